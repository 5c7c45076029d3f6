"""The propagator of a resident system that holds observables (they take no
part in it): the entries of the same system without them, bit for bit, from
the small-system solver (ladder operators), from the general one (a
time-dependent term), and from both precisions."""
import numpy as np
import pytest

from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("driven", [False, True])
@pytest.mark.parametrize("n_e", [1, 3, 9])
def test_observables_take_no_part(qt, n_e, driven, precision):
    d = 6
    a = S.destroy(d)
    td = [(a + S.dag(a), np.array([0.0, 1.0]), np.array([0.0, 0.7]))] if driven else None
    o = qt.qt_opts_default(rtol=1e-6, atol=1e-8,
                           precision=qt.QT_MIXED if precision == "mixed" else qt.QT_FP64)
    tl = torch.tensor([0.0, 0.4, 1.0], dtype=torch.float64, device="cuda")
    out = []
    for e_ops in ([], [S.num(d)] * n_e):
        sysm = qt.System(0.3 * S.num(d) + 0.2 * (a + S.dag(a)), [0.4 * a], e_ops, td=td)
        U = torch.zeros((3, d * d, d * d), dtype=torch.complex128, device="cuda")
        stb = torch.zeros(56, dtype=torch.uint8, device="cuda")
        sysm.qt_propagator_dev(tl, o, U, stats=stb)
        torch.cuda.synchronize()
        assert qt.stats_from_bytes(stb)["status"] == 0
        out.append(U.cpu().numpy())
        sysm.close()
    assert np.array_equal(out[0], out[1]) and np.abs(out[0][2]).max() > 0.5
