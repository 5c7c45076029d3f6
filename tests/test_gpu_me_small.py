"""The small-system master-equation solver (dim <= 64) at the sizes where its
layout changes: one CTA up to 256 entries, clusters of 4 and 8 above; the
upper triangle (kets) and all entries (matrices, QT_ME_SPARSE); real and
complex operators; entry arrays in shared memory and in the workspace; and
operators with more terms than it takes (the general solver).

FP64 against the oracle within 1e-8 at rtol 1e-9 with its step counts (to 2);
mixed within 1e-5 (the mixed path's stated bound)."""
import numpy as np
import pytest

import oracle
from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


def system(kind, d):
    if kind == "real":  # a ladder with hopping, decay and dephasing: real terms
        a = S.destroy(d)
        return dict(H=0.3 * S.num(d) + 0.2 * (a + S.dag(a)), psi0=S.basis(d, min(d - 1, 2)),
                    c_ops=[0.4 * a, 0.1 * S.num(d) / d, 0.2 * S.dag(a)],
                    e_ops=[S.num(d), a], tlist=np.linspace(-0.5, 1.5, 5))
    s = S.random_system(d, 2, 2, seed=d, density=min(1.0, (2.0 if kind == "complex" else 16.0) / d),
                        nt=4, t_end=0.5)
    return s


@pytest.mark.parametrize("kind,d", [("real", 1), ("real", 2), ("real", 22), ("real", 23),
                                    ("real", 44), ("real", 45), ("real", 64), ("complex", 9),
                                    ("complex", 33), ("complex", 64), ("wide", 40)])
@pytest.mark.parametrize("form", ["ket", "matrix", "sparse"])
def test_fp64(qt, kind, d, form):
    s = system(kind, d)
    psi = s["psi0"] / np.linalg.norm(s["psi0"])
    st0 = np.outer(psi, psi.conj()) if form == "matrix" else psi
    o = qt.qt_opts_default(rtol=1e-9, atol=1e-11,
                           me_method=qt.QT_ME_SPARSE if form == "sparse" else qt.QT_ME_AUTO)
    ex, states, st = qt.qt_mesolve(s["H"], s["c_ops"], s["e_ops"], st0, s["tlist"], opts=o,
                                   store_states=True)
    ref, rstates, rst = oracle.mesolve(s["H"], s["c_ops"], s["e_ops"], psi, s["tlist"], rtol=1e-9,
                                       atol=1e-11, store_states=True)
    assert np.abs(ex - ref).max() < 1e-8
    assert np.abs(states - rstates).max() < 1e-8
    assert abs(st["accepted"] - rst["accepted"]) <= 2


@pytest.mark.parametrize("kind,d", [("real", 2), ("real", 22), ("real", 45), ("real", 64),
                                    ("complex", 33), ("complex", 64)])
def test_mixed(qt, kind, d):
    s = system(kind, d)
    o = qt.qt_opts_default(rtol=1e-6, atol=1e-8, precision=qt.QT_MIXED)
    ex, _, _ = qt.qt_mesolve(s["H"], s["c_ops"], s["e_ops"], s["psi0"], s["tlist"], opts=o)
    ref, _, _ = oracle.mesolve(s["H"], s["c_ops"], s["e_ops"], s["psi0"], s["tlist"], rtol=1e-6,
                               atol=1e-8)
    assert np.abs(ex - ref).max() < 1e-5


def test_output_times_that_do_not_advance(qt):
    """Device calls do not check the time list: an output time that is not
    ahead is written from the state already reached."""
    s = system("real", 6)
    dev = torch.device("cuda", 0)
    sysm = qt.System(s["H"], s["c_ops"], s["e_ops"])
    psi = torch.tensor(s["psi0"], dtype=torch.complex128, device=dev)
    tl = torch.tensor([0.0, 0.5, 0.5, 0.25, 1.0], dtype=torch.float64, device=dev)
    ex = torch.zeros((5, 2), dtype=torch.complex128, device=dev)
    sysm.qt_mesolve_dev(psi, tl, qt.qt_opts_default(), ex)
    torch.cuda.synchronize()
    ex = ex.cpu().numpy()
    sysm.close()
    assert np.array_equal(ex[1], ex[2]) and np.array_equal(ex[1], ex[3])
    assert np.abs(ex[4] - ex[3]).max() > 1e-3
