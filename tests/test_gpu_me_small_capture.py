"""Solves of every form of a small system after one ket solve on the same
handle: no further device memory (they can be captured, which allocating and
freeing cannot), and the replayed results are those of the direct calls."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


def wide(d, k):
    """k off-diagonal entries to each side of the diagonal of H."""
    H = np.diag(np.linspace(0.0, 1.0, d)).astype(complex)
    for o in range(1, k + 1):
        v = 0.1 / o + 0.02j * o
        for i in range(d - o):
            H[i, i + o], H[i + o, i] = v, np.conj(v)
    return sp.csr_matrix(H)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("d,k", [(16, 1), (23, 1), (40, 1), (40, 5), (60, 1), (64, 5)])
def test_forms_share_one_workspace(qt, d, k, precision):
    prec = qt.QT_MIXED if precision == "mixed" else qt.QT_FP64
    sysm = qt.System(wide(d, k), [0.3 * S.destroy(d)], [S.num(d)])
    tl = torch.tensor([0.0, 0.2, 0.5], dtype=torch.float64, device="cuda")
    ket = torch.tensor(S.basis(d, 1), dtype=torch.complex128, device="cuda")
    mat = torch.outer(ket, ket.conj()).contiguous()

    def solve(state, method, out):
        o = qt.qt_opts_default(rtol=1e-6, atol=1e-8, precision=prec, me_method=method)
        sysm.qt_mesolve_dev(state, tl, o, out)

    forms = [(ket, qt.QT_ME_AUTO), (mat, qt.QT_ME_AUTO), (ket, qt.QT_ME_SPARSE),
             (mat, qt.QT_ME_SPARSE)]
    new = lambda: torch.zeros((3, 1), dtype=torch.complex128, device="cuda")  # noqa: E731
    solve(*forms[0], new())
    torch.cuda.synchronize()
    graphs, got = [], [new() for _ in forms]
    for f, out in zip(forms, got):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            solve(*f, out)
        graphs.append(g)
    for g in graphs:
        g.replay()
    torch.cuda.synchronize()
    want = [new() for _ in forms]
    for f, out in zip(forms, want):
        solve(*f, out)
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b) and abs(a[0, 0].item() - 1.0) < 1e-6
    sysm.close()
