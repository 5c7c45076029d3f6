"""The GMRES steady state where its sums change: fewer entries than CTAs, a
warp's width of entries per CTA and more than that, and a Krylov space as large
as the problem.  The residual |L rho| (dense, FP64, numpy) stays within the
solver's tolerance 1e-12 of |w I|, w the mean |diagonal of L|, times 100 for
the forming of rho (Hermitian part, unit trace)."""
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


@pytest.mark.parametrize("N,krylov", [(2, 4), (3, 0), (12, 144), (12, 0), (40, 0), (69, 0), (70, 0)])
def test_residual(qt, N, krylov):
    s = S.kerr_cavity(N=N)
    rho, info, _ = qt.qt_steadystate(s["H"], s["c_ops"], krylov_dim=krylov)
    H = s["H"].toarray()
    C = [c.toarray() for c in s["c_ops"]]
    heff = H - 0.5j * sum(c.conj().T @ c for c in C)
    L = -1j * (heff @ rho - rho @ heff.conj().T) + sum(c @ rho @ c.conj().T for c in C)
    assert abs(np.trace(rho) - 1) < 1e-12 and np.abs(rho - rho.conj().T).max() == 0.0
    assert np.linalg.norm(L) <= 100 * 1e-12 * info["w"] * np.sqrt(N)
