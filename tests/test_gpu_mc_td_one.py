"""The mixed Monte-Carlo instances for one narrow time-dependent term against
the general time-dependent instances (the same term and a second, zero one):
the same trajectories bit for bit, at the sizes where the instances change,
with knots inside steps, before and after the interval."""
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


def trajectories(qt, s, td):
    sysm = qt.System(s["H"], s["c_ops"], s["e_ops"], td=td)
    n, nt = 40, len(s["tlist"])
    dev = torch.device("cuda", 0)
    tex = torch.zeros((n, nt, 2), dtype=torch.complex128, device=dev)
    es = torch.zeros((nt, 2), dtype=torch.complex128, device=dev)
    o = qt.qt_opts_default(rtol=1e-6, atol=1e-8, precision=qt.QT_MIXED)
    sysm.qt_mcsolve_dev(torch.tensor(s["psi0"], dtype=torch.complex128, device=dev),
                        torch.tensor(s["tlist"], dtype=torch.float64, device=dev), n, 7, o, es,
                        traj_expect=tex)
    torch.cuda.synchronize()
    sysm.close()
    return tex.cpu().numpy()


@pytest.mark.parametrize("d", [2, 20, 32, 33, 64, 65, 128])
@pytest.mark.parametrize("width", [1, 2])
@pytest.mark.parametrize("wide_h", [False, True])  # H_eff of three or four slots
def test_same_as_general_instance(qt, d, width, wide_h):
    s = S.kerr_cavity(N=d, E=0.3, t_end=3.0, nt=11)
    a = S.destroy(d)
    if wide_h and d > 3:
        s["H"] = s["H"] + sp.diags([0.05, 0.05], [d - 1, 1 - d], shape=(d, d))
    H1 = S.num(d) if width == 1 else (a + S.dag(a)).tocsr()
    knots = (np.array([0.5, 0.77, 1.9, 2.3]), np.array([0.0, 0.8, -0.5, 0.4]))
    zero = (sp.csr_matrix((d, d), dtype=complex), np.array([0.0, 1.0]), np.array([1.0, 2.0]))
    one = trajectories(qt, s, [(H1, *knots)])
    gen = trajectories(qt, s, [(H1, *knots), zero])
    assert np.isfinite(one).all() and np.array_equal(one, gen)
