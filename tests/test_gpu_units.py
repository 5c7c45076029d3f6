"""FP64 solves in extreme units: a generator s L over times t / s is the same
problem for every s.  A step's powers h^k and L^k v leave the FP64 range from
about s = 1e51 (or 1e-51) on, beyond 2^128 the kernels scale them.  Results
within 1e-8 of the solve at s = 1 (rtol 1e-10 on both sides, over |L| t of a
few; the grids differ only by the fixed constants of the first step)."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SCALES = [1e-60, 1e-45, 1e-38, 1e38, 1e45, 1e60]
TOL = 1e-8


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


def opts(qt, s):  # a first step in the units of the problem
    return qt.qt_opts_default(rtol=1e-10, atol=1e-12, h0=1e-3 / s)


def model(d, s):
    a = S.destroy(d)
    H = sp.csr_matrix(sp.diags([np.linspace(0.0, 1.0, d)], [0]) + 0.3 * (a + S.dag(a)))
    return H * s, [np.sqrt(0.2 * s) * a]


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("d,ket", [(5, True), (5, False), (30, True)])  # one CTA, and a cluster
def test_master_equation(qt, d, ket, s):
    psi = np.ones(d) / np.sqrt(d)
    state = psi if ket else np.outer(psi, psi)
    t = np.array([0.0, 0.7, 1.5])
    sol = [qt.qt_mesolve(*model(d, x), [S.num(d)], state, t / x, opts=opts(qt, x),
                         store_states=True)[1] for x in (1.0, s)]
    assert np.abs(sol[1] - sol[0]).max() < TOL


@pytest.mark.parametrize("s", SCALES)
def test_correlation(qt, s):
    d, t = 4, np.array([0.0, 0.5])
    a = S.destroy(d)
    corr = [qt.qt_correlation_2op_2t(*model(d, x), S.dag(a), a, S.basis(d, 2), t / x, t / x,
                                     opts=opts(qt, x))[0] for x in (1.0, s)]
    assert np.abs(corr[1] - corr[0]).max() < TOL


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("d", [5, 60, 150])
def test_trajectory(qt, d, s):
    psi, t = np.ones(d) / np.sqrt(d), np.array([0.0, 0.7, 1.5])
    out = [qt.qt_mcsolve(model(d, x)[0], [], [S.num(d) / d], psi, t / x, 1, opts=opts(qt, x))[0]
           for x in (1.0, s)]
    assert np.abs(out[1] - out[0]).max() < TOL


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("hermitian", [True, False])
def test_adjoint(qt, hermitian, s):
    """Loss and gradients (with respect to omega and gamma in units of s)."""
    d, n_seg, t_seg = 4, 3, 0.4
    a = S.destroy(d)
    rho = np.outer(np.ones(d), np.ones(d)).astype(complex) / d
    if not hermitian:
        rho[0, 1] += 0.2j
    res = []
    for x in (1.0, s):
        adj = qt.Adjoint(S.num(d) * x, (a + S.dag(a)) * x, [a * np.sqrt(x), S.num(d) * np.sqrt(x)],
                         S.num(d), S.num(d) * x, rho, n_seg, t_seg / x, 1, max_per_seg=512)
        om = torch.tensor([[0.3, -0.2, 0.5]], dtype=torch.float64, device="cuda")
        ga = torch.tensor([[0.2, 0.1]], dtype=torch.float64, device="cuda")
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        fixed, go, gg = torch.zeros_like(loss), torch.zeros_like(om), torch.zeros_like(ga)
        adj.forward(om, ga, qt.qt_opts_default(rtol=1e-10, atol=1e-12), loss)
        adj.loss_fixed(om, ga, fixed)
        adj.backward(None, go, gg)
        torch.cuda.synchronize()
        res.append(np.concatenate([v.cpu().numpy().ravel() for v in (loss, fixed, go, gg)]))
    assert np.abs(res[1] - res[0]).max() < TOL
