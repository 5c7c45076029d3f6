"""The adjoint kernels over the operator forms that they treat apart: drives
with a diagonal, complex operators, collapse shapes that are diagonal, real,
complex or with A^dag A off the diagonal, no collapse operator, and initial
matrices that are not Hermitian (all entries instead of the upper triangle);
more steps per segment than the workspace keeps powers for.  Losses and
gradients against the oracle's on the same grid, within 1e-9 of the largest."""
import numpy as np
import pytest
import scipy.sparse as sp

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


def rand(d, rng, herm=False, cplx=True, density=0.4):
    m = rng.standard_normal((d, d)) * (rng.random((d, d)) < density)
    if cplx:
        m = m + 1j * rng.standard_normal((d, d)) * (m != 0)
    return sp.csr_matrix(0.5 * (m + m.conj().T) if herm else m)


@pytest.mark.parametrize("form", ["ladder", "random_real", "random_complex", "no_rates",
                                  "not_hermitian", "many_steps"])
@pytest.mark.parametrize("d", [1, 5, 17])
def test_gradients(qt, form, d):
    rng = np.random.default_rng(d)
    n_seg, batch, t_seg, maxs = 3, 2, 0.5, 64
    cplx = form not in ("ladder", "random_real")
    a = S.destroy(d) if d > 1 else sp.csr_matrix([[0.0]])
    if form == "ladder":
        H0, Hd, A = S.num(d), (a + a.T).tocsr() + 0.1 * S.num(d), [a, S.num(d)]
    else:
        H0, Hd = rand(d, rng, True, cplx), rand(d, rng, True, cplx)
        A = [rand(d, rng, False, cplx), sp.diags(np.exp(1j * np.arange(d))).tocsr()]
    if form == "no_rates":
        A = []
    if form == "many_steps":  # up to 2400 steps a segment at d = 17
        H0, maxs = 40.0 * H0 + 60.0 * S.num(d), 4096
    P1, P2 = rand(d, rng, True), rand(d, rng, True)
    psi = rng.standard_normal(d) + 1j * rng.standard_normal(d)
    if form == "not_hermitian":
        psi = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    adj = qt.Adjoint(H0, Hd, A, P1, P2, psi, n_seg, t_seg, batch, max_per_seg=maxs)
    pr = oracle.AdjointProblem(H0, Hd, A, P1, P2, psi, n_seg, t_seg, max_per_seg=maxs)
    omega = rng.uniform(-0.5, 0.5, (batch, n_seg))
    gamma = rng.uniform(0.0, 0.3, (batch, len(A)))
    t = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")  # noqa: E731
    loss, go = t(np.zeros(batch)), t(np.zeros((batch, n_seg)))
    gg = t(np.zeros((batch, max(len(A), 1))))
    adj.forward(t(omega), t(gamma), qt.qt_opts_default(rtol=1e-7, atol=1e-9), loss)
    adj.backward(None, go, gg)
    torch.cuda.synchronize()
    for b in range(batch):
        ns, hg = adj.grid(b)
        l2, ogo, ogg = pr.grad(omega[b], gamma[b], ns, hg)
        assert abs(l2 - loss[b].item()) <= 1e-9 * max(1.0, abs(l2))
        assert np.abs(go[b].cpu().numpy() - ogo).max() <= 1e-9 * max(1.0, np.abs(ogo).max())
        if A:
            assert np.abs(gg[b].cpu().numpy() - ogg).max() <= 1e-9 * max(1.0, np.abs(ogg).max())
    adj.close()
