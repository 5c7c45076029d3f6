"""Vectors whose forward solve ends early: their loss and gradients are NaN,
their grid holds the completed segments only, and the other vectors of the
batch are those of a batch of their own (bit for bit: a CTA per vector)."""
import numpy as np
import pytest

from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N_SEG = 4


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


def dev(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def handle(qt, batch, max_per_seg):
    s = S.transmon_cavity(N=3, n_seg=N_SEG)
    return qt.Adjoint(s["H0"], s["Hd"], s["A"], s["P1"], s["P2"], s["psi0"], N_SEG, s["t_seg"],
                      batch, max_per_seg=max_per_seg), s["gamma"]


def passes(qt, adj, omega, gamma):
    """Status, and loss, fixed-grid loss and gradients of one round of calls."""
    n = len(omega)
    om, ga = dev(omega), dev(gamma)
    loss, fixed = dev(np.zeros(n)), dev(np.zeros(n))
    go, gg = dev(np.zeros((n, N_SEG))), dev(np.zeros((n, len(gamma[0]))))
    stb = torch.zeros(56, dtype=torch.uint8, device="cuda")
    adj.forward(om, ga, qt.qt_opts_default(), loss, stats=stb)
    adj.loss_fixed(om, ga, fixed)
    adj.backward(None, go, gg)
    torch.cuda.synchronize()
    return qt.stats_from_bytes(stb)["status"], [x.cpu().numpy() for x in (loss, fixed, go, gg)]


def test_step_limit_of_a_segment(qt):
    # a drive of 1 takes a few steps a segment, one of 30 in the third segment many
    omega = np.full((3, N_SEG), 1.0)
    omega[1, 2] = 30.0
    free, gamma = handle(qt, 3, 4096)
    gamma = np.tile(gamma, (3, 1))
    status, _ = passes(qt, free, omega, gamma)
    assert status == 0
    ns = np.array([free.grid(b)[0] for b in range(3)])
    limit = int(ns[0].max())
    assert ns[1, :2].max() <= limit < ns[1, 2]
    adj, _ = handle(qt, 3, limit)
    want = passes(qt, adj, np.ones((3, N_SEG)), gamma)  # a full grid is recorded first
    assert want[0] == 0
    for _ in range(2):
        status, got = passes(qt, adj, omega, gamma)
        assert status == qt.QT_ESTEP
        for g, w in zip(got, want[1]):
            assert np.isnan(g[1]).all() and np.array_equal(g[[0, 2]], w[[0, 2]])
        assert list(adj.grid(1)[0]) == [ns[1, 0], ns[1, 1], 0, 0]
    fresh, _ = handle(qt, 3, limit)  # no grid before
    status, got = passes(qt, fresh, omega, gamma)
    assert status == qt.QT_ESTEP and all(np.isnan(g[1]).all() for g in got)
    # and the handle still solves what it can
    status, again = passes(qt, adj, np.ones((3, N_SEG)), gamma)
    assert status == 0 and all(np.array_equal(g, w) for g, w in zip(again, want[1]))


def test_autograd_with_a_parameter_that_is_not_finite(qt):
    adj, gamma = handle(qt, 2, 64)
    om = np.ones((2, N_SEG))
    om[0, 1] = np.nan
    om, ga = dev(om).requires_grad_(True), dev(np.tile(gamma, (2, 1))).requires_grad_(True)
    loss = qt.master_equation_loss(adj, om, ga, qt.qt_opts_default())
    loss.sum().backward()
    for t in (loss.detach(), om.grad, ga.grad):
        t = t.cpu().numpy()
        assert np.isnan(t[0]).all() and np.isfinite(t[1]).all()
