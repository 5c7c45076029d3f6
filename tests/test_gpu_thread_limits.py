"""Solves of one size while another thread calls the same kernels' entry points
for other sizes: the shared-memory limit of a kernel belongs to the process,
so a caller that sets its own size would have the first thread's launch
refused.  The other thread's calls launch nothing (they are refused for their
size, after the launch has been sized) or launch an ordinary kernel."""
import threading

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


def beside(other, solve, n):
    """solve() n times while other() runs again and again on three threads."""
    stop, errors = threading.Event(), []

    def loop():
        try:
            while not stop.is_set():
                other()
        except Exception as e:  # reported below
            errors.append(e)

    threads = [threading.Thread(target=loop) for _ in range(3)]
    for t in threads:
        t.start()
    try:
        out = [solve() for _ in range(n)]
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert not errors, errors
    return out


def test_steady_state_beside_a_refused_one(qt):
    k = S.kerr_cavity(N=4)
    small = qt.System(k["H"], k["c_ops"], [])
    rho = torch.zeros((4, 4), dtype=torch.complex128, device="cuda")

    def refused():  # krylov_dim 4096 takes more shared memory than a CTA has
        with pytest.raises(qt.QtError) as e:
            small.qt_steadystate_dev(rho, krylov_dim=4096)
        assert e.value.code == qt.QT_ENOTIMPL

    want = qt.qt_steadystate(k["H"], k["c_ops"])[0]
    for got in beside(refused, lambda: qt.qt_steadystate(k["H"], k["c_ops"])[0], 500):
        assert np.array_equal(got, want)


def test_hermitian_solve_beside_a_refused_one(qt):
    d = 70
    a = S.destroy(d)
    args = (0.3 * S.num(d) + 0.2 * (a + S.dag(a)), [0.3 * a, 0.1 * S.num(d)], [S.num(d)],
            S.basis(d, 1), [0.0, 0.05])
    large = qt.System(sp.identity(600, dtype=complex, format="csr"), [], [])
    z = torch.zeros(600, dtype=torch.complex128, device="cuda")
    tl = torch.zeros(1, dtype=torch.float64, device="cuda")
    o = qt.qt_opts_default()

    def refused():  # larger than the preallocated workspace
        with pytest.raises(qt.QtError) as e:
            large.qt_mesolve_dev_noalloc(z, tl, o, z)
        assert e.value.code == qt.QT_EINVAL

    want = qt.qt_mesolve(*args, opts=o)[0]
    for got in beside(refused, lambda: qt.qt_mesolve(*args, opts=o)[0], 200):
        assert np.array_equal(got, want)


def test_trajectories_of_two_sizes(qt):
    def problem(d, w):  # H with 2 w off-diagonal entries a row, 40 distinct values
        H = sp.lil_matrix((d, d), dtype=complex)
        for i in range(d):
            H[i, i] = i / d
            for k in range(1, w + 1):
                j = (i + k) % d
                H[i, j] = H[j, i] = 0.01 * (1 + (7 * i + k) % 40)
        return (sp.csr_matrix(H), [sp.diags([np.full(d - 1, 0.2)], [1], format="csr", dtype=complex)],
                [sp.diags([np.arange(d, dtype=complex)], [0], format="csr")], S.basis(d, 3),
                [0.0, 0.1], 16)

    big, small = problem(500, 18), problem(300, 22)  # 80 KB and 60 KB of operator codes
    o = qt.qt_opts_default(rtol=1e-6, atol=1e-8, precision=qt.QT_MIXED)
    run = lambda p: qt.qt_mcsolve(*p, seed=5, opts=o)[0]  # noqa: E731
    want = run(big), run(small)
    got = beside(lambda: run(small), lambda: run(big), 200)
    for g in got:  # the sums over trajectories are taken in any order
        assert np.allclose(g, want[0], rtol=1e-12, atol=1e-12)
    assert np.allclose(run(small), want[1], rtol=1e-12, atol=1e-12)
