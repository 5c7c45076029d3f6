"""The small-system solver's shared memory at its limits: operators whose
arrays together with the kernels' static variables just exceed what a CTA may
have, and solves of different sizes on several threads at once (the limit that
a launch sets belongs to the process).

FP64 at rtol 1e-10 within 1e-8 of the oracle; the threads' results equal the
one-thread ones."""
import threading

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


def nine_wide(d=20):
    """d = 20, nine complex off-diagonal entries per row of H and one complex
    ladder operator: 232288 bytes of arrays, 160 below 227 KB."""
    H = np.zeros((d, d), dtype=complex)
    for i in range(d):
        for k, v in ((1, 0.2 + 0.1j), (2, 0.1 - 0.05j), (3, 0.05j), (4, 0.04 + 0.02j)):
            H[i, (i + k) % d] += v
            H[(i + k) % d, i] += np.conj(v)
        H[i, (i + 10) % d] = 0.03j if i < 10 else -0.03j
        H[i, i] = 0.1 * i
    return sp.csr_matrix(H), [(0.3 + 0.2j) * S.destroy(d)]


@pytest.mark.parametrize("d", [18, 20, 21])
def test_correlation_at_the_shared_memory_limit(qt, d):
    H, c_ops = nine_wide(20)
    if d != 20:
        H, c_ops = sp.csr_matrix(H[:d, :d]), [(0.3 + 0.2j) * S.destroy(d)]
    a = S.destroy(d)
    psi, t, tau = S.basis(d, 2), [0.0, 0.4], [0.0, 0.3, 0.8]
    if d == 21:  # one more row than the circulant
        H = sp.block_diag([nine_wide(20)[0], sp.csr_matrix([[0.5 + 0j]])], format="csr")
    o = qt.qt_opts_default(rtol=1e-10, atol=1e-12)
    corr, _ = qt.qt_correlation_2op_2t(H, c_ops, S.dag(a), a, psi, t, tau, opts=o)
    ref, _ = oracle.correlation_2op_2t(H, c_ops, S.dag(a), a, psi, t, tau, rtol=1e-10, atol=1e-12)
    assert np.abs(corr - ref).max() < 1e-8


def test_propagator_at_the_shared_memory_limit(qt):
    H, c_ops = nine_wide()
    o = qt.qt_opts_default(rtol=1e-10, atol=1e-12)
    U, _ = qt.qt_propagator(H, c_ops, [0.0, 0.3], opts=o)
    rho = np.outer(S.basis(20, 2), S.basis(20, 2).conj()).astype(complex)
    _, states, _ = oracle.mesolve(H, c_ops, [], rho, [0.0, 0.3], rtol=1e-10, atol=1e-12,
                                  store_states=True)
    assert np.abs((U[1] @ rho.ravel()).reshape(20, 20) - states[1]).max() < 1e-8


def test_sizes_on_several_threads(qt):
    o = qt.qt_opts_default(rtol=1e-8, atol=1e-10)

    def solve(d):
        a = S.destroy(d)
        return qt.qt_mesolve(0.3 * S.num(d) + 0.2 * (a + S.dag(a)), [0.4 * a], [S.num(d)],
                             S.basis(d, 1), [0.0, 0.2], opts=o)[0]

    sizes = [2, 20, 5, 12]  # one CTA each, 13 KB .. 100 KB
    want = {d: solve(d) for d in sizes}
    errors = []

    def work(d):
        try:
            for _ in range(50):
                assert np.array_equal(solve(d), want[d])
        except Exception as e:  # reported by the main thread
            errors.append((d, repr(e)))

    threads = [threading.Thread(target=work, args=(d,)) for d in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
