"""Where the batched kernel keeps a master-equation problem: entry arrays in
shared memory, in the workspace, or (more than 64 terms per entry) the general
solver; kets and matrices, sizes on both sides of each limit, interleaved with
Monte-Carlo problems that use the same shared memory.  Against the oracle, per
observable entry: FP64 at rtol 1e-10 within 1e-8; mixed at rtol 1e-6 within 1e-5
(the solve's tolerance over |H| t of a few, and FP32 rounding).  Monte-Carlo
problems without collapse operators are deterministic."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_1110_0573_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TL = np.array([0.0, 0.3, 0.8])


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


def system(d, k):
    """k off-diagonal entries of H to each side, a ladder collapse operator."""
    H = np.diag(np.linspace(0.0, 1.0, d)).astype(complex)
    for o in range(1, k + 1):
        for i in range(d - o):
            H[i, i + o], H[i + o, i] = 0.2 / k + 0.1j / o, 0.2 / k - 0.1j / o
    return sp.csr_matrix(H), [0.3 * S.destroy(d)], [S.num(d) / d]


def me(d, k, ket):
    H, C, E = system(d, k)
    psi = np.ones(d) / np.sqrt(d)
    return dict(H=H, c_ops=C, e_ops=E, kind="me", state0=psi if ket else np.outer(psi, psi))


def mc(d, dense):
    H, _, E = system(d, 1)
    if dense:  # wide operators: the master equations' arrays go to the workspace
        E = E + [sp.csr_matrix(np.add.outer(np.arange(d), np.arange(d)) / d ** 2)]
    return dict(H=H, c_ops=[0.0 * S.destroy(d)], e_ops=E, kind="mc",
                state0=np.ones(d) / np.sqrt(d), ntraj=4, seed=3)


MES = [(2, 1), (16, 1), (31, 1), (32, 1), (33, 1), (40, 3), (64, 1), (64, 8), (40, 20)]


def solve(qt, problems, precision):
    o = (qt.qt_opts_default(rtol=1e-10, atol=1e-12) if precision == "fp64" else
         qt.qt_opts_default(rtol=1e-6, atol=1e-8, precision=qt.QT_MIXED))
    b = qt.Batch(problems)
    ex = torch.zeros(len(TL) * sum(b.n_e), dtype=torch.complex128, device="cuda")
    stb = torch.zeros(56, dtype=torch.uint8, device="cuda")
    b.qt_batch_solve_dev(torch.tensor(TL, device="cuda"), o, ex, stats=stb)
    torch.cuda.synchronize()
    assert qt.stats_from_bytes(stb)["status"] == 0
    out = b.split(ex.cpu().numpy(), len(TL))
    b.close()
    return out


def reference(p, cache={}):
    key = (p["kind"], p["H"].shape[0], p["H"].nnz, np.ndim(p["state0"]), len(p["e_ops"]))
    if key not in cache:
        cache[key] = oracle.mesolve(p["H"], p["c_ops"], p["e_ops"], p["state0"], TL, rtol=1e-10,
                                    atol=1e-12)[0]
    return cache[key]


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-8), ("mixed", 1e-5)])
@pytest.mark.parametrize("mix", ["alone", "together", "beside_trajectories", "beside_wide"])
def test_placements(qt, mix, precision, tol):
    mes = [me(d, k, ket) for d, k in MES for ket in (True, False)]
    if mix == "alone":  # each problem's own launch size
        batches = [[m] for m in mes]
    elif mix == "together":
        batches = [mes]
    else:
        mcs = [mc(d, mix == "beside_wide") for d in (4, 32, 64)]
        batches = [[m for q in range(len(mes)) for m in (mes[q], mcs[q % 3])]]
    for batch in batches:
        for p, got in zip(batch, solve(qt, batch, precision)):
            assert np.abs(got - reference(p)).max() < tol, (p["kind"], p["H"].shape, p["H"].nnz)
