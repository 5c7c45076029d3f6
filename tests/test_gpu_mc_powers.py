"""The FP64 Monte-Carlo step in powers of H_eff at the sizes where its instances
change (rows per lane 1, 2, 4 and whole CTAs; H_eff in registers or not), with
real and complex off-diagonal entries: jump records as the oracle's, times
within 1e-10 max(1, |tau|) (the search's bracket), values within 1e-8."""
import numpy as np
import pytest

import oracle
from paper_1110_0573_gb300 import systems as S
from tests.parity import compare_jump_records

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


@pytest.mark.parametrize("d", [2, 32, 33, 64, 65, 128, 129])
@pytest.mark.parametrize("phase", [1.0, 1j])
@pytest.mark.parametrize("reach", [1, 3])
def test_fp64_ladder(qt, d, phase, reach):
    a = S.destroy(d)
    hop = sum((phase / (k + 1)) * a ** (k + 1) / d ** (k / 2) for k in range(min(reach, d - 1)))
    H = 0.2 * S.num(d) + 0.3 * (hop + hop.conj().T)
    c_ops = [0.5 * a, 0.2 * S.dag(a) / np.sqrt(d)]
    e_ops, psi0, tl = [S.num(d) / d, a], S.basis(d, min(2, d - 1)), np.linspace(0.0, 2.0, 9)
    o = qt.qt_opts_default(rtol=1e-8, atol=1e-10)
    _, tex, jumps, _ = qt.qt_mcsolve(H, c_ops, e_ops, psi0, tl, 24, seed=d, opts=o, traj_expect=True)
    otex, ojumps, _ = oracle.mcsolve(H, c_ops, e_ops, psi0, tl, 24, seed=d, rtol=1e-8, atol=1e-10)
    n, _ = compare_jump_records(jumps, ojumps, range(24), 2e-10, honour_degenerate=False)
    assert n > 0
    assert np.abs(tex - otex).max() < 1e-8
