"""The FP32 block inversion of the reduction at the edges of its block orders: one leaf of each row
group (up to 160 rows), ragged padding, and blocks split once and twice, with blocks that cannot be
inverted without row exchanges."""
import numpy as np
import pytest

from tests.helpers import custom_problem, nasa_const_cp

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 20, 32, 33, 64, 95, 96, 128, 150, 160, 161, 320, 350])
def test_leaf_orders(S):
    """x of a 3-layer system whose diagonal blocks are cyclic shifts within aligned groups of 32 rows
    (zero diagonals) plus noise.  Bound: FP32 rounding (2^-24, a dozen units per product of the split
    tensor-core path) accumulated over the block order, times the system's condition number."""
    from paper_2512_06729_gb300 import xk
    L = 3
    rng = np.random.default_rng(S)
    A = np.zeros((L, S, S))
    for k in range(L):
        for g in range(0, S, 32):
            m = min(32, S - g)
            A[k, g + np.arange(m), g + (np.arange(m) + 1) % m] = rng.uniform(1.0, 2.0, m)
        A[k] += 0.05 / np.sqrt(S) * rng.normal(size=(S, S))
    lo, up = 0.2 * rng.uniform(-1, 1, (L, S)), 0.2 * rng.uniform(-1, 1, (L, S))
    lo[0] = 0.0
    up[-1] = 0.0
    f = rng.normal(size=(L, S))
    M = np.zeros((L * S, L * S))
    for k in range(L):
        M[k * S:(k + 1) * S, k * S:(k + 1) * S] = A[k]
        i = np.arange(S)
        if k:
            M[k * S + i, (k - 1) * S + i] = lo[k]
        if k + 1 < L:
            M[k * S + i, (k + 1) * S + i] = up[k]
    want = np.linalg.solve(M, f.ravel()).reshape(L, S)
    rx = [{"type": 0, "reac": [0], "prod": [S - 1], "arr": [1e-12, 0.0, 0.0]}]
    p = custom_problem(np.ones((S, 1)), np.full(S, 2.0), rx, [nasa_const_cp(2.5, 0.0, 1.0)] * S,
                       np.geomspace(1.0, 1e-2, L), np.full(L, 1000.0), dcoef=np.full(S, 1e17))
    c = xk.Column(p, "mixed")
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    x = c.block_solve32(dev(A), dev(lo), dev(up), dev(f)).cpu().numpy()
    bound = 12 * 2.0 ** -24 * np.sqrt(S) * 4 * np.linalg.cond(M)
    assert np.max(np.abs(x - want)) <= bound * np.max(np.abs(want)), (S, np.max(np.abs(x - want)), bound)
