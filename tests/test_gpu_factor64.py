"""The FP64 block elimination on few CTAs: columns too many for shared memory, panels of one CTA and of
clusters, one and two panel rows to a thread, one chain and two, ragged last panels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _system(S, L, seed):
    """Blocks 3 I + N / sqrt(S) with their rows shuffled (singular values of 1 to 5, every pivot off the
    diagonal), couplings of 0.3."""
    rng = np.random.default_rng(seed)
    A = np.empty((L, S, S))
    lo, up = np.zeros((L, S)), np.zeros((L, S))
    for k in range(L):
        A[k] = (3.0 * np.eye(S) + rng.normal(size=(S, S)) / np.sqrt(S))[rng.permutation(S)]
        if k > 0:
            lo[k] = 0.3 * rng.uniform(-1.0, 1.0, S)
        if k + 1 < L:
            up[k] = 0.3 * rng.uniform(-1.0, 1.0, S)
    return A, lo, up, rng.normal(size=(L, S))


# (species, layers, CTAs): on 1 to 3 CTAs the matrix in global memory; 4 at 40 species keep their columns;
# 594 species on the CTAs of a batch's slots: clusters of 4, 2 and 1 (two rows to a thread above 512)
@pytest.mark.parametrize("S,L,ctas", [(33, 5, 1), (33, 5, 2), (33, 5, 3), (40, 4, 1), (40, 4, 2), (40, 4, 3), (40, 4, 4),
                                      (40, 4, 8), (250, 4, 4), (250, 4, 9), (594, 4, 38), (594, 4, 19), (594, 3, 9),
                                      (594, 3, 6), (594, 3, 4), (594, 3, 2), (400, 3, 8), (400, 3, 16),
                                      (513, 3, 1), (520, 3, 3), (1024, 3, 2)])
@pytest.mark.parametrize("twisted", [0, 1])
def test_elimination_on_few_ctas(S, L, ctas, twisted):
    """Bound: 100 S roundings of the largest entry, for a system whose condition number is some tens and
    whose eliminated blocks stay as well conditioned as the given ones."""
    from paper_2512_06729_gb300 import synth, xk
    from tests.helpers import independent_block_solve
    p = synth.small_column(S=S, L=L, n_two=2 * S, n_three=S // 2, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    col = xk.Column(p, "fp64", factor_ctas=ctas, twisted=twisted)
    A, lo, up, f = _system(S, L, 7 * S + ctas)
    want = independent_block_solve(A, lo, up, f)
    dev = [torch.as_tensor(a, device="cuda") for a in (A, lo, up, f)]
    for _ in range(2):                           # the barrier words and flags are clean again
        got = col.block_solve(*dev).cpu().numpy()
        assert np.max(np.abs(got - want)) <= 100 * S * 2.0 ** -53 * np.max(np.abs(want))
    col.close()
