"""The analyses at the edges of their work split: equal path lengths, directions without a rate, one
search and as many as there are species to a layer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,layers,nsrc", [(24, 2, 1), (24, 3, 24), (33, 2, 9), (40, 21, 40)])
def test_pathways_ties_bitwise(S, layers, nsrc):
    """Rates of a few powers of two: most path lengths tie, and the tie rules alone decide the tree.
    Both sides add the same IEEE weights in the same order: bit for bit."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column(S=S, L=layers, n_two=2 * S, n_three=S // 2, n_photo=4)
    o, c = Oracle(p), xk.Column(p, "fp64")
    rng = np.random.default_rng(layers)
    q = rng.choice([0.0, 0.25, 0.5, 1.0, 1.0, 1e300], size=(p.L, p.R, 2))
    srcs = list(rng.permutation(p.S)[:nsrc])
    got = {k: v.cpu().numpy() for k, v in c.pathways(torch.as_tensor(q, device="cuda"), srcs).items()}
    for j, s in enumerate(srcs):
        for k in range(p.L):
            ref = o.pathways(q[k], s)
            for key in ("dist", "pred_sp", "pred_edge", "lim_edge", "lim_w"):
                assert np.array_equal(got[key][j, k], ref[key]), (s, k, key)
    c.close()
