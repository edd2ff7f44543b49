"""The FP64 block cyclic reduction at the edges of its blocks and levels: rows per lane of the
inversion, odd orders, ragged product tiles, one to all CTAs of a cluster, layer counts around powers
of two, the largest block and the first that takes the elimination from both ends instead."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,L", [(24, 7), (24, 8), (26, 151), (32, 9), (33, 16), (64, 17), (65, 31), (96, 33), (97, 64),
                                 (128, 10), (129, 9), (152, 12), (153, 12)])
@pytest.mark.parametrize("dt", [1e-8, 1e-2])
def test_reduction_solves_the_step(S, L, dt):
    """The factors are those of the system, so that the refinement around them ends after a few
    iterations at the residual of FP64 (1e-13 of the right-hand side, a thousand roundings), and the
    step is the one the sequential elimination finds, to the system's conditioning: with steps this
    short below 1e9 on these columns, 1e9 x 1e-15 in the 2-norm."""
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column(S=S, L=L, n_two=2 * S, n_three=S // 2, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    a, b = xk.Column(p, "fp64"), xk.Column(p, "fp64", twisted=0)
    a.set_mixing_ratios(p.f0)
    n = a.get_state(device=True)
    got, iters, resid = a.step_delta(n, dt)
    want, _, _ = b.step_delta(n, dt)
    assert iters <= 4 and resid <= 1e-13
    assert float(torch.linalg.norm(got - want) / torch.linalg.norm(want)) <= 1e-6
    a.close()
    b.close()
