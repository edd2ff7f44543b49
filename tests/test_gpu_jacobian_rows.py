"""Jacobian rows of every shape the assembly tells apart: entries of few and of many terms, rows of one
tile and of several, more long entries than a warp has lanes."""
import numpy as np
import pytest

from tests.helpers import custom_problem, nasa_const_cp

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _network(S, R, hubs, seed):
    """A + B -> C + D with a random hub in the first place and random others, equal masses."""
    rng = np.random.default_rng(seed)
    rx = []
    for _ in range(R):
        b, c, d = rng.integers(hubs, S, 3)
        rx.append(dict(type=0, reac=[int(rng.integers(hubs)), int(b)], prod=[int(c), int(d)],
                       arr=[10.0 ** rng.uniform(-14, -10), rng.uniform(-1, 1), rng.uniform(0, 500)]))
    nasa = [nasa_const_cp(2.5 + 0.1 * rng.uniform(), rng.uniform(-1e3, 1e3), rng.uniform(0, 5)) for _ in range(S)]
    return custom_problem(np.ones((S, 1), int), np.full(S, 2.0), rx, nasa, [1.0, 0.1, 1e-3], [1200.0, 1000.0, 800.0],
                          f0=rng.uniform(0.1, 1.0, (3, S)) / S)


@pytest.mark.parametrize("S,R,hubs", [(33, 40, 1), (40, 127, 1), (40, 129, 1), (64, 1024, 1), (64, 1025, 1), (24, 2100, 2),
                                      (80, 3300, 40)])
def test_jacobian_rows(S, R, hubs):
    """Against the oracle, to 1e-12 of the row's largest entry: up to 2,100 terms of either sign in an
    entry, each rounded to 1.1e-16 and added in another order (2,100 x 2.2e-16 = 4.6e-13)."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import xk
    p = _network(S, R, hubs, S + R)
    o, c = Oracle(p), xk.Column(p, "fp64")
    n = o.initial_state()
    A = c.eval_jacobian(torch.as_tensor(n, device="cuda"), 1e-3)[0].cpu().numpy()
    want = o.jacobian(n, 1e-3)[0]
    assert np.max(np.abs(A - want) / np.abs(want).max(axis=2, keepdims=True)) < 1e-12
    c.close()
