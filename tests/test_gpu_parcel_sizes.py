"""The parcel scheme's step at the edges of its kernels' system sizes: one, two and four words of the
vector to a lane, the largest system with its matrices in shared memory and the first without."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [32, 33, 64, 65, 111, 112])
def test_parcel_sizes_match_oracle(S):
    """One iteration over three layers of strong mixing (short visits, which grow a rounding little).
    Bound: 10 x the oracle's own spread under perturbations of 1e-13 relative (at least 1e-9), as for
    the whole columns; step counts agree when the spread's do."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    from tests.test_gpu_parcel import _rel, _spread
    p = synth.small_column(S=S, L=3, n_two=3 * S, n_three=3 * S // 4, n_photo=5, seed=5, W=40,
                           elements="chons" if S < 110 else "full")
    p.Kzz = p.Kzz * 1e8
    o = Oracle(p)
    N0, ngas = o.initial_state(), o.grid()[0]
    ref, spread, hspread, stable = _spread(o, N0, 1e-8, 1, ngas)
    col = xk.Column(p, "fp64")
    col.set_state(N0)
    gi, (N, oi) = col.parcel_iteration(h=1e-8), ref[0]
    if stable:
        assert (gi.steps, gi.rejected) == (oi.steps, oi.rejected)
    assert abs(gi.h - oi.h) <= max(10.0 * hspread, 1e-9) * oi.h
    assert _rel(col.get_state(), N, ngas) <= max(10.0 * spread, 1e-9)
    col.close()
