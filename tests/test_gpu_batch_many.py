"""Batches of more columns than the device has connections for graphs with conditional nodes: every
step's parts are captured without them, and each column still ends where it ends alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_columns_end_where_they_end_alone(precision):
    """Twelve columns to steady state, through late steps (the mixed path's FP64 route among them): 1e-9
    relative on species above 1e-20 mixing ratio, as for batches of up to eight."""
    from paper_2512_06729_gb300 import xk
    from tests.test_gpu_batch import _alone, _problems
    probs = _problems()
    b = xk.Batch(64 << 30, 12)
    cols, slots = [], []
    for i in range(12):
        c = xk.Column(probs[i % 4], precision)
        c.set_mixing_ratios(probs[i % 4].f0)
        slots.append(b.add(c, 1e-8))
        cols.append(c)
    for _ in range(400):
        b.step(8)
        if all(b.poll(s)[1] for s in slots):
            break
    alone = [_alone(p, precision, b.poll(s)[0].steps) for p, s in zip(probs, slots)]
    for i, s in enumerate(slots):
        info, finished, status = b.poll(s)
        assert finished and status == 0
        n_alone, ainfo = alone[i % 4]
        n = b.remove(s).get_state()
        assert info.steps == ainfo.steps
        mask = n_alone > 1e-20 * n_alone.max(axis=1, keepdims=True)
        assert np.max(np.abs(n[mask] - n_alone[mask]) / n_alone[mask]) <= 1e-9
    b.close()


def test_column_off_the_reduction_ends_where_it_ends_alone():
    """A column of 120 species takes the block elimination in a batch of twelve slots and the reduction
    alone: the same steps, and the same steady state to 1e-9."""
    from paper_2512_06729_gb300 import synth, xk
    from tests.test_gpu_batch import _alone
    p = synth.small_column(S=120, L=20, n_two=960, n_three=240, n_photo=40, W=100, elements="full")
    b = xk.Batch(64 << 30, 12)
    cols = [xk.Column(p, "fp64") for _ in range(2)]
    for c in cols:
        c.set_mixing_ratios(p.f0)
    slots = [b.add(c, 1e-8) for c in cols]
    for _ in range(400):
        b.step(8)
        if all(b.poll(s)[1] for s in slots):
            break
    info, finished, status = b.poll(slots[0])
    assert finished and status == 0
    n_alone, ainfo = _alone(p, "fp64", info.steps)
    assert ainfo.steps == info.steps
    mask = n_alone > 1e-20 * n_alone.max(axis=1, keepdims=True)
    for s in slots:
        n = b.remove(s).get_state()
        assert np.max(np.abs(n[mask] - n_alone[mask]) / n_alone[mask]) <= 1e-9
    b.close()
