"""Photolysis rates at the edges of the kernels' tiles: layers and reactions per block, runs of
wavelengths, layers read ahead, direct beam and diffuse field."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,n_photo,W", [(2, 1, 2), (3, 7, 31), (4, 8, 33), (5, 9, 127), (17, 10, 129), (33, 6, 300)])
@pytest.mark.parametrize("diffuse", [0, 1])
def test_photolysis_edges(layers, n_photo, W, diffuse):
    """1e-11 relative: the same exponentials and sums on both sides up to their order, up to 300 terms
    of one sign (300 x 1.1e-16), through optical depths of some hundreds (their rounding times the depth)."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column(S=40, L=layers, n_photo=n_photo, W=W)
    p = synth.with_scattering(p, albedo=0.3, diffuse=diffuse)
    o, c = Oracle(p), xk.Column(p, "fp64")
    n = o.initial_state()
    kph = c.eval_photolysis(torch.as_tensor(n, device="cuda")).cpu().numpy()
    ref = o.photolysis(n)
    m = ref > 1e-300
    assert m.any()
    assert np.max(np.abs(kph[m] - ref[m]) / ref[m]) < 1e-11
    c.close()


@pytest.mark.parametrize("W", [64, 333])
def test_faint_rates_keep_the_products_order(W):
    """Rates near the smallest doubles, from a beam that all but ends: a term (J sigma) dlambda is a few
    units of 5e-324, so that only the definition's order of the product gives the oracle's value; sums of
    such terms are exact (1e-11 covers the rates a little above)."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column(S=40, L=12, n_photo=9, W=W)
    o = Oracle(p)
    n = o.initial_state()
    seen = 0
    for scale in 10.0 ** np.arange(-300.0, -270.0, 3.0):
        q = p.replace(J0=p.J0 * scale)
        ref = Oracle(q).photolysis(n)
        c = xk.Column(q, "fp64")
        kph = c.eval_photolysis(torch.as_tensor(n, device="cuda")).cpu().numpy()
        c.close()
        m = ref > 0.0
        seen += int(np.sum(m & (ref < 1e-307)))
        assert np.array_equal(kph > 0.0, m)
        assert np.max(np.abs(kph[m] - ref[m]) / ref[m]) < 1e-11
    assert seen > 0
