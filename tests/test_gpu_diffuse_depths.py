"""The diffuse field where a layer's optical depth leaves the range in which a quotient may be taken by
the divisor's reciprocal: depths whose reciprocal overflows, the smallest doubles, infinity."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scatter", [0, 1])
@pytest.mark.parametrize("depth", [5e-324, 1e-320, 1e-310, 5.5e-309, 5.6e-309, 2e-308, 1e-300, 1e-290, np.inf])
def test_diffuse_field_at_vanishing_and_infinite_depths(depth, scatter):
    """Every other wavelength bin is absorbed (and, with scatter, as much scattered) by one species only,
    at this optical depth in every layer.  1e-11 relative: up to 64 terms of one sign, through optical
    depths of some hundreds in the other bins; a depth this small or infinite adds no rounding."""
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    p = synth.with_scattering(synth.small_column(S=40, L=12, n_photo=9, W=64), albedo=0.3, diffuse=1)
    o = Oracle(p)
    n, dz = o.initial_state(), o.grid()[2]
    one, faint = 7, np.arange(p.W) % 2 == 1
    sa, ss = p.sigma_abs.copy(), p.sigma_s.copy()
    sa[:, faint] = ss[:, faint] = 0.0
    if np.isinf(depth):
        sa[one, faint] = 1e305
        n[:, one] = 1e6
    else:
        sa[one, faint] = 1e-20
        if scatter:
            ss[one, faint] = 1e-20
        n[:, one] = depth / (1e-20 * dz)
    p = p.replace(sigma_abs=sa, sigma_s=ss)
    ref = Oracle(p).photolysis(n)
    c = xk.Column(p, "fp64")
    kph = c.eval_photolysis(torch.as_tensor(n, device="cuda")).cpu().numpy()
    c.close()
    assert np.isfinite(ref).all() and np.isfinite(kph).all()
    m = ref > 1e-300
    assert m.any()
    assert np.max(np.abs(kph[m] - ref[m]) / ref[m]) < 1e-11
