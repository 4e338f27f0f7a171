"""chi^2 and its gradients do not see map pixels that no sample observes, also where samples without a pixel stand in for
the first one: NaN there changes nothing."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["cache_f64", "cache_mixed", "cache_f32", "on_the_fly"])
@pytest.mark.parametrize("noise", ["white", "banded"])
def test_nan_in_unobserved_pixels(fx, dev, mode, noise):
    nd, ns, nside = 2, 5000, 64
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    q = np.array(o.q_bore)
    q[1000:1010] = np.nan                      # samples without a pixel
    P = fx.Pointing(torch.as_tensor(q, device=dev), torch.as_tensor(o.q_det, device=dev), [nd], [ns], [nside], mode=mode)
    N = fx.Noise.white(P, np.full(nd, 2.0)) if noise == "white" else \
        fx.Noise.banded(P, np.tile(synth.inverse_noise_taps(), (nd, 1)))
    g = np.random.default_rng(8)
    m = torch.as_tensor(synth.gaussian_sky(nside, g), device=dev)
    d = torch.as_tensor(g.normal(size=nd * ns), device=dev)
    seen = P.transpose(torch.ones_like(d), hits=True)[1] > 0
    assert not bool(seen[0]) and int((~seen).sum()) > 1000
    ref = fx.chi2_grad(P, N, d, m)
    bad = m.clone()
    bad[~seen] = float("nan")
    got = fx.chi2_grad(P, N, d, bad)
    for a, b in zip(got, ref):                 # only the order of the sums differs: 5000 terms at most per sum
        assert float((a - b).abs().max()) <= 5000 * 2.0 ** -53 * float(b.abs().max()) * 100
