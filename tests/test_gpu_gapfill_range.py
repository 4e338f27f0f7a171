"""FP64 gap filling of data whose level changes within a tile: what it fills between quiet samples is as accurate as the
FP64 FMA chain's product of those samples.

One CG iteration from 0 fills the gaps with alpha N r, r the observed data (the realisation is 0). alpha = r.r / r.Nr
comes from sums of at most 2^13 terms added in a tree (a thread's 9, then 5 + 4 levels, then the tiles: 40 u each) of
products that are each good to 127 u, and the filled value from one product more: |got - ref| <= (127 + 127 + 2 * 40 + 4) u
alpha |N| |r|, with as much again for the reference's own sums.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import gapfill as og
from oracle import ninv_band

pytestmark = pytest.mark.gpu

BOUND = 2 * (127 + 127 + 2 * 40 + 4) * 2.0 ** -53


@pytest.mark.parametrize("r", [0, 5, 8, 15, 19, 40])
def test_quiet_gaps_beside_a_loud_stretch(fx, dev, r):
    nd, ns = 3, 8192
    o = synth.Observation(8, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    cov = np.tile(synth.noise_covariance_band(64), (nd, 1))
    g = np.random.default_rng(r)
    d = g.normal(size=(nd, ns))
    d[0, 2000:2500] *= 2.0 ** r          # a level change
    d[1, 6000] *= 2.0 ** r               # a glitch that was not cut
    d[2, ::32] *= 2.0 ** r               # one loud sample among every 32
    valid = g.random((nd, ns)) > 0.1
    valid[:, 1000:1120] = False
    valid[:, 7000:7010] = False
    P = fx.Pointing.from_observations([o], mode="cache_f32", device=dev)
    N = fx.Noise.banded(P, cov)
    got, _, _ = fx.gapfill(N, torch.as_tensor(d.ravel(), device=dev), torch.as_tensor(valid.ravel(), device=dev),
                           torch.zeros(nd * ns, dtype=torch.float64, device=dev), maxiter=1, tol=1e-30)
    got = got.cpu().numpy().reshape(nd, ns)
    ref, _ = og.gapfill(cov, d, valid, np.zeros_like(d), maxiter=1, tol=1e-30)
    obs = np.where(valid, d, 0.0)
    nr = np.where(valid, ninv_band(cov, obs), 0.0)
    scale = (obs * obs).sum(1, keepdims=True) / (obs * nr).sum(1, keepdims=True) * ninv_band(np.abs(cov), np.abs(obs))
    assert np.array_equal(got[valid], d[valid])
    gap = ~valid
    worst = np.abs(got - ref)[gap] / np.maximum(scale[gap], 1e-300)
    assert worst.max() <= BOUND, worst.max()
