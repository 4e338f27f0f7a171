"""Bounded waits of the tensor-core kernels: with the products held back (nothing is issued, so nothing is in flight) and a
short budget, every call returns by itself, reports the give-up where its results are asked for, scatters nothing, and
the next call is correct. No fault, no wait without an end."""
import time

import numpy as np
import pytest
import torch

import synth
from parity import rel

pytestmark = pytest.mark.gpu

ETIMEOUT = -5
BUDGET = 1 << 20   # cycles, some 0.5 ms a wait


@pytest.fixture()
def case(fx, dev):
    nd, ns, nside = 3, 9001, 16
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    P = fx.Pointing.from_observations([o], mode="cache_f64", device=dev)
    N = fx.Noise.banded(P, np.tile(synth.inverse_noise_taps(), (nd, 1)))
    g = np.random.default_rng(6)
    return P, N, torch.as_tensor(synth.gaussian_sky(nside, g), device=dev), torch.as_tensor(g.normal(size=nd * ns), device=dev)


def _quick(f):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    out = f()
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 2.0
    return out


@pytest.mark.parametrize("what", ["normal", "f32x2", "rhs", "chi2", "fallback"])
def test_operators_report_and_recover(fx, dev, case, what):
    from paper_2603_19600_gb300 import _native as nat
    P, N, x, d = case
    if what == "fallback":   # no products: the outputs are formed without the tensor cores and nothing gives up
        N = fx.Noise.banded(P, np.tile([[2.0, 0.5]], (3, 1)))
    call = {"normal": lambda: fx.ptnp_apply(P, N, x, precision="f64"), "f32x2": lambda: fx.ptnp_apply(P, N, x, precision="f32x2"),
            "rhs": lambda: fx.rhs(P, N, d), "chi2": lambda: fx.chi2_grad(P, N, d, x)[1],
            "fallback": lambda: fx.ptnp_apply(P, N, x, precision="f64")}[what]
    good = call().clone()
    nat.furax_device_status(P.handle)
    nat.furax_set_wait_budget(P.handle, BUDGET)
    nat.furax_debug_hold_loader(P.handle, True)
    held = _quick(call)
    if what == "fallback":
        nat.furax_device_status(P.handle)
        assert rel(held, good) < 1e-13
    else:
        assert not held.any()          # nothing was added from sums that were never formed
        with pytest.raises(nat.FuraxError) as e:
            nat.furax_device_status(P.handle)
        assert e.value.code == ETIMEOUT
        nat.furax_device_status(P.handle)
    nat.furax_debug_hold_loader(P.handle, False)
    nat.furax_set_wait_budget(P.handle, 0)
    assert rel(call(), good) < 1e-13
    nat.furax_device_status(P.handle)


def test_solver_reports(fx, dev, case):
    from paper_2603_19600_gb300 import _native as nat
    P, N, _, d = case
    nat.furax_set_wait_budget(P.handle, BUDGET)
    nat.furax_debug_hold_loader(P.handle, True)
    with pytest.raises(nat.FuraxError) as e:
        _quick(lambda: fx.mapmaker_cg(P, N, d, maxiter=20))
    assert e.value.code == ETIMEOUT


def test_noise_alone_and_gap_filling(fx, dev, case):
    from paper_2603_19600_gb300 import _native as nat
    P, N, _, d = case
    cov = fx.Noise.banded(P, np.tile(synth.noise_covariance_band(64), (3, 1)))
    valid = torch.rand(d.numel(), device=dev, generator=torch.Generator(dev).manual_seed(1)) > 0.1
    fill = lambda: fx.gapfill(cov, d, valid, torch.zeros_like(d))[0]  # noqa: E731
    good, filled = cov.inv_apply(d), fill()
    nat.furax_noise_status(cov.handle)
    nat.furax_noise_set_wait_budget(cov.handle, BUDGET)
    nat.furax_debug_hold_noise(cov.handle, True)
    assert _quick(lambda: cov.inv_apply(d)).isnan().all()
    with pytest.raises(nat.FuraxError) as e:
        _quick(fill)
    assert e.value.code == ETIMEOUT
    nat.furax_debug_hold_noise(cov.handle, False)
    nat.furax_noise_set_wait_budget(cov.handle, 0)
    assert rel(fill(), filled) < 1e-8                       # not told of the product that gave up before
    with pytest.raises(nat.FuraxError) as e:
        nat.furax_noise_status(cov.handle)                  # which is still reported, once
    assert e.value.code == ETIMEOUT
    nat.furax_noise_status(cov.handle)
    assert torch.equal(cov.inv_apply(d), good)   # one thread per output: the same bits
    with pytest.raises(nat.FuraxError):
        nat.furax_noise_set_wait_budget(cov.handle, -1)
