"""Device work of a call is ordered on the caller's stream alone: a solve on a non-blocking stream must not depend on
what the legacy default stream still holds."""
import glob
import os
import re

import numpy as np
import pytest
import torch

import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_19600_gb300", "csrc")


def test_no_clear_on_the_default_stream():
    """cudaMemset runs on the legacy default stream, which orders nothing with a non-blocking one."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\bcudaMemset\s*\(", code), path


def test_no_copy_on_the_default_stream():
    """cudaMemcpy from pageable memory may return before the copy has reached the device, on that stream."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\bcudaMemcpy\s*\(", code), path


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [{"tol": 1e-10}, {"tol": 1e-10, "binned_only": True},
                                {"tol": 1e-8, "precision": "f32", "acc": "f64"}])
def test_first_solve_beside_a_busy_default_stream(fx, dev, kw):
    """The first solve of a handle (which allocates and clears its workspace) while the default stream is busy,
    against the same solve with nothing else running: their sums differ by their order only, so the maps agree to
    twice the residual they were solved to times a preconditioned condition number below 1e4."""
    nd, ns, nside = 4, 30000, 16
    o = synth.Observation(nside, synth.satellite_scan(ns), synth.hex_focal_plane(nd))
    taps = np.tile(synth.inverse_noise_taps(), (nd, 1))
    d = torch.as_tensor(np.random.default_rng(4).normal(0, 10, nd * ns), device=dev)

    def solve(stream):
        P = fx.Pointing.from_observations([o], mode="cache_mixed", device=dev)
        N = fx.Noise.banded(P, taps)
        a = torch.ones(8192, 8192, device=dev)
        torch.cuda.synchronize()
        for _ in range(10 if stream else 0):
            a = a @ a * (1.0 / 8192)      # some 0.2 s of work on the default stream
        with torch.cuda.stream(stream):
            got = fx.mapmaker_cg(P, N, d, maxiter=1000, **kw)
        torch.cuda.synchronize()
        return got

    ref, rv, ri = solve(None)
    got, gv, gi = solve(torch.cuda.Stream())
    assert torch.equal(rv, gv) and gi.converged and ri.converged
    assert float((got - ref).norm()) <= 2e4 * kw["tol"] * float(ref.norm())
    if "binned_only" in kw:
        assert abs(gi.true_rel_res - ri.true_rel_res) <= 1e-6 * ri.true_rel_res
    else:
        assert gi.true_rel_res <= kw["tol"] * 10
