"""FP32 steps at the ends of the number range.

A step of MPDATA commutes with a scaling of psi, and a power of two scales without rounding, so a
field near either end of the range has to give the scaled result of the same field around 1:
  - flux sums below the smallest normal number (psi itself normal): the limiter still divides by them;
  - 3D cross terms whose psi-sums lie above 2^126, where a flushing reciprocal is 0.
And the tail of a narrow blob, through the subnormal numbers down to zero, stays finite and matches
the FP64 oracle on the kernel families that test_gpu_tiny_values.py leaves out.

Tolerance of the scaled fields: 5 steps of at most 40 roundings each per pass of 2^-24 (a quantum of
the subnormal fluxes, 2^-149, is 2^-24 of the least psi, 2^-125): 200 * 2^-24 = 1.2e-5 of the largest
value and pass, doubled for three passes and more."""
import numpy as np
import pytest
import torch

import oracle
from helpers import boxes, nondivergent
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
# family: shape, passes, options, tuning knobs
FAMILIES = {
    "warp": ((70, 96), 2, 0, {capi.TUNE_KERNEL: 1}), "warp2": ((70, 96), 2, 0, {capi.TUNE_KERNEL: 3}),
    "band": ((70, 96), 2, 0, {capi.TUNE_KERNEL: 2}), "staged2d": ((70, 96), 2, capi.STAGED, {}),
    "blocked": ((70, 96), 2, 0, {capi.TUNE_STEPS_PER_LAUNCH: 3}), "abs": ((70, 96), 2, capi.ABS, {}),
    "dfl": ((70, 96), 2, capi.DFL, {}), "tile": ((70, 96), 3, 0, {}), "tile_tot": ((70, 96), 2, capi.TOT, {}),
    "cluster": ((300,), 2, 0, {}), "cluster3": ((300,), 3, capi.TOT, {}), "block1d": ((300,), 8, 0, {}),
    "staged1d": ((300,), 2, capi.STAGED, {}), "chunks3d": ((9, 20, 128), 2, 0, {}),
    "cells3d": ((9, 20, 61), 3, capi.TOT, {}), "scalar3d": ((9, 20, 21), 2, 0, {}),
}


def run(family, psi, gc, opts, n_steps):
    """The family's FP32 result (FP64 array) and the oracle's for the same, already rounded, inputs."""
    shape, n_iters, extra, knobs = FAMILIES[family]
    t = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)
    with Mpdata(shape, dtype=torch.float32, n_iters=n_iters, opts=extra | opts) as m:
        for k, v in knobs.items():
            m.tune(k, v)
        a = t(psi)
        b = torch.empty_like(a)
        m.advance(a, b, [t(v) for v in gc], n_steps=n_steps)
        torch.cuda.synchronize()
        out = b.double().cpu().numpy()
    return out, oracle.step(psi, gc, n_iters=n_iters, opts=int((extra | opts) & ~capi.STAGED), n_steps=n_steps)


def inputs(shape, seed, values):
    rng = np.random.default_rng(seed)
    gc = [v.astype(np.float32).astype(np.float64) for v in nondivergent(shape, rng, 0.4)]
    return values(shape, rng).astype(np.float32).astype(np.float64), gc


@pytest.mark.parametrize("family", sorted(FAMILIES))
def test_flux_sums_below_the_normal_range_are_limited(family):
    shape, n_iters, _, _ = FAMILIES[family]
    scale = 2.0 ** -125
    psi, gc = inputs(shape, 4, lambda s, r: boxes(s, r) * scale)
    assert psi.min() >= 2 * np.finfo(np.float32).tiny  # psi and its sums are normal, 0.1 of it is not
    out, ref = run(family, psi, gc, capi.FCT, 5)
    tol = 1.2e-5 * (1 if n_iters == 2 else 2)
    assert np.abs(out - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("family", ["chunks3d", "scalar3d"])
@pytest.mark.parametrize("opts", [0, capi.FCT], ids=["basic", "fct"])
def test_cross_terms_at_the_top_of_the_range(family, opts):
    shape = FAMILIES[family][0]
    # pairs of cells sum to less than 2^126, the four cells of a cross term to more
    psi, gc = inputs(shape, 6, lambda s, r: r.uniform(2.1, 3.9, size=s) * 2.0 ** 123)
    out, ref = run(family, psi, gc, opts, 5)
    assert np.abs(out - ref).max() <= 1.2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("family", ["abs", "dfl", "tile", "tile_tot", "cluster", "cluster3", "chunks3d", "cells3d"])
@pytest.mark.parametrize("opts", [0, capi.FCT], ids=["basic", "fct"])
def test_subnormal_tails_stay_finite_and_match_oracle(family, opts):
    def blob(shape, rng):
        r2 = sum((x - n / 2) ** 2 for x, n in zip(np.meshgrid(*map(np.arange, shape), indexing="ij"), shape))
        return np.exp(-r2 / (2 * 1.5 ** 2))

    psi, gc = inputs(FAMILIES[family][0], 5, blob)
    assert ((psi > 0) & (psi < np.finfo(np.float32).tiny)).any()
    out, ref = run(family, psi, gc, opts, 30)
    assert np.isfinite(out).all()
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)
