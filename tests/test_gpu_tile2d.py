"""The 2D shared-memory tile step (third-order terms, more than two passes, open edges, the FP64
divergent-flow option) against the oracle at the edges of its tiles (32 columns,
32 rows in FP32 and 16 in FP64): fields smaller than the halo, one tile, one cell more or less,
several ragged tiles; periodic and every combination of open edges.  Tolerances: the repository's
FP64 1e-12 and FP32 1e-5 bars over 4 steps."""
import numpy as np
import pytest
import torch

import oracle
from helpers import nondivergent, smooth_positive
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
OPTS = {
    "fct3": (3, capi.FCT), "basic3": (3, 0), "fct4": (4, capi.FCT), "tot3_fct": (3, capi.TOT | capi.FCT),
    "tot2": (2, capi.TOT), "iga_tot_fct": (2, capi.IGA | capi.TOT | capi.FCT), "fct": (2, capi.FCT),
    "abs_dfl_fct": (2, capi.ABS | capi.DFL | capi.FCT), "dfl_tot3_fct": (3, capi.DFL | capi.TOT | capi.FCT),
    "nug_tot_fct3": (3, capi.NUG | capi.TOT | capi.FCT), "kahan_fct3": (3, capi.KAHAN | capi.FCT),
    "euler_a_tot": (2, capi.TOT | capi.FCT | capi.RHS_EULER_A),
    "euler_b_tot": (2, capi.TOT | capi.FCT | capi.RHS_EULER_B), "iga_fct_kahan": (2, capi.IGA | capi.FCT | capi.KAHAN),
}
SHAPES = [(2, 3), (5, 4), (16, 32), (17, 33), (15, 65), (33, 31), (50, 70)]
OPEN = {"periodic": 0, "open0": capi.OPEN0, "open1": capi.OPEN1, "open": capi.OPEN0 | capi.OPEN1}


@pytest.mark.parametrize("edges", sorted(OPEN))
@pytest.mark.parametrize("name", sorted(OPTS))
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
def test_tile_step_matches_oracle(dtype, shape, name, edges):
    n_iters, opts = OPTS[name]
    opts = opts | OPEN[edges]
    rng = np.random.default_rng(shape[0] + 100 * shape[1])
    r = (lambda a: a.astype(np.float32).astype(np.float64)) if dtype == torch.float32 else (lambda a: a)
    psi = smooth_positive(shape, rng)
    if opts & (capi.ABS | capi.IGA):
        psi = psi - 1.2
    gc = [0.15 * rng.uniform(-1, 1, size=shape) for _ in range(2)] if opts & capi.DFL else nondivergent(shape, rng, 0.3)
    psi, gc = r(psi), [r(v) for v in gc]
    G = r(1.0 + 0.2 * rng.uniform(size=shape)) if opts & capi.NUG else None
    R = r(0.1 * rng.normal(size=shape)) if opts & (capi.RHS_EULER_A | capi.RHS_EULER_B) else None
    t = lambda a: None if a is None else torch.tensor(a, dtype=dtype, device=DEV)
    bits = int(opts & ~(capi.RHS_EULER_A | capi.RHS_EULER_B | capi.NUG))
    ref = oracle.step(psi, gc, g=G, r=R, dt=0.3, n_iters=n_iters, opts=bits, n_steps=4,
                      rhs="euler_b" if opts & capi.RHS_EULER_B else "euler_a")
    with Mpdata(shape, dtype=dtype, n_iters=n_iters, opts=opts) as m:
        a = t(psi)
        b = torch.empty_like(a)
        m.advance(a, b, [t(v) for v in gc], g=t(G), r=t(R), dt=0.3, n_steps=4)
        torch.cuda.synchronize()
        got = b.double().cpu().numpy()
    if dtype == torch.float64:
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    else:
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("edges", ["periodic", "open"])
@pytest.mark.parametrize("name", ["abs_dfl_fct", "dfl_tot3_fct"])
def test_tall_fp64_tiles_match_oracle(name, edges):
    """FP64 fields with enough tiles for the 32-row form (18 x 17 tiles, the last ones partial)."""
    n_iters, opts = OPTS[name]
    opts = opts | OPEN[edges]
    shape = (563, 530)
    rng = np.random.default_rng(8)
    psi = smooth_positive(shape, rng) - (1.2 if opts & capi.ABS else 0.0)
    gc = [0.15 * rng.uniform(-1, 1, size=shape) for _ in range(2)]
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)
    oracle.set_threads(0)
    ref = oracle.step(psi, gc, n_iters=n_iters, opts=int(opts), n_steps=2)
    with Mpdata(shape, dtype=torch.float64, n_iters=n_iters, opts=opts) as m:
        out = t(psi)
        m.advance(t(psi), out, [t(v) for v in gc], n_steps=2)
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
