"""The 2D tile kernel in FP64 where the dispatch leaves the step to the staged kernels (small fields,
many passes): asked for by MPDATA_TUNE_KERNEL, against the oracle at the edges of its tiles, with both
tile heights.  Tolerance: the repository's FP64 1e-12 bar over 4 steps."""
import numpy as np
import pytest
import torch

import oracle
from helpers import nondivergent, smooth_positive
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
OPEN = capi.OPEN0 | capi.OPEN1
OPTS = {
    "basic3": (3, 0), "fct3": (3, capi.FCT), "tot2": (2, capi.TOT), "tot3_fct": (3, capi.TOT | capi.FCT), "fct5": (5, capi.FCT),
    "iga_tot_fct": (2, capi.IGA | capi.TOT | capi.FCT), "nug_fct3": (3, capi.NUG | capi.FCT),
    "open_fct": (2, capi.FCT | OPEN), "open_fct4": (4, capi.FCT | OPEN), "dfl_fct": (2, capi.DFL | capi.FCT),
    "abs_dfl_open": (2, capi.ABS | capi.DFL | capi.FCT | OPEN), "kahan_fct3": (3, capi.KAHAN | capi.FCT),
    "euler_b_tot": (2, capi.TOT | capi.FCT | capi.RHS_EULER_B),
}


# the last two: 16-row tiles on a ragged field, 32-row tiles (17 x 17 of them)
@pytest.mark.parametrize("shape", [(2, 3), (16, 32), (17, 33), (15, 65), (50, 70), (131, 97), (543, 530)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("name", sorted(OPTS))
def test_asked_for_tile_step_matches_oracle(name, shape):
    n_iters, opts = OPTS[name]
    rng = np.random.default_rng(shape[0] + 100 * shape[1])
    psi = smooth_positive(shape, rng) - (1.2 if opts & (capi.ABS | capi.IGA) else 0.0)
    gc = [0.15 * rng.uniform(-1, 1, size=shape) for _ in range(2)] if opts & capi.DFL else nondivergent(shape, rng, 0.3)
    G = 1.0 + 0.2 * rng.uniform(size=shape) if opts & capi.NUG else None
    R = 0.1 * rng.normal(size=shape) if opts & capi.RHS_EULER_B else None
    t = lambda a: None if a is None else torch.tensor(a, dtype=torch.float64, device=DEV)
    oracle.set_threads(0)
    ref = oracle.step(psi, gc, g=G, r=R, dt=0.3, n_iters=n_iters, opts=int(opts & ~(capi.RHS_EULER_B | capi.NUG)), n_steps=4,
                      rhs="euler_b" if R is not None else "euler_a")
    with Mpdata(shape, dtype=torch.float64, n_iters=n_iters, opts=opts) as m:
        m.tune(capi.TUNE_KERNEL, 1)
        out = t(psi)
        m.advance(t(psi), out, [t(v) for v in gc], g=t(G), r=t(R), dt=0.3, n_steps=4)
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
