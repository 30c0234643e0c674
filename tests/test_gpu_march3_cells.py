"""The FP32 3D z-marches with cell-by-cell staging (x extents that are no multiple of 4, fields of 48
to 127 columns, unaligned arrays) against the oracle at the edges of their tiles (64 or 128
columns, 8 rows) and z-chunks: FP32 bar 1e-5 over 3 steps with per-step advector factors."""
import numpy as np
import pytest
import torch

import oracle
from helpers import nondivergent, smooth_positive
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
CASES = {
    "tot3_fct_G": (3, capi.TOT | capi.FCT | capi.NUG), "iga_tot_fct_G": (2, capi.IGA | capi.TOT | capi.FCT | capi.NUG),
    "fct3": (3, capi.FCT), "abs_fct": (2, capi.ABS | capi.FCT), "tot": (2, capi.TOT),
    "kahan_euler_fct": (2, capi.FCT | capi.KAHAN | capi.RHS_EULER_A),
}
SHAPES = [(1, 1, 49), (3, 2, 63), (6, 9, 65), (17, 8, 127), (5, 7, 129), (33, 3, 191), (2, 17, 258)]


@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "unaligned"])
@pytest.mark.parametrize("shape", SHAPES + [(4, 9, 128)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("name", sorted(CASES))
def test_cell_staging_matches_oracle(name, shape, shift):
    n_iters, opts = CASES[name]
    rng = np.random.default_rng(sum(shape))
    r = lambda a: a.astype(np.float32).astype(np.float64)
    psi = r(smooth_positive(shape, rng) - (1.5 if opts & (capi.IGA | capi.ABS) else 0.0))
    gc = [r(v) for v in nondivergent(shape, rng, 0.3)]
    G = r(1.0 + 0.2 * rng.uniform(size=shape)) if opts & capi.NUG else None
    R = r(0.1 * rng.normal(size=shape)) if opts & capi.RHS_EULER_A else None
    n = psi.size

    def t(a):  # `shift` elements off a 16-byte boundary
        if a is None:
            return None
        buf = torch.empty(n + 4, dtype=torch.float32, device=DEV)
        v = buf[shift:shift + n].view(shape)
        v.copy_(torch.tensor(a, dtype=torch.float32))
        return v

    scales = [1.0, 0.75, -0.5]
    ref = psi
    bits = int(opts & ~(capi.NUG | capi.RHS_EULER_A))
    for s in scales:
        ref = oracle.step(ref, [v * s for v in gc], g=G, r=R, dt=0.2, n_iters=n_iters, opts=bits)
    with Mpdata(shape, dtype=torch.float32, n_iters=n_iters, opts=opts) as m:
        out = t(np.zeros(shape))
        m.advance(t(psi), out, [t(v) for v in gc], g=t(G), r=t(R), dt=0.2, n_steps=3, gc_scale=scales)
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
