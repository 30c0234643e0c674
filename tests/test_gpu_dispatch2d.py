"""The automatic choice of lanes and tile heights of the FP32 2D march, at shapes on both sides of
its rule: padded strips (n1 just above a multiple of a strip), tall and wide fields, one tile: the
automatic step against the oracle (FP32 bar 1e-5 over 4 steps), plain, compensated and with
|psi|; and the recording of a step gives that step's bits."""
import numpy as np
import pytest
import torch

import oracle
from helpers import nondivergent, smooth_positive
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
SHAPES = [(7, 121), (257, 130), (900, 57), (1300, 500), (60, 2500), (701, 803), (1500, 240)]
f = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)
r = lambda a: a.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("name", ["fct", "abs_fct", "compensated"])
def test_automatic_choice_matches_oracle(shape, name):
    rng = np.random.default_rng(shape[1])
    opts = capi.FCT | (capi.ABS if name == "abs_fct" else 0)
    psi = r(smooth_positive(shape, rng) - (1.2 if name == "abs_fct" else 0.0))
    gc = [r(v) for v in nondivergent(shape, rng, 0.3)]
    oracle.set_threads(0)
    ref = oracle.step(psi, gc, n_iters=2, opts=int(opts), n_steps=4)
    with Mpdata(shape, dtype=torch.float32, n_iters=2, opts=opts) as m:
        a, g = f(psi), [f(v) for v in gc]
        out = torch.empty_like(a)
        if name == "compensated":
            m.advance_compensated(a, torch.zeros_like(a), out, torch.empty_like(a), g, n_steps=4)
        else:
            m.advance(a, out, g, n_steps=4)
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
        if name == "fct":
            tape = torch.empty(m.tape_numel(), dtype=torch.float32, device=DEV)
            recorded, step = torch.empty_like(a), torch.empty_like(a)
            m.adjoint_record(a, g, tape, psi_next=recorded)
            m.advance(a, step, g)
            torch.cuda.synchronize()
            assert torch.equal(recorded, step)
