"""The work table of a batched handle outlives a change of a knob that asks for the same table: a
CUDA graph captured before keeps reading it."""
import numpy as np
import pytest
import torch

from helpers import nondivergent, smooth_positive
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


# FP64 lanes own 2 columns whatever the knob says; FP32 with the tile height given takes lanes of 4 for 0 and 1
@pytest.mark.parametrize("dtype,rows", [(torch.float64, 0), (torch.float32, 16)], ids=["f64", "f32"])
def test_captured_steps_survive_a_knob_that_changes_nothing(dtype, rows):
    rng = np.random.default_rng(2)
    shapes = [(40, 50), (33, 61), (64, 48)]
    psi = torch.tensor(np.concatenate([smooth_positive(s, rng).ravel() for s in shapes]), dtype=dtype, device=DEV)
    fields = [nondivergent(s, rng, 0.3) for s in shapes]
    gc = [torch.tensor(np.concatenate([f[d].ravel() for f in fields]), dtype=dtype, device=DEV) for d in range(2)]
    out, other = torch.empty_like(psi), torch.empty_like(psi)
    with Mpdata(shapes, dtype=dtype, n_iters=2, opts=capi.FCT) as m:
        if rows:
            m.tune(capi.TUNE_TILE_ROWS, rows)
        graph = m.capture(psi, out, gc, 3)
        m.tune(capi.TUNE_KERNEL, 1)
        m.advance(psi, other, gc, n_steps=3)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, other)
