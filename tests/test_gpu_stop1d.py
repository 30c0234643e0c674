"""Long calls on the 1D cluster path are split into launches of 256 steps: a stop request ends the
call between them, and the split changes no bit."""
import threading
import time

import numpy as np
import pytest
import torch

from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


def test_stop_request_ends_a_long_call_of_a_1d_system():
    """A call of 1.2 million steps (about 5 s of kernels) returns ESTOPPED: the launch queue fills
    long before its last launch, and the request arrives while the host waits for room in it."""
    n = 1000
    x = torch.arange(n, device=DEV, dtype=torch.float64)
    psi = torch.cat([1 + torch.exp(-((x - 300) / 50) ** 2), torch.zeros_like(x)])
    gc = [torch.full((2 * n,), 0.3, device=DEV, dtype=torch.float64)]
    out = torch.empty_like(psi)
    with Mpdata([(n,), (n,)], dtype=torch.float64, n_iters=2, opts=capi.FCT | capi.RHS_TRAPEZ) as m:
        m.set_rhs_linear(np.array([[0.0, 0.1], [-0.1, 0.0]]))
        m.advance(psi, out, gc, dt=0.1, n_steps=2)
        torch.cuda.synchronize()

        def stop():
            time.sleep(0.2)
            m.request_stop()

        t = threading.Thread(target=stop)
        t.start()
        with pytest.raises(capi.MpdataError, match="stop"):
            m.advance(psi, out, gc, dt=0.1, n_steps=1200000)
        t.join()
        torch.cuda.synchronize()
        assert torch.isfinite(out).all()


@pytest.mark.parametrize("in_place", [False, True], ids=["out_of_place", "in_place"])
@pytest.mark.parametrize("steps", [256, 257, 600])
@pytest.mark.parametrize("trapez", [False, True], ids=["field", "system"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
def test_split_calls_give_the_bits_of_short_ones(dtype, trapez, steps, in_place):
    n, fields = 700, 2 if trapez else 1
    rng = np.random.default_rng(1)
    t = lambda a: torch.tensor(a, dtype=dtype, device=DEV)
    psi = t(1 + rng.uniform(size=fields * n))
    gc = [t(np.full(fields * n, 0.35))]
    opts = capi.FCT | (capi.RHS_TRAPEZ if trapez else 0)
    with Mpdata([(n,)] * fields, dtype=dtype, n_iters=2, opts=opts) as m:
        if trapez:
            m.set_rhs_linear(np.array([[0.0, 0.1], [-0.1, 0.0]]))
        ref = psi.clone()
        for s in range(0, steps, 100):
            m.advance(ref, ref, gc, dt=0.1, n_steps=min(100, steps - s))
        out = psi.clone() if in_place else torch.empty_like(psi)
        m.advance(out if in_place else psi, out, gc, dt=0.1, n_steps=steps)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
