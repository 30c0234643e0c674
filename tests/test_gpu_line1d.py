"""The one-launch 1D path (one thread-block cluster, halos through distributed shared memory)
against the oracle where its work split changes: fields shorter than a step's reach, one chunk, one
chunk more, one chunk per block of the largest cluster and one cell more, several chunks per
block; every option it takes; in place; systems with trapezoidal sources.  Tolerances: the
repository's FP64 1e-12 and FP32 1e-5 bars over 12 steps."""
import numpy as np
import pytest
import torch

import oracle
from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
OPTS = {
    "fct": (2, capi.FCT), "donor": (1, 0), "basic3": (3, 0), "tot3_fct": (3, capi.TOT | capi.FCT),
    "iga_tot": (2, capi.IGA | capi.TOT), "iga_fct_kahan": (2, capi.IGA | capi.FCT | capi.KAHAN),
    "abs_fct": (2, capi.ABS | capi.FCT), "nug_fct": (2, capi.NUG | capi.FCT), "fct6": (6, capi.FCT),
    "euler_a": (2, capi.FCT | capi.RHS_EULER_A), "euler_b": (2, capi.FCT | capi.RHS_EULER_B),
}


def check(got, ref, dtype):
    if dtype == torch.float64:
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    else:
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("name", sorted(OPTS))
@pytest.mark.parametrize("n", [1, 2, 3, 26, 27, 53, 416, 417, 833, 5000])
def test_cluster_path_matches_oracle(n, name, dtype):
    n_iters, opts = OPTS[name]
    rng = np.random.default_rng(n)
    r = (lambda a: a.astype(np.float32).astype(np.float64)) if dtype == torch.float32 else (lambda a: a)
    psi = r(1.0 + rng.uniform(size=n))
    if opts & (capi.IGA | capi.ABS):
        psi = r(psi - 1.5)
    gc = r(np.full(n, 0.4) + 0.1 * rng.uniform(size=n))
    G = r(1.0 + 0.2 * rng.uniform(size=n)) if opts & capi.NUG else None
    R = r(0.1 * rng.normal(size=n)) if opts & (capi.RHS_EULER_A | capi.RHS_EULER_B) else None
    t = lambda a: None if a is None else torch.tensor(a, dtype=dtype, device=DEV)
    bits = int(opts & ~(capi.RHS_EULER_A | capi.RHS_EULER_B | capi.NUG))
    ref = oracle.step(psi, [gc], g=G, r=R, dt=0.3, n_iters=n_iters, opts=bits, n_steps=12,
                      rhs="euler_b" if opts & capi.RHS_EULER_B else "euler_a")
    for in_place in (False, True):
        with Mpdata((n,), dtype=dtype, n_iters=n_iters, opts=opts) as m:
            a = t(psi)
            b = a if in_place else torch.empty_like(a)
            m.advance(a, b, [t(gc)], g=t(G), r=t(R), dt=0.3, n_steps=12)
            torch.cuda.synchronize()
            check(b.double().cpu().numpy(), ref, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("E", [1, 3, 8])
@pytest.mark.parametrize("n", [2, 26, 27, 417, 1700])
def test_systems_match_oracle(n, E, dtype):
    rng = np.random.default_rng(10 * n + E)
    r = (lambda a: a.astype(np.float32).astype(np.float64)) if dtype == torch.float32 else (lambda a: a)
    fields = [r(1.0 + rng.uniform(size=n)) for _ in range(E)]
    b = [r(0.1 * rng.normal(size=n)) for _ in range(E)]
    gc = r(np.full(n, 0.5))
    A = 0.2 * rng.normal(size=(E, E))
    ref = np.stack(oracle.step_trapez(fields, [gc], A, b=b, dt=0.4, n_iters=2, opts=oracle.FCT, n_steps=7))
    t = lambda v: torch.tensor(np.concatenate(v), dtype=dtype, device=DEV)
    with Mpdata([(n,)] * E, dtype=dtype, n_iters=2, opts=capi.FCT | capi.RHS_TRAPEZ) as m:
        psi, bt = t(fields), t(b)
        m.set_rhs_linear(A, bt)
        m.advance(psi, psi, [t([gc] * E)], dt=0.4, n_steps=7)
        torch.cuda.synchronize()
        check(psi.double().cpu().numpy().reshape(E, n), ref, dtype)
