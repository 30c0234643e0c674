"""Rules of the dispatch that only show in time, measured on the device (median of CUDA-event
times, the sides in turn).  The bounds leave room for noise: each faulty rule was at least 20 %
slower than the other side."""
import pytest
import torch

from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.solver import Mpdata

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


def problem(shapes, dtype, n_iters, opts, knobs=None):
    """A call of 4 steps of random fields, ready to be timed."""
    one = not isinstance(shapes, list)
    total = sum(s[0] * s[1] for s in ([shapes] if one else shapes))
    gen = torch.Generator(device=DEV).manual_seed(1)
    psi = 2 + torch.rand(total, generator=gen, device=DEV, dtype=dtype)
    gc = [0.4 * (torch.rand(total, generator=gen, device=DEV, dtype=dtype) - 0.5) for _ in range(2)]
    if one:
        psi, gc = psi.reshape(shapes), [v.reshape(shapes) for v in gc]
    out = torch.empty_like(psi)
    m = Mpdata(shapes, dtype=dtype, n_iters=n_iters, opts=opts)
    for k, v in (knobs or {}).items():
        m.tune(k, v)
    return lambda: m.advance(psi, out, gc, n_steps=4)


def problem3(shape):
    """A call of 4 limited two-pass steps of a random 3D FP32 field, ready to be timed."""
    gen = torch.Generator(device=DEV).manual_seed(1)
    psi = 2 + torch.rand(shape, generator=gen, device=DEV)
    gc = [0.3 * (torch.rand(shape, generator=gen, device=DEV) - 0.5) for _ in range(3)]
    out = torch.empty_like(psi)
    m = Mpdata(shape, dtype=torch.float32, n_iters=2, opts=capi.FCT)
    return lambda: m.advance(psi, out, gc, n_steps=4)


def times(*calls):
    """Median microseconds of each call, timed in turn."""
    got = [[] for _ in calls]
    for rep in range(24):
        for call, ts in zip(calls, got):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            call()
            b.record()
            b.synchronize()
            if rep >= 4:
                ts.append(a.elapsed_time(b) * 1e3)
    return [sorted(ts)[len(ts) // 2] for ts in got]


def test_fp64_tiles_of_one_per_sm_take_the_time_of_one():
    """128 blocks, fewer than SMs, take no longer than 8 (the next step's blocks do not crowd them)."""
    k = {capi.TUNE_KERNEL: 1}
    few, many = times(problem((64, 64), torch.float64, 3, capi.FCT, k), problem((256, 256), torch.float64, 3, capi.FCT, k))
    assert many <= 1.15 * few


@pytest.mark.parametrize("shapes", [[(200, 200)] * 64, [(60 + 7 * k % 241, 60 + 53 * k % 241) for k in range(100)]],
                         ids=["64_of_200", "100_of_60_to_300"])
def test_fp64_ensembles_take_a_tile_height_near_the_best(shapes):
    rows = (0, 12, 16, 24, 32, 48)
    got = times(*[problem(shapes, torch.float64, 2, capi.FCT, {capi.TUNE_TILE_ROWS: r}) for r in rows])
    assert got[0] <= 1.1 * min(got[1:]), dict(zip(rows, got))


@pytest.mark.parametrize("n,dtype,n_iters,opts", [
    (64, torch.float64, 3, capi.FCT), (64, torch.float64, 8, capi.FCT), (64, torch.float64, 3, 0),
    (256, torch.float64, 6, capi.FCT), (512, torch.float64, 5, capi.TOT), (1024, torch.float64, 3, capi.TOT | capi.FCT),
    (1024, torch.float64, 3, 0), (1024, torch.float64, 2, capi.TOT), (64, torch.float32, 8, capi.TOT | capi.FCT),
    (512, torch.float32, 6, capi.FCT), (1024, torch.float32, 8, capi.FCT), (1024, torch.float32, 3, capi.FCT)])
def test_steps_beyond_two_passes_take_the_better_kernels(n, dtype, n_iters, opts):
    auto, tile, staged = times(problem((n, n), dtype, n_iters, opts),
                               problem((n, n), dtype, n_iters, opts, {capi.TUNE_KERNEL: 1}),
                               problem((n, n), dtype, n_iters, opts | capi.STAGED))
    assert auto <= 1.15 * min(tile, staged), (auto, tile, staged)


@pytest.mark.parametrize("pair", [False, True], ids=["one_call", "record_and_replay"])
def test_reverse_step_takes_no_longer_than_its_parts(pair):
    """1024^2 FP32 with the limiter, 20 reverse steps, each in one call or as a recording and a replay,
    against 20 recordings and then 20 replays."""
    n, steps = 1024, 20
    gen = torch.Generator(device=DEV).manual_seed(2)
    psi = 2 + torch.rand((n, n), generator=gen, device=DEV)
    gc = [0.4 * (torch.rand((n, n), generator=gen, device=DEV) - 0.5) for _ in range(2)]
    nxt, pb, gcb = torch.empty_like(psi), torch.rand((n, n), generator=gen, device=DEV), [torch.zeros_like(v) for v in gc]
    m = Mpdata((n, n), dtype=torch.float32, n_iters=2, opts=capi.FCT)
    tape = torch.empty(m.tape_numel(), device=DEV)

    def whole():
        for _ in range(steps):
            if pair:
                m.adjoint_record(psi, gc, tape, psi_next=nxt)
                m.adjoint_replay(psi, gc, tape, pb, gc_bar=gcb)
            else:
                m.adjoint_step(psi, gc, pb, gc_bar=gcb)

    def parts():
        for _ in range(steps):
            m.adjoint_record(psi, gc, tape, psi_next=nxt)
        for _ in range(steps):
            m.adjoint_replay(psi, gc, tape, pb, gc_bar=gcb)

    one, two = times(whole, parts)
    assert one <= 1.08 * two, (one, two)


def test_wide_fields_take_a_tile_height_near_the_best():
    """1250 strips: whole tiles per SM leave few heights to choose from."""
    rows = (0, 32, 64)
    got = times(*[problem((1500, 150000), torch.float32, 2, capi.FCT,
                          {capi.TUNE_TILE_ROWS: r, capi.TUNE_KERNEL: 1} if r else {}) for r in rows])
    assert got[0] <= 1.08 * min(got[1:]), dict(zip(rows, got))


@pytest.mark.parametrize("n,n_iters,opts", [(6000, 4, capi.TOT | capi.FCT), (8000, 3, capi.TOT | capi.FCT), (12000, 2, 0),
                                            (4000, 2, capi.FCT)])
def test_long_fp64_lines_take_the_better_kernels(n, n_iters, opts):
    gen = torch.Generator(device=DEV).manual_seed(3)
    psi = 2 + torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    gc = [torch.full((n,), 0.3, device=DEV, dtype=torch.float64)]
    out = torch.empty_like(psi)

    def steps(extra):
        m = Mpdata((n,), dtype=torch.float64, n_iters=n_iters, opts=opts | extra)
        return lambda: m.advance(psi, out, gc, n_steps=40)

    auto, staged = times(steps(0), steps(capi.STAGED))
    assert auto <= 1.15 * staged, (auto, staged)
