"""Choice of lanes and tile heights of the FP32 2D warp march (csrc/lanes2d.h) over field shapes up to
far more strips than the GPU has warps: every choice is made by an estimated time."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1407_1309_gb300", "csrc")
PROGRAM = r"""
#include "lanes2d.h"
#include <cstdio>
int main() {
  int n0, n1, comp;
  while (std::scanf("%d %d %d", &n0, &n1, &comp) == 3) {
    const mpd::MarchRows a = mpd::march_rows(2, n0, n1, comp), b = mpd::march_rows(4, n0, n1, comp);
    std::printf("%d %.9g %d %.9g %d\n", a.ty, a.us, b.ty, b.us, (int)mpd::narrow_lanes(n0, n1, comp));
  }
}
"""
WIDTHS = [1, 8, 57, 120, 121, 1000, 4096, 33600, 204288, 204289, 300000, 437760, 437761, 2000000]


def test_every_choice_rests_on_a_time(tmp_path):
    src, exe = tmp_path / "lanes.cpp", tmp_path / "lanes"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    cases = [(n0, n1, comp) for n0 in (1, 4, 5, 37, 512, 4096) for n1 in WIDTHS for comp in (0, 1)]
    out = subprocess.run([str(exe)], input="\n".join("%d %d %d" % c for c in cases), text=True, check=True,
                         capture_output=True).stdout.split("\n")
    for case, line in zip(cases, out):
        ty2, us2, ty4, us4, narrow = map(float, line.split())
        assert us2 > 0 and us4 > 0 and ty2 >= 4 and ty4 >= 4, (case, line)
        assert ty2 % 2 == 0 and ty4 % 2 == 0, (case, line)  # an odd height rounds its last row differently
        assert narrow == (us2 < 0.98 * us4), (case, line)


@pytest.mark.gpu
@pytest.mark.parametrize("width", [204290, 437764])
def test_very_wide_fields_give_the_same_bits_with_both_lanes(width):
    import torch
    from paper_1407_1309_gb300 import capi
    from paper_1407_1309_gb300.solver import Mpdata
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(0)
    psi = 1 + torch.rand((5, width), generator=gen, device=dev)
    gc = [0.4 * (torch.rand((5, width), generator=gen, device=dev) - 0.5) for _ in range(2)]
    outs = []
    for kernel in (0, 1, 3):
        with Mpdata((5, width), n_iters=2, opts=capi.FCT) as m:
            m.tune(capi.TUNE_KERNEL, kernel)
            outs.append(torch.empty_like(psi))
            m.advance(psi, outs[-1], gc, n_steps=3)
            torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(538, 791), (600, 510), (1352, 909)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_chosen_heights_give_the_bits_of_a_given_one(shape):
    """Compensated steps (and plain ones where these take the warp march, not the band march) with the
    chosen lanes and height against lanes of 4 and 8 rows."""
    import torch
    from paper_1407_1309_gb300 import capi
    from paper_1407_1309_gb300.solver import Mpdata
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(0)
    psi = 1 + torch.rand(shape, generator=gen, device=dev)
    lo = 1e-7 * (torch.rand(shape, generator=gen, device=dev) - 0.5)
    gc = [0.4 * (torch.rand(shape, generator=gen, device=dev) - 0.5) for _ in range(2)]

    def run(rows):
        with Mpdata(shape, n_iters=2, opts=capi.FCT) as m:
            if rows:
                m.tune(capi.TUNE_KERNEL, 1)
                m.tune(capi.TUNE_TILE_ROWS, rows)
            plain, out, lout = torch.empty_like(psi), torch.empty_like(psi), torch.empty_like(psi)
            if shape[0] * shape[1] > 1000000:
                m.advance(psi, plain, gc, n_steps=3)
            else:
                plain.zero_()
            m.advance_compensated(psi, lo, out, lout, gc, n_steps=3)
            torch.cuda.synchronize()
        return plain, out, lout

    assert all(torch.equal(a, b) for a, b in zip(run(0), run(8)))
