"""Shared-memory layouts of the kernels whose regions mix types, on the CPU,
for every block size and for odd and even bin counts: every region is aligned
for its type, none overlaps the next, and the size asked for at the launch
covers the last."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2308_09348_gb300", "csrc")


def _rows(tmp_path, body):
    """Lines of numbers printed by a program around the layout header."""
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text('#include <cstdio>\n#include "qs_layout.hpp"\nusing namespace qs;\n'
                   "int main() {\n" + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [[int(v) for v in line.split()] for line in out.splitlines()]


def test_batch(tmp_path):
    rows = _rows(tmp_path, """
  for (int warps = 1; warps <= 16; ++warps)
    for (size_t bins = 0; bins < 70; ++bins)
      for (size_t counter = 4; counter <= 8; counter += 4)
        for (size_t smooth = 0; smooth <= 1; ++smooth)
          for (size_t cycle = 0; cycle <= 4096; cycle += 4096) {
            const size_t b[7] = {1092, cycle, 61 * 16, (size_t)warps * 72,
                                 bins ? (bins + 2) * counter : 0, 12, smooth * bins * 8};
            const BatchLayout l = batch_layout(b[0], b[1], b[2], warps, 72, b[4], b[6]);
            printf("0 %zu %zu %zu %zu %zu %zu", l.cycle, l.table, l.red, l.hist, l.item, l.smooth);
            for (size_t x : b) printf(" %zu", x);
            printf(" %zu\\n", l.bytes);
          }""")
    assert len(rows) == 16 * 70 * 2 * 2 * 2
    for r in rows:
        starts, sizes, total = r[:7], r[7:14], r[14]
        # 16-byte loads of the two tables, 8-byte ones of the others
        assert all(s % 8 == 0 for s in starts) and starts[1] % 16 == 0 and starts[2] % 16 == 0
        ends = [s + b for s, b in zip(starts, sizes)]
        assert all(e <= s for e, s in zip(ends, starts[1:] + [total]))


def test_photon(tmp_path):
    rows = _rows(tmp_path, """
  for (int warps = 1; warps <= 8; ++warps)
    for (size_t bins = 1; bins < 70; ++bins)
      for (size_t sums = 1; sums <= 3; sums += 2)
        for (size_t real = 4; real <= 8; real += 4) {
          const bool f = real == 4;
          const size_t b[6] = {61 * (f ? 16u : 8u), f ? 8192u : 0u, bins * real,
                               (size_t)warps * sums * bins * 8, f ? warps * 64 * 32u : 0u,
                               f ? warps * 16 * 128u : 0u};
          const PhotonLayout l = photon_layout(b[0], b[1], b[2], warps, sums * bins * 8,
                                               b[4] / warps, b[5] / warps);
          printf("0 %zu %zu %zu %zu %zu", l.ptab, l.eps, l.part, l.stage, l.state);
          for (size_t x : b) printf(" %zu", x);
          printf(" %zu\\n", l.bytes);
        }""")
    assert len(rows) == 8 * 69 * 2 * 2
    for r in rows:
        starts, sizes, total = r[:6], r[6:12], r[12]
        assert all(s % 8 == 0 for s in starts) and starts[1] % 16 == 0
        assert sizes[4] == 0 or starts[4] % 16 == 0        # the emitters' 16-byte accesses
        ends = [s + b for s, b in zip(starts, sizes)]
        assert all(e <= s for e, s in zip(ends, starts[1:] + [total]))


@pytest.mark.gpu
@pytest.mark.parametrize("block", [32, 96, 160, 224])
@pytest.mark.parametrize("prec,weighted", [("f32", False), ("f32", True), ("f64", False)])
def test_batches_with_odd_numbers_of_warps(block, prec, weighted):
    import torch

    from paper_2308_09348_gb300 import binding as B, build
    from paper_2308_09348_gb300 import inputs as I
    build.build()
    n = 1500
    g = torch.Generator(device="cuda").manual_seed(1)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    # weights on the grid of the fixed-point sums
    w = torch.randint(1, 64, (n,), generator=g, device="cuda") / 16.0 if weighted else None
    beam = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0,
                  sigma_z_um=10.0, div_rad=1e-3)
    lasers = [I.Laser(a0=20.0, w0_um=3.0, n_phase=5, model=I.MODEL_QFP, variant=v)
              for v in (0, 1, 2, 3)] + [I.Laser(a0=20.0, w0_um=3.0, model=I.MODEL_LL)]
    bins = I.Bins(n_bins=33, lo=0.0, hi=5000.0, smooth_sigma_bins=1.5)
    out = []
    for blk in (block, 64):
        bt = B.Batch(lasers, [beam] * 5, None, bins, n, precision=prec, block=blk, tile=512)
        out.append(bt.run(xi, w))
    # the same samples through the same arithmetic: equal counts; moments
    # summed in another grouping (FP32 terms: the bar of the batch tests)
    assert torch.equal(out[0].spectra, out[1].spectra) and bool((out[0].spectra.sum(1) > 0).all())
    assert torch.equal(out[0].spec_smooth, out[1].spec_smooth)
    torch.testing.assert_close(out[0].moments, out[1].moments, atol=0,
                               rtol=1e-12 if prec == "f64" else 1e-7)


@pytest.mark.gpu
@pytest.mark.parametrize("block", [32, 96, 160, 224])
@pytest.mark.parametrize("bins,angles", [(33, False), (33, True), (301, False), (1, True)])
@pytest.mark.parametrize("variant", [0, 1])
def test_photons_with_odd_numbers_of_warps(block, bins, angles, variant):
    import torch

    from paper_2308_09348_gb300 import binding as B, build
    from paper_2308_09348_gb300 import inputs as I
    build.build()
    n = 700
    g = torch.Generator(device="cuda").manual_seed(2)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    beam = I.Beam(gamma_mean=3000.0, rel_spread=0.05, sigma_x_um=1.5, sigma_y_um=1.5,
                  sigma_z_um=3.0, div_rad=2e-3)
    laser = I.Laser(a0=20.0, w0_um=3.0, model=I.MODEL_QFP, n_phase=9, variant=variant)
    pb = I.Bins(n_bins=bins, lo=1e-3, hi=3500.0, log_spaced=1)
    got, ref = (B.qs_photon_spectrum(laser, beam, xi, pb, block=b, theta2=True if angles else None)
                for b in (block, 64))
    if not angles:
        got, ref = (got,), (ref,)
    for a, b in zip(got, ref):
        # the same evaluations; 64 of them summed plainly in 32 bits, then
        # compensated, in another grouping
        assert bool((b > 0).any())
        torch.testing.assert_close(a, b, rtol=64 * 2.0 ** -23, atol=0)
