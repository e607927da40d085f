"""Sizes of a batch's work items, on the CPU: by kind of shot, and never more
items than the workspace has slots for, whatever mixture of shots it holds."""
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2308_09348_gb300", "csrc")


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    """rows of (rule, grid, smoothed bins, slots, totals of the three kinds) -> tiles."""
    d = tmp_path_factory.mktemp("tiles")
    (d / "t.cpp").write_text('''#include <cstdio>
#include "qs_tiles.hpp"
using namespace qs;
int main() {
  long long r, g, s, slots, t[3];
  while (scanf("%lld %lld %lld %lld %lld %lld %lld", &r, &g, &s, &slots, t, t + 1, t + 2) == 7) {
    const int64_t n[kKinds] = {t[0], t[1], t[2]};
    int e[kKinds];
    if (r < 0) {                    // slots of (shots, samples) instead
      printf("%lld 0 0\\n", (long long)open_tiles((int32_t)g, s));
      continue;
    }
    choose_tiles((int)r, (int)g, n, (int)s, slots, e);
    printf("%d %d %d\\n", 1 << e[0], 1 << e[1], 1 << e[2]);
  }
}''')
    exe = str(d / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "t.cpp"), "-o", exe], check=True)

    def run(rows):
        text = "\n".join(" ".join(str(int(v)) for v in r) for r in rows)
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout
        return [[int(v) for v in line.split()] for line in out.splitlines()]

    return run


FORWARD, ADJOINT, MANY = 1, 2, 1 << 60


def test_sizes_follow_each_kinds_own_samples(choose):
    big = 256 * 20000
    rows = [(FORWARD, 0, 0, MANY, big, 0, 0), (FORWARD, 0, 0, MANY, 0, big, 0),
            (FORWARD, 0, 256, MANY, 0, big, 0), (FORWARD, 0, 0, MANY, 0, 0, big),
            (FORWARD, 0, 0, MANY, 20000, big, 20000), (FORWARD, 152, 0, MANY, big, 20000, 20000),
            (ADJOINT, 0, 0, MANY, big, 20000, 20000), (FORWARD, 0, 0, MANY, 0, 0, 0),
            (FORWARD, 0, 4000, MANY, 0, big, 0)]
    got = choose(rows)
    assert [r[0] for r in got[:1]] == [512] and got[1][1] == 4096 and got[2][1] == 512
    assert got[3][2] == 2048 and got[4] == [512, 4096, 512] and got[5] == [2048, 512, 512]
    assert got[6] == [2048] * 3 and got[7] == [512] * 3
    assert got[8][1] == 2048


def test_never_more_items_than_slots(choose):
    rg = random.Random(1)
    cases, asks = [], []
    for _ in range(600):
        shots = rg.choice([1, 2, 3, 16, 400, 4096])
        top = 10 ** rg.uniform(0, 9) / shots
        kinds = rg.choices([0, 1, 2], k=shots, weights=rg.choice([(1, 0, 0), (1, 1, 1), (1, 50, 2),
                                                                 (0, 1, 1), (30, 1, 1)]))
        n = [int(rg.choice([0, 1, rg.uniform(0, 2 * top), top])) for _ in kinds]
        total = sum(n) + rg.choice([0, 0, 1000])         # samples of no shot
        tot = [sum(c for c, k in zip(n, kinds) if k == j) for j in range(3)]
        cases.append((shots, kinds, n, total, tot, rg.choice([FORWARD, ADJOINT]),
                      rg.choice([0, 0, 1, 152]), rg.choice([0, 256, 4000])))
        asks.append((-1, shots, total, 0, 0, 0, 0))
    slots = [r[0] for r in choose(asks)]
    # the workspace of the open size, one made for tiles of 2048, the smallest
    rows, limits = [], []
    for c, s in zip(cases, slots):
        for m in (s, c[3] // 2048 + c[0] + 1, c[3] // 16384 + c[0] + 1):
            rows.append((c[5], c[6], c[7], m - c[0] - 1, *c[4]))
            limits.append((c, m))
    for (c, m), tile in zip(limits, choose(rows)):
        items = sum(-(-v // tile[k]) for v, k in zip(c[2], c[1]))
        assert items <= m, (c[0], c[3:], tile)


def test_sweeps_fit_the_smallest_workspace(choose):
    rows, want = [], []
    for shots in (1, 3, 256, 4096):
        for n in (0, 1, 100, 511, 3000, 16384, 16385, 100000):
            for k in range(3):
                slots = shots * -(-n // 16384) + 1
                tot = [shots * n if j == k else 0 for j in range(3)]
                rows.append((FORWARD, 0, 0, slots - shots - 1, *tot))
                want.append((shots, n, k, slots))
    for (shots, n, k, slots), tile in zip(want, choose(rows)):
        assert shots * -(-n // tile[k]) <= slots


@pytest.mark.gpu
@pytest.mark.parametrize("shared", [False, True])
def test_open_tiles_in_a_smaller_workspace(shared):
    import torch

    from paper_2308_09348_gb300 import binding as B, build
    from paper_2308_09348_gb300 import inputs as I
    build.build()
    shots, per = 5, 30000
    n = per if shared else shots * per
    g = torch.Generator(device="cuda").manual_seed(4)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    beam = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0,
                  sigma_z_um=10.0, div_rad=1e-3)
    lasers = [I.Laser(a0=20.0, w0_um=3.0, n_phase=4, model=m, variant=v) for m, v in
              ((I.MODEL_QFP, 0), (I.MODEL_LL, 0), (I.MODEL_QFP, 1), (I.MODEL_QFP, 2),
               (I.MODEL_LL, 1))]
    off = None if shared else [k * per for k in range(shots + 1)]
    bins = I.Bins(n_bins=40, lo=0.0, hi=4000.0)
    up = torch.zeros(shots, 13, dtype=torch.float64, device="cuda")
    up[:, 1] = 1.0
    out = []
    for tile in (0, 2048, 16384):                     # the workspace's; then left open
        bt = B.Batch(lasers, [beam] * shots, off, bins, n, tile=tile)
        bt.tile = 0
        bt.run(xi)
        out.append((bt.spectra.clone(), bt.moments[:, [0, 1, 11]].clone(), bt.grad(xi, up).clone(),
                    bt))
    for o in out[1:]:
        assert torch.equal(o[0], out[0][0]) and bool((o[1][:, 0] == per).all())
        # FP32 terms summed in another grouping: the bars of the batch tests
        torch.testing.assert_close(o[1], out[0][1], rtol=1e-7, atol=0)
        assert bool(((o[2] - out[0][2]).abs() <= 2e-5 * out[0][2].abs().amax(0)).all())
    bt = out[2][3]
    bt.ws_bytes -= 72 * (5 if shared else 9) + 256    # fewer slots than the largest tiles need
    with pytest.raises(B.QsError):
        bt.run(xi)


@pytest.mark.gpu
def test_ragged_shots_hold_their_own_samples():
    import numpy as np
    import torch

    from paper_2308_09348_gb300 import binding as B, build
    from paper_2308_09348_gb300 import inputs as I
    build.build()
    counts = [513, 1] * 200 + [8193, 0, 16385]
    off = np.concatenate([[0], np.cumsum(counts)])
    n = int(off[-1])
    g = torch.Generator(device="cuda").manual_seed(5)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    beam = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0,
                  sigma_z_um=10.0, div_rad=1e-3)
    bins = I.Bins(n_bins=64, lo=0.0, hi=5000.0)
    kinds = ((I.MODEL_QFP, 0), (I.MODEL_LL, 0), (I.MODEL_QFP, 1), (I.MODEL_QFP, 2))
    lasers = [I.Laser(a0=5.0 + k % 7, w0_um=3.0, n_phase=8, model=kinds[k % 4][0],
                      variant=kinds[k % 4][1]) for k in range(len(counts))]
    bt = B.Batch(lasers, [beam] * len(counts), off, bins, n).run(xi)
    last = len(counts) - 1
    for s in (0, 1, 2, 3, 198, 199, 200, 201, last - 3, last - 2, last):
        x = [t[off[s]:off[s + 1]].clone() for t in xi]
        # the records' bins: the arithmetic of the batch, bit for bit
        rec = B.qs_eval_samples(lasers[s], beam, x, bins)
        b = rec["bin"].long()
        ref = torch.bincount(b[(b >= 0) & (b < 64)], minlength=64).double()
        assert torch.equal(bt.spectra[s], ref), s
        # FP32 terms, compensated: the bar of the batch tests
        mean = float(rec["mu"].double().mean())
        assert abs(float(bt.moments[s, 1]) - mean) <= 1e-7 * mean, s
