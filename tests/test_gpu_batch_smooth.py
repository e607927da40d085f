"""Batched classical shots with smoothed spectra (their own kernel): shots at
the edges of a warp, a block and a tile, against the per-sample path of
single-shot calls."""
import numpy as np
import pytest
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_09348_gb300 import build
    build.build()


BINS = I.Bins(n_bins=40, lo=2000.0, hi=3500.0, smooth_sigma_bins=1.5)
BEAM = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0, sigma_z_um=10.0,
              div_rad=1e-3)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("tile,block", [(0, 0), (64, 32), (512, 256), (8192, 96)])
@pytest.mark.parametrize("shared", [False, True])
def test_shots_equal_single_calls(weighted, tile, block, shared):
    counts = [1000] * 4 if shared else [1, 31, 0, 33, 127, 128, 129, 511, 513, 4097]
    n = counts[0] if shared else sum(counts)
    off = np.concatenate([[0], np.cumsum(counts)])
    g = torch.Generator(device="cuda").manual_seed(n)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    # weights on the grid of the fixed-point sums
    w = torch.randint(1, 64, (n,), generator=g, device="cuda") / 16.0 if weighted else None
    lasers = [I.Laser(a0=10.0 + k, w0_um=3.0, model=I.MODEL_LL) for k in range(len(counts))]
    bt = B.Batch(lasers, [BEAM] * len(counts), None if shared else off, BINS, n, tile=tile,
                 block=block).run(xi, w)
    for s, c in enumerate(counts):
        lo, hi = (0, n) if shared else (int(off[s]), int(off[s + 1]))
        if hi == lo:
            assert not bt.spectra[s].any() and not bt.spec_smooth[s].any()
            continue
        x = [t[lo:hi].clone() for t in xi]
        ref = B.qs_scatter(lasers[s], BEAM, x, BINS, w=None if w is None else w[lo:hi].clone())
        # sums of integers of the same samples' deposits
        assert torch.equal(bt.spectra[s], ref.spectrum)
        assert torch.equal(bt.spec_smooth[s], ref.spec_smooth) and bool(ref.spec_smooth.any())
        # FP32 terms summed in another grouping: the bar of the batch tests
        torch.testing.assert_close(bt.moments[s], ref.moments, rtol=1e-7, atol=0)
