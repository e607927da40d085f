"""The batch workspace with the tile size left open: its size against that of
fixed tiles of 2048 samples, and calls on both sides of the numbers of samples
where the library's tile size changes."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I

BINS = I.Bins(n_bins=64, lo=0.0, hi=5000.0)
BEAM = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0, sigma_z_um=10.0,
              div_rad=1e-3)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2308_09348_gb300 import build
    build.build()


def _bytes(shots, n, tile, shared):
    return B._lib().qs_batch_workspace_bytes(shots, n, C.byref(B.make_bins(BINS)), 64,
                                             C.byref(B.make_exec("f32", 0, 0, 0, None, tile)),
                                             int(shared))


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("shots", [1, 64, 4096])
def test_open_tiles_take_no_more_than_fixed_ones(shots, shared):
    last = 0
    for n in sorted({max(0, 2 ** k + d) for k in range(0, 33) for d in (-1, 0, 1)}):
        b = _bytes(shots, n, 0, shared)
        # at most 19456 slots of less than 200 bytes more
        assert 0 < b <= _bytes(shots, n, 2048, shared) + 19456 * 200, n
        assert b >= last, n              # a workspace for more serves fewer
        last = b


def _streams(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    return [torch.randn(n, generator=g, device="cuda") for _ in range(8)]


@pytest.mark.gpu
@pytest.mark.parametrize("model", [I.MODEL_QFP, I.MODEL_LL])
# 64 shots: the adjoint's tile changes at 77824 samples, the forward's at 155648
@pytest.mark.parametrize("n", [1, 22, 77823, 77824, 155647, 155648, 155649])
def test_sweep_about_the_changes_of_tile(n, model):
    lasers = [I.Laser(a0=5.0 + k, w0_um=3.0, model=model, n_phase=16) for k in range(64)]
    xi = _streams(n)
    upstream = torch.zeros(64, 13, dtype=torch.float64, device="cuda")
    upstream[:, [1, 11]] = 1.0           # the mean energies
    out = []
    for tile in (0, 2048):
        bt = B.Batch(lasers, [BEAM] * 64, None, BINS, n, tile=tile)
        bt.run(xi)
        bt.grad(xi, upstream)
        assert bool((bt.moments[:, 0] == n).all()) and bool(bt.grads.isfinite().all())
        out.append(bt)
    assert torch.equal(out[0].spectra, out[1].spectra)
    # FP32 terms summed in another grouping: the bar of the batch tests
    np.testing.assert_allclose(out[0].moments[:, [0, 1, 11]].cpu().numpy(),
                               out[1].moments[:, [0, 1, 11]].cpu().numpy(), rtol=1e-7)


@pytest.mark.gpu
def test_many_ragged_shots():
    counts = [513, 1] * 2000 + [8193, 0, 16385]
    off = np.concatenate([[0], np.cumsum(counts)])
    xi = _streams(int(off[-1]))
    lasers = [I.Laser(a0=5.0, w0_um=3.0, n_phase=16,
                      model=I.MODEL_QFP if k % 3 else I.MODEL_LL) for k in range(len(counts))]
    bt = B.Batch(lasers, [BEAM] * len(counts), off, BINS, int(off[-1]))
    bt.run(xi)
    assert bt.moments[:, 0].cpu().tolist() == [float(c) for c in counts]
