"""Photon spectrum with a group of 64 samples shared by several warps, each
emitting in its own phase cells: the edges of the split (one sample, a group
plus or minus one, fewer cells than warps) against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_09348_gb300 import build
    build.build()


@pytest.mark.parametrize("n,cells,bins,variant,grid", [
    (1, 1, 1, 0, 0), (1, 67, 33, 0, 0), (63, 5, 64, 1, 0), (65, 64, 33, 0, 0),
    (65, 65, 70, 1, 1), (200, 21, 300, 0, 3)])
def test_shared_groups_match_the_oracle(n, cells, bins, variant, grid):
    L = I.Laser(a0=20.0, w0_um=3.0, model=I.MODEL_QFP, n_phase=cells, variant=variant,
                delay_fs=10.0, dx_um=0.5)
    Bm = I.Beam(gamma_mean=3000.0, rel_spread=0.05, sigma_x_um=1.5, sigma_y_um=1.5,
                sigma_z_um=3.0, div_rad=2e-3)
    pb = I.Bins(n_bins=bins, lo=1e-3, hi=3500.0, log_spaced=1)
    xi = I.sample_streams(n, 31 + n, dtype=np.float32)
    w = I.rng(n).uniform(0.5, 1.5, n).astype(np.float32)
    xt = [torch.from_numpy(a).cuda() for a in xi]
    wt = torch.from_numpy(w).cuda()
    angles = bins <= 256
    got = B.qs_photon_spectrum(L, Bm, xt, pb, w=wt, grid=grid, theta2=True if angles else None)
    xd, wd = [a.astype(np.float64) for a in xi], w.astype(np.float64)
    if angles:
        S, T = (t.cpu().numpy() for t in got)
        Sr, Tr = oracle.photon_spectrum_angles(L, Bm, pb, xd, wd)
        for k in range(2):
            assert np.abs(T[k] - Tr[k]).sum() < 3e-6 * np.abs(Tr[k]).sum()
    else:
        S, Sr = got.cpu().numpy(), oracle.photon_spectrum(L, Bm, pb, xd, wd)
    # FP32 table and coordinate: ~1e-6 in one evaluation, averaged over the
    # cells and samples of a bin (the bar of the unshared sums)
    assert np.abs(S - Sr).sum() < 3e-6 * np.abs(Sr).sum()
