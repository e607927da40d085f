"""Every component of the adjoint by itself, with an upstream gradient on the
spread and the divergences too: its error against the oracle's gradient
relative to the samples' contributions to that component (not to the largest
component), for spots from tight to wide against the beam."""
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


N = 33
BINS = I.Bins(n_bins=64, lo=0.0, hi=3500.0, smooth_sigma_bins=2.0)
UPSTREAM = {"mean": 1e-3, "spread": 2e-3, "rel_spread": 1.0, "div_x": 100.0, "div_y": -70.0,
            "div": 30.0, "mean_aeff": 0.5, "mean_gamma0": 1e-3}


@pytest.mark.parametrize("model,variant", [(I.MODEL_QFP, 0), (I.MODEL_QFP, 1), (I.MODEL_QFP, 2),
                                           (I.MODEL_QFP, 3), (I.MODEL_LL, 0), (I.MODEL_LL, 1)])
@pytest.mark.parametrize("w0,sigma", [(4.0, 3.0), (10.0, 1.0), (40.0, 0.5), (40.0, 0.1)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_each_component(model, variant, w0, sigma, prec):
    L = I.Laser(a0=20.0, w0_um=w0, n_phase=17, model=model, variant=variant, dx_um=0.2 * sigma,
                dy_um=-0.1 * sigma, delay_fs=15.0)
    Bm = I.Beam(gamma_mean=3000.0, rel_spread=0.08, sigma_x_um=sigma, sigma_y_um=sigma,
                sigma_z_um=5.0, div_rad=1e-3)
    xi = I.sample_streams(N, 7, dtype=np.float32)
    w = I.rng(N).uniform(0.5, 1.5, N).astype(np.float32)
    dm = np.zeros(13)
    for k, v in UPSTREAM.items():
        dm[B.MOMENT_FIELDS.index(k)] = v
    xt, dmt = [torch.from_numpy(a).cuda() for a in xi], torch.from_numpy(dm)

    def grad(weights, mom, p):
        return B.qs_scatter_grad(L, Bm, xt, BINS, mom, dmt, w=torch.from_numpy(weights).cuda(),
                                 precision=p).cpu().numpy()

    def forward(p):
        return B.qs_scatter(L, Bm, xt, BINS, w=torch.from_numpy(w).cuda(),
                            precision=p).moments.clone()

    # the samples' contributions: one weight at a time, the moments kept
    mom64 = forward("f64")
    parts = np.stack([grad(np.where(np.arange(N) == i, w, 0).astype(np.float32), mom64, "f64")
                      for i in range(N)])
    ref = oracle.grad(L, Bm, BINS, BINS.smooth_sigma_bins, [a.astype(np.float64) for a in xi],
                      w.astype(np.float64), dL_dm=dm)["grad"]
    err = np.abs(grad(w, forward(prec), prec) - ref)
    scale = np.abs(parts).sum(0)
    assert np.all(scale > 0)
    # FP32: the bar of the large-sample gradient.  The spread's upstream takes
    # mu - mean, a tenth of mu, whose rounding over the cells is some 16 2^-24
    assert np.all(err <= (1e-10 if prec == "f64" else 2e-5) * scale), err / scale
