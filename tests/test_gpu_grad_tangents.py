"""Adjoint with the tangents in logarithmic form, two samples per thread for
every FP32 model with phase cells: odd and single samples, every model and
variant, weak and strong fields, against the oracle's gradient."""
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


SCALE = np.array([20.0, 4.0, 1.0, 1.0, 10.0, 6000.0, 0.08, 1e-3])


@pytest.mark.parametrize("model,variant", [(I.MODEL_QFP, 0), (I.MODEL_QFP, 1), (I.MODEL_QFP, 2),
                                           (I.MODEL_QFP, 3), (I.MODEL_LL, 0), (I.MODEL_LL, 1)])
@pytest.mark.parametrize("n,a0,cells", [(1, 20.0, 33), (2, 0.1, 1), (65, 80.0, 64),
                                        (1027, 20.0, 17)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_gradient_matches_the_oracle(model, variant, n, a0, cells, prec):
    wl = I.fit_qfp(n)
    L = I.Laser(**{**wl.laser.__dict__, "model": model, "variant": variant, "a0": a0,
                   "n_phase": cells})
    xi, _ = I.workload_inputs(wl, n)
    w = I.rng(n).uniform(0.5, 1.5, n).astype(np.float32)
    rg = I.rng(3)
    dm = np.zeros(13)
    # no upstream on the spread and the divergences (singular for one sample
    # of the classical model)
    for k, sc in (("mean", 1e-3), ("mean_aeff", 1.0), ("mean_gamma0", 1e-3)):
        dm[B.MOMENT_FIELDS.index(k)] = rg.normal() * sc
    dS = rg.normal(size=wl.bins.n_bins) * 1e-3
    xt = [torch.from_numpy(a).cuda() for a in xi]
    wt = torch.from_numpy(w).cuda()
    out = B.qs_scatter(L, wl.beam, xt, wl.bins, w=wt, precision=prec)
    g = B.qs_scatter_grad(L, wl.beam, xt, wl.bins, out.moments, torch.from_numpy(dm),
                          torch.from_numpy(dS), w=wt, precision=prec, out=out).cpu().numpy()
    ref = oracle.grad(L, wl.beam, wl.bins, wl.bins.smooth_sigma_bins,
                      [a.astype(np.float64) for a in xi], w.astype(np.float64), dL_dm=dm,
                      dL_dS=dS)["grad"]
    err = np.abs((g - ref) * SCALE) / np.max(np.abs(ref * SCALE))
    # FP32: the bar of the large-sample gradient; a single sample's spectrum
    # slope carries the bin coordinate's rounding (2^-24 of 2^8 bins over a
    # width of 2 bins)
    assert np.all(err <= (1e-10 if prec == "f64" else 2e-5)), err
