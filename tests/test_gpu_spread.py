"""Calls of a few warps' worth of samples, dealt out over all CTAs: the edges
of a warp's step and of one pass of the launch against the per-sample records
and against the oracle."""
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


@pytest.mark.parametrize("prec,model", [("f32", I.MODEL_QFP), ("f32", I.MODEL_LL),
                                        ("f64", I.MODEL_QFP), ("f64", I.MODEL_LL)])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 4097, 64 * 152 + 1, 128 * 152 + 3])
def test_every_sample_once(prec, model, n):
    wl = I.full_qfp(n)
    L = I.Laser(**{**wl.laser.__dict__, "model": model, "n_phase": 7})
    xi, _ = I.workload_inputs(wl, n)
    w = I.rng(n).uniform(0.5, 1.5, n)
    xt = [torch.from_numpy(a).cuda() for a in xi]
    wt = torch.from_numpy(w.astype(np.float32)).cuda()
    out = B.qs_scatter(L, wl.beam, xt, wl.bins, precision=prec)
    rec = B.qs_eval_samples(L, wl.beam, xt, wl.bins, precision=prec)
    b = rec["bin"].long()
    nb = wl.bins.n_bins
    cnt = torch.bincount(torch.where(b < 0, nb + 1, b), minlength=nb + 2).double()
    assert torch.equal(out.spectrum, cnt[:nb])
    m = out.moments_dict()
    assert m["W"] == n
    # sums of n terms: FP64 to its rounding, FP32 terms to theirs (2^-24 each,
    # compensated sums)
    tol = 1e-13 if prec == "f64" else 2e-7
    mu = rec["mu"]
    assert abs(m["mean"] / float(mu.mean()) - 1) < tol
    # weighted, against the oracle's moments
    m = B.qs_scatter(L, wl.beam, xt, wl.bins, w=wt, precision=prec).moments_dict()
    ref = oracle.scatter(L, wl.beam, wl.bins, [a.astype(np.float64) for a in xi],
                         w.astype(np.float32).astype(np.float64))["moments"]
    for k in ("W", "mean", "div_y", "mean_aeff", "mean_gamma0"):
        assert abs(m[k] / ref[k] - 1) < (1e-12 if prec == "f64" else 1e-5), k
