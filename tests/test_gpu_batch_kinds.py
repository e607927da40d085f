"""Batches by kind of shot: classical shots read four samples at a time from
any start, every kind in one call, shots whose pulses differ from the first
one's, against the per-sample records and single-shot calls."""
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


BINS = I.Bins(n_bins=96, lo=0.0, hi=5000.0)
BEAM = I.Beam(gamma_mean=3000.0, rel_spread=0.1, sigma_x_um=3.0, sigma_y_um=3.0, sigma_z_um=10.0,
              div_rad=1e-3)


def _streams(n, skip=0):
    """Eight streams whose first sample lies `skip` elements past an aligned
    allocation (stream 2 one more when skip is 9: streams aligned apart)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    out = []
    for k in range(8):
        s = (skip + (1 if skip == 9 and k == 2 else 0)) % 9
        base = torch.empty(n + s, device="cuda")
        base[s:] = torch.randn(n, generator=g, device="cuda")
        out.append(base[s:])
    return out


def _spectrum(laser, xi, w, prec):
    """Weighted histogram of the per-sample records."""
    b = B.qs_eval_samples(laser, BEAM, xi, BINS, precision=prec)["bin"].long()
    ok = (b >= 0) & (b < BINS.n_bins)
    ww = torch.ones(b.numel(), device="cuda") if w is None else w
    return torch.bincount(b[ok], weights=ww[ok].double(), minlength=BINS.n_bins)


@pytest.mark.parametrize("skip", [0, 1, 3, 9])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("tile", [0, 1024, 4096])
def test_classical_shots_from_any_start(skip, weighted, tile):
    counts = [1, 1023, 1024, 1025, 4097, 8191, 20003, 2]
    off = np.concatenate([[0], np.cumsum(counts)])
    n = int(off[-1])
    xi = _streams(n, skip)
    # weights on the fixed-point grid of the histograms: exact sums
    w = (torch.randint(1, 64, (n,), device="cuda") / 16.0) if weighted else None
    lasers = [I.Laser(a0=10.0 + k, w0_um=3.0, delay_fs=5.0 * k, model=I.MODEL_LL)
              for k in range(len(counts))]
    bt = B.Batch(lasers, [BEAM] * len(counts), off, BINS, n, tile=tile)
    bt.run(xi, w)
    for s in range(len(counts)):
        sub = [x[off[s]:off[s + 1]] for x in xi]
        ws = None if w is None else w[off[s]:off[s + 1]]
        assert torch.equal(bt.spectra[s], _spectrum(lasers[s], sub, ws, "f32")), s
        ref = B.qs_scatter(lasers[s], BEAM, sub, BINS, w=ws).moments
        # FP32 terms summed in another grouping: the bar of the batch tests
        np.testing.assert_allclose(bt.moments[s, [0, 1, 4, 5, 7, 11]].cpu().numpy(),
                                   ref[[0, 1, 4, 5, 7, 11]].cpu().numpy(), rtol=1e-7)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_every_kind_and_pulse_in_one_call(prec):
    n = 700
    xi = _streams(n)
    base = dict(w0_um=3.0, dx_um=0.5)
    lasers = [I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, **base),
              I.Laser(a0=20.0, model=I.MODEL_LL, **base),
              I.Laser(a0=25.0, model=I.MODEL_QFP, n_phase=64, **base),            # shot 0's table
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=48, **base),            # other cells
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, tau_fs=20.0, **base),
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, envelope=I.ENV_SIN2, **base),
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, variant=1, **base),
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, variant=2, **base),
              I.Laser(a0=20.0, model=I.MODEL_LL, n_phase=64, variant=1, **base),
              I.Laser(a0=20.0, model=I.MODEL_QFP, n_phase=64, variant=3, lambda_um=1.0, **base)]
    for order in (range(len(lasers)), reversed(range(len(lasers)))):
        ls = [lasers[k] for k in order]
        bt = B.Batch(ls, [BEAM] * len(ls), None, BINS, n, precision=prec)
        bt.run(xi)
        for s, l in enumerate(ls):
            assert torch.equal(bt.spectra[s], _spectrum(l, xi, None, prec)), s
