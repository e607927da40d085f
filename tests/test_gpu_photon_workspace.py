"""The photon spectrum in workspaces of any size from one partial spectrum per
pass of two samples per thread up to the size asked for."""
import ctypes as C

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


def _least(n, bins, block):
    return -(-max(1, -(-n // (2 * block))) * 24 * bins // 256) * 256


def _asked(n, bins, block, grid=0):
    return B._lib().qs_photon_workspace_bytes(
        C.byref(B.make_bins(I.Bins(n_bins=bins, lo=1.0, hi=3500.0))),
        C.byref(B.make_exec("f32", 0, block, grid, None)), n)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,bins,block", [(1, 33, 256), (600, 33, 96), (2000, 16, 256),
                                          (2000, 16, 32)])
def test_a_smaller_workspace_is_enough(n, bins, block, prec):
    beam = I.Beam(gamma_mean=3000.0, rel_spread=0.05, sigma_x_um=1.5, sigma_y_um=1.5,
                  sigma_z_um=3.0, div_rad=2e-3)
    laser = I.Laser(a0=20.0, w0_um=3.0, model=I.MODEL_QFP, n_phase=3)
    pb = I.Bins(n_bins=bins, lo=1e-3, hi=3500.0, log_spaced=1)
    g = torch.Generator(device="cuda").manual_seed(3)
    xi = [torch.randn(n, generator=g, device="cuda") for _ in range(8)]
    s, keep = B.make_samples(xi, None)
    out = torch.zeros(bins, dtype=torch.float64, device="cuda")
    ws = torch.empty(_asked(n, bins, block) + 256, dtype=torch.uint8, device="cuda")
    ptr = (ws.data_ptr() + 255) // 256 * 256

    def call(size):
        out.fill_(-1.0)
        st = B._lib().qs_photon_spectrum(
            C.byref(B.make_laser(laser)), C.byref(B.make_beam(beam)), C.byref(s),
            C.byref(B.make_bins(pb)), C.byref(B.make_exec(prec, 0, block, 0, None)),
            out.data_ptr(), None, ptr, size, B._stream_ptr(None))
        return st, out.clone()

    least, asked = _least(n, bins, block), _asked(n, bins, block)
    st, ref = call(asked)
    assert st == 0 and least <= asked and bool((ref > 0).any())
    for size in {least, min(asked, least + 24 * bins), (least + asked) // 2, max(least, asked - 1)}:
        st, got = call(size)
        assert st == 0
        # the same evaluations, 64 of them summed plainly in 32 bits
        torch.testing.assert_close(got, ref, rtol=64 * 2.0 ** -23 if prec == "f32" else 1e-13,
                                   atol=0)
    assert call(least - 1)[0] == 3                     # QS_ERR_WORKSPACE


def test_few_samples_ask_for_little():
    # eight CTAs of eight warps for the 64 warps of one group
    assert _asked(64, 512, 256) == 8 * 24 * 512
    assert _asked(1, 512, 256, grid=3) == 3 * 24 * 512
