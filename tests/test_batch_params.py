"""The gradient parameters' columns in a batch's descriptors, by their names."""
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I


def _batch(n=3):
    b = object.__new__(B.Batch)
    b.n_shots = n
    lasers = [I.Laser(a0=1.5 + k, w0_um=2.5, dx_um=0.3, dy_um=0.4, delay_fs=5.0) for k in range(n)]
    beams = [I.Beam(gamma_mean=3000.0 + k, rel_spread=0.06, div_rad=7e-3) for k in range(n)]
    b.d_lasers = B._struct_array_to_device([B.make_laser(x) for x in lasers], B.qs_laser, "cpu")
    b.d_beams = B._struct_array_to_device([B.make_beam(x) for x in beams], B.qs_beam, "cpu")
    return b, lasers, beams


def test_columns_hold_the_named_parameters():
    b, lasers, beams = _batch()
    want = [[getattr(lz, k) for k in B.GRAD_PARAMS[:5]] + [getattr(bm, k) for k in B.GRAD_PARAMS[5:]]
            for lz, bm in zip(lasers, beams)]
    torch.testing.assert_close(b.params(), torch.tensor(want, dtype=torch.float64), rtol=0, atol=0)


def test_writing_leaves_the_other_fields():
    b, _, _ = _batch()
    before = [t.clone() for t in (b.d_lasers, b.d_beams)]
    theta = b.params()
    b.set_params(theta * 2.0)
    torch.testing.assert_close(b.params(), theta * 2.0, rtol=0, atol=0)
    b.set_params(theta)
    assert torch.equal(b.d_lasers, before[0]) and torch.equal(b.d_beams, before[1])
