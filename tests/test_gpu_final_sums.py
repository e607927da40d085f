"""The final sums over CTAs and tiles keep what a plain sum loses: two large
contributions that cancel around a small one."""
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


@pytest.mark.parametrize("order", [(0, 1, 2), (0, 2, 1), (2, 1, 0)])
@pytest.mark.parametrize("batched,per", [(False, 32), (True, 64)])
def test_a_small_gradient_beside_two_that_cancel(order, batched, per):
    laser = I.Laser(a0=10.0, w0_um=3.0, model=I.MODEL_LL)
    beam = I.Beam(gamma_mean=3000.0, sigma_x_um=1.0, sigma_y_um=1.0, sigma_z_um=1.0)
    bins = I.Bins(n_bins=8, lo=0.0, hi=3500.0)
    n = 3 * per                               # one sample with weight per CTA or tile
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    w = torch.zeros_like(x)
    at = [per * k for k in order]
    x[at] = torch.tensor([1.0, -1.0, 1.0], dtype=torch.float64, device="cuda")
    w[at] = torch.tensor([1.0, 1.0, 2.0 ** -60], dtype=torch.float64, device="cuda")
    xi = [x] + [torch.zeros_like(x)] * 7
    dm = torch.zeros(13, dtype=torch.float64, device="cuda")
    dm[B.MOMENT_FIELDS.index("mean")] = 1.0

    if batched:
        bt = B.Batch([laser], [beam], [0, n], bins, n, precision="f64", tile=per)
        mom = bt.run(xi, w).moments.clone()

        def grad(weights):
            return bt.grad(xi, dm[None], w=weights, moments=mom)[0].clone()
    else:
        mom = B.qs_scatter(laser, beam, xi, bins, w=w, precision="f64").moments.clone()

        def grad(weights):
            return B.qs_scatter_grad(laser, beam, xi, bins, mom, dm, w=weights, precision="f64",
                                     block=per, grid=3).clone()

    dx = B.GRAD_PARAMS.index("dx_um")
    alone = torch.zeros_like(w)
    alone[at[0]] = 1.0
    # the three contributions are +-1 and 2^-60 times the same number, exactly
    one = float(grad(alone)[dx])
    assert one != 0.0 and float(grad(w)[dx]) == one * 2.0 ** -60


def test_overflowed_weights_are_not_a_divergence_of_zero():
    laser = I.Laser(a0=10.0, w0_um=3.0, model=I.MODEL_LL)
    beam = I.Beam(gamma_mean=3000.0, sigma_x_um=1.0, sigma_y_um=1.0, sigma_z_um=1.0, div_rad=1e-3)
    xi = [torch.ones(64, dtype=torch.float64, device="cuda") for _ in range(8)]
    xi[4], xi[5] = 1e7 * xi[4], 1e7 * xi[5]             # angles of 1e4: w theta^2 overflows
    w = torch.full((64,), 1e308, dtype=torch.float64, device="cuda")
    out = B.qs_scatter(laser, beam, xi, I.Bins(n_bins=0), w=w, precision="f64").moments_dict()
    assert out["W"] == float("inf") and out["nonfinite"] == 0.0
    assert all(out[k] != out[k] for k in ("div_x", "div_y", "div"))
