"""The fit's losses against their definition written out moment by moment:
value, gradient, unequal weights, one part only, targets that were not
measured (NaN) and carry no weight."""
import pytest
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import fit as F


def _by_definition(mom, S, tm, tS, weights, sw):
    L = 0.0
    for k, c in weights.items():
        i = F.MOMENT_INDEX[k]
        L = L + c * ((mom[..., i] - tm[..., i]) / (tm[..., i].abs() + 1e-30)) ** 2
    if sw and S.numel():
        d = (S - tS) / tS.sum(-1, keepdim=True).clamp_min(1e-30)
        L = L + sw * (d ** 2).sum(-1) * S.shape[-1]
    return L


@pytest.mark.parametrize("weights,sw", [
    (F.DEFAULT_MOMENT_WEIGHTS, 1.0), (F.BATCH_MOMENT_WEIGHTS, 0.0),
    ({"mean": 2.0, "spread": 0.5, "div_x": 1.0}, 3.0), ({"mean": 2.0}, 0.0), ({}, 1.0), ({}, 0.0)])
@pytest.mark.parametrize("shots", [0, 3])
def test_losses_equal_their_definition(weights, sw, shots):
    g = torch.Generator().manual_seed(1)
    shape = (shots,) if shots else ()
    r = lambda n: torch.rand(*shape, n, generator=g, dtype=torch.float64) + 0.5  # noqa: E731
    mom, S, tm, tS = r(13).requires_grad_(), r(20).requires_grad_(), r(13), r(20)
    tm[..., F.MOMENT_INDEX["under"]] = float("nan")       # never selected
    fn = F.loss_batch if shots else F.loss_fn
    L = fn(mom, S, tm, tS, weights, sw)
    ref = _by_definition(mom, S, tm, tS, weights, sw)
    if not torch.is_tensor(ref):
        assert L.shape == shape and L.dtype == torch.float64 and not L.any()
        return
    torch.testing.assert_close(L, ref, rtol=1e-14, atol=0)
    got = torch.autograd.grad(L.sum(), (mom, S), allow_unused=True)
    want = torch.autograd.grad(ref.sum(), (mom, S), allow_unused=True)
    for a, b in zip(got, want):
        assert (a is None) == (b is None)
        if a is not None:
            torch.testing.assert_close(a, b, rtol=1e-13, atol=0)


def test_loss_of_a_spectrum_of_any_shape():
    g = torch.Generator().manual_seed(2)
    r = lambda *n: torch.rand(*n, generator=g, dtype=torch.float64) + 0.5  # noqa: E731
    mom, tm, S, tS = r(13), r(13), r(4, 5), r(4, 5)
    L = F.loss_fn(mom, S, tm, tS, {"mean": 2.0}, 1.0)
    ref = _by_definition(mom, S.reshape(-1), tm, tS.reshape(-1), {"mean": 2.0}, 1.0)
    torch.testing.assert_close(L, ref, rtol=1e-14, atol=0)


def test_targets_of_the_wrong_rank_are_refused():
    mom, S = torch.ones(3, 13, dtype=torch.float64), torch.ones(3, 4, dtype=torch.float64)
    with pytest.raises(IndexError):
        F.loss_batch(mom, S, mom[0], S, {"mean": 1.0}, 0.0)


@pytest.mark.parametrize("cols", [1, 5, 6, 7, 8, 9])
def test_shot_parameters_have_eight_columns(cols):
    b = object.__new__(B.Batch)
    b.n_shots = 3
    b.d_lasers, b.d_beams = (torch.zeros(3 * 80, dtype=torch.uint8) for _ in range(2))
    theta = torch.arange(3.0 * cols, dtype=torch.float64).reshape(3, cols)
    if cols in (6, 8):                     # one column is spread over the beam's three
        b.set_params(theta)
        torch.testing.assert_close(b.params(), theta.clone() if cols == 8 else torch.cat(
            [theta, theta[:, 5:], theta[:, 5:]], dim=1), rtol=0, atol=0)
    else:
        with pytest.raises(RuntimeError):
            b.set_params(theta)


@pytest.mark.gpu
def test_loss_with_a_target_on_the_host():
    g = torch.Generator().manual_seed(3)
    mom, tm = (torch.rand(13, generator=g, dtype=torch.float64) + 0.5 for _ in range(2))
    S = torch.empty(0, dtype=torch.float64)
    L = F.loss_fn(mom.cuda(), S.cuda(), tm, S, F.DEFAULT_MOMENT_WEIGHTS, 1.0)
    ref = _by_definition(mom, S, tm, S, F.DEFAULT_MOMENT_WEIGHTS, 1.0)
    torch.testing.assert_close(L.cpu(), ref, rtol=1e-14, atol=0)
