"""The fit's losses called in other ways than a plain training step: after a
call in another torch mode."""
import pytest
import torch
from torch.fx.experimental.proxy_tensor import make_fx

from paper_2308_09348_gb300 import fit as F

NONE = torch.empty(0, dtype=torch.float64)


def _moments(seed, *shape):
    g = torch.Generator().manual_seed(seed)
    return torch.rand(*shape, 13, generator=g, dtype=torch.float64) + 0.5


def _reference(mom, tm, weights):
    """The moments' part, term by term in the inputs' type, summed in 64 bits."""
    L = torch.zeros(mom.shape[:-1], dtype=torch.float64, device="cpu")
    for k, c in weights.items():
        i = F.MOMENT_INDEX[k]
        L = L + c * ((mom[..., i] - tm[..., i]) / (tm[..., i].abs() + 1e-30)) ** 2
    return L


@pytest.mark.parametrize("weights", [{"mean": 1.5, "div_x": 1.5}, {"mean_aeff": 1.0, "mean": 3.0}])
@pytest.mark.parametrize("mode", ["inference", "default device", "traced"])
def test_a_call_leaves_nothing_behind_for_another_mode(mode, weights):
    mom, tm = _moments(1), _moments(2)

    def loss(m):
        return F.loss_fn(m, NONE, tm, NONE, weights, 0.0)

    if mode == "inference":
        with torch.inference_mode():
            loss(mom)
    elif mode == "default device":
        torch.set_default_device("meta")
        try:
            torch.testing.assert_close(loss(mom), _reference(mom, tm, weights), rtol=1e-14, atol=0)
        finally:
            torch.set_default_device(None)
    else:
        make_fx(lambda m, t: F.loss_fn(m, NONE, t, NONE, weights, 0.0), tracing_mode="fake")(mom, tm)
    m = mom.clone().requires_grad_()
    L, ref = loss(m), _reference(m, tm, weights)
    torch.testing.assert_close(L, ref, rtol=1e-14, atol=0)
    torch.testing.assert_close(torch.autograd.grad(L, m)[0], torch.autograd.grad(ref, m)[0],
                               rtol=1e-13, atol=0)


@pytest.mark.parametrize("weights", [{"mean": 1.0, "spread": 1.0, "div_x": 1.0, "div_y": 1.0},
                                     {"mean": 2.0, "spread": 1.0, "div_x": 1.0, "div_y": 0.5}])
@pytest.mark.parametrize("shots", [0, 3])
@pytest.mark.parametrize("one_by_one", [False, True])
def test_terms_of_32_bits_are_summed_in_64(weights, shots, one_by_one):
    # terms of 1 and of a few 2^-24: every one of them is lost in a 32-bit sum
    mom = torch.ones(*((shots,) if shots else ()), 13, dtype=torch.float32)
    tm = torch.full_like(mom, 1.0 + 2.0 ** -12)
    tm[..., F.MOMENT_INDEX["mean"]] = 0.5
    fn = F.loss_batch if shots else F.loss_fn
    S = torch.empty(*mom.shape[:-1], 0)
    target = tm.unsqueeze(-1) if one_by_one else tm    # another rank: moment by moment
    L = fn(mom, S, target, S, weights, 0.0)
    ref = _reference(mom, tm, weights)
    assert L.dtype == torch.float64 and bool((ref > weights["mean"]).all())
    if one_by_one:                                     # every shot against every target
        L = L.diagonal() if shots else L.squeeze(0)
    torch.testing.assert_close(L, ref, rtol=1e-15, atol=0)


@pytest.mark.parametrize("kind", [list, tuple, lambda t: dict(enumerate(t))])
def test_a_target_of_single_values(kind):
    mom, tm = _moments(3).requires_grad_(), _moments(4)
    weights = F.DEFAULT_MOMENT_WEIGHTS
    L = F.loss_fn(mom, NONE, kind(tm.unbind()), NONE, weights, 0.0)
    torch.testing.assert_close(L, _reference(mom, tm, weights), rtol=1e-15, atol=0)
    assert torch.autograd.grad(L, mom)[0].isfinite().all()


@pytest.mark.parametrize("weights", [{}, {"mean": 1.0}])
def test_one_loss_per_shot_from_a_shared_spectrum(weights):
    mom, tm = _moments(5, 3), _moments(6, 3)
    S, tS = torch.full((1, 4), 1.5, dtype=torch.float64), torch.ones(1, 4, dtype=torch.float64)
    L = F.loss_batch(mom, S, tm, tS, weights, 1.0)
    # 4 bins off by 0.5, normalised by their sum 4, times 4 bins
    torch.testing.assert_close(L, _reference(mom, tm, weights) + 4 * (0.5 / 4) ** 2 * 4, rtol=1e-15,
                               atol=0)


@pytest.mark.parametrize("weights", [{"mean": 2.0, "mean_aeff": 2.0}, {"mean": 2.0, "div_x": 3.0}])
def test_columns_of_moments(weights):
    # moments along the first of two dimensions, and a target with more entries
    mom, tm = _moments(7, 4).T.requires_grad_(), _moments(8, 4).T
    ref = _reference(mom.T, tm.T, weights)
    for target in (tm, torch.cat([tm, tm])):
        L = F.loss_fn(mom, NONE, target, NONE, weights, 0.0)
        torch.testing.assert_close(L, ref, rtol=1e-15, atol=0)
        torch.testing.assert_close(torch.autograd.grad(L.sum(), mom)[0],
                                   torch.autograd.grad(ref.sum(), mom, retain_graph=True)[0],
                                   rtol=1e-14, atol=0)
    with pytest.raises(IndexError):
        F.loss_fn(mom[:5], NONE, tm[:5], NONE, {"mean_aeff": 1.0}, 0.0)


@pytest.mark.parametrize("shots", [0, 3])
def test_moments_without_weight_may_be_anything(shots):
    # neither value, gradient, second derivative nor tangent sees them
    weights = {"mean": 1.5, "spread": 1.5}
    fn = F.loss_batch if shots else F.loss_fn
    mom, tm = (_moments(k, *((shots,) if shots else ())) for k in (9, 10))
    mom[..., F.MOMENT_INDEX["div"]] = float("inf")
    tm[..., F.MOMENT_INDEX["W"]] = float("nan")
    tm[..., F.MOMENT_INDEX["over"]] = 0.0
    mom.requires_grad_()
    S = torch.empty(*mom.shape[:-1], 0)
    L, ref = fn(mom, S, tm, S, weights, 0.0), _reference(mom, tm, weights)
    torch.testing.assert_close(L, ref, rtol=1e-15, atol=0)
    g, gr = (torch.autograd.grad(x.sum(), mom, create_graph=True)[0] for x in (L, ref))
    torch.testing.assert_close(g, gr, rtol=1e-14, atol=0)
    v = torch.ones_like(mom)
    h, hr = (torch.autograd.grad((x[..., 1:3]).sum(), mom)[0] for x in (g, gr))
    torch.testing.assert_close(h, hr, rtol=1e-14, atol=0)
    _, t = torch.func.jvp(lambda m: fn(m, S, tm, S, weights, 0.0), (mom.detach(),), (v,))
    torch.testing.assert_close(t, g.detach()[..., 1:3].sum(-1), rtol=1e-14, atol=0)
    if shots:
        vm = torch.func.vmap(lambda m, s, r: F.loss_fn(m, s, r, s, weights, 0.0))(mom, S, tm)
        torch.testing.assert_close(vm, ref, rtol=1e-15, atol=0)
