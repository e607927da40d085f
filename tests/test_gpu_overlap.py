"""qs_scatter's three kernels overlap at their edges (the evaluation starts
while the accumulators are cleared): calls that follow one another without a
wait, share their workspace and read samples that the kernel just before them
wrote give what separate calls give; also from a captured graph and with
timing events around the kernel."""
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


@pytest.mark.parametrize("model,prec,n", [(I.MODEL_LL, "f32", 300_001), (I.MODEL_LL, "f64", 5_000),
                                          (I.MODEL_QFP, "f32", 20_011), (I.MODEL_QFP, "f64", 999)])
def test_calls_in_a_row(model, prec, n):
    wl = I.full_qfp(n)
    L = I.Laser(**{**wl.laser.__dict__, "model": model, "n_phase": 16})
    sets = []
    for k in range(4):
        g = torch.Generator(device="cuda")
        g.manual_seed(k)
        sets.append([torch.randn(n, generator=g, device="cuda") for _ in range(8)])
    ref = []
    for xi in sets:
        o = B.qs_scatter(L, wl.beam, xi, wl.bins, precision=prec)
        torch.cuda.synchronize()
        ref.append([t.clone() for t in (o.spectrum, o.divmap, o.aeff_hist, o.moments)])
    xi = [torch.empty(n, device="cuda") for _ in range(8)]
    out = B.Outputs(wl.bins, n, precision=prec)

    def chain(events=None):
        got = []
        for s in sets:
            for a, b in zip(xi, s):
                a.copy_(b)                        # written on the stream just before the call
            B.qs_scatter(L, wl.beam, xi, wl.bins, precision=prec, out=out, kernel_events=events)
            got.append([t.clone() for t in (out.spectrum, out.divmap, out.aeff_hist, out.moments)])
        return got

    ev = (torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    for got in (chain(), chain(ev)):
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
    with torch.cuda.stream(stream):
        chain()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        got = chain()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, ref):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
