"""The router of 33 to 255 tokens at the edges of its tiles, stages and waves, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2605_18643_b200 import inputs
from test_gpu_parity import check_route, oracle_route

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,Z,K,gate", [
    (33, 2048, 140, 60, 8, 0),     # a second tile of one token, a last candidate tile of eight
    (64, 1088, 200, 32, 16, 2),    # a last stage of 64 elements: chains of nine steps and of eight
    (65, 2048, 128, 64, 8, 1),     # tiles of 40 tokens by eight CTAs
    (128, 8192, 33, 0, 5, 0),      # eight stages; a last candidate tile of one
    (129, 4096, 300, 100, 8, 0),   # two waves of tiles of 32 tokens by four CTAs
    (255, 2048, 40, 23, 4, 1),     # an odd number of candidates
    (129, 2048, 384, 128, 8, 0),   # two waves of tiles of 40 tokens
    (65, 2048, 64, 32, 4, 0),      # a last tile of one token
    (64, 2048, 64, 32, 4, 0),      # full tiles
    (255, 960, 40, 24, 4, 0),
    (224, 2048, 128, 64, 8, 0),    # tiles of 48 tokens
    (241, 2048, 128, 64, 8, 2),    # tiles of 56 tokens
    (128, 1088, 300, 101, 16, 0),  # tiles of 64 tokens
])
@pytest.mark.parametrize("bias", [0.0, 50.0])
def test_router_of_33_to_255_tokens(T, d, E, Z, K, gate, bias):
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("slices", T=T, d=d, He=64, E=E, Z=Z, K=K, seed=37, zero_fraction=0.4 if Z else None)
    # a bias far above the logits: it has to be added once, behind the products (a sum that carries it loses the logits' last bits)
    b = torch.zeros(E + Z) if wl.router_bias is None else wl.router_bias.clone()
    wl.router_bias = b + bias
    m = zeda.from_workload(wl, gate_mode=gate)
    x = wl.x.to("cuda:0")
    l, idx, w, counts, offsets, perm, P = oracle_route(wl, gate)
    # the logits' error: sums of fp32 products (2e-6 at most at these sizes) and one rounding of a logit of the bias' size
    tol = 2e-6 + 2.0 ** -24 * (bias + np.abs(l).max())
    top = -np.sort(-l.astype(np.float64), axis=1)[:, :K + 1]
    assert float((top[:, :-1] - top[:, 1:]).min()) > 4 * tol  # so that the choice is the oracle's
    for _ in range(2):  # each call clears the histograms that the call before it has filled
        o = m.route(x)
        assert np.array_equal(o["topk_idx"].cpu().numpy(), idx)
        # a weight is a ratio of exponentials of logits: its relative error is at most the errors of two logits, and rounding
        assert np.allclose(o["topk_w"].cpu().numpy(), w, rtol=2 * tol + 1e-6, atol=1e-30)
        check_route(dict(o, topk_w=torch.from_numpy(np.ascontiguousarray(w))), idx, w, counts, offsets, perm, P)
    m.close()


@pytest.mark.parametrize("T", [33, 129, 255])
def test_router_of_33_to_255_tokens_in_a_graph_and_without_dependent_launch(T):
    # it asks for router rows in front of its wait for the kernel before it
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("slices", T=T, d=2112, He=64, E=64, Z=32, K=8, seed=38, zero_fraction=0.4)
    dev = torch.device("cuda:0")
    xs = [wl.x.to(dev), inputs.replica_tokens(wl, 3).to(dev)]
    plain = zeda.from_workload(wl, dev, flags=zeda.FLAG_NO_DEPENDENT_LAUNCH)
    want = [plain.forward(x).view(torch.int16) for x in xs]
    torch.cuda.synchronize()
    m = zeda.from_workload(wl, dev)
    for i in (0, 1, 0):
        assert torch.equal(m.forward(xs[i]).view(torch.int16), want[i])
    x, y, y2 = xs[0].clone(), torch.empty_like(xs[0]), torch.empty_like(xs[0])
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):  # two calls: the second starts under the first
        m.forward(x, y)
        m.forward(y, y2)
    for src in (1, 0, 1):
        x.copy_(xs[src])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(y.view(torch.int16), want[src])
        assert torch.equal(y2.view(torch.int16), plain.forward(y.clone()).view(torch.int16))
    del graph
    m.close()
    plain.close()
