"""The router that also chooses (large batches), at the edges of its tiles, slices and column counts, and the selection
on logits with many ties, both against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_18643_b200 import inputs
from test_gpu_parity import check_route, oracle_route

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,Z,K,gate", [
    (4096, 64, 20, 12, 4, 0),      # one k-step, 32 candidates (the other router)
    (4097, 192, 65, 32, 16, 2),    # three slices of one k-step, 97 candidates, one token in the last tile
    (4400, 320, 129, 0, 1, 0),     # 129 candidates (the other router)
    (5632, 128, 100, 61, 8, 1),    # the same, fewer k-steps than slices
    (5700, 256, 33, 0, 5, 2),      # two accumulators of the large products
    (8449, 192, 200, 55, 8, 0),    # 255 candidates (the other router)
    (33000, 64, 160, 96, 3, 0),    # 256 candidates, more sort blocks than the router counts (the other router)
])
def test_router_with_top_k(T, d, E, Z, K, gate):
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("router", T=T, d=d, He=64, E=E, Z=Z, K=K, seed=31, zero_fraction=0.4 if Z else None)
    m = zeda.from_workload(wl, gate_mode=gate)
    x = wl.x.to("cuda:0")
    l, idx, w, counts, offsets, perm, P = oracle_route(wl, gate)
    for _ in range(2):  # each call clears the histograms that the call before it has filled
        check_route(m.route(x), idx, w, counts, offsets, perm, P)
    f, p, _ = m.stats(x)
    s = oracle.stats(l, idx, E, Z, alpha=1.0, group_w=1.0)
    assert np.allclose(f.cpu().numpy(), s["f"], rtol=1e-5, atol=1e-7)
    assert np.allclose(p.cpu().numpy(), s["P"], rtol=1e-4, atol=1e-7)
    assert np.array_equal(m.token_zero_share(T).cpu().numpy(), oracle.token_zero_share(idx, E).astype(np.float32))
    m.close()


@pytest.mark.parametrize("T,d,E,Z,K,gate,chooses", [
    (4400, 320, 65, 32, 7, 2, True),      # three slices, of one, two and two k-steps
    (5632, 128, 68, 32, 8, 1, True),      # two slices of one k-step
    (8448, 1024, 100, 60, 8, 0, True),    # as many tiles as two slices take
    (8449, 1024, 100, 60, 8, 0, False),   # one more: one slice would take longer than the two kernels
    (9472, 1024, 100, 60, 8, 0, False),   # the most tokens whose logits are one wave there
    (9473, 1024, 100, 60, 8, 0, True),    # one slice; a last tile of one token
    (4096, 1024, 192, 64, 8, 0, False),   # many candidates
    (33000, 256, 100, 30, 3, 2, True),    # more sort blocks than the router counts, two waves of one slice
    (18000, 64, 20, 12, 2, 0, True),      # one k-step, 32 candidates
    (4737, 2048, 200, 55, 8, 1, True),    # 255 candidates, an odd count; a last half tile of one token
    (5003, 2048, 150, 60, 3, 0, True),    # 210 candidates: 224 columns
])
def test_which_router_takes_a_call(T, d, E, Z, K, gate, chooses):
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("router", T=T, d=d, He=64, E=E, Z=Z, K=K, seed=33, zero_fraction=0.4)
    m = zeda.from_workload(wl, gate_mode=gate)
    x = wl.x.to("cuda:0")
    _, idx, w, counts, offsets, perm, P = oracle_route(wl, gate)
    check_route(m.route(x), idx, w, counts, offsets, perm, P)
    m.forward(x)
    place = 1 if T <= 256 * 128 else 3
    assert m.last_counters()[3] == (1 if chooses else 2) + place + 3
    m.close()


@pytest.mark.parametrize("T", [7, 60, 300])
@pytest.mark.parametrize("E,Z,K", [(40, 17, 16), (100, 28, 8), (150, 42, 8), (200, 50, 16), (300, 200, 16)])
def test_selection_among_equal_logits(T, E, Z, K):
    # a handful of distinct values, zeros of both signs among them: equal logits meet within a lane and across lanes
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("ties", T=T, d=64, He=64, E=E, Z=Z, K=K, seed=32, zero_fraction=None)
    m = zeda.from_workload(wl)
    l = np.random.default_rng(T + E).integers(-3, 4, (T, E + Z)).astype(np.float32) / 4
    l[::2][l[::2] == 0] = -0.0
    idx, w = oracle.route(l, E, Z, K, 0)
    check_route(m.route_from_logits(torch.from_numpy(l).to("cuda:0")), idx, w, *oracle.compact(idx, E))
    m.close()


@pytest.mark.parametrize("T,d,E,Z,K,rows", [
    (4097, 1024, 28, 12, 16, 20),    # each row twice, in other lanes
    (4800, 1024, 70, 30, 8, 32),     # up to four times in one lane
    (4737, 1024, 100, 60, 16, 40),   # in other lanes and registers
    (5633, 2048, 180, 70, 8, 32),
    (9473, 2048, 100, 60, 8, 20),    # one slice
])
def test_router_with_top_k_among_equal_logits_and_nan_tokens(T, d, E, Z, K, rows):
    # a few router rows repeated: the logits of their candidates are equal, bit for bit; every seventh token is NaN
    from paper_2605_18643_b200 import zeda
    n = E + Z
    wl = inputs.make_layer("equal", T=T + 256, d=d, He=64, E=E, Z=Z, K=K, seed=34, zero_fraction=None)
    wl.router_w = wl.router_w[torch.arange(n) % rows].contiguous()
    # logits of other rows are further apart than the fp32 sums are exact (4e-6 at these sizes)
    top = torch.topk(wl.x.float() @ wl.router_w[:rows].t(), min(K, rows - 1) + 1, dim=1).values
    wl.x = wl.x[(top[:, :-1] - top[:, 1:]).amin(dim=1) > 5e-5][:T].contiguous()
    wl.T = wl.x.shape[0]
    assert wl.T == T
    nan = np.arange(T) % 7 == 3
    x = wl.x.to("cuda:0")
    x[torch.from_numpy(nan).to(x.device)] = float("nan")
    _, idx, w, *_ = oracle_route(wl)
    idx[nan] = np.arange(K)  # equal keys throughout: the lowest ids
    m = zeda.from_workload(wl)
    m.forward(x)
    assert m.last_counters()[3] == 5  # the router that also chooses
    o = m.route(x)
    counts, offsets, perm, P = oracle.compact(idx, E)
    got = o["topk_w"].cpu().numpy()
    assert np.isnan(got[nan]).all()
    o["topk_w"][torch.from_numpy(nan).to(x.device)] = torch.from_numpy(w[nan]).float().to(x.device)
    check_route(o, idx, w, counts, offsets, perm, P)
    m.close()


@pytest.mark.parametrize("T", [4097, 8448, 9473])
def test_router_with_top_k_in_a_graph_and_without_dependent_launch(T):
    # it fetches router rows in front of its wait for the kernel before it, and clears its own histograms
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("router", T=T, d=1024, He=64, E=64, Z=32, K=8, seed=35)
    dev = torch.device("cuda:0")
    xs = [wl.x.to(dev), inputs.replica_tokens(wl, 3).to(dev)]
    plain = zeda.from_workload(wl, dev, flags=zeda.FLAG_NO_DEPENDENT_LAUNCH)
    want = [plain.forward(x).view(torch.int16) for x in xs]
    torch.cuda.synchronize()
    m = zeda.from_workload(wl, dev)
    for i in (0, 1, 0):
        assert torch.equal(m.forward(xs[i]).view(torch.int16), want[i])
    assert m.last_counters()[3] == 5
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
