"""The expert kernels for the smallest batches (csrc/small_batch.cu) against the CPU oracle, at the edges
of their tiles: 8 pair rows per column tile, 16 weight rows per block, reduction slices with a remainder,
the last batch size that takes them and the first that does not."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_18643_b200 import inputs

pytestmark = pytest.mark.gpu

# bf16 results of fp32 sums against 64 bits: three roundings of 2^-9 (Hmid, expert output, y)
REL_L2, MAX_ABS_RMS = 1e-2, 5e-2


def layer(T, d=256, He=128, E=8, Z=4, K=2, seed=5, zero_fraction=0.5):
    return inputs.make_layer("small", T=T, d=d, He=He, E=E, Z=Z, K=K, seed=seed,
                             zero_fraction=zero_fraction if Z else None)


@pytest.mark.parametrize("T,shape,kind", [
    (1, {}, 0), (2, {}, 1), (5, {}, 0), (8, {}, 0), (9, {}, 1), (16, {}, 0), (17, {}, 0), (32, {}, 0), (33, {}, 0),
    (7, dict(d=320, He=192), 0), (16, dict(d=64, He=64), 1), (3, dict(d=1088, He=832), 0),   # slices with remainders
    (8, dict(E=1, Z=1, K=2), 0), (16, dict(E=1, Z=0, K=1), 0),                               # every token on one expert
    (16, dict(E=40, Z=8, K=16), 0), (9, dict(E=300, Z=100, K=16), 1),                        # widest slot table, many experts
    (16, dict(E=24, Z=8, K=16), 0), (2, dict(E=300, Z=100, K=16), 1), (1, dict(E=384, Z=128, K=16), 0),  # the same on these kernels
    (4, dict(d=2048, He=768, E=16, Z=8, K=8), 0),
])
def test_small_batches_match_the_oracle(T, shape, kind):
    from paper_2605_18643_b200 import zeda
    wl = layer(T, **shape)
    dev = torch.device("cuda:0")
    m = zeda.from_workload(wl, dev, expert_kind=kind)
    x = wl.x.to(dev)
    y = m.forward(x)
    r = torch.randn(wl.T, wl.d, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16).to(dev)
    want_r = (r.float() + y.float()).to(torch.bfloat16)
    want_h = zeda.residual_rmsnorm(want_r.clone(), None)
    h = torch.empty_like(r)
    m.forward_residual(x, r, h)
    torch.cuda.synchronize()
    bias = None if wl.router_bias is None else wl.router_bias.numpy()
    y_ref, idx, _ = oracle.forward(inputs.bits(wl.x), wl.router_w.numpy(), bias, inputs.bits(wl.w_gate_up),
                                   inputs.bits(wl.w_down), wl.E, wl.Z, wl.K, expert_kind=kind)
    got = y.float().cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - y_ref) <= REL_L2 * np.linalg.norm(y_ref)
    assert np.max(np.abs(got - y_ref)) <= MAX_ABS_RMS * max(np.sqrt(np.mean(y_ref ** 2)), 1e-30)
    assert torch.equal(r.view(torch.int16), want_r.view(torch.int16))
    assert torch.equal(h.view(torch.int16), want_h.view(torch.int16))
    if kind == 0:
        dead = np.nonzero((idx >= wl.E).all(axis=1))[0]
        if dead.size:
            assert int(y[torch.as_tensor(dead, device=dev)].view(torch.int16).abs().max().item()) == 0
    P, U, zero_slots = m.last_counters()[:3]  # what the kernels that route themselves leave in the handle
    real = idx[idx < wl.E]
    assert (P, U, zero_slots) == (real.size, np.unique(real).size, idx.size - real.size)
    share = (idx >= wl.E).mean(axis=1).astype(np.float32)
    assert np.array_equal(m.token_zero_share(T).cpu().numpy(), share)
    m.close()


@pytest.mark.parametrize("He,K", [(128, 4), (1024, 2)])
@pytest.mark.parametrize("E,Z,gate", [(32, 32, 0), (64, 64, 1), (100, 60, 2), (150, 100, 0), (200, 200, 1)])
def test_down_kernel_fetches_the_routing_or_repeats_it(E, Z, gate, He, K):
    # Launched in stream order the down kernel always finds gate/up's tables.  With dependent launch it starts as gate/up's
    # CTAs leave, and where these have little to do (H_e 128) nearly all of its CTAs are there before the tables and
    # route for themselves.  Copy experts: the routing weights of zero slots count too.
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("routed", T=8, d=1024, He=He, E=E, Z=Z, K=K, seed=36, zero_fraction=0.5)
    xs = [wl.x.to("cuda:0"), inputs.replica_tokens(wl, 5).to("cuda:0")]
    kw = dict(gate_mode=gate, expert_kind=zeda.EXPERT_COPY)
    plain = zeda.from_workload(wl, flags=zeda.FLAG_NO_DEPENDENT_LAUNCH, **kw)
    m = zeda.from_workload(wl, **kw)
    for T in (1, 2, 5, 8):
        x = [a[:T].contiguous() for a in xs]
        want = [plain.forward(a) for a in x]
        assert plain.last_counters()[3] == 3 and not torch.equal(want[0], want[1])
        got = [torch.empty_like(x[0]) for _ in range(20)]
        torch.cuda.synchronize()
        for i, y in enumerate(got):  # no synchronisation in between
            m.forward(x[i % 2], y)
        torch.cuda.synchronize()
        for i, y in enumerate(got):
            assert torch.equal(y.view(torch.int16), want[i % 2].view(torch.int16)), (T, i)
    m.close()
    plain.close()


@pytest.mark.parametrize("T", [1, 8, 16])
def test_small_batches_in_a_graph_and_without_dependent_launch(T):
    # the expert kernels here read the routing results in front of their wait for the kernel before them
    from paper_2605_18643_b200 import zeda
    wl = layer(T)
    dev = torch.device("cuda:0")
    xs = [wl.x.to(dev), inputs.replica_tokens(wl, 3).to(dev)]
    plain = zeda.from_workload(wl, dev, flags=zeda.FLAG_NO_DEPENDENT_LAUNCH)
    want = [plain.forward(x).view(torch.int16) for x in xs]
    torch.cuda.synchronize()
    m = zeda.from_workload(wl, dev)
    for x, w in zip(xs, want):
        assert torch.equal(m.forward(x).view(torch.int16), w)
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


@pytest.mark.parametrize("T,shape,streams", [
    (8, dict(d=256, He=128, E=64, Z=32, K=4), True),
    (16, dict(d=2048, He=768, E=32, Z=16, K=4), True),
    (2, dict(d=1024, He=256, E=256, Z=0, K=16), True), (8, dict(d=1024, He=256, E=256, Z=0, K=16), False),
    (8, dict(d=1024, He=512, E=192, Z=64, K=16), False), (16, dict(d=4096, He=1536, E=24, Z=8, K=8), False),
])
def test_which_kernels_a_small_batch_takes(T, shape, streams):
    # many active experts per call, or a down projection that leaves SMs idle: the kernels for larger batches
    # (router, routing, two GEMMs, combine) are the faster ones (N 256, K 16, 8 tokens: 52 us against 69)
    from paper_2605_18643_b200 import zeda
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(1)
    E, Z, K, d, He = (shape[k] for k in ("E", "Z", "K", "d", "He"))
    w = [torch.empty(s, dtype=torch.bfloat16, device=dev).normal_(0, 0.02, generator=g) for s in ((E, 2 * He, d), (E, d, He))]
    rw = torch.empty(E + Z, d, device=dev).normal_(0, 0.02, generator=g)
    x = torch.randn(T, d, generator=g, device=dev).to(torch.bfloat16)
    m = zeda.ZedaMoE(rw, None, w[0], w[1], E, Z, K, 40)
    y = m.forward(x)
    assert m.last_counters()[3] == ((3 if T <= 8 else 4) if streams else 5)
    # rows of a batch that is too large for these kernels: the same expert sums in another order
    many = m.forward(torch.cat([x, torch.randn(24, d, generator=g, device=dev).to(torch.bfloat16)]))[:T]
    assert m.last_counters()[3] == 5
    assert float((y.float() - many.float()).norm() / many.float().norm()) <= (REL_L2 if streams else 1e-3)
    m.close()
