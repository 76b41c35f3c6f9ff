"""Calls in a row on one handle, on inputs that route differently and without a host synchronisation in between:
each kernel is launched while the one in front still runs, and must read what that one writes and not what
the call before has left in the same buffers.  (On a repeated input stale results are the right ones.)"""
import pytest
import torch

from paper_2605_18643_b200 import inputs

pytestmark = pytest.mark.gpu

SHAPE = dict(d=512, He=256, E=64, Z=32, K=8)


class Call:
    """One call with outputs of its own, made ahead so that nothing stands between the calls in the stream."""

    def __init__(self, zeda, m, use, x):
        lib, h, T, stream = zeda.lib, m._h, x.shape[0], torch.cuda.current_stream().cuda_stream
        if use == "forward":
            self.out = [torch.empty_like(x)]
            self.run = lambda: m.forward(x, self.out[0])
        elif use == "residual":
            self.out = [x.flip(1).contiguous(), torch.empty_like(x)]
            self.run = lambda: m.forward_residual(x, *self.out)
        elif use == "stats":
            n = m.E + m.Z
            self.out = [torch.empty(k, device=x.device) for k in (n, n, 4, T)]

            def run():
                p = [t.data_ptr() for t in self.out]
                assert lib.zeda_moe_stats(h, x.data_ptr(), T, p[0], p[1], p[2], stream) == zeda.OK
                assert lib.zeda_moe_token_zero_share(h, T, p[3], stream) == zeda.OK
            self.run = run
        else:
            o = m._route_outputs(T)
            self.out = [o[k] for k in ("topk_idx", "topk_w", "counts", "offsets", "perm", "n_pairs")]
            self.run = lambda: self._ok(lib.zeda_route(h, x.data_ptr(), T, *[t.data_ptr() for t in self.out], stream), zeda)

    @staticmethod
    def _ok(status, zeda):
        assert status == zeda.OK

    def same(self, other):
        return all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(self.out, other.out))


def check(zeda, m, plan):
    """plan: list of (key, use, x).  Every call of the row gives the bits of a call of the same key on its own."""
    alone, row = {}, []
    for key, use, x in plan:
        row.append((key, Call(zeda, m, use, x)))
        if key not in alone:
            alone[key] = Call(zeda, m, use, x)
            torch.cuda.synchronize()
            alone[key].run()
            torch.cuda.synchronize()
    for _, c in row:
        c.run()
    torch.cuda.synchronize()
    for i, (key, c) in enumerate(row):
        assert c.same(alone[key]), (i, key)
    m.last_counters()  # no device-side failure recorded
    return alone


@pytest.fixture(scope="module")
def layer():
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("back_to_back", T=2048, seed=41, zero_fraction=0.5, **SHAPE)
    xs = [wl.x.to("cuda:0"), inputs.replica_tokens(wl, 7).to("cuda:0")]
    return zeda, wl, xs


@pytest.mark.parametrize("use", ["forward", "residual", "stats", "route"])
@pytest.mark.parametrize("T", [1, 8, 16, 129, 300, 777, 2048])
def test_alternating_inputs_give_the_bits_of_single_calls(layer, T, use):
    zeda, wl, xs = layer
    m = zeda.from_workload(wl, max_tokens=2048)
    alone = check(zeda, m, [(i % 2, use, xs[i % 2][:T].contiguous()) for i in range(20)])
    assert not alone[0].same(alone[1])
    m.close()


@pytest.fixture(scope="module")
def large_layer():
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("back_to_back", T=9473, d=1024, He=64, E=64, Z=32, K=8, seed=42, zero_fraction=0.5)
    return zeda, wl, [wl.x.to("cuda:0"), inputs.replica_tokens(wl, 7).to("cuda:0")]


@pytest.mark.parametrize("use", ["forward", "residual", "stats", "route"])
@pytest.mark.parametrize("T", [4096, 5633, 8449, 9473])
def test_alternating_large_batches_give_the_bits_of_single_calls(large_layer, T, use):
    # the router with top-K in three slices, two and one, and between them a size that the other router takes
    zeda, wl, xs = large_layer
    m = zeda.from_workload(wl)
    alone = check(zeda, m, [(i % 2, use, xs[i % 2][:T].contiguous()) for i in range(20)])
    assert not alone[0].same(alone[1])
    m.forward(xs[0][:T].contiguous())
    assert m.last_counters()[3] == (6 if T == 8449 else 5)
    m.close()


@pytest.fixture(scope="module")
def long_rows():
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("back_to_back", T=255, d=3136, He=64, E=64, Z=32, K=8, seed=44, zero_fraction=0.5)
    return zeda, wl, [wl.x.to("cuda:0"), inputs.replica_tokens(wl, 7).to("cuda:0")]


@pytest.mark.parametrize("use", ["forward", "stats", "route"])
@pytest.mark.parametrize("T", [40, 129, 255])
def test_alternating_inputs_whose_rows_pass_through_shared_memory_in_stages(long_rows, T, use):
    # the router of 33 to 255 tokens: router rows asked for in front of its wait, and four stages in the room of two
    zeda, wl, xs = long_rows
    m = zeda.from_workload(wl)
    alone = check(zeda, m, [(i % 2, use, xs[i % 2][:T].contiguous()) for i in range(20)])
    assert not alone[0].same(alone[1])
    m.close()


def test_batches_around_the_router_on_clusters_in_any_order(long_rows):
    zeda, wl, xs = long_rows
    m = zeda.from_workload(wl)
    order = [(T, use) for T in (255, 32, 33, 129, 1, 65, 254, 193, 8, 97) for use in ("forward", "stats", "route")]
    check(zeda, m, [((T, use, i % 2), use, xs[i % 2][:T].contiguous()) for i, (T, use) in enumerate(order)])
    m.close()


def test_large_batches_in_any_order(large_layer):
    zeda, wl, xs = large_layer
    m = zeda.from_workload(wl)
    order = [(T, use) for T in (9473, 8449, 300, 4096, 8, 5633, 9473, 4095, 5003) for use in ("forward", "stats", "residual", "route")]
    check(zeda, m, [((T, use, i % 2), use, xs[i % 2][:T].contiguous()) for i, (T, use) in enumerate(order)])
    m.close()


def test_batch_sizes_and_uses_in_any_order(layer):
    zeda, wl, xs = layer
    m = zeda.from_workload(wl, max_tokens=2048)
    order = [(T, use) for T in (2048, 1, 300, 16, 1, 777, 8, 129, 40, 2048, 9, 160) for use in ("forward", "stats", "residual", "route")]
    check(zeda, m, [((T, use, i % 2), use, xs[i % 2][:T].contiguous()) for i, (T, use) in enumerate(order)])
    m.close()


@pytest.mark.parametrize("T", [40, 300, 2048])
def test_expert_parallel_calls_in_a_row(layer, T):
    zeda, wl, xs = layer
    dev = torch.device("cuda:0")
    m = zeda.ZedaMoE(wl.router_w.to(dev), wl.router_bias.to(dev), wl.w_gate_up.to(dev), wl.w_down.to(dev), wl.E, wl.Z, wl.K, T,
                     ep_size=1, max_recv_pairs=T * wl.K)
    xs = [x[:T].contiguous() for x in xs]

    def run(x, n_rows):
        send_rows, send_counts, counts = m.ep_dispatch(x)
        if n_rows is None:
            n_rows = int(send_counts.sum())
        rows = m.ep_experts(send_rows, counts.view(1, -1), n_rows)
        return n_rows, [send_rows, send_counts, counts, m.ep_combine(x, rows)]

    alone = []
    for x in xs:
        alone.append(run(x, None))
        torch.cuda.synchronize()
    got = [run(xs[i % 2], alone[i % 2][0]) for i in range(20)]
    torch.cuda.synchronize()
    for i, (P, out) in enumerate(got):
        want = alone[i % 2][1]
        assert torch.equal(out[0][:P].view(torch.int16), want[0][:P].view(torch.int16)), i
        assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(out[1:], want[1:])), i
    assert not torch.equal(alone[0][1][3], alone[1][1][3])
    m.last_counters()
    m.close()
