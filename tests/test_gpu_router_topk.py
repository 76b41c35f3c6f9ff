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
    (4096, 64, 20, 12, 4, 0),      # one k-step, 32 candidates
    (4097, 192, 65, 32, 16, 2),    # three slices of one k-step, 97 candidates, one token in the last tile
    (4400, 320, 129, 0, 1, 0),     # slices of unequal length, 129 candidates
    (5632, 128, 100, 61, 8, 1),    # as many tiles as three slices take, fewer k-steps than that
    (5700, 256, 33, 0, 5, 2),      # two accumulators of the large products
    (8449, 192, 200, 55, 8, 0),    # one slice, 255 candidates, an empty half tile
    (33000, 64, 160, 96, 3, 0),    # 256 candidates, more sort blocks than the router counts
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
