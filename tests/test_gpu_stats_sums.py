"""The final sums of the routing statistics at the edges of their column groups, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_18643_b200 import inputs
from test_gpu_parity import oracle_route

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,Z,K,d", [
    (40, 3, 2, 2, 64),        # odd: pairs of columns, many threads per group
    (1100, 200, 101, 4, 64),  # odd and more groups than threads: two turns
    (700, 340, 172, 8, 64),   # as many groups of four as threads
    (4500, 5, 5, 3, 64),      # 51 threads per group
    (4500, 200, 312, 8, 64),  # a thread per group of four, 71 rows: three turns of 32
    (3000, 200, 55, 8, 64),   # the same with pairs, 47 rows: two turns
    (32800, 7, 4, 2, 64),     # a kernel of its own: pairs, 93 threads a group
    (32800, 300, 212, 4, 64), # the same, four threads a group
    (33, 128, 64, 8, 2048),   # few tokens of long rows: one row, and four
    (193, 128, 64, 8, 2048),
    (255, 150, 73, 8, 1088),  # (eight logits a lane)
])
def test_final_sums_of_the_statistics(T, E, Z, K, d):
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("stats", T=T, d=d, He=64, E=E, Z=Z, K=K, seed=43, zero_fraction=0.4)
    m = zeda.from_workload(wl)
    x = wl.x.to("cuda:0")
    l, idx, *_ = oracle_route(wl)
    s = oracle.stats(l, idx, E, Z, alpha=1.0, group_w=1.0)
    # counts are whole numbers and exact in fp32; a probability is an fp32 exponential of a logit that is off by up to 2e-5
    f_ref, p_ref = s["f"], s["P"]
    for _ in range(2):
        f, p, o = m.stats(x)
        f, p, o = (t.cpu().numpy().astype(np.float64) for t in (f, p, o))
        assert np.allclose(f, f_ref, rtol=2e-7, atol=0) and np.allclose(p, p_ref, rtol=5e-5, atol=1e-9)
        want = [f_ref[E:].sum() / K, (f_ref * p_ref).sum(), f_ref[:E].sum() * p_ref[:E].sum(), f_ref[E:].sum() * p_ref[E:].sum()]
        assert np.allclose(o, want, rtol=1e-4, atol=1e-9)
    # each result may be left out
    out = torch.empty(4, device=x.device)
    stream = torch.cuda.current_stream().cuda_stream
    assert zeda.lib.zeda_moe_stats(m._h, x.data_ptr(), T, None, None, out.data_ptr(), stream) == zeda.OK
    assert np.array_equal(out.cpu().numpy().astype(np.float64), o)
    assert zeda.lib.zeda_moe_stats(m._h, x.data_ptr(), T, None, None, None, stream) == zeda.OK
    m.last_counters()
    m.close()
