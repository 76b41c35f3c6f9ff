"""The combine at the edges of its forms: rows that end inside a warp's share, K up to 16, few and many warps."""
import pytest
import torch

from paper_2605_18643_b200 import inputs
from test_gpu_parity import check_y, oracle_forward, sample_tokens

pytestmark = pytest.mark.gpu


LINE = 16  # warps of two chunks per lane, per SM, from which on they have two


@pytest.mark.parametrize("T,few,d,E,Z,K,gate,kind", [
    (17, True, 64, 20, 12, 16, 0, 0),     # eight chunks of a row; more slots than are requested at a time
    (40, True, 320, 20, 0, 9, 1, 0),      # a second warp with eight chunks; nine slots, none zero
    ("last", True, 576, 20, 12, 3, 2, 1),    # copy experts, a last share of eight chunks, few warps of one chunk per lane ...
    ("first", False, 576, 20, 12, 3, 2, 1),  # ... and one token more: two chunks per lane
    (4500, False, 576, 20, 12, 5, 0, 1),  # five slots, requested four at a time
    (700, False, 2112, 20, 12, 4, 0, 0),  # a last share of eight chunks behind four full ones
])
def test_layer_against_the_oracle(T, few, d, E, Z, K, gate, kind):
    from paper_2605_18643_b200 import zeda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pieces = -(-d // 512)
    if isinstance(T, str):  # on either side of the line
        T = -(-LINE * sms // pieces) - (T == "last")
    assert (T * pieces < LINE * sms) == few  # the form that the launch takes for this size
    wl = inputs.make_layer("combine", T=T, d=d, He=64, E=E, Z=Z, K=K, seed=47, zero_fraction=0.5 if Z else None)
    m = zeda.from_workload(wl, gate_mode=gate, expert_kind=kind)
    y = m.forward(wl.x.to("cuda:0")).cpu()
    ids = sample_tokens(T, min(T, 200), 5)
    ids[-1] = T - 1
    check_y(y[torch.from_numpy(ids).long()], oracle_forward(wl, token_ids=ids, gate_mode=gate, expert_kind=kind)[0])
    m.close()
