"""Up to 255 tokens a token's routing does not depend on the batch: the bits of its logits and of its routing weights are
those of any other batch of up to 32 tokens, or of 33 to 255, whichever kernel its size and shape send it to."""
import pytest
import torch

from paper_2605_18643_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,E,Z,K,gate", [
    (2048, 128, 64, 8, 0),
    (2048, 64, 32, 4, 2),
    (1024, 64, 32, 8, 1),
    (8192, 200, 60, 8, 0),
    (1088, 300, 101, 16, 0),   # rows that end inside a run of 128; an odd number of candidates
    (192, 40, 24, 4, 0),
])
def test_a_token_is_routed_alike_in_batches_of_any_size(d, E, Z, K, gate):
    from paper_2605_18643_b200 import zeda
    wl = inputs.make_layer("batch_size", T=255, d=d, He=64, E=E, Z=Z, K=K, seed=53, zero_fraction=0.4)
    m = zeda.from_workload(wl, gate_mode=gate)
    x = wl.x.to("cuda:0")
    for sizes in ((32, 1, 2, 4, 7, 17), (255, 33, 64, 65, 96, 97, 128, 129, 160, 193, 224, 254)):
        ref = None
        for T in sizes:
            part = x[:T].contiguous()
            logits, o = m.router_logits(part), m.route(part)
            own = m.route_from_logits(logits)  # what the logits that the library shows give
            assert torch.equal(o["topk_idx"], own["topk_idx"]) and torch.equal(o["topk_w"].view(torch.int32), own["topk_w"].view(torch.int32)), T
            if ref is None:
                ref = (logits, o["topk_idx"], o["topk_w"])
            assert torch.equal(logits.view(torch.int32), ref[0][:T].view(torch.int32)), T
            assert torch.equal(o["topk_idx"], ref[1][:T]) and torch.equal(o["topk_w"].view(torch.int32), ref[2][:T].view(torch.int32)), T
    m.close()
