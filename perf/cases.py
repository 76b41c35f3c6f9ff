"""Timed cases of the zero-expert MoE layer: the calls that a user of the library makes.

The layer shapes are the two of the benchmark: the Qwen3-30B-A3B-shaped layer (d 2048, H_e 768, N 128, N_Z 64,
K 8) and the GLM-shaped one (d 2048, H_e 1536, N 64, N_Z 32, K 4).  A case names one of five uses:

  forward  one layer call on device tensors (ZedaMoE.forward)
  stack    a residual stream through several layers, each with weights of its own (residual_rmsnorm in front,
           then ZedaMoE.forward_residual per layer)
  host     one layer call on pinned host buffers (ZedaMoE.forward_host)
  ep       one expert-parallel layer call of a group of one (ExpertParallelMoE over a LoopbackExchange)
  stats    the routing statistics that the load-balancing losses are built from (ZedaMoE.stats,
           ZedaMoE.token_zero_share)
"""
import functools
import math

import numpy as np
import torch

from paper_2605_18643_b200 import ep, zeda

DEVICE = "cuda:0"
QWEN = {"d": 2048, "He": 768, "E": 128, "Z": 64, "K": 8}
GLM = {"d": 2048, "He": 1536, "E": 64, "Z": 32, "K": 4}
EPS = 1e-6
TIE_MARGIN = 2e-3        # smallest gap between neighbours of a token's top K+1 logits
SMALL_STACK_TOKENS = 64  # up to here a stack's tokens are drawn so that no layer decides on a near-tie


def _case(name, use, T, shape, zero=0.5, zipf=0.0, shift=0.0, gate=zeda.GATE_TOPK_NORM, copy=False, layers=1):
    c = dict(use=use, T=T, **shape)
    c.update(zero=zero, zipf=zipf, shift=shift, gate=gate, copy=copy, layers=layers)
    if name is not None:
        c["name"] = name
    return c


def listed():
    static = dict(QWEN, Z=0)
    return [
        # one sequence being decoded: one token through consecutive layers, every layer's weights cold
        _case("decode_stack_t1", "stack", 1, QWEN, layers=4),
        # the decode batch of the benchmark: per-token zero share spread over 0..100 %
        _case("decode_t64", "forward", 64, QWEN, shift=2.5),
        # a mixed serving step: decoding sequences and the tail of a prompt
        _case("mixed_t193", "forward", 193, QWEN),
        # a prompt chunk of odd length, copy experts with the renormalised gate (Eq. 7, Appendix B)
        _case("chunk_t777_copy", "forward", 777, QWEN, zero=0.4, gate=zeda.GATE_RENORM_REAL, copy=True),
        # the zero-fraction sweep's batch, even load
        _case("batch_t2048", "forward", 2048, QWEN),
        # the benchmark's prefill batch: Zipf load
        _case("prefill_t8192", "forward", 8192, QWEN, zipf=1.1),
        # the static top-K layer (no zero experts) that the zero-expert layer is compared with
        _case("static_t8192", "forward", 8192, static, zero=0.0, zipf=1.1),
        # the second model shape, ragged batch
        _case("glm_t5003", "forward", 5003, GLM, zipf=1.1),
        # the layer-stack workload, four of its layers
        _case("stack_t4096", "stack", 4096, QWEN, layers=4),
        # activations that live in host memory
        _case("host_t8192", "host", 8192, QWEN, zipf=1.1),
        # the expert-parallel path of one rank
        _case("ep_t4096", "ep", 4096, QWEN, zipf=1.1),
        # routing statistics of a training batch
        _case("stats_t8192", "stats", 8192, QWEN),
    ]


def draw(rng):
    use = rng.choice(["forward"] * 6 + ["stack"] * 2 + ["host", "ep", "stats"])
    shape = dict(QWEN if rng.random() < 0.7 else GLM)
    lo, hi = {"forward": (1, 8192), "stack": (1, 4096), "host": (16, 8192), "ep": (16, 4096), "stats": (256, 8192)}[use]
    T = min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))
    zero = round(rng.uniform(0.3, 0.75), 2)
    if use == "forward" and rng.random() < 0.2:
        shape["Z"], zero = 0, 0.0
    zipf = 1.1 if use != "stack" and rng.random() < 0.4 else 0.0
    shift = 2.5 if use == "forward" and shape["Z"] and rng.random() < 0.3 else 0.0
    gate = rng.choice([zeda.GATE_TOPK_NORM, zeda.GATE_TOPK_NORM, zeda.GATE_SOFTMAX_RAW, zeda.GATE_RENORM_REAL])
    copy = bool(shape["Z"]) and use != "stack" and rng.random() < 0.2
    return _case(None, use, T, shape, zero, zipf, shift, gate, copy, rng.randint(2, 4) if use == "stack" else 1)


# ---------------------------------------------------------------------------------------- inputs

def _zero_bias(logits, E, K, share):
    """Offset on the zero experts' logits that puts `share` of the top-K slots on them (bisection)."""
    lo, hi = -40.0, 40.0
    trial = logits.clone()
    for _ in range(24):
        c = 0.5 * (lo + hi)
        trial[:, E:] = logits[:, E:] + c
        got = float((torch.topk(trial, K, dim=1).indices >= E).double().mean())
        lo, hi = (c, hi) if got < share else (lo, c)
    return 0.5 * (lo + hi)


def _gaps(logits, K):
    k = min(K + 1, logits.shape[1])
    top = torch.topk(logits, k, dim=1).values
    return (top[:, :-1] - top[:, 1:]).amin(dim=1) if k > 1 else torch.full((logits.shape[0],), math.inf, device=logits.device)


def _logits(x, layer):
    return x.double() @ layer["router_w"].double().t() + layer["bias"].double()


def _layer(case, g):
    """Weights of one layer, on the GPU: N(0, 0.02^2), the recipe of the benchmark."""
    d, He, E, Z, K = (case[k] for k in ("d", "He", "E", "Z", "K"))

    def normal(shape, std, dtype):
        return torch.empty(shape, dtype=dtype, device=DEVICE).normal_(0.0, std, generator=g)

    layer = {"w_gate_up": normal((E, 2 * He, d), 0.02, torch.bfloat16), "w_down": normal((E, d, He), 0.02, torch.bfloat16)}
    layer["router_w"] = normal((E + Z, d), 0.02, torch.float32)
    layer["bias"] = torch.zeros(E + Z, dtype=torch.float32, device=DEVICE)
    if case["shift"] and Z:
        u = normal((d,), 1.0, torch.float32)
        layer["router_w"][E:] += case["shift"] * u / u.norm()
    if case["zipf"]:
        p = torch.arange(1, E + 1, dtype=torch.float64, device=DEVICE).pow(-case["zipf"])
        order = torch.randperm(E, generator=g, device=DEVICE)
        layer["bias"][:E] = (p / p.sum())[order].log().float()
    if Z:
        proxy = normal((1024, d), 1.0, torch.bfloat16)
        layer["bias"][E:] += _zero_bias(_logits(proxy, layer), E, K, case["zero"])
    return layer


def _tokens(case, g, gaps):
    """x ~ N(0, 1); tokens whose smallest gap (gaps(x)) is below the margin are drawn again."""
    x = torch.empty((case["T"], case["d"]), dtype=torch.bfloat16, device=DEVICE).normal_(0.0, 1.0, generator=g)
    for _ in range(60):
        bad = torch.nonzero(gaps(x) < TIE_MARGIN).flatten()
        if not bad.numel():
            return x
        x[bad] = torch.empty((bad.numel(), case["d"]), dtype=torch.bfloat16, device=DEVICE).normal_(0.0, 1.0, generator=g)
    raise RuntimeError("could not reach the tie margin")


def _rmsnorm(r):
    rf = r.float()
    return (rf * torch.rsqrt(rf.pow(2).mean(dim=-1, keepdim=True) + EPS)).to(torch.bfloat16)


def _stack_gaps(case, layers, r):
    """Smallest gap per token over the layers of a stack, on a plain PyTorch pass of the (few) tokens."""
    E, K, He = case["E"], case["K"], case["He"]
    least = None
    for layer in layers:
        h = _rmsnorm(r)
        logits = _logits(h, layer)
        gap = _gaps(logits, K)
        least = gap if least is None else torch.minimum(least, gap)
        top = torch.topk(logits, K, dim=1)
        w = torch.softmax(logits, dim=1).gather(1, top.indices)
        real = top.indices < E
        if case["gate"] == zeda.GATE_TOPK_NORM:
            w = w / w.sum(dim=1, keepdim=True)
        elif case["gate"] == zeda.GATE_RENORM_REAL:
            w = w / (w * real).sum(dim=1, keepdim=True).clamp_min(1e-30)
        y = torch.zeros(r.shape, dtype=torch.float32, device=DEVICE)
        for k in range(K):
            e = top.indices[:, k].clamp(max=E - 1)
            gu = torch.bmm(layer["w_gate_up"][e], h.unsqueeze(2)).squeeze(2).float()
            mid = (torch.nn.functional.silu(gu[:, :He]) * gu[:, He:]).to(torch.bfloat16)
            o = torch.bmm(layer["w_down"][e], mid.unsqueeze(2)).squeeze(2).float()
            y += (w[:, k] * real[:, k]).float().unsqueeze(1) * o
        r = (r.float() + y.to(torch.bfloat16).float()).to(torch.bfloat16)
    return least


def prepare(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(1000003 * seed + 17)
    T, E, Z, K, use = case["T"], case["E"], case["Z"], case["K"], case["use"]
    layers = [_layer(case, g) for _ in range(case["layers"])]
    if use != "stack":
        x = _tokens(case, g, lambda x: _gaps(_logits(x, layers[0]), K))
    elif T <= SMALL_STACK_TOKENS:
        x = _tokens(case, g, lambda x: _stack_gaps(case, layers, x))
    else:  # a decision that flips on the last bits of one token's logits is lost in a batch's residual stream
        x = torch.empty((T, case["d"]), dtype=torch.bfloat16, device=DEVICE).normal_(0.0, 1.0, generator=g)
    kw = {"ep_size": 1, "ep_rank": 0, "max_recv_pairs": T * K} if use == "ep" else {}
    moes = [zeda.ZedaMoE(l["router_w"], l["bias"], l["w_gate_up"], l["w_down"], E, Z, K, T, gate_mode=case["gate"],
                         expert_kind=zeda.EXPERT_COPY if case["copy"] else zeda.EXPERT_ZERO, **kw) for l in layers]
    s = {"use": use, "moes": moes}
    if use == "stack":
        s.update(r0=x, r=torch.empty_like(x), h=[torch.empty_like(x), torch.empty_like(x)])
    elif use == "host":
        s.update(x=x.cpu().pin_memory(), y=torch.empty(x.shape, dtype=x.dtype).pin_memory())
    elif use == "ep":
        s.update(x=x, rank=ep.ExpertParallelMoE(moes[0], ep.LoopbackExchange()))
    else:
        s.update(x=x)
    return s


def run(s):
    m = s["moes"][0]
    if s["use"] == "forward":
        return m.forward(s["x"])
    if s["use"] == "stack":
        r, h = s["r"], s["h"]
        r.copy_(s["r0"])  # what an embedding lookup would write
        zeda.residual_rmsnorm(r, None, h[0], EPS)
        for i, layer in enumerate(s["moes"]):
            layer.forward_residual(h[i % 2], r, h[(i + 1) % 2], EPS)
        return r, h[len(s["moes"]) % 2]
    if s["use"] == "host":
        return m.forward_host(s["x"], s["y"])
    if s["use"] == "ep":
        return s["rank"].forward(s["x"])
    f, p_mean, sums = m.stats(s["x"])
    return f, p_mean, sums, m.token_zero_share(s["x"].shape[0])


# ---------------------------------------------------------------------------------------- work, tolerance

@functools.lru_cache(maxsize=None)
def _expected_load(E, Z, K, d, zero, zipf):
    """Chance that a token selects each normal expert, from a model of the router: logits are normal with the
    router rows' spread, the experts carry their prior, the zero experts the offset that gives their share."""
    rng = np.random.default_rng(0)
    logits = rng.standard_normal((2048, E + Z)) * 0.02 * math.sqrt(d)
    if zipf:
        p = np.arange(1, E + 1, dtype=np.float64) ** -zipf
        logits[:, :E] += np.log(p / p.sum())
    if Z:
        lo, hi = -40.0, 40.0
        for _ in range(24):
            c = 0.5 * (lo + hi)
            trial = logits.copy()
            trial[:, E:] += c
            got = (np.argpartition(-trial, K - 1, axis=1)[:, :K] >= E).mean()
            lo, hi = (c, hi) if got < zero else (lo, c)
        logits[:, E:] += 0.5 * (lo + hi)
    top = np.argpartition(-logits, K - 1, axis=1)[:, :K]
    return tuple(np.bincount(top.ravel(), minlength=E + Z)[:E] / 2048.0)


def work(case):
    """Active experts' weights, router rows and activations once; the pairs' three products and the router's."""
    T, d, He, E, Z, K, L = (case[k] for k in ("T", "d", "He", "E", "Z", "K", "layers"))
    n = E + Z
    router_bytes, router_flops = 4.0 * n * d, 2.0 * T * n * d
    if case["use"] == "stats":
        return {"bytes": 2.0 * T * d + router_bytes + 8.0 * n + 4.0 * T, "flops": router_flops}
    q = np.array(_expected_load(E, Z, K, d, case["zero"], case["zipf"]))
    pairs, active = T * float(q.sum()), float((1.0 - (1.0 - q) ** T).sum())
    layer_bytes = active * 6.0 * d * He + router_bytes
    act = 2.0 * T * d
    # a stack reads the residual stream once and returns it with the next input; other uses read x, write y
    return {"bytes": L * layer_bytes + act * (3 if case["use"] == "stack" else 2), "flops": L * (6.0 * pairs * d * He + router_flops)}


def tolerance(case):
    """About four times the distance of the path from the same case in 64 bits: bf16 intermediate results and outputs
    (2.9e-3 in the 2-norm, 1.7e-2 at most; a small stack's residual 1.3e-3 and 8e-3, a large one's 5.7e-3 and
    0.15, near-ties that fall the other way included); fp32 sums for the statistics (1.7e-7, 5e-7; their order
    is free, so a little more)."""
    if case["use"] == "stats":
        return {"rel": 2e-6, "max": 1e-5}
    if case["use"] == "stack":
        return {"rel": 6e-3, "max": 0.04} if case["T"] <= SMALL_STACK_TOKENS else {"rel": 2e-2, "max": 0.5}
    return {"rel": 1e-2, "max": 0.06}
