"""The layer calls whose speed is followed: what a program that uses the BigMac MoE layer has it do.

Every case is one call (or one training step) of `binding.Layer` on one GPU.  The widths are those of the configurations
in `workloads.py`: small (d 1024, 32 experts, top-4), medium and decode (d 2048, 64 experts, top-8), large (d 4096, 128
experts, top-8), BF16 with GELU, and the fp32 ReLU configuration (tiny).  Inputs follow the same recipe as there: x and
dy are N(0, 1), weights N(0, 1/fan_in), the medium training workload has the Zipf gate bias that gives its experts very
different loads.  Tokens whose k + 1 largest gate logits lie closer than MARGIN are drawn again, as everywhere in this
repository: the routing of a batch is then the same whatever the order in which a logit's products are added.
"""
import math

import torch

from paper_2502_16927_b200 import binding
from paper_2502_16927_b200.workloads import ACT_GELU_ERF, ACT_RELU, WORKLOADS, zipf_log_popularity

MARGIN = 1e-3

SMALL, MEDIUM, LARGE, TINY = (dict((n, getattr(WORKLOADS[w], n)) for n in ("d", "r", "h", "E", "k"))
                              for w in ("small", "medium", "large", "tiny"))


def _case(path, widths, T, dtype="bf16", zipf=False, accumulate=False, capacity=0.0, aux=0.0):
    return dict(path=path, T=T, dtype=dtype, zipf=zipf, accumulate=accumulate, capacity=capacity, aux=aux, **widths)


def _named(name, *args, **kw):
    return dict(_case(*args, **kw), name=name)


def listed():
    return [
        # Generation: one new token per running sequence.  A single sequence, a handful, a busy server, a full one.
        _named("decode 1", "forward", MEDIUM, 1),
        _named("decode 8", "forward", MEDIUM, 8),
        _named("decode 64", "forward", MEDIUM, 64),
        _named("decode 512", "forward", MEDIUM, 512),
        # Reading prompts: a batch of prompts packed without padding has whatever length it has; a big batch, large widths.
        _named("prefill 3001", "forward", MEDIUM, 3001),
        _named("prefill large 16384", "forward", LARGE, 16384),
        # Routing alone: the tables for a program that moves the tokens itself.
        _named("route 16384", "route", MEDIUM, 16384, zipf=True),
        # Training, forward and backward: the fp32 configuration (gradient checks, small studies) ...
        _named("train fp32 256", "train", TINY, 256, dtype="fp32"),
        # ... the three BF16 sizes: two sequences of 2048, eight with a skewed gate, sixteen ...
        _named("train small 4096", "train", SMALL, 4096),
        _named("train medium 16384", "train", MEDIUM, 16384, zipf=True),
        _named("train large 32768", "train", LARGE, 32768),
        # ... and a micro-batch of unpadded documents whose gradients are added to those of the ones before, with the
        # pre-training recipe's capacity factor and load-balancing loss.
        _named("train recipe 2999", "train", MEDIUM, 2999, accumulate=True, capacity=1.2, aux=0.001),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "prefill", "route", "fp32", "train", "train", "train", "recipe"])
    if kind == "decode":
        return _case("forward", rng.choice([SMALL, MEDIUM, MEDIUM, LARGE]), _log_uniform(rng, 1, 600))
    if kind == "prefill":
        return _case("forward", rng.choice([SMALL, MEDIUM, LARGE]), _log_uniform(rng, 600, 20000), zipf=rng.random() < 0.3)
    if kind == "route":
        return _case("route", rng.choice([SMALL, MEDIUM, LARGE]), _log_uniform(rng, 64, 32768), zipf=rng.random() < 0.5)
    if kind == "fp32":
        return _case("train", TINY, _log_uniform(rng, 32, 2048), dtype="fp32")
    widths = rng.choice([SMALL, MEDIUM, LARGE])
    if kind == "recipe":
        return _case("train", widths, _log_uniform(rng, 512, 12000), zipf=rng.random() < 0.3, accumulate=True, capacity=1.2, aux=0.001)
    return _case("train", widths, _log_uniform(rng, 512, 30000), zipf=rng.random() < 0.3, accumulate=rng.random() < 0.3)


def _tokens_with_margin(normal, T, d, w_gate, b_gate, k):
    x = normal(T, d)
    if w_gate.shape[0] < 2:
        return x
    gate = w_gate.float().t()
    rows = torch.arange(T, device=x.device)
    for _ in range(64):
        logits = x[rows].float() @ gate
        if b_gate is not None:
            logits += b_gate
        top = torch.topk(logits, min(k + 1, w_gate.shape[0]), dim=1).values
        rows = rows[(top[:, :-1] - top[:, 1:]).amin(dim=1) < MARGIN]
        if rows.numel() == 0:
            return x
        x[rows] = normal(rows.numel(), d)
    raise RuntimeError("no tokens with the wanted margin between gate logits")


def prepare(case, seed):
    """The handle, the weights and the batch; for a training step also the upstream gradient and the gradient buffers."""
    T, d, r, h, E, k = (case[n] for n in ("T", "d", "r", "h", "E", "k"))
    bf16 = case["dtype"] == "bf16"
    tdtype = torch.bfloat16 if bf16 else torch.float32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape, std=1.0):
        t = torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)
        return (t if std == 1.0 else t.mul_(std)).to(tdtype)

    W = {"w_gate": normal(E, d, std=d ** -0.5), "w_down": normal(r, d, std=d ** -0.5), "w1": normal(E, h, r, std=r ** -0.5),
         "w2": normal(E, r, h, std=h ** -0.5), "w_up": normal(d, r, std=r ** -0.5)}
    if case["zipf"]:
        W["b_gate"] = torch.from_numpy(zipf_log_popularity(E)).cuda()
    x = _tokens_with_margin(normal, T, d, W["w_gate"], W.get("b_gate"), k)
    layer = binding.Layer(d, r, h, E, k, T, binding.BIGMAC_BF16 if bf16 else binding.BIGMAC_F32, ACT_GELU_ERF if bf16 else ACT_RELU,
                          capacity_factor=case["capacity"], aux_loss_coef=case["aux"])
    state = {"case": case, "layer": layer, "W": W, "x": x}
    if case["path"] == "train":
        state["dy"] = normal(T, d)
        # an accumulating step finds the gradients of the micro-batches before it
        fill = normal if case["accumulate"] else lambda *shape: torch.empty(*shape, device="cuda", dtype=tdtype)
        state["G"] = {"d" + n: fill(*W[n].shape) for n in ("w_gate", "w_down", "w1", "w2", "w_up")}
        if case["zipf"]:
            state["G"]["db_gate"] = torch.zeros(E, device="cuda", dtype=torch.float32)
    return state


def run(state):
    case, layer, W, x = state["case"], state["layer"], state["W"], state["x"]
    if case["path"] == "route":
        R = layer.route(x, W)
        return {n: R[n] for n in ("topk_idx", "topk_w", "counts", "offsets", "row_of_slot", "slot_of_row")}
    if case["path"] == "forward":
        return layer.forward(x, W)
    out = {}
    if case["aux"] > 0:                                # a training program logs the loss and the experts' loads
        out["y"], R = layer.forward(x, W, training=True, want_routing=True)
        out["aux_loss"], out["counts"] = R["aux_loss"], R["counts"]
    else:
        out["y"] = layer.forward(x, W, training=True)
    out["dx"] = layer.backward(x, state["dy"], W, state["G"], accumulate=case["accumulate"])
    out.update(state["G"])
    return out


def work(case):
    """Every input once, every output once; of the experts' weights those of the experts that a batch of this size chooses
    (expected number for even loads).  A backward pass has twice the forward's multiply-adds."""
    T, d, r, h, E, k = (case[n] for n in ("T", "d", "r", "h", "E", "k"))
    es = 2 if case["dtype"] == "bf16" else 4
    if case["path"] == "route":
        return {"bytes": T * d * es + E * d * es + 16.0 * T * k + 8.0 * E, "flops": 2.0 * T * d * E}
    experts = E * (1.0 - (1.0 - k / E) ** T)
    shared = (2.0 * d * r + d * E) * es
    forward = 2.0 * T * d * (E + 2 * r) + 4.0 * T * k * r * h
    if case["path"] == "forward":
        return {"bytes": 2.0 * T * d * es + shared + experts * 2 * r * h * es, "flops": forward}
    grads = (2.0 * d * r + d * E + 2.0 * E * r * h) * es * (2 if case["accumulate"] else 1)
    return {"bytes": 4.0 * T * d * es + shared + experts * 2 * r * h * es + grads, "flops": 3.0 * forward}


def tolerance(case):
    if case["path"] == "route":                        # tables are whole numbers with one right value; gate values are fp32
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.0}
    if case["dtype"] == "fp32":                        # max: a ReLU unit within rounding of zero may fall on either side
        return {"rel": 1e-5, "max": 0.5}
    # bf16 between the stages; the bias gradient of a skewed gate is a difference of large sums of both signs
    return {"rel": 2e-2 if case["zipf"] and case["path"] == "train" else 1e-2, "max": 0.5, "differ": 0.0}
