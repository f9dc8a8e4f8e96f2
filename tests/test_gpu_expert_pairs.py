"""Both contractions of an expert in one kernel.  On CTA pairs: one chunk of the hidden width or an odd number of them, experts
without rows, with one row, with a half-used pair of row tiles, more items than SM pairs, the tables of many experts; forward,
backward and inference.  The sums are the separate contractions' in the same order, so every result has their bits.
On the fp32 path: widths that are no multiple of a tile or of a warp, two chunks, blocks of 16 and of 32 rows, of padding rows alone."""
import numpy as np
import pytest

from paper_2502_16927_b200 import workloads as wl
from helpers import empty_grads, make_layer, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,h,E,k,T,skew,act", [
    (256, 128, 5, 2, 300, 3.0, wl.ACT_GELU_ERF),        # one chunk; loads from a few rows to several pairs
    (128, 384, 4, 4, 129, 0.0, wl.ACT_GELU_ERF),        # three chunks; every expert has 129 rows
    (256, 640, 96, 2, 40, 0.0, wl.ACT_GELU_ERF),        # experts without rows, with one
    (128, 256, 3, 1, 20000, 1.0, wl.ACT_GELU_ERF),      # more items than SM pairs
    (256, 256, 300, 4, 3000, 2.0, wl.ACT_RELU),         # the tables take the place of a ring stage
    (256, 256, 200, 2, 777, 1.0, wl.ACT_GELU_TANH),
    (128, 1024, 1, 1, 257, 0.0, wl.ACT_IDENTITY),
])
def test_equals_the_separate_contractions(r, h, E, k, T, skew, act):
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("pairs", T=T, d=128, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_BF16, act=act, seed=900 + T)
    inp = wl.make_inputs(w)
    inp["b_gate"] = (skew * np.linspace(1.0, -1.0, w.E) ** 3).astype(np.float32)
    dev = to_device(w, inp)
    out = {}
    for mode in (0, 2):
        try:
            binding.bigmac_debug_set("ffn", mode)           # read at creation
            layer = make_layer(w)
            binding.bigmac_debug_set("fused_mlp", 0)
            infer = layer.forward(dev["x"], dev)
            y = layer.forward(dev["x"], dev, training=True)
            grads = empty_grads(w, dev)
            dx = layer.backward(dev["x"], dev["dy"], dev, grads)
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        assert layer.status() == 0
        out[mode] = dict(grads, infer=infer, y=y, dx=dx)
        layer.close()
    for name, ref in out[0].items():
        assert torch.equal(ref, out[2][name]), name
        assert torch.isfinite(ref.float()).all(), name


@pytest.mark.parametrize("variant,r,h,E,k,T", [("capacity", 256, 256, 6, 3, 500), ("capacity", 128, 128, 8, 2, 900), ("cdac", 128, 256, 5, 2, 300),
                                               ("cdac", 256, 128, 3, 1, 700), ("gate_low", 256, 384, 6, 2, 333), ("accumulate", 128, 256, 7, 3, 400),
                                               ("accumulate", 256, 128, 4, 2, 129), ("nan", 256, 256, 9, 2, 300), ("nan", 128, 384, 5, 1, 650)])
def test_variants_equal_the_separate_contractions(variant, r, h, E, k, T):
    """A capacity limit, the layer without projections, the gate on x', gradients added to others; tokens of NaN, whose rows lie beside the
    unused half of another expert's last pair and leave no trace there."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("variant", T=T, d=r if variant == "cdac" else 192, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=50 + T,
                    cdac=variant == "cdac", gate_low=variant == "gate_low")
    inp = wl.make_inputs(w)
    inp["b_gate"] = np.linspace(1.0, -1.0, w.E).astype(np.float32)
    if variant == "nan":
        inp["x"][[0, T // 2, T - 1]] = np.nan
    dev = to_device(w, inp)
    out = {}
    for mode in (0, 2):
        try:
            binding.bigmac_debug_set("ffn", mode)
            layer = make_layer(w, capacity_factor=0.6 if variant == "capacity" else 0.0)
            binding.bigmac_debug_set("fused_mlp", 0)
            infer = layer.forward(dev["x"], dev)
            y = layer.forward(dev["x"], dev, training=True)
            grads = empty_grads(w, dev, fill=0.25)
            dx = layer.backward(dev["x"], dev["dy"], dev, grads, accumulate=variant == "accumulate")
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        assert layer.status() == 0
        out[mode] = dict(grads, infer=infer, y=y, dx=dx)
        layer.close()
    for name, ref in out[0].items():
        got = out[2][name]
        assert torch.equal(ref.isnan(), got.isnan()) and torch.equal(ref.nan_to_num(), got.nan_to_num()), name
    rest = torch.ones(T, dtype=torch.bool, device="cuda")
    if variant == "nan":
        rest[[0, T // 2, T - 1]] = False
        assert out[2]["y"][~rest].isnan().all()
    for name in ("infer", "y", "dx"):
        assert torch.isfinite(out[2][name][rest].float()).all(), name


@pytest.mark.parametrize("d,r,h,E,k,T,capacity", [(128, 32, 128, 8, 2, 33, 0.0), (64, 4, 4, 3, 1, 7, 0.0), (64, 12, 132, 5, 2, 130, 0.0),
                                                 (128, 32, 256, 6, 3, 200, 0.7), (64, 20, 60, 4, 2, 5000, 0.0), (64, 28, 252, 40, 2, 300, 0.0)])
def test_fp32_in_one_launch(d, r, h, E, k, T, capacity):
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("narrow", T=T, d=d, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_F32, act=wl.ACT_GELU_ERF, seed=40 + T)
    dev = to_device(w, wl.make_inputs(w))
    out = {}
    for mode in (0, 1):
        try:
            binding.bigmac_debug_set("ffn", mode)
            layer = make_layer(w, capacity_factor=capacity)
            infer = layer.forward(dev["x"], dev)
            y = layer.forward(dev["x"], dev, training=True)
            grads = empty_grads(w, dev)
            dx = layer.backward(dev["x"], dev["dy"], dev, grads)
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        out[mode] = dict(grads, infer=infer, y=y, dx=dx)
        layer.close()
    # The same products in another order: sums of at most 256 terms, four in a row, of unit roundoff 6e-8, i.e. 16 x 6e-8 x 4 for random
    # signs; the weight gradients then sum these errors like their terms.  The gate's gradients are differences of dp: ten times that
    # (and exactly zero with one expert a token).
    for name, ref in out[0].items():
        err = (ref.double() - out[1][name].double()).norm()
        assert err <= (4e-5 if "gate" in name else 4e-6) * ref.double().norm(), (name, float(err), float(ref.double().norm()))


def test_inference_under_a_capacity_limit_keeps_u_in_fp32():
    """1250 tokens of 16 experts top-8, eight of them favoured: the capacity limit leaves 48 row tiles, for which the experts' kernel of
    few rows cuts the hidden width and keeps u in fp32.  Such a call does not go to the pairs, which would round u to bf16."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("limit", T=1250, d=128, r=256, h=1024, E=16, k=8, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=77)
    inp = wl.make_inputs(w)
    inp["b_gate"] = np.where(np.arange(w.E) < 8, 30.0, 0.0).astype(np.float32)
    dev = to_device(w, inp)
    out = {}
    for mode in (0, 1):
        try:
            binding.bigmac_debug_set("ffn", mode)
            layer = make_layer(w, capacity_factor=1.2)
            out[mode] = layer.forward(dev["x"], dev)
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        assert layer.status() == 0
        layer.close()
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("dtype,r,h,T", [(wl.DTYPE_BF16, 256, 256, 300), (wl.DTYPE_F32, 32, 128, 90)])
@pytest.mark.parametrize("before,after", [(2, 0), (0, 2)])
def test_switch_between_a_forward_and_its_backward(dtype, r, h, T, before, after):
    """The kernels of the two directions agree on where sigma' lies: what the switch says when the handle is created holds for both."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("switch", T=T, d=128, r=r, h=h, E=5, k=2, dtype=dtype, act=wl.ACT_GELU_ERF, seed=5)
    dev = to_device(w, wl.make_inputs(w))
    out = []
    for later in (before, after):
        try:
            binding.bigmac_debug_set("ffn", before)
            layer = make_layer(w)
            layer.forward(dev["x"], dev, training=True)
            binding.bigmac_debug_set("ffn", later)
            grads = empty_grads(w, dev)
            dx = layer.backward(dev["x"], dev["dy"], dev, grads)
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        out.append(dict(grads, dx=dx))
        layer.close()
    for name, ref in out[0].items():
        assert torch.equal(ref, out[1][name]), name


def _step_in_64_bits(w, dev, idx):
    """y and the gradients of a layer without biases or limit, for the given routing, by torch in 64 bits."""
    import torch

    P = {n: dev[n].double().requires_grad_() for n in ("w_gate", "w_down", "w1", "w2", "w_up")}
    x = dev["x"].double().requires_grad_()
    weight = torch.softmax((x @ P["w_gate"].t()).gather(1, idx), 1)
    low = x @ P["w_down"].t()
    mixed = torch.zeros_like(low)
    for e in range(w.E):
        t, j = (idx == e).nonzero(as_tuple=True)
        u = torch.nn.functional.gelu(low[t] @ P["w1"][e].t()) @ P["w2"][e].t()
        mixed = mixed.index_add(0, t, weight[t, j, None] * u)
    y = mixed @ P["w_up"].t()
    y.backward(dev["dy"].double())
    return dict({"d" + n: p.grad for n, p in P.items()}, y=y.detach(), dx=x.grad)


@pytest.mark.parametrize("d,r,h,E,k,T", [(128, 32, 128, 8, 2, 2048), (128, 32, 256, 16, 4, 700), (256, 16, 252, 12, 3, 700), (64, 32, 128, 4, 2, 6000)])
def test_fp32_in_one_launch_is_as_exact(d, r, h, E, k, T):
    """Distance from 64 bits: no larger than that of the separate contractions, whose sums are of short parts.  (Distances of these
    sizes repeat within 4 % from seed to seed; one running sum of h terms was 1.15 to 1.6 times as far off.)"""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("exact", T=T, d=d, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_F32, act=wl.ACT_GELU_ERF, seed=12 + T)
    dev = to_device(w, wl.make_inputs(w))
    far = {}
    for mode in (0, 1):
        try:
            binding.bigmac_debug_set("ffn", mode)
            layer = make_layer(w)
            y, R = layer.forward(dev["x"], dev, training=True, want_routing=True)
            grads = empty_grads(w, dev)
            dx = layer.backward(dev["x"], dev["dy"], dev, grads)
            torch.cuda.synchronize()
        finally:
            binding.bigmac_debug_set("defaults")
        ref = _step_in_64_bits(w, dev, R["topk_idx"].view(T, k).long())
        far[mode] = {n: float((g.double() - ref[n]).norm() / ref[n].norm()) for n, g in dict(grads, y=y, dx=dx).items() if n in ref}
        layer.close()
    for name, before in far[0].items():
        assert far[1][name] <= 1.08 * before, (name, far[1][name], before)
