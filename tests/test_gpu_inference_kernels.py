"""Kernels of the inference forward at the sizes where their tiling can go wrong: the experts in one kernel (token counts
around its 16-token groups, 64- and 128-token tiles, hidden widths that end inside a 128-wide chunk, one to eight slices
of the hidden width) and the two routing launches (one to many blocks, expert counts around the lanes' loads)."""
import numpy as np
import pytest

import oracle
from oracle import margin
from paper_2502_16927_b200 import workloads as wl
from helpers import empty_grads, make_layer, to_device, to_numpy

pytestmark = pytest.mark.gpu


def _inputs(w, skew):
    inp = wl.make_inputs(w)
    inp["b_gate"] = (skew * np.linspace(1.0, -1.0, w.E) ** 3).astype(np.float32)
    margin.enforce_margin(w, inp, 1e-3)
    return inp


def _launches(layer, start=False):
    """Counts the layer's launches from `start` on."""
    from paper_2502_16927_b200 import binding

    if start:
        return binding.bigmac_profile_enable(layer.handle, True)
    return binding.bigmac_profile_read(layer.handle)["launches"]


def _check_tables(R, rt):
    for name in ("topk_idx", "counts", "counts_chosen", "offsets", "row_of_slot", "slot_of_row"):
        np.testing.assert_array_equal(to_numpy(R[name]), getattr(rt, name).reshape(-1), err_msg=name)
    # softmax of fp32 logits (rounding about 1e-6 of values of order one)
    np.testing.assert_allclose(to_numpy(R["topk_w"]), rt.topk_p.reshape(-1), rtol=0, atol=2e-5)


@pytest.mark.parametrize("r,h", [(64, 64), (128, 192), (192, 512), (256, 1024), (320, 256), (512, 384)])
@pytest.mark.parametrize("T,skew", [(17, 0.0), (40, 4.0), (129, 0.0), (333, 2.0)])
def test_experts_in_one_kernel(r, h, T, skew):
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("mlp", T=T, d=128, r=r, h=h, E=12, k=3, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=500 + T)
    inp = _inputs(w, skew)
    dev = to_device(w, inp)
    layer = make_layer(w)
    try:
        binding.bigmac_debug_set("fused_mlp", 2)
        y, R = layer.forward(dev["x"], dev, want_routing=True)
        again = layer.forward(dev["x"], dev)
        torch.cuda.synchronize()
    finally:
        binding.bigmac_debug_set("defaults")
    assert layer.status() == 0
    rt = oracle.route(inp, w.k)
    _check_tables(R, rt)
    ref = oracle.forward_tokens(inp, rt, w.act)["y"]
    # four bf16 stores (x', a, y', y; u too with one slice) of unit roundoff 2^-8 each, i.e. about 0.17 % of the rms per store
    err = np.linalg.norm(to_numpy(y) - ref) / np.linalg.norm(ref)
    assert err <= 8e-3, err
    assert torch.equal(y, again)
    layer.close()


@pytest.mark.parametrize("r,h,E", [(128, 512, 64), (64, 256, 320), (320, 256, 40)])
def test_experts_in_one_kernel_many_units(r, h, E):
    """More tiles than SMs, and the tables of many experts in shared memory; every token against the separate contractions."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("mlp", T=2601, d=128, r=r, h=h, E=E, k=8, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=77)
    dev = to_device(w, _inputs(w, 1.0))
    out = {}
    for mode in (0, 2):
        layer = make_layer(w)
        try:
            binding.bigmac_debug_set("fused_mlp", mode)
            out[mode] = to_numpy(layer.forward(dev["x"], dev))
        finally:
            binding.bigmac_debug_set("defaults")
        assert layer.status() == 0
        layer.close()
    # both sides keep a and y in bf16, the separate contractions u as well: sqrt(5) stores of 0.17 % of the rms each
    err = np.linalg.norm(out[2] - out[0], axis=1) / np.linalg.norm(out[0], axis=1)
    assert err.max() <= 2e-2 and np.sqrt((err ** 2).mean()) <= 6e-3, (err.max(), np.sqrt((err ** 2).mean()))


@pytest.mark.parametrize("E,k", [(4, 1), (8, 8), (36, 3), (64, 8), (100, 5), (256, 8)])
@pytest.mark.parametrize("T", [1, 4, 31, 33, 128, 4737, 20003])
def test_routing_in_two_launches(E, k, T):
    """With a load-balancing loss every size goes through two launches (the top-k with the blocks' counts, the placement); without one, up to
    512 tokens of at most 128 experts go through one."""
    import torch

    w = wl.Workload("route", T=T, d=32, r=8, h=8, E=E, k=k, dtype=wl.DTYPE_F32, act=wl.ACT_RELU, seed=33)
    inp = _inputs(w, 1.0)
    dev = to_device(w, inp)
    for f in (0.0, 0.6):
        rt = oracle.route(inp, w.k, capacity_factor=f)
        for aux in (0.0, 0.01):
            layer = make_layer(w, capacity_factor=f, aux_loss_coef=aux)
            _launches(layer, True)
            R = layer.route(dev["x"], dev)
            torch.cuda.synchronize()
            # the logits' launch, then one or two
            assert _launches(layer) == (2 if aux == 0 and T <= 512 and E <= 128 else 3)
            assert layer.status() == 0
            _check_tables(R, rt)
            layer.close()


@pytest.mark.parametrize("E,k,T", [(4, 1, 1), (64, 8, 5), (128, 8, 127), (132, 3, 129), (256, 8, 300), (36, 3, 512), (64, 8, 513), (128, 8, 1500), (32, 4, 3000)])
def test_routing_call_with_logits_in_parts(E, k, T):
    """bf16, d = 1088 (17 slices: parts of unequal length): the routing call adds the parts of its logits in the top-k; up to 512 tokens
    and 128 experts in one launch.  The call without scratch of its own returns the same bits."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("route", T=T, d=1088, r=64, h=64, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_RELU, seed=36)
    inp = _inputs(w, 1.0)
    dev = to_device(w, inp)
    for f in (0.0, 0.6):
        layer = make_layer(w, capacity_factor=f)
        R, S = layer.route(dev["x"], dev), layer.empty_routing(T)
        binding.bigmac_route_static(layer.handle, dev["x"], T, dev, S)
        torch.cuda.synchronize()
        assert layer.status() == 0
        _check_tables(R, oracle.route(inp, w.k, capacity_factor=f))
        assert all(torch.equal(R[name], S[name]) for name in ("topk_idx", "topk_w", "counts", "offsets", "row_of_slot", "slot_of_row"))
        layer.close()


@pytest.mark.parametrize("E,k", [(8, 8), (32, 1), (36, 3), (64, 8), (128, 8)])
@pytest.mark.parametrize("T", [1, 7, 33, 259, 511, 512])
def test_routing_in_one_launch(E, k, T):
    """A forward of up to 512 tokens routes in one launch (clusters that share the tokens): rows from a matrix (r 8, fp32) and from
    partial results (bf16, contraction of d = 1024 in parts; a training forward also wants the padding rows as zeros, which its
    weight gradients contract over), with and without a capacity limit."""
    import torch
    from paper_2502_16927_b200 import binding

    for dtype, d, r, h, training in ((wl.DTYPE_F32, 32, 8, 8, True), (wl.DTYPE_BF16, 1024, 128, 64, False), (wl.DTYPE_BF16, 1024, 128, 64, True)):
        w = wl.Workload("route", T=T, d=d, r=r, h=h, E=E, k=k, dtype=dtype, act=wl.ACT_RELU, seed=35)
        inp = _inputs(w, 1.0)
        dev = to_device(w, inp)
        for f in (0.0, 0.6):
            layer = make_layer(w, capacity_factor=f, flags=0)
            if training:                                             # what lies in the workspaces must not reach a gradient
                layer._workspaces(T, True)
                layer._scratch.fill_(255)
                layer._saved.fill_(255)
            y, R = layer.forward(dev["x"], dev, want_routing=True, training=training)
            if training:
                G = empty_grads(w, "cuda", fill=float("nan"))
                dx = layer.backward(dev["x"], dev["dy"], dev, G)
                assert all(bool(torch.isfinite(v).all()) for v in (*G.values(), dx))
            torch.cuda.synchronize()
            assert layer.status() == 0
            rt = oracle.route(inp, w.k, capacity_factor=f)
            _check_tables(R, rt)
            ref = oracle.forward_tokens(inp, rt, w.act)["y"]
            tol = 1e-4 if dtype == wl.DTYPE_F32 else 8e-3          # bf16: four or five stores of 0.17 % of the rms each
            err = np.linalg.norm(to_numpy(y) - ref) / max(np.linalg.norm(ref), 1e-30)
            assert err <= tol, (dtype, f, err)
            layer.close()


@pytest.mark.parametrize("E,k", [(4, 4), (36, 8), (64, 8), (128, 8), (256, 8)])
def test_equal_and_nonfinite_logits(E, k):
    """Logits that are nothing but the gate bias: a handful of values that many experts share (in one lane's quad, across its
    quads, across lanes), both zeros, infinities and NaN: order by value, then by id, NaN as -inf."""
    import torch

    T = 70
    w = wl.Workload("ties", T=T, d=32, r=8, h=8, E=E, k=k, dtype=wl.DTYPE_F32, act=wl.ACT_RELU, seed=3)
    inp = wl.make_inputs(w)
    inp["x"] = np.zeros_like(inp["x"])
    rng = np.random.default_rng(E)
    for values in ([1.0], [0.0, -0.0, -1.0], [2.0, 2.0, -3.0], [-np.inf, np.nan], [np.inf, 1.0, np.nan, -np.inf]):
        bias = rng.choice(np.array(values, dtype=np.float32), E)
        inp["b_gate"] = bias
        layer = make_layer(w)
        R = layer.route(to_device(w, inp)["x"], to_device(w, inp))
        torch.cuda.synchronize()
        assert layer.status() == 0
        key = np.where(np.isnan(bias), -np.inf, bias)
        want = np.array(sorted(range(E), key=lambda e: (-key[e], e))[:k])
        np.testing.assert_array_equal(to_numpy(R["topk_idx"]).reshape(T, k), np.tile(want, (T, 1)))
        layer.close()


@pytest.mark.parametrize("E,k", [(4, 4), (33, 8), (64, 8), (100, 40), (256, 16)])
@pytest.mark.parametrize("T", [1, 3, 16])
def test_small_batch_orders_equal_and_nonfinite_logits(E, k, T):
    """The same order in the one-kernel forward of a few tokens, every token with a bias pattern of its own column order."""
    import torch

    w = wl.Workload("ties", T=T, d=64, r=64, h=64, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=3)
    inp = wl.make_inputs(w)
    inp["x"] = np.zeros_like(inp["x"])
    rng = np.random.default_rng(E)
    layer = make_layer(w)
    for values in ([1.0], [0.0, -0.0, -1.0], [2.0, 2.0, -3.0], [-np.inf, np.nan], [np.inf, 1.0, np.nan, -np.inf], None):
        bias = (rng.standard_normal(E) if values is None else rng.choice(np.array(values), E)).astype(np.float32)
        inp["b_gate"] = bias
        dev = to_device(w, inp)
        R = layer.forward(dev["x"], dev, want_routing=True)[1]
        torch.cuda.synchronize()
        assert layer.status() == 0
        key = np.where(np.isnan(bias), -np.inf, bias)
        want = np.array(sorted(range(E), key=lambda e: (-key[e], e))[:k])
        np.testing.assert_array_equal(to_numpy(R["topk_idx"]).reshape(T, k), np.tile(want, (T, 1)))
    layer.close()


def _small_batch(w, one_kernel):
    """A forward of a few tokens against the oracle, in one kernel or not."""
    import torch
    from paper_2502_16927_b200 import binding

    inp = _inputs(w, 0.0)
    dev = to_device(w, inp)
    layer = make_layer(w)
    binding.bigmac_profile_enable(layer.handle, True)
    y = layer.forward(dev["x"], dev)
    launches = binding.bigmac_profile_read(layer.handle)["launches"]
    assert (launches == 1) == one_kernel, launches
    binding.bigmac_profile_enable(layer.handle, False)
    again = layer.forward(dev["x"], dev)
    torch.cuda.synchronize()
    assert layer.status() == 0 and torch.equal(y, again)
    ref = oracle.forward_tokens(inp, oracle.route(inp, w.k), w.act)["y"]
    err = np.linalg.norm(to_numpy(y) - ref) / np.linalg.norm(ref)
    # bf16 stores of 0.17 % of the rms each: y alone in the one kernel, x', a, u, y' and y in the launch chain
    assert err <= (4e-3 if one_kernel else 8e-3), err
    layer.close()


@pytest.mark.parametrize("r,h,E,k,T", [
    (64, 8192, 8, 4, 1), (64, 8192, 8, 5, 3), (64, 16384, 4, 3, 2), (64, 32768, 4, 1, 2),    # one pass over the slots, two, of unequal length
    (64, 64, 64, 64, 9),                                                                      # 576 slots
    (256, 9408, 8, 4, 4)])                                                                    # the last batch in front of the launch chain
def test_small_batch_with_many_hidden_units(r, h, E, k, T):
    _small_batch(wl.Workload("hidden", T=T, d=128, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=900 + T), True)


@pytest.mark.parametrize("r,h,E,k,T", [(256, 9408, 8, 4, 5), (64, 32832, 4, 1, 1)])
def test_small_batch_left_to_the_launch_chain(r, h, E, k, T):
    _small_batch(wl.Workload("chain", T=T, d=128, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=900 + T), False)


@pytest.mark.parametrize("d,r,h,E,k,T", [
    (8192, 512, 64, 8, 2, 2), (8192, 512, 64, 8, 2, 4),          # W'_up rows of a block: 57 KB of shared memory ...
    (8192, 1024, 64, 8, 2, 4),                                    # ... and more than it takes
    (128, 64, 1024, 16, 8, 2), (128, 64, 1088, 16, 8, 2)])       # two tokens on either side of the change of variant
def test_small_batch_variants(d, r, h, E, k, T):
    _small_batch(wl.Workload("var", T=T, d=d, r=r, h=h, E=E, k=k, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=950 + T), True)


def test_first_call_on_another_stream_while_the_default_stream_is_busy():
    """Handles made behind queued work of the default stream, more of them than the pool has places, first used on a stream that
    is not ordered with it: nothing that making them left behind may come between (or after) their launches."""
    import torch

    w = wl.Workload("busy", T=3, d=128, r=64, h=128, E=8, k=2, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=41)
    inp = _inputs(w, 0.0)
    dev = to_device(w, inp)
    layer = make_layer(w)
    want = layer.forward(dev["x"], dev)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    torch.cuda._sleep(200_000_000)                       # about 0.1 s of the default stream
    layers = [layer]
    with torch.cuda.stream(side):
        outs = []
        for _ in range(8):
            layers.append(make_layer(w))
            outs += [layers[-1].forward(dev["x"], dev) for _ in range(3)]
        side.synchronize()
    torch.cuda.synchronize()
    outs += [one.forward(dev["x"], dev) for one in layers]
    for y in outs:
        assert torch.equal(y, want)
    for one in layers:
        assert one.status() == 0
        one.close()


@pytest.mark.parametrize("more_handles", [0, 4])
def test_launch_count_of_the_small_batch_kernel_wraps(more_handles):
    """Hand-over words carry the low 32 bits of a launch count.  A batch size that was last used 2^32 launches ago, with calls of
    one token in between, must not find its old words valid; nor may the counts around the wrap.  In the pool and outside it."""
    import torch
    from paper_2502_16927_b200 import binding

    w = wl.Workload("wrap", T=16, d=128, r=64, h=128, E=8, k=4, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=43)
    inp = _inputs(w, 0.0)
    dev = to_device(w, inp)
    others = [make_layer(w) for _ in range(more_handles)]
    layer = make_layer(w)
    first, single = dev["x"].clone(), dev["x"][:1].clone()
    second = dev["x"].flip(0).contiguous()
    want, one = layer.forward(second, dev), layer.forward(single, dev)
    start = (1 << 30) + (more_handles << 20)                        # far from the counts of other tests
    for _ in range(2):
        binding.bigmac_debug_decode_launches(layer.handle, start)
        layer.forward(first, dev)                                   # its words carry start + 1
        for _ in range(2500):                                       # in place of 2^32 - 1 calls of one token
            y = layer.forward(single, dev)
        assert torch.equal(y, one)
        binding.bigmac_debug_decode_launches(layer.handle, start)
        for _ in range(3):
            assert torch.equal(layer.forward(second, dev), want)
    binding.bigmac_debug_decode_launches(layer.handle, 2 ** 32 - 3)
    for _ in range(6):
        assert torch.equal(layer.forward(second, dev), want)
        assert torch.equal(layer.forward(single, dev), one)
    assert layer.status() == 0
    binding.bigmac_debug_decode_launches(layer.handle, start + 10000)      # above all tags but those around the wrap
    for each in others + [layer]:
        each.close()


def test_small_batch_memory_goes_from_call_to_call_and_from_handle_to_handle():
    """The kernel's launch counts and hand-over words outlive a call and, in the pool of four places, a handle: batch sizes in any
    order on one handle, handles of other widths in a place, more handles than places, on two streams at a time.  Bit for bit
    what a handle that is alone computes."""
    import torch

    shapes = [dict(d=128, r=64, h=128, E=8, k=4), dict(d=256, r=192, h=320, E=12, k=2), dict(d=64, r=64, h=64, E=33, k=8)]
    sizes = [16, 1, 3, 8, 2, 16, 5, 1]
    cases = []
    for n, shape in enumerate(shapes):
        w = wl.Workload("pool", T=16, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=60 + n, **shape)
        dev = to_device(w, _inputs(w, 0.0))
        xs = {T: dev["x"][16 - T:].contiguous() for T in sizes}
        want = {}
        for T in sizes:
            layer = make_layer(w)
            want[T] = layer.forward(xs[T], dev)
            layer.close()
        cases.append((w, dev, xs, want))

    def run(layer, case, order):
        return [(layer.forward(case[2][T], case[1]), case[3][T]) for T in order]

    got = []
    for case in cases * 2:                                           # one handle after another
        layer = make_layer(case[0])
        for _ in range(3):
            got += run(layer, case, sizes)
        assert layer.status() == 0
        layer.close()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    layers = [make_layer(case[0]) for case in cases * 2]           # six at a time, three on each stream
    for n in range(20):
        for i, (layer, case) in enumerate(zip(layers, cases * 2)):
            with torch.cuda.stream(streams[i // 3]):
                got += run(layer, case, [sizes[(n + i) % len(sizes)]])
    torch.cuda.synchronize()
    assert all(torch.equal(y, want) for y, want in got)
    for layer in layers:
        assert layer.status() == 0
        layer.close()


@pytest.mark.parametrize("T", [1, 2, 16])
def test_small_batch_forward_in_a_graph(T):
    """The launch count is kept on the device: a captured call can be replayed, with other tokens, between plain calls."""
    import torch

    w = wl.Workload("graph", T=16, d=128, r=64, h=128, E=8, k=4, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=71)
    dev = to_device(w, _inputs(w, 0.0))
    batches = [dev["x"][i:i + T].contiguous() for i in range(0, 17 - T, max(1, T // 2))]
    layer = make_layer(w)
    want = [layer.forward(x, dev) for x in batches]
    x, y = batches[0].clone(), torch.empty_like(batches[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layer.forward(x, dev, y=y)
    for _ in range(3):
        for batch, ref in zip(batches, want):
            x.copy_(batch)
            graph.replay()
            assert torch.equal(y, ref)
            assert torch.equal(layer.forward(batches[-1], dev), want[-1])
    assert layer.status() == 0
    del graph
    layer.close()


@pytest.mark.parametrize("T", [300, 651])
def test_weights_hint_beside_few_and_many_descend_tiles(T):
    """Descend launches of 72 and of 144 tiles: SMs without a tile are given the experts' weights to bring to L2, or not."""
    import torch

    w = wl.Workload("hint", T=T, d=8192, r=256, h=64, E=32, k=4, dtype=wl.DTYPE_BF16, act=wl.ACT_GELU_ERF, seed=81)
    inp = _inputs(w, 0.0)
    dev = to_device(w, inp)
    layer = make_layer(w)
    y = layer.forward(dev["x"], dev)
    torch.cuda.synchronize()
    assert layer.status() == 0
    ref = oracle.forward_tokens(inp, oracle.route(inp, w.k), w.act)["y"]
    err = np.linalg.norm(to_numpy(y) - ref) / np.linalg.norm(ref)
    assert err <= 8e-3, err                              # four or five bf16 stores of 0.17 % of the rms each
    layer.close()


@pytest.mark.parametrize("r,h", [(64, 3200), (256, 1408), (320, 1664), (512, 1088), (512, 320)])
@pytest.mark.parametrize("T,skew", [(17, 0.0), (40, 4.0), (333, 2.0)])
def test_experts_in_slices_of_unequal_length(r, h, T, skew):
    """Hidden widths of 3 to 25 chunks in one to eight slices, which then differ by a chunk."""
    test_experts_in_one_kernel(r, h, T, skew)
