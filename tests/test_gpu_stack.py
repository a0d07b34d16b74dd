"""The dependent stack (snn_conv_stack_*: layers chained through their packed thresholded signs, one
persistent launch) against the same chain through the CPU oracle: every layer's signs are an integer
decision, so the chain is compared bit for bit.  Where at most 2^17 words lie between two members the
words carry tags, else the members' tiles are counted: two variants of the kernel, and each of the
shapes that need care runs on both (tests/test_plan.py checks which of them a chain gets)."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def snn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_09195_b200 import build
    build.build()
    import paper_2110_09195_b200 as m
    m.load_library()
    return m


def _pack_signs(y, shift):
    """fl(Y + shift) >= 0 in fp32, packed along c_out into little-endian uint32 words (oracle side)."""
    y = (y.astype(np.float32) + shift.astype(np.float32)[None, None, None, :]).astype(np.float32)
    bits = y >= 0
    n, h, w, k = bits.shape
    kw = (k + 31) // 32
    pad = np.zeros((n, h, w, kw * 32), dtype=np.uint64)
    pad[..., :k] = bits
    weights = np.uint64(1) << np.arange(32, dtype=np.uint64)
    return (pad.reshape(n, h, w, kw, 32) * weights).sum(axis=-1).astype(np.uint32)


def _build_chain(snn, oracle_mod, shapes, tau, n, seed):
    """Draws the layers, runs the chain through the oracle; returns (layers, first input, per-layer packed
    signs, last layer's (S, Y))."""
    layers, mids = [], []
    x = wl.pack_activation_bits(wl.draw_activation_bits(shapes[0], n, seed))
    first = x
    last = None
    for i, shape in enumerate(shapes):
        p = wl.draw_layer_params(shape, tau, seed + i)
        rng = np.random.default_rng(seed + 100 + i)
        alpha = p.alpha.copy()
        alpha[::7] *= -1.0
        # thresholds of the size of the sums' spread keep the signs balanced through the chain
        shift = (rng.normal(0.0, 1.0, size=shape.c_out) * np.sqrt(9.0 * shape.c_in) * 0.5).astype(np.float32)
        if shape.ksize == 1:
            s_ref, y_ref = oracle_mod.conv1x1_bin(p.codebook, tau, p.idx_packed, alpha, shape.c_in, shape.c_out, shape.stride, x)
        else:
            s_ref, y_ref = oracle_mod.conv_bin(p.codebook, tau, p.idx_packed, alpha, shape.c_in, shape.c_out, shape.stride,
                                               shape.pad, x)
        last = (s_ref, y_ref)
        x = _pack_signs(y_ref, shift)
        mids.append(x)
        layers.append(snn.SnnConv(shape.c_in, shape.c_out, tau, p.codebook, p.idx_packed, alpha, shape.stride,
                                  shape.pad, snn.ACT_BIN, shift=shift, ksize=shape.ksize))
    return layers, first, mids, last


def _check_chain(snn, oracle_mod, shapes, tau, n, seed, repeats=2):
    layers, first, mids, (s_ref, y_ref) = _build_chain(snn, oracle_mod, shapes, tau, n, seed)
    stack = snn.SnnConvStack(layers, n, shapes[0].h, shapes[0].w)
    act = torch.from_numpy(first.view(np.int32)).cuda()
    for _ in range(repeats):
        bits = stack.forward(act, out_type=snn.OUT_BITS)
        sums = stack.forward(act, out_type=snn.OUT_I32)
        outs = stack.forward(act, out_type=snn.OUT_F32)
        torch.cuda.synchronize()
        assert (bits.cpu().numpy().view(np.uint32) == mids[-1]).all()
        assert (sums.cpu().numpy() == s_ref).all()
        assert (outs.cpu().numpy() == y_ref).all()
    stack.destroy()
    for l in layers:
        l.destroy()


def test_stack_of_one(snn, oracle_mod):
    _check_chain(snn, oracle_mod, [wl.LayerShape(16, 16, 32, 32, 1, 1)], 5, 1, 301)


def test_stack_small_ragged_chain(snn, oracle_mod):
    shapes = [wl.LayerShape(33, 40, 13, 11, 1, 1), wl.LayerShape(40, 70, 13, 11, 2, 1), wl.LayerShape(70, 24, 7, 6, 1, 0),
              wl.LayerShape(24, 130, 5, 4, 1, 1), wl.LayerShape(130, 9, 5, 4, 2, 1)]
    _check_chain(snn, oracle_mod, shapes, 5, 3, 311)


@pytest.mark.parametrize("n", [2, 64])
def test_stack_resnet18_full_depth(snn, oracle_mod, n):
    """The 16 ResNet-18-shaped layers as one dependent chain, at batch 2 and at the benchmark's batch 64."""
    wk = wl.get_workload("resnet18")
    _check_chain(snn, oracle_mod, list(wk.layers), wk.tau, n, 321, repeats=1 if n == 64 else 2)


def test_stack_resnet20_full_depth(snn, oracle_mod):
    wk = wl.get_workload("resnet20")
    _check_chain(snn, oracle_mod, list(wk.layers), wk.tau, 4, 331)


def test_stack_argument_errors(snn):
    a = wl.draw_layer_params(wl.LayerShape(16, 32, 8, 8), 5, 3)
    b = wl.draw_layer_params(wl.LayerShape(16, 16, 8, 8), 5, 4)
    la = snn.SnnConv(16, 32, 5, a.codebook, a.idx_packed, a.alpha)
    lb = snn.SnnConv(16, 16, 5, b.codebook, b.idx_packed, b.alpha)
    lf = snn.SnnConv(16, 16, 5, b.codebook, b.idx_packed, b.alpha, act_type=snn.ACT_F16)
    with pytest.raises(snn.SnnError) as ei:
        snn.SnnConvStack([la, lb], 1, 8, 8)          # 32 channels out, 16 in
    assert ei.value.status == 1
    with pytest.raises(snn.SnnError) as ei:
        snn.SnnConvStack([lf], 1, 8, 8)              # fp16 activations do not chain
    assert ei.value.status == 1
    st = snn.SnnConvStack([lb, la], 1, 8, 8)
    with pytest.raises(snn.SnnError) as ei:
        st.forward(torch.zeros((2, 8, 8, 1), dtype=torch.int32, device="cuda"))
    assert ei.value.status == 1
    st.destroy()
    for l in (la, lb, lf):
        l.destroy()


@pytest.mark.parametrize("chans,hw,n", [
    ((33, 64, 96, 128, 40), 9, 2),          # one and two words a pixel, blocks of two and four chunks
    ((160, 192, 256, 288, 70), 8, 1),       # five to nine words: blocks of six and eight chunks, odd word counts
    ((16, 16, 16), 32, 128),                # as many words between the members as may carry tags ...
    ((16, 16, 16), 32, 129),                # ... and one image more
])
def test_stack_words_between_members(snn, oracle_mod, chans, hw, n):
    """Chains whose words carry tags and the first that runs on counters; several launches of one stack, and its graph."""
    shapes = [wl.LayerShape(a, b, hw, hw, 1, 1) for a, b in zip(chans, chans[1:])]
    _check_chain(snn, oracle_mod, shapes, 6, n, 341, repeats=1 if n > 2 else 3)


def test_stack_replayed_as_a_graph(snn, oracle_mod):
    """A replay is a launch like any other to the tags: new inputs in the same buffer give new outputs every time."""
    shapes = [wl.LayerShape(64, 64, 10, 10, 1, 1), wl.LayerShape(64, 128, 10, 10, 2, 1), wl.LayerShape(128, 96, 5, 5, 1, 1)]
    layers, first, _, _ = _build_chain(snn, oracle_mod, shapes, 5, 2, 351)
    stack = snn.SnnConvStack(layers, 2, 10, 10)
    inputs = [torch.from_numpy(first.view(np.int32)).cuda()]
    inputs += [torch.randint(-2 ** 31, 2 ** 31, inputs[0].shape, dtype=torch.int32, device="cuda") for _ in range(3)]
    want = [stack.forward(x).clone() for x in inputs]
    act, out = inputs[0].clone(), stack.alloc_out()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            stack.forward(act, out)
            stack.forward(act, out)
        for i in (1, 2, 3, 0, 2):
            act.copy_(inputs[i])
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want[i])
    del graph
    stack.destroy()
    for l in layers:
        l.destroy()


@pytest.mark.parametrize("h,w,n", [(40, 50, 4), (100, 150, 5)])   # words with tags, and counters
def test_stack_whose_ctas_pass_members_by(snn, oracle_mod, h, w, n):
    """Members of a few tiles in a row, then one of more: most CTAs have no tile in several members, and some have one again."""
    chans, strides = (64, 40, 16, 16, 16, 16, 16, 512, 24), (1, 2, 2, 2, 2, 1, 1, 1)
    shapes = []
    for a, b, s in zip(chans, chans[1:], strides):
        shapes.append(wl.LayerShape(a, b, h, w, s, 1))
        h, w = shapes[-1].h_out, shapes[-1].w_out
    _check_chain(snn, oracle_mod, shapes, 5, n, 361, repeats=1)


def chain_shapes(chans, h, w, strides, pads, ksizes):
    shapes = []
    for a, b, s, p, k in zip(chans, chans[1:], strides, pads, ksizes):
        shapes.append(wl.LayerShape(a, b, h, w, s, p, k))
        h, w = shapes[-1].h_out, shapes[-1].w_out
    return shapes


# channels, map, strides, pads, kernel sizes, batch with tags, batch with counters
CHAINS = [
    # two and three words a pixel, a last word of few channels, no padding, channel tiles of 2 and 9 channels
    ((33, 40, 70, 24, 130, 9), 13, 11, (1, 2, 1, 1, 2), (1, 1, 0, 1, 1), (3,) * 5, 458, 480),
    # five, seven and nine words a pixel: one word a load, blocks of several chunks; an odd map without padding
    ((160, 200, 257, 288, 70), 15, 9, (1, 1, 2, 1), (1, 0, 1, 1), (3,) * 4, 138, 175),
    # groups of two, four and eight pixels a position, stride 2
    ((20, 64, 17, 31, 16, 48), 37, 29, (1, 1, 2, 1, 2), (1, 1, 1, 0, 1), (3,) * 5, 61, 67),
    # a bottleneck: 1x1, 3x3 at stride 2, 1x1
    ((256, 72, 136, 512), 28, 28, (1, 2, 1), (0, 1, 0), (1, 3, 1), 55, 58),
    # one member: nothing lies between members (tags whatever the batch)
    ((40, 70), 13, 11, (2,), (1,), (3,), 5, None),
]


@pytest.mark.parametrize("chain,n", [(c, n) for c in CHAINS for n in c[6:] if n],
                         ids=lambda v: "-".join(map(str, v[0])) if isinstance(v, tuple) else str(v))
def test_stack_by_tags_and_by_counters(snn, oracle_mod, chain, n):
    _check_chain(snn, oracle_mod, chain_shapes(*chain[:6]), 6, n, 371, repeats=1)
