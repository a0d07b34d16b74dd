"""Shapes at the edges of the tensor-core kernel's tiles: the channel counts at which a position starts to stand for
2, 4 or 8 output pixels, maps whose width is no multiple of them, one activation word per pixel (two taps per K step),
channel counts around a tile of 128, tiles of fewer than 32 positions, and fp16 units fetched by TMA or by copies.
Sums and signs of binary layers are exact; fp16 outputs are checked at the tolerance of fp32 sums of exact products."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def snn():
    import paper_2110_09195_b200 as snn
    return snn


@pytest.fixture(scope="module")
def oracle_mod():
    import oracle
    oracle.build()
    return oracle


def _signs(y):
    n, h, w, k = y.shape
    bits = np.zeros((n, h, w, (k + 31) // 32 * 32), np.uint32)
    bits[..., :k] = y >= 0
    return (bits.reshape(n, h, w, -1, 32) << np.arange(32, dtype=np.uint32)).sum(axis=-1, dtype=np.uint32)


@pytest.mark.parametrize("stride,pad", [(1, 1), (1, 0), (2, 1), (2, 0)])
@pytest.mark.parametrize("c_in,c_out,h,w,n", [
    (1, 1, 3, 3, 1), (16, 15, 7, 9, 2), (31, 16, 8, 16, 3), (32, 17, 9, 13, 2), (33, 32, 5, 31, 2), (64, 33, 11, 6, 2),
    (20, 64, 6, 33, 3), (65, 65, 4, 40, 2), (96, 128, 10, 10, 2), (70, 129, 3, 57, 2), (160, 257, 6, 7, 3), (16, 16, 57, 3, 5),
])
def test_binary_tile_edges(snn, oracle_mod, c_in, c_out, h, w, n, stride, pad):
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, 6, 300 + c_in + c_out)
    alpha = p.alpha.copy()
    alpha[::3] *= -1.0
    packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, n, 301 + w))
    s_ref, y_ref = oracle_mod.conv_bin(p.codebook, 6, p.idx_packed, alpha, c_in, c_out, stride, pad, packed)
    shift = np.random.default_rng(7).normal(0, np.sqrt(9 * c_in), c_out).astype(np.float32)
    shift[::5] = -0.0   # a negative zero sum counts as +1 like a positive one
    layer = snn.SnnConv(c_in, c_out, 6, p.codebook, p.idx_packed, alpha, stride, pad, snn.ACT_BIN, shift=shift)
    act = torch.from_numpy(packed.view(np.int32)).cuda()
    assert layer.path_supported(snn.PATH_DECODED_TC, n, h, w)
    sums = layer.forward(act, out_type=snn.OUT_I32, path=snn.PATH_DECODED_TC).cpu().numpy()
    assert (sums == s_ref).all()
    y = layer.forward(act, out_type=snn.OUT_F32, path=snn.PATH_DECODED_TC).cpu().numpy()
    assert (y == s_ref.astype(np.float32) * alpha).all()
    bits = layer.forward(act, out_type=snn.OUT_BITS).cpu().numpy().view(np.uint32)
    assert (bits == _signs(s_ref.astype(np.float32) * alpha + shift)).all()
    layer.destroy()


@pytest.mark.parametrize("c_in", [65, 96, 160, 214, 224])
@pytest.mark.parametrize("c_out,h,w,n,stride,pad", [(20, 14, 14, 5, 2, 1), (130, 9, 40, 3, 2, 0), (48, 30, 31, 2, 1, 1), (16, 6, 70, 2, 1, 0)])
def test_binary_split_blocks(snn, oracle_mod, c_in, c_out, h, w, n, stride, pad):
    """Odd numbers of activation words: the one tile of a CTA as several units."""
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, 6, 340 + c_in)
    packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, n, 341 + w))
    s_ref, _ = oracle_mod.conv_bin(p.codebook, 6, p.idx_packed, p.alpha, c_in, c_out, stride, pad, packed)
    layer = snn.SnnConv(c_in, c_out, 6, p.codebook, p.idx_packed, p.alpha, stride, pad)
    act = torch.from_numpy(packed.view(np.int32)).cuda()
    assert (layer.forward(act, out_type=snn.OUT_I32).cpu().numpy() == s_ref).all()
    out = torch.full(s_ref.shape, -7, dtype=torch.int32, device="cuda")
    snn.forward_static(c_in, c_out, 6, p.codebook, p.idx_packed, p.alpha, act, out, stride, pad, snn.OUT_I32)
    assert (out.cpu().numpy() == s_ref).all()
    layer.destroy()


def test_binary_tile_edges_in_one_launch(snn, oracle_mod):
    """Members of every group size in one launch: one ring geometry for all of them."""
    shapes = [(wl.LayerShape(16, 16, 32, 32, 1, 1), 9), (wl.LayerShape(40, 32, 9, 13, 2, 1), 2), (wl.LayerShape(64, 64, 20, 21, 1, 1), 6),
              (wl.LayerShape(96, 200, 7, 7, 1, 1), 4), (wl.LayerShape(24, 16, 6, 5, 1, 0, 1), 3), (wl.LayerShape(512, 300, 5, 5, 1, 1), 2)]
    layers, acts, refs = [], [], []
    for i, (s, n) in enumerate(shapes):
        p = wl.draw_layer_params(s, 5, 400 + i)
        packed = wl.pack_activation_bits(wl.draw_activation_bits(s, n, 400 + i))
        if s.ksize == 1:
            refs.append(oracle_mod.conv1x1_bin(p.codebook, 5, p.idx_packed, p.alpha, s.c_in, s.c_out, s.stride, packed)[0])
        else:
            refs.append(oracle_mod.conv_bin(p.codebook, 5, p.idx_packed, p.alpha, s.c_in, s.c_out, s.stride, s.pad, packed)[0])
        layers.append(snn.SnnConv(s.c_in, s.c_out, 5, p.codebook, p.idx_packed, p.alpha, s.stride, s.pad, ksize=s.ksize))
        acts.append(torch.from_numpy(packed.view(np.int32)).cuda())
    group = snn.SnnConvGroup(layers, [(n, s.h, s.w) for s, n in shapes])
    for out, ref in zip(group.forward(acts, out_type=snn.OUT_I32), refs):
        assert (out.cpu().numpy() == ref).all()
    group.destroy()
    for l in layers:
        l.destroy()


@pytest.mark.parametrize("c_in,c_out,h,w,stride,pad,n", [
    (8, 16, 5, 4, 1, 1, 2),        # fewer channels than a box
    (72, 40, 9, 11, 1, 0, 3),      # a second channel block that is mostly out of bounds
    (128, 130, 30, 17, 2, 1, 2),   # parity planes as units of their own, two channel tiles
    (64, 64, 3, 255, 1, 1, 1),     # the widest row of positions a box takes at stride 1 ...
    (64, 64, 3, 256, 1, 1, 1),     # ... and one more: copied
    (16, 24, 5, 250, 2, 1, 2),     # the same at stride 2
    (16, 24, 5, 256, 2, 1, 2),
    (20, 24, 6, 7, 1, 1, 2),       # rows that are no multiple of 16 bytes: copied element by element
])
def test_fp16_units(snn, oracle_mod, c_in, c_out, h, w, stride, pad, n):
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, 5, 500 + w)
    act = wl.draw_activation_f16(shape, n, 501 + c_in)
    ref = oracle_mod.conv_f16(p.codebook, 5, p.idx_packed, p.alpha, c_in, c_out, stride, pad, act).astype(np.float64)
    layer = snn.SnnConv(c_in, c_out, 5, p.codebook, p.idx_packed, p.alpha, stride, pad, snn.ACT_F16)
    assert layer.path_supported(snn.PATH_DECODED_TC, n, h, w)
    y = layer.forward(torch.from_numpy(act).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy().astype(np.float64)
    # 9 * c_in exact products summed in fp32: each addition rounds by at most 2^-24 of the sum of magnitudes
    mag = p.alpha.astype(np.float64) * 9 * c_in * np.abs(act.astype(np.float64)).max()
    assert (np.abs(y - ref) <= 9 * c_in * 2.0 ** -24 * mag).all()
    assert np.linalg.norm(y - ref) <= 1e-5 * np.linalg.norm(ref)
    # an infinity reaches the outputs whose window holds it, and no other
    at = (0, h // 2, w // 2, c_in // 2)
    bad = act.copy()
    bad[at] = np.inf
    z = layer.forward(torch.from_numpy(bad).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy()
    hit = np.zeros(z.shape[1:3], bool)
    for i in range(z.shape[1]):
        for j in range(z.shape[2]):
            hit[i, j] = abs(i * stride - pad + 1 - at[1]) <= 1 and abs(j * stride - pad + 1 - at[2]) <= 1
    assert np.isinf(z[0][hit]).all()
    assert (z[0][~hit] == y[0][~hit].astype(np.float32)).all() and (z[1:] == y[1:].astype(np.float32)).all()
    layer.destroy()


def _whole_f16(shape, n, seed):
    """fp16 activations of small whole numbers: every sum is exact in fp32, and one multiplication by the scale rounds."""
    return np.random.default_rng(seed).integers(-8, 9, size=(n, shape.h, shape.w, shape.c_in)).astype(np.float16)


# units that the threads copy (rows that are no multiple of 16 bytes, or longer than a box), more of them per tile than the
# ring has slots: three in flight, slots reused behind them
COPIED = [(260, 24, 14, 14, 1, 1, 40), (330, 40, 12, 20, 1, 0, 9), (256, 16, 5, 300, 1, 1, 6), (260, 40, 14, 14, 2, 1, 40), (1, 3, 40, 40, 1, 1, 30)]


@pytest.mark.parametrize("c_in,c_out,h,w,stride,pad,n", COPIED)
def test_fp16_copied_units(snn, oracle_mod, c_in, c_out, h, w, stride, pad, n):
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, 5, 900 + w)
    act = _whole_f16(shape, n, 901 + c_in)
    ref = oracle_mod.conv_f16(p.codebook, 5, p.idx_packed, p.alpha, c_in, c_out, stride, pad, act).astype(np.float64)
    layer = snn.SnnConv(c_in, c_out, 5, p.codebook, p.idx_packed, p.alpha, stride, pad, snn.ACT_F16)
    y = layer.forward(torch.from_numpy(act).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy().astype(np.float64)
    assert (np.abs(y - ref) <= 2.0 ** -23 * np.abs(ref)).all()
    layer.destroy()


def test_fp16_copied_and_fetched_members_in_one_launch(snn, oracle_mod):
    """Members whose units are copied and members whose units are fetched by TMA take turns, with several tiles per CTA: the
    copies in flight are finished before the next member's units, and the ring carries on."""
    shapes = [(wl.LayerShape(260, 24, 14, 14, 1, 1), 40), (wl.LayerShape(72, 40, 20, 20, 1, 1), 90), (wl.LayerShape(330, 16, 12, 20, 1, 0), 30),
              (wl.LayerShape(256, 32, 14, 14, 2, 1), 60), (wl.LayerShape(36, 130, 16, 16, 2, 1), 60), (wl.LayerShape(64, 64, 28, 28, 1, 1), 40)]
    layers, acts, refs = [], [], []
    for i, (s, n) in enumerate(shapes):
        p = wl.draw_layer_params(s, 5, 950 + i)
        act = _whole_f16(s, n, 960 + i)
        refs.append(oracle_mod.conv_f16(p.codebook, 5, p.idx_packed, p.alpha, s.c_in, s.c_out, s.stride, s.pad, act).astype(np.float64))
        layers.append(snn.SnnConv(s.c_in, s.c_out, 5, p.codebook, p.idx_packed, p.alpha, s.stride, s.pad, snn.ACT_F16))
        acts.append(torch.from_numpy(act).cuda())
    group = snn.SnnConvGroup(layers, [(n, s.h, s.w) for s, n in shapes])
    for _ in range(2):
        for out, ref in zip(group.forward(acts), refs):
            assert (np.abs(out.cpu().numpy().astype(np.float64) - ref) <= 2.0 ** -23 * np.abs(ref)).all()
    group.destroy()
    for l in layers:
        l.destroy()


@pytest.mark.parametrize("c_out", [1, 16, 17, 32, 33, 64, 65])
@pytest.mark.parametrize("c_in,h,w,n,stride", [(16, 32, 32, 40, 1), (24, 9, 11, 3, 2), (20, 40, 28, 36, 1)])
def test_fp16_few_channels(snn, oracle_mod, c_in, c_out, h, w, n, stride):
    """Lanes that hold copies of the channels: tiles of one slice and of many, fetched and copied units."""
    shape = wl.LayerShape(c_in, c_out, h, w, stride, 1)
    p = wl.draw_layer_params(shape, 5, 800 + c_out)
    act = wl.draw_activation_f16(shape, n, 801 + c_in)
    ref = oracle_mod.conv_f16(p.codebook, 5, p.idx_packed, p.alpha, c_in, c_out, stride, 1, act).astype(np.float64)
    layer = snn.SnnConv(c_in, c_out, 5, p.codebook, p.idx_packed, p.alpha, stride, 1, snn.ACT_F16)
    y = layer.forward(torch.from_numpy(act).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy().astype(np.float64)
    # 9 * c_in exact products summed in fp32: each addition rounds by at most 2^-24 of the sum of magnitudes
    mag = p.alpha.astype(np.float64) * 9 * c_in * np.abs(act.astype(np.float64)).max()
    assert (np.abs(y - ref) <= 9 * c_in * 2.0 ** -24 * mag).all()
    layer.destroy()


@pytest.mark.parametrize("stride,pad", [(1, 1), (2, 0)])
@pytest.mark.parametrize("c_in,c_out,h,w,n,tau", [
    (1, 1, 3, 3, 1, 1), (16, 16, 9, 8, 2, 3), (31, 33, 6, 7, 2, 9), (64, 64, 5, 12, 2, 5), (70, 20, 8, 5, 3, 7), (129, 200, 4, 6, 2, 8),
    (512, 128, 4, 4, 1, 9), (3, 512, 5, 6, 1, 2),
])
def test_operand_from_the_stored_form(snn, oracle_mod, c_in, c_out, h, w, n, tau, stride, pad):
    """forward_static writes the weight operand from the index stream itself: indices of any width that straddle bytes and
    end the stream, ragged words, groups of pixels, two taps per step."""
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, tau, 600 + c_in)
    packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, n, 601 + w))
    s_ref, _ = oracle_mod.conv_bin(p.codebook, tau, p.idx_packed, p.alpha, c_in, c_out, stride, pad, packed)
    act = torch.from_numpy(packed.view(np.int32)).cuda()
    out = torch.full(s_ref.shape, -7, dtype=torch.int32, device="cuda")
    snn.forward_static(c_in, c_out, tau, p.codebook, p.idx_packed, p.alpha, act, out, stride, pad, snn.OUT_I32)
    assert (out.cpu().numpy() == s_ref).all()
    # pinned arrays are copied from where they are, in stream order
    pinned = torch.from_numpy(p.idx_packed).pin_memory()
    out.fill_(-7)
    snn.forward_static(c_in, c_out, tau, p.codebook, pinned.numpy(), p.alpha, act, out, stride, pad, snn.OUT_I32)
    assert (out.cpu().numpy() == s_ref).all()


def test_stored_form_under_capture(snn, oracle_mod):
    """A captured call copies the layer's arrays at every replay, as it did before it was gathered into one copy."""
    shape, n, tau = wl.LayerShape(64, 48, 8, 8, 1, 1), 2, 5
    p, q = wl.draw_layer_params(shape, tau, 700), wl.draw_layer_params(shape, tau, 701)
    packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, n, 702))
    refs = [oracle_mod.conv_bin(l.codebook, tau, l.idx_packed, l.alpha, 64, 48, 1, 1, packed)[0] for l in (p, q)]
    act = torch.from_numpy(packed.view(np.int32)).cuda()
    out = torch.zeros(refs[0].shape, dtype=torch.int32, device="cuda")
    arrays = [torch.from_numpy(a.copy()).pin_memory() for a in (p.codebook.view(np.int16), p.idx_packed, p.alpha)]
    args = (arrays[0].numpy().view(np.uint16), arrays[1].numpy(), arrays[2].numpy())
    snn.forward_static(64, 48, tau, *args, act, out, out_type=snn.OUT_I32)   # the first call resolves the array
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        snn.forward_static(64, 48, tau, *args, act, out, out_type=snn.OUT_I32)
    graph.replay()
    torch.cuda.synchronize()
    assert (out.cpu().numpy() == refs[0]).all()
    for a, new in zip(arrays, (q.codebook.view(np.int16), q.idx_packed, q.alpha)):
        a.copy_(torch.from_numpy(new.copy()))
    graph.replay()
    torch.cuda.synchronize()
    assert (out.cpu().numpy() == refs[1]).all()


@pytest.mark.parametrize("c_in,c_out,h,w,n", [(40, 48, 5, 6, 1), (64, 70, 9, 29, 4), (33, 16, 20, 21, 3), (128, 256, 14, 14, 12)])
def test_signs_where_scaled_sums_round_or_cancel(snn, oracle_mod, c_in, c_out, h, w, n):
    """The kernel compares a sum with the integer at which fl(fl(alpha*S) + shift) changes its sign: scales of zero, subnormal and
    overflowing products, shifts that cancel a product exactly or miss it by a rounding, and shifts beyond every sum; tiles
    of one slice of 32 positions, of several, and of an odd number."""
    shape = wl.LayerShape(c_in, c_out, h, w, 1, 1)
    p = wl.draw_layer_params(shape, 6, 500 + c_in)
    packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, n, 501 + w))
    rng = np.random.default_rng(c_out)
    f32 = np.float32
    scales = np.array([1.0, -1.0, 0.0, -0.0, 1e-45, -1e-45, 1.2e-38, 3e38, -3e38, 0.1, -0.1, 0.3333333, 1.0000001], f32)
    alpha = scales[rng.integers(0, len(scales), c_out)]
    near = rng.integers(-30, 31, c_out).astype(f32)
    with np.errstate(over="ignore"):
        shift = np.clip(-(alpha * near), f32(-3.3e38), f32(3.3e38))
        kind = rng.integers(0, 6, c_out)
        shift = np.where(kind == 1, np.nextafter(shift, f32(-1)), np.where(kind == 2, np.nextafter(shift, f32(1)), shift))
        shift = np.where(kind == 3, f32(-0.0), np.where(kind == 4, f32(1e30), np.where(kind == 5, f32(-1e30), shift))).astype(f32)
        s_ref, _ = oracle_mod.conv_bin(p.codebook, 6, p.idx_packed, p.alpha, c_in, c_out, 1, 1, packed)
        want = _signs((s_ref.astype(f32) * alpha) + shift)
    layer = snn.SnnConv(c_in, c_out, 6, p.codebook, p.idx_packed, alpha, 1, 1, snn.ACT_BIN, shift=shift)
    got = layer.forward(torch.from_numpy(packed.view(np.int32)).cuda(), out_type=snn.OUT_BITS).cpu().numpy().view(np.uint32)
    assert (got == want).all()
    layer.destroy()


@pytest.mark.parametrize("stride,pad", [(1, 1), (1, 0), (2, 1), (2, 0)])
@pytest.mark.parametrize("c_in,c_out,h,w,n", [(8, 33, 5, 5, 1), (64, 64, 15, 15, 3), (72, 48, 9, 31, 2), (128, 40, 20, 57, 4), (16, 64, 30, 30, 12)])
def test_fp16_layers_of_33_to_64_channels(snn, oracle_mod, c_in, c_out, h, w, n, stride, pad):
    """Two kernel columns in the rows of the weight operand: sums put together over two columns of the accumulator, tiles that overlap by
    one position, one and several slices and channel blocks; an infinity reaches the outputs whose windows hold it and no others."""
    shape = wl.LayerShape(c_in, c_out, h, w, stride, pad)
    p = wl.draw_layer_params(shape, 6, 700 + c_in + c_out)
    rng = np.random.default_rng(31)
    x = rng.standard_normal((n, h, w, c_in)).astype(np.float16)
    layer = snn.SnnConv(c_in, c_out, 6, p.codebook, p.idx_packed, p.alpha, stride, pad, snn.ACT_F16)
    assert layer.path_supported(snn.PATH_DECODED_TC, n, h, w)
    for k in range(2):
        if k:
            x[rng.random(x.shape) < 0.4 / (9 * c_in)] = np.inf
            x[rng.random(x.shape) < 0.2 / (9 * c_in)] = -np.inf
        with np.errstate(invalid="ignore"):
            want = oracle_mod.conv_f16(p.codebook, 6, p.idx_packed, p.alpha, c_in, c_out, stride, pad, x)
        got = layer.forward(torch.from_numpy(x).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy()
        finite = np.isfinite(want)
        assert finite.all() or k
        assert (np.isnan(got) == np.isnan(want)).all() and (got[np.isinf(want)] == want[np.isinf(want)]).all()
        # exact products, fp32 sums of 9*c_in terms: 2^-24 a step of the sum at most, on terms of size one
        assert (np.abs(got[finite] - want[finite]) <= 2.0 ** -24 * 9 * c_in * 1.5 * 4 * np.sqrt(9 * c_in)).all()
    layer.destroy()


@pytest.mark.parametrize("unit", [2.0 ** -24, 1024.0])
@pytest.mark.parametrize("c_in,c_out,h,w,n", [(32, 33, 5, 5, 1), (64, 64, 13, 31, 3), (72, 48, 20, 57, 2)])
def test_fp16_halves_of_kernel_columns_are_exact(snn, oracle_mod, c_in, c_out, h, w, n, unit):
    """Activations of whole units, from the smallest fp16 number to near the largest: half a unit is exact, and so is every sum (below 2^24 halves)."""
    shape = wl.LayerShape(c_in, c_out, h, w, 1, 1)
    p = wl.draw_layer_params(shape, 6, 800 + c_in)
    x = (np.random.default_rng(32).integers(-63, 64, (n, h, w, c_in)) * unit).astype(np.float16)
    want = oracle_mod.conv_f16(p.codebook, 6, p.idx_packed, np.ones(c_out, np.float32), c_in, c_out, 1, 1, x)
    layer = snn.SnnConv(c_in, c_out, 6, p.codebook, p.idx_packed, np.ones(c_out, np.float32), 1, 1, snn.ACT_F16)
    got = layer.forward(torch.from_numpy(x).cuda(), path=snn.PATH_DECODED_TC).cpu().numpy()
    assert (got == want).all()
    layer.destroy()
