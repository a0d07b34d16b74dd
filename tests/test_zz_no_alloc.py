"""The no-allocation entry point against the ordinary one and against the oracle.

`snn_conv_forward_static` serves hosts that cannot let this library allocate
device memory (the application owns the whole device through its own pool, or
runs with a fixed memory budget, or sits in a loop that cannot take the
synchronisation an allocation may cause).  It keeps its working data in one
fixed array inside the library, shared by all calls.  This test calls it twice
in a row through the C ABI, on two different layers, and checks both results
against `snn_conv_forward` on a handle and against the CPU oracle: the second
call must not be affected by what the first one left in the shared array.  It
is collected last so that a run stopping at the first failure has already run
every other test.
"""
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


def _handle_path(snn, shape, p, act, out_type):
    layer = snn.SnnConv(shape.c_in, shape.c_out, p.tau, p.codebook, p.idx_packed, p.alpha, shape.stride, shape.pad)
    ref = layer.forward(act, out_type=out_type, path=snn.PATH_DECODED)
    torch.cuda.synchronize()
    layer.destroy()
    return ref


def _check_case(snn, oracle_mod, shape, tau, n, seed):
    p = wl.draw_layer_params(shape, tau, seed)
    bits = wl.draw_activation_bits(shape, n, seed)
    packed = wl.pack_activation_bits(bits)
    s_ref, y_ref = oracle_mod.conv_bin(p.codebook, tau, p.idx_packed, p.alpha, shape.c_in, shape.c_out, shape.stride,
                                       shape.pad, packed)
    act = torch.from_numpy(packed.view(np.int32)).cuda()
    ho, wo = shape.h_out, shape.w_out
    for out_type, dtype in ((snn.OUT_I32, torch.int32), (snn.OUT_F32, torch.float32)):
        ref = _handle_path(snn, shape, p, act, out_type)
        out = torch.full((n, ho, wo, shape.c_out), -7, dtype=dtype, device="cuda")
        snn.forward_static(shape.c_in, shape.c_out, tau, p.codebook, p.idx_packed, p.alpha, act, out,
                           stride=shape.stride, pad=shape.pad, out_type=out_type)
        torch.cuda.synchronize()
        if out_type == snn.OUT_I32:
            assert torch.equal(out, ref)                       # the existing entry point: bit-exact
            assert (out.cpu().numpy() == s_ref).all()          # the oracle: bit-exact integer sums
        else:
            r = ref.cpu().numpy()
            o = out.cpu().numpy()
            assert (np.abs(o - r) <= 1e-6 * np.abs(r)).all()
            assert (np.abs(o - y_ref) <= 1e-6 * np.abs(y_ref)).all()


def test_two_calls_in_a_row_match_the_handle_path_and_the_oracle(snn, oracle_mod):
    cases = [
        (wl.LayerShape(96, 130, 9, 11, 1, 1), 6, 3, 11),   # first call: larger layer, fills more of the array
        (wl.LayerShape(33, 20, 7, 6, 2, 1), 3, 2, 12),     # second call: smaller layer over stale contents
    ]
    for shape, tau, n, seed in cases:
        _check_case(snn, oracle_mod, shape, tau, n, seed)


def test_largest_layer_the_array_holds(snn, oracle_mod):
    """512 -> 512 channels with the full 512-kernel codebook: the documented upper limit."""
    _check_case(snn, oracle_mod, wl.LayerShape(512, 512, 3, 3, 1, 1), 9, 1, 13)


def test_a_warmed_call_leaves_device_memory_alone(snn):
    shape = wl.LayerShape(64, 48, 8, 8, 1, 1)
    p = wl.draw_layer_params(shape, 5, 14)
    act = torch.from_numpy(wl.pack_activation_bits(wl.draw_activation_bits(shape, 2, 14)).view(np.int32)).cuda()
    out = torch.empty((2, 8, 8, 48), dtype=torch.float32, device="cuda")
    snn.forward_static(64, 48, 5, p.codebook, p.idx_packed, p.alpha, act, out)   # the first call resolves the array
    torch.cuda.synchronize()
    free_before = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        snn.forward_static(64, 48, 5, p.codebook, p.idx_packed, p.alpha, act, out)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free_before


def test_sizes_beyond_the_fixed_array_are_refused(snn):
    shape = wl.LayerShape(520, 16, 5, 5, 1, 1)
    p = wl.draw_layer_params(shape, 2, 1)
    act = torch.zeros((1, 5, 5, 17), dtype=torch.int32, device="cuda")
    out = torch.zeros((1, 5, 5, 16), dtype=torch.float32, device="cuda")
    with pytest.raises(snn.SnnError) as ei:
        snn.forward_static(520, 16, 2, p.codebook, p.idx_packed, p.alpha, act, out)
    assert ei.value.status == 2 and "512" in str(ei.value)


def test_wrong_buffers_are_refused_on_the_host(snn):
    """The C entry point cannot see buffer sizes, so the binding checks them: nothing is launched."""
    shape = wl.LayerShape(64, 48, 8, 8, 1, 1)
    p = wl.draw_layer_params(shape, 5, 15)
    act = torch.zeros((2, 8, 8, 2), dtype=torch.int32, device="cuda")
    good = torch.zeros((2, 8, 8, 48), dtype=torch.float32, device="cuda")
    before = snn.kernel_launches()
    bad_calls = [
        dict(act=torch.zeros((2, 8, 8, 1), dtype=torch.int32, device="cuda"), out=good),            # too few words
        dict(act=act, out=torch.zeros((2, 8, 8, 40), dtype=torch.float32, device="cuda")),          # wrong c_out
        dict(act=act, out=torch.zeros((2, 4, 4, 48), dtype=torch.float32, device="cuda")),          # wrong map
        dict(act=act, out=torch.zeros((2, 8, 8, 48), dtype=torch.int32, device="cuda")),            # wrong dtype
        dict(act=act.to(torch.float32), out=good),                                                   # wrong act dtype
    ]
    for kw in bad_calls:
        with pytest.raises(snn.SnnError) as ei:
            snn.forward_static(64, 48, 5, p.codebook, p.idx_packed, p.alpha, kw["act"], kw["out"])
        assert ei.value.status == 1
    with pytest.raises(snn.SnnError):
        snn.forward_static(64, 48, 5, p.codebook, p.idx_packed, p.alpha, act, good, stride=2)       # out is stride-1 sized
    assert snn.kernel_launches() == before


@pytest.mark.parametrize("c_in,c_out,h,w,stride,pad,tau,n", [
    (1, 1, 5, 4, 1, 1, 1, 1),          # one channel of a word, one row of the operand
    (31, 5, 9, 9, 2, 1, 9, 3),         # pairs of taps, groups of pixels, indices across byte borders
    (32, 16, 32, 32, 1, 1, 5, 8),      # eight pixels a position: sixteen rows each
    (33, 17, 12, 7, 1, 0, 7, 2),       # words without any channel in a block of two chunks
    (65, 64, 14, 14, 2, 1, 6, 4),
    (160, 127, 9, 26, 1, 1, 3, 2),     # blocks of six chunks
    (200, 129, 6, 6, 1, 1, 8, 2),      # a second channel tile of one row
])
def test_operand_from_the_stored_form(snn, oracle_mod, c_in, c_out, h, w, stride, pad, tau, n):
    _check_case(snn, oracle_mod, wl.LayerShape(c_in, c_out, h, w, stride, pad), tau, n, 17)


@pytest.mark.parametrize("c_in,c_out,tau", [(32, 64, 7), (33, 64, 7), (96, 128, 7), (97, 128, 7), (272, 128, 7), (273, 128, 7), (17, 500, 9), (1, 1, 1)])
def test_stored_forms_around_the_sizes_that_go_with_the_launch(snn, oracle_mod, c_in, c_out, tau):
    """3072, 12288 and 32000 bytes and a little more: parameters of three sizes, and beyond them a copy.  Calls follow one another
    without a wait, each with another layer's arrays, which are overwritten as soon as the call returns."""
    shape = wl.LayerShape(c_in, c_out, 6, 9, 1, 1)
    calls = []
    for seed in range(4):
        p = wl.draw_layer_params(shape, tau, 70 + seed)
        packed = wl.pack_activation_bits(wl.draw_activation_bits(shape, 2, 90 + seed))
        ref = oracle_mod.conv_bin(p.codebook, tau, p.idx_packed, p.alpha, c_in, c_out, 1, 1, packed)[1]
        calls.append((p, torch.from_numpy(packed.view(np.int32)).cuda(), torch.empty((2, 6, 9, c_out), device="cuda"), ref))
    book, stream, alpha = (np.array(a) for a in (calls[0][0].codebook, calls[0][0].idx_packed, calls[0][0].alpha))
    for p, act, out, _ in calls:
        book[:], stream[:], alpha[:] = p.codebook, p.idx_packed, p.alpha
        snn.forward_static(c_in, c_out, tau, book, stream, alpha, act, out)
        book[:], stream[:], alpha[:] = 0, 0, 0
    for _, _, out, ref in calls:
        assert (out.cpu().numpy() == ref).all()


@pytest.mark.parametrize("n,h,w", [(2, 6, 9), (8, 28, 28)])
def test_calls_behind_the_kernel_that_writes_their_activations(snn, oracle_mod, n, h, w):
    """A layer's launch writes the activations right before each call, no wait between; calls whose stored form goes with the launch (64
    outputs) and calls whose arrays are copied (500, tau 9) in turn, each with scales of its own; few tiles, and one on every SM."""
    first = wl.LayerShape(48, 64, h, w, 1, 1)
    p = wl.draw_layer_params(first, 6, 300)
    producer = snn.SnnConv(48, 64, 6, p.codebook, p.idx_packed, p.alpha, 1, 1)
    act = torch.empty((n, h, w, 2), dtype=torch.int32, device="cuda")
    calls = []
    for k, (c_out, tau) in enumerate([(64, 7), (500, 9), (64, 7), (64, 7), (500, 9), (64, 7)]):
        packed = wl.pack_activation_bits(wl.draw_activation_bits(first, n, 310 + k))
        sums = oracle_mod.conv_bin(p.codebook, 6, p.idx_packed, p.alpha, 48, 64, 1, 1, packed)[0]
        q = wl.draw_layer_params(wl.LayerShape(64, c_out, h, w, 1, 1), tau, 320 + k)
        ref = oracle_mod.conv_bin(q.codebook, tau, q.idx_packed, q.alpha, 64, c_out, 1, 1, wl.pack_activation_bits(sums >= 0))[1]
        calls.append((torch.from_numpy(packed.view(np.int32)).cuda(), q, c_out, torch.empty((n, h, w, c_out), device="cuda"), ref))
    torch.cuda.synchronize()
    for x, q, c_out, out, _ in calls:
        producer.forward(x, out=act, out_type=snn.OUT_BITS)
        snn.forward_static(64, c_out, q.tau, q.codebook, q.idx_packed, q.alpha, act, out)
    for *_, out, ref in calls:
        assert (out.cpu().numpy() == ref).all()
    producer.destroy()
