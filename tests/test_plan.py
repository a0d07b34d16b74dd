"""The planner of the tensor-core kernel, compiled for the host: every shape the path takes can be planned, fits shared and
tensor memory, and keeps the kernel's reads inside what is staged."""
import ctypes
import random
import subprocess
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parent.parent
WORDS, CHAIN, SIGNS = 0, 1, 2
SMS = 148


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("plan") / "plan.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", f"-I{ROOT}/include", f"-I{ROOT}/paper_2110_09195_b200/csrc",
                    "-I/usr/local/cuda/include", "-o", str(so), str(ROOT / "tests/plan_harness.cpp")], check=True)
    lib = ctypes.CDLL(str(so))
    lib.plan_make.restype = ctypes.c_char_p
    return lib


def _array(shapes):
    return np.array(shapes, np.int32).ctypes.data_as(ctypes.POINTER(ctypes.c_int))


def takes(lib, shape, f16):
    return bool(lib.plan_takes(_array(shape), int(f16)))


def make(lib, shapes, f16=False, kind=WORDS):
    """[(lg, Np, tma, tiles, channel blocks)] of the problems (N, H, W, C, K, stride, pad, ksize)."""
    out = np.zeros((len(shapes), 5), np.int32)
    err = lib.plan_make(_array(shapes), len(shapes), int(f16), kind, SMS, out.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))
    assert err is None, (err, shapes, f16, kind)
    return out.tolist()


def draw(rng):
    log = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    ksize = rng.choice((3, 3, 3, 1))
    return (log(1, 300), log(3, 700), log(3, 700), log(1, 1200), log(1, 1200), rng.choice((1, 2)),
            0 if ksize == 1 else rng.choice((0, 1)), ksize)


@pytest.mark.parametrize("f16", [False, True])
def test_every_shape_the_path_takes_can_be_planned(lib, f16):
    rng = random.Random(5)
    taken = 0
    for _ in range(4000):
        shape = draw(rng)
        if not takes(lib, shape, f16):
            continue
        taken += 1
        for kind in (WORDS,) if f16 else (WORDS, SIGNS, CHAIN):
            make(lib, [shape], f16, kind)
    assert taken > 500


@pytest.mark.parametrize("f16", [False, True])
def test_every_group_of_such_shapes_can_be_planned(lib, f16):
    rng = random.Random(6)
    for _ in range(60):
        shapes = [s for s in (draw(rng) for _ in range(80)) if takes(lib, s, f16)][:rng.randint(2, 32)]
        for kind in (WORDS,) if f16 else (WORDS, SIGNS):
            make(lib, shapes, f16, kind)


@pytest.mark.parametrize("shape,kind,tiles", [
    # N, H, W, C, K, stride, pad, ksize: what packs each of these into fewer tiles takes 1.2 to 3 times as long
    ((16, 14, 14, 96, 20, 2, 1, 3), WORDS, 32), ((4, 14, 14, 512, 16, 1, 1, 3), WORDS, 16), ((4, 46, 33, 93, 31, 2, 1, 3), WORDS, 50),
    ((1, 30, 30, 96, 16, 1, 1, 3), WORDS, 20), ((4, 56, 56, 256, 16, 1, 1, 3), SIGNS, 100), ((21, 10, 43, 214, 24, 2, 1, 3), SIGNS, 31),
    ((4, 56, 56, 96, 16, 1, 0, 1), SIGNS, 98),
])
def test_a_small_layer_of_few_channels_is_spread_over_the_machine(lib, shape, kind, tiles):
    (lg, _, _, got, _), = make(lib, [shape], kind=kind)
    assert lg <= 1 and got >= tiles   # (a tile of a group of pixels takes two to eight times the MMAs of one of pixels)


@pytest.mark.parametrize("shape,blocks", [
    # both teams of expanders stage the one tile of a CTA where words come one at a time ...
    ((16, 14, 14, 96, 20, 2, 1, 3), 2), ((9, 43, 55, 83, 48, 2, 1, 3), 2), ((4, 14, 14, 160, 300, 2, 1, 3), 3), ((2, 14, 14, 214, 24, 2, 1, 3), 2),
    # ... but not where loads are wider, or there are few of them
    ((4, 14, 14, 128, 64, 2, 1, 3), 1), ((4, 14, 14, 96, 64, 1, 1, 3), 1),
])
def test_a_single_tile_is_staged_by_both_teams(lib, shape, blocks):
    (_, _, _, _, got), = make(lib, [shape])
    assert got == blocks


@pytest.mark.parametrize("c_out", [1, 8, 16, 17, 31, 32, 33, 48, 64, 65, 96, 128, 129, 160, 300])
@pytest.mark.parametrize("lg", [0, 1, 2, 3])
@pytest.mark.parametrize("np_", [16, 32, 48, 112, 160, 240])
def test_the_warps_that_write_share_the_columns(lib, c_out, lg, np_):
    """Every (channel, 32-column slice) is written by exactly one warp and lane; with few channels and single pixels by as many
    warps as there are slices; and a chain's counters expect the warps that do write."""
    rows = ctypes.c_int(0)
    warps = lib.plan_tile(_array((4, 20, 20, 32, c_out, 1, 1, 3)), 0, WORDS, lg, np_, ctypes.byref(rows))
    if not warps:
        return   # no such tile
    rows, slices = rows.value, (np_ + 31) // 32
    written, writing = {}, 0
    for co in range(0, c_out, 128):
        for warp in range(8):   # the kernel's epilogue: lane quarter warp % 4, half warp // 4
            first = 32 * (warp % 4)
            copy = 0 if lg else first // rows
            mine = range(warp // 4 + 2 * copy, slices, 2 if lg else 2 * (128 // rows))
            if co + first % rows >= c_out or not mine:
                continue
            writing += 1
            for row in range(first, first + 32):
                pixel, channel = (row // rows if lg else 0), co + row % rows
                for s in mine if channel < c_out else ():
                    written[pixel, channel, s] = written.get((pixel, channel, s), 0) + 1
    assert writing == warps
    assert written == {(g, c, s): 1 for g in range(1 << lg) for c in range(c_out) for s in range(slices)}
    if lg == 0 and c_out <= 32:
        assert warps == min(8, slices)


@pytest.mark.parametrize("c_in,c_out,copies", [(16, 16, True), (16, 64, True), (32, 32, True), (64, 64, False), (512, 16, False), (512, 32, False)])
def test_copies_only_where_the_stores_take_longer_than_the_mmas(lib, c_in, c_out, copies):
    rows = ctypes.c_int(0)
    assert lib.plan_tile(_array((64, 32, 32, c_in, c_out, 1, 1, 3)), 1, WORDS, 0, 256, ctypes.byref(rows))
    assert (rows.value < 128) == copies


def test_division_by_run_time_constants_is_exact_below_2_to_the_31(lib):
    lib.plan_divide.restype = ctypes.c_uint32
    rng = random.Random(9)
    top = (1 << 31) - 1
    for d in [*range(1, 130), *(1 << k for k in range(31)), *((1 << k) - 1 for k in range(2, 32)), *(rng.randint(1, top) for _ in range(200))]:
        last = top // d * d   # the largest multiple: the quotient changes there
        for q in (0, 1, d - 1, d, min(2 * d - 1, top), last - 1 if last else 0, last, top, *(rng.randint(0, top) for _ in range(20))):
            assert lib.plan_divide(q, d) == q // d, (q, d)


@pytest.mark.parametrize("ctas", [1, 2, 3, 7, 64, 100, 147, 148, 160])
def test_launches_of_a_chain_are_counted_whole(lib, ctas):
    """The upper half of the count is the same for every CTA of a launch, and right again after launches that overlapped."""
    lib.plan_launches.restype = ctypes.c_uint64
    rng = random.Random(ctas)

    def count(ended):
        a = np.array(ended, np.uint32)
        return lib.plan_launches(ctas, a.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32)), len(a))

    once, twice = list(range(ctas)), list(range(ctas)) * 2
    for _ in range(20):
        rng.shuffle(once)
        rng.shuffle(twice)   # two launches whose CTAs end in any order
        assert [count(once[:k]) >> 32 for k in range(ctas)] == [0] * ctas   # a CTA that starts late takes the same tag
        assert count(once) == 1 << 32 and count(twice) == 2 << 32


def test_every_cta_finds_its_next_tile(lib):
    """Tiles are dealt once each, and a CTA is told the next problem in which it has one, whatever it passes by."""
    rng = random.Random(12)
    for tiles in [[1], [1, 1, 1], [148] * 3, [414, 1, 1, 1, 1, 109, 1, 1, 1], [267, 135, 106, 88, 28, 28, 112, 28],
                  *([rng.choice((1, 2, 5, 30, 147, 148, 149, 400)) for _ in range(rng.randint(1, 32))] for _ in range(40))]:
        grid = min(SMS, sum(tiles))
        ranks = np.zeros((len(tiles), grid), np.uint32)
        lib.plan_assign(_array(tiles), len(tiles), grid, ranks.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32)))
        assert (np.sort(ranks & 0xffff, axis=1) == np.arange(grid)).all()
        has = (ranks & 0xffff) < np.array(tiles)[:, None]
        for i in range(len(tiles)):
            for b in range(grid):
                assert ranks[i, b] >> 16 == next((k for k in range(i + 1, len(tiles)) if has[k, b]), len(tiles))


def _words(shapes, n):
    return max((n * s.h_out * s.w_out * ((s.c_out + 31) // 32) for s in shapes[:-1]), default=0)


def test_which_chains_of_the_gpu_tests_carry_tags(lib):
    """The stacks that are compared on the GPU stand on the sides of the rule that they are meant to."""
    import test_gpu_stack as gpu
    import workloads as wl
    lib.plan_tagged.argtypes = [ctypes.c_uint64]
    assert lib.plan_tagged(0) and lib.plan_tagged(1 << 17) and not lib.plan_tagged((1 << 17) + 1)
    for chain in gpu.CHAINS:
        shapes = gpu.chain_shapes(*chain[:6])
        assert lib.plan_tagged(_words(shapes, chain[6])), chain
        assert chain[7] is None or not lib.plan_tagged(_words(shapes, chain[7])), chain
    pair = [wl.LayerShape(16, 16, 32, 32, 1, 1)] * 2
    assert _words(pair, 128) == 1 << 17 and not lib.plan_tagged(_words(pair, 129))
    for net, n, tags in (("resnet18", 2, True), ("resnet18", 64, False), ("resnet20", 4, True)):
        assert bool(lib.plan_tagged(_words(wl.get_workload(net).layers, n))) == tags


GIVEN, HEAVY_FIRST, IN_TURN = 0, 1, 2


def group_order(lib, shapes, f16=False, kind=WORDS, by=-1):
    """(which order, the problems in it, cycles of a tile's MMAs, cycles of its stores)"""
    order, mma, drain = (ctypes.c_int * 32)(), (ctypes.c_double * 32)(), (ctypes.c_double * 32)()
    by = lib.plan_order(_array(shapes), len(shapes), int(f16), kind, SMS, by, order, mma, drain)
    assert by >= 0
    return by, order[:len(shapes)], mma[:len(shapes)], drain[:len(shapes)]


@pytest.mark.parametrize("f16", [False, True])
def test_heavy_problems_of_a_group_come_first(lib, f16):
    """The order is a permutation by the tiles' MMAs, and keeps the order given among problems whose tiles are small or alike."""
    rng = random.Random(11)
    for _ in range(60):
        shapes = [s for s in (draw(rng) for _ in range(rng.randint(1, 32))) if takes(lib, s, f16)]
        if not shapes:
            continue
        shapes += shapes[:32 - len(shapes)]
        _, order, cycles, _ = group_order(lib, shapes, f16, by=HEAVY_FIRST)
        assert sorted(order) == list(range(len(shapes)))
        assert order == sorted(order, key=lambda i: (-max(cycles[i], 1200.0), i))


def test_problems_bound_by_their_stores_come_in_turn_with_the_others(lib):
    rng = random.Random(12)
    for count in (1, 2, 3, 7, 32):
        shapes = []
        while len(shapes) < count:
            shapes += [s for s in (draw(rng),) if takes(lib, s, False)]
        _, order, mma, drain = group_order(lib, shapes, by=IN_TURN)
        assert sorted(order) == list(range(count))
        bound = [drain[i] / mma[i] for i in order]
        most, least = bound[::2], bound[1::2]
        assert most == sorted(most, reverse=True) and least == sorted(least) and (not least or min(most) >= max(least))


@pytest.mark.parametrize("net,n,f16,kind,by", [
    ("resnet18", 64, False, WORDS, GIVEN), ("resnet18", 32, False, WORDS, HEAVY_FIRST), ("resnet34", 64, False, WORDS, GIVEN),
    ("resnet18", 64, True, WORDS, GIVEN), ("resnet20", 128, False, WORDS, HEAVY_FIRST),
    # stores take most of the time: large groups and small ones, but one image, fp16 activations and packed signs
    ("resnet50_1x1", 64, False, WORDS, IN_TURN), ("resnet50_1x1", 8, False, WORDS, IN_TURN), ("resnet50_1x1", 1, False, WORDS, HEAVY_FIRST),
    ("resnet50_1x1", 64, True, WORDS, GIVEN), ("resnet50_1x1", 64, False, SIGNS, HEAVY_FIRST)])
def test_the_order_of_the_networks_groups(lib, net, n, f16, kind, by):
    import workloads as wl
    shapes = [(n, s.h, s.w, s.c_in, s.c_out, s.stride, s.pad, s.ksize) for s in getattr(wl, net + "_layers")()]
    got, order, *_ = group_order(lib, shapes, f16, kind)
    assert got == by and (by != GIVEN or order == sorted(order))


@pytest.mark.parametrize("net,n,kind,streams", [("resnet50_1x1", 64, WORDS, True), ("resnet50_1x1", 9, WORDS, True), ("resnet50_1x1", 8, WORDS, False),
                                                ("resnet50_1x1", 64, SIGNS, False), ("resnet18", 64, WORDS, False), ("resnet34", 64, WORDS, False)])
def test_which_outputs_leave_the_l2_first(lib, net, n, kind, streams):
    """More than twice what it holds, where the stores take most of the time."""
    import workloads as wl
    shapes = [(n, s.h, s.w, s.c_in, s.c_out, s.stride, s.pad, s.ksize) for s in getattr(wl, net + "_layers")()]
    assert lib.plan_streams(_array(shapes), len(shapes), 0, kind, SMS) == streams


def test_the_large_group_of_the_gpu_tests_leaves_the_l2_first(lib):
    shapes = [(22, 56, 57, 64, 250, 1, 0, 1)] * 2 + [(3, 7, 7, 2048, 33, 1, 0, 1), (22, 113, 113, 72, 250, 2, 0, 1), (31, 29, 57, 40, 333, 1, 0, 1)]
    assert lib.plan_streams(_array(shapes), len(shapes), 0, WORDS, SMS) == 1


@pytest.mark.parametrize("c_in", [32, 64, 72, 512])
@pytest.mark.parametrize("c_out", [33, 48, 64])
@pytest.mark.parametrize("n,h,w,pad", [(1, 5, 5, 1), (3, 15, 15, 0), (2, 9, 31, 1), (8, 56, 56, 1)])
def test_pairs_of_kernel_columns_make_every_product_once(lib, c_in, c_out, n, h, w, pad):
    """Rows and steps of the weight operand, as the kernel lays them out and the epilogue adds them up: each (channel, kernel row, kernel
    column) of an output has the weight one in all, on its own position; a tile's position more is the next tile's first."""
    rows = np.zeros((6 * 128, 5), np.int32)
    shape = _array((n, h, w, c_in, c_out, 1, pad, 3))
    assert lib.plan_pair_products(shape, rows.ctypes.data_as(ctypes.POINTER(ctypes.c_int))) == len(rows)
    tiles = (ctypes.c_int * 5)()
    lib.plan_pair_tiles(shape, tiles)
    positions, own, multiplied, count, pitch = tiles
    halves = {}
    for channel, ky, kx, at, weight in rows.tolist():
        assert at == ky * pitch + kx
        halves[channel, ky, kx] = halves.get((channel, ky, kx), 0) + weight
    assert halves == {(c, ky, kx): 2 for c in range(64) for ky in range(3) for kx in range(3)}
    assert own == multiplied - 1 and (count - 1) * own < positions <= count * own


@pytest.mark.parametrize("c_in,c_out,stride,ksize", [(64, 32, 1, 3), (64, 65, 1, 3), (64, 64, 2, 3), (64, 64, 1, 1), (36, 64, 1, 3), (24, 64, 1, 3)])
def test_other_layers_hold_no_pairs(lib, c_in, c_out, stride, ksize):
    rows = np.zeros((6 * 128, 5), np.int32)
    assert not lib.plan_pair_products(_array((2, 20, 20, c_in, c_out, stride, 0, ksize)), rows.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))


@pytest.mark.parametrize("threshold", [0.0, 1.0, -1.0, 4608.0, float("inf")])
@pytest.mark.parametrize("value", [0.0, -0.0, 1.0, -1.0, 2.0, 4608.0, -4608.0])
def test_a_sum_at_its_threshold_has_the_bit_whatever_its_zero(lib, value, threshold):
    lib.plan_sign.argtypes = [ctypes.c_float, ctypes.c_float, ctypes.c_int]
    assert lib.plan_sign(value, threshold, 0) == (value >= threshold)
    assert lib.plan_sign(value, threshold, 1) == (value < threshold)
