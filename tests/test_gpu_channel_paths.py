"""The grouped kernel's channel paths at the sizes where their bookkeeping can go wrong (needs a B200):
1x1 rows around every group size and vector remainder, kernels of every specialised size around the
group sizes, rows that start anywhere, all output forms, many flips and massive ties (the selection's
exact search).  Whole numbers and raw float words must equal the checker's."""
import time

import numpy as np
import pytest
import torch

import oracle
import paper_2202_07471_b200 as sq
from paper_2202_07471_b200 import workloads as W

from cases import adversarial_layer, coarse

pytestmark = pytest.mark.gpu

ROWS = (1, 2, 3, 5, 31, 32, 33, 252, 253, 256, 257, 509, 512, 1021, 1024, 1025, 2045, 2048, 4093, 4096, 8181, 8188, 8192)
KERNELS = (1, 2, 3, 31, 33, 127, 128, 129, 256, 257, 511, 512, 513, 1025)


def layers(shape, seed):
    """Special channels; one-signed values (hundreds of flips per channel); a coarse grid (ties)."""
    out = [adversarial_layer(shape, seed)]
    if shape[1] >= 100:
        out += [np.abs(W.random_layer((3,) + shape[1:], seed)), coarse(W.random_layer((3,) + shape[1:], seed), steps=24, div=4)]
    return out


def check(ws, bits, mode=sq.MODE_EKC, flags=sq.FLAG_NARROW_RANGE, start=0, outputs=False, clip=None, sums=True):
    pack = bool(flags & sq.FLAG_PACK_INT4)
    bufs, scales = [], []
    for i, w in enumerate(ws):
        t = torch.zeros(w.size + 4, device="cuda")[start:start + w.size].view(w.shape)
        t.copy_(torch.from_numpy(w))
        b = sq.alloc_outputs(t, pack_int4=pack, dequant=outputs, dequant_bf16=outputs, kernel_err=sums, channel_err=sums)
        b.codes.fill_(-128)
        if sums:
            b.kernel_err.fill_(float("nan"))
        sc = None
        if clip:
            a = np.abs(w).reshape(w.shape[0], -1).max(1)
            sc = (np.where(a > 0, a, 1) * clip / (2 ** (bits - 1) - 1)).astype(np.float32)
            b.scales_in = torch.from_numpy(sc).cuda()
        scales.append(sc)
        bufs.append(b)
    sq.squant_quantize_model(bufs, bits=bits, mode=mode, flags=flags)
    sq.squant_device_status()
    for b, w, sc in zip(bufs, ws, scales):
        r = oracle.quantize_layer(w, bits=bits, mode=mode, flags=flags, details=True, scales_in=sc)
        pairs = [(b.codes, r.codes), (b.scales, r.scales)]
        if sums:
            pairs += [(b.kernel_err, r.kernel_err), (b.channel_err, r.channel_err)]
        if outputs:
            pairs += [(b.dequant, r.dequant), (b.dequant_bf16.view(torch.int16), r.dequant_bf16.view(np.int16))]
        for k, (got, want) in enumerate(pairs):
            got = got.cpu().numpy()
            assert np.array_equal(got.view(np.uint8), np.ascontiguousarray(want).view(np.uint8)), (w.shape, bits, mode, flags, start, clip, k)


def shapes(kind):
    if kind == "rows":
        return [(5 if n > 1000 else 37, n, 1, 1) for n in ROWS]
    return [(5 if n > 200 else 19, n) + k for k in ((3, 3), (1, 7), (3, 1), (2, 2), (5, 5)) for n in KERNELS if n * k[0] * k[1] <= 14000]


@pytest.mark.parametrize("kind", ["rows", "kernels"])
@pytest.mark.parametrize("bits,mode,flags", [(4, 7, 1), (8, 7, 0), (2, 7, 1), (4, 3, 1), (4, 1, 0)])
def test_channel_paths(kind, bits, mode, flags):
    ws = [w for i, s in enumerate(shapes(kind)) for w in layers(s, 40 * bits + i)]
    check(ws, bits, mode, flags)
    check(ws, bits, mode, flags, start=1, outputs=True)
    if bits <= 4:
        check(ws, bits, mode, flags | sq.FLAG_PACK_INT4, start=3)
    check(ws, bits, mode, flags, start=2, clip=0.6)
    check(ws, bits, mode, flags, outputs=True, clip=0.9)


@pytest.mark.parametrize("shape", [(3, 1254, 17, 17), (3, 897, 20, 20), (2, 11, 120, 120), (2, 16, 1, 20000), (2, 3, 150, 150)])
def test_cluster_runs_of_an_even_number_of_kernels(shape):
    """Channels of few large kernels whose thread blocks take a number of kernels that is no multiple of four."""
    assert sq.squant_plan_kernels([shape]) == ["cluster"]
    w = [adversarial_layer(shape, seed=shape[1])]
    check(w, 4)
    check(w, 4, mode=sq.MODE_E | sq.MODE_K, start=1, outputs=True)
    check(w, 3, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=2, outputs=True)
    check(w, 8, flags=0, clip=0.98)


@pytest.mark.parametrize("shape", [(4096, 250, 1, 1), (2048, 512, 1, 1), (1024, 1024, 1, 1), (300, 2048, 1, 1)])
def test_rows_with_full_lists(shape):
    """So many rows of normal weights that some have more candidates above the bound than their list holds: groups
    that share a warp, of one warp and of two."""
    w = W.random_layer(shape, seed=shape[1])
    check([w, np.sign(w) * np.abs(w) ** np.float32(1.5)], 4)
    check([w], 8, flags=0, start=1)
    check([w], 4, start=2, clip=0.9)


@pytest.mark.parametrize("n", [64, 175, 176, 177, 255, 258, 513, 1030, 4100])
def test_rows_whose_list_starts_at_a_guess(n):
    """SQuant-C of rows from 176 weights on lists from a guessed bound first: rows for which the guess is good, too high
    (two bits and outliers: few candidates come near one half) and too low (one-signed weights, ties: a full list)."""
    shape = (400 if n < 1000 else 100, n, 1, 1)
    w = W.random_layer(shape, seed=n)
    ws = [w, np.where(W.random_layer(shape, seed=n + 1) > 2.0 * w.std(), 8 * w, w)] + layers((5,) + shape[1:], n)
    for bits in (2, 4, 8):
        check(ws, bits, start=bits % 3)


@pytest.mark.parametrize("n", [180, 256, 512, 1024, 2048, 4096])
def test_rows_of_every_number_of_flips(n):
    """A row for each number of flips up to a quarter of its weights: first lists with and without room, searches among
    too few maxima, exact searches from the bound of a list that was full; spread and coarse values, other rows between them."""
    flips = np.arange(n // 4)
    rng = np.random.default_rng(n)
    x = rng.integers(-6, 7, (2 * flips.size, n)) + np.where(rng.random((2 * flips.size, n)) < 0.5, 0, rng.uniform(-0.49, 0.49, (2 * flips.size, n)))
    x[::2] = rng.integers(-6, 7, (flips.size, n))
    for k in flips:   # the first elements add up to about k
        up = rng.uniform(0.3, 0.49, n)
        x[2 * k, :] += np.where((np.cumsum(up) < k) if k % 3 else (np.arange(n) < k / 0.4), up if k % 3 else 0.4, 0.0)
    x[:, 0] = 7
    w = x.astype(np.float32)[..., None, None] / np.float32(7)
    check([w, -w], 4)
    check([w], 4, start=1, clip=0.99)
    check([w], 4, clip=0.6)


@pytest.mark.parametrize("rows,n", [(1, 25001), (3, 24004), (3, 100352), (2, 65541)])
def test_long_rows_whose_list_starts_at_a_guess(rows, n):
    """Long and wide rows: a guess from the number of elements seen near one half, too few of them (two bits and outliers),
    one-signed weights and ties."""
    if rows == 1:   # enough of them for the long form
        rows = torch.cuda.get_device_properties(0).multi_processor_count + 1
    shape = (rows, n, 1, 1)
    w = W.random_layer(shape, seed=n)
    ws = [w, np.where(W.random_layer(shape, seed=n + 1) > 2.0 * w.std(), 8 * w, w)] + layers((3,) + shape[1:], n)
    for bits in (2, 4, 8):
        check(ws, bits, start=bits % 3)


@pytest.mark.parametrize("bits,clip", [(2, 0.97), (4, 0.7), (8, 0.5), (3, 0.2), (8, 0.1), (6, 0.04)])
def test_elements_at_and_far_beyond_the_clip_range(bits, clip):
    """Scales of the caller's from just below absmax (elements on the last code) to far below (sums of many whole codes, kernels
    whose every candidate is flipped), rows in groups of every kind and 3x3 kernels; with absmax layers in the same call too."""
    ws = [w for i, s in enumerate([(37, 100, 1, 1), (20, 300, 1, 1), (9, 701, 1, 1), (5, 3000, 1, 1), (19, 33, 3, 3), (5, 513, 3, 3)]) for w in layers(s, 7 * bits + i)]
    check(ws, bits, clip=clip)
    check(ws, bits, flags=0, start=1, outputs=True, clip=clip)
    bufs = []
    for i, w in enumerate(ws):
        b = sq.alloc_outputs(torch.from_numpy(w).cuda())
        if i % 2:
            a = np.abs(w).reshape(w.shape[0], -1).max(1)
            b.scales_in = torch.from_numpy((np.where(a > 0, a, 1) * clip / (2 ** (bits - 1) - 1)).astype(np.float32)).cuda()
        bufs.append(b)
    sq.squant_quantize_model(bufs, bits=bits)
    for b, w in zip(bufs, ws):
        r = oracle.quantize_layer(w, bits=bits, scales_in=None if b.scales_in is None else b.scales_in.cpu().numpy(), details=True)
        assert np.array_equal(b.codes.cpu().numpy(), r.codes) and np.array_equal(b.kernel_err.cpu().numpy().view(np.int32), r.kernel_err.view(np.int32))


@pytest.mark.parametrize("shape", [(2, 1, 1, 45857), (3, 2, 1, 22928), (2, 9, 1, 5095), (2, 200, 1, 229), (5, 106, 7, 7), (9, 52, 7, 7), (9, 103, 5, 5)])
def test_larger_kernels_at_the_sizes_that_share_a_thread_block(shape):
    """The longest channels of few large kernels that one thread block, or two and four channels that share one, hold;
    in the table variant too."""
    assert sq.squant_plan_kernels([shape]) == ["grouped"]
    w = [adversarial_layer(shape, seed=shape[1])]
    check(w, 4)
    check(w, 8, flags=0, start=1, outputs=True)
    check(w, 4, mode=sq.MODE_E | sq.MODE_K, start=3, clip=0.8)
    b = sq.alloc_outputs(torch.from_numpy(w[0]).cuda())
    sq.squant_quantize_layer_noalloc(b, bits=4)
    sq.squant_device_status()
    r = oracle.quantize_layer(w[0], bits=4)
    assert np.array_equal(b.codes.cpu().numpy(), r.codes)
    assert np.array_equal(b.kernel_err.cpu().numpy().view(np.uint32), r.kernel_err.view(np.uint32))


@pytest.mark.parametrize("n", [1184, 1188, 1412, 2048])
def test_long_channels_with_packed_and_dequantized_outputs(n):
    """Long 3x3 channels with further outputs: one, two, three and many channels per persistent thread block
    (the outputs follow three steps behind), partial last warps, rows that start on two-byte boundaries."""
    for m in (1, 149, 297, 450, 700):
        w = [adversarial_layer((m, n, 3, 3), seed=m + n)]
        check(w, 4, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, outputs=m < 400)
        check(w, 6, outputs=True)


@pytest.mark.parametrize("n", [1188, 1500, 2044])
def test_no_lane_overtakes_the_further_outputs(n):
    """The further outputs of a long channel are written by whole warps from codes that other lanes own and
    overwrite in the next step.  The checked build sees a lane that begins the next step while another is still
    reading (trip counts that differ by lane: 144 packed words over 32 lanes, the row's tail); many steps per
    thread block, and the outputs must be right in either build."""
    from paper_2202_07471_b200 import build as lib_build
    ws = [adversarial_layer((1200, n, 3, 3), seed=n)]
    flags = sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4
    check(ws, 4, flags=flags)
    sq.use_library(lib_build.LIB_DEBUG)
    try:
        sq.squant_debug_violations()
        check(ws, 4, flags=flags)
        check([w[:400] for w in ws], 4, flags=flags, outputs=True)
        check([w[:400] for w in ws], 5, outputs=True)
        checked, failed, site = sq.squant_debug_violations()
        assert checked and failed == 0, (failed, site)
    finally:
        sq.use_library(None)


def test_checked_build_takes_every_error_sum_a_second_time():
    """Groups of 8 threads to a thread block, the row kernel, kernels of every body; each channel once."""
    from paper_2202_07471_b200 import build as lib_build
    shapes = [(37, 64, 3, 3), (33, 5, 1, 1), (9, 300, 1, 1), (5, 4097, 1, 1), (3, 9001, 1, 1), (4, 3, 5, 5), (6, 70, 1, 7), (11, 9, 3, 1), (3, 1100, 3, 3)]
    ws = [adversarial_layer(s, seed=s[1]) for s in shapes]
    sq.use_library(lib_build.LIB_DEBUG)
    try:
        sq.squant_debug_violations()
        sq.squant_debug_sums_checked()
        for bits, mode in ((4, sq.MODE_EKC), (8, sq.MODE_EKC), (3, sq.MODE_E | sq.MODE_K)):
            check(ws, bits, mode, start=bits & 3)
            assert sq.squant_debug_sums_checked() == sum(s[0] for s in shapes)
            checked, failed, site = sq.squant_debug_violations()
            assert checked and failed == 0, (failed, site)
    finally:
        sq.use_library(None)
    assert sq.squant_debug_sums_checked() == 0   # the regular build takes none


def test_long_channels_with_packed_codes_in_a_capture():
    """The first call of a plan inside a stream capture can allocate nothing: the grouped kernel takes it."""
    w = adversarial_layer((40, 1536, 3, 3), seed=5)
    b = sq.alloc_outputs(torch.from_numpy(w).cuda(), pack_int4=True)
    flags = sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sq.squant_quantize_model([b], bits=4, flags=flags)
    b.codes.fill_(-128)
    graph.replay()
    sq.squant_device_status()
    r = oracle.quantize_layer(w, bits=4, flags=flags)
    assert np.array_equal(b.codes.cpu().numpy(), r.codes)
    assert np.array_equal(b.kernel_err.cpu().numpy().view(np.uint32), r.kernel_err.view(np.uint32))


def test_scratch_of_a_captured_call_lives_as_long_as_the_graph():
    """A graph keeps the scratch memory its streaming launch points to after the plan has left the cache."""
    area = 70 << 10   # bytes per multiprocessor; 72 KB are allocated
    area *= torch.cuda.get_device_properties(0).multi_processor_count
    w = adversarial_layer((40, 1536, 3, 3), seed=6)
    b = sq.alloc_outputs(torch.from_numpy(w).cuda(), pack_int4=True)
    flags = sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4
    small = [sq.alloc_outputs(torch.randn(1, 3, device="cuda")) for _ in range(66)]
    again = sq.alloc_outputs(torch.from_numpy(w).cuda(), pack_int4=True)

    def evict():   # the cache holds 64 plans; the last call is one that can free
        for s in small:
            sq.squant_quantize_model([s], bits=4)

    evict()
    sq.squant_quantize_model([again], bits=4, flags=flags)   # its own area, and what earlier tests left is freed
    call = sq.ModelCall([b], bits=4, flags=flags)
    call.run()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call.run()
    sq.squant_quantize_model([again], bits=4, flags=flags)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for s in small[:62]:
        sq.squant_quantize_model([s], bits=4)
    sq.squant_quantize_model([again], bits=4, flags=flags)   # most recent: stays
    for s in small[62:]:
        sq.squant_quantize_model([s], bits=4)                # the captured plan has left by now
    sq.squant_quantize_model([again], bits=4, flags=flags)
    assert torch.cuda.mem_get_info()[0] < free0 + area       # (checked before the replay)
    b.codes.fill_(-128)
    graph.replay()
    sq.squant_device_status()
    r = oracle.quantize_layer(w, bits=4, flags=flags)
    assert np.array_equal(b.codes.cpu().numpy(), r.codes)
    assert np.array_equal(b.kernel_err.cpu().numpy().view(np.uint32), r.kernel_err.view(np.uint32))
    free1 = torch.cuda.mem_get_info()[0]
    del graph
    torch.cuda.synchronize()
    for _ in range(200):   # the graph's resources go in a callback of the driver
        sq.squant_quantize_model([again], bits=4, flags=flags)
        if torch.cuda.mem_get_info()[0] >= free1 + area:
            break
        time.sleep(0.01)
    assert torch.cuda.mem_get_info()[0] >= free1 + area


def test_a_captured_call_keeps_its_work_counter():
    """A graph of a streaming launch and a call whose plan was made a thousand plans later overlap on the GPU:
    each draws its channels from a counter of its own, so none is left out."""
    shape = (700, 1536, 3, 3)
    w = W.random_layer(shape, seed=15)
    r = oracle.quantize_layer(w, bits=4)
    t = torch.from_numpy(w).cuda()
    a, *later = [sq.alloc_outputs(t.clone()) for _ in range(4)]
    assert sq.squant_plan_kernels([a]) == ["stream"]
    call = sq.ModelCall([a], bits=4)
    call.run()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call.run()
    small = sq.alloc_outputs(torch.randn(1, 1184, 3, 3, device="cuda"))
    base = torch.randn(10656 + 4 * 1024, device="cuda")
    for i in range(1023):   # further plans: the same outputs, other weights
        small.w = base[4 * i:4 * i + 10656].view(1, 1184, 3, 3)
        sq.squant_quantize_model([small], bits=4)
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    for b in later * 2:
        for x in (a, b):
            x.codes.fill_(-128)
            x.kernel_err.fill_(float("nan"))
        torch.cuda.synchronize()
        for _ in range(3):
            graph.replay()
            sq.squant_quantize_model([b], bits=4, stream=other)
        sq.squant_device_status()
        for x in (a, b):
            assert np.array_equal(x.codes.cpu().numpy(), r.codes)
            assert np.array_equal(x.kernel_err.cpu().numpy().view(np.uint32), r.kernel_err.view(np.uint32))
            assert np.array_equal(x.channel_err.cpu().numpy().view(np.uint32), r.channel_err.view(np.uint32))


def free_memory():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_scratch_is_given_back():
    """The streaming kernel's scratch memory (72 KB per multiprocessor) goes with its plan: at squant_shutdown, and
    when the plan leaves the cache although no further streaming call follows."""
    area = (70 << 10) * torch.cuda.get_device_properties(0).multi_processor_count
    long_call = sq.ModelCall([sq.alloc_outputs(torch.randn(3, 1536, 3, 3, device="cuda"))])
    small = [sq.ModelCall([sq.alloc_outputs(torch.randn(1, 3, device="cuda"))]) for _ in range(65)]
    for call in [long_call] + small:   # loads what there is to load
        call.run()
    for again in range(2):
        sq.squant_shutdown()
        free0 = free_memory()
        long_call.run()
        assert free_memory() <= free0 - area
        if again:
            for call in small:         # the cache holds 64 plans
                call.run()
        else:
            sq.squant_shutdown()
        assert free_memory() >= free0


def test_scratch_of_a_graph_survives_shutdown_and_goes_after_it():
    area = (70 << 10) * torch.cuda.get_device_properties(0).multi_processor_count
    w = adversarial_layer((40, 1536, 3, 3), seed=8)
    b = sq.alloc_outputs(torch.from_numpy(w).cuda())
    call = sq.ModelCall([b])
    small = sq.ModelCall([sq.alloc_outputs(torch.randn(1, 3, device="cuda"))])
    call.run()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call.run()
    sq.squant_shutdown()
    small.run()
    b.codes.fill_(-128)
    graph.replay()
    sq.squant_device_status()
    assert np.array_equal(b.codes.cpu().numpy(), oracle.quantize_layer(w, bits=4).codes)
    free0 = free_memory()
    del graph
    for _ in range(200):   # the graph's resources go in a callback of the driver
        small.run()        # not a streaming call
        if free_memory() >= free0 + area:
            break
        time.sleep(0.01)
    assert free_memory() >= free0 + area


def test_freeing_scratch_leaves_captures_of_other_streams_alone():
    """A call that frees scratch memory of an evicted plan, on a stream that is not captured, while another stream is."""
    long_call = sq.ModelCall([sq.alloc_outputs(torch.randn(3, 1536, 3, 3, device="cuda"))])
    small = [sq.ModelCall([sq.alloc_outputs(torch.randn(1, 3, device="cuda"))]) for _ in range(66)]
    w = W.random_layer((8, 64, 3, 3), seed=9)
    b = sq.alloc_outputs(torch.from_numpy(w).cuda())
    captured = sq.ModelCall([b])
    side = torch.cuda.Stream()
    for call in small:
        call.run()
    long_call.run()
    captured.run()
    free0 = free_memory()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured.run()
        for call in small:   # the plan of long_call leaves the cache
            call.run(side)
    assert free_memory() > free0
    b.codes.fill_(-128)
    graph.replay()
    sq.squant_device_status()
    assert np.array_equal(b.codes.cpu().numpy(), oracle.quantize_layer(w, bits=4).codes)


@pytest.mark.parametrize("n", [8193, 8196, 12290, 16384, 16387, 32767])
def test_long_rows(n):
    """1x1 rows of the row kernel: both of its sizes, lengths around their limits, rows that start anywhere, hundreds
    of flips and massive ties (full lists, the exact search), every output form."""
    assert sq.squant_plan_kernels([(3, n, 1, 1)]) == ["row"]
    ws = layers((3, n, 1, 1), n)
    check(ws + ([adversarial_layer((600, n, 1, 1), seed=1)] if n <= 16384 else []), 4)   # more than one wave: the smaller thread blocks
    check(ws, 8, flags=0, start=1, outputs=True)
    check(ws, 3, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=2)
    check(ws, 4, mode=sq.MODE_E, outputs=True)
    check(ws, 4, start=3, clip=0.7)
    check(ws[:1], 2, flags=0, outputs=True, clip=0.98)


def test_wide_rows_without_supplied_scales():
    """Rows of a cluster on either side of 2^16 elements, from where a flip can be barred without a supplied scale too:
    every alignment and output form, hundreds of flips."""
    shapes = [(2, 100353, 1, 1), (3, 65541, 1, 1), (1, 65536, 1, 1), (2, 50000, 1, 1)]
    assert set(sq.squant_plan_kernels(shapes)) == {"cluster"}
    ws = [adversarial_layer(s, seed=i) for i, s in enumerate(shapes)] + [np.abs(W.random_layer((1, 70001, 1, 1), 9))]
    check(ws, 4, start=1)
    check(ws, 8, flags=0, outputs=True)
    check(ws, 4, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=2)
    check(ws, 4, clip=0.8)


@pytest.mark.parametrize("n", [8193, 8196, 9001, 16387, 25002, 32767, 46501, 65535, 65541, 100352])
def test_long_and_wide_rows_without_sums(n):
    """Codes and scales only (rows of the row and the cluster kernel): every start of a row, packed codes, supplied
    scales; many rows and few."""
    assert sq.squant_plan_kernels([(3, n, 1, 1)]) == ["row" if n <= 32768 else "cluster"]
    ws = layers((3, n, 1, 1), n)
    m = 12 * torch.cuda.get_device_properties(0).multi_processor_count + 8
    if n < 10000:   # more rows than four waves of the smaller thread blocks, both sides of a vector's start
        check([W.random_layer((m, n, 1, 1), seed=2)], 4, sums=False, start=n & 3)
    for start in (0, 1, 2, 3):
        check(ws, 4, start=start, sums=False)
    check(ws, 8, flags=0, sums=False)
    check(ws, 4, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=1, sums=False)
    check(ws, 3, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, outputs=True, sums=False)
    check(ws, 4, clip=0.7, sums=False)


@pytest.mark.parametrize("n,form", [(8193, "256"), (10985, "256"), (10986, "256"), (13500, "256"), (14877, "256"), (14878, "512"), (16387, "512"), (22313, "512"),
                                    (22314, "long"), (25001, "long"), (26869, "long"), (26870, "512")])
def test_forms_of_long_rows(n, form):
    """Rows of the row kernel on either side of the lengths (four and three thread blocks of 256 threads on a multiprocessor;
    two of 512 only in long_row_body) and of the numbers of rows (two and a quarter a multiprocessor; one) from which they take
    another form, every output form in each.  The form shows in the number of launches of a call that has another
    layer in row_body with 512 threads."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few = 9 * sms // 4 if n < 20000 else sms
    w, other = adversarial_layer((few + 1, n, 1, 1), seed=n), adversarial_layer((1, 14900, 1, 1), seed=1)

    def launches(w, *args, **kw):
        n0 = sq.squant_launch_count()
        check([w, other], *args, **kw)
        return sq.squant_launch_count() - n0

    apart, small = (1 if form == "512" else 2), (2 if form == "256" else 1)   # long_row_body: neither packed codes nor supplied scales
    assert launches(w, 4) == apart
    assert launches(w[1:], 4) == 1
    assert launches(w, 4, sums=False, start=1) == apart
    assert launches(w, 4, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=2) == small
    if n not in (10985, 10986, 22313, 26870):
        assert launches(w, 8, flags=0, outputs=True, start=3) == apart
        if n < 15000:   # (longer rows with supplied scales go to the cluster kernel)
            assert launches(w, 4, clip=0.8) == small
        assert launches(w, 3, mode=sq.MODE_E | sq.MODE_C) == apart
        assert launches(w, 4, mode=sq.MODE_E, outputs=True) == apart


def test_call_with_every_form_of_long_rows():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes = [(sms, 14877, 1, 1), (9 * sms // 4, 8201, 1, 1), (5, 12000, 1, 1), (sms + 1, 25001, 1, 1), (7, 32768, 1, 1), (11, 17000, 1, 1), (3, 50000, 1, 1), (40, 64, 3, 3)]
    ws = [adversarial_layer(s, seed=s[1]) for s in shapes]
    n0 = sq.squant_launch_count()
    check(ws, 4, start=1)
    # 256 threads of which three and of which four thread blocks fit a multiprocessor, both forms with 512; the wide layer, the grouped launch
    assert sq.squant_launch_count() - n0 == 4 + 1 + 1


@pytest.mark.parametrize("n", [46501, 48000, 50999])
def test_wide_rows_in_clusters_of_two_and_four(n):
    """On either side of the number of rows up to which clusters of two are not taken."""
    m = 7 * torch.cuda.get_device_properties(0).multi_processor_count // 16
    w = adversarial_layer((m + 1, n, 1, 1), seed=n)
    assert sq.squant_plan_kernels([w.shape]) == ["cluster"]
    for part in (w, w[1:]):
        check([part], 4)
        check([part], 4, sums=False, start=1)
        check([part], 4, flags=sq.FLAG_NARROW_RANGE | sq.FLAG_PACK_INT4, start=3)
    check([w[:9]], 8, flags=0, outputs=True, clip=0.9)


@pytest.mark.parametrize("shapes,kernels", [([(100, 16384, 1, 1), (1, 50000, 1, 1)], ["row", "cluster"]), ([(100, 8000, 1, 1), (1, 50000, 1, 1)], ["grouped", "cluster"]),
                                            ([(100, 8000, 1, 1), (5, 9000, 1, 1), (1, 50000, 1, 1)], ["grouped", "row", "cluster"])])
def test_what_follows_a_call_follows_all_of_its_launches(shapes, kernels):
    """The first launch (every row flips thousands of weights that tie) outlasts those that may start before it ends.  Its
    outputs are copied, its weights overwritten and the call made again on the same stream, with no synchronization."""
    assert sq.squant_plan_kernels(shapes) == kernels
    ws = [((np.arange(np.prod(s)) % 7 - 3 + 0.4) / 7).astype(np.float32).reshape(s) if i == 0 else W.random_layer(s, seed=i) for i, s in enumerate(shapes)]
    ws[0][:, 0] = 1.0   # scales of 1/7
    refs = [oracle.quantize_layer(w, bits=4) for w in ws]
    weights = [torch.from_numpy(w).cuda() for w in ws]
    bufs = [sq.alloc_outputs(w.clone()) for w in weights]
    call = sq.ModelCall(bufs)

    def time_of(c):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        start.record()
        for _ in range(10):
            c.run()
        end.record()
        end.synchronize()
        return start.elapsed_time(end)

    call.run()
    first, rest = sq.ModelCall(bufs[:1]), sq.ModelCall(bufs[1:])
    time_of(first), time_of(rest)
    assert time_of(first) > 1.5 * time_of(rest)
    seen = []
    for _ in range(10):
        for b, w in zip(bufs, weights):
            b.w.copy_(w)
            b.codes.fill_(-128)
        call.run()
        got = [(b.codes.clone(), b.kernel_err.clone(), b.channel_err.clone()) for b in bufs]
        for b in bufs:
            b.w.fill_(0.0)
        call.run()
        seen.append((got, [b.codes.clone() for b in bufs]))
    torch.cuda.synchronize()
    for got, again in seen:
        for g, a, r in zip(got, again, refs):
            for x, want in zip(g, (r.codes, r.kernel_err, r.channel_err)):
                assert np.array_equal(x.cpu().numpy().view(np.uint8), np.ascontiguousarray(want).view(np.uint8))
            assert not a.any()
