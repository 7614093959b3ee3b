"""Host-side checks that need no GPU: the library loads, exports what include/squant.h declares,
validates arguments and plans launches."""
import ctypes
import os
import re

import pytest

import paper_2202_07471_b200 as sq
from paper_2202_07471_b200 import binding, workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    lib = sq.load_library()
    header = open(os.path.join(ROOT, "include", "squant.h")).read()
    declared = set(re.findall(r"\b(squant_[a-z_]+)\s*\(", header))
    assert declared, "no declarations found"
    for name in declared:
        assert hasattr(lib, name), f"{name} is declared in squant.h but not exported"
    assert declared == set(binding.EXPORTS)


def test_strerror_covers_all_codes():
    lib = sq.load_library()
    texts = {lib.squant_strerror(c).decode() for c in range(0, -12, -1)}
    assert len(texts) == 12 and all(texts)
    assert "unknown" in lib.squant_strerror(-99).decode()


def _info(shapes, **kw):
    return sq.squant_plan_info(shapes, **kw)


def test_plan_geometry_for_the_five_configs():
    for name, wl in W.WORKLOADS.items():
        info = _info(wl.shapes)
        assert info["cta_threads"] == 256
        assert 0 < info["dynamic_smem_bytes"] <= 232448
        assert info["grid_ctas"] >= 1
    # one CTA per output channel for the large layers
    assert _info(W.WORKLOADS["large_layer"].shapes)["grid_ctas"] == 8 * 2048
    # small channels share a CTA: 8 warps, one channel each
    assert _info([(64, 64, 3, 3)])["grid_ctas"] == 8   # 64 channels, 8 one-warp groups per 256-thread block
    assert _info([(33, 7, 3, 3)])["grid_ctas"] == 5
    assert _info([(600, 1, 3, 3)])["grid_ctas"] == 3   # depthwise: a whole channel per thread, 256 per block


@pytest.mark.parametrize("shape,kw,code", [
    ((0, 3, 3, 3), {}, -2), ((4, -1, 3, 3), {}, -2), ((4, 3, 0, 3), {}, -2),
    ((4, 3, 3, 3), {"bits": 1}, -3), ((4, 3, 3, 3), {"bits": 9}, -3),
    ((4, 3, 3, 3), {"mode": 2}, -4), ((4, 3, 3, 3), {"mode": 8 | 1}, -4),
    ((4, 3, 3, 3), {"mode": 16 | 1}, -4), ((4, 3, 3, 3), {"flags": 16}, -4),
    ((4, 3, 3, 3), {"bits": 6, "flags": 3}, -3),
    ((4, 70000, 1, 1), {}, -6), ((4, 8000, 3, 3), {}, -6),
])
def test_invalid_arguments_are_rejected(shape, kw, code):
    with pytest.raises(sq.SquantError) as ei:
        _info([shape], **kw)
    assert ei.value.code == code


@pytest.mark.parametrize("n,k", [(13207, 65041), (13210, 65026), (13270, 64732), (262143, 3277), (16384, 52429), (16384, 65535)])
def test_sizes_beyond_32_bits_are_rejected(n, k):
    """5 B a weight of such a channel are a small number modulo 2^32."""
    for mode in (sq.MODE_EKC, sq.MODE_E | sq.MODE_C, sq.MODE_E):
        for plan in (sq.squant_plan_info, sq.squant_plan_kernels):
            with pytest.raises(sq.SquantError) as ei:
                plan([(1, n, 1, k)], mode=mode)
            assert ei.value.code == -6, (plan, mode)


def test_valid_edge_arguments():
    assert _info([], bits=4)["grid_ctas"] == 0
    assert _info([(4, 300, 1, 1)], mode=1 | 4)["grid_ctas"] >= 1      # E|C ablation mode
    assert _info([(4, 30, 3, 3)], mode=1 | 4)["grid_ctas"] >= 1
    assert _info([(1, 1, 1, 1)], bits=2)["grid_ctas"] == 1
    assert _info([(2, 4000, 3, 3)])["grid_ctas"] == 2


@pytest.mark.parametrize("shape", [(50, 1254, 17, 17), (700, 897, 20, 20), (8, 48, 1, 7600), (3, 16, 1, 20000), (4, 12, 120, 120), (3, 3, 150, 150)])
def test_channels_of_few_large_kernels_fit_a_cluster(shape):
    """Of kernels of more than one element each thread block of a cluster takes an even number, not a multiple of
    four: rounding up further would cost such a channel the shared memory of up to two kernels more."""
    assert sq.squant_plan_kernels([shape]) == ["cluster"]


@pytest.mark.parametrize("k", [1, 9, 16, 25, 49, 81, 121, 169, 225, 289, 400, 1024, 2500, 7600, 14400, 22500])
def test_limit_of_the_cluster_kernel(k):
    """A channel is taken if an eighth of its kernels, rounded up to an even number, fits one thread block at 5 B a
    weight and, of larger kernels, 10 B a kernel."""
    up = lambda v: (v + 15) // 16 * 16
    def fits(n):
        n8 = ((n + 7) // 8 + 1) // 2 * 2
        return up(4 * n8 * k) + up(n8 * k) + (2 * up(4 * n8) + up(2 * n8) if k > 1 else 0) + 2304 <= 232448
    lo, hi = 1, 262143
    while lo < hi:   # the widest channel that fits
        mid = (lo + hi + 1) // 2
        lo, hi = (mid, hi) if fits(mid) else (lo, mid - 1)
    for n in {max(lo + d, 1) for d in (-40, -17, -16, -9, -8, -7, -5, -4, -3, -2, -1, 0, 1, 2, 3, 8, 15, 16, 17, 40)}:
        if n > 262143:
            continue
        if fits(n):
            assert sq.squant_plan_kernels([(3, n, 1, k)])[0] in ("cluster", "row", "grouped"), n
        else:
            with pytest.raises(sq.SquantError) as ei:
                sq.squant_plan_kernels([(3, n, 1, k)])
            assert ei.value.code == -6, n


@pytest.mark.parametrize("n,k", [(1, 45857), (2, 22928), (3, 15285), (9, 5095), (17, 2697), (191, 240), (200, 229)])
def test_limit_of_few_large_kernels_in_one_thread_block(n, k):
    """Channels of few large kernels are taken up to these sizes: what a thread block holds at 5 B a weight beside
    3,120 B for the selection."""
    for mode in (sq.MODE_EKC, sq.MODE_E | sq.MODE_K):
        assert _info([(2, n, 1, k)], mode=mode)["grid_ctas"] == 2
        assert len(sq.squant_plan_kernels([(2, n, 1, k)], mode=mode)) == 1
    with pytest.raises(sq.SquantError) as ei:
        _info([(2, n, 1, k + 1)])
    assert ei.value.code == -6


@pytest.mark.parametrize("n,kh,kw,groups", [(106, 7, 7, 2), (108, 7, 7, 2), (212, 5, 5, 2), (13, 20, 20, 2), (18, 17, 17, 2),
                                            (52, 7, 7, 4), (103, 5, 5, 4), (109, 7, 7, 1), (213, 5, 5, 1), (54, 7, 7, 2)])
def test_channels_of_larger_kernels_that_share_a_thread_block(n, kh, kw, groups):
    """As many channels of larger kernels share a thread block as leave room for four blocks on a multiprocessor."""
    assert _info([(16, n, kh, kw)])["grid_ctas"] == 16 // groups


def test_kernel_of_a_layer():
    shapes = [(64, 64, 3, 3), (8, 8192, 1, 1), (8, 8193, 1, 1), (8, 32768, 1, 1), (8, 40000, 1, 1), (8, 70000, 1, 1),
              (8, 2048, 3, 3), (8, 2049, 3, 3), (8, 2052, 3, 3), (8, 600, 5, 5), (8, 8192, 3, 3)]
    want = ["grouped", "grouped", "row", "row", "grouped", "cluster", "stream", "grouped", "grouped", "grouped", "cluster"]
    assert sq.squant_plan_kernels(shapes) == want
    assert sq.squant_plan_kernels([(8, 2048, 3, 3)], mode=sq.MODE_E) == ["grouped"]   # without SQuant-K
    assert sq.squant_plan_kernels([]) == []


def test_null_pointers_are_rejected_before_any_cuda_call():
    lib = sq.load_library()
    layer = binding.Layer(None, 4, 3, 3, 3, None, None, None, None, None, None, None)
    opt = binding.Options(4, 7, 1)
    assert lib.squant_quantize_layer(ctypes.byref(layer), ctypes.byref(opt), None) == -1
    assert lib.squant_quantize_model(None, 2, ctypes.byref(opt), None) == -1
    assert lib.squant_quantize_model(None, 0, ctypes.byref(opt), None) == 0
    assert lib.squant_quantize_layer(None, ctypes.byref(opt), None) == -1
    layer = binding.Layer(1026, 4, 3, 3, 3, 64, 128, None, None, None, None, None)      # weights not 4-byte aligned
    assert lib.squant_quantize_layer(ctypes.byref(layer), ctypes.byref(opt), None) == -5


def test_missing_library_fails_loudly(monkeypatch):
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", os.path.join(ROOT, "no_such_dir", "libsquant.so"))
    with pytest.raises(RuntimeError, match="no CPU or PyTorch fallback"):
        binding.load_library()
