"""Host-side checks of the C ABI: the library loads without a GPU, exports every declared
symbol, and rejects bad arguments with an error code before anything is launched."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2411_07762_b200 import build
    build.build()
    from paper_2411_07762_b200 import binding
    return binding.lib


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "aser.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(aser_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    from paper_2411_07762_b200 import binding
    names = declared_symbols()
    assert len(names) >= 14
    for nm in names:
        assert getattr(lib, nm) is not None
    assert set(names) == set(binding.EXPORTED_SYMBOLS)


def test_version_and_sizes(lib):
    assert lib.aser_version() >= 1000
    assert lib.aser_repacked_bytes(128, 128) == 8192
    assert lib.aser_repacked_bytes(129, 256) == 2 * 2 * 8192     # rows padded to 128
    assert lib.aser_repacked_bytes(0, 128) == 0
    assert lib.aser_workspace_bytes(8, 4096, 4096, 64) >= 256
    assert lib.aser_workspace_bytes(8, 4096, 4100, 64) == 0      # bad K


def test_bad_arguments_are_rejected_before_launch(lib):
    OK, NULL, ALIGN, SHAPE, WORKSPACE = 0, -1, -2, -3, -4
    good = C.c_void_p(0x1000)
    odd = C.c_void_p(0x1004)
    # shape errors
    assert lib.aser_pack_w4(good, None, 128, 100, good, good, None) == SHAPE
    assert lib.aser_quant_act(good, None, good, 4, 256, 24, good, good, good, None) == SHAPE
    assert lib.aser_quant_act(good, None, good, 4, 256, 512, good, good, good, None) == SHAPE
    assert lib.aser_linear_w4a8(good, good, good, good, -1, 128, 128, good, None, good, 1 << 20, None) == SHAPE
    # empty problems are no-ops
    assert lib.aser_quant_act(None, None, None, 0, 256, 16, None, None, None, None) == OK
    assert lib.aser_pack_w4(None, None, 0, 256, None, None, None) == OK
    assert lib.aser_linear_w4a8(None, None, None, None, 0, 128, 128, None, None, None, 0, None) == OK
    # null / misaligned pointers
    assert lib.aser_pack_w4(None, None, 128, 128, good, good, None) == NULL
    assert lib.aser_pack_w4(good, None, 128, 128, odd, good, None) == ALIGN
    assert lib.aser_quant_act(good, odd, None, 4, 256, 0, good, good, None, None) == ALIGN
    assert lib.aser_quant_act(good, None, None, 4, 256, 16, good, good, good, None) == NULL
    assert lib.aser_linear_w4a8_lr(good, good, good, good, None, good, 4, 128, 128, 16, good, None,
                                   good, 1 << 20, None) == NULL
    # workspace missing or too small
    assert lib.aser_linear_w4a8(good, good, good, good, 4, 128, 128, good, None, None, 0, None) == WORKSPACE
    assert lib.aser_linear_w4a8(good, good, good, good, 4, 128, 128, good, None, good, 8, None) == WORKSPACE
    assert lib.aser_workspace_init(None, 1024, None) == WORKSPACE
    assert lib.aser_last_error() != b""
    # a fused shared-input group: layer count, N a multiple of 128, one rank within the stacked limit
    i3 = (C.c_int * 3)(256, 128, 128)
    bad_n = (C.c_int * 2)(256, 136)
    i5 = (C.c_int * 5)(128, 128, 128, 128, 128)
    cat = lambda n, N, r, ws=good, nbytes=1 << 24: lib.aser_linear_w4a8_lr_cat(
        good, good, good, good, good, good, n, N, r, 64, 256, good, ws, nbytes, None)
    assert cat(5, i5, 16) == SHAPE
    assert cat(2, bad_n, 16) == SHAPE
    assert cat(3, i3, 192) == SHAPE                 # 3 x 192 stacked rows of T
    assert cat(0, i3, 16) == SHAPE
    assert cat(3, None, 16) == SHAPE
    assert cat(3, i3, 16, None, 0) == WORKSPACE
    assert lib.aser_forward_shared_cat_workspace_bytes(3, i3, 16, 64, 256) >= lib.aser_workspace_bytes(64, 512, 256, 16)
    assert lib.aser_forward_shared_cat_workspace_bytes(2, bad_n, 16, 64, 256) == 0
    assert lib.aser_forward_shared_cat(good, None, good, 3, good, good, good, i3, 16, 64, 256, good, good, good,
                                       None, good, 1 << 24, None) == NULL      # Y missing


def test_binding_refuses_cpu_tensors(lib):
    import torch
    import paper_2411_07762_b200 as aser
    with pytest.raises(TypeError):
        aser.pack_w4(torch.zeros(128, 128, dtype=torch.float16), None)


def test_forward_host_parts(lib):
    """Whole 128-token groups dealt evenly, a short rest joined to the last part, no part below 128 tokens or below
    1.5 MiB in the smaller direction."""
    first = (C.c_int * 5)()
    for N, K in ((264, 512), (1024, 4096), (4096, 4096), (4104, 14336), (28672, 8192)):
        for M in (1, 127, 128, 255, 256, 257, 260, 384, 385, 512, 513, 640, 1024, 1030, 2047, 4096, 70001):
            parts = lib.aser_forward_host_parts(M, N, K, first)
            assert parts == lib.aser_forward_host_parts(M, N, K, None)
            assert parts == max(1, min(4, M // 128, M * 2 * min(N, K) // (3 << 19)))
            begin = list(first)[:parts + 1]
            assert begin[0] == 0 and begin[-1] == M
            if parts > 1:
                sizes = [b - a for a, b in zip(begin, begin[1:])]
                assert min(sizes) >= 128 and max(sizes) - min(sizes) < 256
                assert all(b % 128 == 0 for b in begin[:-1])
    assert lib.aser_forward_host_parts(0, 128, 128, None) == 0
    assert lib.aser_forward_host_parts(512, 128, 100, None) == 0


def test_construct_workspace_of_large_layers(lib):
    """What one way through the construction holds at a time: through the whitening factor A, E [N, K], G [K, K] and
    the tokens, or the matrix [N, K + tokens] and the tokens; the iterated vectors and split sums come to less than a
    tenth of that and half a gigabyte."""
    for N, K, tokens, r in ((8192, 28672, 512, 64), (14336, 4096, 4096, 128), (32768, 32768, 512, 64),
                            (32768, 32768, 32768, 256), (4096, 4096, 262144, 64)):
        wide = N * (K + tokens) if tokens <= K else 0
        held = 8 * (max(2 * N * K + K * K, wide) + tokens * K)
        got = lib.aser_construct_workspace_bytes(N, K, tokens, r, 0)
        assert held <= got <= 1.1 * held + (1 << 29), (N, K, tokens, r, got / held)


def test_activation_path_of_a_forward_pass(lib):
    """One launch or two (many tokens, and ranks above 128 from 33 on): 448 tokens are seven whole clusters of the
    cluster kernel, the last of the one-launch kernels, at 4096 columns and more."""
    for K in (4096, 8192, 14336):
        assert [lib.aser_forward_act_launches(M, K, 128) for M in (1, 32, 33, 447, 448, 449, 4096)] == [1, 1, 1, 1, 1, 2, 2]
    assert [lib.aser_forward_act_launches(M, 2048, 128) for M in (1023, 1024)] == [1, 2]
    assert [lib.aser_forward_act_launches(M, 1024, 128) for M in (4096, 4097)] == [1, 2]
    assert [lib.aser_forward_act_launches(M, 4096, 144) for M in (32, 33)] == [1, 2]


def test_activation_path_without_a_projection_is_one_launch(lib):
    """The kernel that quantizes rows is the only one then, whatever the number of tokens."""
    for K in (1024, 4096, 8192, 14336):
        assert {lib.aser_forward_act_launches(M, K, 0) for M in (1, 32, 33, 448, 449, 4097)} == {1}
    assert lib.aser_forward_act_launches(0, 4096, 0) == 0 and lib.aser_forward_act_launches(8, 4100, 0) == 0


def test_activation_scratch_of_a_larger_pass_is_enough_for_a_smaller_one(lib):
    """A caller sizes it once, for his largest pass, although only few tokens go through it up to 8192 columns."""
    for K in (128, 512, 1024, 3072, 4096, 6144, 7680, 8192):
        for r in (0, 16, 128, 144, 256, 384):
            if K > 4096 and r > 128:
                continue            # partial sums at every size
            sizes = [lib.aser_quant_workspace_bytes(M, K, r) for M in (1, 32, 33, 63, 64, 100, 333, 399, 400, 599, 600, 1599, 1600, 4096, 70000)]
            assert sizes == sorted(sizes) and sizes[0] > 0
            slices = max(k for k in range(1, max(1, K // 256) + 1) if (K // 64) % k == 0)       # of one tile: the most there are
            if r > 128 and K <= 2048:
                assert sizes[3] >= 1024 + slices * 63 * (1 + (r + 127) // 128 * 128) * 4


def test_linear_kernel_rejects_bad_shapes(lib):
    assert lib.aser_linear_kernel(8, 4096, 4096) == 0
    for bad in ((8, 4096, 4100), (8, 4100, 4096), (0, 4096, 4096), (-1, 128, 128)):
        assert lib.aser_linear_kernel(*bad) == -3
