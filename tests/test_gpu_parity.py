"""GPU parity: the CUDA library (through its C ABI) against the CPU oracle on the same
seeded inputs.  Integer stages bit-exact; fp16 outputs within 2e-3 * max|y_ref| per row."""
import numpy as np
import pytest
import torch

import aser_synth as synth
from oracle import forward as F
from gpu_util import to_dev, oracle_layer, assert_rows_close, assert_T_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aser(cuda_device):
    import os
    import paper_2411_07762_b200 as aser
    # the oracle's row loops are independent: all host cores for the full-size cases
    F.set_threads(len(os.sched_getaffinity(0)))
    yield aser
    F.set_threads(1)


def bits(a):
    return np.ascontiguousarray(a).view(np.uint32)


# ---------------------------------------------------------------------------
# aser_pack_w4 / repack
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("N,K,smooth", [(512, 512, True), (136, 1024, True), (8, 128, False),
                                        (1024, 4096, True), (264, 14336, True)])
def test_pack_w4_bit_exact(aser, N, K, smooth):
    lay = synth.make_layer(1, N, K, seed=100 + N + K, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 11.5) if smooth else None
    W = lay.W.copy()
    if N >= 136:
        W[3] = 0                        # zero row: scale 0, codes 0
        W[5, :] = 0
        W[5, 7] = np.float16(3.5)       # single element: code 7 and exact ties elsewhere
        W[6, :8] = np.array([7, .5, 1.5, 2.5, -2.5, 6.5, -6.5, -7], np.float16)
        W[6, 8:] = 0
    q, w_scale = F.quant_w4(W, s)
    Wq, wsc = aser.pack_w4(to_dev(W), None if s is None else to_dev(s))
    assert np.array_equal(Wq.cpu().numpy(), F.pack_w4(q))
    assert np.array_equal(bits(wsc.cpu().numpy()), bits(w_scale))
    Wk = aser.repack_w4(Wq)
    assert Wk.numel() == aser.repacked_bytes(N, K)
    back = aser.unrepack_w4(Wk, N, K)
    assert torch.equal(back, Wq)


@pytest.mark.parametrize("N,K", [(16, 2176), (8, 4224), (136, 6272), (24, 8320), (8, 16384), (16, 16512), (8, 24704), (8, 32768)])
def test_pack_w4_chunks_per_thread(aser, N, K):
    """A row length for every chunk count a thread may hold (its last chunk partly missing where the
    length allows), with a row of exact ties and smoothing factors so small that the scale is below
    the range where its reciprocal is used."""
    lay = synth.make_layer(1, N, K, seed=300 + N + K, n_cal=8)
    W = lay.W.copy()
    W[1] = (np.arange(K) % 15 - 7).astype(np.float16) / 2      # halves, so ties against a scale of 1
    W[1, 0] = np.float16(7)
    W[2] = np.float16(2.0 ** -24)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 11.5)
    for sv in (None, s, (s * np.float32(2.0 ** -120)).astype(np.float32)):
        q, w_scale = F.quant_w4(W, sv)
        Wq, wsc = aser.pack_w4(to_dev(W), None if sv is None else to_dev(sv))
        assert np.array_equal(Wq.cpu().numpy(), F.pack_w4(q))
        assert np.array_equal(bits(wsc.cpu().numpy()), bits(w_scale))
    Wk = aser.repack_w4(Wq)
    assert torch.equal(aser.unrepack_w4(Wk, N, K), Wq)


def test_repack_layout_by_definition(aser):
    """Word w of sub-block `sub`, row `row` covers columns 32*sub + 8*w .. +7 with column
    c0+i in nibble 2i and column c0+4+i in nibble 2i+1."""
    N, K = 256, 384
    rng = np.random.default_rng(5)
    q = rng.integers(-8, 8, (N, K)).astype(np.int8)
    Wq = to_dev(F.pack_w4(q))
    Wk = aser.repack_w4(Wq).cpu().numpy().view(np.uint32).reshape(N // 128, K // 128, 4, 128, 4)
    for (nb, kb, sub, row, w) in [(0, 0, 0, 0, 0), (1, 2, 3, 127, 3), (0, 1, 2, 77, 1), (1, 0, 1, 5, 2)]:
        word = int(Wk[nb, kb, sub, row, w])
        c0 = kb * 128 + sub * 32 + w * 8
        n = nb * 128 + row
        for i in range(4):
            assert (word >> (8 * i)) & 0xF == int(q[n, c0 + i]) & 0xF
            assert (word >> (8 * i + 4)) & 0xF == int(q[n, c0 + 4 + i]) & 0xF


# ---------------------------------------------------------------------------
# aser_quant_act
# ---------------------------------------------------------------------------
ACT_CASES = [  # M, K, r
    (1, 512, 16), (3, 4096, 64), (8, 4096, 64), (16, 512, 16), (17, 1024, 0), (32, 8192, 32),
    (33, 512, 16), (127, 1024, 64), (129, 4096, 128), (300, 2048, 256), (64, 14336, 64),
    # cluster kernel: one stage per CTA, r = 0, ranks that leave accumulator rows unused, ragged
    # last token tile, every cluster size
    (65, 128, 0), (200, 128, 48), (96, 8192, 32), (1000, 2048, 112), (2049, 512, 16), (40, 28672, 64),
    # few tokens, long rows (two to eight chunks per thread, the last partly missing), with one, two
    # and four tokens per projection CTA and a last CTA that has fewer
    (1, 8320, 64), (5, 14336, 256), (17, 16512, 48), (32, 32768, 64), (3, 14336, 256), (7, 32768, 256), (31, 8320, 64), (2, 16384, 0),
]


@pytest.mark.parametrize("M,K,r", ACT_CASES)
def test_quant_act_parity(aser, M, K, r):
    lay = synth.make_layer(M, 8, K, seed=200 + M + K + r, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 13.0)
    X = lay.X.copy()
    if M >= 3:
        X[1] = 0                                   # zero token: scale 0, codes 0
        X[2, :] = 0
        X[2, :6] = np.array([127, .5, 1.5, 2.5, -2.5, -126.5], np.float16)   # exact ties
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0] if r else None
    xs = F.smooth_act(X, s)
    Xq_ref, sc_ref = F.quant_act(xs)
    Xq, sc, T = aser.quant_act(to_dev(X), to_dev(s), None if L_A is None else to_dev(L_A))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    if r:
        T_ref = F.down_proj(xs, L_A)
        assert_T_close(T.float().cpu().numpy(), T_ref, xs, L_A)


@pytest.mark.parametrize("M,K,r", [(8, 1024, 16), (300, 1024, 64), (2048, 512, 32)])
def test_quant_act_dense_smoothing_vector(aser, M, K, r):
    """Every divisor differs from 1 (a SmoothQuant-style vector): the division path everywhere,
    including divisors below 1."""
    lay = synth.make_layer(M, 8, K, seed=400 + M + K + r, n_cal=8)
    rng = np.random.default_rng(M + K)
    s = rng.uniform(0.25, 6.0, size=K).astype(np.float32)
    s[::7] = 1.0
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    xs = F.smooth_act(lay.X, s)
    Xq_ref, sc_ref = F.quant_act(xs)
    Xq, sc, T = aser.quant_act(to_dev(lay.X), to_dev(s), to_dev(L_A))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.parametrize("M,r", [(1, 32), (3, 256), (7, 256)])       # one, two and four tokens per projection CTA
@pytest.mark.parametrize("K", [512, 8320])
def test_quant_act_few_tokens_extreme_divisors(aser, M, r, K):
    """Divisors whose reciprocal is infinite (below 2^-128) or subnormal (above 2^126), with zeros and
    the smallest activations against them: x~ is the quotient, for the codes and for T alike."""
    lay = synth.make_layer(M, 8, K, seed=450 + M + r, n_cal=8)
    s = np.ones(K, np.float32)
    X = lay.X.copy()
    s[3], s[70], s[300], s[301] = 1e-40, 1e-40, 3e38, 7.0
    X[:, 3] = 0
    X[:, 70] = np.where(np.arange(M) % 2, 0, 2.0 ** -24).astype(np.float16)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    xs = F.smooth_act(X, s)
    assert np.isfinite(xs).all()
    Xq_ref, sc_ref = F.quant_act(xs)
    Xq, sc, T = aser.quant_act(to_dev(X), to_dev(s), to_dev(L_A))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.parametrize("path,M,K,r", [("cluster", 4096, 4096, 64), ("ws", 4800, 8192, 16)])
def test_quant_act_dense_smoothing_long_slices(aser, path, M, K, r):
    """Every divisor differs from 1 on slices long enough that a CTA meets more units with a
    divisor than it keeps in shared memory (the cluster kernel keeps 62 of its 128, the
    projection kernel 254 of its 256): the rest read their divisors from global memory."""
    lay = synth.make_layer(M, 8, K, seed=430 + M + K + r, n_cal=8)
    rng = np.random.default_rng(M + K + 1)
    s = rng.uniform(0.25, 6.0, size=K).astype(np.float32)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    xs = F.smooth_act(lay.X, s)
    Xq_ref, sc_ref = F.quant_act(xs)
    fn = aser.quant_act if path == "cluster" else aser.quant_act_ws
    Xq, sc, T = fn(to_dev(lay.X), to_dev(s), to_dev(L_A))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


def test_quant_act_without_smoothing_vector(aser):
    lay = synth.make_layer(5, 8, 256, seed=9, n_cal=8)
    Xq, sc, _ = aser.quant_act(to_dev(lay.X), None, None)
    Xq_ref, sc_ref = F.quant_act(F.smooth_act(lay.X, None))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref) and np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))


WS_ACT_CASES = [  # M, K, r, t_pair
    (33, 512, 16, False), (127, 1024, 64, False), (129, 4096, 128, False), (300, 2048, 256, False),
    (64, 14336, 64, False), (200, 128, 48, False), (65, 256, 0, False), (1000, 2048, 112, False),
    (2049, 512, 16, False), (40, 28672, 64, False),
    # stacked down projections of several layers (more than 256 rows), the pair storage of T,
    # and enough tokens at K = 14336 for the pass to be cut into chunks
    (700, 4096, 384, False), (260, 1024, 512, False), (300, 2048, 96, True), (4096, 14336, 128, False),
]


@pytest.mark.parametrize("M,K,r,t_pair", WS_ACT_CASES)
def test_quant_act_ws_parity(aser, M, K, r, t_pair):
    """aser_quant_act_ws (two kernels, caller's scratch): codes and scales bit-exact against the
    oracle, T within the derived bound, on ragged token tiles, zero rows and exact ties."""
    lay = synth.make_layer(M, 8, K, seed=250 + M + K + r, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 13.0)
    X = lay.X.copy()
    X[1] = 0
    X[2, :] = 0
    X[2, :6] = np.array([127, .5, 1.5, 2.5, -2.5, -126.5], np.float16)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0] if r else None
    xs = F.smooth_act(X, s)
    Xq_ref, sc_ref = F.quant_act(xs)
    Xq, sc, T = aser.quant_act_ws(to_dev(X), to_dev(s), None if L_A is None else to_dev(L_A), t_pair=t_pair)
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    if r:
        T_ref = F.down_proj(xs, L_A)
        if t_pair:
            assert_T_close(T[:, :r].float().cpu().numpy(), T_ref, xs, L_A)
            T_sum = T[:, :r].double().cpu().numpy() + T[:, r:].double().cpu().numpy()
            xs64, la64 = xs.astype(np.float64), L_A.astype(np.float64)
            tol = 2.0 ** -16 * np.abs(T_ref) + 2.0 ** -9.2 * np.sqrt((xs64 ** 2) @ (la64 ** 2).T) + \
                2.0 ** -20 * (np.abs(xs64) @ np.abs(la64).T) + 1e-30
            assert np.all(np.abs(T_sum - T_ref) <= tol)
        else:
            assert_T_close(T.float().cpu().numpy(), T_ref, xs, L_A)


def test_quant_act_ws_dense_smoothing_and_6_bits(aser):
    """Every divisor differs from 1, and 6-bit codes, through the two-kernel path."""
    M, K, r = 300, 1024, 64
    lay = synth.make_layer(M, 8, K, seed=471, n_cal=8)
    rng = np.random.default_rng(M + K)
    s = rng.uniform(0.25, 6.0, size=K).astype(np.float32)
    s[::7] = 1.0
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    xs = F.smooth_act(lay.X, s)
    for bits_ in (8, 6):
        Xq_ref, sc_ref = F.quant_act(xs, act_bits=bits_)
        Xq, sc, T = aser.quant_act_ws(to_dev(lay.X), to_dev(s), to_dev(L_A), act_bits=bits_)
        assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
        assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
        assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.parametrize("entry,M,K,r,divided,act_bits,t_pair", [
    # one launch (33 to a few hundred tokens): every cluster size and chunk count, one, two and four rows per CTA
    ("one", 33, 128, 16, 1, 8, False), ("one", 129, 1152, 48, 3, 8, True), ("one", 600, 1024, 16, 10, 6, False),
    ("one", 200, 2176, 64, 513, 8, False), ("one", 131, 4224, 80, 42, 8, False), ("one", 65, 8192, 32, 8192, 6, True),
    ("one", 40, 14336, 112, 143, 8, False), ("one", 34, 28672, 16, 600, 8, False), ("one", 47, 512, 0, 5, 8, False),
    # rows quantized beside the projection, and without one: every number of warps per row, ragged last rows
    ("ws", 35, 128, 16, 2, 8, False), ("ws", 1201, 1152, 16, 70, 8, True), ("ws", 333, 4096, 144, 512, 8, False),
    ("ws", 50, 4224, 16, 513, 6, False), ("ws", 1187, 8192, 32, 81, 8, False), ("ws", 305, 14336, 0, 143, 8, False),
    ("ws", 37, 28672, 0, 28672, 8, False), ("ws", 2500, 640, 0, 0, 8, False)])
def test_quant_act_beside_projection(aser, entry, M, K, r, divided, act_bits, t_pair):
    """Codes and scales bit-exact and T within the derived bound where codes and T are made by different CTAs
    (or kernels), with none, a few, a full list of and more divided columns than the list holds."""
    rng = np.random.default_rng(7 * M + K + r)
    X = rng.standard_normal((M, K)).astype(np.float16)
    X[1] = 0
    X[M - 1, :6] = np.array([127, .5, 1.5, 2.5, -2.5, -126.5], np.float16)
    X[M - 1, 6:] = 0
    s = np.ones(K, np.float32)
    cols = rng.choice(K, divided, replace=False)
    s[cols] = rng.uniform(0.02, 40.0, divided).astype(np.float32)
    X[:, cols[:3]] *= np.float16(30)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0] if r else None
    xs = F.smooth_act(X, s)
    Xq_ref, sc_ref = F.quant_act(xs, act_bits=act_bits)
    fn = aser.quant_act if entry == "one" else aser.quant_act_ws
    Xq, sc, T = fn(to_dev(X), to_dev(s), None if L_A is None else to_dev(L_A), act_bits=act_bits, t_pair=t_pair)
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    if r:
        assert_T_close(T[:, :r].float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.parametrize("M,K,r", [
    (63, 4096, 48), (64, 4096, 48), (99, 2048, 144), (100, 2048, 144), (599, 3712, 256), (600, 3712, 256),
    (99, 512, 384), (100, 512, 384), (1599, 1024, 272), (1600, 1024, 272), (99, 6144, 32), (100, 6144, 32), (99, 3200, 384),
    (100, 3200, 384), (399, 8192, 80), (400, 8192, 80)])
def test_quant_act_ws_on_both_sides_of_each_line(aser, M, K, r):
    """The two kernels one after the other below, beside each other above, with the scratch of a larger pass."""
    rng = np.random.default_rng(M + K + r)
    X = rng.standard_normal((M, K)).astype(np.float16)
    s = np.ones(K, np.float32)
    cols = rng.choice(K, K // 100, replace=False)
    s[cols] = 4.0
    X[:, cols] *= np.float16(20)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    ws = torch.full((aser.quant_workspace_bytes(4096, K, r),), 0x7f, dtype=torch.uint8, device="cuda")
    Xq, sc, T = aser.quant_act_ws(to_dev(X), to_dev(s), to_dev(L_A), ws=ws)
    xs = F.smooth_act(X, s)
    Xq_ref, sc_ref = F.quant_act(xs)
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.parametrize("entry", ["one", "ws"])
@pytest.mark.parametrize("M,K", [(20, 1024), (40, 8192), (300, 2048), (900, 4096), (333, 14336)])
@pytest.mark.parametrize("divided,s_value", [(3, 1e36), (3, 3e37), (0, 3e37), (600, 1e-36)])
def test_quant_act_rows_with_tiny_scales(aser, entry, M, K, divided, s_value):
    """Rows whose only elements that are not zero were divided by huge factors: the reciprocal of the scale overflows.
    divided 0: every column (the loop without a list)."""
    rng = np.random.default_rng(M + K + divided)
    X = rng.standard_normal((M, K)).astype(np.float16)
    s = np.ones(K, np.float32)
    cols = rng.choice(K, divided or K, replace=False)
    s[cols] = s_value
    X[::2, s == 1] = 0
    Xq_ref, sc_ref = F.quant_act(F.smooth_act(X, s))
    Xq, sc, _ = (aser.quant_act if entry == "one" else aser.quant_act_ws)(to_dev(X), to_dev(s), None)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)


# ---------------------------------------------------------------------------
# whole path: quant_act -> linear
# ---------------------------------------------------------------------------
def run_path(aser, lay, s, Wq_ref, w_scale_ref, L_A, L_B, impl, rows=None, use_dgemm=False,
             t_pair=False, timed_config=False, ws=None, ref=None):
    """Pack, quantize and multiply on the GPU, run the oracle on the same arrays, compare every
    stage.  `rows`: the oracle's products cover these token rows only (None = all).
    `t_pair`: T as bf16 pairs with the up projection written twice.  `timed_config`: the linear
    kernel runs once more without the accumulator dump (the configuration that is timed) and
    that output is compared with the oracle as well.  `ws`: a caller-owned workspace (reuse
    across calls).  `ref`: a precomputed oracle result for these inputs."""
    M, K = lay.X.shape
    N = lay.W.shape[0]
    r = 0 if L_A is None else L_A.shape[0]
    dW, ds = to_dev(lay.W), to_dev(s)
    Wq, wsc = aser.pack_w4(dW, ds)
    assert np.array_equal(Wq.cpu().numpy(), Wq_ref)
    assert np.array_equal(bits(wsc.cpu().numpy()), bits(w_scale_ref))
    del dW
    dLA = None if r == 0 else to_dev(L_A)
    dLB = None if r == 0 else to_dev(L_B)
    Xq, sc, T = aser.quant_act(to_dev(lay.X), ds, dLA, t_pair=t_pair)
    if t_pair:
        dLB = aser.pair_up_projection(dLB)
    r_lin = 2 * r if t_pair else r
    acc = torch.full((M, N), -7, dtype=torch.int32, device="cuda")
    Y_timed = None
    if impl == "simt":
        Y = aser.linear_w4a8_lr_simt(Xq, sc, Wq, wsc, T, dLB, acc_debug=acc)
    else:
        Wk = aser.repack_w4(Wq)
        if ws is None:
            ws = aser.new_workspace(M, N, K, r_lin)

        def call(acc_debug):
            if r:
                return aser.linear_w4a8_lr(Xq, sc, Wk, wsc, T, dLB, N, ws, acc_debug=acc_debug)
            return aser.linear_w4a8(Xq, sc, Wk, wsc, N, ws, acc_debug=acc_debug)
        Y = call(acc)
        if timed_config:
            Y_timed = call(None)
        aser.check_status(ws)
    torch.cuda.synchronize()
    if ref is None:
        ref = F.forward(lay.X, s, Wq_ref, w_scale_ref, L_A, L_B, rows=rows, use_dgemm=use_dgemm)
    assert np.array_equal(Xq.cpu().numpy(), ref.Xq)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(ref.a_scale))
    acc_h = acc.cpu().numpy()
    assert np.array_equal(acc_h if rows is None else acc_h[rows], ref.acc)
    assert_rows_close(Y.cpu().numpy(), ref.y, rows)
    if Y_timed is not None:
        assert_rows_close(Y_timed.cpu().numpy(), ref.y, rows)
    return Y


PATH_CASES = [  # M, N, K, r
    (16, 512, 512, 16), (1, 256, 512, 16), (7, 136, 1024, 32), (33, 264, 512, 0),
    (130, 384, 1024, 64), (257, 520, 2048, 128), (40, 128, 384, 256),
    # 17..32 tokens: the 32-token tile of the tensor-core kernel
    (19, 264, 1024, 32), (32, 384, 512, 16), (17, 1152, 2048, 64),
]


@pytest.mark.parametrize("impl", ["simt", "tc"])
@pytest.mark.parametrize("M,N,K,r", PATH_CASES)
def test_path_parity_small(aser, impl, M, N, K, r):
    lay = synth.make_layer(M, N, K, seed=300 + M + N + K + r, n_cal=64,
                           n_out=max(1, K // 100))
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=(K <= 1024 and r > 0))
    if r == 0:
        L_A = L_B = None
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, impl, timed_config=(impl == "tc"))


PAIR_CASES = [  # M, N, K, r: shapes the kernel on CTA pairs serves (256 channels x 256 tokens, 256 columns per stage)
    (333, 264, 384, 48),        # odd column blocks (half a stage), ragged channels, a whole and a short token column
    (260, 640, 512, 0),         # no low-rank term; odd number of 128-row blocks; four tokens in the short column
    (100, 520, 512, 80),        # a single half; two chunks, the second 16 wide
    (1300, 2056, 512, 144),     # three chunks; whole tiles, then single halves
    (513, 768, 640, 256),       # four chunks; tiles cut into single halves; one token in the short column
    (2100, 4104, 512, 64),      # more than one item per pair: whole, cut and short
]


@pytest.mark.parametrize("M,N,K,r", PAIR_CASES)
def test_pair_kernel_edges(aser, M, N, K, r):
    assert aser.lib.aser_linear_kernel(M, N, K) == 2
    lay = synth.make_layer(M, N, K, seed=900 + M + N + K + r, n_cal=16, n_out=max(1, K // 100))
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    if r == 0:
        L_A = L_B = None
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", timed_config=True, use_dgemm=True)


SHARED_TILE_CASES = [  # M, N, K, r: more than 64 tokens on the kernel whose CTAs may share tiles
    (130, 3080, 512, 64),       # whole tiles, ragged tokens and channels
    (257, 2056, 512, 128),      # whole tiles; one token in the last token tile
    (513, 1160, 512, 0),
    (77, 136, 7168, 80),        # every tile shared by many CTAs; two chunks, the second 16 wide
    (130, 392, 7168, 144),      # three chunks
    (257, 264, 7168, 0),
    (333, 264, 7168, 256),      # four chunks
    (263, 9480, 6144, 80),      # shared tiles before and after whole ones in a CTA's range
    (263, 9480, 8192, 32),      # the same with the shared tiles first
]


@pytest.mark.parametrize("M,N,K,r", SHARED_TILE_CASES)
def test_shared_tile_kernel_edges(aser, M, N, K, r):
    assert aser.lib.aser_linear_kernel(M, N, K) == 1
    lay = synth.make_layer(M, N, K, seed=950 + M + N + K + r, n_cal=16, n_out=max(1, K // 100))
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    if r == 0:
        L_A = L_B = None
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", timed_config=True, use_dgemm=True)


SPLIT_CASES = [  # M, N, K, r: 17 to 512 tokens, a tile's slices of K in a cluster
    (17, 520, 1024, 16),        # two CTAs of a cluster finish sixteen tokens each, the others none; ragged channels
    (33, 18944, 1024, 64),      # as many tiles as SMs: not split
    (64, 2056, 2176, 0),        # an odd number of column blocks, slices of unequal length
    (101, 4104, 4096, 80),      # the last CTA of a cluster has fewer tokens to finish; two chunks, the second 16 wide
    (128, 1160, 7168, 256),     # four chunks, eight slices
    (257, 2048, 1152, 144),     # three token tiles, three chunks
    (512, 1032, 1024, 128),     # four full token tiles
]


@pytest.mark.parametrize("M,N,K,r", SPLIT_CASES)
def test_split_kernel_edges(aser, M, N, K, r):
    assert aser.lib.aser_linear_kernel(M, N, K) == 3
    lay = synth.make_layer(M, N, K, seed=990 + M + N + K + r, n_cal=16, n_out=max(1, K // 100))
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    if r == 0:
        L_A = L_B = None
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", timed_config=True, use_dgemm=True)


@pytest.mark.parametrize("M", [1, 8])
@pytest.mark.parametrize("N,K,r", [(14336, 384, 128), (14344, 640, 0), (18944, 384, 16), (14216, 512, 64)])
def test_streaming_kernel_four_ctas_per_sm(aser, M, N, K, r):
    """Up to eight tokens and three to four 32-channel tiles for every SM of the part (445 to 592 on 148), with odd
    numbers of column blocks and a ragged last tile."""
    assert aser.lib.aser_linear_kernel(M, N, K) == 0
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 148:
        assert 3 * sms < (N + 31) // 32 <= 4 * sms
    lay = synth.make_layer(M, N, K, seed=970 + M + N + K + r, n_cal=16, n_out=max(1, K // 100))
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    if r == 0:
        L_A = L_B = None
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", timed_config=True, use_dgemm=True)


@pytest.mark.parametrize("impl", ["simt", "tc"])
def test_config1_tiny_with_constructed_factors(aser, impl):
    lay, r = synth.config1_tiny()
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=True)
    Y = run_path(aser, lay, s, Wq, w_scale, L_A, L_B, impl)
    # the compensated output is closer to the fp product than the plain W4A8 one
    plain = run_path(aser, lay, s, Wq, w_scale, None, None, impl)
    ref = lay.X.astype(np.float64) @ lay.W.astype(np.float64).T
    e_lr = np.linalg.norm(Y.cpu().numpy().astype(np.float64) - ref)
    e_plain = np.linalg.norm(plain.cpu().numpy().astype(np.float64) - ref)
    assert e_lr < e_plain


@pytest.mark.parametrize("impl", ["tc"])
@pytest.mark.parametrize("M", [1, 8])
def test_config2_decode_full_size(aser, impl, M):
    lay, r = synth.config2_decode(M)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=(M == 8))
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, impl, use_dgemm=True, timed_config=True)


@pytest.mark.parametrize("impl", ["tc"])
@pytest.mark.parametrize("which", ["gate_up", "down"])
def test_config3_prefill_full_size_all_rows(aser, impl, which):
    """Both prefill layers at full size: every accumulator bit-exact and every output element
    within the bound, with and without the accumulator dump (the timed configuration)."""
    lay, r = synth.config3_prefill(which)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, impl, use_dgemm=True, timed_config=True)


FORWARD_CASES = [  # M, N, K, r
    (8, 512, 4096, 64), (1, 256, 512, 16), (33, 264, 512, 0), (130, 384, 1024, 64),
    (300, 1152, 2048, 128), (2048, 512, 4096, 64),
]


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,r", FORWARD_CASES)
def test_forward_overlapped_is_bit_identical_to_separate_calls(aser, M, N, K, r):
    """aser_forward launches the linear kernel as a programmatic dependent of the quantization
    kernel; every output must equal that of the two plain calls, on repeated back-to-back runs
    with alternating inputs (a missing wait would show as stale Xq, a_scale or T)."""
    lay = synth.make_layer(M, N, K, seed=900 + M + N + K + r, n_cal=8, n_out=max(1, K // 100))
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 9.0)
    L_A, L_B = synth.standin_factors(N, K, r, seed=M + r, scale_a=0.02, scale_b=0.02) if r else (None, None)
    layer = aser.AserLinear(to_dev(lay.W), to_dev(s), None if r == 0 else to_dev(L_A),
                            None if r == 0 else to_dev(L_B), M)
    X0 = to_dev(lay.X)
    X1 = torch.roll(X0, shifts=3, dims=1).contiguous() * 0.5
    want = []
    for X in (X0, X1):
        layer.quant(X)
        layer.linear(M)
        want.append((layer.Y[:M].clone(), layer.Xq[:M].clone(), layer.a_scale[:M].clone(),
                     layer.T[:M].clone()))
    aser.check_status(layer.ws)
    for it in range(12):
        X = (X0, X1)[it & 1]
        Y = layer(X)
        got = (Y, layer.Xq[:M], layer.a_scale[:M], layer.T[:M])
        for g, w in zip(got, want[it & 1]):
            assert torch.equal(g.view(torch.uint8), w.view(torch.uint8)), it
    aser.check_status(layer.ws)


@pytest.mark.parametrize("name", ["q", "k", "gate", "down"])
def test_config4_block_linears_full_size_all_rows(aser, name):
    """Decoder-block linears at 4096 tokens, rank 128 (the square projection with eight whole
    tiles per CTA, the GQA projection, the widest and the deepest layer): every code, scale,
    accumulator and output element.  The widest layer also runs a 32-token call first on the
    workspace sized for 4096 tokens: one workspace serves calls of different shapes in turn."""
    lay, r = synth.config4_block_layer(name)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    ref = F.forward(lay.X, s, Wq, w_scale, L_A, L_B, use_dgemm=True)
    M, K = lay.X.shape
    N = lay.W.shape[0]
    ws = aser.new_workspace(M, N, K, r)
    if name == "gate":
        m = 32
        small = synth.LayerInputs(X=lay.X[:m], W=lay.W, X_cal=lay.X_cal, outlier_idx=lay.outlier_idx,
                                  outlier_gain=lay.outlier_gain, meta=lay.meta)
        ref_small = F.ForwardResult(xs=ref.xs[:m], Xq=ref.Xq[:m], a_scale=ref.a_scale[:m],
                                    acc=ref.acc[:m], T=ref.T[:m], y=ref.y[:m], rows=None)
        run_path(aser, small, s, Wq, w_scale, L_A, L_B, "tc", ws=ws, ref=ref_small)
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", ws=ws, ref=ref, timed_config=True)
    if name == "gate":     # and back to the small shape on the same workspace
        run_path(aser, small, s, Wq, w_scale, L_A, L_B, "tc", ws=ws, ref=ref_small)


C5_POINTS = [  # M, N, r, all rows?
    (1, 8192, 64, True), (16, 8192, 32, True), (16, 28672, 64, True), (128, 8192, 0, True),
    (128, 28672, 256, True), (1024, 8192, 128, True), (1024, 28672, 32, False),
    (4096, 8192, 128, True), (4096, 8192, 0, False), (4096, 28672, 64, True), (4096, 8192, 256, False),
]


@pytest.mark.parametrize("M,N,r,full", C5_POINTS)
def test_config5_sweep_points(aser, M, N, r, full):
    """Points of the 70B-class sweep (K = 8192): few tokens on both few-token paths (streaming
    kernel up to 64 MB of packed weights, tensor-core kernel above), rank 256 (two launches of
    the quantization cluster kernel), rank 0 (plain W4A8), and 4096 tokens at both widths
    compared on every row (the remaining points on token rows spread over every 128-token tile)."""
    lay = synth.config5_point(M, N)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    if r == 0:
        L_A = L_B = None
    rows = None
    if not full:
        base = np.arange(0, M, 128)
        rows = np.unique(np.concatenate([base, base + 127, base + 61]).clip(0, M - 1))
    run_path(aser, lay, s, Wq, w_scale, L_A, L_B, "tc", rows=rows, use_dgemm=True,
             timed_config=(M == 4096))


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,r", [(4096, 8192, 8192, 256), (4096, 4096, 4096, 128), (2048, 1024, 14336, 192)])
def test_many_chunks_on_long_tiles_repeated_launches(aser, M, N, K, r):
    """Several low-rank chunks per 128-token tile on tiles long enough for the mid-tile schedule,
    several tiles per CTA, launched back to back: no bounded wait may give up (a chunk that is
    late must never make a role wait for something only a stalled role can provide) and every
    launch must give the same bits."""
    lay = synth.make_layer(M, N, K, seed=900 + r, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 16.0)
    L_A, L_B = synth.standin_factors(N, K, r, seed=3, scale_a=0.01, scale_b=0.01)
    L = aser.AserLinear(to_dev(lay.W), to_dev(s), to_dev(L_A), to_dev(L_B), M)
    X = to_dev(lay.X)
    first = L(X).clone()
    aser.check_status(L.ws)
    for rep in range(30):
        L.linear(M, True)
    torch.cuda.synchronize()
    aser.check_status(L.ws)
    assert torch.equal(L.Y[:M], first)
    for rep in range(10):
        Y = L(X)
    torch.cuda.synchronize()
    aser.check_status(L.ws)
    assert torch.equal(Y, first)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,r", [(8, 256, 1024, 40), (200, 384, 2048, 72)])
def test_rank_not_a_multiple_of_16_is_padded_with_zeros(aser, M, N, K, r):
    """A per-layer rank from the singular-value threshold (Sec. 4.1) is any integer: pad_rank
    appends zero rows / columns; the result must match the oracle run on the UNPADDED factors."""
    lay = synth.make_layer(M, N, K, seed=700 + r, n_cal=8)
    s, Wq_ref, w_scale_ref, L_A, L_B = oracle_layer(lay, r, construct=False)
    dLA, dLB = aser.pad_rank(to_dev(L_A), to_dev(L_B))
    assert dLA.shape[0] % 16 == 0 and dLB.shape[1] == dLA.shape[0]
    ds = to_dev(s)
    Wq, wsc = aser.pack_w4(to_dev(lay.W), ds)
    Wk = aser.repack_w4(Wq)
    Xq, sc, T = aser.quant_act(to_dev(lay.X), ds, dLA)
    ws = aser.new_workspace(M, N, K, dLA.shape[0])
    acc = torch.zeros((M, N), dtype=torch.int32, device="cuda")
    Y = aser.linear_w4a8_lr(Xq, sc, Wk, wsc, T, dLB, N, ws, acc_debug=acc)
    aser.check_status(ws)
    torch.cuda.synchronize()
    ref = F.forward(lay.X, s, Wq_ref, w_scale_ref, L_A, L_B)
    assert np.array_equal(acc.cpu().numpy(), ref.acc)
    assert bool((T[:, r:] == 0).all())
    assert_rows_close(Y.cpu().numpy(), ref.y)


@pytest.mark.gpu
@pytest.mark.parametrize("M", [16, 200])
def test_paper_smoothing_rule_with_outlier_split_runs_through_the_same_path(aser, M):
    """The paper's own variant (Sec. 4.2): m_i = X-bar_i / min over the f outlier channels
    (Eq. 11), and the outlier columns W_o kept out of the int4 matrix and carried by the low-rank
    factors (Eq. 12).  For the GPU this is the same path with different inputs: the caller zeroes
    the outlier columns of W before packing.  The low-rank term is then as large as the output,
    so T is stored as bf16 pairs (aser_quant_act_ex); with that the output meets the same
    2e-3 * max|y_ref| bound as everywhere else.  Packed weights and accumulators bit-exact; and
    the split layer's output is closer to the fp product than plain W4A8 on the same codes.
    M = 16 takes the few-token kernels, M = 200 the tensor-core kernels."""
    from oracle import construct as Cn
    lay, r = synth.config1_tiny()
    if M != 16:
        lay = synth.make_layer(M, 512, 512, seed=synth.seed_for(1, M), n_out=4, outlier_gain=40.0,
                               sigma_w=0.02, n_cal=128)
    s, idx = Cn.smoothing_vector_paper(lay.X_cal, lay.W, f=4)
    assert np.array_equal(idx, lay.outlier_idx)
    L = Cn.construct_layer(lay.W, lay.X_cal, s, r=r, split_outliers=idx)
    W_split = lay.W.copy()
    W_split[:, idx] = 0
    lay_split = synth.LayerInputs(X=lay.X, W=W_split, X_cal=lay.X_cal, outlier_idx=lay.outlier_idx,
                                  outlier_gain=lay.outlier_gain, meta=lay.meta)
    Y = run_path(aser, lay_split, s, L.Wq, L.w_scale, L.L_A, L.L_B, "tc", t_pair=True,
                 timed_config=True)
    plain = run_path(aser, lay_split, s, L.Wq, L.w_scale, None, None, "tc")
    ref = lay.X.astype(np.float64) @ lay.W.astype(np.float64).T
    e_lr = np.linalg.norm(Y.cpu().numpy().astype(np.float64) - ref)
    e_plain = np.linalg.norm(plain.cpu().numpy().astype(np.float64) - ref)
    assert e_lr < 0.5 * e_plain        # without the factors the outlier columns are simply missing


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,r", [(8, 1024, 16), (300, 2048, 64), (129, 4096, 128), (40, 512, 48)])
def test_quant_act_pair_storage_of_T(aser, M, K, r):
    """aser_quant_act_ex with t_pair: hi + lo reproduces the fp64 projection to 2^-16 of each
    entry (plus the fp16 rounding of x~ inside the tensor-core product), codes and scales are
    those of the plain call, and hi is the plain call's T."""
    lay = synth.make_layer(M, 8, K, seed=800 + M + K + r, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 13.0)
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0]
    dX, ds, dLA = to_dev(lay.X), to_dev(s), to_dev(L_A)
    Xq0, sc0, T0 = aser.quant_act(dX, ds, dLA)
    Xq, sc, T = aser.quant_act(dX, ds, dLA, t_pair=True)
    assert T.shape == (M, 2 * r)
    assert torch.equal(Xq, Xq0) and torch.equal(sc, sc0)
    assert torch.equal(T[:, :r].contiguous().view(torch.int16), T0.view(torch.int16))
    xs = F.smooth_act(lay.X, s)
    T_ref = F.down_proj(xs, L_A)
    T_sum = T[:, :r].double().cpu().numpy() + T[:, r:].double().cpu().numpy()
    xs64, la64 = xs.astype(np.float64), L_A.astype(np.float64)
    rms = np.sqrt((xs64 ** 2) @ (la64 ** 2).T)
    l1 = np.abs(xs64) @ np.abs(la64).T
    tol = 2.0 ** -16 * np.abs(T_ref) + 2.0 ** -9.2 * rms * (M > 32) + 2.0 ** -20 * l1 + 1e-30
    assert np.all(np.abs(T_sum - T_ref) <= tol)
    with pytest.raises(aser.AserError) as err:      # 2 r beyond the kernels' 256
        aser.quant_act(dX, ds, to_dev(synth.standin_factors(8, K, 144, seed=1)[0]), t_pair=True)
    assert err.value.code == -3


@pytest.mark.gpu
def test_rank_from_threshold_end_to_end(aser):
    """Sec. 4.1 Eq. 9 end to end: the oracle picks the rank from the singular-value threshold
    alpha (any integer, here not a multiple of 16), pad_rank brings the factors to the kernels'
    granularity, and the GPU output matches the oracle run on the UNPADDED factors."""
    from oracle import construct as Cn
    lay = synth.make_layer(48, 384, 512, seed=synth.seed_for(1, 77), n_out=5, outlier_gain=40.0, n_cal=256)
    s = Cn.smoothing_vector_config(lay.X_cal, lay.W, lay.outlier_idx)
    seen = set()
    for alpha in (0.05, 0.12, 0.3):
        L = Cn.construct_layer(lay.W, lay.X_cal, s, r=None, alpha=alpha)
        r = L.L_A.shape[0]
        assert r == Cn.rank_from_alpha(L.sigma, alpha) and 0 < r < 256
        seen.add(r % 16 != 0)
        dLA, dLB = aser.pad_rank(to_dev(L.L_A), to_dev(L.L_B))
        ds = to_dev(s)
        Wq, wsc = aser.pack_w4(to_dev(lay.W), ds)
        assert np.array_equal(Wq.cpu().numpy(), L.Wq)
        Xq, sc, T = aser.quant_act(to_dev(lay.X), ds, dLA)
        ws = aser.new_workspace(48, 384, 512, dLA.shape[0])
        acc = torch.zeros((48, 384), dtype=torch.int32, device="cuda")
        Y = aser.linear_w4a8_lr(Xq, sc, aser.repack_w4(Wq), wsc, T, dLB, 384, ws, acc_debug=acc)
        aser.check_status(ws)
        ref = F.forward(lay.X, s, L.Wq, L.w_scale, L.L_A, L.L_B)
        assert np.array_equal(acc.cpu().numpy(), ref.acc)
        assert_rows_close(Y.cpu().numpy(), ref.y)
    assert True in seen                 # at least one rank that needed padding


@pytest.mark.gpu
def test_status_word_reports_a_timeout_and_clears(aser):
    """aser_check_status without any kernel timing out: a status word planted by a memset must
    come back as ASER_ERR_DEVICE_TIMEOUT once, then the workspace is clean (word and counters)."""
    ws = aser.new_workspace(64, 256, 512, 16)
    aser.check_status(ws)
    ws[0] = 1
    ws[256:260] = 3                     # a tile counter left behind by the same launch
    with pytest.raises(aser.AserError) as err:
        aser.check_status(ws)
    assert err.value.code == -6 and "status word" in str(err.value)
    aser.check_status(ws)
    assert int(ws[:1024].to(torch.int32).sum()) == 0


SHARED_CASES = [  # M, K, [(N, r), ...]
    (8, 1024, [(256, 32), (128, 16), (128, 16)]),
    (8, 1024, [(256, 32), (128, 32), (384, 32), (128, 32)]),
    (16, 2048, [(1024, 64), (256, 64)]),
    (200, 1024, [(384, 64), (128, 64)]),
    (1100, 1024, [(256, 128), (128, 128), (128, 128)]),
    (200, 1024, [(384, 64), (136, 48), (128, 0)]),
    (300, 2048, [(512, 128), (256, 128), (256, 128)]),
]


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,spec", SHARED_CASES)
def test_forward_shared_matches_oracle_per_layer(aser, M, K, spec):
    """aser_forward_shared: one activation pass for layers that read the same X.  Codes and
    scales bit-exact; every layer's output within the bound of the oracle run on that layer
    alone; and the stacked T agrees with the per-layer T of each layer's own activation step."""
    check_shared_group(aser, M, K, spec, seed0=1200 + M + K, construct=False)


def check_shared_group(aser, M, K, spec, seed0, construct, gain=30.0):
    base = synth.make_layer(M, spec[0][0], K, seed=seed0, n_cal=64, n_out=max(1, K // 100), outlier_gain=gain)
    s = synth.standin_smoothing_vector(K, base.outlier_idx, 11.0)
    ds = to_dev(s)
    layers, refs = [], []
    for li, (N, r) in enumerate(spec):
        rng = np.random.default_rng(seed0 + 17 * li + 1)
        W = (rng.standard_normal((N, K), dtype=np.float32) * np.float32(0.02)).astype(np.float16)
        q, w_scale = F.quant_w4(W, s)
        L_A, L_B = synth.standin_factors(N, K, max(r, 16), seed=seed0 + li, scale_a=0.01, scale_b=0.01)
        L_A, L_B = (L_A[:r], np.ascontiguousarray(L_B[:, :r])) if r else (None, None)
        lay = aser.AserLinear(to_dev(W), ds, None if r == 0 else to_dev(L_A), None if r == 0 else to_dev(L_B), M)
        assert np.array_equal(lay.Wq.cpu().numpy(), F.pack_w4(q))
        layers.append(lay)
        refs.append(F.forward(base.X, s, F.pack_w4(q), w_scale, L_A, L_B, use_dgemm=True))
    group = aser.AserSharedInput(layers, M)
    X = to_dev(base.X)
    for rep in range(2):                    # twice: the workspace is reused
        Ys = group(X)
        aser.check_status(group.ws)
        torch.cuda.synchronize()
        assert np.array_equal(group.Xq[:M].cpu().numpy(), refs[0].Xq)
        assert np.array_equal(bits(group.a_scale[:M].cpu().numpy()), bits(refs[0].a_scale))
        col = 0
        for lay, ref, Y in zip(layers, refs, Ys):
            assert_rows_close(Y.cpu().numpy(), ref.y)
            if lay.r:
                # the layer's own activation step may run other kernels (another summation
                # order): equal up to the last bf16 bit wherever T is not a cancellation
                lay.quant(X)
                a = group.T[:M, col:col + lay.r].float()
                b = lay.T[:M].float()
                assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 2.0 ** -9 * b.abs().max()).all())
                col += lay.r
    # the same group stored as one fused projection (one linear launch over the concatenated N)
    ranks = {r for _, r in spec}
    if len(ranks) == 1 and all(N % 128 == 0 for N, _ in spec) and len(spec) <= 4:
        per_layer = [y.clone() for y in group(X)]
        cat = aser.AserSharedInputCat(layers, M)
        for rep in range(2):
            Ys = cat(X)
            aser.check_status(cat.ws)
            torch.cuda.synchronize()
            assert np.array_equal(cat.Xq[:M].cpu().numpy(), refs[0].Xq)
            for ref, Y, Y1 in zip(refs, Ys, per_layer):
                assert_rows_close(Y.cpu().numpy(), ref.y)
                # same operands, same arithmetic per element as the layer's own launch
                assert torch.equal(Y, Y1)
        Ys = cat.linear(M)                  # the linear step alone on the codes already there
        torch.cuda.synchronize()
        for ref, Y in zip(refs, Ys):
            assert_rows_close(Y.cpu().numpy(), ref.y)


@pytest.mark.gpu
@pytest.mark.parametrize("which", ["qkv", "gate_up"])
def test_forward_shared_decoder_block_groups_full_size(aser, which):
    """The two shared-input groups of the decoder block at 4096 tokens, rank 128: query/key/value
    (384 stacked rows) and gate/up (256)."""
    spec = [(4096, 128), (1024, 128), (1024, 128)] if which == "qkv" else [(14336, 128), (14336, 128)]
    check_shared_group(aser, 4096, 4096, spec, seed0=synth.seed_for(4, 50 + len(spec)), construct=False)


# ---------------------------------------------------------------------------
# 6-bit activation codes (the W4A6 setting): same kernels, narrower code range
# ---------------------------------------------------------------------------
@pytest.mark.gpu
@pytest.mark.parametrize("M,K,r", [(5, 1024, 16), (33, 512, 0), (200, 2048, 64), (300, 2048, 256),
                                   (129, 4096, 128)])
def test_quant_act_6bit_parity(aser, M, K, r):
    lay = synth.make_layer(M, 8, K, seed=600 + M + K + r, n_cal=8)
    s = synth.standin_smoothing_vector(K, lay.outlier_idx, 13.0)
    X = lay.X.copy()
    X[1] = 0                                       # zero token: scale 0, codes 0
    X[2, :] = 0
    X[2, :6] = np.array([31, .5, 1.5, 2.5, -2.5, -30.5], np.float16)   # exact ties at scale 1
    L_A = synth.standin_factors(8, K, r, seed=M, scale_a=0.05)[0] if r else None
    xs = F.smooth_act(X, s)
    Xq_ref, sc_ref = F.quant_act(xs, act_bits=6)
    Xq, sc, T = aser.quant_act(to_dev(X), to_dev(s), None if L_A is None else to_dev(L_A), act_bits=6)
    assert np.array_equal(Xq.cpu().numpy(), Xq_ref)
    assert np.array_equal(bits(sc.cpu().numpy()), bits(sc_ref))
    assert int(Xq.abs().max()) == 31
    if r:
        assert_T_close(T.float().cpu().numpy(), F.down_proj(xs, L_A), xs, L_A)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,r", [(8, 256, 1024, 16), (130, 384, 1024, 64)])
def test_w4a6_path_parity(aser, M, N, K, r):
    """W4A6: 6-bit codes through the unchanged linear kernels; accumulators bit-exact, output
    within the bound, against the oracle run with act_bits = 6."""
    lay = synth.make_layer(M, N, K, seed=650 + M, n_cal=8)
    s, Wq_ref, w_scale_ref, L_A, L_B = oracle_layer(lay, r, construct=False)
    ds, dLA, dLB = to_dev(s), to_dev(L_A), to_dev(L_B)
    Wq, wsc = aser.pack_w4(to_dev(lay.W), ds)
    Wk = aser.repack_w4(Wq)
    Xq, sc, T = aser.quant_act(to_dev(lay.X), ds, dLA, act_bits=6)
    ws = aser.new_workspace(M, N, K, r)
    acc = torch.zeros((M, N), dtype=torch.int32, device="cuda")
    Y = aser.linear_w4a8_lr(Xq, sc, Wk, wsc, T, dLB, N, ws, acc_debug=acc)
    aser.check_status(ws)
    torch.cuda.synchronize()
    ref = F.forward(lay.X, s, Wq_ref, w_scale_ref, L_A, L_B, act_bits=6)
    assert np.array_equal(Xq.cpu().numpy(), ref.Xq)
    assert np.array_equal(acc.cpu().numpy(), ref.acc)
    assert_rows_close(Y.cpu().numpy(), ref.y)


@pytest.mark.gpu
def test_quant_act_bits_rejects_other_widths(aser):
    X = torch.zeros((4, 128), dtype=torch.float16, device="cuda")
    for bad in (1, 9, 0):
        with pytest.raises(aser.AserError) as err:
            aser.quant_act(X, None, None, act_bits=bad)
        assert err.value.code == -3


@pytest.mark.gpu
@pytest.mark.parametrize("N,K", [(264, 512), (6152, 6144)])
@pytest.mark.parametrize("M", [200, 256, 333, 700, 1030])
def test_forward_host_in_parts(aser, M, N, K):
    """Pinned buffers: undivided where there is too little to overlap, else one part, two and four with a ragged last
    one; pageable buffers take the undivided path.  Both against the oracle, and again on two streams in turn
    and from two threads at once (each with a layer of its own)."""
    import threading
    r = 32
    assert aser.lib.aser_forward_host_parts(M, N, K, None) == (1 if K == 512 else {200: 1, 256: 2, 333: 2, 700: 4, 1030: 4}[M])
    lay = synth.make_layer(M, N, K, seed=1200 + M, n_cal=8)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    ref = F.forward(lay.X, s, Wq, w_scale, L_A, L_B, use_dgemm=True)
    X = torch.from_numpy(lay.X.copy())

    def make():
        return (aser.AserLinear(to_dev(lay.W), to_dev(s), to_dev(L_A), to_dev(L_B), M), X.pin_memory(),
                torch.zeros((M, N), dtype=torch.float16).pin_memory())

    layer, X_pin, Y_pin = make()
    torch.cuda.synchronize()
    layer.forward_host(X_pin, Y_pin)
    torch.cuda.current_stream().synchronize()
    assert_rows_close(Y_pin.numpy(), ref.y)
    Y_page = torch.zeros((M, N), dtype=torch.float16)
    layer.forward_host(X, Y_page)
    torch.cuda.current_stream().synchronize()
    assert_rows_close(Y_page.numpy(), ref.y)

    sets = [make(), make()]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(3):
        for st, (l, x, y) in zip(streams, sets):
            with torch.cuda.stream(st):
                l.forward_host(x, y)
    for st in streams:
        st.synchronize()
    for _, _, y in sets:
        assert_rows_close(y.numpy(), ref.y)
        y.zero_()

    def work(st, l, x, y):
        with torch.cuda.stream(st):
            for _ in range(5):
                l.forward_host(x, y)
            st.synchronize()
    threads = [threading.Thread(target=work, args=(st, *t)) for st, t in zip(streams, sets)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for l, _, y in sets:
        assert_rows_close(y.numpy(), ref.y)
        aser.check_status(l.ws)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,r,parts", [
    (1024, 4096, 5120, 64, 4),      # whole: two-kernel activation path; a quarter alone would take the cluster kernel
    (2050, 1032, 1024, 48, 2),      # cluster kernel, whose split of K depends on the number of tokens; a ragged last part
    (520, 6144, 14336, 16, 4),      # long rows; parts of 128 tokens share tiles of the linear kernel
    (700, 3072, 7168, 256, 2),      # four low-rank chunks; two-kernel path, whose split depends on the number too
])
def test_forward_host_bits_do_not_depend_on_the_cut(aser, M, N, K, r, parts):
    """A pass from pinned buffers, cut into parts on any number of streams, has the bits of one undivided pass."""
    assert aser.lib.aser_forward_host_parts(M, N, K, None) == parts
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N)
    W = torch.randn(N, K, device="cuda", generator=g).half() * 0.02
    # the second half of K all but cancels the first, so that T shows the order in which it was summed
    half = torch.randn(M, K // 2, device="cuda", generator=g).half()
    X = torch.cat([half, half], dim=1)
    a = torch.randn(r, K // 2, device="cuda", generator=g).half()
    L_A = torch.cat([a, 0.01 * torch.randn(r, K // 2, device="cuda", generator=g).half() - a], dim=1)
    L_B = torch.randn(N, r, device="cuda", generator=g).half()
    layer = aser.AserLinear(W, None, L_A, L_B, M)
    whole, whole_T = layer(X).cpu(), layer.T.clone()
    X_pin, Y_pin = X.cpu().pin_memory(), torch.empty((M, N), dtype=torch.float16).pin_memory()
    torch.cuda.synchronize()
    for st in [torch.cuda.Stream() for _ in range(6)]:       # more streams than a thread keeps copy streams for
        for _ in range(2):
            Y_pin.zero_()
            with torch.cuda.stream(st):
                layer.forward_host(X_pin, Y_pin)
            st.synchronize()
            assert torch.equal(layer.T, whole_T)
            assert torch.equal(Y_pin, whole)
    aser.check_status(layer.ws)


@pytest.mark.gpu
@pytest.mark.parametrize("host,device", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("N,K", [(4096, 3072), (3072, 4096), (3072, 3072)])
def test_forward_host_output_in_the_place_of_the_input(aser, N, K, host, device):
    """Y over X in the pinned host buffer, in the device staging buffer, or both: no row of X is overwritten before it
    is read, whether or not the pass is cut into parts."""
    M, r = 512, 32
    assert aser.lib.aser_forward_host_parts(M, N, K, None) == 2
    lay = synth.make_layer(M, N, K, seed=1300 + N + K, n_cal=8)
    s, Wq, w_scale, L_A, L_B = oracle_layer(lay, r, construct=False)
    ref = F.forward(lay.X, s, Wq, w_scale, L_A, L_B, use_dgemm=True)
    layer = aser.AserLinear(to_dev(lay.W), to_dev(s), to_dev(L_A), to_dev(L_B), M)
    if device:
        both = torch.empty((M * max(N, K),), dtype=torch.float16, device="cuda")
        layer.X_dev, layer.Y = both[:M * K].view(M, K), both[:M * N].view(M, N)
    X = torch.empty((M * max(N, K),), dtype=torch.float16).pin_memory()
    Y = X if host else torch.empty((M * N,), dtype=torch.float16).pin_memory()
    for _ in range(3):
        X[:M * K] = torch.from_numpy(lay.X.copy()).view(-1)
        layer.forward_host(X[:M * K].view(M, K), Y[:M * N].view(M, N))
        torch.cuda.current_stream().synchronize()
        assert_rows_close(Y[:M * N].view(M, N).numpy(), ref.y)
    aser.check_status(layer.ws)


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,spec", [
    (5, 640, [(520, 16), (24, 0), (2056, 48)]), (16, 1024, [(9480, 64), (9480, 64)]),               # few tokens: any ranks
    (333, 384, [(264, 48)] * 4), (1300, 512, [(2056, 144)] * 2), (513, 640, [(768, 0)] * 3),      # CTA pairs: one rank
])
def test_shared_group_in_one_launch_has_the_bits_of_its_layers(aser, M, K, spec):
    """Layers that read the same codes, each with operands of its own, served by one launch: ragged channels in every
    layer, so that tiles end inside the group."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K)
    s = torch.ones(K, device="cuda")
    s[::97] = 3.0
    half = lambda *shape, scale: (torch.randn(*shape, device="cuda", generator=g) * scale).half()
    layers = [aser.AserLinear(half(n, K, scale=0.02), s, half(r, K, scale=0.02) if r else None,
                              half(n, r, scale=0.02) if r else None, M) for n, r in spec]
    assert len({aser.lib.aser_linear_kernel(M, n, K) for n, _ in spec}) == 1
    group = aser.AserSharedInput(layers, M)
    Ys = [y.clone() for y in group(half(M, K, scale=1.0))]
    aser.check_status(group.ws)
    col = 0
    for (n, r), lay, Y in zip(spec, layers, Ys):
        if r:
            ref = aser.binding.linear_w4a8_lr_ld(group.Xq, group.a_scale, lay.Wk, lay.w_scale, group.T, col, lay.L_B, n, group.ws)
        else:
            ref = aser.linear_w4a8(group.Xq, group.a_scale, lay.Wk, lay.w_scale, n, group.ws)
        assert torch.equal(Y, ref)
        col += r


@pytest.mark.gpu
@pytest.mark.parametrize("r", [128, 192])
def test_fused_group_is_bit_identical_across_the_two_tensor_core_kernels(aser, r):
    """1024 tokens, K = 4096, two layers of 2048 channels: the fused launch (4096 channels) is served by CTA pairs,
    a layer alone by the kernel that may share tiles.  Both add the low-rank chunks in order, so the bits agree."""
    import ctypes as C
    M, K, N = 1024, 4096, 2048
    assert [aser.lib.aser_linear_kernel(M, n, K) for n in (N, 2 * N)] == [1, 2]
    g = torch.Generator(device="cuda")
    g.manual_seed(77 + r)
    Xq = torch.randint(-127, 128, (M, K), device="cuda", dtype=torch.int8, generator=g)
    a = torch.rand(M, device="cuda", generator=g) * 1e-3
    T = torch.randn(M, 2 * r, device="cuda", generator=g).bfloat16()
    packed = [aser.pack_w4(torch.randn(N, K, device="cuda", generator=g).half(), None) for _ in range(2)]
    Wk = [aser.repack_w4(w) for w, _ in packed]
    LB = [torch.randn(N, r, device="cuda", generator=g).half() * 0.1 for _ in range(2)]
    ws = aser.new_workspace(M, 2 * N, K, r)
    Y = torch.empty((M, 2 * N), device="cuda", dtype=torch.float16)
    wk, sc, lb = torch.cat(Wk), torch.cat([s for _, s in packed]), torch.cat(LB).contiguous()
    P = lambda t: C.c_void_p(t.data_ptr())
    rc = aser.lib.aser_linear_w4a8_lr_cat(P(Xq), P(a), P(wk), P(sc), P(T), P(lb), 2, (C.c_int * 2)(N, N), r, M, K, P(Y),
                                          P(ws), ws.numel(), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    for i in range(2):
        y = aser.linear_w4a8_lr_ld(Xq, a, Wk[i], packed[i][1], T, i * r, LB[i], N, ws)
        assert torch.equal(Y[:, i * N:(i + 1) * N], y)
    aser.check_status(ws)


@pytest.mark.gpu
@pytest.mark.parametrize("M,more,N,K,r,kernel", [
    (17, 2000, 512, 1152, 48, 1),         # an odd number of column blocks: the last stage of a slice is half a stage
    (101, 1200, 4096, 4096, 128, 2), (384, 900, 2048, 2176, 192, 1), (512, 2000, 1024, 1024, 256, 1), (32, 2048, 14336, 1024, 0, 2)])
def test_split_kernel_has_the_bits_of_the_other_tensor_core_kernels(aser, M, more, N, K, r, kernel):
    """The first tokens of a call that another kernel serves: integer sums, and the low-rank chunks in order."""
    assert [aser.lib.aser_linear_kernel(m, N, K) for m in (M, more)] == [3, kernel]
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + r)
    Xq = torch.randint(-127, 128, (more, K), device="cuda", dtype=torch.int8, generator=g)
    a = torch.rand(more, device="cuda", generator=g) * 1e-3
    T = torch.randn(more, max(r, 1), device="cuda", generator=g).bfloat16()
    Wq, sc = aser.pack_w4(torch.randn(N, K, device="cuda", generator=g).half(), None)
    Wk, LB = aser.repack_w4(Wq), torch.randn(N, max(r, 1), device="cuda", generator=g).half() * 0.1
    ws = aser.new_workspace(more, N, K, r)
    Y = [aser.linear_w4a8_lr(Xq[:m], a[:m], Wk, sc, T[:m], LB, N, ws) if r else aser.linear_w4a8(Xq[:m], a[:m], Wk, sc, N, ws)
         for m in (M, more)]
    assert torch.equal(Y[0], Y[1][:M])
    if r and N % 256 == 0:          # the same channels as a fused group of two layers, each with its columns of T
        import ctypes as C
        T2 = torch.randn(M, 2 * r, device="cuda", generator=g).bfloat16()
        P = lambda t: C.c_void_p(t.data_ptr())
        Yc = torch.empty((M, N), device="cuda", dtype=torch.float16)
        h = N // 2
        rc = aser.lib.aser_linear_w4a8_lr_cat(P(Xq), P(a), P(Wk), P(sc), P(T2), P(LB), 2, (C.c_int * 2)(h, h), r, M, K, P(Yc),
                                              P(ws), ws.numel(), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        for i in range(2):
            y = aser.linear_w4a8_lr(Xq[:M], a[:M], Wk, sc, T2[:, i * r:(i + 1) * r].contiguous(), LB, N, ws)
            assert torch.equal(Yc[:, i * h:(i + 1) * h], y[:, i * h:(i + 1) * h])
    aser.check_status(ws)
