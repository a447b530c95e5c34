"""Per-kernel parity: each operator called through the C ABI against the oracle's definition."""
import numpy as np
import pytest
import torch

from oracle import d3_oracle as o
from paper_2601_07568_b200 import binding as d3
from paper_2601_07568_b200 import synth_inputs as si
from gpu_utils import DEV, Ctx

pytestmark = pytest.mark.gpu

BF16_SHAPE = si.scaled_shape(si.LLADA8B, name="ops-bf16", n_layers=1, d_model=256, n_q_heads=4, n_kv_heads=2,
                             d_ffn=512, vocab=1000, d_head=64)
F32_SHAPE = si.scaled_shape(si.TINY, name="ops-f32", n_layers=1, d_model=128, n_q_heads=4, n_kv_heads=2,
                            d_ffn=256, vocab=1000, d_head=32)


@pytest.fixture(scope="module")
def ctx_bf16():
    with Ctx(BF16_SHAPE, None, block=32, max_batch=32, max_seq=640) as c:
        yield c


@pytest.fixture(scope="module")
def ctx_f32():
    with Ctx(F32_SHAPE, None, block=16, max_batch=8, max_seq=256) as c:
        yield c


def rand_bf16(rng, shape, scale=1.0):
    x = (rng.standard_normal(shape) * scale).astype(np.float32)
    t = torch.from_numpy(x).to(torch.bfloat16)
    return t, t.float().numpy().astype(np.float64)


def swiglu_ref(y, n):
    # packed columns: 2j = gate of hidden unit j, 2j+1 = its up value
    return o.silu(y[:, 0::2]) * y[:, 1::2]


LINEAR_SHAPES = [(32, 9000, 128), (32, 256, 128), (16, 128, 64), (48, 200, 192), (130, 384, 256), (1, 128, 4096), (32, 4096, 4096),
                 (256, 640, 1024), (1024, 256, 512)]


@pytest.mark.parametrize("m,n,k", LINEAR_SHAPES)
@pytest.mark.parametrize("splits", [0, 1, 3, 7, 148])
def test_linear_bf16_tensor_core(ctx_bf16, m, n, k, splits):
    rng = np.random.default_rng(m * 7 + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    # fp32 out
    y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y, 0, splits)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
    # residual: y += x w^T
    y0 = rng.standard_normal((m, n)).astype(np.float32)
    y = torch.from_numpy(y0).to(DEV)
    d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y, 2, splits)
    assert np.max(np.abs(y.cpu().numpy() - (ref + y0))) <= tol + 1e-6
    # bf16 out
    y = torch.zeros((m, n), dtype=torch.bfloat16, device=DEV)
    d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y, 1, splits)
    assert np.max(np.abs(y.float().cpu().numpy() - ref)) <= tol + 2 ** -8 * np.abs(ref).max()
    # SwiGLU
    if n % 2 == 0:
        y = torch.zeros((m, n // 2), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y, 3, splits)
        sref = swiglu_ref(ref, n)
        assert np.max(np.abs(y.float().cpu().numpy() - sref)) <= 2 ** -7 * np.abs(sref).max() + 4 * tol
    assert ctx_bf16.error_word() == 0


@pytest.mark.parametrize("m,n,k", [(32, 9000, 128), (48, 200, 192), (130, 384, 256), (1, 128, 4096), (32, 4096, 4096),
                                   (7, 100, 72), (256, 640, 1024)])
@pytest.mark.parametrize("splits", [0, 1, 5])
def test_linear_bf16_packed_weights(ctx_bf16, m, n, k, splits):
    """Weights in the tiled layout (contiguous 128 x 64 blocks, zero-padded) give the same products as
    the row-major form, ragged edges included."""
    rng = np.random.default_rng(m * 11 + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    packed = torch.full((d3.d3_packed_weight_elems(n, k),), 3.0, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wd, packed)
    y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, splits)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
    y2 = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y2, 0, splits)
    if not (128 < m <= 256 and n % 128 == 0 and splits == 0):  # (there the packed form takes the weights-as-rows kernel)
        assert torch.equal(y, y2)  # same units, same order of sums: identical bits
    if n % 2 == 0:
        h = torch.zeros((m, n // 2), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, h, n, 3, splits)
        want = swiglu_ref(ref, n)
        assert np.max(np.abs(h.float().cpu().numpy() - want)) <= 2 ** -7 * np.abs(want).max() + tol
    assert ctx_bf16.error_word() == 0


@pytest.mark.parametrize("m,n,k,cluster", [(130, 384, 256, 1), (256, 512, 2048, 8), (200, 1024, 1024, 4), (192, 256, 512, 2),
                                           (256, 3584, 3584, 4), (129, 128, 4096, 8), (256, 4096, 1024, 4), (160, 12288, 256, 1)])
def test_linear_bf16_weights_as_rows(ctx_bf16, m, n, k, cluster):
    """Matmuls of 129..256 rows with at most one 128-column tile per SM: the weights are the MMA's 128-row
    operand, all rows of X its column operand, a cluster per tile splits K (1, 2, 4 or 8 parts) and adds
    the staged partial sums in rank order.  fp32, bf16 and residual epilogues against the fp64 product;
    the residual epilogue also leaves the bf16 copy and the chunk sums of squares of the rows (checked
    through a second matmul that uses them: the folded RMSNorm factor)."""
    rng = np.random.default_rng(m + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    packed = torch.full((d3.d3_packed_weight_elems(n, k),), 3.0, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wd, packed)
    n0 = d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_xt_kernel")
    y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, 0)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
    y0 = rng.standard_normal((m, n)).astype(np.float32)
    y = torch.from_numpy(y0).to(DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 2, 0)
    assert np.max(np.abs(y.cpu().numpy() - (ref + y0))) <= tol + 1e-6
    y = torch.zeros((m, n), dtype=torch.bfloat16, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 1, 0)
    assert np.max(np.abs(y.float().cpu().numpy() - ref)) <= tol + 2 ** -8 * np.abs(ref).max()
    assert d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_xt_kernel") == n0 + 3
    # the same through the unit-range kernel (switch off): same products up to the order of the fp32 sums
    d3.d3_set_tuning(ctx_bf16.ctx, weights_as_rows=0)
    y2 = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y2, n, 0, 0)
    d3.d3_set_tuning(ctx_bf16.ctx)
    assert d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_xt_kernel") == n0 + 3
    assert np.max(np.abs(y2.cpu().numpy() - ref)) <= tol
    assert ctx_bf16.error_word() == 0


@pytest.mark.parametrize("m,n,k", [(1, 16, 4), (16, 128, 512), (17, 130, 260), (33, 384, 128), (48, 200, 1028), (5, 514, 64), (3, 96, 256), (9, 48, 292)])
@pytest.mark.parametrize("epi", [0, 2, 3])
def test_linear_fp32_small_tiles_same_bits(ctx_f32, m, n, k, epi):
    """fp32 matmuls of few tiles run on 16 x 16 tiles: against the fp64 product, and bit for bit what a matmul of many
    rows (the 32 x 128 tiles) gives for the same rows, since a sum is one chain of multiply-adds in either."""
    rng = np.random.default_rng(m + n + k + epi)
    big = (74 * 32 // ((n + 127) // 128) + 32) // 32 * 32 + 32  # rows at which the tiles are more than half the SMs
    x = rng.standard_normal((big, k)).astype(np.float32)
    w = (rng.standard_normal((n, k)) * 0.05).astype(np.float32)
    y0 = rng.standard_normal((big, n // 2 if epi == 3 else n)).astype(np.float32)
    xd, wd = torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV)
    few, many = torch.from_numpy(y0[:m]).to(DEV), torch.from_numpy(y0).to(DEV)
    n0 = d3.d3_launch_count_of(ctx_f32.ctx, "gemm_simt_small_kernel")
    d3.d3_op_linear(ctx_f32.ctx, xd[:m].contiguous(), wd, few, epi, 0)
    assert d3.d3_launch_count_of(ctx_f32.ctx, "gemm_simt_small_kernel") == n0 + 1
    d3.d3_op_linear(ctx_f32.ctx, xd, wd, many, epi, 0)
    assert d3.d3_launch_count_of(ctx_f32.ctx, "gemm_simt_small_kernel") == n0 + 1
    assert torch.equal(few, many[:m])
    ref = x[:m].astype(np.float64) @ w.T.astype(np.float64)
    want = ref + y0[:m] if epi == 2 else swiglu_ref(ref, n) if epi == 3 else ref
    assert np.max(np.abs(few.cpu().numpy() - want)) <= 1e-6 * np.sqrt(k) * (np.abs(ref).max() ** (2 if epi == 3 else 1) + 1) + 1e-6


@pytest.mark.parametrize("m,n,k", [(1, 256, 64), (32, 512, 4096), (33, 3584, 3584), (96, 256, 8192), (128, 12288, 512), (129, 4096, 1024),
                                   (200, 768, 2048), (256, 4096, 4096), (257, 1280, 1920), (501, 3584, 1024), (640, 19200, 256),
                                   (96, 19456, 256), (288, 21760, 1024)])
def test_linear_bf16_k_cut_pairs(ctx_bf16, m, n, k):
    """Weights as the row operand of CTA pairs with the tiles of an incomplete wave cut along K: one tile and no cut,
    one tile shared by all pairs, ranges that touch two tiles, a whole wave behind cut tiles (640 x 19200, 288 x 21760), a
    wave and two tiles none of which is cut (96 x 19456), one to three tiles of rows, row counts on both sides of a multiple of 16, 32 and 256; fp32, residual, bf16 and SwiGLU
    epilogues against the fp64 product (bounds as in the other matmul tests), twice with the same bits."""
    rng = np.random.default_rng(m + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    packed = torch.full((d3.d3_packed_weight_elems(n, k),), 3.0, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wd, packed)
    d3.d3_set_k_cut_pairs(ctx_bf16.ctx, 1)
    try:
        n0 = d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_sk_kernel")
        y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, 0)
        assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
        y2 = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y2, n, 0, 0)
        assert torch.equal(y, y2)
        y0 = rng.standard_normal((m, n)).astype(np.float32)
        yr = torch.from_numpy(y0).to(DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, yr, n, 2, 0)
        assert np.max(np.abs(yr.cpu().numpy() - (ref + y0))) <= tol + 1e-6
        yb = torch.zeros((m, n), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, yb, n, 1, 0)
        assert np.max(np.abs(yb.float().cpu().numpy() - ref)) <= tol + 2 ** -8 * np.abs(ref).max()
        h = torch.zeros((m, n // 2), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, h, n, 3, 0)
        want = swiglu_ref(ref, n)
        assert np.max(np.abs(h.float().cpu().numpy() - want)) <= 2 ** -7 * np.abs(want).max() + tol
        assert d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_sk_kernel") == n0 + 5
    finally:
        d3.d3_set_k_cut_pairs(ctx_bf16.ctx, -1)
    assert ctx_bf16.error_word() == 0


def test_tensor_maps_of_thousands_of_buffers(ctx_bf16):
    """One operand against 4400 others at other addresses: the maps kept for earlier calls are dropped in between, never
    under a call that uses one."""
    rng = np.random.default_rng(11)
    _, x = rand_bf16(rng, (160, 64))
    xd = torch.from_numpy(x).to(torch.bfloat16).to(DEV)
    size = d3.d3_packed_weight_elems(256, 64)
    wt, w = rand_bf16(rng, (256, 64), 0.05)
    one = torch.zeros(size, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wt.to(DEV), one)
    want, room = x @ w.T, torch.zeros(size + 8 * 4400, dtype=torch.bfloat16, device=DEV)
    y = torch.zeros((160, 256), dtype=torch.float32, device=DEV)
    for i in range(4400):
        packed = room[8 * i:8 * i + size]
        if i % 40 == 0 or i > 4050:
            packed.copy_(one)
            y.zero_()
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, 256, 0, 0)
        if i % 40 == 0 or i > 4050:
            assert np.max(np.abs(y.cpu().numpy() - want)) <= 2e-5 * 8 * np.abs(want).max() + 1e-6
    assert ctx_bf16.error_word() == 0


@pytest.mark.parametrize("m,n,k", [(512, 256, 64), (1024, 512, 512), (640, 768, 1024), (1000, 256, 4096), (2048, 4096, 1024),
                                   (513, 12288, 256), (256, 19200, 128), (130, 19200, 64)])
def test_linear_bf16_cta_pairs(ctx_bf16, m, n, k):
    """Matmuls of more than 128 rows on tiled weights (the 130- and 256-row cases have more column tiles than the
    weights-as-rows kernel takes): 256 x 256 tiles, each computed by one MMA of 256 rows that a
    pair of CTAs shares (each stages its own 128 rows of X and 128 of the tile's weight rows).  Row counts that end
    inside the leader's half, inside the peer's half and on a tile border; one K slab and many; more tiles than
    pairs (two accumulators in turn) and fewer; fp32, residual, bf16 and SwiGLU epilogues against the fp64 product,
    and the same through single CTAs."""
    rng = np.random.default_rng(m + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    packed = torch.full((d3.d3_packed_weight_elems(n, k),), 3.0, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wd, packed)
    n0 = d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_pair_kernel")
    y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, 0)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
    y0 = rng.standard_normal((m, n)).astype(np.float32)
    yr = torch.from_numpy(y0).to(DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, yr, n, 2, 0)
    assert np.max(np.abs(yr.cpu().numpy() - (ref + y0))) <= tol + 1e-6
    yb = torch.zeros((m, n), dtype=torch.bfloat16, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, yb, n, 1, 0)
    assert np.max(np.abs(yb.float().cpu().numpy() - ref)) <= tol + 2 ** -8 * np.abs(ref).max()
    h = torch.zeros((m, n // 2), dtype=torch.bfloat16, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, h, n, 3, 0)
    want = swiglu_ref(ref, n)
    assert np.max(np.abs(h.float().cpu().numpy() - want)) <= 2 ** -7 * np.abs(want).max() + tol
    assert d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_pair_kernel") == n0 + 4
    # the same through single CTAs (switch off): same products up to the order of the fp32 sums
    d3.d3_set_tuning(ctx_bf16.ctx, cta_pairs=0)
    y2 = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
    d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y2, n, 0, 0)
    d3.d3_set_tuning(ctx_bf16.ctx)
    assert d3.d3_launch_count_of(ctx_bf16.ctx, "gemm_pair_kernel") == n0 + 4
    assert np.max(np.abs(y2.cpu().numpy() - ref)) <= tol
    assert np.max(np.abs(y.cpu().numpy() - y2.cpu().numpy())) <= tol
    assert ctx_bf16.error_word() == 0


@pytest.mark.parametrize("m,n,k,widths", [(32, 2400, 256, [16, 48, 80, 96, 240]), (64, 2400, 200, [48, 160]),
                                          (7, 4736, 1024, [32, 128]), (1, 512, 4096, [16, 256]),
                                          (100, 2400, 256, [48, 240]), (128, 4736, 512, [128, 64])])
def test_linear_bf16_column_strips(ctx_bf16, m, n, k, widths):
    """The column-strip kernel (one CTA per strip of S columns, whole K range) against the fp64 product:
    strips that start and end inside the 128-row weight blocks, span three blocks, end in half a
    32-column chunk; ragged K; all four epilogues."""
    rng = np.random.default_rng(m * 13 + n + k)
    xt, x = rand_bf16(rng, (m, k))
    wt, w = rand_bf16(rng, (n, k), 0.05)
    ref = x @ w.T
    tol = 2e-5 * np.sqrt(k) * np.abs(ref).max() + 1e-6
    xd, wd = xt.to(DEV), wt.to(DEV)
    packed = torch.full((d3.d3_packed_weight_elems(n, k),), 3.0, dtype=torch.bfloat16, device=DEV)
    d3.d3_pack_weight(ctx_bf16.ctx, wd, packed)
    y0 = rng.standard_normal((m, n)).astype(np.float32)
    sref = swiglu_ref(ref, n)
    for S in widths:
        y = torch.full((m, n), 7.0, dtype=torch.float32, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, -S)
        assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol, S
        y = torch.from_numpy(y0).to(DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 2, -S)
        assert np.max(np.abs(y.cpu().numpy() - (ref + y0))) <= tol + 1e-6, S
        y = torch.zeros((m, n), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 1, -S)
        assert np.max(np.abs(y.float().cpu().numpy() - ref)) <= tol + 2 ** -8 * np.abs(ref).max(), S
        h = torch.zeros((m, n // 2), dtype=torch.bfloat16, device=DEV)
        d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, h, n, 3, -S)
        assert np.max(np.abs(h.float().cpu().numpy() - sref)) <= 2 ** -7 * np.abs(sref).max() + 4 * tol, S
    # widths the kernel cannot take are refused, not rounded
    y = torch.zeros((m, n), dtype=torch.float32, device=DEV)
    for bad in (-24, -272, -(n + 16)):
        with pytest.raises(d3.D3Error):
            d3.d3_op_linear_packed(ctx_bf16.ctx, xd, packed, y, n, 0, bad)
    assert ctx_bf16.error_word() == 0


def test_linear_bf16_repeated_launches_keep_split_counters_clean(ctx_bf16):
    rng = np.random.default_rng(3)
    xt, x = rand_bf16(rng, (32, 1024))
    wt, w = rand_bf16(rng, (256, 1024), 0.05)
    ref = x @ w.T
    xd, wd = xt.to(DEV), wt.to(DEV)
    outs = []
    for _ in range(4):
        y = torch.zeros((32, 256), dtype=torch.float32, device=DEV)
        d3.d3_op_linear(ctx_bf16.ctx, xd, wd, y, 0, 4)
        outs.append(y.cpu().numpy())
    assert all(np.array_equal(outs[0], a) for a in outs[1:])  # deterministic split-K
    assert np.max(np.abs(outs[0] - ref)) <= 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("m,n,k", [(16, 128, 128), (5, 100, 100), (33, 256, 72), (64, 512, 128)])
def test_linear_fp32_simt(ctx_f32, m, n, k):
    rng = np.random.default_rng(m + n + k)
    x = rng.standard_normal((m, k)).astype(np.float32)
    w = (rng.standard_normal((n, k)) * 0.05).astype(np.float32)
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    tol = 2e-6 * np.sqrt(k) * np.abs(ref).max()
    xd, wd = torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV)
    y = torch.zeros((m, n), dtype=torch.float32, device=DEV)
    d3.d3_op_linear(ctx_f32.ctx, xd, wd, y, 0)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol
    y2 = torch.zeros((m, n), dtype=torch.float32, device=DEV)
    d3.d3_op_linear(ctx_f32.ctx, xd, wd, y2, 1)
    assert torch.equal(y, y2)
    d3.d3_op_linear(ctx_f32.ctx, xd, wd, y2, 2)
    assert np.max(np.abs(y2.cpu().numpy() - 2 * ref)) <= 2 * tol
    if n % 2 == 0:
        y3 = torch.zeros((m, n // 2), dtype=torch.float32, device=DEV)
        d3.d3_op_linear(ctx_f32.ctx, xd, wd, y3, 3)
        sref = swiglu_ref(ref, n)
        assert np.max(np.abs(y3.cpu().numpy() - sref)) <= 1e-5 * np.abs(sref).max() + 4 * tol


def _stats_case(ctx, bf16, m, V, k, mask_id, scale, seed):
    rng = np.random.default_rng(seed)
    if bf16:
        xt, x = rand_bf16(rng, (m, k))
        wt, w = rand_bf16(rng, (V, k), 0.05)
    else:
        x32 = rng.standard_normal((m, k)).astype(np.float32)
        w32 = (rng.standard_normal((V, k)) * 0.05).astype(np.float32)
        xt, wt, x, w = torch.from_numpy(x32), torch.from_numpy(w32), x32.astype(np.float64), w32.astype(np.float64)
    lg = scale * (x @ w.T)
    p, conf, tok, ent = o.softmax_stats(lg, mask_id)
    part = np.partition(p, -2, axis=-1)
    gap = part[:, -1] - part[:, -2]
    c = torch.zeros(m, dtype=torch.float32, device=DEV)
    e = torch.zeros(m, dtype=torch.float32, device=DEV)
    a = torch.zeros(m, dtype=torch.int32, device=DEV)
    d3.d3_op_lm_head_stats(ctx.ctx, xt.to(DEV), wt.to(DEV), scale, mask_id, c, e, a)
    c, e, a = c.cpu().numpy(), e.cpu().numpy(), a.cpu().numpy()
    tol = 3e-3 if bf16 else 2e-4
    assert np.max(np.abs(c - conf)) <= tol
    assert np.max(np.abs(e - ent)) <= 3 * tol
    bad = (a != tok) & (gap >= 1e-3)
    assert not bad.any()
    assert np.all(a != mask_id)


@pytest.mark.parametrize("V,mask_id", [(1000, 999), (1000, 500), (512, 511), (128, 0), (300, 130)])
def test_lm_head_stats_bf16(ctx_bf16, V, mask_id):
    _stats_case(ctx_bf16, True, 32, V, 256, mask_id, 20.0, V + mask_id)
    _stats_case(ctx_bf16, True, 17, V, 128, mask_id, 3.0, V + mask_id + 1)


@pytest.mark.parametrize("V,mask_id", [(1000, 999), (512, 511), (77, 3)])
def test_lm_head_stats_fp32(ctx_f32, V, mask_id):
    _stats_case(ctx_f32, False, 16, V, 128, mask_id, 20.0, V)
    _stats_case(ctx_f32, False, 7, V, 100, mask_id, 2.0, V + 1)


def test_lm_head_stats_special_rows(ctx_f32):
    # all-equal logits -> conf = 1/(V-1), H = ln(V-1), token 0; one dominant column -> conf ~ 1, H ~ 0
    V, k = 300, 64
    x = np.zeros((2, k), dtype=np.float32)
    x[1, 0] = 1.0
    w = np.zeros((V, k), dtype=np.float32)
    w[123, 0] = 5.0
    c = torch.zeros(2, dtype=torch.float32, device=DEV)
    e = torch.zeros(2, dtype=torch.float32, device=DEV)
    a = torch.zeros(2, dtype=torch.int32, device=DEV)
    d3.d3_op_lm_head_stats(ctx_f32.ctx, torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV), 20.0, V - 1, c, e, a)
    c, e, a = c.cpu().numpy(), e.cpu().numpy(), a.cpu().numpy()
    assert abs(c[0] - 1.0 / (V - 1)) < 1e-7 and abs(e[0] - np.log(V - 1)) < 1e-5 and a[0] == 0
    assert c[1] > 1 - 1e-6 and e[1] < 1e-5 and a[1] == 123


def _attention_case(ctx, shape, bf16, bs, rows, kv_lens, seed, ramp=0.0):
    rng = np.random.default_rng(seed)
    hq, hkv, dh = shape.n_q_heads, shape.n_kv_heads, shape.d_head
    rnd = (lambda s: rand_bf16(rng, s)) if bf16 else (
        lambda s: (lambda a: (torch.from_numpy(a), a.astype(np.float64)))(rng.standard_normal(s).astype(np.float32)))
    qt, q = rnd((bs * rows, hq * dh))
    refs = []
    for b in range(bs):
        L = kv_lens[b]
        kt, k = rnd((hkv, L, dh))
        if ramp:  # keys grow along the sequence: the running maximum of a row keeps rising from tile to tile
            grow = (1.0 + ramp * np.arange(L))[None, :, None]
            kt = (kt.float() * torch.from_numpy(grow).float()).to(torch.bfloat16)
            k = kt.float().numpy().astype(np.float64)
        vt, v = rnd((hkv, L, dh))
        d3.d3_op_write_kv(ctx.ctx, 0, b, 0, kt.float().to(DEV).contiguous(), vt.float().to(DEV).contiguous())
        qb = q[b * rows:(b + 1) * rows].reshape(rows, hq, dh)
        refs.append(o.attention(qb, k.transpose(1, 0, 2), v.transpose(1, 0, 2)).reshape(rows, hq * dh))
    ref = np.concatenate(refs)
    out = torch.zeros_like(qt, device=DEV)
    d3.d3_op_attention(ctx.ctx, qt.to(DEV), 0, bs, rows, torch.tensor(kv_lens, dtype=torch.int32, device=DEV), out)
    got = out.float().cpu().numpy()
    tol = (2 ** -7 if bf16 else 2e-5) * np.abs(ref).max()
    assert np.max(np.abs(got - ref)) <= tol
    assert ctx.error_word() == 0


@pytest.mark.parametrize("rows,kv_lens", [(32, [64, 33, 1]), (7, [40, 300, 5]), (32, [600, 32, 257])])
def test_attention_bf16(ctx_bf16, rows, kv_lens):
    _attention_case(ctx_bf16, BF16_SHAPE, True, 3, rows, kv_lens, rows + sum(kv_lens))


ATT_GQA = si.scaled_shape(si.QWEN7B, name="att-gqa7", n_layers=1, d_model=256, n_q_heads=14, n_kv_heads=2,
                          d_ffn=256, vocab=1000, d_head=128)
ATT_MHA = si.scaled_shape(si.LLADA8B, name="att-mha", n_layers=1, d_model=256, n_q_heads=3, n_kv_heads=3,
                          d_ffn=256, vocab=1000, d_head=128)


@pytest.mark.parametrize("shape", [ATT_GQA, ATT_MHA], ids=["gqa7", "mha"])
@pytest.mark.parametrize("rows,kv_lens", [(32, [64, 33, 1]), (32, [600, 65, 257]), (64, [640, 63, 128]),
                                          (7, [40, 300, 5]), (100, [100, 37, 129]), (300, [300, 5, 64])])
def test_attention_bf16_tensor_core(shape, rows, kv_lens):
    """d_head 128 runs the TMA-staged tensor-core kernel: decode-sized row counts take several key
    splits (partials merged by the last CTA), prefill-sized ones several query tiles; group 7 packs
    the query heads of one kv head into shared tiles."""
    with Ctx(shape, None, block=32, max_batch=3, max_seq=640, max_prefill_rows=3 * 300) as ctx:
        _attention_case(ctx, shape, True, 3, rows, kv_lens, rows + sum(kv_lens))
        # same inputs again: split counters must have been left clean
        _attention_case(ctx, shape, True, 3, rows, kv_lens, rows + sum(kv_lens))


@pytest.mark.parametrize("shape", [ATT_GQA, ATT_MHA], ids=["gqa7", "mha"])
@pytest.mark.parametrize("rows,kv_lens", [(32, [64, 33, 1]), (32, [600, 65, 257]), (64, [640, 63, 128]),
                                          (7, [40, 300, 5]), (100, [100, 37, 129]), (300, [300, 5, 64]),
                                          (32, [128, 256, 384]), (40, [129, 127, 640])])
@pytest.mark.parametrize("keys_per_tile", [64, 128])
def test_attention_bf16_tensor_memory(shape, rows, kv_lens, keys_per_tile):
    """The same cases on the tcgen05 kernel (S, P, O and Q in tensor memory, V as an MN-major operand), in both
    shapes (64-key tiles with one S buffer, 128-key tiles with two): whole and partly filled 128-row tiles, one to
    ten key tiles, ragged last tiles, key splits over a cluster."""
    with Ctx(shape, None, block=32, max_batch=3, max_seq=640, max_prefill_rows=3 * 300) as ctx:
        d3.d3_set_tuning(ctx.ctx, attention_tmem=keys_per_tile)
        _attention_case(ctx, shape, True, 3, rows, kv_lens, rows + sum(kv_lens))
        _attention_case(ctx, shape, True, 3, rows, kv_lens, rows + sum(kv_lens))
        assert d3.d3_launch_count_of(ctx.ctx, "attn_tmem_kernel") == 2
        # row maxima that rise by far more than 2^8 over the tiles: the reference moves and O is rescaled in place
        _attention_case(ctx, shape, True, 3, rows, kv_lens, 7 + rows + sum(kv_lens), ramp=0.05)


ATT_GQA2 = si.scaled_shape(si.QWEN7B, name="att-gqa2", n_layers=1, d_model=256, n_q_heads=4, n_kv_heads=2,
                           d_ffn=256, vocab=1000, d_head=128)


@pytest.mark.parametrize("shape,rows,bs", [(ATT_MHA, 32, 64), (ATT_MHA, 64, 50), (ATT_GQA2, 32, 90), (ATT_GQA2, 64, 3),
                                           (ATT_MHA, 8, 120), (ATT_MHA, 128, 70)], ids=["mha32", "mha64", "gqa2x32", "gqa2x64", "mha8", "mha128"])
def test_attention_bf16_tensor_memory_persistent(shape, rows, bs):
    """The persistent form: one CTA per SM walks through its (sequence, kv head) pairs and treats their key tiles as
    one stream.  More pairs than SMs (CTAs with one, two and three pairs) and fewer, ragged key ranges from 1 key to
    5 tiles, one or two query heads per kv head, part-filled and full 128-row tiles; then the row maxima that keep
    rising."""
    rng = np.random.default_rng(rows + bs)
    kv_lens = [int(v) for v in rng.integers(1, 640, size=bs)]
    kv_lens[1] = 640
    kv_lens[2] = 128
    kv_lens[5 % bs] = 1
    with Ctx(shape, None, block=32, max_batch=bs, max_seq=640, max_prefill_rows=bs * rows) as ctx:
        d3.d3_set_tuning(ctx.ctx, attention_tmem=2)
        _attention_case(ctx, shape, True, bs, rows, kv_lens, rows + bs)
        _attention_case(ctx, shape, True, bs, rows, kv_lens, rows + bs)
        assert d3.d3_launch_count_of(ctx.ctx, "attn_tmem_stream_kernel") == 2
        _attention_case(ctx, shape, True, bs, rows, kv_lens, 7 + rows + bs, ramp=0.05)


@pytest.mark.parametrize("rows,kv_lens", [(16, [48, 17]), (5, [5, 200])])
def test_attention_fp32(ctx_f32, rows, kv_lens):
    _attention_case(ctx_f32, F32_SHAPE, False, 2, rows, kv_lens, rows)


@pytest.mark.parametrize("mode", [0, 1])
def test_unmask_matches_oracle_decision(mode):
    shape = F32_SHAPE
    with Ctx(shape, None, block=32, max_batch=64, max_seq=64, decide_mode=mode) as c:
        rng = np.random.default_rng(mode)
        bs, B = 64, 32
        grid = np.array([0.05, 0.3, 0.3, 0.6, 0.9, 0.9, 0.95], dtype=np.float32)
        conf = rng.choice(grid, size=(bs, B)).astype(np.float32)
        ent = rng.choice(grid, size=(bs, B)).astype(np.float32)
        tok = rng.integers(0, 900, size=(bs, B)).astype(np.int32)
        mask = rng.random((bs, B)) < 0.6
        mask[0] = False
        mask[1] = True
        ids = np.where(mask, shape.mask_id, 5).astype(np.int32)
        for tau in (0.3, 0.6, 1.0, 0.0):
            t = lambda a, dt: torch.tensor(a, dtype=dt, device=DEV)
            idt, mt = t(ids, torch.int32), t(mask.astype(np.uint8), torch.uint8)
            pos = torch.full((bs, B), -1, dtype=torch.int32, device=DEV)
            oid = torch.full((bs, B), -1, dtype=torch.int32, device=DEV)
            cnt = torch.zeros(bs, dtype=torch.int32, device=DEV)
            d3.d3_op_unmask(c.ctx, t(conf.reshape(-1), torch.float32), t(ent.reshape(-1), torch.float32),
                            t(tok.reshape(-1), torch.int32), idt, mt, tau, pos, oid, cnt)
            idn, mn, pos, oid, cnt = (a.cpu().numpy() for a in (idt, mt, pos, oid, cnt))
            for b in range(bs):
                commit = o.decide(conf[b], ent[b], mask[b], np.float32(tau), mode)
                assert cnt[b] == commit.sum()
                assert np.array_equal(pos[b, :cnt[b]], np.flatnonzero(commit))
                assert np.array_equal(oid[b, :cnt[b]], tok[b][commit])
                assert np.array_equal(mn[b].astype(bool), mask[b] & ~commit)
                assert np.array_equal(idn[b], np.where(commit, tok[b], ids[b]))


def test_argument_errors(ctx_f32):
    L = d3.lib()
    import ctypes as C
    assert L.d3_create(None, None, None) == d3.D3_ERR_INVALID_ARG
    bad = d3.make_config(F32_SHAPE, block=16, max_batch=1, max_seq=64)
    bad.d_head = 48
    out = C.c_void_p(0)
    assert L.d3_create(C.byref(bad), None, C.byref(out)) == d3.D3_ERR_UNSUPPORTED
    ids = torch.zeros((1, 16), dtype=torch.int32, device=DEV)
    m = torch.ones((1, 16), dtype=torch.uint8, device=DEV)
    cnt = torch.zeros(1, dtype=torch.int32, device=DEV)
    with pytest.raises(d3.D3Error) as ei:
        d3.d3_denoise_step(ctx_f32.ctx, ids, m, 0.9, ids.clone(), ids.clone(), cnt)
    assert ei.value.code == d3.D3_ERR_STATE  # no weights / prefill yet
    with pytest.raises(d3.D3Error) as ei:
        d3.d3_denoise_step(ctx_f32.ctx, ids, m, float("nan"), ids.clone(), ids.clone(), cnt)
    assert ei.value.code == d3.D3_ERR_INVALID_ARG
    with pytest.raises(d3.D3Error) as ei:
        d3.d3_prefill(ctx_f32.ctx, ids, cnt)
    assert ei.value.code == d3.D3_ERR_STATE
    assert d3.lib().d3_strerror(-5).decode().startswith("bounded")
