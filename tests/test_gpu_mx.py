"""GPU parity of the block-scaled (MX) FP8 path against the oracle.

- fp8_quantize_mx: codes and E8M0 scales bit-exact against the oracle's
  mx_quantize (row-major scales) for E4M3 and E5M2, ragged shapes, zero
  blocks, huge, tiny and subnormal inputs; the tiled layout equals the
  oracle's scales placed by the header's layout formula (written out here).
- fp8_mx_scales_to_tiled: the oracle's row-major scales, tiled on the GPU.
- gemm_fp8_mx: structured cases first (scales varying by row group, by
  column group and by 32-element block, so a misplaced scale shows as a
  pattern), then small-integer inputs bit-exact against the FP64 oracle
  (every partial sum an integer below 2^24), then N(0,1) inputs within the
  FP32 / BF16 tolerances of tests/parity.py, all four format pairings, the
  swapped skinny path, and a large product checked on row/column blocks.
"""
import numpy as np
import pytest
import torch

import workloads
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2602_10262_gb300 as gb
    gb.library()
    return gb


def tiled_layout(sc_rowmajor, rows, cols):
    """The tiled scale layout of include/gb300fp8.h, from row-major scales."""
    kb = (cols + 127) // 128
    rt = (rows + 127) // 128
    out = np.full(rt * kb * 512, 127, np.uint8)
    r = np.arange(rows)[:, None]
    b = np.arange(cols // 32)[None, :]
    off = 512 * ((r // 128) * kb + b // 4) + 16 * (r % 32) + 4 * ((r % 128) // 32) + b % 4
    out[off] = sc_rowmajor
    return out


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _mx_inputs(rows, cols, seed):
    x = workloads.randn_f32((rows, cols), seed=seed)
    # vary the block magnitudes over many binades, with zero, tiny and huge blocks
    g = np.random.default_rng(seed)
    mag = 2.0 ** g.integers(-30, 30, size=(rows, cols // 32)).astype(np.float32)
    x = (x.reshape(rows, cols // 32, 32) * mag[:, :, None]).reshape(rows, cols).astype(np.float32)
    if rows > 2 and cols >= 96:
        x[0, :32] = 0.0                                   # an all-zero block
        x[0, 32:64] = -0.0
        x[1, 32:64] *= np.float32(2.0 ** -130)            # subnormal block
        x[2, 64:96] = np.float32(3.0e38)                  # near fp32 max
    return x


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 32), (130, 160), (256, 512), (77, 4096), (300, 96)])
def test_mx_quantize_bit_exact(gb, orc, fmt, rows, cols):
    x = _mx_inputs(rows, cols, seed=rows * 7 + cols + fmt)
    q_ref, s_ref = orc.mx_quantize(x, fmt)
    xd = _dev(x)
    q, s = gb.fp8_quantize_mx(xd, fmt, scale_layout=0)
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    assert np.array_equal(q.cpu().numpy(), q_ref)
    assert np.array_equal(s.cpu().numpy(), s_ref)
    q2, st = gb.fp8_quantize_mx(xd, fmt, scale_layout=1)
    torch.cuda.synchronize()
    assert np.array_equal(q2.cpu().numpy(), q_ref)
    assert np.array_equal(st.cpu().numpy(), tiled_layout(s_ref, rows, cols))
    # the layout converter gives the same tiled array from row-major scales
    st2 = gb.fp8_mx_scales_to_tiled(_dev(s_ref), rows, cols)
    torch.cuda.synchronize()
    assert np.array_equal(st2.cpu().numpy(), tiled_layout(s_ref, rows, cols))


def test_mx_quantize_rejects_nonfinite(gb):
    x = torch.zeros((4, 64), device="cuda")
    x[2, 40] = float("inf")
    gb.fp8_quantize_mx(x, 0)
    assert gb.fp8_last_device_error() == -4


def _gemm(gb, A, SA, B, SB, fmt=(0, 0), alpha=1.0, out_dtype=0):
    M, K = A.shape
    N = B.shape[0]
    C = gb.gemm_fp8_mx(_dev(A), _dev(tiled_layout(SA, M, K)), _dev(B), _dev(tiled_layout(SB, N, K)), alpha,
                       out_dtype, fmt[0], fmt[1])
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    return C.float().cpu().numpy()


ONE = 0x38          # E4M3 1.0


@pytest.mark.parametrize("case", ["a_rows", "a_blocks", "b_cols", "b_blocks"])
def test_mx_structured_scales(gb, orc, case):
    """All codes 1.0; scales 2^j with j set by A's row group, A's 32-element
    block, B's row (output column) group or B's block."""
    M, N, K = 256, 256, 256
    A = np.full((M, K), ONE, np.uint8)
    B = np.full((N, K), ONE, np.uint8)
    SA = np.full((M, K // 32), 127, np.uint8)
    SB = np.full((N, K // 32), 127, np.uint8)
    if case == "a_rows":
        SA += ((np.arange(M) // 32) % 8).astype(np.uint8)[:, None]
    elif case == "a_blocks":
        SA += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    elif case == "b_cols":
        SB += ((np.arange(N) // 32) % 8).astype(np.uint8)[:, None]
    else:
        SB += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    C = _gemm(gb, A, SA, B, SB)
    ref = orc.gemm_mx(A, SA, B, SB)
    assert np.array_equal(C.astype(np.float64), ref), (C[::32, ::32], ref[::32, ::32])


@pytest.mark.parametrize("fmt", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K", [(256, 256, 256), (200, 72, 320), (128, 384, 1024), (16, 512, 2048),
                                   (300, 130, 4096)])
def test_mx_small_integers_bit_exact(gb, orc, fmt, M, N, K):
    A = workloads.small_int_codes((M, K), seed=M + K, fmt=fmt[0])
    B = workloads.small_int_codes((N, K), seed=N + K + 1, fmt=fmt[1])
    g = np.random.default_rng(M * N + K)
    SA = g.integers(127, 129, size=(M, K // 32)).astype(np.uint8)      # scales 1 or 2
    SB = g.integers(126, 128, size=(N, K // 32)).astype(np.uint8)      # scales 1/2 or 1
    C = _gemm(gb, A, SA, B, SB, fmt)
    ref = orc.gemm_mx(A, SA, B, SB, a_fmt=fmt[0], b_fmt=fmt[1])
    assert np.array_equal(C.astype(np.float64), ref)


@pytest.mark.parametrize("fmt", [(0, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("M,N,K", [(256, 256, 256), (1000, 600, 1024), (64, 2048, 1024), (512, 512, 4096)])
def test_mx_normal_inputs(gb, orc, fmt, M, N, K):
    x = workloads.randn_f32((M, K), seed=M + 3)
    w = workloads.randn_f32((N, K), seed=N + 4)
    A, SA = orc.mx_quantize(x, fmt[0])
    B, SB = orc.mx_quantize(w, fmt[1])
    ref = orc.gemm_mx(A, SA, B, SB, alpha=0.75, a_fmt=fmt[0], b_fmt=fmt[1])
    C = _gemm(gb, A, SA, B, SB, fmt, alpha=0.75, out_dtype=0)
    parity.check_fp32(C, ref)
    Cb = _gemm(gb, A, SA, B, SB, fmt, alpha=0.75, out_dtype=1)
    S = orc.gemm_mx(parity.abs_codes(A), SA, parity.abs_codes(B), SB, alpha=0.75, a_fmt=fmt[0],
                    b_fmt=fmt[1])
    parity.check_bf16(Cb, ref, S, K)


@pytest.mark.parametrize("M,N,K", [(1024, 1024, 1024), (16, 4096, 4096)])
def test_mx_pipeline_quantized_on_gpu(gb, orc, M, N, K):
    """fp32 -> fp8_quantize_mx (tiled scales) -> gemm_fp8_mx on the GPU,
    against the oracle's quantisation and product."""
    x = workloads.randn_f32((M, K), seed=11)
    w = workloads.randn_f32((N, K), seed=12)
    A, SAt = gb.fp8_quantize_mx(_dev(x), 0, scale_layout=1)
    B, SBt = gb.fp8_quantize_mx(_dev(w), 0, scale_layout=1)
    C = gb.gemm_fp8_mx(A, SAt, B, SBt, 1.0, gb.OUT_F32)
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    Ao, SAo = orc.mx_quantize(x, 0)
    Bo, SBo = orc.mx_quantize(w, 0)
    assert np.array_equal(A.cpu().numpy(), Ao) and np.array_equal(B.cpu().numpy(), Bo)
    parity.check_fp32(C.cpu().numpy(), orc.gemm_mx(Ao, SAo, Bo, SBo))


def test_mx_large_blocks(gb, orc):
    """8192^3 on the GPU; the oracle takes the first and last 128 rows of A
    against the first and last 128 rows of B (four 128 x 128 blocks)."""
    M = N = K = 8192
    x = workloads.randn_f32((M, K), seed=21)
    w = workloads.randn_f32((N, K), seed=22)
    A, SAt = gb.fp8_quantize_mx(_dev(x), 0, scale_layout=1)
    B, SBt = gb.fp8_quantize_mx(_dev(w), 0, scale_layout=1)
    C = gb.gemm_fp8_mx(A, SAt, B, SBt, 1.0, gb.OUT_BF16)
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    C = C.float().cpu().numpy()
    rows = np.r_[0:128, M - 128:M]
    Ao, SAo = orc.mx_quantize(x[rows], 0)
    Bo, SBo = orc.mx_quantize(w[rows], 0)
    ref = orc.gemm_mx(Ao, SAo, Bo, SBo)
    S = orc.gemm_mx(parity.abs_codes(Ao), SAo, parity.abs_codes(Bo), SBo)
    parity.check_bf16(C[np.ix_(rows, rows)], ref, S, K)


# Shapes whose N tiles are 256 wide (the planner keeps 256 while 2 x row
# blocks x column blocks reach the SM count): one accumulator, B's scales
# in two 128-row chunks per k-block, ring after the accumulator.  N = 800
# leaves the last tile's second 128-row scale chunk outside B (not loaded).
WIDE = [(4096, 1024, 256), (4096, 1000, 640), (4096, 800, 1024)]


def test_mx_wide_tiles_are_planned(gb):
    for M, N, K in WIDE:
        info = gb.gemm_fp8_mx_plan(M, N, K)
        assert info["mt"] == 1 and info["bn"] == 256 and info["cluster"] == 0, (M, N, K, info)
    assert gb.gemm_fp8_mx_plan(1024, 1024, 1024)["bn"] == 128


@pytest.mark.parametrize("case", ["a_rows", "a_blocks", "b_cols", "b_blocks"])
def test_mx_wide_tiles_structured_scales(gb, orc, case):
    M, N, K = 4096, 1024, 256
    A = np.full((M, K), ONE, np.uint8)
    B = np.full((N, K), ONE, np.uint8)
    SA = np.full((M, K // 32), 127, np.uint8)
    SB = np.full((N, K // 32), 127, np.uint8)
    if case == "a_rows":
        SA += ((np.arange(M) // 32) % 8).astype(np.uint8)[:, None]
    elif case == "a_blocks":
        SA += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    elif case == "b_cols":
        SB += ((np.arange(N) // 32) % 8).astype(np.uint8)[:, None]
    else:
        SB += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    C = _gemm(gb, A, SA, B, SB)
    rows = np.r_[0:160, M - 160:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB)
    assert np.array_equal(C[rows].astype(np.float64), ref), (C[rows][::32, ::32], ref[::32, ::32])


@pytest.mark.parametrize("fmt", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K", WIDE)
def test_mx_wide_tiles_small_integers_bit_exact(gb, orc, fmt, M, N, K):
    A = workloads.small_int_codes((M, K), seed=M + K + 3, fmt=fmt[0])
    B = workloads.small_int_codes((N, K), seed=N + K + 4, fmt=fmt[1])
    g = np.random.default_rng(M + N + K)
    SA = g.integers(127, 129, size=(M, K // 32)).astype(np.uint8)
    SB = g.integers(126, 128, size=(N, K // 32)).astype(np.uint8)
    C = _gemm(gb, A, SA, B, SB, fmt)
    rows = np.r_[0:128, 1900:2100, M - 128:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB, a_fmt=fmt[0], b_fmt=fmt[1])
    assert np.array_equal(C[rows].astype(np.float64), ref)


@pytest.mark.parametrize("M,N,K", WIDE)
def test_mx_wide_tiles_normal_inputs(gb, orc, M, N, K):
    x = workloads.randn_f32((M, K), seed=M + 13)
    w = workloads.randn_f32((N, K), seed=N + 14)
    A, SA = orc.mx_quantize(x, 0)
    B, SB = orc.mx_quantize(w, 0)
    rows = np.r_[0:128, M - 256:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB, alpha=0.5)
    C = _gemm(gb, A, SA, B, SB, alpha=0.5, out_dtype=0)
    parity.check_fp32(C[rows], ref)
    Cb = _gemm(gb, A, SA, B, SB, alpha=0.5, out_dtype=1)
    S = orc.gemm_mx(parity.abs_codes(A[rows]), SA[rows], parity.abs_codes(B), SB, alpha=0.5)
    parity.check_bf16(Cb[rows], ref, S, K)


# CTA pairs (256 x 256 tiles over two CTAs, each holding its 128 rows of A
# and of B, their scale chunks loaded by TMA into each CTA's tensor memory):
# problems whose 256-row tiles fill the SMs.  Ragged N and M put part of the
# odd CTA's half outside B or A.
PAIRS = [(4096, 2048, 256), (4096, 2000, 640), (4000, 2048, 1024)]


def test_mx_pairs_are_planned(gb):
    for M, N, K in PAIRS + [(8192, 8192, 8192)]:
        info = gb.gemm_fp8_mx_plan(M, N, K)
        assert info["mt"] == 3 and info["bn"] == 256 and info["cluster"] == 2, (M, N, K, info)


@pytest.mark.parametrize("case", ["a_rows", "a_blocks", "b_cols", "b_blocks"])
def test_mx_pairs_structured_scales(gb, orc, case):
    M, N, K = PAIRS[0]
    A = np.full((M, K), ONE, np.uint8)
    B = np.full((N, K), ONE, np.uint8)
    SA = np.full((M, K // 32), 127, np.uint8)
    SB = np.full((N, K // 32), 127, np.uint8)
    if case == "a_rows":
        SA += ((np.arange(M) // 32) % 8).astype(np.uint8)[:, None]
    elif case == "a_blocks":
        SA += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    elif case == "b_cols":
        SB += ((np.arange(N) // 32) % 8).astype(np.uint8)[:, None]
    else:
        SB += (np.arange(K // 32) % 8).astype(np.uint8)[None, :]
    C = _gemm(gb, A, SA, B, SB)
    rows = np.r_[0:288, M - 160:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB)
    assert np.array_equal(C[rows].astype(np.float64), ref), (C[rows][::32, ::32], ref[::32, ::32])


@pytest.mark.parametrize("fmt", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K", PAIRS)
def test_mx_pairs_small_integers_bit_exact(gb, orc, fmt, M, N, K):
    A = workloads.small_int_codes((M, K), seed=M + K + 5, fmt=fmt[0])
    B = workloads.small_int_codes((N, K), seed=N + K + 6, fmt=fmt[1])
    g = np.random.default_rng(M + 2 * N + K)
    SA = g.integers(127, 129, size=(M, K // 32)).astype(np.uint8)
    SB = g.integers(126, 128, size=(N, K // 32)).astype(np.uint8)
    C = _gemm(gb, A, SA, B, SB, fmt)
    rows = np.r_[0:300, 1900:2100, M - 300:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB, a_fmt=fmt[0], b_fmt=fmt[1])
    assert np.array_equal(C[rows].astype(np.float64), ref)


@pytest.mark.parametrize("M,N,K", PAIRS)
def test_mx_pairs_normal_inputs(gb, orc, M, N, K):
    x = workloads.randn_f32((M, K), seed=M + 23)
    w = workloads.randn_f32((N, K), seed=N + 24)
    A, SA = orc.mx_quantize(x, 0)
    B, SB = orc.mx_quantize(w, 0)
    rows = np.r_[0:256, M - 256:M]
    ref = orc.gemm_mx(A[rows], SA[rows], B, SB, alpha=0.5)
    C = _gemm(gb, A, SA, B, SB, alpha=0.5, out_dtype=0)
    parity.check_fp32(C[rows], ref)
    Cb = _gemm(gb, A, SA, B, SB, alpha=0.5, out_dtype=1)
    S = orc.gemm_mx(parity.abs_codes(A[rows]), SA[rows], parity.abs_codes(B), SB, alpha=0.5)
    parity.check_bf16(Cb[rows], ref, S, K)


def test_mx_pairs_stalled_launch_times_out(gb):
    """The failure path on block-scaled pairs: loads withheld, every wait
    bounded (50 ms here), FP8_ERR_TIMEOUT recorded, C unwritten, and the
    next launch exact."""
    M, N, K = PAIRS[0]
    A = workloads.small_int_codes((M, K), seed=41)
    B = workloads.small_int_codes((N, K), seed=42)
    SA = np.full((M, K // 32), 127, np.uint8)
    SB = np.full((N, K // 32), 128, np.uint8)
    ref = _gemm(gb, A, SA, B, SB)
    At, Bt = _dev(A), _dev(B)
    SAt, SBt = _dev(tiled_layout(SA, M, K)), _dev(tiled_layout(SB, N, K))
    C = torch.full((M, N), float("nan"), device="cuda")
    gb.fp8_test_stall_gemm_loads(1, 50.0)
    try:
        gb.gemm_fp8_mx(At, SAt, Bt, SBt, 1.0, gb.OUT_F32, C=C)
        assert gb.fp8_last_device_error() == -7
    finally:
        gb.fp8_test_stall_gemm_loads(0, 0.0)
    assert torch.isnan(C).all()
    gb.gemm_fp8_mx(At, SAt, Bt, SBt, 1.0, gb.OUT_F32, C=C)
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    assert np.array_equal(C.cpu().numpy(), ref)


# pairs with one tile each (one accumulator) and with several (accumulators
# with shared columns): odd and even tile counts per pair, one k-block, an
# odd number of k-blocks, a partial last k-block, an unaligned output
@pytest.mark.parametrize("M,N,K,out", [(2560, 2560, 4096, 0), (5120, 2816, 128, 0), (5200, 2800, 416, 1),
                                       (5120, 5001, 672, 0), (7680, 7680, 160, 1)])
def test_mx_pair_tile_counts_exact(gb, M, N, K, out):
    assert gb.gemm_fp8_mx_plan(M, N, K, out)["mt"] == 3
    _check_mx_exact(gb, M, N, K, out)


# skinny products split along K within clusters: partial sums beside the ring
# and in it, two to eight slices, ragged everything
@pytest.mark.parametrize("out", [0, 1])
@pytest.mark.parametrize("M,N,K", [(1, 520, 4096), (16, 8192, 4096), (17, 1029, 4128), (33, 4096, 8192),
                                   (64, 1544, 8224), (100, 777, 8192), (128, 8192, 8192), (128, 256, 16384)])
def test_mx_split_clusters_exact(gb, M, N, K, out):
    plan = gb.gemm_fp8_mx_plan(M, N, K, out)
    assert plan["mt"] == 1 and plan["splits"] > 1, plan
    _check_mx_exact(gb, M, N, K, out)


def _check_mx_exact(gb, M, N, K, out):
    """Integers times powers of two: every partial sum is exact in FP32, so
    the product equals float64's."""
    A = _dev(workloads.small_int_codes((M, K), seed=M))
    B = _dev(workloads.small_int_codes((N, K), seed=N + 1))
    g = torch.Generator().manual_seed(K)

    def scales(rows):
        s = torch.randint(126, 129, (rows, K // 32), generator=g, dtype=torch.int32).to(torch.uint8).cuda()
        return s, gb.fp8_mx_scales_to_tiled(s, rows, K)

    def value(codes, s):
        v = codes.view(torch.float8_e4m3fn).double().reshape(codes.shape[0], K // 32, 32)
        return (v * torch.exp2(s.double() - 127)[:, :, None]).reshape(codes.shape)

    (sa, ta), (sb, tb) = scales(M), scales(N)
    C = gb.gemm_fp8_mx(A, ta, B, tb, out_dtype=out)
    assert gb.fp8_last_device_error() == 0
    ref = value(A, sa) @ value(B, sb).T
    if out == gb.OUT_F32:
        assert torch.equal(C.double(), ref)
    else:
        assert torch.equal(C, ref.float().bfloat16())


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 32), (3, 224), (129, 256), (5, 288), (128, 384), (300, 4128)])
def test_mx_quantize_alignments(gb, orc, layout, rows, cols):
    """256-column windows that end in a row, padding rows, and every row
    alignment of x and q; bytes between q's rows untouched."""
    x = _mx_inputs(rows, cols, seed=rows + cols)
    q_ref, s_ref = orc.mx_quantize(x, 0)
    want = s_ref if layout == 0 else tiled_layout(s_ref, rows, cols)
    for pad, off, qpad, qoff in ((0, 0, 0, 0), (4, 4, 4, 4), (1, 1, 1, 1)):
        xb = torch.full((rows * (cols + pad) + off,), float("nan"), device="cuda")
        xt = xb[off:].view(rows, cols + pad)[:, :cols]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((rows * (cols + qpad) + qoff,), 0xA5, dtype=torch.uint8, device="cuda")
        qt = qb[qoff:].view(rows, cols + qpad)[:, :cols]
        _, s = gb.fp8_quantize_mx(xt, 0, scale_layout=layout, q=qt)
        assert np.array_equal(qt.cpu().numpy(), q_ref)
        assert np.array_equal(s.cpu().numpy(), want)
        assert bool((qb[qoff:].view(rows, cols + qpad)[:, cols:] == 0xA5).all())
    assert gb.fp8_last_device_error() == 0


# rows: one column of tiles of each width, odd ones among them; N: few tiles
# in many slices, as many clusters of eight as there are SMs / 8, and more
# than fit; K from the first split length up
@pytest.mark.parametrize("M", [1, 16, 17, 33, 48, 64, 70, 96, 100, 127, 128])
def test_mx_needs_no_workspace(gb, M):
    """gemm_fp8_mx promises to need none: a product split along K adds its
    slices up within clusters, whatever its size."""
    for N in (129, 256, 777, 1024, 2048, 2176, 2304, 2432, 3000, 4096, 8192, 9728, 14336):
        for K in (4096, 4128, 8192, 14336, 16384, 32768):
            plan = gb.gemm_fp8_mx_plan(M, N, K)
            assert plan["workspace_bytes"] == 0, (N, K, plan)
            assert plan["splits"] == 1 or plan["cluster"] == plan["splits"], (N, K, plan)


@pytest.mark.parametrize("out", [0, 1])
@pytest.mark.parametrize("M,N,K", [(128, 1024, 8192), (128, 2048, 8192), (64, 2048, 8192), (96, 2048, 14336),
                                   (70, 1024, 8192), (48, 2432, 8192), (16, 2432, 8192)])
def test_mx_few_tiles_split_exact(gb, M, N, K, out):
    assert gb.gemm_fp8_mx_plan(M, N, K, out)["splits"] > 1
    _check_mx_exact(gb, M, N, K, out)


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 32), (5, 288), (130, 512), (129, 4128)])
def test_mx_quantize_mixed_alignments(gb, orc, layout, fmt, rows, cols):
    """x and q of different alignment (either may rule the whole vectors
    out); blocks of zeros, and a non-finite value reported from either form."""
    x = _mx_inputs(rows, cols, seed=rows + cols)
    x[rows - 1, :32] = 0.0
    q_ref, s_ref = orc.mx_quantize(x, fmt)
    want = s_ref if layout == 0 else tiled_layout(s_ref, rows, cols)
    for pad, off, qpad, qoff in ((0, 0, 1, 0), (0, 4, 0, 3), (3, 0, 0, 0), (0, 8, 0, 4)):
        xt = torch.zeros(rows * (cols + pad) + off, device="cuda")[off:].view(rows, cols + pad)[:, :cols]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((rows * (cols + qpad) + qoff,), 0xA5, dtype=torch.uint8, device="cuda")
        qt = qb[qoff:].view(rows, cols + qpad)[:, :cols]
        _, s = gb.fp8_quantize_mx(xt, fmt, scale_layout=layout, q=qt)
        assert np.array_equal(qt.cpu().numpy(), q_ref)
        assert np.array_equal(s.cpu().numpy(), want)
        assert bool((qb[:qoff] == 0xA5).all())
        assert bool((qb[qoff:].view(rows, cols + qpad)[:, cols:] == 0xA5).all())
        assert gb.fp8_last_device_error() == 0
        xt[rows // 2, cols - 1] = float("inf")
        gb.fp8_quantize_mx(xt, fmt, scale_layout=layout, q=qt)
        assert gb.fp8_last_device_error() == -4
