"""GPU parity: fp8_quantize_e4m3 (scale selection + E4M3 encode) against the
oracle, bit-exact on codes and scales."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2602_10262_gb300 as gb
    gb.library()
    return gb


def _run(gb, x: np.ndarray, mode: int):
    xt = torch.from_numpy(x).cuda()
    q, d = gb.fp8_quantize_e4m3(xt, mode)
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0
    return q.cpu().numpy(), d.cpu().numpy()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1), (3, 5), (33, 3), (256, 256), (257, 1000), (64, 4096),
                                   (1000, 1029)])
def test_parity_small(gb, orc, mode, shape):
    x = workloads.randn_f32(shape, seed=shape[0] + 10 * shape[1])
    q, d = _run(gb, x, mode)
    qo, do = orc.quantize(x, mode)
    assert np.array_equal(q, qo)
    assert np.array_equal(d, do)


@pytest.mark.parametrize("mode", [0, 1])
def test_parity_full_size(gb, orc, mode):
    # the square-sweep operand size used by the benchmark (8192 x 8192 fp32)
    x = workloads.randn_f32((8192, 8192), seed=workloads.SEED_A)
    q, d = _run(gb, x, mode)
    qo, do = orc.quantize(x, mode)
    assert np.array_equal(d, do)
    assert np.array_equal(q, qo)


def test_strided_rows(gb, orc):
    wide = workloads.randn_f32((40, 100), seed=3)
    xt = torch.from_numpy(wide).cuda()[:, 7:67]       # ld = 100, unaligned start
    q, d = gb.fp8_quantize_e4m3(xt, 1)
    qo, do = orc.quantize(wide[:, 7:67], 1)
    assert np.array_equal(q.cpu().numpy(), qo) and np.array_equal(d.cpu().numpy(), do)


def test_zero_rows(gb):
    x = np.zeros((4, 64), np.float32)
    x[2, 5] = -3.0
    q, d = _run(gb, x, 1)
    assert np.array_equal(d, np.array([1, 1, 3 / 448, 1], np.float32))
    assert np.all(q[[0, 1, 3]] == 0) and q[2, 5] == 0xFE


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("mode", [0, 1])
def test_nonfinite_reported(gb, mode, bad):
    x = np.ones((8, 64), np.float32)
    x[3, 9] = bad
    xt = torch.from_numpy(x).cuda()
    gb.fp8_quantize_e4m3(xt, mode)
    assert gb.fp8_last_device_error() == -4          # FP8_ERR_NONFINITE
    assert gb.fp8_last_device_error() == 0           # cleared by the read


def test_device_encoder_all_in_range_fp32(gb, orc):
    """Every fp32 bit pattern with |x| <= 448 through the device encoder.

    A tensor whose amax is exactly 448 gets s = 448/448 = 1, so the codes are
    enc(x) itself; each chunk carries a sentinel row of 448."""
    top = 0x43E00000                                     # bits of 448.0f
    chunk = 1 << 26
    cols = 1024
    for sign in (0, 0x80000000):
        for lo in range(0, top + 1, chunk):
            hi = min(lo + chunk, top + 1)
            n = hi - lo
            rows = (n + cols - 1) // cols
            bits = torch.arange(lo, lo + rows * cols, dtype=torch.int64, device="cuda")
            bits = torch.clamp(bits, max=hi - 1) | sign
            bits = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits)     # as signed int32
            x = bits.to(torch.int32).view(torch.float32).reshape(rows, cols)
            x = torch.cat([x, torch.full((1, cols), 448.0, device="cuda")])
            q, d = gb.fp8_quantize_e4m3(x, 0)
            assert d.item() == 1.0
            got = q[:-1].reshape(-1)[:n].cpu().numpy()
            ref = orc.encode_pattern_range(lo | sign, (hi - 1 | sign) + 1)
            assert np.array_equal(got, ref), f"chunk at {lo | sign:#x}"


# every threads-per-row / vectors-per-thread shape at its first and last
# column counts, few rows and many (the rule counts rows per SM), and rows
# longer than registers hold; each row stride and start: 32-byte, 16-byte
# and no alignment of x, 8-, 4- and 1-byte alignment of the codes
@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("rows,cols", [(r, c) for r in (9, 401) for c in
                                       (1, 31, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4096, 4097, 6144, 6145,
                                        8192, 8199, 12288, 12289, 16384, 16385, 32768, 32769)])
def test_row_shapes(gb, orc, fmt, rows, cols):
    x = workloads.randn_f32((rows, cols), seed=rows + cols)
    x[rows // 2] = 0.0
    x[0, cols - 1] = -1e4                                  # the row's amax in its last element
    qo, do = orc.quantize(x, 1, fmt=fmt)
    quantize = gb.fp8_quantize_e5m2 if fmt else gb.fp8_quantize_e4m3
    for pad, off, qpad, qoff in ((-cols % 8, 0, -cols % 8, 0), (-cols % 4 + 4, 4, -cols % 4 + 4, 4), (1, 1, 1, 1)):
        xb = torch.full((rows * (cols + pad) + off,), float("nan"), device="cuda")
        xt = xb[off:].view(rows, cols + pad)[:, :cols]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((rows * (cols + qpad) + qoff,), 0xA5, dtype=torch.uint8, device="cuda")
        qt = qb[qoff:].view(rows, cols + qpad)[:, :cols]
        _, d = quantize(xt, 1, q=qt)
        assert np.array_equal(d.cpu().numpy(), do)
        assert np.array_equal(qt.cpu().numpy(), qo)
        if qpad:                                           # nothing written between the rows
            assert bool((qb[qoff:].view(rows, cols + qpad)[:, cols:] == 0xA5).all())
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0


@pytest.mark.parametrize("cols", [64, 1000, 4096, 4097, 8192, 16384, 16400])
def test_grouped_rows_equal_single(gb, cols):
    """fp8_quantize_e4m3_rows_grouped over matrices of mixed alignment and
    length equals the single calls, for each register size it runs with."""
    from paper_2602_10262_gb300._lib import FP8QuantJob
    g = torch.Generator(device="cuda").manual_seed(cols)
    mats, jobs, want = [], [], []
    for rows, c, pad in ((3, cols, 0), (1, max(1, cols - 3), 1), (7, 17, 4)):
        for aligned in (True, False):
            x = torch.randn((rows, c + pad), generator=g, device="cuda")[:, :c]
            q = torch.empty((rows, c + (0 if aligned else 1)), dtype=torch.uint8, device="cuda")[:, :c]
            d = torch.empty(rows, device="cuda")
            mats.append((x, q, d))
            want.append(gb.fp8_quantize_e4m3(x, 1))
            jobs.append(FP8QuantJob(x.data_ptr(), rows, c, x.stride(0), q.data_ptr(), q.stride(0), d.data_ptr()))
    for subset in (slice(0, None), slice(0, 1)):
        for _, q, d in mats:
            q.zero_(), d.zero_()
        arr = (FP8QuantJob * len(jobs[subset]))(*jobs[subset])
        assert gb.library().fp8_quantize_e4m3_rows_grouped(arr, len(arr), torch.cuda.current_stream().cuda_stream) == 0
        for (_, q, d), (qw, dw) in list(zip(mats, want))[subset]:
            assert torch.equal(q, qw) and torch.equal(d, dw)
    assert gb.fp8_last_device_error() == 0


def test_dependent_launches_keep_stream_order(gb):
    """Back-to-back calls whose buffers feed one another (the kernels are
    launched with programmatic serialization): eager and from a captured
    graph, every pass equals the calls made one by one."""
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((64, 2048), generator=g, device="cuda")
    w = torch.randn((512, 2048), generator=g, device="cuda")

    def chain(x, sync=lambda: None):
        outs, h = [], x
        for _ in range(3):
            A, dA = gb.fp8_quantize_e4m3(h, 1)
            sync()
            B, dB, v, m = gb.fp8_quantize_e4m3_prune24(w)
            sync()
            C = gb.gemm_fp8_dense(A, B, dA, 1, dB, 1, out_dtype=gb.OUT_F32)
            sync()
            P = gb.prune24_decompress(*gb.prune24_compress(B), 2048)
            sync()
            h = torch.cat([gb.gemm_fp8_dense(A, P, dA, 1, dB, 1, out_dtype=gb.OUT_F32), C, C, C], 1)
            sync()
            outs += [A, dA, C, h]
        return outs

    want = chain(x, torch.cuda.synchronize)
    for _ in range(5):
        assert all(torch.equal(a, b) for a, b in zip(chain(x), want))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        chain(x)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = chain(x)
    for _ in range(3):
        for t in got:
            t.zero_()
        graph.replay()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert gb.fp8_last_device_error() == 0


# one cluster with 1, 2, 4 and 8 vectors a thread at their first and last
# sizes, then the three-kernel form: flat and strided, rows shorter than a
# warp's vectors, single elements, ragged ends; each alignment of x and q
@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 7), (7, 9), (256, 128), (257, 128), (4096, 8), (4097, 8), (128, 512),
                                       (129, 512), (256, 512), (512, 512), (513, 512), (1, 262144), (1, 262145),
                                       (32769, 3), (100000, 5), (5000, 100), (700, 1001), (64, 8200), (3, 200001)])
def test_tensor_shapes(gb, orc, fmt, rows, cols):
    x = workloads.randn_f32((rows, cols), seed=rows + 3 * cols)
    x[-1, -1] = -77.0                                      # amax in the last element
    qo, do = orc.quantize(x, 0, fmt=fmt)
    quantize = gb.fp8_quantize_e5m2 if fmt else gb.fp8_quantize_e4m3
    for pad, off, qpad, qoff in ((0, 0, 0, 0), (0, 4, 0, 4), (-cols % 8, 0, -cols % 16, 0), (1, 1, 3, 1),
                                 (-cols % 4 + 4, 4, -cols % 4 + 4, 4)):
        xb = torch.full((rows * (cols + pad) + off,), float("nan"), device="cuda")
        xt = xb[off:].view(rows, cols + pad)[:, :cols]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((rows * (cols + qpad) + qoff,), 0xA5, dtype=torch.uint8, device="cuda")
        qt = qb[qoff:].view(rows, cols + qpad)[:, :cols]
        for _ in range(2):                                 # the scale slot holds the first pass's scale
            _, d = quantize(xt, 0, q=qt)
        assert np.array_equal(d.cpu().numpy(), do)
        assert np.array_equal(qt.cpu().numpy(), qo)
        if qpad:
            assert bool((qb[qoff:].view(rows, cols + qpad)[:, cols:] == 0xA5).all())
    torch.cuda.synchronize()
    assert gb.fp8_last_device_error() == 0


@pytest.mark.parametrize("rows,cols", [(64, 64), (700, 1001)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_tensor_nonfinite_reported(gb, rows, cols, bad):
    x = torch.randn((rows, cols), device="cuda")
    x[rows - 1, cols - 2] = bad
    gb.fp8_quantize_e4m3(x, 0)
    assert gb.fp8_last_device_error() == -4
    assert gb.fp8_last_device_error() == 0


def test_reused_buffers_follow_their_writers(gb):
    """One code buffer and one scale buffer per kind of quantiser, rewritten
    on every pass with other values and read by the product right behind (the
    kernels are launched with programmatic serialization): eager and from a
    captured graph, every pass equals the calls made one by one.  Covers the
    per-row, per-tensor (one cluster, and the four-kernel chain), grouped,
    long-row and block-scaled quantisers, the scale re-layout, and the fused
    quantise + compress, each before the dense, block-scaled or 2:4 product."""
    from paper_2602_10262_gb300._lib import FP8QuantJob
    g = torch.Generator(device="cuda").manual_seed(7)
    passes, R, K, KL, N = 4, 600, 512, 32896, 512

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    xs = [randn(R, K) * 3.0 ** p for p in range(passes)]
    longs = [randn(16, KL) * 5.0 ** p for p in range(passes)]
    W, dW = gb.fp8_quantize_e4m3(randn(N, K), 1)
    WL, dWL = gb.fp8_quantize_e4m3(randn(N, KL), 1)
    WX, sWX = gb.fp8_quantize_mx(randn(N, K))

    def codes(rows, cols):
        return torch.empty((rows, cols), dtype=torch.uint8, device="cuda")

    q, ql, qs = codes(R, K), codes(16, KL), codes(256, K)
    d, dl, dt = torch.empty(R, device="cuda"), torch.empty(16, device="cuda"), torch.empty(1, device="cuda")
    v, m = codes(R, K // 2), codes(R, K // 8)
    sr = codes(R, K // 32)
    st = torch.empty(gb.fp8_mx_scale_tiled_bytes(R, K), dtype=torch.uint8, device="cuda")

    def outputs():
        f = lambda r: torch.full((r, N), float("nan"), device="cuda")
        return [[f(R), f(256), f(R), f(R), f(16), f(R), f(R), f(R)] for _ in range(passes)]

    def grouped(x):
        job = (FP8QuantJob * 1)(FP8QuantJob(x.data_ptr(), R, K, K, q.data_ptr(), K, d.data_ptr()))
        stream = torch.cuda.current_stream().cuda_stream
        assert gb.library().fp8_quantize_e4m3_rows_grouped(job, 1, stream) == 0

    def run(outs, sync=lambda: None):
        for x, xl, o in zip(xs, longs, outs):
            for step in (
                    lambda: gb.fp8_quantize_e4m3(x, 1, q=q, dequant_scale=d),
                    lambda: gb.gemm_fp8_dense(q, W, d, 1, dW, 1, 1.0, gb.OUT_F32, C=o[0]),
                    lambda: gb.fp8_quantize_e4m3(x[:256], 0, q=qs, dequant_scale=dt),
                    lambda: gb.gemm_fp8_dense(qs, W, dt, 0, dW, 1, 1.0, gb.OUT_F32, C=o[1]),
                    lambda: gb.fp8_quantize_e4m3(x, 0, q=q, dequant_scale=dt),
                    lambda: gb.gemm_fp8_dense(q, W, dt, 0, dW, 1, 1.0, gb.OUT_F32, C=o[2]),
                    lambda: grouped(x),
                    lambda: gb.gemm_fp8_dense(W, q, dW, 1, d, 1, 1.0, gb.OUT_F32, C=o[3].view(N, R)),
                    lambda: gb.fp8_quantize_e4m3(xl, 1, q=ql, dequant_scale=dl),
                    lambda: gb.gemm_fp8_dense(ql, WL, dl, 1, dWL, 1, 1.0, gb.OUT_F32, C=o[4]),
                    lambda: gb.fp8_quantize_mx(x, q=q, scales=st),
                    lambda: gb.gemm_fp8_mx(q, st, WX, sWX, out_dtype=gb.OUT_F32, C=o[5]),
                    lambda: gb.fp8_quantize_mx(x, scale_layout=0, q=q, scales=sr),
                    lambda: gb.fp8_mx_scales_to_tiled(sr, R, K, st),
                    lambda: gb.gemm_fp8_mx(q, st, WX, sWX, out_dtype=gb.OUT_F32, C=o[6]),
                    lambda: gb.fp8_quantize_e4m3_prune24(x, q=q, dequant_scale=d, a_vals=v, a_meta=m),
                    lambda: gb.gemm_fp8_sparse24(v, m, W, d, 1, dW, 1, 1.0, gb.OUT_F32, C=o[7])):
                step()
                sync()

    want = outputs()
    run(want, torch.cuda.synchronize)
    assert not any(torch.isnan(t).any() for o in want for t in o)
    assert torch.equal(want[0][5], want[0][6])
    assert not torch.equal(want[0][0], want[1][0])

    def check(outs):
        for a, b in zip(outs, want):
            assert all(torch.equal(s, t) for s, t in zip(a, b))

    for _ in range(3):
        got = outputs()
        run(got)
        check(got)
    got = outputs()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(got)
    for _ in range(3):
        for o in got:
            for t in o:
                t.fill_(float("nan"))
        graph.replay()
        check(got)
    assert gb.fp8_last_device_error() == 0


@pytest.mark.parametrize("rows,cols", [(r, c) for r in (3, 401) for c in
                                       (1, 33, 255, 512, 1024, 1031, 4096, 4100, 6144, 12288, 14336, 16384, 32768)])
def test_row_mixed_alignments(gb, orc, rows, cols):
    """x and q of different alignment (either may rule the whole vectors
    out), by the single call and by the grouped one."""
    from paper_2602_10262_gb300._lib import FP8QuantJob
    x = workloads.randn_f32((rows, cols), seed=rows + cols)
    x[rows - 1, cols - 1] = 3e4
    qo, do = orc.quantize(x, 1)
    for pad, off, qpad, qoff in ((-cols % 8, 0, 1 - cols % 2, 1), (-cols % 8, 4, -cols % 16, 4),
                                 (1 - cols % 2, 0, -cols % 8, 0), (-cols % 4, 4, 3, 2)):
        xt = torch.zeros(rows * (cols + pad) + off, device="cuda")[off:].view(rows, cols + pad)[:, :cols]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((rows * (cols + qpad) + qoff,), 0xA5, dtype=torch.uint8, device="cuda")
        qt = qb[qoff:].view(rows, cols + qpad)[:, :cols]
        d = torch.empty(rows, device="cuda")
        gb.fp8_quantize_e4m3(xt, 1, q=qt, dequant_scale=d)
        single = qb.clone()
        assert np.array_equal(qt.cpu().numpy(), qo) and np.array_equal(d.cpu().numpy(), do)
        qb.fill_(0xA5), d.zero_()
        job = (FP8QuantJob * 1)(FP8QuantJob(xt.data_ptr(), rows, cols, xt.stride(0), qt.data_ptr(), qt.stride(0),
                                            d.data_ptr()))
        assert gb.library().fp8_quantize_e4m3_rows_grouped(job, 1, torch.cuda.current_stream().cuda_stream) == 0
        assert torch.equal(qb, single) and np.array_equal(d.cpu().numpy(), do)
    assert gb.fp8_last_device_error() == 0


@pytest.mark.parametrize("rows", [1, 15, 17, 130])
@pytest.mark.parametrize("lengths", [(1,), (256, 257), (512, 513, 100), (4096, 40, 4097), (8192, 3, 513),
                                     (16384, 64, 8193, 256, 1024, 2049), (16385, 64)])
def test_grouped_units_of_mixed_lengths(gb, orc, rows, lengths):
    """Rows of every threads-per-row shape in one launch (a block takes as
    many short rows as it has warps), row counts that end inside a block,
    aligned and unaligned jobs side by side; nothing written between rows."""
    from paper_2602_10262_gb300._lib import FP8QuantJob
    mats, jobs = [], []
    for i, c in enumerate(lengths * 2):
        n = rows + i
        x = workloads.randn_f32((n, c), seed=100 * i + c)
        x[n - 1, c - 1] = 500.0
        pad = -c % 8 if i < len(lengths) else 1
        xt = torch.zeros((n, c + pad), device="cuda")[:, :c]
        xt.copy_(torch.from_numpy(x))
        qb = torch.full((n, c + pad), 0xA5, dtype=torch.uint8, device="cuda")
        d = torch.empty(n, device="cuda")
        mats.append((x, xt, qb, d, c))
        jobs.append(FP8QuantJob(xt.data_ptr(), n, c, xt.stride(0), qb.data_ptr(), qb.stride(0), d.data_ptr()))
    arr = (FP8QuantJob * len(jobs))(*jobs)
    for _ in range(2):
        assert gb.library().fp8_quantize_e4m3_rows_grouped(arr, len(arr), torch.cuda.current_stream().cuda_stream) == 0
    for x, _, qb, d, c in mats:
        qo, do = orc.quantize(x, 1)
        assert np.array_equal(qb[:, :c].cpu().numpy(), qo) and np.array_equal(d.cpu().numpy(), do)
        assert bool((qb[:, c:] == 0xA5).all())
    assert gb.fp8_last_device_error() == 0
