"""GPU parity: prune24_compress / prune24_decompress against the oracle,
bit-exact on kept codes and metadata."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import paper_2602_10262_gb300 as gb
    gb.library()
    return gb


def _ties(a):
    a = a.copy()
    a[:, 1::5] = a[:, 0::5][:, : a[:, 1::5].shape[1]]      # equal neighbours
    a[:, 2::9] ^= 0x80                                       # equal magnitude, other sign
    return a


@pytest.mark.parametrize("shape", [(1, 4), (3, 36), (5, 48), (7, 1028), (33, 1040), (128, 256),
                                   (257, 4096), (64, 100), (2, 16)])
def test_parity(gb, orc, shape):
    a = _ties(workloads.random_codes(shape, seed=shape[1]))
    v, m = gb.prune24_compress(torch.from_numpy(a).cuda())
    vo, mo = orc.prune24(a)
    assert np.array_equal(v.cpu().numpy(), vo)
    assert np.array_equal(m.cpu().numpy(), mo)


def test_parity_full_size(gb, orc):
    x = workloads.randn_f32((8192, 8192), seed=workloads.SEED_A)
    q, _ = orc.quantize(x, 1)
    v, m = gb.prune24_compress(torch.from_numpy(q).cuda())
    vo, mo = orc.prune24(q)
    assert np.array_equal(m.cpu().numpy(), mo)
    assert np.array_equal(v.cpu().numpy(), vo)


def test_strided_input(gb, orc):
    wide = workloads.random_codes((50, 300), seed=9)
    at = torch.from_numpy(wide).cuda()[:, 4:260]            # lda = 300, K = 256
    v, m = gb.prune24_compress(at)
    vo, mo = orc.prune24(wide[:, 4:260])
    assert np.array_equal(v.cpu().numpy(), vo) and np.array_equal(m.cpu().numpy(), mo)


def test_decompress(gb, orc):
    a = _ties(workloads.random_codes((33, 512), seed=10))
    v, m = gb.prune24_compress(torch.from_numpy(a).cuda())
    d = gb.prune24_decompress(v, m, 512)
    assert np.array_equal(d.cpu().numpy(), orc.decompress24(*orc.prune24(a), 512))


def test_bad_k(gb):
    with pytest.raises(gb.Fp8Error) as e:
        gb.prune24_compress(torch.zeros((2, 6), dtype=torch.uint8, device="cuda"))
    assert e.value.status == -2


@pytest.mark.parametrize("M,K,pad", [(1, 16, 0), (3, 16, 0), (1025, 16, 0), (7, 1024, 0), (5, 1040, 16),
                                     (2, 16400, 0), (33, 4096, 32), (6, 24, 0), (6, 24, 8), (4, 1028, 0), (1, 4, 0),
                                     (5, 4, 4), (9, 12, 0), (9, 20, 12), (300, 1032, 0), (301, 1036, 4), (64, 8, 8),
                                     (2100, 132, 0), (3, 4100, 3), (1, 40, 0)])
def test_contiguous_and_strided_rows(orc, M, K, pad):
    """Rows as one run of 16-code pieces (lda == K), row by row (padded
    rows) and the scalar path (K % 16 != 0), at the edges of a block's 1024
    pieces; the expansion of each on its vector and scalar paths."""
    import paper_2602_10262_gb300 as gb
    a = workloads.random_codes((M, K), seed=11 + M)
    t = torch.zeros((M, K + pad), dtype=torch.uint8, device="cuda")
    t[:, :K] = torch.from_numpy(a).cuda()
    vals, meta = gb.prune24_compress(t[:, :K])
    vo, mo = orc.prune24(a)
    assert np.array_equal(vals.cpu().numpy(), vo) and np.array_equal(meta.cpu().numpy(), mo)
    out = gb.prune24_decompress(vals, meta, K)
    assert np.array_equal(out.cpu().numpy(), orc.decompress24(vo, mo, K))
    # an output that starts off a 16-byte boundary takes the scalar path
    buf = torch.zeros(M * K + 4, dtype=torch.uint8, device="cuda")
    off = buf[4:].reshape(M, K)
    gb.prune24_decompress(vals, meta, K, out=off)
    assert torch.equal(off, out)


def test_expand_any_index_nibble(orc):
    """Metadata is the caller's: equal or descending indices expand the same
    on the vector and the scalar path."""
    import paper_2602_10262_gb300 as gb
    M, K = 4, 512
    g = torch.Generator().manual_seed(3)
    vals = torch.randint(0, 256, (M, K // 2), generator=g, dtype=torch.int32).to(torch.uint8).cuda()
    meta = torch.randint(0, 256, (M, K // 8), generator=g, dtype=torch.int32).to(torch.uint8).cuda()
    out = gb.prune24_decompress(vals, meta, K)
    buf = torch.zeros(M * K + 4, dtype=torch.uint8, device="cuda")
    off = buf[4:].reshape(M, K)
    gb.prune24_decompress(vals, meta, K, out=off)
    assert torch.equal(off, out)


@pytest.mark.parametrize("M,K", [(1, 4), (1, 8), (3, 12), (7, 20), (5, 132), (320, 4100), (129, 1032), (9, 4096),
                                 (1300, 4100)])
@pytest.mark.parametrize("pad,off", [(0, 1), (1, 0), (5, 3)])
def test_compress_from_any_byte(orc, M, K, pad, off):
    """Codes that start on any byte: two groups a thread while there is little
    work (the last shape is past that), outputs aligned and not, nothing
    written beside them."""
    import paper_2602_10262_gb300 as gb
    a = workloads.random_codes((M, K), seed=5 + M + K)
    t = torch.zeros(M * (K + pad) + off, dtype=torch.uint8, device="cuda")[off:].view(M, K + pad)[:, :K]
    t.copy_(torch.from_numpy(a))
    vo, mo = orc.prune24(a)
    for shift in (0, 1, 2):
        vb = torch.full((M * (K // 2) + shift + 4,), 0xA5, dtype=torch.uint8, device="cuda")
        mb = torch.full((M * ((K + 7) // 8) + shift + 4,), 0xA5, dtype=torch.uint8, device="cuda")
        v, m = vb[shift:-4].view(M, -1), mb[shift:-4].view(M, -1)
        gb.prune24_compress(t, v, m)
        assert np.array_equal(v.cpu().numpy(), vo) and np.array_equal(m.cpu().numpy(), mo)
        for b in (vb, mb):
            assert bool((b[:shift] == 0xA5).all()) and bool((b[-4:] == 0xA5).all())


@pytest.mark.parametrize("M,K", [(1, 4), (1, 8), (3, 12), (7, 20), (5, 132), (33, 28), (320, 4100), (129, 1032),
                                 (9, 4096), (1300, 4100), (40000, 4), (20000, 12), (700, 8200)])
def test_expand_to_any_byte(orc, M, K):
    """Outputs that start off a 4-byte boundary (one group a thread, with few
    groups and many, rows of whole and of half metadata bytes) equal the
    oracle; nothing is written beside them."""
    import paper_2602_10262_gb300 as gb
    vo, mo = orc.prune24(workloads.random_codes((M, K), seed=9 + M + K))
    want = orc.decompress24(vo, mo, K)
    for shift, off in ((0, 1), (0, 2), (1, 3), (2, 7)):
        vb = torch.zeros(M * (K // 2) + shift, dtype=torch.uint8, device="cuda")
        v, m = vb[shift:].view(M, -1), torch.from_numpy(mo).cuda()
        v.copy_(torch.from_numpy(vo))
        buf = torch.full((M * K + off + 5,), 0xA5, dtype=torch.uint8, device="cuda")
        out = buf[off:-5].view(M, K)
        gb.prune24_decompress(v, m, K, out=out)
        assert np.array_equal(out.cpu().numpy(), want)
        assert bool((buf[:off] == 0xA5).all()) and bool((buf[-5:] == 0xA5).all())


def test_expand_any_index_nibble_by_value():
    """Every metadata byte against the rule itself, on the vector path, the
    piece path and the group path: code 0 of a group at index nibble & 3,
    code 1 at nibble >> 2, both OR-ed where the indices agree."""
    import paper_2602_10262_gb300 as gb
    M, K = 8, 1024                                        # 256 metadata bytes in each two rows
    g = np.random.default_rng(4)
    vals = g.integers(0, 256, (M, K // 2), dtype=np.uint8)
    meta = np.stack([g.permutation(256).astype(np.uint8) for _ in range(M // 2)]).reshape(M, K // 8)
    nib = np.stack([meta & 15, meta >> 4], -1).reshape(M, K // 4)
    want = np.zeros((M, K // 4, 4), np.uint8)
    r, c = np.indices(nib.shape)
    pair = vals.reshape(M, K // 4, 2)
    want[r, c, nib & 3] |= pair[..., 0]
    want[r, c, nib >> 2] |= pair[..., 1]
    v, m = torch.from_numpy(vals).cuda(), torch.from_numpy(meta).cuda()
    for off in (0, 4, 1):
        out = torch.zeros(M * K + off, dtype=torch.uint8, device="cuda")[off:].view(M, K)
        gb.prune24_decompress(v, m, K, out=out)
        assert np.array_equal(out.cpu().numpy(), want.reshape(M, K))
