// 2:4 selection of one or two groups of four E4M3/E5M2 codes, shared by
// prune24_compress (prune.cu) and the fused quantise + compress
// (fp8_quantize_e4m3_prune24, quant.cu): both keep the two codes of largest
// magnitude (code & 0x7F, the lower index on a tie) and write the same
// kept-code and index layout.
#pragma once
#include <cstdint>

namespace gb300 {

// One group of four codes (byte i of w = element i).  Element j outranks
// element i when key_j > key_i, or key_j == key_i and j < i (key = code &
// 0x7F); the two highest-ranked elements are kept.  score_i = key_i * 4 +
// (3 - i) orders the elements exactly that way and makes every score
// distinct, so the kept pair is the top two of four scores: a two-round
// max/min tournament.  Returns the two kept codes in the low 16 bits (lower
// index first) and the nibble i0 | i1 << 2 in bits 16..19.
__device__ __forceinline__ uint32_t select_group(uint32_t w)
{
    const uint32_t s0 = ((w << 2) & 0x1FCu) | 3u;
    const uint32_t s1 = ((w >> 6) & 0x1FCu) | 2u;
    const uint32_t s2 = ((w >> 14) & 0x1FCu) | 1u;
    const uint32_t s3 = (w >> 22) & 0x1FCu;
    const uint32_t a = max(s0, s1), b = min(s0, s1), c = max(s2, s3), d = min(s2, s3);
    const uint32_t t1 = max(a, c);
    const uint32_t t2 = max(min(a, c), max(b, d));
    const uint32_t i0 = 3u - max(t1 & 3u, t2 & 3u);
    const uint32_t i1 = 3u - min(t1 & 3u, t2 & 3u);
    const uint32_t vals = __byte_perm(w, 0u, i0 | (i1 << 4)) & 0xFFFFu;
    return vals | ((i0 | (i1 << 2)) << 16);
}

// 0xFF in every byte of v whose bit 7 is set, 0 in the others (a selector
// nibble of prmt with its top bit set replicates the byte's sign; the
// __byte_perm intrinsic ignores that bit).
__device__ __forceinline__ uint32_t byte_sign_mask(uint32_t v)
{
    uint32_t m;
    asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(m) : "r"(v));
    return m;
}

// Four groups at once (word g = group g), the groups side by side in the
// bytes of a register: after a 4 x 4 byte transpose, t_j holds element j of
// every group.  Element a < b is preferred over b when key_a >= key_b, and
// bit 7 of byte g of (key_a | 0x80) - key_b says so for group g without any
// borrow between bytes (keys are 7 bits).  An element is kept when it wins at
// least two of its three comparisons, a majority, which is one three-input
// logic instruction for all four groups.  The same pair as select_group's
// tournament in about 12 instructions a group (the two-groups-per-register
// tournament this replaced took about 30, and they were what limited
// prune24_compress: 23.3 -> 17.3 us at 8192 x 8192 with rows taken as one
// run).  Returns the four index
// nibbles (group g in bits 4g .. 4g + 3) and the kept codes of groups 0, 1
// and 2, 3 in v01 and v23 (lower index first).
__device__ __forceinline__ uint32_t select_groups4(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                                   uint32_t* v01, uint32_t* v23)
{
    const uint32_t kHigh = 0x80808080u, kKey = 0x7F7F7F7Fu;
    const uint32_t a = __byte_perm(w0, w1, 0x5140u), b = __byte_perm(w0, w1, 0x7362u);
    const uint32_t c = __byte_perm(w2, w3, 0x5140u), d = __byte_perm(w2, w3, 0x7362u);
    const uint32_t t0 = __byte_perm(a, c, 0x5410u), t1 = __byte_perm(a, c, 0x7632u);
    const uint32_t t2 = __byte_perm(b, d, 0x5410u), t3 = __byte_perm(b, d, 0x7632u);
    const uint32_t k1 = t1 & kKey, k2 = t2 & kKey, k3 = t3 & kKey;
    const uint32_t h0 = t0 | kHigh, h1 = t1 | kHigh, h2 = t2 | kHigh;
    // bit 7 of each byte: the lower-indexed element of the pair is preferred
    const uint32_t c01 = h0 - k1, c02 = h0 - k2, c03 = h0 - k3;
    const uint32_t c12 = h1 - k2, c13 = h1 - k3, c23 = h2 - k3;
    const auto maj = [](uint32_t x, uint32_t y, uint32_t z) { return (x & y) | (x & z) | (y & z); };
    const uint32_t e0 = maj(c01, c02, c03), e1 = maj(~c01, c12, c13);
    const uint32_t e2 = maj(~c02, ~c12, c23), e3 = maj(~c03, ~c13, ~c23);
    const uint32_t m0 = byte_sign_mask(e0), m1 = byte_sign_mask(e1);
    const uint32_t m2 = byte_sign_mask(e2), m3 = byte_sign_mask(e3);
    // first kept: element 0, else 1, else 2; second: element 3, else 2, else 1
    const uint32_t f1 = (t1 & m1) | (t2 & ~m1), f = (t0 & m0) | (f1 & ~m0);
    const uint32_t s1 = (t2 & m2) | (t1 & ~m2), s = (t3 & m3) | (s1 & ~m3);
    *v01 = __byte_perm(f, s, 0x5140u);
    *v23 = __byte_perm(f, s, 0x7362u);
    // nibble i0 | i1 << 2 of group g in the low half of byte g
    const uint32_t n = (~m0 & m1 & 0x01010101u) | (~m0 & ~m1 & 0x02020202u) |
                       ((m3 | ~m2) & 0x04040404u) | ((m3 | m2) & 0x08080808u);
    const uint32_t p = n | (n >> 4);
    return __byte_perm(p, 0u, 0x4420u);
}

}  // namespace gb300
