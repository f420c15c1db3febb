// Site updates on single words (32 sites of one class in one row), four
// neighbouring lanes of a warp sharing the Philox outputs of a 128-site
// group.  Included by the .cu files only.
//
// Lane q of a quad holds word q of its group.  The random planes of a group
// are drawn four at a time: lane q computes plane 4b + q (one Philox output,
// the plane's four words) and the quad transposes the 4 x 4 words, so that
// lane q ends with word q of planes 4b .. 4b + 3.  A group's planes take a
// quarter of the time they take one thread, and a warp holds 8 groups.
#pragma once

#include "tl_device.cuh"

namespace tl {

// What Philox4x32-10 with counter (grp, sweep, (plane << 16) | slot, stream)
// needs of the group alone after two rounds: the first round multiplies grp
// by M0, the second that product's high half (with stream and key mixed in)
// by M1, whatever the sweep and plane are.
struct GroupKey {
    uint32_t a, bh, bl;
    TL_DEV void set(uint32_t grp, const DevRng& r)
    {
        a = grp * 0xD2511F53u;
        const uint32_t c2 = __umulhi(grp, 0xD2511F53u) ^ r.stream ^ r.k1;
        bl = c2 * 0xCD9E8D57u;
        bh = __umulhi(c2, 0xCD9E8D57u);
    }
};
// The same of the plane and pass alone (shared by a thread's groups).
struct PlaneKey {
    uint32_t l1, l0, h0;
    TL_DEV void set(uint32_t plane, uint32_t slot, uint32_t sweep, const DevRng& r)
    {
        const uint32_t c2 = (plane << 16) | slot;
        l1 = c2 * 0xCD9E8D57u;
        const uint32_t c0 = __umulhi(c2, 0xCD9E8D57u) ^ sweep ^ r.k0;
        l0 = c0 * 0xD2511F53u;
        h0 = __umulhi(c0, 0xD2511F53u);
    }
};
// Rounds 3 to 10 (the first two are in the keys): 16 products instead of 20.
TL_DEV uint4 philox_keyed(const GroupKey& g, const PlaneKey& p, const DevRng& r)
{
    uint32_t k0 = r.k0 + 0x9E3779B9u, k1 = r.k1 + 0xBB67AE85u;
    uint32_t c0 = g.bh ^ p.l1 ^ k0, c1 = g.bl, c2 = p.h0 ^ g.a ^ k1, c3 = p.l0;
#pragma unroll
    for (int i = 2; i < 10; ++i) {
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
        const uint32_t lo0 = c0 * 0xD2511F53u, hi0 = __umulhi(c0, 0xD2511F53u);
        const uint32_t lo1 = c2 * 0xCD9E8D57u, hi1 = __umulhi(c2, 0xCD9E8D57u);
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// Planes 4 b0 .. 4 (b0 + B) - 1 of this lane's word (every lane of the warp
// calls it): B Philox calls in flight together, then B transposes of 4 x 4
// words over the quad, through shared memory (`buf`: this quad's 16 B words,
// quads 16 B + 4 words apart, so that the reads are free of bank conflicts; by
// shuffles a transpose takes 12 selects more, and the ALU is as busy as the
// multiplier).
constexpr int kMaxBlocks = 2, kQuadPitch = 16 * kMaxBlocks + 4, kWarpTrans = 8 * kQuadPitch;
template <int B>
TL_DEV void quad_planes(const GroupKey& g, uint32_t b0, uint32_t slot, uint32_t sweep, const DevRng& r, int q,
                        uint32_t* buf, uint4 (&w)[B])
{
    uint4 o[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        PlaneKey pk;
        pk.set(4u * (b0 + (uint32_t)b) + (uint32_t)q, slot, sweep, r);
        o[b] = philox_keyed(g, pk, r);
    }
    __syncwarp();
#pragma unroll
    for (int b = 0; b < B; ++b) *reinterpret_cast<uint4*>(buf + 16 * b + 4 * q) = o[b];
    __syncwarp();
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const uint32_t* p = buf + 16 * b + q;
        w[b] = make_uint4(p[0], p[4], p[8], p[12]);
    }
}

// The comparison u < t of four planes as a subtraction, least significant
// plane first: lt is the borrow (one three-input operation a plane), eq the
// sites where all planes agree.
TL_DEV void cmp_block(uint4 u, const uint32_t (&t)[4], uint32_t& lt, uint32_t& eq)
{
    lt = ~u.w & t[3];
    lt = (~u.z & t[2]) | (~(u.z ^ t[2]) & lt);
    lt = (~u.y & t[1]) | (~(u.y ^ t[1]) & lt);
    lt = (~u.x & t[0]) | (~(u.x ^ t[0]) & lt);
    eq = ~(u.w ^ t[3]);
    eq &= ~(u.z ^ t[2]);
    eq &= ~(u.y ^ t[1]);
    eq &= ~(u.x ^ t[0]);
}

// Six-vertex threshold bits as XORs of products of the corner bits (algebraic
// normal form): per plane 16 coefficients (all ones or zero) of the products
// of TL, TR, BR, BL in index order, or, in the count form, 5 of 1, n0, n1,
// n0 n1, n2.  One three-input operation per product and plane, the coefficient
// straight from the parameter bank.
struct AnfTable {
    uint32_t c[32][16];
};
TL_DEV void anf_products(uint32_t tl, uint32_t tr, uint32_t br, uint32_t bl, uint32_t (&m)[16])
{
    m[0] = 0xFFFFFFFFu;
    m[1] = tl;
    m[2] = tr;
    m[4] = br;
    m[8] = bl;
    m[3] = tl & tr;
    m[5] = tl & br;
    m[6] = tr & br;
    m[9] = tl & bl;
    m[10] = tr & bl;
    m[12] = br & bl;
    m[7] = m[3] & br;
    m[11] = m[3] & bl;
    m[13] = m[5] & bl;
    m[14] = m[6] & bl;
    m[15] = m[7] & bl;
}
// Bits [lo, hi] of a word, clipped to it (lo, hi any integers).
TL_DEV uint32_t span_mask(int lo, int hi)
{
    const int a = lo > 0 ? lo : 0, b = hi < 31 ? 31 - hi : 0;
    return __funnelshift_lc(0u, 0xFFFFFFFFu, (uint32_t)a) & __funnelshift_rc(0xFFFFFFFFu, 0u, (uint32_t)b);
}

// Edges of one word's sites: `row` points at plane 0, word k of row y in rows
// of P planes of K words, RW words apart.  `e` is the edge that is set in the
// UP state; flips are XORed into every edge of the site.  Words that two words'
// sites share (planes read one site over) are changed by atomicXor alone.
struct DominoWord {
    uint32_t he, ho, n, s;
    TL_DEV uint32_t read(const uint32_t* row, int K, int RW, int k, int p, uint32_t& e)
    {
        he = row[0];
        ho = row[K];
        n = row[(2 + p) * K];
        s = row[(2 + p) * K - RW];
        const uint32_t hp = (!p && k > 0) ? row[K - 1] : 0u;
        e = p ? ho : he;
        const uint32_t w = p ? he : (ho << 1) | (hp >> 31);
        return (e & w & ~(n | s)) | (n & s & ~(e | w));
    }
    TL_DEV void flip(uint32_t* row, int K, int RW, int k, int p, uint32_t fl) const
    {
        row[0] = he ^ fl;
        row[(2 + p) * K] = n ^ fl;
        row[(2 + p) * K - RW] = s ^ fl;
        if (p) {
            row[K] = ho ^ fl;
        } else {
            if (fl >> 1) atomicXor(row + K, fl >> 1);
            if ((fl & 1u) && k > 0) atomicXor(row + K - 1, 0x80000000u);
        }
    }
};

struct LozengeWord {
    uint32_t e0, e1, e2, e5, w3, w4;   // w3, w4: the words holding e3, e4
    TL_DEV uint32_t read(const uint32_t* row, int K, int RW, int k, int r, uint32_t& e)
    {
        e0 = row[r * K];
        e1 = row[(6 + r) * K];
        e2 = row[(3 + r) * K];
        e5 = row[(3 + r) * K - RW];
        const int c = r ? r - 1 : 2;
        w3 = row[c * K];
        w4 = row[(6 + c) * K - RW];
        uint32_t e3 = w3, e4 = w4;
        if (!r) {
            const uint32_t p3 = k > 0 ? row[c * K - 1] : 0u, p4 = k > 0 ? row[(6 + c) * K - RW - 1] : 0u;
            e3 = (w3 << 1) | (p3 >> 31);
            e4 = (w4 << 1) | (p4 >> 31);
        }
        e = e0;
        return (e0 & e2 & e4 & ~(e1 | e3 | e5)) | (e1 & e3 & e5 & ~(e0 | e2 | e4));
    }
    TL_DEV void flip(uint32_t* row, int K, int RW, int k, int r, uint32_t fl) const
    {
        row[r * K] = e0 ^ fl;
        row[(6 + r) * K] = e1 ^ fl;
        row[(3 + r) * K] = e2 ^ fl;
        row[(3 + r) * K - RW] = e5 ^ fl;
        if (r) {
            row[(r - 1) * K] = w3 ^ fl;
            row[(6 + r - 1) * K - RW] = w4 ^ fl;
        } else {
            if (fl >> 1) {
                atomicXor(row + 2 * K, fl >> 1);
                atomicXor(row + 8 * K - RW, fl >> 1);
            }
            if ((fl & 1u) && k > 0) {
                atomicXor(row + 2 * K - 1, 0x80000000u);
                atomicXor(row + 8 * K - RW - 1, 0x80000000u);
            }
        }
    }
};

struct SixvWord {
    uint32_t b, t, l, r;           // r: the word holding the R edges
    uint32_t tl, tr, br, bl;
    // row: face row Y; RW above it the next vertex row
    TL_DEV uint32_t read(const uint32_t* row, int K, int RW, int k, int px, uint32_t& e)
    {
        uint32_t rr;
        if (!px) {
            b = row[0];
            t = row[RW];
            l = row[2 * K];
            r = rr = row[3 * K];
            br = row[K];
            tr = row[RW + K];
            tl = row[RW + 2 * K];
            bl = (br << 1) | (k > 0 ? row[K - 1] >> 31 : 0u);
        } else {
            const bool more = k + 1 < K;
            b = row[K];
            t = row[RW + K];
            l = row[3 * K];
            tl = row[RW + 3 * K];
            bl = row[0];
            r = row[2 * K];
            const uint32_t tw = row[RW];
            br = (bl >> 1) | (more ? row[1] << 31 : 0u);
            tr = (tw >> 1) | (more ? row[RW + 1] << 31 : 0u);
            rr = (r >> 1) | (more ? row[2 * K + 1] << 31 : 0u);
        }
        e = b;
        return (b & l & ~(rr | t)) | (rr & t & ~(b | l));
    }
    TL_DEV void flip(uint32_t* row, int K, int RW, int k, int px, uint32_t fl) const
    {
        if (!px) {
            row[0] = b ^ fl;
            row[RW] = t ^ fl;
            row[2 * K] = l ^ fl;
            row[3 * K] = r ^ fl;
        } else {
            row[K] = b ^ fl;
            row[RW + K] = t ^ fl;
            row[3 * K] = l ^ fl;
            if (fl << 1) atomicXor(row + 2 * K, fl << 1);
            if ((fl >> 31) && k + 1 < K) atomicXor(row + 2 * K + 1, 1u);
        }
    }
};

template <int LAT>
struct WordOf {
    using type = DominoWord;
};
template <>
struct WordOf<LAT_LOZENGE> {
    using type = LozengeWord;
};
template <>
struct WordOf<LAT_SIXV> {
    using type = SixvWord;
};

}  // namespace tl
