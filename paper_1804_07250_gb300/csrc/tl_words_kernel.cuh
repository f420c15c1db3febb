// Resident multi-sweep kernel of every chain but the dominoes at t = 2^31 and
// large stripes with thresholds of few bits (cooperative launch, one CTA per SM).
//
// The paper launches Rotate and Update once per half-step and moves the whole
// tiling through device memory every time (Sec. 2.2).  Here one launch runs
// many sweeps: each CTA keeps a horizontal stripe of the packed state and
// `halo` rows above and below it in shared memory.  A pass updates every row
// whose inputs are still exact; a site only reads edges within one row of it,
// so the exact region shrinks by one row per pass and side, and after `halo`
// passes the CTA publishes its boundary rows and refreshes its halos from its
// neighbours (64-bit words of a launch and cycle tag and 32 data bits, double
// buffered by cycle parity; every wait is bounded).  A domain that one CTA
// holds has no exchange at all.
//
// Every thread owns up to M words (32 sites of one class each; the four words
// of a 128-site group in the four lanes of a quad, tl_words.cuh) for the whole
// launch, so the bookkeeping of a group is done once.  A pass has two halves:
//  - the update, on the chain's critical path: read the edges around the
//    word, find the flippable sites, flip those whose draw says so;
//  - the draws of the NEXT pass, which depend on no state: the first 4 NB
//    random planes, and for lozenges and dominoes also the comparison with
//    the thresholds of all 32 sites (two words are carried over the barrier:
//    sites decided UP, sites undecided).  Six-vertex thresholds depend on the
//    corner bits, so there the planes are carried and compared in the update.
// A warp whose flippable sites are not all decided by then draws four more
// planes at a time.  One CTA barrier per pass.
//
// Bound: the latency of the update and the barrier, and the multiplier rate
// of the draws (68 cycles of a scheduler per 32 Philox calls).
#pragma once

#include "tl_words.cuh"

#include <cstdint>

namespace tl {

struct WordParams {
    uint32_t* rows0;            // global row 0 (after the pad row)
    Geom g;
    const int* stripe_lo;
    int halo, nblk;             // passes per exchange; blocks of four planes drawn ahead (dominoes, lozenges)
    const uint8_t* colours;     // random pass order: colour of every slot of the launch, else nullptr
    uint32_t sweep0, nsweeps;
    DevRng rng;
    uint32_t scalar;            // THR_SCALAR
    int kmax;
    const uint32_t* planes;     // THR_SITE
    int cpol;                   // six-vertex count form: polarity
    const int2* grange;
    unsigned long long* xbuf;   // [C][2][2][halo row_words] tagged exchange words
    int* status;
    unsigned int* loaded;       // [C] epoch of the last launch without an exchange that a stripe has loaded in
    unsigned long long* ring;
    uint32_t* counts;           // bit-sliced density counter planes, or nullptr
    uint64_t burn;
    uint32_t stride;
    unsigned int epoch;
    unsigned long long* flips;  // accepted-flip counter, or nullptr
    AnfTable anf;               // six-vertex threshold bits
};

TL_DEV uint64_t wd_globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
TL_DEV void wd_ld2(const unsigned long long* p, unsigned long long* a, unsigned long long* b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(*a), "=l"(*b) : "l"(p) : "memory");
}
TL_DEV void wd_st2(unsigned long long* p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
constexpr uint64_t kWordWaitLimitNs = 2000000000ull;   // 2 s: far beyond any healthy exchange

// A thread's word: `off` its shared-memory word offset (plane 0, word k of its
// row), `ym` its row mod 2 (dominoes) or 3 (lozenges), lim[] the last pass of
// a cycle its row is exact in (0: none; six-vertex: the two face rows of its
// pair), and what its sites need of the constants: threshold planes of residue
// 0 (per-site), sites inside the square by residue (six-vertex).
struct WordItem {
    int off, k;
    uint8_t ym;
    uint8_t lim[2];
    bool own[2];
    GroupKey key;
    const uint32_t* tp;
    uint32_t inside[2];
};

// FIXED: every cycle is whole sweeps in the fixed colour order, so the pass
// loop is unrolled by slot and slot and colour are constants.
template <int LAT, int TK, bool CNT, int MAXT, int M, int NB, bool FIXED>
__global__ void __launch_bounds__(MAXT, 1) words_kernel(const __grid_constant__ WordParams P)
{
    extern __shared__ uint4 smem4[];
    __shared__ unsigned long long s_red[MAXT / 32];
    __shared__ __align__(16) uint32_t s_tr[(MAXT / 32) * kWarpTrans];
    constexpr bool SIX = LAT == LAT_SIXV;
    using Word = typename WordOf<LAT>::type;
    const Geom& g = P.g;
    const int K = g.K, RW = (int)g.row_words, nt = blockDim.x;
    const int c = blockIdx.x, C = gridDim.x;
    const int tid = threadIdx.x, q = tid & 3;
    const int lo = P.stripe_lo[c], hi = P.stripe_lo[c + 1];
    const bool bot = c == 0, top = c == C - 1;
    const int h = P.halo;
    const int slo = bot ? -1 : lo - h, shi = top ? g.H + 1 : hi + h;
    const int nloc = shi - slo;
    uint32_t* const sm = reinterpret_cast<uint32_t*>(smem4);
    int* const off = reinterpret_cast<int*>(sm + (size_t)nloc * RW);   // [rows + 1] first item of a local row (pair)
    uint32_t* const tbuf = s_tr + (tid >> 5) * kWarpTrans + ((tid & 31) >> 2) * kQuadPitch;

    {
        uint4* d = smem4;
        const uint4* s = reinterpret_cast<const uint4*>(P.rows0 + (int64_t)slo * RW);
        for (int i = tid; i < nloc * (RW / 4); i += nt) d[i] = __ldcg(s + i);
    }
    // ---- items: the active groups of every row of the stripe and its halos
    // (six-vertex: of every pair of face rows 2r, 2r + 1) ----
    const int r0 = SIX ? (slo > 0 ? slo >> 1 : 0) : (slo > 0 ? slo : 0);
    const int r1 = SIX ? ((shi < g.H ? shi : g.H) + 1) >> 1 : (shi < g.H ? shi : g.H);
    auto row_groups = [&](int r) {
        if (!SIX) return P.grange[r];
        int2 a = P.grange[2 * r];
        if (2 * r + 1 < g.H) {
            const int2 b = P.grange[2 * r + 1];
            if (a.y <= a.x) a = b;
            else if (b.y > b.x) a = make_int2(a.x < b.x ? a.x : b.x, a.y > b.y ? a.y : b.y);
        }
        return a;
    };
    for (int r = r0 + tid; r < r1; r += nt) {
        const int2 gr = row_groups(r);
        off[r - r0 + 1] = gr.y > gr.x ? gr.y - gr.x : 0;
    }
    __syncthreads();
    if (tid == 0) {
        off[0] = 0;
        for (int r = r0; r < r1; ++r) off[r - r0 + 1] += off[r - r0];
    }
    __syncthreads();
    const int nitems = r1 > r0 ? off[r1 - r0] : 0;
    WordItem it[M];
#pragma unroll
    for (int s = 0; s < M; ++s) {
        const int i = (tid >> 2) + s * (nt >> 2);
        it[s].lim[0] = it[s].lim[1] = 0;
        it[s].own[0] = it[s].own[1] = false;
        it[s].off = it[s].k = 0;
        it[s].ym = 0;
        it[s].tp = P.planes;
        it[s].inside[0] = it[s].inside[1] = 0u;
        it[s].key.set(0u, P.rng);
        if (i >= nitems) continue;
        int a = 0, b = r1 - r0 - 1;
        while (a < b) {   // last row whose first item is <= i
            const int mid = (a + b + 1) >> 1;
            if (off[mid] <= i) a = mid;
            else b = mid - 1;
        }
        const int r = r0 + a, m = row_groups(r).x + (i - off[a]);
        const int y0 = SIX ? 2 * r : r;
        it[s].k = 4 * m + q;
        it[s].off = (y0 - slo) * RW + it[s].k;
        it[s].ym = (uint8_t)(LAT == LAT_LOZENGE ? y0 % 3 : y0 & 1);
        if (TK == THR_SITE) it[s].tp = P.planes + ((size_t)y0 * g.npar * 32) * K + it[s].k;
        if (SIX)
#pragma unroll
            for (int px = 0; px < 2; ++px)
                it[s].inside[px] = span_mask((px ? 0 : 1) - 32 * it[s].k, ((g.N - 1 - px) >> 1) - 32 * it[s].k);
        it[s].key.set((uint32_t)(r * g.Kg + m), P.rng);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int y = y0 + (SIX ? v : 0);
            int l;
            if (SIX) {
                // face row y reads vertex rows y and y + 1; interior faces 1 .. N - 1
                const int lb = bot ? 255 : y - slo + 1, lt = top ? 255 : shi - 1 - y;
                l = y >= 1 && y <= g.N - 1 ? (lb < lt ? lb : lt) : 0;
            } else {
                // row y reads rows y - 1 and y
                const int lb = bot ? 255 : y - slo, lt = top ? 255 : shi - y;
                l = lb < lt ? lb : lt;
            }
            it[s].lim[v] = (uint8_t)(l < 0 ? 0 : (l > 255 ? 255 : l));
            it[s].own[v] = y >= lo && y < hi;
        }
#ifdef TL_DEBUG
        // the words read and written: rows y - 1 and y (six-vertex face rows
        // y .. y + 1, vertex rows up to y + 2), words 4m .. 4m + 3
        const int ylo = SIX ? y0 + (it[s].lim[0] ? 0 : 1) : y0 - 1;
        const int yhi = SIX ? y0 + (it[s].lim[1] ? 2 : 1) : y0;
        if ((it[s].lim[0] || it[s].lim[1]) &&
            !(TL_IN(ylo - slo, nloc, 201) && TL_IN(yhi - slo, nloc, 202) && TL_IN(4 * m + 3, K, 203)))
            it[s].lim[0] = it[s].lim[1] = 0;
#endif
    }
    __syncthreads();

    const int passes = g.passes;
    const uint64_t total = (uint64_t)P.nsweeps * passes;
    if (C > 1 && total <= (uint64_t)h && tid == 0) stripe_mark_loaded(P.loaded, P.epoch);
    // the next density sample: sweeps s (counted after the sweep, 1-based)
    // with s >= burn and (s - burn) % stride == 0, tracked incrementally
    uint64_t next_sample = ~0ull;
    if (P.counts && P.stride) {
        const uint64_t first = (uint64_t)P.sweep0 + 1;
        next_sample = first <= P.burn ? P.burn : P.burn + ((first - P.burn + P.stride - 1) / P.stride) * P.stride;
    }
    uint32_t nflip = 0;   // accepted flips of this thread's owned sites

    // colour of a pass slot (the slot itself unless the order is random)
    auto colour_of = [&](uint32_t sweep, uint32_t slot) -> uint32_t {
        return P.colours ? P.colours[(size_t)(sweep - P.sweep0) * passes + slot] : slot;
    };
    // face row of the pair and residue of an item in a pass of colour `col`
    auto row_v = [&](uint32_t col) { return SIX ? sixv_py(col) : 0; };
    auto residue = [&](const WordItem& w, uint32_t col) {
        if (LAT == LAT_DOMINO) return (int)((col + w.ym) & 1u);
        if (LAT == LAT_LOZENGE) return (int)col - (int)w.ym + (col < w.ym ? 3 : 0);
        return sixv_px(col);
    };
    auto site_bits = [&](const WordItem& w, int res, int b, bool in, uint32_t (&t)[4]) {
        const uint32_t* tp = w.tp + (size_t)(32 * res + 4 * b) * K;
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = in ? __ldg(tp + (size_t)j * K) : 0u;
    };
    auto scalar_bits = [&](int b, uint32_t (&t)[4]) {
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = 0u - ((P.scalar >> (31 - 4 * b - j)) & 1u);
    };

    // carried over the barrier: the draws of the coming pass
    uint32_t lt_[SIX ? 1 : M], und_[SIX ? 1 : M];   // dominoes, lozenges
    uint4 rp_[SIX ? M : 1][SIX ? NB : 1];           // six-vertex: random planes
    // A warp none of whose sites was flippable in its last two sweeps' worth
    // of passes (`cold` counts them) draws nothing ahead: in the frozen corners
    // it will hardly need it, and draws in the update if it does.
    int cold[M];
    bool drawn[M];
#pragma unroll
    for (int s = 0; s < M; ++s) cold[s] = 0;
    const int frozen = 2 * passes;
    // draws of pass `slot` (colour col) of `sweep`, the i-th of its cycle
    auto draw = [&](uint32_t sweep, uint32_t slot, uint32_t col, int i) {
        const int v = row_v(col);
        bool any = false;
#pragma unroll
        for (int s = 0; s < M; ++s) {
            drawn[s] = cold[s] < frozen && __any_sync(0xFFFFFFFFu, i <= (v ? it[s].lim[1] : it[s].lim[0]));
            any |= drawn[s];
        }
        if (!any) return;
        if constexpr (SIX) {
#pragma unroll
            for (int s = 0; s < M; ++s)
                if (drawn[s]) quad_planes<NB>(it[s].key, 0u, slot, sweep, P.rng, q, tbuf, rp_[s]);
        } else {
#pragma unroll
            for (int s = 0; s < M; ++s) {
                if (!drawn[s]) continue;
                const int res = residue(it[s], col);
                const bool in = i <= (v ? it[s].lim[1] : it[s].lim[0]);
                uint32_t lt = 0u, und = TK == THR_SCALAR && P.kmax < 0 ? 0u : 0xFFFFFFFFu, l, eq;
                int b = 0;
                for (; b + 2 <= P.nblk; b += 2) {
                    uint32_t t0[4], t1[4];
                    uint4 w[2];
                    if (TK == THR_SITE) {
                        site_bits(it[s], res, b, in, t0);
                        site_bits(it[s], res, b + 1, in, t1);
                    } else {
                        scalar_bits(b, t0);
                        scalar_bits(b + 1, t1);
                    }
                    quad_planes<2>(it[s].key, (uint32_t)b, slot, sweep, P.rng, q, tbuf, w);
                    cmp_block(w[0], t0, l, eq);
                    lt |= und & l;
                    und &= eq;
                    cmp_block(w[1], t1, l, eq);
                    lt |= und & l;
                    und &= eq;
                }
                if (b < P.nblk) {
                    uint32_t t[4];
                    uint4 w[1];
                    if (TK == THR_SITE) site_bits(it[s], res, b, in, t);
                    else scalar_bits(b, t);
                    quad_planes<1>(it[s].key, (uint32_t)b, slot, sweep, P.rng, q, tbuf, w);
                    cmp_block(w[0], t, l, eq);
                    lt |= und & l;
                    und &= eq;
                }
                lt_[s] = lt;
                und_[s] = und;
            }
            // past the last set threshold bit an undecided u is >= t
            if (TK == THR_SCALAR && 4 * P.nblk > P.kmax) {
#pragma unroll
                for (int s = 0; s < M; ++s) und_[s] = 0u;
            }
        }
    };

    // update of item s in pass `slot` (colour col) of `sweep`, the i-th of its
    // cycle
    auto update = [&](int s, uint32_t sweep, uint32_t slot, uint32_t col, int i) {
        const int v = row_v(col);
        const bool act = i <= (v ? it[s].lim[1] : it[s].lim[0]);
        const int res = residue(it[s], col);
        const int k = it[s].k;
        uint32_t* const row = sm + it[s].off + (SIX ? v * RW : 0);
        Word w;
        uint32_t e = 0u, f = 0u;
        if (act) {
            f = w.read(row, K, RW, k, res, e);
            if constexpr (SIX) f &= res ? it[s].inside[1] : it[s].inside[0];
        }
        if (!__any_sync(0xFFFFFFFFu, f != 0u)) {
            ++cold[s];
            return;
        }
        cold[s] = 0;
        constexpr int NM = CNT ? 5 : 16;
        uint32_t m[NM];
        if constexpr (SIX) {
            if constexpr (CNT) {
                uint32_t n0, n1, n2;
                corner_count(w.tl ^ polmask(P.cpol, 0), w.tr ^ polmask(P.cpol, 1), w.br ^ polmask(P.cpol, 2),
                             w.bl ^ polmask(P.cpol, 3), n0, n1, n2);
                m[0] = 0xFFFFFFFFu;
                m[1] = n0;
                m[2] = n1;
                m[3] = n0 & n1;
                m[4] = n2;
            } else {
                anf_products(w.tl, w.tr, w.br, w.bl, m);
            }
        }
        auto table_bits = [&](int b, uint32_t (&t)[4]) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                t[j] = P.anf.c[4 * b + j][0];
#pragma unroll
                for (int x = 1; x < NM; ++x) t[j] ^= P.anf.c[4 * b + j][x] & m[x];
            }
        };
        uint32_t lt = 0u, und = f;
        int b = 0;
        if (drawn[s]) {
            if constexpr (SIX) {
#pragma unroll
                for (int a = 0; a < NB; ++a) {
                    uint32_t t[4], l, eq;
                    table_bits(a, t);
                    cmp_block(rp_[s][a], t, l, eq);
                    lt |= und & l;
                    und &= eq;
                }
                b = NB;
            } else {
                lt = lt_[s];
                und &= und_[s];
                b = P.nblk;
            }
        }
        for (; b < 8 && __any_sync(0xFFFFFFFFu, und != 0u); ++b) {
            uint32_t t[4], l, eq;
            uint4 u[1];
            if constexpr (SIX) table_bits(b, t);
            else if (TK == THR_SITE) site_bits(it[s], res, b, act, t);
            else scalar_bits(b, t);
            quad_planes<1>(it[s].key, (uint32_t)b, slot, sweep, P.rng, q, tbuf, u);
            cmp_block(u[0], t, l, eq);
            lt |= und & l;
            und &= eq;
        }
        // a flippable site with `e` set is UP now; it flips iff the draw disagrees
        const uint32_t fl = f & (lt ^ e);
        if (fl) {
            w.flip(row, K, RW, k, res, fl);
            if (P.flips && (v ? it[s].own[1] : it[s].own[0])) nflip += __popc(fl);
        }
    };

    auto update_all = [&](uint32_t sweep, uint32_t slot, uint32_t col, int i) {
#pragma unroll
        for (int s = 0; s < M; ++s) update(s, sweep, slot, col, i);
    };
    auto end_of_sweep = [&](uint32_t swept) {
        // end of a sweep: the owned rows are exact (i <= halo)
        const bool sample = (uint64_t)swept + 1 == next_sample;
        if (sample) next_sample += P.stride;
        if (P.ring || sample) {
            const int nw = (hi - lo) * RW;
            const uint32_t* rb = sm + (lo - slo) * RW;
            uint64_t acc = 0;
            for (int w = tid; w < nw; w += nt) {
                const uint32_t x = rb[w];
                if (!x) continue;
                const int rr = w / RW;
                const int rem = w - rr * RW;
                const int pl = rem / K, k = rem - pl * K;
                if (P.ring) acc += word_hash(x, g, lo + rr, pl, k);
                if (sample) word_count_sliced(x, (int64_t)(lo + rr) * RW + rem, (int64_t)g.H * RW, P.counts);
            }
            if (P.ring) {
                for (int o = 16; o; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
                if ((tid & 31) == 0) s_red[tid >> 5] = acc;
                __syncthreads();
                if (tid == 0) {
                    unsigned long long t = 0;
                    for (int wv = 0; wv < nt / 32; ++wv) t += s_red[wv];
#ifdef TL_DEBUG
                    if (TL_IN(swept - P.sweep0, P.nsweeps, 209))
#endif
                        atomicAdd(P.ring + (swept - P.sweep0), t);
                }
            }
            __syncthreads();
        }
    };

    constexpr int passes_c = LAT == LAT_DOMINO ? 2 : LAT == LAT_LOZENGE ? 3 : 4;
    uint32_t sweep = P.sweep0, slot = 0;
    uint64_t done = 0;
    int cyc = 0;
    uint32_t col = colour_of(sweep, 0);
    draw(sweep, 0, col, 1);
    while (true) {
        const int hc = (int)((total - done) < (uint64_t)h ? (total - done) : (uint64_t)h);
        const bool last = done + (uint64_t)hc >= total;
        if constexpr (FIXED) {
            for (int i = 1; i <= hc; i += passes_c) {
#pragma unroll
                for (int p = 0; p < passes_c; ++p) {
                    update_all(sweep, (uint32_t)p, (uint32_t)p, i + p);
                    // the next pass's draws; after the last of a cycle they
                    // are made while the neighbours' rows are on their way
                    if (p + 1 < passes_c) draw(sweep, (uint32_t)p + 1u, (uint32_t)p + 1u, i + p + 1);
                    else if (i + p < hc) draw(sweep + 1u, 0u, 0u, i + p + 1);
                    __syncthreads();
                }
                end_of_sweep(sweep);
                ++sweep;
            }
        } else {
            for (int i = 1; i <= hc; ++i) {
                update_all(sweep, slot, col, i);
                const bool eos = slot + 1 == (uint32_t)passes;
                const uint32_t swept = sweep;
                slot = eos ? 0u : slot + 1;
                sweep += eos ? 1u : 0u;
                if (i < hc) {
                    col = colour_of(sweep, slot);
                    draw(sweep, slot, col, i + 1);
                }
                __syncthreads();
                if (eos) end_of_sweep(swept);
            }
        }
        done += (uint64_t)hc;
        if (last) break;
        col = colour_of(sweep, slot);
        if (C == 1) {
            draw(sweep, slot, col, 1);
            continue;
        }
        // ---- exchange: tagged 64-bit words, double-buffered by cycle parity ----
        // a status word raised anywhere (a wait that gave up in another CTA,
        // or raised by the host) ends every CTA at its next exchange: read
        // here, used at the end, so that its latency hides behind the exchange
        const int raised = tid == 0 ? *(volatile int*)P.status : 0;
        const size_t side_words = (size_t)h * RW;
        const int par = cyc & 1, half = h * RW / 2;   // 16-byte units per side
        const unsigned long long tag =
            ((unsigned long long)(((P.epoch & 0xFFFFu) << 16) | (unsigned)((cyc + 1) & 0xFFFF))) << 32;
        unsigned long long* const mine = P.xbuf + ((size_t)c * 4 + (size_t)par * 2) * side_words;
        for (int u = tid; u < 2 * half; u += nt) {
            const int side = u >= half, x = 2 * (u - (side ? half : 0));
            if (side ? top : bot) continue;
            const uint32_t* src = sm + ((side ? hi - h : lo) - slo) * RW + x;
            wd_st2(mine + (size_t)side * side_words + x, tag | src[0], tag | src[1]);
        }
        draw(sweep, slot, col, 1);
        int ok = 1;
        {
            constexpr int MAXU = 4;
            uint64_t t_wait = 0;
            // the stripe below publishes its upper rows as side 1, the one above its lower rows as side 0
            const unsigned long long* th0 = bot ? nullptr : P.xbuf + ((size_t)(c - 1) * 4 + (size_t)par * 2 + 1) * side_words;
            const unsigned long long* th1 = top ? nullptr : P.xbuf + ((size_t)(c + 1) * 4 + (size_t)par * 2) * side_words;
            for (int u0 = tid; u0 < 2 * half && ok; u0 += MAXU * nt) {
                unsigned long long a[MAXU], b[MAXU];
                unsigned need = 0;
#pragma unroll
                for (int j = 0; j < MAXU; ++j) {
                    const int u = u0 + j * nt, side = u >= half;
                    const unsigned long long* src = side ? th1 : th0;
                    if (u < 2 * half && src) {
                        need |= 1u << j;
                        wd_ld2(src + 2 * (u - (side ? half : 0)), &a[j], &b[j]);
                    }
                }
                for (unsigned spin = 1; need; ++spin) {
#pragma unroll
                    for (int j = 0; j < MAXU; ++j) {
                        if (!(need >> j & 1u)) continue;
                        if ((a[j] & 0xFFFFFFFF00000000ull) == tag && (b[j] & 0xFFFFFFFF00000000ull) == tag) {
                            const int u = u0 + j * nt, side = u >= half;
                            uint32_t* d = sm + ((side ? hi : lo - h) - slo) * RW + 2 * (u - (side ? half : 0));
                            d[0] = (uint32_t)a[j];
                            d[1] = (uint32_t)b[j];
                            need &= ~(1u << j);
                        }
                    }
                    if (!need) break;
                    // the limit and the status word are looked at every 16th
                    // round: their reads take as long as the poll's own
                    if ((spin & 15u) == 0u) {
                        const uint64_t now = wd_globaltimer();
                        if (!t_wait) t_wait = now;
                        if (*(volatile int*)P.status || now - t_wait > kWordWaitLimitNs) {
                            atomicExch(P.status, 1);
                            ok = 0;
                            break;
                        }
                    }
                    __nanosleep(32);
#pragma unroll
                    for (int j = 0; j < MAXU; ++j) {
                        if (!(need >> j & 1u)) continue;
                        const int u = u0 + j * nt, side = u >= half;
                        wd_ld2((side ? th1 : th0) + 2 * (u - (side ? half : 0)), &a[j], &b[j]);
                    }
                }
            }
        }
        if (raised) ok = 0;
        if (!__syncthreads_and(ok)) return;   // the state is undefined; the host reports TL_ETIMEOUT
        ++cyc;
    }
    if (gridDim.x > 1 && cyc == 0 &&
        !__syncthreads_and(tid != 0 || stripe_neighbours_loaded(P.loaded, P.epoch, P.status)))
        return;
    {
        uint4* d = reinterpret_cast<uint4*>(P.rows0 + (int64_t)lo * RW);
        const uint4* s = smem4 + (size_t)(lo - slo) * (RW / 4);
        for (int i = tid; i < (hi - lo) * (RW / 4); i += nt) __stcg(d + i, s[i]);
    }
    if (P.flips && nflip) atomicAdd(P.flips, (unsigned long long)nflip);
}

// Builds by threads and words per thread: fewer threads leave more registers
// (512: 128 each, 768: 80, 1024: 64).  A six-vertex word carries 8 random
// planes (12: 5.55 us a sweep of the square 2048 against 4.78, and 4: 4.89; the
// planes it carries are compared in the update's chain), 4 with four words a
// thread.
template <int LAT, int TK, bool CNT>
static const void* words_build(int threads, int slots, bool fixed)
{
    if (slots > 2) return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 1024, 4, 1, false>);
    if (slots == 2) return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 1024, 2, 2, false>);
    if (fixed) {
        if (threads <= 512) return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 512, 1, 2, true>);
        if (threads <= 768) return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 768, 1, 2, true>);
        return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 1024, 1, 2, true>);
    }
    if (threads <= 512) return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 512, 1, 2, false>);
    return reinterpret_cast<const void*>(&words_kernel<LAT, TK, CNT, 1024, 1, 2, false>);
}

}  // namespace tl
