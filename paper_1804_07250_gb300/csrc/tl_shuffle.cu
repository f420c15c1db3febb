// Domino shuffling: exact uniform random tilings of the Aztec diamond (the
// shuffling algorithms the paper names as an alternative exact sampler,
// Sec. 3; Elkies, Kuperberg, Larsen and Propp), in the face-local form of
// Propp's generalized domino-shuffling.
//
// Cells are unit squares with lower-left corner (x, y), x, y in [-n, n); in
// order k a horizontal domino with left cell (x, y) goes north if x + y + k
// is even, else south, a vertical one with bottom cell (x, y) east or west.
// Seen from the 2x2 blocks of cells with x + y + K odd (K = k + 1), every
// domino of order k lies along one side of exactly one such block of the
// order-K diamond and moves to the opposite side of it; two dominoes of one
// block destroy each other, and a block without any gets a new pair.  So a
// step is one bitwise update of the four edges of every block of one colour
// class, on the same packed edge planes as the chain's passes: with (X, Y)
// the canonical vertex in the middle of the block (X = x + 1 + n, Y = y + 1 +
// n), E = Hz(X, Y), W = Hz(X-1, Y), N = Vt(X, Y), S = Vt(X, Y-1):
//   E' = W & ~E | v,  W' = E & ~W | v,  N' = S & ~N | h,  S' = N & ~S | h,
// h and v the blocks with no edge whose draw picks a horizontal or a vertical
// pair.  All K^2 blocks cover all edges of the diamond, so a step rewrites
// every word in reach and the buffers alternate.
//
// Packed rows: planes He, Ho, Ve, Vo (edges at even and odd X), Kw words each.
// A row's class alternates its parity p = (Y + K + 1) & 1 every step.  At
// p = 0 the W edges are the odd plane moved up by one site; the step leaves
// them there (word j of Ho then holds the odd edges left of its sites), and
// the next step of the row, at p = 1, moves them back as it reads.  No
// word is ever shared by two writers.
#include "tl_words.cuh"

#include <cstdint>

namespace tl {

constexpr int kShufThreads = 512, kShufWarps = kShufThreads / 32;
// per warp: the blocks to fill of 32 words (at most 1024), and their draws
struct ShufScratch {
    uint16_t list[1024];
    uint32_t coin[32];
};
struct ShufParams {
    int n, Kw;                  // order, words per plane row (multiple of 4)
    int h;                      // halo rows per side = steps per exchange
    int K0, K1;                 // the launch runs steps K0 .. K1
    const int* stripe_lo;       // [C + 1] vertex rows, n - K1 .. n + K1 + 1
    DevRng rng;
    unsigned long long* xbuf;   // [C][2][2][4 h Kw] tagged words, cleared before step 1
    uint32_t* rows0;            // packed rows (chain layout), row 0: as step K0 - 1 left them, then as step K1 does
    int* status;
};
TL_DEV void sh_ld2(const unsigned long long* p, unsigned long long* a, unsigned long long* b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(*a), "=l"(*b) : "l"(p) : "memory");
}
TL_DEV void sh_st2(unsigned long long* p, unsigned long long a, unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
TL_DEV uint64_t sh_globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
constexpr uint64_t kShufWaitLimitNs = 2000000000ull;   // 2 s: far beyond any healthy exchange

// The draws of step K: bit 31 of word 0 of Philox4x32-10 with counter
// (c0, K, 0xFFFE0000, stream), clear for a horizontal pair.  Only c0 differs
// between the blocks of a step: the second product of round 1 is a constant
// and the first of round 2 the same for the whole step, and the last two
// rounds need one word each.  17 products per draw instead of 20.
struct ShufDraw {
    uint32_t a1, m2lo, m2hi;   // of the step
    uint32_t stream, k0, k1;
    TL_DEV ShufDraw(uint32_t K, const DevRng& rng)
    {
        constexpr uint64_t m = (uint64_t)0xFFFE0000u * 0xCD9E8D57u;
        a1 = (uint32_t)m;
        const uint32_t a0 = (uint32_t)(m >> 32) ^ K ^ rng.k0;
        m2lo = a0 * 0xD2511F53u;
        m2hi = __umulhi(a0, 0xD2511F53u);
        stream = rng.stream;
        k0 = rng.k0;
        k1 = rng.k1;
    }
    TL_DEV bool horizontal(uint32_t c0) const
    {
        uint32_t q0 = k0, q1 = k1;
        const uint32_t a2 = __umulhi(c0, 0xD2511F53u) ^ stream ^ q1, a3 = c0 * 0xD2511F53u;
        q0 += 0x9E3779B9u;
        q1 += 0xBB67AE85u;
        uint32_t x0 = __umulhi(a2, 0xCD9E8D57u) ^ a1 ^ q0, x1 = a2 * 0xCD9E8D57u, x2 = m2hi ^ a3 ^ q1, x3 = m2lo;
#pragma unroll
        for (int r = 2; r < 10; ++r) {
            q0 += 0x9E3779B9u;
            q1 += 0xBB67AE85u;
            const uint32_t lo0 = x0 * 0xD2511F53u, hi0 = __umulhi(x0, 0xD2511F53u);
            const uint32_t lo1 = x2 * 0xCD9E8D57u, hi1 = __umulhi(x2, 0xCD9E8D57u);
            x0 = hi1 ^ x1 ^ q0;
            x1 = lo1;
            x2 = hi0 ^ x3 ^ q1;
            x3 = lo0;
        }
        return (int)x0 >= 0;
    }
};

// Columns that step K can touch in rows at distance >= d from the middle row:
// words [lo, hi] of a plane row.
TL_DEV void sh_words(int n, int K, int d, int& lo, int& hi)
{
    const int w = K - 1 - d;
    lo = ((n - w - 1) >> 1) >> 5;
    hi = ((n + w) >> 1) >> 5;
}

// One warp's words of step K: lane's word k of row Y (`live` if it has one),
// read from `src` and written to `dst`, both pointing at row Y (pitch RW
// words; row Y - 1 holds the S edges).  The blocks to fill are sparse (a
// quarter of the blocks in the disordered region, none in the frozen
// corners) and uneven (8 +- 2.4 a word), and a draw costs a warp 68 cycles of
// its scheduler's multiplier, so the warp lists them and its lanes share the
// draws evenly, two in flight each.  Measured at order 2048 (512 threads): 7.3 ms a sample;
// 9.5 with every lane drawing for its own word, 8.6 with the lanes drawing
// for their own words until fewer than 20 have a block left.
TL_DEV void sh_step_words(const uint32_t* src, uint32_t* dst, int Kw, int n, int K, int Y, int k, bool live,
                          const ShufDraw& draw, ShufScratch& sc)
{
    const int lane = threadIdx.x & 31;
    const int RW = 4 * Kw;
    const int p = (Y + K + 1) & 1;
    uint32_t A = 0, B = 0, N = 0, S = 0, fill = 0;
    if (live) {
        const uint32_t* V = src + (2 + p) * Kw + k;
        A = src[k];
        const uint32_t ho = src[Kw + k];
        const bool in = p ? k + 1 < Kw : k > 0;
        const uint32_t adj = in ? src[Kw + k + (p ? 1 : -1)] : 0u;
        B = p ? (ho >> 1) | (adj << 31) : (ho << 1) | (adj >> 31);
        N = V[0];
        S = V[-RW];
        const int w = K - 1 - (Y > n ? Y - n : n - Y);
        fill = ~(A | B | N | S) & span_mask(((n - w - p) >> 1) - 32 * k, ((n + w - p) >> 1) - 32 * k);
    }
    uint32_t hor = 0;
    if (__any_sync(0xFFFFFFFFu, fill != 0u)) {
        // counter word 0 of bit 0 of this lane's word: (Y - 1) << 16 | (X - 1)
        const uint32_t base = ((uint32_t)(Y - 1) << 16) + (uint32_t)(64 * k + p - 1);
        const int cnt = __popc(fill);
        int off = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, off, o);
            if (lane >= o) off += v;
        }
        const int total = __shfl_sync(0xFFFFFFFFu, off, 31);
        off -= cnt;
        sc.coin[lane] = 0u;
        // from the top: one trip to the special-function unit a block (lowest
        // first takes two, and the list as long as the draws)
        for (uint32_t m = fill; m;) {
            const int j = 31 - __clz((int)m);
            sc.list[off++] = (uint16_t)((lane << 5) | j);
            m ^= 1u << j;
        }
        __syncwarp();
        for (int i0 = 0; i0 < total; i0 += 64) {
            // two draws a lane in flight
            const int ia = i0 + lane, ib = ia + 32;
            const uint32_t ea = ia < total ? sc.list[ia] : 0u, eb = ib < total ? sc.list[ib] : 0u;
            const uint32_t ca = __shfl_sync(0xFFFFFFFFu, base, ea >> 5) + 2u * (ea & 31u);
            if (i0 + 32 < total) {
                const uint32_t cb = __shfl_sync(0xFFFFFFFFu, base, eb >> 5) + 2u * (eb & 31u);
                const bool ha = draw.horizontal(ca), hb = draw.horizontal(cb);
                if (ha) atomicOr(&sc.coin[ea >> 5], 1u << (ea & 31u));
                if (hb && ib < total) atomicOr(&sc.coin[eb >> 5], 1u << (eb & 31u));
            } else if (draw.horizontal(ca) && ia < total) {
                atomicOr(&sc.coin[ea >> 5], 1u << (ea & 31u));
            }
        }
        __syncwarp();
        hor = sc.coin[lane];
        __syncwarp();
    }
    if (live) {
        const uint32_t ver = fill & ~hor;
        uint32_t* V = dst + (2 + p) * Kw + k;
        dst[k] = (B & ~A) | ver;
        dst[Kw + k] = (A & ~B) | ver;
        V[0] = (S & ~N) | hor;
        V[-RW] = (N & ~S) | hor;
    }
}

// The odd plane of row Y after step K, moved back if the row's class had p = 0.
TL_DEV uint32_t sh_plain_odd(const uint32_t* row, int Kw, int Y, int K, int k)
{
    const uint32_t o = row[Kw + k];
    if ((Y + K + 1) & 1) return o;
    return (o >> 1) | ((k + 1 < Kw ? row[Kw + k + 1] : 0u) << 31);
}

// Steps K0 .. K1 in one cooperative launch: every CTA keeps a stripe of rows
// and h rows on each side in shared memory (two copies, alternating by step),
// runs h steps while the exact region shrinks by one row per step and side,
// then swaps boundary rows with its neighbours (64-bit words: cycle tag,
// data).  Stripes the diamond has not reached yet do nothing, and a seam
// starts its exchanges a few rows before the diamond arrives.
//
// Bound: the draws (about K^2 / 6 Philox calls in step K) in the middle
// stripes, and below order 500 the latency of a step (a dependent read, list,
// draw and write per word, one barrier).
template <int NT>
__global__ void __launch_bounds__(NT, 1) shuffle_kernel(const ShufParams P)
{
    extern __shared__ uint4 smem4[];
    __shared__ ShufScratch s_scr[NT / 32];
    const int n = P.n, Kw = P.Kw, RW = 4 * Kw, h = P.h;
    const int c = blockIdx.x, C = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lo = P.stripe_lo[c], hi = P.stripe_lo[c + 1];
    const bool bot = c == 0, top = c == C - 1;
    const int slo = bot ? lo : lo - h, shi = top ? hi : hi + h;
    const int nloc = shi - slo;
    uint32_t* const buf0 = reinterpret_cast<uint32_t*>(smem4);
    const int bwords = nloc * RW;
    {
        // rows of the diamond so far into the first copy; the second is
        // written before it is read, except where the diamond has not been
        const uint4* g = reinterpret_cast<const uint4*>(P.rows0 + (int64_t)slo * RW);
        for (int i = tid; i < bwords / 4; i += NT) {
            smem4[i] = P.K0 > 1 ? __ldcg(g + i) : make_uint4(0u, 0u, 0u, 0u);
            smem4[bwords / 4 + i] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    __syncthreads();
    int cur = 0;
    const size_t side_words = (size_t)h * RW;
    for (int Kc = P.K0;; Kc += h) {
        const int hc = P.K1 - Kc + 1 < h ? P.K1 - Kc + 1 : h;
        // for all steps of the cycle: the words of the widest row that its last
        // step reaches, and the same number of words for every warp and turn
        // (fewer than 32 spread a small step's draws over more warps)
        uint32_t nw = 1, per = 4;
        int klo = 0;
        {
            const int K = Kc + hc - 1, ya = slo + 1, yb = shi;
            const int r0 = ya > n - K + 1 ? ya : n - K + 1, r1 = yb < n + K ? yb : n + K;
            if (r1 > r0) {
                const int dmin = r0 > n ? r0 - n : (r1 <= n ? n - (r1 - 1) : 0);
                int khi;
                sh_words(n, K, dmin, klo, khi);
                nw = (uint32_t)(khi - klo + 1);
                const uint32_t total = (uint32_t)(r1 - r0) * nw;
                const uint32_t turns = (total + NT - 1) / NT;
                per = (uint32_t)__float2int_ru(__fdividef((float)total, (float)(turns * (NT / 32))));
                per = per < 4u ? 4u : (per > 32u ? 32u : per);
            }
        }
        // t / nw: exact, since t < 2^20 keeps the rounding below half of 1 / nw
        const float inv = __frcp_rn((float)nw);
        for (int i = 1; i <= hc; ++i) {
            const int K = Kc + i - 1;
            // rows whose inputs are exact and that the order-K diamond reaches
            const int ya = bot ? slo + 1 : slo + i, yb = top ? shi : shi - (i - 1);
            const int r0 = ya > n - K + 1 ? ya : n - K + 1, r1 = yb < n + K ? yb : n + K;
            if (r1 <= r0) continue;
            const uint32_t total = (uint32_t)(r1 - r0) * nw;
            const uint32_t* src = buf0 + cur * bwords;
            uint32_t* dst = buf0 + (cur ^ 1) * bwords;
            const ShufDraw draw((uint32_t)K, P.rng);
            for (uint32_t t0 = (uint32_t)warp * per; t0 < total; t0 += per * (NT / 32)) {
                const uint32_t t = t0 + (uint32_t)lane;
                const uint32_t rr = (uint32_t)(((float)t + 0.5f) * inv);
                const int Y = r0 + (int)rr, k = klo + (int)(t - rr * nw);
                bool live = t < total && (uint32_t)lane < per;
#ifdef TL_DEBUG
                // rows Y - 1 and Y are local, word k lies in a plane row
                if (live && !(TL_IN(Y - 1 - slo, nloc, 501) && TL_IN(Y - slo, nloc, 501) && TL_IN(k, Kw, 502)))
                    live = false;
#endif
                sh_step_words(src + (Y - slo) * RW, dst + (Y - slo) * RW, Kw, n, K, Y, k, live, draw,
                              s_scr[warp]);
            }
            cur ^= 1;
            __syncthreads();
        }
        const int K = Kc + hc - 1;
        if (K >= P.K1) break;
        // ---- exchange with the stripes below and above, where the diamond is
        // within reach of the seam (both sides decide alike) ----
        const int reach = K + 2 * h + 2;
        const bool xb = !bot && lo - n <= reach && n - lo <= reach, xt = !top && hi - n <= reach && n - hi <= reach;
        if (!xb && !xt) continue;
        // the order of the rows names the exchange (never 0, increasing over
        // the launches of a sample); the copy alternates within a launch
        const unsigned long long tag = (unsigned long long)(uint32_t)K << 32;
        const int raised = tid == 0 ? *(volatile int*)P.status : 0;   // used at the end of the exchange
        const int par = ((Kc - P.K0) / h) & 1;
        // words that can be non-zero after step K, in pairs
        const int e0 = (n - K) >> 1, e1 = ((n + K) >> 1) + 1;
        const int xk0 = ((e0 > 0 ? e0 - 1 : 0) >> 5) & ~1;
        const int xk1 = ((e1 >> 5) < Kw ? (e1 >> 5) : Kw - 1) | 1;
        const int npw = (xk1 - xk0 + 1) >> 1, units = 4 * h * npw;
        uint32_t* const st = buf0 + cur * bwords;
        unsigned long long* const mine = P.xbuf + ((size_t)c * 2 + par) * 2 * side_words;
        for (int u = tid; u < 2 * units; u += NT) {
            const int s = u >= units, v = u - (s ? units : 0);
            if (!(s ? xt : xb)) continue;
            const int rp = v / npw, wd = rp * Kw + xk0 + 2 * (v - rp * npw);   // (row, plane) block, word pair
#ifdef TL_DEBUG
            if (!TL_IN(wd + 1, (int64_t)side_words, 503)) continue;
#endif
            const uint32_t* a = st + ((s ? hi - h : lo) - slo) * RW + wd;
            sh_st2(mine + (size_t)s * side_words + wd, tag | a[0], tag | a[1]);
        }
        int ok = 1;
        uint64_t t_wait = 0;
        for (int u = tid; u < 2 * units && ok; u += NT) {
            const int s = u >= units, v = u - (s ? units : 0);
            if (!(s ? xt : xb)) continue;
            const int rp = v / npw, wd = rp * Kw + xk0 + 2 * (v - rp * npw);
#ifdef TL_DEBUG
            if (!TL_IN(wd + 1, (int64_t)side_words, 504)) continue;
#endif
            // the neighbour below publishes its upper rows as side 1, the one above its lower rows as side 0
            const unsigned long long* from =
                P.xbuf + (((size_t)(s ? c + 1 : c - 1) * 2 + par) * 2 + (s ? 0 : 1)) * side_words + wd;
            unsigned long long a, b;
            for (unsigned spin = 1;; ++spin) {
                sh_ld2(from, &a, &b);
                if ((a >> 32) == (tag >> 32) && (b >> 32) == (tag >> 32)) break;
                // the limit and the status word are looked at every 16th
                // round: their reads take as long as the poll's own
                if ((spin & 15u) == 0u) {
                    const uint64_t now = sh_globaltimer();
                    if (!t_wait) t_wait = now;
                    if (*(volatile int*)P.status || now - t_wait > kShufWaitLimitNs) {
                        atomicExch(P.status, 1);
                        ok = 0;
                        break;
                    }
                }
                __nanosleep(32);
            }
            uint32_t* d = st + ((s ? hi : lo - h) - slo) * RW + wd;
            d[0] = (uint32_t)a;
            d[1] = (uint32_t)b;
        }
        if (raised) ok = 0;
        if (!__syncthreads_and(ok)) return;   // the host reports the timeout
    }
    const uint32_t* st = buf0 + cur * bwords;
    for (int i = tid; i < (hi - lo) * RW; i += NT) {
        const int rr = i / RW, rem = i - rr * RW, pl = rem / Kw, k = rem - pl * Kw;
        const uint32_t* row = st + (lo + rr - slo) * RW;
        P.rows0[(int64_t)lo * RW + i] = pl == 1 && P.K1 == n ? sh_plain_odd(row, Kw, lo + rr, n, k) : row[rem];
    }
}

// One step with the rows in global memory (diamonds whose stripes do not fit
// the SMs' shared memory): A is read, B written, both with a pad row below row
// 0 and zero wherever the diamond has not been.
__global__ void __launch_bounds__(kShufThreads) shuffle_step_kernel(const uint32_t* __restrict__ A,
                                                                    uint32_t* __restrict__ B, int n, int Kw, int K,
                                                                    DevRng rng)
{
    __shared__ ShufScratch s_scr[kShufWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t RW = 4 * (int64_t)Kw;
    const int d = (int)blockIdx.y < K ? K - 1 - (int)blockIdx.y : (int)blockIdx.y - (K - 1);
    const int Y = n - (K - 1) + (int)blockIdx.y;
    int klo, khi;
    sh_words(n, K, d, klo, khi);
    const ShufDraw draw((uint32_t)K, rng);
    for (int k0 = klo + (int)(blockIdx.x * kShufWarps + warp) * 32; k0 <= khi; k0 += (int)gridDim.x * kShufThreads) {
        bool live = k0 + lane <= khi;
#ifdef TL_DEBUG
        if (live && !(TL_IN(Y, 2 * n + 1, 505) && TL_IN(k0 + lane, Kw, 506))) live = false;
#endif
        sh_step_words(A + (int64_t)Y * RW, B + (int64_t)Y * RW, Kw, n, K, Y, k0 + lane, live, draw, s_scr[warp]);
    }
}

// The odd planes of B after the last step, moved back, into A (whose other
// planes are copied).
__global__ void shuffle_plain_kernel(const uint32_t* __restrict__ B, uint32_t* __restrict__ A, int n, int Kw)
{
    const int64_t RW = 4 * (int64_t)Kw, total = (2 * (int64_t)n + 1) * RW;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int Y = (int)(i / RW), rem = (int)(i - Y * RW), pl = rem / Kw, k = rem - pl * Kw;
        A[i] = pl == 1 ? sh_plain_odd(B + Y * RW, Kw, Y, n, k) : B[i];
    }
}

static inline cudaStream_t SS_(void* s) { return reinterpret_cast<cudaStream_t>(s); }

size_t shuffle_smem_bytes(int nloc, int Kw) { return (size_t)nloc * 4 * Kw * 4 * 2; }

static const void* shuffle_pick(int threads)
{
    return threads > 512 ? reinterpret_cast<const void*>(&shuffle_kernel<768>)
                         : reinterpret_cast<const void*>(&shuffle_kernel<512>);
}

int shuffle_prepare_kernel(int threads, size_t smem_bytes, int* blocks_per_sm)
{
    *blocks_per_sm = 0;
    const void* k = shuffle_pick(threads);
    // one limit for all orders: a context must not lower another's
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, threads, smem_bytes);
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

size_t shuffle_static_smem(int threads) { return sizeof(ShufScratch) * (size_t)(threads / 32); }

int launch_shuffle(const ShufflePlan* seg, int nseg, int n, int Kw, size_t total_words, size_t xbuf_words,
                   uint32_t* rows, const DevRng& rng, void* stream)
{
    cudaError_t e = cudaMemsetAsync(seg[0].xbuf, 0, xbuf_words * sizeof(unsigned long long), SS_(stream));
    // rows the first launches do not cover
    if (e == cudaSuccess) e = cudaMemsetAsync(rows, 0, total_words * 4, SS_(stream));
    for (int i = 0; i < nseg && e == cudaSuccess; ++i) {
        ShufParams P;
        P.n = n;
        P.Kw = Kw;
        P.h = seg[i].halo;
        P.K0 = i ? seg[i - 1].last + 1 : 1;
        P.K1 = seg[i].last;
        P.stripe_lo = seg[i].stripe_lo;
        P.rng = rng;
        P.xbuf = seg[i].xbuf;
        P.rows0 = rows + 4 * (size_t)Kw;
        P.status = seg[i].status;
        void* args[] = {&P};
        e = cudaLaunchCooperativeKernel(shuffle_pick(seg[i].threads), dim3(seg[i].ctas), dim3(seg[i].threads), args,
                                        seg[i].smem_bytes, SS_(stream));
    }
    return (int)e;
}

int launch_shuffle_global(int n, int Kw, size_t total_words, uint32_t* A, uint32_t* B, const DevRng& rng, void* stream)
{
    const cudaStream_t s = SS_(stream);
    cudaError_t e = cudaMemsetAsync(A, 0, total_words * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(B, 0, total_words * 4, s);
    if (e != cudaSuccess) return (int)e;
    uint32_t *src = A + 4 * (size_t)Kw, *dst = B + 4 * (size_t)Kw;   // row 0, after the pad row
    for (int K = 1; K <= n; ++K) {
        const int words = ((2 * K) >> 6) + 2;   // of the widest row, with both ragged ends
        const dim3 grid((words + kShufThreads - 1) / kShufThreads, 2 * K - 1);
        shuffle_step_kernel<<<grid, kShufThreads, 0, s>>>(src, dst, n, Kw, K, rng);
        uint32_t* t = src;
        src = dst;
        dst = t;
    }
    // src holds the sample; the plain planes go to A
    shuffle_plain_kernel<<<2048, 256, 0, s>>>(src, dst, n, Kw);
    if (dst != A + 4 * (size_t)Kw) {
        e = cudaMemcpyAsync(A, B, total_words * 4, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return (int)e;
    }
    return (int)cudaGetLastError();
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_shuffle(unsigned long long* out, bool clear)
{
#ifdef TL_DEBUG
    return tl_dbg_fetch(out, clear);
#else
    (void)out;
    (void)clear;
    return (int)cudaErrorNotSupported;
#endif
}

}  // namespace tl
