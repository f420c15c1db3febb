// One-block kernel for small domino domains at t = 2^31: no stripes, no
// exchange, a thread per 32 sites.
//
// Up to 1,024 words of sites fit one CTA (Aztec diamonds to order 127), and
// then a pass is nothing but its own latency: the register kernel, a thread
// per 2 x 128 sites, spends 700 cycles a pass in one warp's chain of two
// Philox calls and two row updates.  Here
//  - the four lanes of a quad share the Philox outputs of their 128-site
//    group over time: lane q draws the plane of pass t + q, and a 4 x 4
//    transpose deals every lane its word of the next four passes, so a thread
//    draws once in four passes (one plane decides at t = 2^31);
//  - a thread keeps its row's horizontal edges (He, Ho) in registers; shared
//    memory holds the vertical planes, which two rows use in turn, and copies
//    of Ho for the word to the right;
//  - at parity p = 0 a word's first site also flips the top bit of the word
//    to its left: it leaves that bit in shared memory and the left word
//    applies it at its next pass (parity 1), so no word has two writers.
// Rows are laid out by parity, so that a warp's words are consecutive (in the
// packed layout they fall on the same banks: 0.46 us a sweep at order 32).
//
// Bound: the latency of a pass (two shared-memory round trips and a barrier)
// below order 40, then the issue of 20 instructions a warp and pass.  us a
// sweep of Aztec diamonds, register kernel -> this one: order 8 0.71 -> 0.20,
// 32 0.70 -> 0.24, 64 0.71 -> 0.35, 96 0.72 -> 0.45, 127 0.70 -> 0.57.
#include "tl_words.cuh"

#include <cstdint>

namespace tl {

struct SmallParams {
    uint32_t *rows_a, *rows_b;   // global row 0 of each chain (one block each)
    Geom g;
    uint32_t sweep0, nsweeps;
    DevRng rng;
    const int2* grange;
};

__global__ void __launch_bounds__(1024, 1) small_kernel(const SmallParams P)
{
    extern __shared__ uint4 smem4[];
    __shared__ __align__(16) uint32_t s_tr[32 * 8 * 20];
    const Geom& g = P.g;
    const int K = g.K, RW = (int)g.row_words, nt = blockDim.x, tid = threadIdx.x, q = tid & 3;
    uint32_t* const rows = (blockIdx.x ? P.rows_b : P.rows_a) - RW;   // row -1 (the pad row below)
    // shared memory: per plane (0: straddling flips, 1: Ho, 2: Ve, 3: Vo) the
    // even rows, then the odd rows from -1 on, K words each: a warp's rows have
    // one parity, so its words are consecutive, its own as well as those of the
    // rows below
    const int H = g.H, he_ = (H + 1) >> 1, PW = (H + 3) * K;
    uint32_t* const sm = reinterpret_cast<uint32_t*>(smem4);
    int* const off = reinterpret_cast<int*>(sm + (size_t)4 * PW);
    auto pos = [&](int y) { return (y & 1) ? he_ + 1 + (y >> 1) : y >> 1; };   // y >= -1 (-1 >> 1 is -1)
    uint32_t* const buf = s_tr + (tid >> 5) * 160 + ((tid & 31) >> 2) * 20;
    for (int i = tid; i < (H + 1) * RW; i += nt) {   // rows -1 .. H - 1
        const int yy = i / RW, rem = i - yy * RW, pl = rem / K;
        sm[pl * PW + pos(yy - 1) * K + (rem - pl * K)] = pl == 0 ? 0u : __ldcg(rows + i);
    }
    // items: the groups with sites and the one left of them (it holds the
    // edge their first site shares)
    auto row_groups = [&](int y) {
        int2 gr = P.grange[y];
        if (gr.y > gr.x && gr.x > 0) --gr.x;
        return gr;
    };
    // even rows first, then odd rows from the next warp on: a warp's rows have
    // one parity in every pass, so its branch on the parity is uniform
    auto slot_row = [&](int i) { return i < he_ ? 2 * i : 2 * (i - he_) + 1; };
    for (int i = tid; i < H; i += nt) {
        const int2 gr = row_groups(slot_row(i));
        off[i + 1] = gr.y > gr.x ? gr.y - gr.x : 0;
    }
    __syncthreads();
    if (tid == 0) {
        off[0] = 0;
        for (int i = 0; i < H; ++i) off[i + 1] += off[i];
    }
    __syncthreads();
    const int ne = off[he_], ne8 = (ne + 7) & ~7;
    const bool odd = (tid >> 2) >= ne8;
    const int item = odd ? (tid >> 2) - ne8 + ne : (tid >> 2);
    const bool act = item < (odd ? off[H] : ne);
    int y = odd ? 1 : 0, k = 0;
    uint32_t grp = 0;
    if (act) {
        int a = odd ? he_ : 0, b = (odd ? H : he_) - 1;
        while (a < b) {   // last slot whose first item is <= item
            const int mid = (a + b + 1) >> 1;
            if (off[mid] <= item) a = mid;
            else b = mid - 1;
        }
        y = slot_row(a);
        const int m = row_groups(y).x + (item - off[a]);
        k = 4 * m + q;
        grp = (uint32_t)(y * g.Kg + m);
    }
#ifdef TL_DEBUG
    const bool ok = !act || (TL_IN(y, g.H, 601) && TL_IN(k, K, 602));
#else
    constexpr bool ok = true;
#endif
    uint32_t* const row = sm + pos(y) * K + k;   // plane 0, word k of row y
    const bool left = k > 0, right = k + 1 < K;
    uint32_t he = 0, ho = 0;
    const bool live = act && ok;
    if (live) {
        he = __ldcg(rows + (y + 1) * RW + k);
        ho = row[PW];
    }
    GroupKey key;
    key.set(grp, P.rng);
    // words of passes 4u .. 4u + 3 (two sweeps)
    auto draws = [&](uint32_t u) {
        PlaneKey pk;
        pk.set(0u, (uint32_t)q & 1u, P.sweep0 + 2u * u + ((uint32_t)q >> 1), P.rng);
        const uint4 o = philox_keyed(key, pk, P.rng);
        __syncwarp();
        *reinterpret_cast<uint4*>(buf + 4 * q) = o;
        __syncwarp();
        return make_uint4(buf[q], buf[4 + q], buf[8 + q], buf[12 + q]);
    };
    // the pass at parity p of this row, with random word u
    uint32_t *const n0 = row + 2 * PW, *const s0 = sm + 2 * PW + pos(y - 1) * K + k;
    auto pass = [&](int p, uint32_t u) {
        if (live) {
            if (p) {
                const uint32_t n = n0[PW], s = s0[PW];
                // the flip that the word to the right left at p = 0
                ho ^= right ? row[1] << 31 : 0u;
                const uint32_t f = (ho & he & ~(n | s)) | (n & s & ~(ho | he));
                const uint32_t fl = f & (~u ^ ho);
                n0[PW] = n ^ fl;
                s0[PW] = s ^ fl;
                he ^= fl;
                ho ^= fl;
                row[PW] = ho;
            } else {
                const uint32_t n = n0[0], s = s0[0];
                // left edge of the first site: the top of the word to the left
                const uint32_t w = (ho << 1) | (left ? row[PW - 1] >> 31 : 0u);
                const uint32_t f = (he & w & ~(n | s)) | (n & s & ~(he | w));
                const uint32_t fl = f & (~u ^ he);
                n0[0] = n ^ fl;
                s0[0] = s ^ fl;
                he ^= fl;
                ho ^= fl >> 1;
                row[PW] = ho;
                row[0] = fl & 1u;
            }
        }
        __syncthreads();
    };
    __syncthreads();
    const int p0 = odd ? 1 : 0;   // parity of slot 0
    uint4 w = draws(0);
    const uint32_t blocks = P.nsweeps >> 1;
    for (uint32_t u = 0; u < blocks; ++u) {
        const uint4 c = w;
        pass(p0, c.x);
        w = draws(u + 1);
        pass(p0 ^ 1, c.y);
        pass(p0, c.z);
        pass(p0 ^ 1, c.w);
    }
    if (P.nsweeps & 1u) {
        pass(p0, w.x);
        pass(p0 ^ 1, w.y);
    }
    if (live) {
        // after the last pass (slot 1): a row at parity 0 there has flips to apply
        if (p0 == 1 && right) ho ^= row[1] << 31;
        uint32_t* const o = rows + (y + 1) * RW + k;
        o[0] = he;
        o[K] = ho;
    }
    for (int i = tid; i < H * RW; i += nt) {
        const int yy = i / RW, rem = i - yy * RW, pl = rem / K;
        if (pl >= 2) rows[RW + i] = sm[pl * PW + pos(yy) * K + (rem - pl * K)];
    }
}

size_t small_smem_bytes(const Geom& g) { return (size_t)(g.H + 3) * g.K * 16 + (size_t)(g.H + 1) * 4; }

// Threads for `even` and `odd` groups in even and odd rows.
int small_threads(long even, long odd) { return (int)(((even + 7) / 8 + (odd + 7) / 8) * 32 < 4096 ? ((even + 7) / 8 + (odd + 7) / 8) * 32 : 4096); }

// One limit for all chains: a plan must not lower another chain's.
int small_prepare(size_t smem_bytes, int threads, bool* fits)
{
    *fits = false;
    int dev = 0, optin = 0, bps = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, small_kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, small_kernel, threads, smem_bytes);
    if (e != cudaSuccess) cudaGetLastError();
    else *fits = bps > 0;
    return (int)e;
}

int launch_small(const Geom& g, uint32_t* rows_a, uint32_t* rows_b, int threads, uint32_t sweep0, uint32_t nsweeps,
                 const DevRng& rng, const int2* grange, void* stream)
{
    SmallParams P;
    P.rows_a = rows_a + g.row_words;
    P.rows_b = (rows_b ? rows_b : rows_a) + g.row_words;
    P.g = g;
    P.sweep0 = sweep0;
    P.nsweeps = nsweeps;
    P.rng = rng;
    P.grange = grange;
    small_kernel<<<rows_b ? 2 : 1, threads, small_smem_bytes(g), reinterpret_cast<cudaStream_t>(stream)>>>(P);
    return (int)cudaGetLastError();
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_small(unsigned long long* out, bool clear)
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
