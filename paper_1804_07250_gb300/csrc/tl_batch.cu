// Batched chains: one launch advances every tile of every chain by R sweeps.
//
// Many independent chains of uneven size (the batched workload of Sec. 4's
// sampling experiments) are cut into row stripes ("tiles").  A CTA takes
// tiles from a work list ordered largest first, loads a tile plus a halo of
// passes * R rows from the chain's source buffer into shared memory, runs the
// R sweeps there with the exact region shrinking one row per pass, and writes
// only the tile's own rows to the destination buffer.  Because tiles of one
// chain run concurrently within a launch, a launch reads one buffer and
// writes the other; consecutive launches alternate.  Sweep indices come from
// a per-chain device counter, so a block of launches captured in a CUDA graph
// can be replayed: the graph ends with a kernel that advances the counters.
#include "tl_words.cuh"

#include <cstdint>

namespace tl {

// Bulk asynchronous copies (the copy engine of sm_90+, cp.async.bulk) between
// global and shared memory, completed through an mbarrier (loads) or a bulk
// group (stores).  Addresses 16-byte aligned, sizes multiples of 16 bytes.
TL_DEV uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
TL_DEV void mbar_init(unsigned long long* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
TL_DEV void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
TL_DEV bool mbar_try_wait(unsigned long long* bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
TL_DEV uint64_t batch_globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Wait for the phase of `parity` to complete, at most about two seconds.
TL_DEV bool mbar_wait_bounded(unsigned long long* bar, uint32_t parity)
{
    const uint64_t t0 = batch_globaltimer();
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0 && batch_globaltimer() - t0 > 2000000000ull) return false;
    }
}
TL_DEV void bulk_store(void* dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
TL_DEV void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
TL_DEV void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
TL_DEV void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

struct TileView {
    uint32_t* sm;              // row slo
    const uint32_t* items;     // (row - slo) << 8 | group; six-vertex: of the even row of the pair
    const int* off;            // first item of every row (pair) from r0 on
    const uint32_t* ttab;      // six-vertex table, expanded; or
    const uint32_t* ctab;      // its count form, expanded (nullptr: general)
    uint4* pk;                 // [2][32] plane keys of a pass, by its parity
    int r0;
    int slo, shi;
    bool bot, top;
};

// Random planes of one group: 16 of Philox's 20 products, the rest in the
// group's key and in the pass's table of plane keys.
struct RndKeyed {
    GroupKey key;
    const uint4* pk;
    DevRng rng;
    TL_DEV uint4 operator()(int k) const
    {
        const uint4 v = pk[k];
        const PlaneKey p{v.x, v.y, v.z};
        return philox_keyed(key, p, rng);
    }
};
// Two planes compared as one subtraction (borrow out: less; no difference:
// undecided).
TL_DEV void hb_pair(uint32_t& lt, uint32_t& und, uint32_t u0, uint32_t t0, uint32_t u1, uint32_t t1)
{
    const uint32_t l = (~u0 & t0) | (~(u0 ^ t0) & ~u1 & t1);
    lt |= und & l;
    und &= ~(u0 ^ t0) & ~(u1 ^ t1);
}
template <class TB>
TL_DEV uint4 heat_bath(uint4 f, int kmax, const RndKeyed& rnd, const TB& tb)
{
    uint4 und = f;
    uint4 lt = make_uint4(0u, 0u, 0u, 0u);
    int k = 0;
    for (; k + 1 <= kmax; k += 2) {
        if (!any4(und)) return lt;
        const uint4 o0 = rnd(k), o1 = rnd(k + 1);
        const uint4 t0 = tb(k), t1 = tb(k + 1);
        hb_pair(lt.x, und.x, o0.x, t0.x, o1.x, t1.x);
        hb_pair(lt.y, und.y, o0.y, t0.y, o1.y, t1.y);
        hb_pair(lt.z, und.z, o0.z, t0.z, o1.z, t1.z);
        hb_pair(lt.w, und.w, o0.w, t0.w, o1.w, t1.w);
    }
    if (k <= kmax && any4(und)) hb_compare(lt, und, rnd(k), tb(k));
    return lt;
}

template <int LAT, int TK, int NT>
TL_DEV void tile_passes(const BatchChain& ch, const TileView& t, uint32_t sweep0, int R)
{
    constexpr bool SIX = LAT == LAT_SIXV;
    const Geom& g = ch.g;
    const int64_t RW = g.row_words;
    const int Kg = g.Kg, passes = g.passes;
    const DevRng rng = ch.rng;
    int i = 0;
    for (int r = 0; r < R; ++r) {
        const uint32_t sweep = sweep0 + (uint32_t)r;
        for (int p = 0; p < passes; ++p, ++i) {
            const uint32_t pass = (uint32_t)p;
            const int vlo = t.bot ? -1 : t.slo + i;
            const int vhi = t.top ? g.H + 1 : t.shi - i;
            // exact rows [a, b) (six-vertex: face rows), and their items
            int a, b;
            if (SIX) {
                a = vlo > 1 ? vlo : 1;
                b = ((vhi - 2) < (g.N - 1) ? (vhi - 2) : (g.N - 1)) + 1;
            } else {
                a = (vlo + 1) > 0 ? (vlo + 1) : 0;
                b = vhi < g.H ? vhi : g.H;
            }
            const int v = SIX ? sixv_py(pass) : 0;
            int s = 0, e = 0;
            if (b > a) {
                s = t.off[(SIX ? a >> 1 : a) - t.r0];
                e = t.off[(SIX ? ((b - 1) >> 1) + 1 : b) - t.r0];
            }
            // the next pass's plane keys
            if (threadIdx.x < 32) {
                const bool wrap = p + 1 == passes;
                PlaneKey k;
                k.set(threadIdx.x, wrap ? 0u : pass + 1u, wrap ? sweep + 1u : sweep, rng);
                t.pk[((i + 1) & 1) * 32 + threadIdx.x] = make_uint4(k.l1, k.l0, k.h0, 0u);
            }
            for (int x = s + (int)threadIdx.x; x < e; x += NT) {
                const uint32_t en = t.items[x];
                const int y = t.slo + (int)(en >> 8) + v, m = (int)(en & 255u);
                if (SIX && (y < a || y >= b)) continue;
                RndKeyed rnd;
                rnd.key.set((uint32_t)((SIX ? y >> 1 : y) * Kg + m), rng);
                rnd.pk = t.pk + (i & 1) * 32;
                rnd.rng = rng;
                group_update<LAT, TK>(t.sm + (int64_t)(y - t.slo) * RW, RW, g, y, m, pass, rnd, ch.th, t.ttab, t.ctab);
            }
            __syncthreads();
        }
    }
}

// NT threads per tile: the plan's 256 or 128, or 512 where a launch has too few
// tiles to fill the SMs that way.  Registers without spills (128 a
// thread) beat more threads: 128 weighted diamonds of order 16 to 512, read
// out after 500 sweeps, take 6.9 ms at 512 threads an SM, 7.4 at 768 (80
// registers), 7.7 at 1,024; a lane per 32 sites instead of per 128 (a quad
// sharing the Philox outputs) 9.6: its update costs as much per word as this
// one per group.
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) batch_kernel(const BatchChain* __restrict__ chains,
                                                              const BatchTile* __restrict__ tiles, int ntiles, int R,
                                                              uint32_t sweep_off, int src, unsigned int* cursor,
                                                              int* __restrict__ status)
{
    extern __shared__ uint4 smem4[];
    __shared__ int s_tile;
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ uint4 s_pk[2 * 32];
    __shared__ __align__(16) uint32_t s_ttab[32 * 16];   // expanded six-vertex table
    const int tid = threadIdx.x;
    uint32_t* sm = reinterpret_cast<uint32_t*>(smem4);
    if (tid == 0) mbar_init(&s_bar, 1);
    __syncthreads();
    uint32_t parity = 0;
    // a block's first tile is its own index, and a grid that covers the tiles
    // asks for no second one
    for (bool own = true;; own = false) {
        if (!own && (int)gridDim.x >= ntiles) break;
        // a raised status word (a wait that gave up elsewhere, or raised by
        // the host) stops the block before it issues another copy
        if (tid == 0)
            s_tile = *(volatile int*)status ? ntiles
                     : own                  ? (int)blockIdx.x
                                            : (int)(gridDim.x + atomicAdd(cursor, 1u));
        __syncthreads();
        const int t = s_tile;
        __syncthreads();
        if (t >= ntiles) break;
        const BatchTile tile = tiles[t];
        const BatchChain& ch = chains[tile.chain];
        const Geom& g = ch.g;
        const int64_t RW = g.row_words;
        const int halo = g.passes * R;
        const bool bot = tile.lo == 0, top = tile.hi == g.H;
        TileView tv;
        tv.slo = bot ? -1 : (tile.lo - halo > -1 ? tile.lo - halo : -1);
        tv.shi = top ? g.H + 1 : (tile.hi + halo < g.H + 1 ? tile.hi + halo : g.H + 1);
        // a halo clamped at a pad row is exact from then on
        tv.bot = tv.slo == -1;
        tv.top = tv.shi == g.H + 1;
        const int nloc = tv.shi - tv.slo;
        const uint32_t* srcp = ch.rows[src] + RW;   // global row 0
        uint32_t* dstp = ch.rows[src ^ 1] + RW;
        // rows (pairs of face rows) with items, and their prefix counts
        const bool six = g.lattice == LAT_SIXV;
        const int r1 = tv.shi < g.H ? tv.shi : g.H;
        tv.r0 = tv.slo > 0 ? tv.slo : 0;
        if (six) tv.r0 >>= 1;
        const int nr = (six ? (r1 + 1) >> 1 : r1) - tv.r0;
        int* const off = reinterpret_cast<int*>(sm + (int64_t)nloc * RW);
        uint32_t* const items = reinterpret_cast<uint32_t*>(off + nr + 1);
#ifdef TL_DEBUG
        {
            // the tile, its halo rows and its item table fit the block's shared memory
            uint32_t dyn;
            asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
            const int64_t need = (int64_t)nloc * RW * 4 + 4 * (nr + 1) + 4 * (int64_t)(ch.gpre[tv.r0 + nr] - ch.gpre[tv.r0]);
            if (!TL_IN(need - 1, (int64_t)dyn, 301)) continue;
        }
#endif
        // the tile and its halo rows are contiguous: one bulk copy into shared
        // memory (rows are whole 16-byte units, buffers 256-byte aligned)
        if (tid == 0) bulk_load(sm, srcp + (int64_t)tv.slo * RW, (uint32_t)((int64_t)nloc * RW * 4), &s_bar);
        const int first = ch.gpre[tv.r0];
        for (int r = tid; r <= nr; r += NT) off[r] = ch.gpre[tv.r0 + r] - first;
        for (int r = tid; r < nr; r += NT) {
            const int x0 = ch.gpre[tv.r0 + r] - first, n = ch.gpre[tv.r0 + r + 1] - first - x0;
            const int m0 = ch.gfirst[tv.r0 + r], y = (six ? 2 : 1) * (tv.r0 + r);
            for (int j = 0; j < n; ++j) items[x0 + j] = (uint32_t)(y - tv.slo) << 8 | (uint32_t)(m0 + j);
        }
        if (six) {
            // threshold bits by corner index, or (count form) by corner count
            if (ch.th.cpol < 0)
                for (int x = tid; x < 32 * 16; x += NT)
                    s_ttab[x] = ((ch.th.tmask[x >> 4] >> (x & 15)) & 1u) ? 0xFFFFFFFFu : 0u;
            else
                for (int x = tid; x < 32 * 8; x += NT) {
                    const int n = x & 7;
                    s_ttab[x] = (n < 5 && ((ch.th.t5[n] >> (31 - (x >> 3))) & 1u)) ? 0xFFFFFFFFu : 0u;
                }
        }
        const uint32_t sweep0 = *ch.sweep_base + sweep_off;
        if (tid < 32) {
            PlaneKey k;
            k.set((uint32_t)tid, 0u, sweep0, ch.rng);
            s_pk[tid] = make_uint4(k.l1, k.l0, k.h0, 0u);
        }
        const int arrived = __syncthreads_and(mbar_wait_bounded(&s_bar, parity) ? 1 : 0);
        parity ^= 1u;
        if (!arrived) {
            // the copy did not complete in two seconds: report, give the copy
            // one more bounded wait so that nothing is left writing this
            // block's shared memory, and stop (every thread of the block
            // takes this branch together)
            if (tid == 0) {
                atomicExch(status, 1);
                mbar_wait_bounded(&s_bar, parity ^ 1u);
            }
            __syncthreads();
            return;
        }
        tv.sm = sm;
        tv.items = items;
        tv.off = off;
        tv.ttab = s_ttab;
        tv.ctab = six && ch.th.cpol >= 0 ? s_ttab : nullptr;
        tv.pk = s_pk;
        if (g.lattice == LAT_DOMINO) {
            if (ch.th.kind == THR_SITE) tile_passes<LAT_DOMINO, THR_SITE, NT>(ch, tv, sweep0, R);
            else tile_passes<LAT_DOMINO, THR_SCALAR, NT>(ch, tv, sweep0, R);
        } else if (g.lattice == LAT_LOZENGE) {
            if (ch.th.kind == THR_SITE) tile_passes<LAT_LOZENGE, THR_SITE, NT>(ch, tv, sweep0, R);
            else tile_passes<LAT_LOZENGE, THR_SCALAR, NT>(ch, tv, sweep0, R);
        } else {
            tile_passes<LAT_SIXV, THR_TABLE, NT>(ch, tv, sweep0, R);
        }
        // the tile's own rows back in one bulk copy; shared memory is reused
        // by the next tile once the copy has read it
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            bulk_store(dstp + (int64_t)tile.lo * RW, sm + (int64_t)(tile.lo - tv.slo) * RW,
                       (uint32_t)((int64_t)(tile.hi - tile.lo) * RW * 4));
            bulk_wait_read();
        }
        // the pad rows of the destination stay zero: they are never written
        __syncthreads();
    }
    if (tid == 0) bulk_wait_all();
}

__global__ void batch_advance_kernel(const BatchChain* __restrict__ chains, int nchains, uint32_t k,
                                     unsigned int* cursors, int ncursors)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nchains; i += gridDim.x * blockDim.x)
        *chains[i].sweep_base += k;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncursors; i += gridDim.x * blockDim.x) cursors[i] = 0u;
}

static const void* batch_pick(int threads)
{
    return threads == 128   ? reinterpret_cast<const void*>(&batch_kernel<128>)
           : threads == 256 ? reinterpret_cast<const void*>(&batch_kernel<256>)
                            : reinterpret_cast<const void*>(&batch_kernel<512>);
}

int batch_prepare(size_t smem_bytes, int threads, int* blocks_per_sm)
{
    const void* k = batch_pick(threads);
    // the largest limit, whatever this plan needs: a plan must not lower
    // another batch's
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, threads, smem_bytes);
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

int launch_batch(const BatchChain* chains, const BatchTile* tiles, int ntiles, int R, uint32_t sweep_off, int src,
                 unsigned int* cursor, int grid, int threads, size_t smem_bytes, int* status, void* stream)
{
    void* args[] = {&chains, &tiles, &ntiles, &R, &sweep_off, &src, &cursor, &status};
    return (int)cudaLaunchKernel(batch_pick(threads), dim3(grid), dim3(threads), args, smem_bytes,
                                 reinterpret_cast<cudaStream_t>(stream));
}

int launch_batch_advance(const BatchChain* chains, int nchains, uint32_t k, unsigned int* cursors, int ncursors,
                         void* stream)
{
    const int n = nchains > ncursors ? nchains : ncursors;
    batch_advance_kernel<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(chains, nchains, k,
                                                                                             cursors, ncursors);
    return (int)cudaGetLastError();
}

// Per-chain state hash over all tiles (out[chain] must be zeroed).  A block
// takes one slice of a tile's words, every gridDim.y-th run of 256: a word of a
// frozen region is a chain of 32 64-bit mixes in one lane, so what a lane takes
// one after the other sets the time, and a block per tile left it 10 to 60 words
// (12 chains in 120 tiles: 165 -> 25 us).
__global__ void batch_hash_kernel(const BatchChain* __restrict__ chains, const BatchTile* __restrict__ tiles,
                                  int ntiles, int buf, unsigned long long* out)
{
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const BatchTile tile = tiles[t];
        const BatchChain& ch = chains[tile.chain];
        const Geom& g = ch.g;
        const int64_t RW = g.row_words;
        const uint32_t* base = ch.rows[buf] + RW + (int64_t)tile.lo * RW;
        const int nw = (tile.hi - tile.lo) * (int)RW;
        uint64_t acc = 0;
        for (int w = blockIdx.y * blockDim.x + threadIdx.x; w < nw; w += gridDim.y * blockDim.x) {
            const uint32_t v = base[w];
            if (!v) continue;
            const int rr = w / (int)RW;
            const int rem = w - rr * (int)RW;
            const int pl = rem / g.K, k = rem - pl * g.K;
            acc += word_hash(v, g, tile.lo + rr, pl, k);
        }
        for (int o = 16; o; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
        if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out + tile.chain, (unsigned long long)acc);
    }
}

int launch_batch_hash(const BatchChain* chains, const BatchTile* tiles, int ntiles, int buf,
                      unsigned long long* out, void* stream)
{
    // 4,096 blocks or a little more, at most 64 slices a tile
    const int grid = ntiles < 1 ? 1 : ntiles < 4096 ? ntiles : 4096;
    const int slices = grid < 64 ? 64 : (4096 + grid - 1) / grid;
    batch_hash_kernel<<<dim3(grid, slices), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(chains, tiles, ntiles,
                                                                                            buf, out);
    return (int)cudaGetLastError();
}

// Copy every tile's rows from buffer `from` to the other buffer.
__global__ void batch_copy_kernel(const BatchChain* __restrict__ chains, const BatchTile* __restrict__ tiles,
                                  int ntiles, int from)
{
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const BatchTile tile = tiles[t];
        const BatchChain& ch = chains[tile.chain];
        const int64_t RW = ch.g.row_words;
        const uint4* s4 = reinterpret_cast<const uint4*>(ch.rows[from] + RW + (int64_t)tile.lo * RW);
        uint4* d4 = reinterpret_cast<uint4*>(ch.rows[from ^ 1] + RW + (int64_t)tile.lo * RW);
        const int64_t n4 = (int64_t)(tile.hi - tile.lo) * RW / 4;
        for (int64_t i = threadIdx.x; i < n4; i += blockDim.x) d4[i] = s4[i];
    }
}

int launch_batch_copy(const BatchChain* chains, const BatchTile* tiles, int ntiles, int from, void* stream)
{
    const int grid = ntiles < 4096 ? ntiles : 4096;
    batch_copy_kernel<<<grid > 0 ? grid : 1, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(chains, tiles, ntiles,
                                                                                             from);
    return (int)cudaGetLastError();
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_batch(unsigned long long* out, bool clear)
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
