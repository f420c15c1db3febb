// Launches of the word kernel (tl_words_kernel.cuh).
#include "tl_words_kernel.cuh"

#include <numeric>

namespace tl {

// ---- host side ----

const void* words_kernel_domino(int tk, int threads, int slots, bool fixed);
const void* words_kernel_lozenge(int tk, int threads, int slots, bool fixed);
const void* words_kernel_sixv(bool count, int threads, int slots, bool fixed);

static const void* pick(int lattice, int tk, int cpol, int threads, int slots, bool fixed)
{
    if (lattice == LAT_DOMINO) return words_kernel_domino(tk, threads, slots, fixed);
    if (lattice == LAT_LOZENGE) return words_kernel_lozenge(tk, threads, slots, fixed);
    return words_kernel_sixv(cpol >= 0, threads, slots, fixed);
}

// Threads of a launch with a hash after every sweep: up to 512, whatever the
// passes need, share the words, in a number of warps that does not divide the
// 32-word runs of a row (or the same warps would take the same planes, the full
// ones, in every row).  us a sweep with the plan's threads -> these: Aztec 40 6.4
// -> 4.7, 300 8.3 -> 5.9, hexagon 200 12.7 -> 8.5, domain-wall square 30 12.7 ->
// 5.0, 500 12.2 -> 7.0; Aztec 900 (128 words a row) 17 with 480 threads, 42 with 512.
static int hash_threads(const Geom& g, const ResidentPlan& plan)
{
    if (plan.slots != 1 || plan.threads >= 512) return plan.threads;
    const int runs = g.row_words % 32 ? 1 : (int)(g.row_words / 32);
    for (int w = 16; 32 * w > plan.threads && w > 12; --w)
        if (std::gcd(w, runs) == 1) return 32 * w;
    return plan.threads;
}

size_t words_smem_bytes(const Geom& g, int local_rows) { return (size_t)local_rows * g.row_words * 4 + (size_t)(local_rows + 2) * 4; }

int words_prepare(const Geom& g, const ThrView& th, int threads, int slots, size_t smem_bytes, int* blocks_per_sm)
{
    *blocks_per_sm = 0;
    // one limit for all chains: a plan must not lower another chain's
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int least = 1 << 30;
    for (int fixed = 0; fixed < 2 && e == cudaSuccess; ++fixed) {
        const void* k = pick(g.lattice, th.kind, th.cpol, threads, slots, fixed != 0);
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
        int bps = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k, threads, smem_bytes);
        least = bps < least ? bps : least;
    }
    if (e == cudaSuccess) *blocks_per_sm = least;
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

int launch_words(const Geom& g, uint32_t* rows, const ResidentPlan& plan, uint32_t sweep0, uint32_t nsweeps,
                 const DevRng& rng, const ThrView& th, const int2* grange, unsigned int epoch, unsigned long long* ring,
                 uint32_t* counts, uint64_t burn, uint32_t stride, const uint8_t* colours, unsigned long long* flips,
                 void* stream)
{
    WordParams P;
    P.rows0 = rows + g.row_words;
    P.g = g;
    P.stripe_lo = plan.stripe_lo;
    P.halo = plan.halo;
    P.nblk = (plan.npre + 3) / 4;
    P.colours = colours;
    P.sweep0 = sweep0;
    P.nsweeps = nsweeps;
    P.rng = rng;
    P.scalar = th.scalar;
    P.kmax = th.kmax;
    P.planes = th.planes;
    P.cpol = th.cpol;
    P.grange = grange;
    P.xbuf = plan.xbuf;
    P.status = plan.status;
    P.loaded = plan.loaded;
    P.ring = ring;
    P.counts = counts;
    P.burn = burn;
    P.stride = stride;
    P.epoch = epoch;
    P.flips = flips;
    if (g.lattice == LAT_SIXV) {
        for (int k = 0; k < 32; ++k) {
            uint32_t coef;   // bit s: coefficient of product s
            if (th.cpol >= 0) {
                uint32_t b[5];
                for (int n = 0; n < 5; ++n) b[n] = (th.t5[n] >> (31 - k)) & 1u;
                coef = b[0] | (b[0] ^ b[1]) << 1 | (b[0] ^ b[2]) << 2 | (b[0] ^ b[1] ^ b[2] ^ b[3]) << 3 | (b[0] ^ b[4]) << 4;
            } else {
                // Moebius transform of the 16-entry truth table
                coef = th.tmask[k] & 0xFFFFu;
                coef ^= (coef & 0x5555u) << 1;
                coef ^= (coef & 0x3333u) << 2;
                coef ^= (coef & 0x0F0Fu) << 4;
                coef ^= (coef & 0x00FFu) << 8;
            }
            for (int s = 0; s < 16; ++s) P.anf.c[k][s] = 0u - ((coef >> s) & 1u);
        }
    }
    void* args[] = {&P};
    const bool fixed = !colours && plan.halo % g.passes == 0;
    const void* k = pick(g.lattice, th.kind, th.cpol, plan.threads, plan.slots, fixed);
    return (int)cudaLaunchCooperativeKernel(k, dim3(plan.ctas), dim3(ring ? hash_threads(g, plan) : plan.threads), args,
                                            plan.smem_bytes, reinterpret_cast<cudaStream_t>(stream));
}

}  // namespace tl
