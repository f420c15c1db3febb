// CUDA kernels for colour-class-parallel heat-bath Glauber dynamics on
// bit-packed tilings (Keating & Sridhar, "Random Tilings with the GPU",
// Sec. 1.1.3 cluster rotations, Sec. 1.2.1 lozenges, Sec. 1.2.4 six-vertex,
// Sec. 2.2 Rotate / Update kernels).  Written for sm_103a.
//
// Every thread updates one 128-site group (four 32-bit words, one Philox
// output) of one colour class in one row: the flippable mask is built with
// bitwise logic over the four neighbouring edge words, the heat-bath draw
// compares a bit-plane transposed Philox stream against the threshold MSB
// first and stops as soon as every flippable site is decided, and the flip is
// applied as an XOR of the four (or six) edge words.  Because each edge has a
// single owner inside a pass, there are no write conflicts except for the one
// word that straddles two groups when a plane is shifted by one site; that
// word is updated with atomicXor.  The paper's second kernel (UpdateBlack /
// UpdateWhite, which rebuilt the redundant 4-bit states of the other colour)
// has no counterpart: the packed state stores every edge once.
#include "tl_device.cuh"

#include <cstdint>
#include <mutex>
#include <type_traits>

namespace tl {

// ---------------------------------------------------------------------------
// One launch per pass, state in global memory (L2-resident for mid sizes).
// Thread = (site row, group).  grange[y] = [first, last+1) groups of row y
// that hold sites of the domain.
// ---------------------------------------------------------------------------
template <int LAT, int TK>
__global__ void __launch_bounds__(256) pass_global_kernel(uint32_t* __restrict__ rows0, Geom g,
                                                          uint32_t pass, uint32_t slot, uint32_t sweep,
                                                          DevRng rng, ThrView th,
                                                          const int2* __restrict__ grange,
                                                          unsigned long long* __restrict__ flips)
{
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int nrow = (LAT == LAT_SIXV) ? ((g.H + 1) >> 1) : g.H;
    const int rix = tid / g.Kg;
    const int m = tid - rix * g.Kg;
    if (rix >= nrow) return;
    int y, rr;
    if (LAT == LAT_SIXV) {
        y = 2 * rix + sixv_py(pass);
        if (y < 1 || y > g.N - 1) return;
        rr = rix;
    } else {
        y = rix;
        rr = y;
    }
#ifdef TL_DEBUG
    if (!TL_IN(y, g.H, 401)) return;
#endif
    const int2 gr = grange[y];
    if (m < gr.x || m >= gr.y) return;
#ifdef TL_DEBUG
    if (!TL_IN(4 * m + 3, g.K, 402)) return;
#endif
    const uint32_t grp = (uint32_t)(rr * g.Kg + m);
    uint32_t* row = rows0 + (int64_t)y * g.row_words;
    const RndPhilox rnd{grp, sweep, slot, rng};
    uint32_t nfl = 0;
    group_update<LAT, TK>(row, g.row_words, g, y, m, pass, rnd, th, nullptr, nullptr, flips ? &nfl : nullptr);
    if (nfl) atomicAdd(flips, (unsigned long long)nfl);
}

static inline cudaStream_t S(void* s) { return reinterpret_cast<cudaStream_t>(s); }

int launch_pass_global(const Geom& g, uint32_t* rows, uint32_t pass, uint32_t slot, uint32_t sweep,
                       const DevRng& rng, const ThrView& th, const int2* grange, unsigned long long* flips,
                       void* stream)
{
    const int nrow = (g.lattice == LAT_SIXV) ? ((g.H + 1) >> 1) : g.H;
    const int64_t threads = (int64_t)nrow * g.Kg;
    const int blocks = (int)((threads + 255) / 256);
    uint32_t* rows0 = rows + g.row_words;
    if (g.lattice == LAT_DOMINO) {
        if (th.kind == THR_SITE)
            pass_global_kernel<LAT_DOMINO, THR_SITE><<<blocks, 256, 0, S(stream)>>>(rows0, g, pass, slot, sweep, rng, th, grange, flips);
        else
            pass_global_kernel<LAT_DOMINO, THR_SCALAR><<<blocks, 256, 0, S(stream)>>>(rows0, g, pass, slot, sweep, rng, th, grange, flips);
    } else if (g.lattice == LAT_LOZENGE) {
        if (th.kind == THR_SITE)
            pass_global_kernel<LAT_LOZENGE, THR_SITE><<<blocks, 256, 0, S(stream)>>>(rows0, g, pass, slot, sweep, rng, th, grange, flips);
        else
            pass_global_kernel<LAT_LOZENGE, THR_SCALAR><<<blocks, 256, 0, S(stream)>>>(rows0, g, pass, slot, sweep, rng, th, grange, flips);
    } else {
        pass_global_kernel<LAT_SIXV, THR_TABLE><<<blocks, 256, 0, S(stream)>>>(rows0, g, pass, slot, sweep, rng, th, grange, flips);
    }
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Layout conversion.  Canonical: uint8 [ntype][H][W].
// ---------------------------------------------------------------------------
// A thread per word, for planes of one group a row (at most 128 columns each): the
// rows are too short for a warp.
__global__ void pack_narrow_kernel(const uint8_t* __restrict__ canon, uint32_t* __restrict__ rows, Geom g)
{
    const uint32_t n = (uint32_t)g.H * (uint32_t)g.row_words;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t y = i / (uint32_t)g.row_words, rem = i - y * (uint32_t)g.row_words;
        const int pl = (int)rem / g.K, k = (int)rem - pl * g.K, type = pl / g.npar, res = pl - type * g.npar;
        const uint8_t* src = canon + ((size_t)type * g.H + y) * g.W;
        uint32_t w = 0;
        for (int b = 0; b < 32; ++b) {
            const int x = g.npar * (32 * k + b) + res;
            if (x < g.W && src[x]) w |= 1u << b;
        }
        rows[g.row_words + i] = w;
    }
}

// A warp per 32 words of a (row, plane): lane l looks at the byte of bit l of a
// word, and a ballot is the word.  (Indices fit 32 bits: at most 65,536 rows of
// 9 planes of 32 such runs.)
// us: square 2048 18 with a thread a word, 9.4 with a warp a row, 10 so; 60000 x 4
// 4.0, 52, 3.4; 12000 x 60 5.9, 13, 4.1.
__global__ void pack_kernel(const uint8_t* __restrict__ canon, uint32_t* __restrict__ rows, Geom g)
{
    const int lane = threadIdx.x & 31;
    const uint32_t runs = (uint32_t)(g.K + 31) >> 5, n = (uint32_t)g.H * (uint32_t)g.P * runs,
                   step = gridDim.x * (blockDim.x >> 5);
    for (uint32_t u = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < n; u += step) {
        const uint32_t r = runs == 1u ? u : u / runs, y = r / (uint32_t)g.P;
        const int pl = (int)(r - y * (uint32_t)g.P), k0 = 32 * (int)(u - r * runs);
        const int type = pl / g.npar, res = pl - type * g.npar;
        const uint8_t* src = canon + ((size_t)type * g.H + y) * g.W;
        uint32_t* dst = rows + g.row_words + (int64_t)y * g.row_words + (int64_t)pl * g.K;
        const int nk = g.K - k0 < 32 ? g.K - k0 : 32;   // a multiple of 4
        uint32_t keep = 0;
        auto words = [&](int k, auto cnt) {
            constexpr int N = decltype(cnt)::value;
            uint32_t w[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int x = g.npar * (32 * (k0 + k + j) + lane) + res;
                w[j] = x < g.W ? src[x] : 0u;
            }
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const uint32_t v = __ballot_sync(0xFFFFFFFFu, w[j] != 0u);
                if (lane == k + j) keep = v;
            }
        };
        // the words that hold columns of the domain's box
        const int nw = (g.W + 32 * g.npar - 1) / (32 * g.npar) - k0, nv = nk < nw ? nk : nw;
        int k = 0;
        for (; k + 8 <= nv; k += 8) words(k, std::integral_constant<int, 8>{});
        for (; k < nv; k += 2) words(k, std::integral_constant<int, 2>{});
        if (lane < nk) dst[k0 + lane] = keep;
    }
}

// Bits j0 .. j0 + 31 of a plane row of K words (0 outside it).
TL_DEV uint32_t plane_bits(const uint32_t* p, int K, int j0)
{
    const int k = j0 >> 5;
    const uint32_t a = k >= 0 && k < K ? p[k] : 0u, b = k + 1 >= 0 && k + 1 < K ? p[k + 1] : 0u;
    return __funnelshift_r(a, b, j0 & 31);
}
// Bits [lo, hi] of 16, clipped to them.
TL_DEV uint32_t cell_span(int lo, int hi)
{
    lo = lo > 0 ? lo : 0;
    hi = hi < 15 ? hi : 15;
    return hi < lo ? 0u : (2u << hi) - (1u << lo);
}
// Bit i of the low 16 to position 2 i; of the low 8 to position 3 i.
TL_DEV uint32_t spread2(uint32_t x)
{
    x &= 0xFFFFu;
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}
// Edges x0 .. x0 + 16 (at least) of a row from its planes of even and odd x.
TL_DEV uint32_t bits2(const uint32_t* p, int K, int x0)
{
    const int j0 = x0 >> 1;
    return (spread2(plane_bits(p, K, j0)) | spread2(plane_bits(p + K, K, j0)) << 1) >> (x0 & 1);
}
TL_DEV uint32_t spread3(uint32_t x)
{
    x &= 0xFFu;
    x = (x | (x << 8)) & 0x0000F00Fu;
    x = (x | (x << 4)) & 0x000C30C3u;
    return (x | (x << 2)) & 0x00249249u;
}

// 16 bytes a thread: the bits of 16 neighbouring edges of a canonical row
// interleaved from the row's planes, four bits at a time spread into bytes by
// a product, and one aligned 16-byte store (the row's ragged ends by bytes).
// A row's units at its own alignment (at most `units`) are consecutive threads,
// whatever the shape: with a warp a row, few wide rows leave the chip idle and
// narrow ones the lanes.
// us: square 2048 36 with a thread a byte, 6.0 with a warp a row, 5.9 so; 60000 x 4
// 5.7, 39, 1.9; 200 x 20000 35, 15, 7.9; 2 x 30000 2.9, 20, 3.1.
//
// CHECK: dominoes, the units of horizontal edges also look at the other edges of
// their 16 cells: exactly one domino on every cell of the diamond of order n and
// none elsewhere, or the status word is raised (domino shuffling's steps look at
// edges only and would not notice; a launch of its own took 4 us, a check of every
// block the steps read 1 to 3% of a sample).
template <bool CHECK>
__global__ void unpack_kernel(const uint32_t* __restrict__ rows, uint8_t* __restrict__ canon, Geom g, int order, int* status)
{
    const uint32_t units = (uint32_t)(g.W + 30) >> 4, n = (uint32_t)(g.ntype * g.H) * units;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const uint32_t r = u / units;
        const int type = (int)(r / (uint32_t)g.H), y = (int)(r - (uint32_t)type * (uint32_t)g.H);
        const uint32_t* p = rows + g.row_words + (int64_t)y * g.row_words + (int64_t)type * g.npar * g.K;
        uint8_t* o = canon + (size_t)r * g.W;
        const int lead = (int)(reinterpret_cast<uintptr_t>(o) & 15u);
        const int x0 = 16 * (int)(u - r * units) - lead;   // may be negative: those bits are not stored
        if (x0 >= g.W) continue;
        uint32_t v;
        if (CHECK || g.npar == 2) {
            v = bits2(p, g.K, x0);
            if (CHECK && type == 0 && y < 2 * order) {
                const uint32_t b = bits2(p + g.row_words, g.K, x0), c = bits2(p + 2 * g.K, g.K, x0), d = c >> 1;
                const int w = y < order ? y + 1 : 2 * order - y;   // cells order - w .. order + w - 1 of the row
                const uint32_t in = cell_span(order - w - x0, order + w - 1 - x0);
                const uint32_t one = (v ^ b ^ c ^ d) & ~((v & b) | (c & d)), any = v | b | c | d;
                if (((one ^ in) | (any & ~in)) & 0xFFFFu) atomicCAS(status, 0, 2);
            }
        } else {
            const int j0 = (x0 + 18) / 3 - 6;   // floor, x0 > -16
            v = (spread3(plane_bits(p, g.K, j0)) | spread3(plane_bits(p + g.K, g.K, j0)) << 1 |
                 spread3(plane_bits(p + 2 * g.K, g.K, j0)) << 2) >>
                (x0 - 3 * j0);
        }
        const uint32_t b0 = ((v & 15u) * 0x00204081u) & 0x01010101u, b1 = (((v >> 4) & 15u) * 0x00204081u) & 0x01010101u,
                       b2 = (((v >> 8) & 15u) * 0x00204081u) & 0x01010101u,
                       b3 = (((v >> 12) & 15u) * 0x00204081u) & 0x01010101u;
        if (x0 >= 0 && x0 + 16 <= g.W) {
            *reinterpret_cast<uint4*>(o + x0) = make_uint4(b0, b1, b2, b3);
        } else {
            for (int t = 0; t < 16; ++t)
                if (x0 + t >= 0 && x0 + t < g.W) o[x0 + t] = (uint8_t)((v >> t) & 1u);
        }
    }
}

static int grid_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 32) b = 152 * 32;
    if (b < 1) b = 1;
    return (int)b;
}

int launch_pack(const Geom& g, const uint8_t* canon_dev, uint32_t* rows, void* stream)
{
    cudaError_t e = cudaMemsetAsync(rows, 0, (size_t)g.total_words * 4, S(stream));
    if (e != cudaSuccess) return (int)e;
    if (g.K == 4) pack_narrow_kernel<<<grid_for((int64_t)g.H * g.row_words, 256), 256, 0, S(stream)>>>(canon_dev, rows, g);
    else pack_kernel<<<grid_for((int64_t)g.H * g.P * ((g.K + 31) / 32) * 32, 256), 256, 0, S(stream)>>>(canon_dev, rows, g);
    return (int)cudaGetLastError();
}

int launch_unpack(const Geom& g, const uint32_t* rows, uint8_t* canon_dev, void* stream)
{
    unpack_kernel<false><<<grid_for((int64_t)g.ntype * g.H * ((g.W + 30) / 16), 256), 256, 0, S(stream)>>>(rows, canon_dev, g, 0,
                                                                                                          nullptr);
    return (int)cudaGetLastError();
}

int launch_unpack_diamond(const Geom& g, const uint32_t* rows, uint8_t* canon_dev, int n, int* status, void* stream)
{
    unpack_kernel<true><<<grid_for((int64_t)g.ntype * g.H * ((g.W + 30) / 16), 256), 256, 0, S(stream)>>>(rows, canon_dev, g, n,
                                                                                                         status);
    return (int)cudaGetLastError();
}

// Per-site thresholds [H][W] -> bit planes [H][npar][32][K]; plane k holds
// bit (31-k) of t for each site of the (row, residue) plane row.
__global__ void threshold_planes_kernel(const uint32_t* __restrict__ t, uint32_t* __restrict__ planes, Geom g)
{
    const int64_t n = (int64_t)g.H * g.npar * g.K;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(i % g.K);
        const int64_t r = i / g.K;
        const int res = (int)(r % g.npar);
        const int y = (int)(r / g.npar);
        uint32_t tv[32];
        for (int b = 0; b < 32; ++b) {
            const int x = g.npar * (32 * k + b) + res;
            tv[b] = (x < g.W) ? t[(size_t)y * g.W + x] : 0u;
        }
        uint32_t* out = planes + ((size_t)(y * g.npar + res) * 32) * g.K + k;
        for (int pl = 0; pl < 32; ++pl) {
            uint32_t w = 0;
            for (int b = 0; b < 32; ++b) w |= ((tv[b] >> (31 - pl)) & 1u) << b;
            out[(size_t)pl * g.K] = w;
        }
    }
}

int launch_threshold_planes(const Geom& g, const uint32_t* t_site_dev, uint32_t* planes, void* stream)
{
    const int64_t n = (int64_t)g.H * g.npar * g.K;
    threshold_planes_kernel<<<grid_for(n, 128), 128, 0, S(stream)>>>(t_site_dev, planes, g);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Validation of a canonical state against its domain, on the device: every
// byte 0 or 1; dominoes: no edge outside the box, every face of the domain
// covered once and no other; lozenges: every triangle covered as the domain
// says; six-vertex: no bit off the lattice, the external edges those of the
// boundary, the ice rule at every vertex.  The first failure in the order of
// a row-major scan (kinds in this order) is kept as the smallest code
// (kind << 48 | position) by an atomic min; *first stays ~0 if the state is
// valid.  Kinds: 1 byte (position = byte index), 2 domino edge right of the
// box (y), 3 domino edge above the box (x), 4 domino face (y (W-1) + x),
// 5 lozenge triangles ((y+1)(W+1) + x+1), 6 six-vertex bit off the lattice
// (Y W + X), 7 six-vertex boundary (k), 8 six-vertex ice rule (Y W + X).
// ---------------------------------------------------------------------------
struct DevCanon {
    const uint8_t* s;
    int W, H;
    TL_DEV int at(int type, int x, int y) const
    {
        if (x < 0 || y < 0 || x >= W || y >= H) return 0;
        return s[((size_t)type * H + y) * W + x];
    }
};

TL_DEV void vfail(unsigned long long* first, int kind, uint64_t pos)
{
    atomicMin(first, ((unsigned long long)kind << 48) | (unsigned long long)pos);
}

// 16 bytes at a time where they are aligned, the ends of the buffer by bytes.
__global__ void validate_bytes_kernel(const uint8_t* __restrict__ s, size_t n, unsigned long long* first)
{
    const size_t lead = (16u - (reinterpret_cast<uintptr_t>(s) & 15u)) & 15u, head = lead < n ? lead : n;
    const size_t units = (n - head) >> 4, t0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const uint4* v = reinterpret_cast<const uint4*>(s + head);
    for (size_t i = t0; i < units; i += (size_t)gridDim.x * blockDim.x) {
        const uint4 w = v[i];
        if (((w.x | w.y | w.z | w.w) & 0xFEFEFEFEu) == 0u) continue;
        for (int b = 0; b < 16; ++b)
            if (s[head + 16 * i + b] > 1) vfail(first, 1, head + 16 * i + b);
    }
    const size_t tail = head + 16 * units;
    if (t0 < head && s[t0] > 1) vfail(first, 1, t0);
    if (t0 < n - tail && s[tail + t0] > 1) vfail(first, 1, tail + t0);
}

// The lattice checks: a warp per 256 columns of a row.
constexpr int kCheckCols = 256;
struct WarpSpan {
    uint32_t u, n, step;   // 32 bits: at most 65,537 rows of 257 spans
    uint32_t segs;
    int cols;
    TL_DEV WarpSpan(int rows, int cols_)
        : u(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), step(gridDim.x * (blockDim.x >> 5)), cols(cols_)
    {
        segs = (uint32_t)(cols + kCheckCols - 1) / kCheckCols;
        n = (uint32_t)rows * segs;
    }
    TL_DEV int row() const { return (int)(segs == 1u ? u : u / segs); }
    // this lane's first column and the end of the span
    TL_DEV void span(int row, int& x0, int& x1) const
    {
        const int c = (int)(u - (uint32_t)row * segs) * kCheckCols;
        x0 = c + (int)(threadIdx.x & 31);
        x1 = c + kCheckCols < cols ? c + kCheckCols : cols;
    }
};

// aux: face cover [(H-1)][(W-1)]
__global__ void validate_domino_kernel(const uint8_t* __restrict__ s, Geom g, const uint8_t* __restrict__ cover,
                                       unsigned long long* first)
{
    const DevCanon c{s, g.W, g.H};
    const int FW = g.W - 1;
    const uint8_t *hz = s, *vt = s + (size_t)g.H * g.W;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t0; i < g.H + g.W; i += nt) {
        if (i < g.H) {
            if (c.at(0, g.W - 1, (int)i)) vfail(first, 2, (uint64_t)i);
        } else if (c.at(1, (int)(i - g.H), g.H - 1)) {
            vfail(first, 3, (uint64_t)(i - g.H));
        }
    }
    for (WarpSpan w(g.H - 1, FW); w.u < w.n; w.u += w.step) {
        const int y = w.row();
        int x, x1;
        w.span(y, x, x1);
        const size_t o = (size_t)y * g.W;
        const uint8_t* cv = cover + (size_t)y * FW;
#pragma unroll 4
        for (; x < x1; x += 32) {
            const int k = hz[o + x] + hz[o + g.W + x] + vt[o + x] + vt[o + x + 1];
            if (k != cv[x]) vfail(first, 4, (uint64_t)y * FW + x);
        }
    }
}

// aux: triangle cover, up then down, [(H+1)][(W+1)] each
__global__ void validate_lozenge_kernel(const uint8_t* __restrict__ s, Geom g, const uint8_t* __restrict__ cover,
                                        unsigned long long* first)
{
    const DevCanon c{s, g.W, g.H};
    const int TW = g.W + 1, TH = g.H + 1;
    const int64_t nt = (int64_t)TW * TH;
    for (WarpSpan w(TH, TW); w.u < w.n; w.u += w.step) {
        const int r = w.row(), y = r - 1;
        int c0, c1;
        w.span(r, c0, c1);
        for (; c0 < c1; c0 += 32) {
            const int x = c0 - 1;
            const int64_t i = (int64_t)r * TW + c0;
            const int e3 = c.at(2, x, y);
            const int u = c.at(0, x, y) + c.at(1, x + 1, y) + e3;
            const int v = e3 + c.at(1, x, y) + c.at(0, x, y + 1);
            if (u != cover[i] || v != cover[nt + i]) vfail(first, 5, (uint64_t)i);
        }
    }
}

// aux: the boundary edges of the domain, [4][N]: for k = 1..N (index k - 1)
// type 0 at (0, k), type 0 at (N, k), type 1 at (k, 0), type 1 at (k, N)
__global__ void validate_sixv_kernel(const uint8_t* __restrict__ s, Geom g, const uint8_t* __restrict__ bnd,
                                     unsigned long long* first)
{
    const DevCanon c{s, g.W, g.H};
    const int N = g.N;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t0; i < N; i += nt) {
        const int k = (int)i + 1;
        if (c.at(0, 0, k) != bnd[k - 1] || c.at(0, N, k) != bnd[N + k - 1] || c.at(1, k, 0) != bnd[2 * N + k - 1] ||
            c.at(1, k, N) != bnd[3 * N + k - 1])
            vfail(first, 7, (uint64_t)k);
    }
    for (WarpSpan w(g.H, g.W); w.u < w.n; w.u += w.step) {
        const int Y = w.row();
        int X, x1;
        w.span(Y, X, x1);
        for (; X < x1; X += 32) {
            const int64_t i = (int64_t)Y * g.W + X;
            const int R = c.at(0, X, Y), U = c.at(1, X, Y);
            const bool hreal = Y >= 1 && Y <= N && X <= N;
            const bool vreal = X >= 1 && X <= N && Y <= N;
            if ((R && !hreal) || (U && !vreal)) vfail(first, 6, (uint64_t)i);
            if (Y < 1 || Y > N || X < 1 || X > N) continue;
            const int L = c.at(0, X - 1, Y), D = c.at(1, X, Y - 1);
            if (L + U != D + R) vfail(first, 8, (uint64_t)i);
        }
    }
}

int launch_validate(const Geom& g, const uint8_t* canon, const uint8_t* aux, unsigned long long* first, void* stream)
{
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(first, 0xFF, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return (int)e;
    const size_t n = (size_t)g.ntype * g.W * g.H;
    validate_bytes_kernel<<<grid_for((int64_t)(n + 15) / 16, 256), 256, 0, st>>>(canon, n, first);
    if (g.lattice == LAT_DOMINO)
        validate_domino_kernel<<<grid_for((int64_t)g.H * ((g.W + kCheckCols) / kCheckCols) * 32, 256), 256, 0, st>>>(canon, g, aux, first);
    else if (g.lattice == LAT_LOZENGE)
        validate_lozenge_kernel<<<grid_for((int64_t)(g.H + 1) * ((g.W + kCheckCols) / kCheckCols) * 32, 256), 256, 0, st>>>(canon, g, aux, first);
    else
        validate_sixv_kernel<<<grid_for((int64_t)g.H * ((g.W + kCheckCols) / kCheckCols) * 32, 256), 256, 0, st>>>(canon, g, aux, first);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Observables.
// ---------------------------------------------------------------------------
__global__ void hash_kernel(const uint32_t* __restrict__ rows0, Geom g, unsigned long long* out)
{
    const int64_t n = (int64_t)g.H * g.row_words;
    uint64_t acc = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t w = rows0[i];
        if (!w) continue;
        const int y = (int)(i / g.row_words);
        const int rem = (int)(i - (int64_t)y * g.row_words);
        const int pl = rem / g.K, k = rem - pl * g.K;
        acc += word_hash(w, g, y, pl, k);
    }
    for (int off = 16; off; off >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, off);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, (unsigned long long)acc);
}

// The same in one block, writing the result itself: one launch instead of a
// clear and a launch, where a thread takes one word.  A word is a chain of up
// to 32 mixes, and one SM has room for 32 warps of them: us a hash in one block
// / in two launches, Aztec diamonds 8 3.6 / 5.1, 24 5.2 / 5.8, 32 (1,040 words)
// 6.2 / 6.2, 40 7.2 / 6.3, 127 20.7 / 8.3; domain-wall squares (denser) 30 5.6 /
// 6.3, 40 (672 words) 6.3 / 6.4, 50 7.9 / 6.8, 180 20.8 / 8.2; hexagons 10 4.3 /
// 5.0, 20 6.3 / 6.1, 40 11.5 / 6.4.
static bool small_hash(const Geom& g)
{
    return (int64_t)g.H * g.row_words <= (g.lattice == LAT_SIXV ? 704 : 1040);
}
__global__ void __launch_bounds__(1024) hash_small_kernel(const uint32_t* __restrict__ rows0, Geom g,
                                                          unsigned long long* out)
{
    __shared__ unsigned long long part[32];
    const int n = g.H * (int)g.row_words, RW = (int)g.row_words;
    uint64_t acc = 0;
    for (int i = threadIdx.x; i < n; i += 1024) {
        const uint32_t w = rows0[i];
        if (!w) continue;
        const int y = i / RW, rem = i - y * RW, pl = rem / g.K;
        acc += word_hash(w, g, y, pl, rem - pl * g.K);
    }
    for (int off = 16; off; off >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < 32; ++w) t += part[w];
        *out = t;
    }
}

int launch_hash(const Geom& g, const uint32_t* rows, unsigned long long* out, void* stream)
{
    if (small_hash(g)) {
        hash_small_kernel<<<1, 1024, 0, S(stream)>>>(rows + g.row_words, g, out);
        return (int)cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), S(stream));
    if (e != cudaSuccess) return (int)e;
    const int64_t n = (int64_t)g.H * g.row_words;
    hash_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(rows + g.row_words, g, out);
    return (int)cudaGetLastError();
}

// Edge-occupancy counters, bit-sliced in the packed layout (word_count_sliced).
__global__ void density_acc_kernel(const uint32_t* __restrict__ rows0, Geom g, uint32_t* __restrict__ cplanes)
{
    const int64_t n = (int64_t)g.H * g.row_words;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t w = rows0[i];
        if (w) word_count_sliced(w, i, n, cplanes);
    }
}

int launch_density_accumulate(const Geom& g, const uint32_t* rows, uint32_t* cplanes, void* stream)
{
    const int64_t n = (int64_t)g.H * g.row_words;
    density_acc_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(rows + g.row_words, g, cplanes);
    return (int)cudaGetLastError();
}

// Canonical counters counts[type][y][x] from the bit-sliced planes; only the
// `nbits` low planes can be non-zero (samples < 2^nbits).
__global__ void density_decode_kernel(const uint32_t* __restrict__ cplanes, Geom g, int nbits,
                                      uint32_t* __restrict__ counts)
{
    const int64_t n = (int64_t)g.ntype * g.H * g.W, plane = (int64_t)g.H * g.row_words;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % g.W);
        const int64_t r = i / g.W;
        const int y = (int)(r % g.H), type = (int)(r / g.H);
        const int res = x % g.npar, j = x / g.npar;
        const int64_t w = (int64_t)y * g.row_words + (int64_t)(type * g.npar + res) * g.K + (j >> 5);
        uint32_t v = 0;
        for (int b = 0; b < nbits; ++b) v |= ((cplanes[(int64_t)b * plane + w] >> (j & 31)) & 1u) << b;
        counts[i] = v;
    }
}

int launch_density_decode(const Geom& g, const uint32_t* cplanes, uint64_t samples, uint32_t* counts, void* stream)
{
    int nbits = 0;
    while (nbits < 32 && (samples >> nbits)) ++nbits;
    const int64_t n = (int64_t)g.ntype * g.H * g.W;
    density_decode_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(cplanes, g, nbits, counts);
    return (int)cudaGetLastError();
}

__global__ void density_read_kernel(const uint32_t* __restrict__ counts, uint64_t n, double inv,
                                    double* __restrict__ out)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = (double)counts[i] * inv;
}

int launch_density_read(const uint32_t* counts, uint64_t n, uint64_t samples, double* out, void* stream)
{
    const double inv = samples ? 1.0 / (double)samples : 0.0;
    density_read_kernel<<<grid_for((int64_t)n, 256), 256, 0, S(stream)>>>(counts, n, inv, out);
    return (int)cudaGetLastError();
}

// Domino type densities per face from the bit-sliced edge counters.  Face (x,y)
// of colour c = (x+y) mod 2 is covered by a domino crossing exactly one of its
// edges: right Vt(x+1,y) or left Vt(x,y) (horizontal), top Hz(x,y+1) or bottom
// Hz(x,y) (vertical).  Horizontal: north iff the left square has colour kappa,
// so the face's north density is that of its right edge if c == kappa, else of
// its left edge, and the south density the other one's.  Vertical: west iff the
// bottom square has colour != kappa.
//
// A block takes a run of face rows: it decodes the counters of a row of Hz and
// of Vt into shared memory (nbits planes of 32 edges a thread, its lanes
// starting at different edges so that the stores hit all banks) and writes the
// four densities.  count / samples comes from a table in shared memory (count
// <= samples): the same products, without an FP64 conversion and product for
// every value (FP64 is far below the write bandwidth here).  Aztec 2048 with
// 31 samples: 634 us before, decoding the counters to memory first.
constexpr int kNsewTable = 2048;
TL_DEV void decode_row(const uint32_t* __restrict__ cplanes, const Geom& g, int type, int y, int nbits, uint32_t* out,
                       int tid, int nt)
{
    const int64_t plane = (int64_t)g.H * g.row_words, base = (int64_t)y * g.row_words + (int64_t)type * 2 * g.K;
    for (int w = tid; w < 2 * g.K; w += nt) {
        const int res = w >= g.K, k = w - (res ? g.K : 0);
        for (int b0 = 0; b0 < nbits || b0 == 0; b0 += 8) {
            uint32_t v[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) v[b] = b0 + b < nbits ? cplanes[(int64_t)(b0 + b) * plane + base + w] : 0u;
            for (int jj = 0; jj < 32; ++jj) {
                const int j = (jj + tid) & 31, x = 2 * (32 * k + j) + res;
                if (x >= g.W) continue;
                uint32_t c = 0;
#pragma unroll
                for (int b = 0; b < 8; ++b) c |= ((v[b] >> j) & 1u) << b;
                out[x] = b0 ? out[x] | c << b0 : c;
            }
        }
    }
}

__global__ void __launch_bounds__(256) nsew_kernel(const uint32_t* __restrict__ cplanes, Geom g, int nbits,
                                                   uint32_t samples, double inv, int kappa, double* __restrict__ out)
{
    extern __shared__ double s_val[];   // [kNsewTable], then three rows of counts
    const int FW = g.W - 1, FH = g.H - 1, tid = threadIdx.x;
    const int64_t n = (int64_t)FW * FH;
    uint32_t* bottom = reinterpret_cast<uint32_t*>(s_val + kNsewTable);
    uint32_t *top = bottom + g.W, *side = top + g.W;
    const bool table = samples < kNsewTable;
    if (table)
        for (uint32_t i = tid; i <= samples; i += 256) s_val[i] = (double)i * inv;
    auto val = [&](uint32_t c) { return table ? s_val[c] : (double)c * inv; };
    const int y0 = (int)((int64_t)FH * blockIdx.x / gridDim.x), y1 = (int)((int64_t)FH * (blockIdx.x + 1) / gridDim.x);
    if (y0 < y1) decode_row(cplanes, g, 0, y0, nbits, bottom, tid, 256);
    for (int y = y0; y < y1; ++y) {
        // Hz of the next row by the first half, Vt of this one by the second
        if (tid < 128) decode_row(cplanes, g, 0, y + 1, nbits, top, tid, 128);
        else decode_row(cplanes, g, 1, y, nbits, side, tid - 128, 128);
        __syncthreads();
        double* o = out + (int64_t)y * FW;
        for (int x = tid; x < FW; x += 256) {
            const bool ck = ((x + y) & 1) == kappa;   // this face has colour kappa
            const uint32_t l = side[x], r = side[x + 1], t = top[x], b = bottom[x];
            o[x] = val(ck ? r : l);
            o[n + x] = val(ck ? l : r);
            o[2 * n + x] = val(ck ? t : b);
            o[3 * n + x] = val(ck ? b : t);
        }
        __syncthreads();
        uint32_t* z = bottom;
        bottom = top;
        top = z;
    }
}

// Few wide rows, or many narrow ones: from canonical counters in memory.
__global__ void nsew_counts_kernel(const uint32_t* __restrict__ counts, Geom g, double inv, int kappa,
                                   double* __restrict__ out)
{
    const int FW = g.W - 1, FH = g.H - 1;
    const int64_t n = (int64_t)FW * FH;
    const uint32_t* hz = counts;
    const uint32_t* vt = counts + (size_t)g.H * g.W;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % FW), y = (int)(i / FW);
        const bool ck = ((x + y) & 1) == kappa;
        const uint32_t right = vt[(size_t)y * g.W + x + 1], left = vt[(size_t)y * g.W + x];
        const uint32_t top = hz[(size_t)(y + 1) * g.W + x], bottom = hz[(size_t)y * g.W + x];
        out[i] = (double)(ck ? right : left) * inv;
        out[n + i] = (double)(ck ? left : right) * inv;
        out[2 * n + i] = (double)(ck ? top : bottom) * inv;
        out[3 * n + i] = (double)(ck ? bottom : top) * inv;
    }
}

int launch_nsew(const Geom& g, const uint32_t* cplanes, uint32_t* counts, uint64_t samples, int kappa, int smem_optin,
                double* out, int* launches, void* stream)
{
    const double inv = samples ? 1.0 / (double)samples : 0.0;
    const size_t smem = sizeof(double) * kNsewTable + 3 * sizeof(uint32_t) * (size_t)g.W;
    // A block per row leaves the chip idle where a domain has few rows, and
    // spends 3 us a row however narrow it is where a block takes several.  us
    // fused / through memory: 16000 x 2 27 / 8, 8000 x 8 17 / 10, 2000 x 8 10 / 8,
    // 8000 x 31 17 / 17, 12000 x 60 21 / 33; 20 x 20000 68 / 23, 100 x 20000 100 /
    // 78, 200 x 20000 107 / 148, 30 x 900 9.8 / 8.5.
    const bool flat = g.H <= 32 && g.W > 1600, narrow = g.W < 160 && g.H > 880;
    if (!flat && !narrow && smem <= (size_t)smem_optin) {
        int nbits = 0;
        while (nbits < 32 && (samples >> nbits)) ++nbits;
        cudaError_t e = cudaFuncSetAttribute(nsew_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return (int)e;
        const int per_sm = smem <= 36 * 1024 ? 6 : (smem <= 72 * 1024 ? 3 : 1);
        const int grid = g.H - 1 < 152 * per_sm ? g.H - 1 : 152 * per_sm;
        nsew_kernel<<<grid > 0 ? grid : 1, 256, smem, S(stream)>>>(
            cplanes, g, nbits, samples < 0xFFFFFFFFull ? (uint32_t)samples : 0xFFFFFFFFu, inv, kappa, out);
        *launches = 1;
        return (int)cudaGetLastError();
    }
    const int e = launch_density_decode(g, cplanes, samples, counts, stream);
    if (e) return e;
    const int64_t n = (int64_t)(g.W - 1) * (g.H - 1);
    nsew_counts_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(counts, g, inv, kappa, out);
    *launches = 2;
    return (int)cudaGetLastError();
}

// Height function: (1) prefix sums of horizontal steps along each segment
// of a row, (2) one block links every segment to its parent through a
// vertical step and adds the offsets up along the parents, (3) offsets are added.
template <int NPAR>
TL_DEV uint32_t bit_at(const uint32_t* rows0, const Geom& g, int type, int x, int y)
{
    if (x < 0 || y < 0 || x >= g.W || y >= g.H) return 0u;
    const int j = x / NPAR, res = x - j * NPAR;
    const uint32_t w = rows0[(int64_t)y * g.row_words + (int64_t)(type * NPAR + res) * g.K + (j >> 5)];
    return (w >> (j & 31)) & 1u;
}

// Step from grid point (x,y) to (x+1,y) / from (x,y-1) to (x,y).
template <int LAT>
TL_DEV int hstep(const uint32_t* rows0, const Geom& g, int x, int y)
{
    if (LAT == LAT_DOMINO) {
        const int s = ((x + y) & 1) ? -1 : 1;
        return bit_at<2>(rows0, g, 0, x, y) ? -3 * s : s;
    }
    if (LAT == LAT_LOZENGE) return -(int)bit_at<3>(rows0, g, 0, x, y);
    return bit_at<2>(rows0, g, 1, x + 1, y) ? 1 : -1;   // faces: cross Vt(x+1, y)
}
template <int LAT>
TL_DEV int vstep(const uint32_t* rows0, const Geom& g, int x, int y)
{
    if (LAT == LAT_DOMINO) {
        const int s = ((x - 1 + y - 1) & 1) ? -1 : 1;
        return bit_at<2>(rows0, g, 1, x, y - 1) ? -3 * s : s;
    }
    if (LAT == LAT_LOZENGE) return -(int)bit_at<3>(rows0, g, 1, x, y - 1);
    return bit_at<2>(rows0, g, 0, x, y) ? 1 : -1;       // faces: cross Hz(x, y)
}

// Height segments: seg[6 s .. 6 s + 5] = (y, lo, hi, parent, xs, dir): a
// maximal run [lo, hi] of row y joined by domain steps, the segment it is
// linked to (-1 for the first, which holds the reference vertex) and the
// column xs of the linking vertical step, dir = +1 if this segment lies one
// row above its parent and -1 if below.  Parents precede children.
__global__ void height_fill_kernel(int32_t* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = INT32_MIN;
}

// Heights of vertices [a, b) of row y (a warp, 32 at a time), from `run` at a;
// the row's segment ends at hi.
template <int LAT>
TL_DEV void scan_steps(const uint32_t* rows0, const Geom& g, int y, int a, int b, int hi, int run, int32_t* o)
{
    const int lane = threadIdx.x & 31;
    for (int x0 = a; x0 < b; x0 += 32) {
        const int x = x0 + lane;
        const int st = x < hi && x < b ? hstep<LAT>(rows0, g, x, y) : 0;
        int inc = st;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += v;
        }
        if (x < b) o[x] = run + inc - st;
        run += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
}

// Heights along each segment relative to its left end: each of the block's
// warps takes an eighth of it, sums its steps, and then scans them 32 at a
// time from the sum of the warps before it.
template <int LAT>
__global__ void __launch_bounds__(256) height_seg_kernel(const uint32_t* __restrict__ rows0, Geom g,
                                                         const int* __restrict__ seg, int hw,
                                                         int32_t* __restrict__ out)
{
    const int* sg = seg + 6 * (size_t)blockIdx.x;
    const int y = sg[0], lo = sg[1], hi = sg[2];
#ifdef TL_DEBUG
    // a segment of row y spans vertices lo .. hi of a row of hw heights
    if (!(TL_IN(y, g.H, 403) && TL_IN(lo, hw, 404) && TL_IN(hi, hw, 404))) return;
#endif
    int32_t* o = out + (size_t)y * hw;
    __shared__ int part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = ((hi - lo + 32) / 32 + 7) / 8 * 32;   // vertices a warp
    const int a = lo + warp * per, b = a + per < hi + 1 ? a + per : hi + 1;
    int sum = 0;
    for (int x = a + lane; x < b; x += 32)
        if (x < hi) sum += hstep<LAT>(rows0, g, x, y);   // step x -> x+1
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) part[warp] = sum;
    __syncthreads();
    int run = 0;   // height of the warp's first vertex relative to lo
    for (int w = 0; w < warp; ++w) run += part[w];
    scan_steps<LAT>(rows0, g, y, a, b, hi, run, o);
}

// Offsets of the segments, 1,024 at a time: the differences to the parents,
// then every segment follows its parents within the batch, doubling its reach
// each round (parents come first, so those of earlier batches are done).
template <int LAT>
TL_DEV void link_segments(const uint32_t* rows0, const Geom& g, const int* seg, int nseg, int hw, const int32_t* rel,
                          int* base, int* val, int* up)
{
    const int t = threadIdx.x;
    for (int c0 = 0; c0 < nseg; c0 += 1024) {
        const int s = c0 + t;
        int v = 0, q = -1;
        if (s < nseg) {
            const int* sg = seg + 6 * (size_t)s;
            const int y = sg[0], p = sg[3], xs = sg[4], dir = sg[5];
            if (p >= 0) {
                const int py = seg[6 * (size_t)p];
                const int step = dir > 0 ? vstep<LAT>(rows0, g, xs, y) : -vstep<LAT>(rows0, g, xs, y + 1);
                v = rel[(size_t)py * hw + xs] + step - rel[(size_t)y * hw + xs];
                if (p < c0) v += base[p];
                else q = p - c0;
            }
        }
        val[t] = v;
        up[t] = q;
        while (__syncthreads_or(q >= 0)) {
            const int v2 = q >= 0 ? val[q] : 0, q2 = q >= 0 ? up[q] : -1;
            __syncthreads();
            v += v2;
            q = q2;
            val[t] = v;
            up[t] = q;
        }
        if (s < nseg) base[s] = v;
        __syncthreads();
    }
}

template <int LAT>
__global__ void __launch_bounds__(1024) height_link_kernel(const uint32_t* __restrict__ rows0, Geom g,
                                                           const int* __restrict__ seg, int nseg, int hw,
                                                           const int32_t* __restrict__ rel, int* __restrict__ base)
{
    __shared__ int val[1024], up[1024];
    link_segments<LAT>(rows0, g, seg, nseg, hw, rel, base, val, up);
}

// All of it in one block, for grids so small that four launches take longer:
// its 32 warps take the segments in turn, 32 vertices at a time.
template <int LAT>
__global__ void __launch_bounds__(1024) height_small_kernel(const uint32_t* __restrict__ rows0, Geom g,
                                                            const int* __restrict__ seg, int nseg, int hw, int n,
                                                            int32_t* out, int* base)
{
    __shared__ int val[1024], up[1024];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < n; i += 1024) out[i] = INT32_MIN;
    __syncthreads();
    for (int s = warp; s < nseg; s += 32) {
        const int y = seg[6 * s], lo = seg[6 * s + 1], hi = seg[6 * s + 2];
        scan_steps<LAT>(rows0, g, y, lo, hi + 1, hi, 0, out + (size_t)y * hw);
    }
    __syncthreads();
    link_segments<LAT>(rows0, g, seg, nseg, hw, out, base, val, up);
    __syncthreads();
    for (int s = warp; s < nseg; s += 32) {
        const int y = seg[6 * s], lo = seg[6 * s + 1], hi = seg[6 * s + 2], b = base[s];
        for (int x = lo + lane; x <= hi; x += 32) out[(size_t)y * hw + x] += b;
    }
}

__global__ void __launch_bounds__(256) height_add_kernel(int32_t* __restrict__ out, const int* __restrict__ seg,
                                                         const int* __restrict__ base, int hw)
{
    const int* sg = seg + 6 * (size_t)blockIdx.x;
    const int y = sg[0], lo = sg[1], hi = sg[2];
    const int b = base[blockIdx.x];
    int32_t* o = out + (size_t)y * hw;
    for (int x = lo + threadIdx.x; x <= hi; x += 256) o[x] += b;
}

// One block or four launches.  us in one block / four launches: Aztec diamonds 32
// 8.3 / 17.6, 64 12.5 / 17.8, 100 (40,401 heights) 19.6 / 18.2, 127 28.0 / 18.6;
// domain-wall squares 100 12.7 / 17.5, 140 (19,881) 17.8 / 17.6, 180 23.7 / 17.5;
// squares of 11 columns 300 (301 segments) 15.3 / 18.5, 1000 36.7 / 18.5; flat ones
// 1000 x 4 (32 turns a segment) 12.5 / 17.5, 2000 x 4 20.7 / 19.7, 15000 x 1 119 / 37.
int height_launches(int nseg, int hw, int hh)
{
    const int64_t turns = (int64_t)((nseg + 31) / 32) * ((hw + 31) / 32);
    return nseg <= 0 || ((int64_t)hw * hh <= 20000 && nseg <= 320 && turns <= 32) ? 1 : 4;
}

int launch_height(const Geom& g, const uint32_t* rows, const int* seg, int nseg, int hw, int hh, int32_t* out,
                  int* base_scratch, void* stream)
{
    const uint32_t* rows0 = rows + g.row_words;
    const int64_t n = (int64_t)hw * hh;
    auto run = [&](auto lat) {
        constexpr int LAT = decltype(lat)::value;
        if (nseg > 0 && height_launches(nseg, hw, hh) == 1) {
            height_small_kernel<LAT><<<1, 1024, 0, S(stream)>>>(rows0, g, seg, nseg, hw, (int)n, out, base_scratch);
            return;
        }
        height_fill_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(out, n);
        if (nseg <= 0) return;
        height_seg_kernel<LAT><<<nseg, 256, 0, S(stream)>>>(rows0, g, seg, hw, out);
        height_link_kernel<LAT><<<1, 1024, 0, S(stream)>>>(rows0, g, seg, nseg, hw, out, base_scratch);
        height_add_kernel<<<nseg, 256, 0, S(stream)>>>(out, seg, base_scratch, hw);
    };
    if (g.lattice == LAT_DOMINO) run(std::integral_constant<int, LAT_DOMINO>{});
    else if (g.lattice == LAT_LOZENGE) run(std::integral_constant<int, LAT_LOZENGE>{});
    else run(std::integral_constant<int, LAT_SIXV>{});
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Generated log-normal weights and their heat-bath thresholds, on the device.
// Weight of item i (an edge or a vertex, by canonical index) = exp(sigma Z),
// Z standard normal by the Box-Muller transform of two 32-bit words of
// Philox4x32-10(key = seed, counter = (i lo, i hi, 0x6C6F676E, 0)).  The
// threshold arithmetic uses correctly rounded FP64 operations in the order of
// the host formulas (no fused multiply-add), so for equal weights it equals
// the host result bit for bit.
// ---------------------------------------------------------------------------
TL_DEV double lognormal_weight(uint64_t i, double sigma, uint32_t k0, uint32_t k1)
{
    const uint4 o = philox10((uint32_t)i, (uint32_t)(i >> 32), 0x6C6F676Eu, 0u, k0, k1);
    const double u1 = ((double)o.x + 1.0) * (1.0 / 4294967296.0);   // (0, 1]
    const double u2 = (double)o.y * (1.0 / 4294967296.0);           // [0, 1)
    const double z = sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
    return exp(sigma * z);
}

TL_DEV uint32_t prob_threshold(double p)
{
    const double t = floor(__dmul_rn(p, 4294967296.0));
    if (!(t > 0.0)) return 0u;
    if (t >= 4294967295.0) return 0xFFFFFFFFu;
    return (uint32_t)t;
}

// Dominoes: edge weights on the canonical [2][H][W] layout; t at every vertex
// from up = wE * wW, down = wN * wS, P = up / (up + down) (1.0 off the box).
__global__ void lognormal_domino_kernel(int W, int H, double sigma, uint32_t k0, uint32_t k1, uint32_t* t)
{
    const int64_t n = (int64_t)W * H;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(v % W), y = (int)(v / W);
        auto wt = [&](int type, int xx, int yy) -> double {
            if (xx < 0 || yy < 0 || xx >= W || yy >= H) return 1.0;
            return lognormal_weight(((uint64_t)type * H + yy) * W + xx, sigma, k0, k1);
        };
        const double up = __dmul_rn(wt(0, x, y), wt(0, x - 1, y));
        const double down = __dmul_rn(wt(1, x, y), wt(1, x, y - 1));
        t[v] = prob_threshold(__ddiv_rn(up, __dadd_rn(up, down)));
    }
}

// Lozenges: volume weight q_v per vertex; P(add a cube) = q / (1 + q).
__global__ void lognormal_lozenge_kernel(int W, int H, double sigma, uint32_t k0, uint32_t k1, uint32_t* t)
{
    const int64_t n = (int64_t)W * H;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const double q = lognormal_weight((uint64_t)v, sigma, k0, k1);
        t[v] = prob_threshold(__ddiv_rn(q, __dadd_rn(1.0, q)));
    }
}

int launch_lognormal_thresholds(int lattice, int W, int H, double sigma, uint64_t seed, uint32_t* t, void* stream)
{
    const int64_t n = (int64_t)W * H;
    if (lattice == LAT_DOMINO)
        lognormal_domino_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(W, H, sigma, (uint32_t)seed,
                                                                       (uint32_t)(seed >> 32), t);
    else
        lognormal_lozenge_kernel<<<grid_for(n, 256), 256, 0, S(stream)>>>(W, H, sigma, (uint32_t)seed,
                                                                        (uint32_t)(seed >> 32), t);
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Height function without any allocation.  For callers that cannot allocate
// device memory at the time they need the heights (for example code running
// under a memory budget that forbids cudaMalloc, or a real-time loop that
// must not synchronise the device the way cudaMalloc / cudaFree can), the
// per-segment offsets that launch_height keeps in chain-owned memory live here
// in one file-scope device array instead.  The array holds kNoAllocMaxSegs
// ints (256 KiB): one per height segment, a maximal run of domain vertices in
// one row (one segment per row for the Aztec diamond, rectangles, hexagons and
// the domain-wall square; a row of a non-convex domain from a boundary path
// can hold several).  Domains with more segments are rejected.  Every GPU
// that loads the library keeps the array until the process exits.  All calls
// on a device share it: each call rewrites every entry it reads, so nothing
// needs clearing, but calls whose kernels overlap on the GPU (concurrent
// streams) race on it and must be serialised by the caller.
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxSegs = 65536;
static __device__ __align__(256) int g_noalloc_height_base[kNoAllocMaxSegs];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static int* g_noalloc_base_dev[kNoAllocMaxDevices];   // device address per device ordinal

int noalloc_height_max_segments() { return kNoAllocMaxSegs; }

// The device address of the scratch array must come from cudaGetSymbolAddress
// with the device current: in host code the symbol names a host-side stand-in.
// Looked up once per device, when a context is created on it (the lookup can
// load this module, which allocates), so the entry point itself never does.
int noalloc_prepare(int device)
{
    if (device < 0 || device >= kNoAllocMaxDevices) return (int)cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_base_dev[device]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_height_base);
        if (e != cudaSuccess) return (int)e;
        g_noalloc_base_dev[device] = static_cast<int*>(p);
    }
    return 0;
}

static int noalloc_scratch(int device, int** out)
{
    if (device < 0 || device >= kNoAllocMaxDevices) return (int)cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    *out = g_noalloc_base_dev[device];
    return *out ? 0 : (int)cudaErrorInitializationError;
}

int launch_height_noalloc(const Geom& g, const uint32_t* rows, const int* seg, int nseg, int hw, int hh,
                          int32_t* out, int device, void* stream)
{
    if (nseg > kNoAllocMaxSegs) return (int)cudaErrorInvalidValue;
    int* base = nullptr;
    const int e = noalloc_scratch(device, &base);
    if (e) return e;
    return launch_height(g, rows, seg, nseg, hw, hh, out, base, stream);
}

// This file's debug word (failures, then the id, index and bound of the
// first failed check); cudaErrorNotSupported in the normal build.
int dbg_fetch_kernels(unsigned long long* out, bool clear)
{
#ifdef TL_DEBUG
    return tl_dbg_fetch(out, clear);
#else
    (void)out;
    (void)clear;
    return (int)cudaErrorNotSupported;
#endif
}

#ifdef TL_DEBUG
// One check on an index out of its range (5 of 3, id 999) and none of the
// access it guards: the failure must be recorded, nothing else happens.
__global__ void dbg_selftest_kernel(int* out)
{
    int x = 0;
    if (TL_IN(threadIdx.x + 5, 3, 999)) x = 1;
    out[threadIdx.x] = x;
}
#endif

int dbg_selftest()
{
#ifdef TL_DEBUG
    int* d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(int));
    if (e == cudaSuccess) {
        dbg_selftest_kernel<<<1, 1>>>(d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d);
    return (int)e;
#else
    return (int)cudaErrorNotSupported;
#endif
}

}  // namespace tl
