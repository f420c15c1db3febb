// Host runtime of the C-ABI in include/tiling.h: domain builders, FP64
// heat-bath thresholds, chain state management and the launch planner.
#include "tiling.h"
#include "tl_internal.h"
#include "tl_thurston.h"

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <mutex>
#include <new>
#include <tuple>
#include <string>
#include <vector>

// NVTX ranges around the library's launches, graph blocks and exact
// samplers, named after the C-ABI call (visible in Nsight Systems / ncu
// with NVTX enabled; without a tool attached each costs a pointer check).
namespace {
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};
}  // namespace

using namespace tl;

#define TL_API extern "C" __attribute__((visibility("default")))

// ---------------------------------------------------------------------------
// Errors
// ---------------------------------------------------------------------------
static thread_local std::string g_err;

static int fail(int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

#define TL_TRY(expr)                   \
    do {                               \
        int rc_ = (expr);              \
        if (rc_ != TL_OK) return rc_;  \
    } while (0)

#define CUDA_TRY(expr)                                                                  \
    do {                                                                                \
        cudaError_t e_ = (cudaError_t)(expr);                                           \
        if (e_ != cudaSuccess)                                                          \
            return fail(TL_ECUDA, "%s failed: %s", #expr, cudaGetErrorString(e_));     \
    } while (0)

TL_API const char* tl_last_error(void) { return g_err.c_str(); }
TL_API const char* tl_version(void) { return "tiling-gb300 0.1 (sm_103a)"; }

// ---------------------------------------------------------------------------
// Context
// ---------------------------------------------------------------------------
// Domino shuffling of one order n, kept per context: the packed rows of the
// sample, and the stripes and exchange buffer of the resident kernel or, for
// orders whose rows do not fit on chip, the second buffer of the per-step one.
struct ShuffleCache {
    int n = 0;
    Geom g{};
    uint32_t *rows = nullptr, *alt = nullptr;
    uint8_t* canon = nullptr;   // staging of results read to host memory
    int* stripe = nullptr;
    unsigned long long* xbuf = nullptr;
    int* status = nullptr;
    std::vector<ShufflePlan> seg;   // empty: one launch per step
    size_t xbuf_words = 0;
    void release()
    {
        cudaFree(rows); cudaFree(alt); cudaFree(canon); cudaFree(stripe); cudaFree(xbuf); cudaFree(status);
        *this = ShuffleCache();
    }
};

struct tl_ctx {
    // one reference for the caller's handle and one per chain or batch on
    // the context: it is freed when the last of them goes, whatever the order
    std::atomic<int> refs{1};
    int device;
    int sms;
    int smem_optin;
    int l2_bytes;
    std::mutex shuffle_mu;   // one shuffling sample at a time per context
    ShuffleCache shuffle;
};

TL_API int tl_ctx_create_opts(int cuda_device, const tl_ctx_opts* opts, tl_ctx** out)
{
    if (opts && opts->max_sms < 0) return fail(TL_EINVAL, "tl_ctx_create_opts: max_sms < 0");
    const int rc = tl_ctx_create(cuda_device, out);
    if (rc != TL_OK || !opts) return rc;
    if (opts->max_sms > 0) (*out)->sms = std::min((*out)->sms, opts->max_sms);
    return TL_OK;
}

TL_API int tl_ctx_create(int cuda_device, tl_ctx** out)
{
    if (!out) return fail(TL_EINVAL, "tl_ctx_create: out is NULL");
    int n = 0;
    CUDA_TRY(cudaGetDeviceCount(&n));
    if (cuda_device < 0 || cuda_device >= n)
        return fail(TL_EINVAL, "tl_ctx_create: device %d of %d", cuda_device, n);
    CUDA_TRY(cudaSetDevice(cuda_device));
    tl_ctx* c = new (std::nothrow) tl_ctx();
    if (!c) return fail(TL_ENOMEM, "tl_ctx_create: host allocation");
    c->device = cuda_device;
    cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, cuda_device);
    cudaDeviceGetAttribute(&c->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, cuda_device);
    cudaDeviceGetAttribute(&c->l2_bytes, cudaDevAttrL2CacheSize, cuda_device);
    // the allocation-free height call's static scratch: its device address
    // is looked up here, once per device, so that call itself loads nothing
    const int e = noalloc_prepare(cuda_device);
    if (e) {
        delete c;
        return fail(TL_ECUDA, "tl_ctx_create: static scratch lookup: %s", cudaGetErrorString((cudaError_t)e));
    }
    *out = c;
    return TL_OK;
}

static void ctx_release(tl_ctx* c)
{
    if (!c || c->refs.fetch_sub(1) != 1) return;
    if (c->shuffle.n) {
        cudaSetDevice(c->device);
        cudaDeviceSynchronize();
        c->shuffle.release();
    }
    delete c;
}

TL_API void tl_ctx_destroy(tl_ctx* c) { ctx_release(c); }

// ---------------------------------------------------------------------------
// Domains
// ---------------------------------------------------------------------------
struct tl_domain {
    Geom g;
    std::vector<uint8_t> init;        // canonical starting configuration
    std::vector<uint8_t> cover;       // domino: faces [H-1][W-1]; lozenge: up/down [2][H][W]
    uint64_t sites = 0, edges = 0;
    std::vector<int2> grange;         // per site row: [first, last+1) active groups
    int hw = 0, hh = 0;
    std::vector<int> hseg;            // height segments, 6 ints each (see plan_heights)
    int nseg = 0;
    int kappa = 0;
};

static Geom make_geom(int lattice, int W, int H, int N)
{
    Geom g{};
    g.lattice = lattice;
    g.W = W;
    g.H = H;
    g.N = N;
    g.npar = (lattice == LAT_LOZENGE) ? 3 : 2;
    g.ntype = (lattice == LAT_LOZENGE) ? 3 : 2;
    g.P = g.npar * g.ntype;
    const int64_t wj = (W + g.npar - 1) / g.npar;
    const int64_t rp = (wj + 127) / 128 * 128;
    g.K = (int)(rp / 32);
    g.Kg = g.K / 4;
    g.passes = (lattice == LAT_DOMINO) ? 2 : (lattice == LAT_LOZENGE ? 3 : 4);
    g.row_words = (int64_t)g.P * g.K;
    g.total_words = (int64_t)(H + 2) * g.row_words;
    return g;
}

static bool box_ok(int64_t W, int64_t H)
{
    return W >= 2 && H >= 2 && W <= 65536 && H <= 65536 && W * H <= (int64_t)1 << 31;
}

// Edge access on a canonical array, zero outside the box.
struct Canon {
    const uint8_t* s;
    int W, H;
    int at(int type, int x, int y) const
    {
        if (x < 0 || y < 0 || x >= W || y >= H) return 0;
        return s[((size_t)type * H + y) * W + x];
    }
};

// Groups of a row that hold sites of the domain.
static void set_group_range(tl_domain* d, int row, int jmin, int jmax)
{
    if (jmin > jmax) d->grange[row] = make_int2(0, 0);
    else d->grange[row] = make_int2(jmin >> 7, (jmax >> 7) + 1);
}

// Height segments over a grid of hw x hh points, given membership tests
// for points, for the horizontal step (x,y)-(x+1,y) and for the vertical
// step (x,y-1)-(x,y).  A segment is a maximal run of domain points of one
// row joined by domain steps; segments are linked into a tree by vertical
// steps, breadth first from the segment holding the first domain point in
// (y, x) order, so every parent precedes its children.  Entry s of hseg is
// (y, lo, hi, parent, xs, dir), dir = +1 if the segment lies above its
// parent.  A domain whose segments are not all linked is not connected.
template <class InV, class InH, class InVert>
static int plan_heights(tl_domain* d, int hw, int hh, InV inv, InH inh, InVert invert)
{
    d->hw = hw;
    d->hh = hh;
    struct Seg {
        int y, lo, hi;
    };
    std::vector<Seg> segs;
    std::vector<int> row_first(hh + 1, 0);
    for (int y = 0; y < hh; ++y) {
        row_first[y] = (int)segs.size();
        int x = 0;
        while (x < hw) {
            if (!inv(x, y)) {
                ++x;
                continue;
            }
            const int lo = x;
            while (x + 1 < hw && inv(x + 1, y) && inh(x, y)) ++x;
            segs.push_back(Seg{y, lo, x});
            ++x;
        }
    }
    row_first[hh] = (int)segs.size();
    const int n = (int)segs.size();
    d->nseg = n;
    d->hseg.assign((size_t)6 * n, 0);
    if (n == 0) return TL_OK;
    // breadth-first linking; `order` lists segments parent first
    std::vector<int> parent(n, -2), xs(n, -1), dir(n, 0), order;
    order.reserve(n);
    parent[0] = -1;
    order.push_back(0);
    for (size_t qi = 0; qi < order.size(); ++qi) {
        const Seg& sg = segs[order[qi]];
        for (int dy = -1; dy <= 1; dy += 2) {
            const int ny = sg.y + dy;
            if (ny < 0 || ny >= hh) continue;
            // unlinked segments of the neighbouring row that overlap this one
            for (int t = row_first[ny]; t < row_first[ny + 1]; ++t) {
                if (parent[t] != -2 || segs[t].hi < sg.lo || segs[t].lo > sg.hi) continue;
                const int a = std::max(sg.lo, segs[t].lo), b = std::min(sg.hi, segs[t].hi);
                for (int x = a; x <= b; ++x)
                    if (invert(x, dy > 0 ? ny : sg.y)) {
                        parent[t] = order[qi];
                        xs[t] = x;
                        dir[t] = dy;
                        order.push_back(t);
                        break;
                    }
            }
        }
    }
    if ((int)order.size() != n) return fail(TL_ENOTSIMPLY, "height: the domain is not connected");
    std::vector<int> pos(n);
    for (int i = 0; i < n; ++i) pos[order[i]] = i;
    for (int i = 0; i < n; ++i) {
        const int sidx = order[i];
        int* e = &d->hseg[(size_t)6 * i];
        e[0] = segs[sidx].y;
        e[1] = segs[sidx].lo;
        e[2] = segs[sidx].hi;
        e[3] = parent[sidx] < 0 ? -1 : pos[parent[sidx]];
        e[4] = xs[sidx];
        e[5] = dir[sidx];
    }
    return TL_OK;
}

// Derive the face set, sites, group ranges and height plan of a domino
// domain from a tiling of it.
static int analyse_domino(tl_domain* d, int aztec_n)
{
    const Geom& g = d->g;
    const int W = g.W, H = g.H;
    Canon c{d->init.data(), W, H};
    d->cover.assign((size_t)(W - 1) * (H - 1), 0);
    auto face = [&](int x, int y) -> int {
        if (x < 0 || y < 0 || x >= W - 1 || y >= H - 1) return 0;
        return d->cover[(size_t)y * (W - 1) + x];
    };
    for (int y = 0; y < H - 1; ++y)
        for (int x = 0; x < W - 1; ++x) {
            const int k = c.at(0, x, y) + c.at(0, x, y + 1) + c.at(1, x, y) + c.at(1, x + 1, y);
            if (k > 1) return fail(TL_EINVAL, "domino: face (%d,%d) covered twice", x, y);
            d->cover[(size_t)y * (W - 1) + x] = (uint8_t)k;
        }
    d->grange.assign(H, make_int2(0, 0));
    d->sites = 0;
    for (int y = 0; y < H; ++y) {
        int jmin = 1 << 30, jmax = -1;
        for (int x = 0; x < W; ++x)
            if (face(x - 1, y - 1) && face(x, y - 1) && face(x - 1, y) && face(x, y)) {
                ++d->sites;
                jmin = std::min(jmin, x >> 1);
                jmax = std::max(jmax, x >> 1);
            }
        set_group_range(d, y, jmin, jmax);
    }
    d->edges = 0;
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x) {
            d->edges += face(x, y - 1) && face(x, y);   // horizontal edge between two faces
            d->edges += face(x - 1, y) && face(x, y);   // vertical edge between two faces
        }
    d->kappa = aztec_n > 0 ? (aztec_n & 1) : 0;
    auto inv = [&](int x, int y) { return face(x, y) || face(x - 1, y) || face(x, y - 1) || face(x - 1, y - 1); };
    auto inh = [&](int x, int y) { return face(x, y) || face(x, y - 1); };
    auto invert = [&](int x, int y) { return face(x - 1, y - 1) || face(x, y - 1); };
    return plan_heights(d, W, H, inv, inh, invert);
}

static int analyse_lozenge(tl_domain* d)
{
    const Geom& g = d->g;
    const int W = g.W, H = g.H;
    Canon c{d->init.data(), W, H};
    // triangles with lower-left corner in [-1, W) x [-1, H) stored with offset 1
    const int TW = W + 1, TH = H + 1;
    d->cover.assign((size_t)2 * TW * TH, 0);
    auto tu = [&](int x, int y) -> int {
        if (x < -1 || y < -1 || x >= W || y >= H) return 0;
        return d->cover[(size_t)(y + 1) * TW + (x + 1)];
    };
    auto td = [&](int x, int y) -> int {
        if (x < -1 || y < -1 || x >= W || y >= H) return 0;
        return d->cover[(size_t)TW * TH + (size_t)(y + 1) * TW + (x + 1)];
    };
    for (int y = -1; y < H; ++y)
        for (int x = -1; x < W; ++x) {
            const int u = c.at(0, x, y) + c.at(1, x + 1, y) + c.at(2, x, y);
            const int v = c.at(2, x, y) + c.at(1, x, y) + c.at(0, x, y + 1);
            if (u > 1 || v > 1) return fail(TL_EINVAL, "lozenge: triangle at (%d,%d) covered twice", x, y);
            d->cover[(size_t)(y + 1) * TW + (x + 1)] = (uint8_t)u;
            d->cover[(size_t)TW * TH + (size_t)(y + 1) * TW + (x + 1)] = (uint8_t)v;
        }
    d->grange.assign(H, make_int2(0, 0));
    d->sites = 0;
    for (int y = 0; y < H; ++y) {
        int jmin = 1 << 30, jmax = -1;
        for (int x = 0; x < W; ++x)
            if (tu(x, y) && td(x, y) && tu(x - 1, y) && td(x - 1, y - 1) && tu(x - 1, y - 1) && td(x, y - 1)) {
                ++d->sites;
                jmin = std::min(jmin, x / 3);
                jmax = std::max(jmax, x / 3);
            }
        set_group_range(d, y, jmin, jmax);
    }
    d->edges = 0;
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x) {
            d->edges += tu(x, y) && td(x, y - 1);       // E1(x,y)
            d->edges += td(x, y) && tu(x - 1, y);       // E2(x,y)
            d->edges += tu(x, y) && td(x, y);           // E3(x,y)
        }
    auto inv = [&](int x, int y) {
        return tu(x, y) || td(x, y) || tu(x - 1, y) || td(x - 1, y - 1) || tu(x - 1, y - 1) || td(x, y - 1);
    };
    auto inh = [&](int x, int y) { return tu(x, y) || td(x, y - 1); };
    auto invert = [&](int x, int y) { return td(x, y - 1) || tu(x - 1, y - 1); };
    return plan_heights(d, W, H, inv, inh, invert);
}

static int analyse_sixv(tl_domain* d)
{
    const int N = d->g.N;
    d->grange.assign(d->g.H, make_int2(0, 0));
    const int gmax = (((N - 1) >> 1) >> 7) + 1;
    for (int Y = 1; Y <= N - 1; ++Y) d->grange[Y] = make_int2(0, gmax);
    d->sites = (uint64_t)(N - 1) * (N - 1);
    d->edges = (uint64_t)2 * N * (N - 1);
    d->hw = d->hh = N + 1;
    d->nseg = N + 1;
    d->hseg.assign((size_t)6 * (N + 1), 0);
    for (int y = 0; y <= N; ++y) {
        int* e = &d->hseg[(size_t)6 * y];
        e[0] = y;
        e[1] = 0;
        e[2] = N;
        e[3] = y - 1;
        e[4] = 0;
        e[5] = 1;
    }
    return TL_OK;
}

static int finish_domain(tl_domain* d, int aztec_n, tl_domain** out)
{
    int rc;
    if (d->g.lattice == LAT_DOMINO) rc = analyse_domino(d, aztec_n);
    else if (d->g.lattice == LAT_LOZENGE) rc = analyse_lozenge(d);
    else rc = analyse_sixv(d);
    if (rc != TL_OK) {
        delete d;
        return rc;
    }
    *out = d;
    return TL_OK;
}

// Aztec diamond of order n.  Each row of faces is an interval centred on
// x = n; the start tiles every row with horizontal dominoes from its left end.
TL_API int tl_domain_aztec(int n, tl_domain** out)
{
    if (!out || n < 1 || !box_ok(2 * (int64_t)n + 1, 2 * (int64_t)n + 1))
        return fail(TL_EINVAL, "tl_domain_aztec: bad order %d", n);
    tl_domain* d = new (std::nothrow) tl_domain();
    if (!d) return fail(TL_ENOMEM, "tl_domain_aztec: host allocation");
    const int W = 2 * n + 1;
    d->g = make_geom(LAT_DOMINO, W, W, 0);
    d->init.assign((size_t)2 * W * W, 0);
    uint8_t* vt = d->init.data() + (size_t)W * W;
    for (int fy = 0; fy < 2 * n; ++fy) {
        const int half = (fy < n) ? fy + 1 : 2 * n - fy;   // faces per half-row
        for (int fx = n - half; fx < n + half; fx += 2) vt[(size_t)fy * W + fx + 1] = 1;
    }
    return finish_domain(d, n, out);
}

TL_API int tl_domain_rect(int w, int h, tl_domain** out)
{
    if (!out || w < 1 || h < 1 || !box_ok((int64_t)w + 1, (int64_t)h + 1))
        return fail(TL_EINVAL, "tl_domain_rect: bad size %dx%d", w, h);
    if ((int64_t)w * h % 2) return fail(TL_ENOTTILEABLE, "tl_domain_rect: %dx%d has odd area", w, h);
    tl_domain* d = new (std::nothrow) tl_domain();
    if (!d) return fail(TL_ENOMEM, "tl_domain_rect: host allocation");
    const int W = w + 1, H = h + 1;
    d->g = make_geom(LAT_DOMINO, W, H, 0);
    d->init.assign((size_t)2 * W * H, 0);
    uint8_t* hz = d->init.data();
    uint8_t* vt = d->init.data() + (size_t)W * H;
    for (int fy = 0; fy < h; ++fy)
        for (int fx = 0; fx < w; ++fx) {
            if (w % 2 == 0) {
                if (fx % 2 == 0) vt[(size_t)fy * W + fx + 1] = 1;
            } else if (fy % 2 == 0) {
                hz[(size_t)(fy + 1) * W + fx] = 1;
            }
        }
    return finish_domain(d, 0, out);
}

// Hexagon a x b x c: the tiling of a plane partition pi (heights of the
// cube stacks over the a x b floor) seen along (1,1,1).  A unit square of
// the stepped surface is a lozenge whose short diagonal is an edge of the
// triangular lattice; a point (i,j,k) maps to the box vertex
// (i - k + c, j - k + c).  The start is pi = 0 (the empty box).
TL_API int tl_domain_hexagon(int a, int b, int c, tl_domain** out)
{
    if (!out || a < 1 || b < 1 || c < 1 || !box_ok((int64_t)a + c + 1, (int64_t)b + c + 1))
        return fail(TL_EINVAL, "tl_domain_hexagon: bad sides %d,%d,%d", a, b, c);
    tl_domain* d = new (std::nothrow) tl_domain();
    if (!d) return fail(TL_ENOMEM, "tl_domain_hexagon: host allocation");
    const int W = a + c + 1, H = b + c + 1;
    d->g = make_geom(LAT_LOZENGE, W, H, 0);
    d->init.assign((size_t)3 * W * H, 0);
    auto mark = [&](int type, int i, int j, int k) {
        // short diagonal from the corner (i,j,k) of a unit square
        int x = i - k + c, y = j - k + c;
        if (type == 0) x -= 1;        // square normal to e1: diagonal to (-1, 0)
        else if (type == 1) y -= 1;   // square normal to e2: diagonal to (0, -1)
        d->init[((size_t)type * H + y) * W + x] = 1;
    };
    for (int i = 0; i < a; ++i)
        for (int j = 0; j < b; ++j) mark(2, i, j, 0);   // floor, normal e3
    for (int j = 0; j < b; ++j)
        for (int k = 0; k < c; ++k) mark(0, 0, j, k);   // wall x = 0, normal e1
    for (int i = 0; i < a; ++i)
        for (int k = 0; k < c; ++k) mark(1, i, 0, k);   // wall y = 0, normal e2
    return finish_domain(d, 0, out);
}

// Domain-wall boundary: bottom and left external edges occupied.  Start:
// the path entering column k+1 goes up to row k+1 and leaves to the left.
TL_API int tl_domain_dwbc(int N, tl_domain** out)
{
    if (!out || N < 2 || !box_ok((int64_t)N + 2, (int64_t)N + 2))
        return fail(TL_EINVAL, "tl_domain_dwbc: bad size %d", N);
    tl_domain* d = new (std::nothrow) tl_domain();
    if (!d) return fail(TL_ENOMEM, "tl_domain_dwbc: host allocation");
    const int B = N + 2;
    d->g = make_geom(LAT_SIXV, B, B, N);
    d->init.assign((size_t)2 * B * B, 0);
    uint8_t* hz = d->init.data();
    uint8_t* vt = d->init.data() + (size_t)B * B;
    for (int col = 1; col <= N; ++col) {
        for (int Y = 0; Y < col; ++Y) vt[(size_t)Y * B + col] = 1;     // up column `col`
        for (int X = 0; X < col; ++X) hz[(size_t)col * B + X] = 1;     // left along row `col`
    }
    return finish_domain(d, 0, out);
}

// ---------------------------------------------------------------------------
// Extreme configurations and domains from a boundary path (Sec. 1.1: the
// maximal and minimal tilings; tileability by Thurston's algorithm).
// ---------------------------------------------------------------------------

// Height edges of a domino region, faces given by F(x, y) (lower-left
// corner (x, y)).  Along an edge the height rises by 1 if the face on its
// left is black (x + y even) and falls by 1 otherwise; across a domino the
// step is -3 times that (Fig. 2).
template <class Face>
static void domino_region(int W, int H, Face F, std::vector<uint8_t>& active, std::vector<HEdge>& edges)
{
    active.assign((size_t)W * H, 0);
    edges.clear();
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x)
            active[(size_t)y * W + x] = F(x, y) || F(x - 1, y) || F(x, y - 1) || F(x - 1, y - 1);
    for (int y = 0; y < H; ++y)
        for (int x = 0; x + 1 < W; ++x) {
            const bool a = F(x, y), b = F(x, y - 1);   // above, below (left, right of the step +x)
            if (!a && !b) continue;
            const int8_t af = ((x + y) & 1) == 0 ? 1 : -1;
            edges.push_back(HEdge{y * W + x, y * W + x + 1, af, (int8_t)(-3 * af), (uint8_t)(a && b),
                                  (int64_t)y * W + x});
        }
    for (int y = 0; y + 1 < H; ++y)
        for (int x = 0; x < W; ++x) {
            const bool l = F(x - 1, y), r = F(x, y);   // left, right of the step +y
            if (!l && !r) continue;
            const int8_t af = ((x - 1 + y) & 1) == 0 ? 1 : -1;
            edges.push_back(HEdge{y * W + x, (y + 1) * W + x, af, (int8_t)(-3 * af), (uint8_t)(l && r),
                                  (int64_t)H * W + (int64_t)y * W + x});
        }
}

// Height edges of a lozenge region, triangles given by U(x, y) (vertices
// (x,y), (x+1,y), (x+1,y+1)) and D(x, y) (vertices (x,y), (x+1,y+1),
// (x,y+1)).  The height is the k-coordinate of the stepped surface: a free
// E1 or E2 step keeps it and a crossed one (a lozenge's short diagonal)
// lowers it by one; a free E3 step lowers it by one and a crossed one keeps it.
template <class Up, class Dn>
static void lozenge_region(int W, int H, Up U, Dn D, std::vector<uint8_t>& active, std::vector<HEdge>& edges)
{
    active.assign((size_t)W * H, 0);
    edges.clear();
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x)
            active[(size_t)y * W + x] =
                U(x, y) || D(x, y) || U(x - 1, y) || D(x - 1, y - 1) || U(x - 1, y - 1) || D(x, y - 1);
    const int64_t plane = (int64_t)W * H;
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x) {
            const int v = y * W + x;
            if (x + 1 < W) {   // E1: up(x,y) | down(x,y-1)
                const bool a = U(x, y), b = D(x, y - 1);
                if (a || b) edges.push_back(HEdge{v, v + 1, 0, -1, (uint8_t)(a && b), (int64_t)v});
            }
            if (y + 1 < H) {   // E2: down(x,y) | up(x-1,y)
                const bool a = D(x, y), b = U(x - 1, y);
                if (a || b) edges.push_back(HEdge{v, v + W, 0, -1, (uint8_t)(a && b), plane + v});
            }
            if (x + 1 < W && y + 1 < H) {   // E3: up(x,y) | down(x,y)
                const bool a = U(x, y), b = D(x, y);
                if (a || b) edges.push_back(HEdge{v, v + W + 1, -1, 0, (uint8_t)(a && b), 2 * plane + v});
            }
        }
}

// Configuration with the maximal (`up`) or minimal height function.  For
// lozenges and the six-vertex model these are the configurations with every
// rotatable site UP (a cube added; paths through B and L) or DOWN; for
// dominoes a rotation raises the height at sites of one colour and lowers
// it at the other, so T_max and T_min mix both kinds of blocks.
static int extreme_config(const tl_domain* d, bool up, std::vector<uint8_t>& out)
{
    const Geom& g = d->g;
    const int W = g.W, H = g.H;
    out.assign(d->init.size(), 0);
    if (g.lattice == LAT_SIXV) {
        if (!up) {
            out = d->init;
            return TL_OK;
        }
        // paths hug the top right: the path entering column X rises to row N+1-X
        const int N = g.N, B = N + 2;
        uint8_t* hz = out.data();
        uint8_t* vt = out.data() + (size_t)B * B;
        for (int Y = 1; Y <= N; ++Y)
            for (int X = 0; X <= N - Y; ++X) hz[(size_t)Y * B + X] = 1;
        for (int X = 1; X <= N; ++X)
            for (int Y = 0; Y <= N - X; ++Y) vt[(size_t)Y * B + X] = 1;
        return TL_OK;
    }
    std::vector<uint8_t> active;
    std::vector<HEdge> edges;
    bool top;
    if (g.lattice == LAT_DOMINO) {
        auto F = [&](int x, int y) {
            return x >= 0 && y >= 0 && x < W - 1 && y < H - 1 && d->cover[(size_t)y * (W - 1) + x] != 0;
        };
        domino_region(W, H, F, active, edges);
        top = up;
    } else {
        const int TW = W + 1, TH = H + 1;
        auto U = [&](int x, int y) {
            return x >= -1 && y >= -1 && x < W && y < H && d->cover[(size_t)(y + 1) * TW + (x + 1)] != 0;
        };
        auto D = [&](int x, int y) {
            return x >= -1 && y >= -1 && x < W && y < H &&
                   d->cover[(size_t)TW * TH + (size_t)(y + 1) * TW + (x + 1)] != 0;
        };
        lozenge_region(W, H, U, D, active, edges);
        top = up;
    }
    std::vector<int> h;
    std::string why;
    const int rc = thurston_heights(W * H, active, edges, top, h, why);
    if (rc != TL_OK) return fail(rc, "extreme configuration: %s", why.c_str());
    tiling_from_heights(edges, h, out.data());
    return TL_OK;
}

TL_API int tl_domain_extreme_state(const tl_domain* d, int which, uint8_t* canon, size_t cap)
{
    if (!d || !canon || (which != TL_EXTREME_BOTTOM && which != TL_EXTREME_TOP))
        return fail(TL_EINVAL, "tl_domain_extreme_state: bad argument");
    if (cap < d->init.size()) return fail(TL_EINVAL, "tl_domain_extreme_state: cap %zu < %zu", cap, d->init.size());
    std::vector<uint8_t> cfg;
    TL_TRY(extreme_config(d, which == TL_EXTREME_TOP, cfg));
    std::memcpy(canon, cfg.data(), cfg.size());
    return TL_OK;
}

// Face (triangle) membership by winding number: for each cell the signed
// count of path steps crossing a ray from its centre towards +x.
TL_API int tl_domain_from_boundary(int lattice, const int8_t* steps, size_t nsteps, tl_domain** out)
{
    if (!out || !steps || (lattice != TL_DOMINO && lattice != TL_LOZENGE))
        return fail(TL_EINVAL, "tl_domain_from_boundary: bad argument");
    if (nsteps < 3 || nsteps > ((size_t)1 << 28)) return fail(TL_EINVAL, "tl_domain_from_boundary: %zu steps", nsteps);
    static const int DX[2][6] = {{1, 0, -1, 0, 0, 0}, {1, 0, 1, -1, 0, -1}};
    static const int DY[2][6] = {{0, 1, 0, -1, 0, 0}, {0, 1, 1, 0, -1, -1}};
    const int L = lattice == TL_DOMINO ? 0 : 1, ndir = L ? 6 : 4;
    std::vector<int64_t> px(nsteps + 1), py(nsteps + 1);
    px[0] = py[0] = 0;
    for (size_t i = 0; i < nsteps; ++i) {
        const int s = steps[i];
        if (s < 0 || s >= ndir) return fail(TL_EINVAL, "tl_domain_from_boundary: step %zu = %d", i, s);
        px[i + 1] = px[i] + DX[L][s];
        py[i + 1] = py[i] + DY[L][s];
    }
    if (px[nsteps] != 0 || py[nsteps] != 0) return fail(TL_EINVAL, "tl_domain_from_boundary: path is not closed");
    const int64_t x0 = *std::min_element(px.begin(), px.end()), y0 = *std::min_element(py.begin(), py.end());
    const int64_t W = *std::max_element(px.begin(), px.end()) - x0 + 1;
    const int64_t H = *std::max_element(py.begin(), py.end()) - y0 + 1;
    if (!box_ok(W, H)) return fail(TL_EINVAL, "tl_domain_from_boundary: box %lldx%lld", (long long)W, (long long)H);
    {
        std::vector<uint8_t> seen((size_t)W * H, 0);
        for (size_t i = 0; i < nsteps; ++i) {
            uint8_t& v = seen[(size_t)(py[i] - y0) * W + (px[i] - x0)];
            if (v) return fail(TL_ENOTSIMPLY, "tl_domain_from_boundary: path visits a point twice (step %zu)", i);
            v = 1;
        }
    }
    // signed crossings per row band [y, y+1]: vertical (E2) steps at x, and
    // for lozenges diagonal (E3) steps leaving row y at x
    std::vector<int> cv((size_t)W * H, 0), cd((size_t)W * H, 0);
    for (size_t i = 0; i < nsteps; ++i) {
        const int64_t x = px[i] - x0, y = py[i] - y0;
        const int s = steps[i], dx = DX[L][s], dy = DY[L][s];
        if (dy == 0) continue;
        const int64_t yb = dy > 0 ? y : y - 1;           // band crossed
        const int64_t xb = dy > 0 ? x : x + dx;           // x of the step's lower end
        int* arr = dx == 0 ? cv.data() : cd.data();
        arr[(size_t)yb * W + xb] += dy;
    }
    // suffix sums: cells to the left of a crossing see it
    for (int64_t y = 0; y < H; ++y)
        for (int64_t x = W - 2; x >= 0; --x) {
            cv[(size_t)y * W + x] += cv[(size_t)y * W + x + 1];
            cd[(size_t)y * W + x] += cd[(size_t)y * W + x + 1];
        }
    auto SV = [&](int64_t x, int64_t y) { return x < W ? cv[(size_t)y * W + x] : 0; };
    auto SD = [&](int64_t x, int64_t y) { return x < W ? cd[(size_t)y * W + x] : 0; };
    tl_domain* d = new (std::nothrow) tl_domain();
    if (!d) return fail(TL_ENOMEM, "tl_domain_from_boundary: host allocation");
    std::vector<uint8_t> active;
    std::vector<HEdge> edges;
    int64_t cells = 0;
    const bool top = false;   // start: T_min
    if (!L) {
        d->g = make_geom(LAT_DOMINO, (int)W, (int)H, 0);
        std::vector<uint8_t> face((size_t)(W - 1) * (H - 1), 0);
        for (int64_t y = 0; y + 1 < H; ++y)
            for (int64_t x = 0; x + 1 < W; ++x) {
                face[(size_t)y * (W - 1) + x] = SV(x + 1, y) != 0;   // centre (x + 1/2, y + 1/2)
                cells += face[(size_t)y * (W - 1) + x];
            }
        auto F = [&](int x, int y) {
            return x >= 0 && y >= 0 && x < W - 1 && y < H - 1 && face[(size_t)y * (W - 1) + x] != 0;
        };
        domino_region((int)W, (int)H, F, active, edges);
    } else {
        d->g = make_geom(LAT_LOZENGE, (int)W, (int)H, 0);
        // up (x,y): centre (x + 2/3, y + 1/3); down (x,y): centre (x + 1/3, y + 2/3).
        // A vertical step at x' crosses the ray iff x' >= x + 1; a diagonal
        // step leaving row y at x' crosses at x' + 1/3 (up) or x' + 2/3 (down).
        std::vector<uint8_t> up((size_t)W * H, 0), dn((size_t)W * H, 0);
        for (int64_t y = 0; y + 1 < H; ++y)
            for (int64_t x = 0; x + 1 < W; ++x) {
                up[(size_t)y * W + x] = (SV(x + 1, y) + SD(x + 1, y)) != 0;
                dn[(size_t)y * W + x] = (SV(x + 1, y) + SD(x, y)) != 0;
                cells += up[(size_t)y * W + x] + dn[(size_t)y * W + x];
            }
        auto U = [&](int x, int y) { return x >= 0 && y >= 0 && x < W && y < H && up[(size_t)y * W + x] != 0; };
        auto D = [&](int x, int y) { return x >= 0 && y >= 0 && x < W && y < H && dn[(size_t)y * W + x] != 0; };
        lozenge_region((int)W, (int)H, U, D, active, edges);
    }
    if (cells == 0 || cells % 2) {
        delete d;
        return fail(TL_ENOTTILEABLE, "tl_domain_from_boundary: %lld cells", (long long)cells);
    }
    std::vector<int> h;
    std::string why;
    const int rc = thurston_heights((int)(W * H), active, edges, top, h, why);
    if (rc != TL_OK) {
        delete d;
        return fail(rc, "tl_domain_from_boundary: %s", why.c_str());
    }
    d->init.assign((size_t)d->g.ntype * W * H, 0);
    tiling_from_heights(edges, h, d->init.data());
    return finish_domain(d, 0, out);
}

TL_API void tl_domain_destroy(tl_domain* d) { delete d; }

TL_API int tl_domain_get_info(const tl_domain* d, tl_domain_info* o)
{
    if (!d || !o) return fail(TL_EINVAL, "tl_domain_get_info: NULL argument");
    o->lattice = d->g.lattice;
    o->width = d->g.W;
    o->height = d->g.H;
    o->planes = d->g.ntype;
    o->passes = d->g.passes;
    o->sites = d->sites;
    o->edges = d->edges;
    o->canon_bytes = (uint64_t)d->g.ntype * d->g.W * d->g.H;
    o->packed_bytes = (uint64_t)d->g.total_words * 4;
    o->site_box = (uint64_t)d->g.W * d->g.H;
    o->height_count = (uint64_t)d->hw * d->hh;
    o->height_width = d->hw;
    o->height_height = d->hh;
    return TL_OK;
}

TL_API int tl_domain_initial_state(const tl_domain* d, uint8_t* canon, size_t cap)
{
    if (!d || !canon) return fail(TL_EINVAL, "tl_domain_initial_state: NULL argument");
    if (cap < d->init.size()) return fail(TL_EINVAL, "tl_domain_initial_state: cap %zu < %zu", cap, d->init.size());
    std::memcpy(canon, d->init.data(), d->init.size());
    return TL_OK;
}

// A canonical configuration is valid for the domain if it covers exactly
// the domain's faces (triangles) once each, or for six-vertex if every model
// vertex obeys the ice rule and the external edges match the boundary.
static int validate(const tl_domain* d, const uint8_t* s)
{
    const Geom& g = d->g;
    Canon c{s, g.W, g.H};
    const size_t n = (size_t)g.ntype * g.W * g.H;
    for (size_t i = 0; i < n; ++i)
        if (s[i] > 1) return fail(TL_EINVAL, "state byte %zu is %d (must be 0 or 1)", i, s[i]);
    if (g.lattice == LAT_DOMINO) {
        for (int y = 0; y < g.H; ++y)
            if (c.at(0, g.W - 1, y)) return fail(TL_EINVAL, "domino: edge outside the box set");
        for (int x = 0; x < g.W; ++x)
            if (c.at(1, x, g.H - 1)) return fail(TL_EINVAL, "domino: edge outside the box set");
        for (int y = 0; y < g.H - 1; ++y)
            for (int x = 0; x < g.W - 1; ++x) {
                const int k = c.at(0, x, y) + c.at(0, x, y + 1) + c.at(1, x, y) + c.at(1, x + 1, y);
                if (k != d->cover[(size_t)y * (g.W - 1) + x])
                    return fail(TL_EINVAL, "domino: face (%d,%d) covered %d times", x, y, k);
            }
        return TL_OK;
    }
    if (g.lattice == LAT_LOZENGE) {
        const int TW = g.W + 1, TH = g.H + 1;
        for (int y = -1; y < g.H; ++y)
            for (int x = -1; x < g.W; ++x) {
                const int u = c.at(0, x, y) + c.at(1, x + 1, y) + c.at(2, x, y);
                const int v = c.at(2, x, y) + c.at(1, x, y) + c.at(0, x, y + 1);
                if (u != d->cover[(size_t)(y + 1) * TW + (x + 1)] ||
                    v != d->cover[(size_t)TW * TH + (size_t)(y + 1) * TW + (x + 1)])
                    return fail(TL_EINVAL, "lozenge: triangles at (%d,%d) not covered once", x, y);
            }
        return TL_OK;
    }
    const int N = g.N;
    for (int Y = 0; Y < g.H; ++Y)
        for (int X = 0; X < g.W; ++X) {
            const bool hreal = Y >= 1 && Y <= N && X <= N;
            const bool vreal = X >= 1 && X <= N && Y <= N;
            if ((c.at(0, X, Y) && !hreal) || (c.at(1, X, Y) && !vreal))
                return fail(TL_EINVAL, "six-vertex: bit set off the lattice at (%d,%d)", X, Y);
        }
    for (int k = 1; k <= N; ++k)
        if (c.at(0, 0, k) != d->init[(size_t)k * g.W] || c.at(0, N, k) != d->init[(size_t)k * g.W + N] ||
            c.at(1, k, 0) != d->init[(size_t)g.W * g.H + k] ||
            c.at(1, k, N) != d->init[(size_t)g.W * g.H + (size_t)N * g.W + k])
            return fail(TL_EINVAL, "six-vertex: external edges differ from the boundary");
    for (int Y = 1; Y <= N; ++Y)
        for (int X = 1; X <= N; ++X) {
            const int L = c.at(0, X - 1, Y), R = c.at(0, X, Y), D = c.at(1, X, Y - 1), U = c.at(1, X, Y);
            if (L + U != D + R) return fail(TL_EINVAL, "six-vertex: ice rule fails at (%d,%d)", X, Y);
        }
    return TL_OK;
}

// ---------------------------------------------------------------------------
// Thresholds (FP64 on the host)
// ---------------------------------------------------------------------------
static uint32_t to_threshold(double p)
{
    const double t = std::floor(p * 4294967296.0);
    if (!(t > 0.0)) return 0u;
    if (t >= 4294967295.0) return 0xFFFFFFFFu;
    return (uint32_t)t;
}

TL_API int tl_thresholds_domino_edge_weights(const tl_domain* d, const double* w, size_t n_w,
                                             uint32_t* t, size_t n_t)
{
    if (!d || !w || !t) return fail(TL_EINVAL, "domino thresholds: NULL argument");
    if (d->g.lattice != LAT_DOMINO) return fail(TL_EINVAL, "domino thresholds: not a domino domain");
    const int W = d->g.W, H = d->g.H;
    if (n_w != (size_t)2 * W * H || n_t != (size_t)W * H)
        return fail(TL_EINVAL, "domino thresholds: sizes %zu/%zu, want %zu/%zu", n_w, n_t,
                    (size_t)2 * W * H, (size_t)W * H);
    for (size_t i = 0; i < n_w; ++i)
        if (!(w[i] > 0.0) || !std::isfinite(w[i])) return fail(TL_EINVAL, "domino thresholds: weight %zu not positive", i);
    const double* hz = w;
    const double* vt = w + (size_t)W * H;
    auto H_ = [&](int x, int y) { return (x < 0 || y < 0 || x >= W || y >= H) ? 1.0 : hz[(size_t)y * W + x]; };
    auto V_ = [&](int x, int y) { return (x < 0 || y < 0 || x >= W || y >= H) ? 1.0 : vt[(size_t)y * W + x]; };
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x) {
            const double up = H_(x, y) * H_(x - 1, y);
            const double down = V_(x, y) * V_(x, y - 1);
            t[(size_t)y * W + x] = to_threshold(up / (up + down));
        }
    return TL_OK;
}

TL_API int tl_thresholds_volume(const tl_domain* d, const double* q, size_t n_q, uint32_t* t, size_t n_t)
{
    if (!d || !q || !t) return fail(TL_EINVAL, "volume thresholds: NULL argument");
    if (d->g.lattice == LAT_SIXV) return fail(TL_EINVAL, "volume thresholds: six-vertex uses tl_thresholds_6v");
    const int W = d->g.W, H = d->g.H;
    if (n_q != (size_t)W * H || n_t != (size_t)W * H)
        return fail(TL_EINVAL, "volume thresholds: sizes %zu/%zu, want %zu", n_q, n_t, (size_t)W * H);
    for (size_t i = 0; i < n_q; ++i)
        if (!(q[i] >= 1e-75 && q[i] <= 1e75))   // q^4 stays a normal double
            return fail(TL_EINVAL, "volume thresholds: q[%zu] = %g outside [1e-75, 1e75]", i, q[i]);
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < W; ++x) {
            const double qv = q[(size_t)y * W + x];
            double p;
            if (d->g.lattice == LAT_DOMINO) {
                const double q4 = (qv * qv) * (qv * qv);
                p = ((x + y) & 1) == 0 ? q4 / (1.0 + q4) : 1.0 / (1.0 + q4);
            } else {
                p = qv / (1.0 + qv);
            }
            t[(size_t)y * W + x] = to_threshold(p);
        }
    return TL_OK;
}

TL_API int tl_thresholds_lognormal_device(const tl_domain* d, double sigma, uint64_t seed, uint32_t* t_dev,
                                          size_t n_t, void* stream)
{
    if (!d || !t_dev || !(sigma >= 0.0) || !std::isfinite(sigma))
        return fail(TL_EINVAL, "tl_thresholds_lognormal_device: bad argument");
    if (d->g.lattice == LAT_SIXV) return fail(TL_EINVAL, "tl_thresholds_lognormal_device: six-vertex uses tl_thresholds_6v");
    if (n_t < (size_t)d->g.W * d->g.H) return fail(TL_EINVAL, "tl_thresholds_lognormal_device: n_t too small");
    const int e = launch_lognormal_thresholds(d->g.lattice, d->g.W, d->g.H, sigma, seed, t_dev, stream);
    if (e) return fail(TL_ECUDA, "tl_thresholds_lognormal_device: %s", cudaGetErrorString((cudaError_t)e));
    return TL_OK;
}

TL_API int tl_thresholds_lozenge_q(double q, uint32_t* t_add, uint32_t* t_rem)
{
    if (!t_add || !t_rem || !(q > 0.0) || !std::isfinite(q)) return fail(TL_EINVAL, "lozenge thresholds: bad q");
    const uint32_t ta = to_threshold(q / (1.0 + q));
    if (ta == 0) return fail(TL_EINVAL, "lozenge thresholds: q=%g gives t_add = 0", q);
    *t_add = ta;
    *t_rem = (uint32_t)((((uint64_t)1) << 32) - ta);
    return TL_OK;
}

// Corner vertex types of a face in its two states (Fig. 5A types
// a1=0 a2=1 b1=2 b2=3 c1=4 c2=5), keyed by the corner's external bit.
// Rows: top-left (bit Vt(X,Y+1)), top-right (Hz(X+1,Y+1)), bottom-right
// (Hz(X+1,Y)), bottom-left (Hz(X-1,Y)); entries {A-type, B-type} for the
// bit = 0 and bit = 1.
static const int kCorner[4][2][2] = {
    {{2, 4}, {5, 3}},   // TL: 0 -> (b1, c1), 1 -> (c2, b2)
    {{4, 0}, {1, 5}},   // TR: 0 -> (c1, a1), 1 -> (a2, c2)
    {{3, 4}, {5, 2}},   // BR: 0 -> (b2, c1), 1 -> (c2, b1)
    {{0, 5}, {4, 1}},   // BL: 0 -> (a1, c2), 1 -> (c1, a2)
};

TL_API int tl_thresholds_6v(const double w6[6], uint32_t t16[16])
{
    if (!w6 || !t16) return fail(TL_EINVAL, "six-vertex thresholds: NULL argument");
    for (int i = 0; i < 6; ++i)
        if (!(w6[i] > 0.0) || !std::isfinite(w6[i])) return fail(TL_EINVAL, "six-vertex thresholds: weight %d", i);
    for (int idx = 0; idx < 16; ++idx) {
        const int b[4] = {idx & 1, (idx >> 1) & 1, (idx >> 2) & 1, (idx >> 3) & 1};
        const double wa = w6[kCorner[0][b[0]][0]] * w6[kCorner[1][b[1]][0]] * w6[kCorner[2][b[2]][0]] *
                          w6[kCorner[3][b[3]][0]];
        const double wb = w6[kCorner[0][b[0]][1]] * w6[kCorner[1][b[1]][1]] * w6[kCorner[2][b[2]][1]] *
                          w6[kCorner[3][b[3]][1]];
        t16[idx] = to_threshold(wb / (wa + wb));
    }
    return TL_OK;
}

// ---------------------------------------------------------------------------
// Chains
// ---------------------------------------------------------------------------
struct tl_chain {
    tl_ctx* ctx = nullptr;
    Geom g{};
    uint64_t sites = 0;
    int kappa = 0;
    std::vector<uint8_t> cover;        // for validation of written states
    std::vector<uint8_t> init;         // boundary reference (six-vertex)
    tl_domain dom_copy;                // host copy of the domain description
    uint32_t* rows = nullptr;          // packed state
    uint32_t* rows0 = nullptr;         // packed starting state (for reset)
    int2* grange = nullptr;
    uint8_t* canon = nullptr;          // staging buffer [ntype][H][W]
    uint32_t* tplanes = nullptr;       // per-site threshold planes
    ThrView th{};
    DevRng rng{};
    uint64_t seed = 0;
    uint32_t stream_id = 0;
    uint64_t sweep = 0;
    uint64_t launches = 0;
    // observables
    unsigned long long* hash = nullptr;
    uint32_t* counts = nullptr;        // canonical counters, decoded at readback
    uint32_t* cplanes = nullptr;       // bit-sliced counters [32][H][row_words]
    uint64_t samples = 0;
    uint32_t stride = 0;
    uint64_t burn = 0;
    bool density_on = false;
    bool counts_dirty = false;         // counters to be zeroed on the next run's stream
    int* hseg = nullptr;
    int* hbase = nullptr;
    int32_t* hscratch = nullptr;
    // planner
    int kernel = 0;
    int spl = 0;
    int halo_req = 0;
    bool res_ready = false, res_failed = false;
    ResidentPlan res{};
    int* stripe_d = nullptr;
    unsigned long long* xbuf_d = nullptr;
    int* status_d = nullptr;           // error word, then a word per stripe (ResidentPlan::loaded)
    int threads_req = 0, npre_req = 0;
    int random_order = 0;   // colours of the pass slots drawn per sweep
    uint8_t* colours = nullptr;   // device colours of one resident launch's slots
    size_t colours_cap = 0;
    unsigned int epoch = 0;
    std::string res_why;
    // accepted-flip counter (tl_chain_count_flips)
    unsigned long long* flips_d = nullptr;
    bool count_flips = false;
    // thresholds as given, for checkpoints
    int thr_api_kind = 0;
    std::vector<uint32_t> thr_site;    // TL_T_SITE: [H][W]
    uint32_t thr_table16[16] = {};
    // register-resident domino kernel (dominoes at t = 2^31)
    bool use_reg = false;
    RegPlan reg{};
    int small_threads = 0;             // > 0: plain runs take the one-block kernel
    int2* hull_d = nullptr;
    // device validation of written states: the domain's cover or boundary
    // edges, and the first failure found
    uint8_t* vaux_d = nullptr;
    unsigned long long* vfirst_d = nullptr;
    // device staging of density read-backs to host memory (grown on demand)
    double* dscratch = nullptr;
    size_t dscratch_n = 0;
};

static void chain_free(tl_chain* c)
{
    if (!c) return;
    cudaFree(c->rows);
    cudaFree(c->rows0);
    cudaFree(c->grange);
    cudaFree(c->canon);
    cudaFree(c->tplanes);
    cudaFree(c->hash);
    cudaFree(c->counts);
    cudaFree(c->cplanes);
    cudaFree(c->colours);
    cudaFree(c->hseg);
    cudaFree(c->hbase);
    cudaFree(c->hscratch);
    cudaFree(c->stripe_d);
    cudaFree(c->xbuf_d);
    cudaFree(c->status_d);
    cudaFree(c->hull_d);
    cudaFree(c->flips_d);
    cudaFree(c->vaux_d);
    cudaFree(c->vfirst_d);
    cudaFree(c->dscratch);
    tl_ctx* ctx = c->ctx;
    delete c;
    ctx_release(ctx);
}

static bool is_device_ptr(const void* p)
{
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// A caller's buffer in device memory of a GPU other than `device`: the
// chain's kernels and copies would fault on it (no peer access is set up),
// so it is rejected with TL_EINVAL.  Host and managed memory pass.
static int require_local(const void* p, int device, const char* fn)
{
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return TL_OK;
    }
    if (a.type == cudaMemoryTypeDevice && a.device != device)
        return fail(TL_EINVAL, "%s: the buffer is on device %d, the chain on device %d", fn, a.device, device);
    return TL_OK;
}

static cudaStream_t SS(void* s) { return reinterpret_cast<cudaStream_t>(s); }

template <class T>
static int dev_alloc(T** p, size_t count, const char* what)
{
    cudaError_t e = cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return fail(e == cudaErrorMemoryAllocation ? TL_ENOMEM : TL_ECUDA, "cudaMalloc(%s, %zu B): %s", what,
                    count * sizeof(T), cudaGetErrorString(e));
    }
    return TL_OK;
}

static int upload_state(tl_chain* c, const uint8_t* canon, bool device_src, void* stream)
{
    const size_t n = (size_t)c->g.ntype * c->g.W * c->g.H;
    CUDA_TRY(cudaMemcpyAsync(c->canon, canon, n, device_src ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                             SS(stream)));
    CUDA_TRY(launch_pack(c->g, c->canon, c->rows, stream));
    c->launches += 1;
    return TL_OK;
}

// Active groups [x, y) of every row; six-vertex: of every pair of face rows.
static std::vector<int2> unit_groups(const tl_domain& d)
{
    const Geom& g = d.g;
    if (g.lattice != LAT_SIXV) return d.grange;
    std::vector<int2> u;
    for (int y = 0; y < g.H; y += 2) {
        int2 a = d.grange[y];
        if (y + 1 < g.H) {
            const int2 b = d.grange[y + 1];
            if (a.y <= a.x) a = b;
            else if (b.y > b.x) a = make_int2(std::min(a.x, b.x), std::max(a.y, b.y));
        }
        u.push_back(a);
    }
    return u;
}

TL_API int tl_chain_create(tl_ctx* ctx, const tl_domain* d, const uint8_t* canon_init, uint64_t seed,
                           uint32_t stream_id, const tl_thresholds* th, tl_chain** out)
{
    if (!ctx || !d || !th || !out) return fail(TL_EINVAL, "tl_chain_create: NULL argument");
    const Geom& g = d->g;
    if (g.lattice == LAT_SIXV && th->kind != TL_T_TABLE16)
        return fail(TL_EINVAL, "tl_chain_create: six-vertex needs a 16-entry table");
    if (g.lattice != LAT_SIXV && th->kind == TL_T_TABLE16)
        return fail(TL_EINVAL, "tl_chain_create: 16-entry tables are for six-vertex only");
    if (th->kind == TL_T_SITE && !th->site) return fail(TL_EINVAL, "tl_chain_create: per-site thresholds missing");
    if (th->kind < 0 || th->kind > 2) return fail(TL_EINVAL, "tl_chain_create: bad threshold kind");
    const uint8_t* start = canon_init ? canon_init : d->init.data();
    if (canon_init) TL_TRY(validate(d, canon_init));
    CUDA_TRY(cudaSetDevice(ctx->device));
    tl_chain* c = new (std::nothrow) tl_chain();
    if (!c) return fail(TL_ENOMEM, "tl_chain_create: host allocation");
    c->ctx = ctx;
    ctx->refs.fetch_add(1);
    c->g = g;
    c->sites = d->sites;
    c->kappa = d->kappa;
    c->dom_copy = *d;
    c->seed = seed;
    c->stream_id = stream_id;
    c->rng.k0 = (uint32_t)seed;
    c->rng.k1 = (uint32_t)(seed >> 32);
    c->rng.stream = stream_id;
    int rc = TL_OK;
    const size_t ncanon = (size_t)g.ntype * g.W * g.H;
    if ((rc = dev_alloc(&c->rows, (size_t)g.total_words, "state")) ||
        (rc = dev_alloc(&c->rows0, (size_t)g.total_words, "start state")) ||
        (rc = dev_alloc(&c->grange, (size_t)g.H + ((size_t)g.H + 2), "group ranges")) ||
        (rc = dev_alloc(&c->canon, ncanon, "staging")) || (rc = dev_alloc(&c->hash, 1, "hash")) ||
        (rc = dev_alloc(&c->hseg, (size_t)6 * std::max(d->nseg, 1), "height plan")) ||
        (rc = dev_alloc(&c->hbase, (size_t)std::max(d->nseg, 1), "height plan"))) {
        chain_free(c);
        return rc;
    }
    // group ranges, then (for batches) the prefix counts and first groups of
    // the rows, for the six-vertex model of the pairs of face rows
    std::vector<int2> gr(d->grange);
    gr.resize((size_t)g.H + ((size_t)g.H + 2), make_int2(0, 0));
    {
        const std::vector<int2> u = unit_groups(*d);
        int* const pre = reinterpret_cast<int*>(gr.data() + g.H);
        int* const first = pre + g.H + 2;
        for (size_t r = 0; r < u.size(); ++r) {
            pre[r + 1] = pre[r] + std::max(0, u[r].y - u[r].x);
            first[r] = u[r].x;
        }
    }
    cudaError_t e = cudaMemcpy(c->grange, gr.data(), sizeof(int2) * gr.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && d->nseg)
        e = cudaMemcpy(c->hseg, d->hseg.data(), sizeof(int) * 6 * d->nseg, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        chain_free(c);
        return fail(TL_ECUDA, "tl_chain_create: upload: %s", cudaGetErrorString(e));
    }
    // thresholds
    c->th.kind = th->kind == TL_T_SITE ? THR_SITE : (th->kind == TL_T_TABLE16 ? THR_TABLE : THR_SCALAR);
    c->thr_api_kind = th->kind;
    if (th->kind == TL_T_TABLE16)
        for (int i = 0; i < 16; ++i) c->thr_table16[i] = th->table16[i];
    c->th.scalar = th->scalar;
    c->th.kmax = th->scalar ? 31 - __builtin_ctz(th->scalar) : -1;
    c->th.planes = nullptr;
    if (th->kind == TL_T_TABLE16) {
        for (int k = 0; k < 32; ++k) {
            uint32_t m = 0;
            for (int idx = 0; idx < 16; ++idx) m |= ((th->table16[idx] >> (31 - k)) & 1u) << idx;
            c->th.tmask[k] = m;
        }
        // tables that depend only on how many corner bits differ from a fixed
        // polarity (the symmetric weights a1 = a2 = b1 = b2, c1 = c2 among
        // them) take a cheaper lookup: a bit-sliced corner count and a
        // 5-entry table
        c->th.cpol = -1;
        for (int pol = 0; pol < 16 && c->th.cpol < 0; ++pol) {
            uint32_t t5[5];
            bool seen[5] = {false, false, false, false, false}, ok = true;
            for (int idx = 0; idx < 16 && ok; ++idx) {
                const int n = __builtin_popcount((unsigned)(idx ^ pol));
                if (!seen[n]) {
                    seen[n] = true;
                    t5[n] = th->table16[idx];
                } else if (t5[n] != th->table16[idx]) {
                    ok = false;
                }
            }
            if (ok) {
                c->th.cpol = pol;
                for (int n = 0; n < 5; ++n) c->th.t5[n] = t5[n];
            }
        }
    } else {
        c->th.cpol = -1;
    }
    if (th->kind == TL_T_SITE) {
        const size_t nplanes = (size_t)g.H * g.npar * 32 * g.K;
        uint32_t* tdev = nullptr;
        if ((rc = dev_alloc(&c->tplanes, nplanes, "threshold planes")) ||
            (rc = dev_alloc(&tdev, (size_t)g.W * g.H, "thresholds"))) {
            cudaFree(tdev);
            chain_free(c);
            return rc;
        }
        e = cudaMemcpy(tdev, th->site, sizeof(uint32_t) * g.W * g.H,
                       is_device_ptr(th->site) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice);
        c->thr_site.resize((size_t)g.W * g.H);
        if (e == cudaSuccess)
            e = cudaMemcpy(c->thr_site.data(), tdev, sizeof(uint32_t) * g.W * g.H, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = (cudaError_t)launch_threshold_planes(g, tdev, c->tplanes, nullptr);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        cudaFree(tdev);
        if (e != cudaSuccess) {
            chain_free(c);
            return fail(TL_ECUDA, "tl_chain_create: threshold planes: %s", cudaGetErrorString(e));
        }
        c->th.planes = c->tplanes;
        c->launches += 1;
    }
    rc = upload_state(c, start, false, nullptr);
    if (rc == TL_OK) {
        e = cudaMemcpyAsync(c->rows0, c->rows, (size_t)g.total_words * 4, cudaMemcpyDeviceToDevice, nullptr);
        if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
        if (e != cudaSuccess) rc = fail(TL_ECUDA, "tl_chain_create: %s", cudaGetErrorString(e));
    }
    if (rc != TL_OK) {
        chain_free(c);
        return rc;
    }
    *out = c;
    return TL_OK;
}

TL_API void tl_chain_destroy(tl_chain* c)
{
    if (c) cudaSetDevice(c->ctx->device);
    chain_free(c);
}

TL_API int tl_chain_reset(tl_chain* c, void* stream)
{
    if (!c) return fail(TL_EINVAL, "tl_chain_reset: NULL chain");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    CUDA_TRY(cudaMemcpyAsync(c->rows, c->rows0, (size_t)c->g.total_words * 4, cudaMemcpyDeviceToDevice, SS(stream)));
    c->sweep = 0;
    c->density_on = false;
    c->samples = 0;
    return TL_OK;
}

TL_API uint64_t tl_chain_sweep(const tl_chain* c) { return c ? c->sweep : 0; }
TL_API uint64_t tl_chain_launches(const tl_chain* c) { return c ? c->launches : 0; }

static bool want_resident(tl_chain* c);
static void free_resident(tl_chain* c);

TL_API int tl_chain_set_plan(tl_chain* c, const tl_plan* p)
{
    if (!c || !p || p->kernel < 0 || p->kernel > 3 || p->sweeps_per_launch < 0 || p->halo < 0 ||
        p->halo > 64 || (p->threads != 0 && p->threads != 512 && p->threads != 1024) || p->npre < 0 ||
        p->npre > 16)
        return fail(TL_EINVAL, "tl_chain_set_plan: bad plan");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    const bool kernel_changed = (p->kernel >= 2) != (c->kernel >= 2) || (c->kernel >= 2 && p->kernel != c->kernel);
    c->spl = p->sweeps_per_launch;
    if (p->halo != c->halo_req || p->threads != c->threads_req || p->npre != c->npre_req || kernel_changed) {
        CUDA_TRY(cudaDeviceSynchronize());
        free_resident(c);
        c->use_reg = false;
        c->res_ready = c->res_failed = false;
        c->halo_req = p->halo;
        c->threads_req = p->threads;
        c->npre_req = p->npre;
    }
    c->kernel = p->kernel;
    if (p->kernel >= 2 && (!want_resident(c) || (p->kernel == 3) != c->use_reg))
        return fail(TL_EUNSUPPORTED, "%s kernel unavailable: %s", p->kernel == 3 ? "register-resident" : "resident",
                    c->res_why.c_str());
    return TL_OK;
}

TL_API int tl_chain_get_plan(tl_chain* c, tl_plan* p)
{
    if (!c || !p) return fail(TL_EINVAL, "tl_chain_get_plan: NULL argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    const bool res = want_resident(c);
    p->kernel = res ? (c->use_reg ? 3 : 2) : 1;
    p->sweeps_per_launch = c->spl;
    p->halo = res ? c->res.halo : 0;
    p->threads = res ? c->res.threads : 256;
    p->npre = res ? c->res.npre : 0;
    p->ctas = res ? c->res.ctas : 0;
    p->smem_bytes = res ? (int)c->res.smem_bytes : 0;
    return TL_OK;
}

// Sweeps [c->sweep, c->sweep + n) with no density sample inside, one launch
// per pass over global memory.
// Philox4x32-10 on the host (Salmon et al., SC'11), for the colour draws of
// the random pass order: ten rounds of two 32x32 -> 64-bit products by the
// round multipliers, high halves mixed into the other words and the key.
static void philox_host(uint32_t c[4], uint32_t k0, uint32_t k1)
{
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c[0], p1 = (uint64_t)0xCD9E8D57u * c[2];
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c[1] ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = (uint32_t)p1;
        c[2] = n2;
        c[3] = (uint32_t)p0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// Colour of pass slot `slot` of sweep `sweep` (same rule as the kernels).
static uint32_t slot_colour_host(const DevRng& rng, uint32_t sweep, uint32_t slot, int P)
{
    uint32_t c[4] = {0xFFFFFFFFu, sweep, 0xFFFF0000u | slot, rng.stream};
    philox_host(c, rng.k0, rng.k1);
    return (uint32_t)(((uint64_t)c[0] * (uint64_t)P) >> 32);
}

static int run_segment(tl_chain* c, uint64_t n, void* stream)
{
    const Geom& g = c->g;
    for (uint64_t s = 0; s < n; ++s) {
        const uint32_t sw = (uint32_t)(c->sweep + s);
        for (int p = 0; p < g.passes; ++p) {
            const uint32_t colour = c->random_order ? slot_colour_host(c->rng, sw, (uint32_t)p, g.passes) : (uint32_t)p;
            const int e = launch_pass_global(g, c->rows, colour, (uint32_t)p, sw, c->rng, c->th, c->grange,
                                             c->count_flips ? c->flips_d : nullptr, stream);
            if (e) return fail(TL_ECUDA, "pass kernel: %s", cudaGetErrorString((cudaError_t)e));
        }
        c->launches += (uint64_t)g.passes;
    }
    c->sweep += n;
    return TL_OK;
}

static uint64_t next_sample(const tl_chain* c)
{
    // smallest s > sweep with s >= burn and (s - burn) % stride == 0
    const uint64_t s0 = std::max<uint64_t>(c->burn, c->sweep + 1);
    const uint64_t k = (s0 - c->burn + c->stride - 1) / c->stride;
    return c->burn + k * c->stride;
}

// Number of sample points s <= x (s = sweeps done, s >= burn, stride apart).
static uint64_t samples_upto(const tl_chain* c, uint64_t x)
{
    return x >= c->burn ? (x - c->burn) / c->stride + 1 : 0;
}

static int take_sample(tl_chain* c, void* stream)
{
    const int e = launch_density_accumulate(c->g, c->rows, c->cplanes, stream);
    if (e) return fail(TL_ECUDA, "density kernel: %s", cudaGetErrorString((cudaError_t)e));
    c->samples += 1;
    c->launches += 1;
    return TL_OK;
}

// Dominoes at t = 2^31 take the single-plane updates when they fit.
static bool fast_candidate(const tl_chain* c)
{
    return c->g.lattice == LAT_DOMINO && c->th.kind == THR_SCALAR && c->th.scalar == 0x80000000u &&
           c->npre_req <= 1;
}

// Groups one pass of the single-plane domino update can hold: each of the
// threads / 2 updater threads takes up to two groups (one with 1024 threads).
static int fast_capacity(int threads) { return (threads / 2) * (threads >= 1024 ? 1 : 2); }

// Local rows of stripe [lo, hi) of `C`, with halo h, clamped to the pads.
static void stripe_local(int lo, int hi, int k, int C, int h, int H, int* slo, int* shi)
{
    *slo = k == 0 ? -1 : lo - h;
    *shi = k == C - 1 ? H + 1 : hi + h;
}

// Groups that the register-resident domino kernel holds of each row pair.
struct RegHull {
    std::vector<int2> hull;
    std::vector<long> w, pre;   // their number, prefix sums
};

static RegHull reg_hull(const tl_chain* c)
{
    const Geom& g = c->g;
    const tl_domain& d = c->dom_copy;
    RegHull rh;
    const int H = g.H, W = g.W;
    const int npairs = (H + 1) / 2;
    // extents of the domain's faces per face row
    std::vector<int> fmin(std::max(H - 1, 0), 1 << 30), fmax(std::max(H - 1, 0), -1);
    for (int fy = 0; fy + 1 < H; ++fy) {
        const uint8_t* cv = d.cover.data() + (size_t)fy * (W - 1);
        int a = 0, b = W - 2;
        while (a < W - 1 && !cv[a]) ++a;
        if (a == W - 1) continue;
        while (!cv[b]) --b;
        fmin[fy] = a;
        fmax[fy] = b;
    }
    auto join = [](int2 a, int2 b) {
        if (a.y <= a.x) return b;
        if (b.y <= b.x) return a;
        return make_int2(std::min(a.x, b.x), std::max(a.y, b.y));
    };
    // groups of row y holding sites or edges of domain faces (Hz(x,y) lies
    // between faces (x,y-1) and (x,y), Vt(x,y) between (x-1,y) and (x,y))
    auto row_groups = [&](int y) {
        if (y < 0 || y >= H) return make_int2(0, 0);
        int2 r = d.grange[y];
        for (int fy = y - 1; fy <= y; ++fy) {
            if (fy < 0 || fy + 1 >= H || fmax[fy] < 0) continue;
            r = join(r, make_int2(fmin[fy] >> 8, ((fmax[fy] + 1) >> 8) + 1));
        }
        return r;
    };
    std::vector<int2> hull(npairs);
    std::vector<long> w(npairs), pre(npairs + 1, 0);
    for (int q = 0; q < npairs; ++q) {
        int2 r = join(row_groups(2 * q), row_groups(2 * q + 1));
        if (2 * q + 2 < H) r = join(r, d.grange[2 * q + 2]);
        hull[q] = r.y > r.x ? r : make_int2(0, 0);
        w[q] = hull[q].y - hull[q].x;
        pre[q + 1] = pre[q] + w[q];
    }
    rh.hull = std::move(hull);
    rh.w = std::move(w);
    rh.pre = std::move(pre);
    return rh;
}

// Register-resident domino kernel with `h` passes per exchange: a stripe
// partition of the row pairs that balances the work of a cycle (owned pairs
// every pass, halo pairs while they can still reach the stripe), and buffers.
//
// `max_threads`: threads a stripe may take (512, or fewer to find out whether a
// deeper halo keeps the stripes that small).
static int plan_regdom(tl_chain* c, const RegHull& rh, int h, int max_threads)
{
    const Geom& g = c->g;
    const tl_domain& d = c->dom_copy;
    if (h & 1) {
        c->res_why = "the register-resident kernel needs an even halo";
        return TL_EUNSUPPORTED;
    }
    const int H = g.H;
    const int npairs = (H + 1) / 2;
    const int hp = h / 2;
    const std::vector<int2>& hull = rh.hull;
    const std::vector<long>&w = rh.w, &pre = rh.pre;
    auto items = [&](int a, int b) {
        const int lo = a > 0 ? std::max(0, a - hp) : a, hi = b < npairs ? std::min(npairs, b + hp) : b;
        return pre[hi] - pre[lo];
    };
    if (max_threads < 512) {
        // a quick answer where the stripes cannot be that small: the fewest
        // stripes that hold the groups, halos included
        int stripes = 0;
        for (int a = 0; a < npairs; ++stripes) {
            int b = std::min(npairs, a + hp);
            if (items(a, b) > max_threads || stripes >= c->ctx->sms) return TL_EUNSUPPORTED;
            while (b < npairs && items(a, b + 1) <= max_threads) ++b;
            a = b;
        }
    }
    // Work of one exchange cycle, in warp-passes: threads take the held
    // groups of the stripe's local pairs in order, 32 to a warp, and a warp
    // runs in the passes where any of its pairs is still useful (owned pairs
    // every pass; halo pair k below the stripe in the first h - (2k - 1)
    // passes, above it in the first h - (2k - 2)).  A pass costs at least
    // as much as four warps (one per scheduler: below that it is bound by
    // the latency of one warp's chain, not by issue).  The slowest stripe
    // sets the pace of all, since neighbours wait for each other at every
    // exchange.
    std::vector<int> live(h + 1);
    auto cost = [&](int a, int b) {
        const int plo = a > 0 ? std::max(0, a - hp) : a, phi = b < npairs ? std::min(npairs, b + hp) : b;
        std::fill(live.begin(), live.end(), 0);   // live[p]: warps whose useful passes are the first p
        long t = 0;
        int warp_min = h;   // smallest halo distance in the current warp
        for (int q = plo; q < phi; ++q) {
            const int d = q < a ? 2 * (a - q) - 1 : (q >= b ? 2 * (q - b) : 0);
            for (long i = 0; i < w[q]; ++i) {
                warp_min = std::min(warp_min, d);
                if (++t % 32 == 0) {
                    live[std::max(0, h - warp_min)] += 1;
                    warp_min = h;
                }
            }
        }
        if (t % 32) live[std::max(0, h - warp_min)] += 1;
        long v = 0;
        int active = 0;   // warps running in pass ip, counted from the last pass down
        for (int ip = h; ip >= 1; --ip) {
            active += live[ip];
            v += std::max(4, active);
        }
        return v;
    };
    // greedy stripes under a cost bound; bounds empty if infeasible
    auto partition = [&](long T, std::vector<int>& lo) {
        lo.assign(1, 0);
        int a = 0;
        while (a < npairs) {
            int b = std::min(npairs, a + hp);
            if (cost(a, b) > T || items(a, b) > max_threads) return false;
            while (b < npairs && cost(a, b + 1) <= T && items(a, b + 1) <= max_threads) ++b;
            if (b < npairs && npairs - b < hp) {
                b = npairs - hp;
                if (b - a < hp) return false;
            }
            lo.push_back(b);
            a = b;
            if ((int)lo.size() - 1 > c->ctx->sms) return false;
        }
        return true;
    };
    if (npairs < 2 * hp) {
        c->res_why = "domain too small for register-resident stripes";
        return TL_EUNSUPPORTED;
    }
    std::vector<int> best;
    long tlo = 0, thi = cost(0, npairs) + 1;
    {
        std::vector<int> tmp;
        if (!partition(thi, tmp)) {
            // even one stripe per SM does not fit the thread limit at any bound
            long big = 1L << 60;
            if (!partition(big, tmp)) {
                c->res_why = "a stripe holds more groups than the register-resident kernel takes";
                return TL_EUNSUPPORTED;
            }
            thi = big;
        }
        best = tmp;
    }
    while (tlo + 1 < thi) {
        const long mid = tlo + (thi - tlo) / 2;
        std::vector<int> tmp;
        if (partition(mid, tmp)) {
            thi = mid;
            best = tmp;
        } else {
            tlo = mid;
        }
    }
    const int C = (int)best.size() - 1;
    int max_items = 0, max_npl = 0;
    for (int k = 0; k < C; ++k) {
        max_items = std::max(max_items, (int)items(best[k], best[k + 1]));
        const int plo = k > 0 ? best[k] - hp : best[k], phi = k < C - 1 ? best[k + 1] + hp : best[k + 1];
        max_npl = std::max(max_npl, phi - plo);
    }
    const int threads = std::max(32, (max_items + 31) / 32 * 32);
    size_t smem = regdom_smem_bytes(threads, max_npl);
    // one CTA per SM: ask for more than half of an SM's shared memory
    smem = std::max(smem, (size_t)c->ctx->smem_optin / 2 + 1024);
    if ((long)smem > (long)c->ctx->smem_optin) {
        c->res_why = "register-resident tables do not fit in shared memory";
        return TL_EUNSUPPORTED;
    }
    int bps = 0;
    if (regdom_prepare(threads, smem, c->ctx->smem_optin, &bps) != 0 || bps < 1) {
        c->res_why = "register-resident kernel does not fit on an SM";
        return TL_EUNSUPPORTED;
    }
    if (C > bps * c->ctx->sms) {
        c->res_why = "too many stripes for a cooperative launch";
        return TL_EUNSUPPORTED;
    }
    std::vector<int> rows_lo(C + 1);
    for (int k = 0; k <= C; ++k) rows_lo[k] = 2 * best[k];
    int rc;
    if ((rc = dev_alloc(&c->stripe_d, (size_t)C + 1, "stripes")) ||
        (rc = dev_alloc(&c->hull_d, (size_t)npairs, "pair hulls")) ||
        (rc = dev_alloc(&c->xbuf_d, (size_t)C * 4 * h * g.row_words, "exchange buffer")) ||
        (rc = dev_alloc(&c->status_d, 1 + (size_t)C, "status")))
        return rc;
    CUDA_TRY(cudaMemcpy(c->stripe_d, rows_lo.data(), sizeof(int) * (C + 1), cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(c->hull_d, hull.data(), sizeof(int2) * npairs, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemset(c->xbuf_d, 0, sizeof(unsigned long long) * C * 4 * h * g.row_words));
    CUDA_TRY(cudaMemset(c->status_d, 0, sizeof(int) * (1 + (size_t)C)));
    c->reg.ctas = C;
    c->reg.threads = threads;
    c->reg.halo = h;
    c->reg.smem_bytes = smem;
    c->reg.smem_optin = c->ctx->smem_optin;
    c->reg.stripe_lo = c->stripe_d;
    c->reg.hull = c->hull_d;
    c->reg.xbuf = c->xbuf_d;
    c->reg.status = c->status_d;
    c->reg.loaded = reinterpret_cast<unsigned int*>(c->status_d + 1);
    // the common fields, for reporting and the launch loop
    c->res = ResidentPlan{};
    c->res.ctas = C;
    c->res.threads = threads;
    c->res.halo = h;
    c->res.npre = 1;
    c->res.fast = true;
    c->res.smem_bytes = smem;
    c->res.stripe_lo = c->stripe_d;
    c->res.xbuf = c->xbuf_d;
    c->res.status = c->status_d;
    c->res.loaded = reinterpret_cast<unsigned int*>(c->status_d + 1);
    c->use_reg = true;
    c->res_ready = true;
    // domains of at most 1,024 words of sites: plain runs take the one-block
    // kernel (automatic plans only); hashed, sampled, counted and randomly
    // ordered runs stay here
    c->small_threads = 0;
    if (c->kernel == 0 && c->halo_req == 0) {
        long groups[2] = {0, 0};
        for (int y = 0; y < H; ++y) {
            const int2 r = d.grange[y];
            groups[y & 1] += r.y > r.x ? r.y - std::max(0, r.x - 1) : 0;
        }
        const int st = small_threads(groups[0], groups[1]);
        bool fits = false;
        if (st <= 1024 && small_prepare(small_smem_bytes(g), st, &fits) == 0 && fits) c->small_threads = st;
    }
    return TL_OK;
}

// Device buffers of a resident plan with stripe bounds `lo` (C + 1).
static int alloc_resident(tl_chain* c, const std::vector<int>& lo, int h)
{
    const Geom& g = c->g;
    const int C = (int)lo.size() - 1;
    int rc;
    if ((rc = dev_alloc(&c->stripe_d, (size_t)C + 1, "stripes")) ||
        (rc = dev_alloc(&c->xbuf_d, (size_t)C * 4 * h * g.row_words, "exchange buffer")) ||
        (rc = dev_alloc(&c->status_d, 1 + (size_t)C, "status")))
        return rc;
    CUDA_TRY(cudaMemcpy(c->stripe_d, lo.data(), sizeof(int) * (C + 1), cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemset(c->xbuf_d, 0, sizeof(unsigned long long) * C * 4 * h * g.row_words));
    CUDA_TRY(cudaMemset(c->status_d, 0, sizeof(int) * (1 + (size_t)C)));
    c->res.ctas = C;
    c->res.halo = h;
    c->res.stripe_lo = c->stripe_d;
    c->res.xbuf = c->xbuf_d;
    c->res.status = c->status_d;
    c->res.loaded = reinterpret_cast<unsigned int*>(c->status_d + 1);
    c->res_ready = true;
    return TL_OK;
}

// Row bounds of C stripes of at least h rows each with equal shares of the
// weights (prefix sums `pre`, one more than rows); bounds are rounded up to
// multiples of `step` where that keeps h rows.
static std::vector<int> even_stripes(const std::vector<double>& pre, int C, int h, int step)
{
    const int H = (int)pre.size() - 1;
    std::vector<int> lo(C + 1, 0);
    int y = 0;
    for (int k = 1; k < C; ++k) {
        const double target = pre[H] * k / C;
        const int ymin = lo[k - 1] + h, ymax = H - h * (C - k);
        while (y < H && pre[y] < target) ++y;
        int v = std::min(std::max(y, ymin), ymax);
        if (v % step && v + step - v % step <= ymax) v += step - v % step;
        lo[k] = v;
    }
    lo[C] = H;
    return lo;
}

// Kernels of a thread per 128-site group (tl_resident.cu).  `fast`: dominoes at
// t = 2^31 with the single-plane update, 1024 threads and 6 passes per exchange
// (fastest on the Aztec diamond of order 2048).  Else 512 threads, 8 (dominoes)
// or 6 (lozenges) passes.
static int plan_groups(tl_chain* c, bool fast)
{
    const Geom& g = c->g;
    const tl_domain& d = c->dom_copy;
    const bool half = fast_candidate(c);
    const int h = c->halo_req > 0 ? c->halo_req : half || g.lattice == LAT_LOZENGE ? 6 : 8;
    const int threads = c->threads_req > 0 && g.lattice == LAT_DOMINO ? c->threads_req : half ? 1024 : 512;
    const int planes = c->th.kind == THR_SITE ? 32 : std::max(1, c->th.kmax + 1);
    const int npre = fast ? 1 : c->npre_req > 0 ? c->npre_req : std::min(8, planes);
    std::vector<int> pre(g.H + 1, 0);
    std::vector<double> w(g.H + 1, 0.0);
    for (int y = 0; y < g.H; ++y) {
        // fast: and the group left of them, which writes the word they share
        // (it counts in the weights of both forms: rows of few groups cost
        // shared memory, and the outer stripes have many of them)
        const int2 gr = d.grange[y];
        const int act = gr.y > gr.x ? gr.y - std::max(0, gr.x - 1) : 0;
        pre[y + 1] = pre[y] + (fast || act == 0 ? act : gr.y - gr.x);
        w[y + 1] = w[y] + 0.1 + act;
    }
    auto items_in = [&](int a, int b) {
        a = std::max(a, 0);
        b = std::min(b, g.H);
        return b <= a ? 0 : pre[b] - pre[a];
    };
    const int C = std::min(c->ctx->sms, g.H / h);
    if (C < 2) {
        c->res_why = "domain too small for stripes";
        return TL_EUNSUPPORTED;
    }
    const std::vector<int> lo = even_stripes(w, C, h, 1);
    int max_nloc = 0, cap_items = 0, cap_cycle = 0, max_pass = 0;
    for (int k = 0; k < C; ++k) {
        int slo, shi;
        stripe_local(lo[k], lo[k + 1], k, C, h, g.H, &slo, &shi);
        max_nloc = std::max(max_nloc, shi - slo);
        cap_items = std::max(cap_items, items_in(slo, shi));
        int cyc = 0;
        for (int i = 1; i <= h; ++i) {
            const int n = items_in(k == 0 ? 0 : slo + i, k == C - 1 ? g.H + 1 : shi - (i - 1));
            cyc += n;
            max_pass = std::max(max_pass, n);
        }
        cap_cycle = std::max(cap_cycle, cyc);
    }
    size_t smem = (size_t)max_nloc * g.row_words * 4 + (size_t)npre * cap_cycle * 16 + (size_t)cap_items * 4 +
                  (size_t)(max_nloc + 1) * 4 + 16;
    if (fast) smem += (size_t)cap_items * 8 + 8;
    int bps = 0;
    if ((fast && max_pass > fast_capacity(threads)) || (long)smem > (long)c->ctx->smem_optin ||
        resident_prepare(g, c->th.kind, threads, fast, smem, c->ctx->smem_optin, &bps) != 0 || bps < 1 || C > bps * c->ctx->sms) {
        c->res_why = fast ? "a pass does not fit the single-plane update" : "stripe does not fit in shared memory";
        return TL_EUNSUPPORTED;
    }
    c->res = ResidentPlan{};
    c->res.threads = threads;
    c->res.npre = npre;
    c->res.cap_items = cap_items;
    c->res.cap_cycle = cap_cycle;
    c->res.fast = fast;
    c->res.smem_bytes = smem;
    return alloc_resident(c, lo, h);
}

// Words a stripe of the word kernel holds from which the group form is the
// better one (tl_resident.cu has the figures).  The word kernel's cost goes by
// blocks of four planes, the group form's by planes.
static int group_form_from(const tl_chain* c)
{
    const bool dom = c->g.lattice == LAT_DOMINO;
    if (c->th.kind == THR_SITE && c->g.lattice == LAT_LOZENGE) return 801;
    if (c->th.kind != THR_SCALAR || c->g.lattice == LAT_SIXV) return 1 << 30;
    const int planes = c->th.kmax + 1;
    if (planes > 6) return 1 << 30;
    if (planes == 5 || planes <= (dom ? 2 : 1)) return 513;
    return planes == 6 ? 881 : dom ? 641 : 801;
}

// Words a stripe of the word kernel may hold for it to beat a launch per pass.
// Over 2,048 a thread owns four, with 64 registers and spills.  us a sweep, four
// words / per pass, at the words a stripe: six-vertex 13.4 / 33.9 (2,304) and 13.1 /
// 40.8 (3,456); dominoes with one threshold 8.3 / 12.3 (2,176, 2 to 4 planes), 12.6 /
// 13.2 (3,968), 18.6 / 24.6 (32 planes), but with 5 planes 10.6 / 12.3 (2,176),
// 12.6 / 12.3 (2,432), 14.4 / 12.3 (3,328); with one a site 16.7 / 19.4 (2,176),
// 19.3 / 20.3 (2,432), 16.8 / 14.1 (3,072); lozenges of 2 to 4 planes 14.4 / 18.5
// (2,176), 15.6 / 18.5 (2,432), 21.6 / 18.5 (2,688), of more 17.3 / 18.5, 19.0 / 18.5
// and 24.5 / 18.5, with one a site 25.3 / 19.0 (2,176).
static int word_form_to(const tl_chain* c)
{
    if (c->g.lattice == LAT_SIXV) return 4096;
    const bool dom = c->g.lattice == LAT_DOMINO;
    if (c->th.kind == THR_SITE) return dom ? 2432 : 2048;
    const int planes = c->th.kmax + 1;
    if (dom) return planes == 5 ? 2176 : 4096;
    return planes <= 4 ? 2432 : 2176;
}

// The word kernel: stripes, passes per exchange, threads and words per thread.
//
// A pass is modelled as a fixed chain (update and barrier), a cost per
// 128-site group of the CTA (owned, and half of the halo rows on average: they
// fall out one by one), the exchange spread over the `halo` passes of a cycle
// (none with one stripe), and what the builds of fewer registers cost:
//   T = 1000 + 24 groups + 3500 / halo + 350 (over 512 threads) + 1500 (more
//   than one word a thread) cycles,
// fitted to the passes measured with halos of 2 to 12 on the hexagons 1024^3
// and 301 x 467 x 214, the domain-wall squares 333 and 2048 and the Aztec
// diamond 1333; the minimum is flat.
static int plan_words(tl_chain* c)
{
    const Geom& g = c->g;
    const tl_domain& d = c->dom_copy;
    const bool sixv = g.lattice == LAT_SIXV;
    // groups of every row; six-vertex items are pairs of face rows
    const int step = sixv ? 2 : 1, U = (g.H + step - 1) / step;
    std::vector<int> pre(U + 1, 0);
    std::vector<double> w(g.H + 1, 0.0);
    int maxact = 0;
    const std::vector<int2> unit = unit_groups(d);
    for (int r = 0; r < U; ++r) {
        const int2 gr = unit[r];
        const int act = std::max(0, gr.y - gr.x);
        pre[r + 1] = pre[r] + act;
        maxact = std::max(maxact, act);
        for (int y = step * r; y < std::min(g.H, step * r + step); ++y) w[y + 1] = w[y] + 0.1 + act;
    }
    auto items_in = [&](int slo, int shi) {
        const int a = std::max(slo, 0) / step, b = (std::min(shi, g.H) + step - 1) / step;
        return b <= a ? 0 : pre[b] - pre[a];
    };
    if (c->kernel == 2 && std::min(c->ctx->sms, g.H / (c->halo_req > 0 ? c->halo_req : g.lattice == LAT_LOZENGE ? 6 : 8)) < 2) {
        c->res_why = "domain too small for stripes";
        return TL_EUNSUPPORTED;
    }
    struct Cand {
        double t;
        int h, C;
    };
    auto model = [](double own, double halo, int h) {
        const double lanes = 4 * (own + 2 * halo);
        return 1000 + 24 * (own + halo) + (h ? 3500.0 / h : 0) + (lanes > 512 ? 350 : 0) + (lanes > 1024 ? 1500 : 0);
    };
    std::vector<Cand> cand;
    // whole sweeps per exchange (the pass loop is then unrolled)
    const int hs[3][4] = {{4, 6, 8, 12}, {3, 6, 9, 12}, {4, 8, 12, 16}};
    for (int hi = 0; hi < 4; ++hi) {
        const int h = c->halo_req > 0 ? c->halo_req : hs[g.lattice][hi];
        const int cmax = std::min(c->ctx->sms, g.H / h);
        for (int C = 2; C <= cmax; C = C < 16 ? C + 1 : (C < cmax && C + C / 8 > cmax ? cmax : C + C / 8))
            cand.push_back(Cand{model((double)pre[U] / C, (double)h * maxact / step, h), h, C});
        if (c->halo_req > 0) break;
    }
    cand.push_back(Cand{model(pre[U], 0, 0), c->halo_req > 0 ? c->halo_req : 60, 1});
    std::stable_sort(cand.begin(), cand.end(), [](const Cand& a, const Cand& b) { return a.t < b.t; });
    c->res_why = "stripe does not fit in shared memory";
    bool groups_tried = false;
    for (const Cand& cd : cand) {
        const int h = cd.h, C = cd.C;
        const std::vector<int> lo = even_stripes(w, C, h, step);
        int max_nloc = 0, max_own = 0, items = 0;
        for (int k = 0; k < C; ++k) {
            int slo, shi;
            stripe_local(lo[k], lo[k + 1], k, C, h, g.H, &slo, &shi);
            max_nloc = std::max(max_nloc, shi - slo);
            max_own = std::max(max_own, lo[k + 1] - lo[k]);
            items = std::max(items, items_in(slo, shi));
        }
        const int lanes = std::max(32, 4 * items);
        const size_t smem = words_smem_bytes(g, max_nloc);
        if (smem > (size_t)c->ctx->smem_optin || lanes > 4096) continue;
        if (!groups_tried && lanes >= group_form_from(c)) {
            groups_tried = true;
            if (plan_groups(c, false) == TL_OK) return TL_OK;
            free_resident(c);
        }
        if (c->kernel != 2 && lanes > word_form_to(c)) {
            c->res_why = "a launch per pass is the faster one";
            continue;
        }
        // `threads` asks for at most that many; results never depend on it
        const int cap = c->threads_req == 512 && lanes <= 2048 ? 512 : 1024;
        int slots = 1;
        while (slots * cap < lanes) slots *= 2;
        const int threads = ((lanes + slots - 1) / slots + 31) / 32 * 32;
        int bps = 0;
        if (words_prepare(g, c->th, threads, slots, smem, &bps) != 0 || bps < 1 || C > bps * c->ctx->sms) {
            c->res_why = "resident kernel does not fit on an SM";
            continue;
        }
        c->res = ResidentPlan{};
        c->res.threads = threads;
        c->res.slots = slots;
        c->res.max_words = (int)std::min<int64_t>(max_own * g.row_words, 1 << 30);
        // six-vertex words carry 8 or 4 planes by their build
        c->res.npre = sixv ? (slots <= 2 ? 8 : 4)
                           : c->npre_req > 0 ? c->npre_req
                                             : (c->th.kind == THR_SCALAR ? std::max(1, std::min(8, c->th.kmax + 1)) : 8);
        c->res.smem_bytes = smem;
        return alloc_resident(c, lo, h);
    }
    // stripes of more words than the word kernel takes
    if (c->th.kind == THR_SCALAR && !sixv && !groups_tried) return plan_groups(c, false);
    return TL_EUNSUPPORTED;
}

static void free_resident(tl_chain* c)
{
    cudaFree(c->stripe_d);
    cudaFree(c->hull_d);
    cudaFree(c->xbuf_d);
    cudaFree(c->status_d);
    c->stripe_d = nullptr;
    c->hull_d = nullptr;
    c->xbuf_d = nullptr;
    c->status_d = nullptr;
}

// Plan of the chain's resident kernel: registers for dominoes at t = 2^31
// where they fit, else shared memory.
static int plan_resident(tl_chain* c)
{
    if (c->kernel != 2 && fast_candidate(c) && c->g.Kg <= 4096) {
        // Passes per exchange: 8, or the deepest halo with which no stripe
        // needs more than four warps.  Up to one warp per scheduler a pass
        // costs the latency of one warp's chain, so halo rows are free and
        // every exchange (about 3,500 cycles) counts; beyond, halo rows cost
        // more than the exchanges they save.  us a sweep at 8 -> the chosen
        // halo: Aztec 140 0.96 -> 0.73 (24), 300 1.01 -> 0.76 (24), 450 1.02
        // -> 0.79 (20), 700 1.05 -> 0.91 (12), 1000 1.04 -> 0.96 (10); at 1400
        // and 2048 8 stays (1.15 and 1.41; 1.23 and 1.80 with 10).
        int rc = TL_EUNSUPPORTED;
        const RegHull rh = reg_hull(c);
        if (c->halo_req <= 0)
            for (int h : {24, 20, 16, 12, 10}) {
                rc = plan_regdom(c, rh, h, 128);
                if (rc == TL_OK) return TL_OK;
                free_resident(c);
            }
        rc = plan_regdom(c, rh, c->halo_req > 0 ? c->halo_req : 8, 512);
        if (rc == TL_OK) return TL_OK;
        if (c->kernel == 3) return rc;
        free_resident(c);
    }
    if (c->kernel == 3) {
        c->res_why = "the register-resident kernel covers dominoes at t = 2^31 only";
        return TL_EUNSUPPORTED;
    }
    if (fast_candidate(c)) {
        if (plan_groups(c, true) == TL_OK) return TL_OK;
        free_resident(c);
    }
    return plan_words(c);
}

static bool want_resident(tl_chain* c)
{
    if (c->kernel == 1) return false;
    if (!c->res_ready && !c->res_failed) {
        if (plan_resident(c) != TL_OK) c->res_failed = true;
    }
    return c->res_ready;
}

// Pass slots of one resident launch at most: exchange tags carry 16 bits of
// cycle, so a launch runs at most 60,000 cycles, each of at most 64 passes
// (the largest halo a plan takes).
constexpr size_t kMaxLaunchSlots = (size_t)60000 * 64;

// Whether a plain run of the (planned) chain takes the one-block kernel.
static bool small_run(const tl_chain* c)
{
    return c->use_reg && c->small_threads > 0 && !c->density_on && !c->random_order && !c->count_flips;
}

// Sweeps of one resident launch at most: exchange tags carry 16 bits of cycle
// and 16 bits of launch epoch, and a launch ends in a time that a user can wait
// for (well under a second).
static uint64_t max_launch_sweeps(const tl_chain* c)
{
    return std::max<uint64_t>(1, 60000ull * c->res.halo / c->g.passes);
}

// Resident launches over [c->sweep, c->sweep + k), at most spl sweeps each.
static int run_resident(tl_chain* c, uint64_t k, unsigned long long* ring, void* stream)
{
    const uint64_t max_sweeps = max_launch_sweeps(c);
    uint64_t done = 0;
    while (done < k) {
        uint64_t n = c->spl > 0 ? std::min<uint64_t>((uint64_t)c->spl, k - done) : k - done;
        n = std::min(n, max_sweeps);
        const bool dens = c->density_on;
        if (((c->epoch + 1) & 0xFFFFu) == 0) {
            const size_t nx = (size_t)c->res.ctas * 4 * c->res.halo * c->g.row_words;
            CUDA_TRY(cudaMemsetAsync(c->xbuf_d, 0, nx * sizeof(unsigned long long), SS(stream)));
        }
        if (c->random_order) {
            const size_t need = (size_t)n * c->g.passes;
            if (need > c->colours_cap) {
                CUDA_TRY(cudaStreamSynchronize(SS(stream)));
                cudaFree(c->colours);
                c->colours = nullptr;
                c->colours_cap = 0;
                TL_TRY(dev_alloc(&c->colours, need, "pass colours"));
                c->colours_cap = need;
            }
            const int ec = launch_slot_colours(c->colours, (uint32_t)c->sweep, (uint32_t)n, c->g.passes, c->rng, stream);
            if (ec) return fail(TL_ECUDA, "colour kernel: %s", cudaGetErrorString((cudaError_t)ec));
            c->launches += 1;
        }
        const bool small = small_run(c) && !ring;
        if (c->use_reg && !small && (uint64_t)n * c->g.passes > (uint64_t)c->reg.halo) {
            // the register kernel's exchange tags count cycles within one
            // launch: its buffers start every launch cleared
            CUDA_TRY(cudaMemsetAsync(c->xbuf_d, 0,
                                     (size_t)c->reg.ctas * 4 * c->reg.halo * c->g.row_words * sizeof(unsigned long long),
                                     SS(stream)));
        }
        const int e =
            small
                ? launch_small(c->g, c->rows, nullptr, c->small_threads, (uint32_t)c->sweep, (uint32_t)n, c->rng,
                               c->grange, stream)
            : c->use_reg
                ? launch_regdom(c->g, c->rows, c->reg, (uint32_t)c->sweep, (uint32_t)n, c->rng, ++c->epoch,
                                ring ? ring + done : nullptr, dens ? c->cplanes : nullptr, c->burn,
                                dens ? c->stride : 0, c->random_order ? c->colours : nullptr,
                                c->count_flips ? c->flips_d : nullptr, stream)
            : c->res.slots == 0
                ? launch_resident(c->g, c->rows, c->res, (uint32_t)c->sweep, (uint32_t)n, c->rng, c->th, c->grange,
                                  ++c->epoch, ring ? ring + done : nullptr, dens ? c->cplanes : nullptr, c->burn,
                                  dens ? c->stride : 0, c->random_order ? c->colours : nullptr,
                                  c->count_flips ? c->flips_d : nullptr, stream)
                : launch_words(c->g, c->rows, c->res, (uint32_t)c->sweep, (uint32_t)n, c->rng, c->th, c->grange,
                               ++c->epoch, ring ? ring + done : nullptr, dens ? c->cplanes : nullptr, c->burn,
                               dens ? c->stride : 0, c->random_order ? c->colours : nullptr,
                               c->count_flips ? c->flips_d : nullptr, stream);
        if (e) return fail(TL_ECUDA, "resident kernel: %s", cudaGetErrorString((cudaError_t)e));
        if (dens) c->samples += samples_upto(c, c->sweep + n) - samples_upto(c, c->sweep);
        c->sweep += n;
        c->launches += 1;
        done += n;
    }
    return TL_OK;
}

TL_API const char* tl_chain_kernel(tl_chain* c)
{
    if (!c || cudaSetDevice(c->ctx->device) != cudaSuccess) return nullptr;
    if (!want_resident(c)) return "pass_global_kernel";
    if (small_run(c)) return "small_kernel";
    return c->use_reg ? "regdom_kernel" : c->res.slots == 0 ? "resident_kernel" : "words_kernel";
}

static int zero_counts_if_needed(tl_chain* c, void* stream)
{
    if (c->counts_dirty) {
        const size_t n = (size_t)32 * c->g.H * c->g.row_words;
        CUDA_TRY(cudaMemsetAsync(c->cplanes, 0, n * sizeof(uint32_t), SS(stream)));
        c->counts_dirty = false;
    }
    return TL_OK;
}

static bool is_capturing(void* stream)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(SS(stream), &st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return st != cudaStreamCaptureStatusNone;
}

// Planning allocates and copies, which a capture does not take: a chain not
// planned yet is captured as one launch per pass.
static bool want_resident_on(tl_chain* c, void* stream)
{
    const bool planned = c->kernel == 1 || c->res_ready || c->res_failed;
    return (planned || !is_capturing(stream)) && want_resident(c);
}

TL_API int tl_run_sweeps(tl_chain* c, uint64_t k, void* stream)
{
    NvtxRange nvtx_("tl_run_sweeps");
    if (!c) return fail(TL_EINVAL, "tl_run_sweeps: NULL chain");
    if (c->sweep + k > 0x100000000ull) return fail(TL_EINVAL, "tl_run_sweeps: sweep index beyond 2^32 - 1");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(zero_counts_if_needed(c, stream));
    if (k == 0) return TL_OK;
    if (want_resident_on(c, stream)) return run_resident(c, k, nullptr, stream);
    if (c->kernel == 2) return fail(TL_EUNSUPPORTED, "resident kernel unavailable: %s", c->res_why.c_str());
    const uint64_t end = c->sweep + k;
    while (c->sweep < end) {
        uint64_t stop = end;
        bool sample = false;
        if (c->density_on) {
            const uint64_t ns = next_sample(c);
            if (ns <= end) {
                stop = ns;
                sample = true;
            }
        }
        TL_TRY(run_segment(c, stop - c->sweep, stream));
        if (sample) TL_TRY(take_sample(c, stream));
    }
    return TL_OK;
}

TL_API int tl_chain_sync(tl_chain* c, void* stream)
{
    if (!c) return fail(TL_EINVAL, "tl_chain_sync: NULL chain");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    if (c->status_d) {
        int st = 0;
        CUDA_TRY(cudaMemcpy(&st, c->status_d, sizeof(int), cudaMemcpyDeviceToHost));
        if (st) {
            CUDA_TRY(cudaMemset(c->status_d, 0, sizeof(int)));
            return fail(TL_ETIMEOUT, "a bounded wait in the resident kernel gave up; chain state undefined");
        }
    }
    return TL_OK;
}

static int batch_raise_status(tl_batch* b);

TL_API int tl_debug_build(void)
{
#ifdef TL_DEBUG
    return 1;
#else
    return 0;
#endif
}

TL_API int tl_debug_checks(int clear, uint64_t* failures, int* first_id, int64_t* index, int64_t* bound)
{
#ifdef TL_DEBUG
    CUDA_TRY(cudaDeviceSynchronize());
    int (*const fetch[])(unsigned long long*, bool) = {dbg_fetch_kernels, dbg_fetch_regdom, dbg_fetch_small, dbg_fetch_resident,
                                                       dbg_fetch_words_domino, dbg_fetch_words_lozenge, dbg_fetch_words_sixv,
                                                       dbg_fetch_batch, dbg_fetch_shuffle};
    uint64_t n = 0;
    int id = 0;
    int64_t ix = 0, bd = 0;
    for (auto f : fetch) {
        unsigned long long w[4] = {0, 0, 0, 0};
        const int e = f(w, clear != 0);
        if (e) return fail(TL_ECUDA, "tl_debug_checks: %s", cudaGetErrorString((cudaError_t)e));
        if (w[0] && !n) {
            id = (int)w[1];
            ix = (int64_t)w[2];
            bd = (int64_t)w[3];
        }
        n += w[0];
    }
    if (failures) *failures = n;
    if (first_id) *first_id = id;
    if (index) *index = ix;
    if (bound) *bound = bd;
    return TL_OK;
#else
    (void)clear;
    (void)failures;
    (void)first_id;
    (void)index;
    (void)bound;
    return fail(TL_EUNSUPPORTED, "tl_debug_checks: not the checked build (build with --debug, load with TL_DEBUG=1)");
#endif
}

TL_API int tl_debug_selftest(void)
{
#ifdef TL_DEBUG
    const int e = dbg_selftest();
    if (e) return fail(TL_ECUDA, "tl_debug_selftest: %s", cudaGetErrorString((cudaError_t)e));
    return TL_OK;
#else
    return fail(TL_EUNSUPPORTED, "tl_debug_selftest: not the checked build");
#endif
}

TL_API int tl_debug_raise_status(tl_chain* c, tl_batch* b)
{
    if (!c && !b) return fail(TL_EINVAL, "tl_debug_raise_status: NULL argument");
    const int one = 1;
    if (c) {
        CUDA_TRY(cudaSetDevice(c->ctx->device));
        if (!want_resident(c) || !c->status_d)
            return fail(TL_EUNSUPPORTED, "tl_debug_raise_status: the chain has no resident kernel");
        CUDA_TRY(cudaMemcpy(c->status_d, &one, sizeof(int), cudaMemcpyHostToDevice));
    }
    if (b) TL_TRY(batch_raise_status(b));
    return TL_OK;
}

TL_API int tl_run_sweeps_hashed(tl_chain* c, uint64_t k, uint64_t* ring, void* stream)
{
    NvtxRange nvtx_("tl_run_sweeps_hashed");
    if (!c || (!ring && k)) return fail(TL_EINVAL, "tl_run_sweeps_hashed: NULL argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    if (k) TL_TRY(require_local(ring, c->ctx->device, "tl_run_sweeps_hashed"));
    const bool dev = k ? is_device_ptr(ring) : true;
    uint64_t* dring = reinterpret_cast<uint64_t*>(ring);
    uint64_t* tmp = nullptr;
    if (!dev && k) {
        TL_TRY(dev_alloc(&tmp, (size_t)k, "hash ring"));
        dring = tmp;
    }
    int rc = TL_OK;
    if (k && want_resident_on(c, stream)) {
        rc = zero_counts_if_needed(c, stream);
        cudaError_t e = cudaMemsetAsync(dring, 0, k * 8, SS(stream));
        if (rc == TL_OK && e != cudaSuccess) rc = fail(TL_ECUDA, "hash ring: %s", cudaGetErrorString(e));
        // A stripe hashes its own words.  The outer stripes of large diamonds
        // hold many rows of few, full words each, a lane's work and not a warp's:
        // there a launch per sweep and a hash over the whole chip are faster (us a
        // sweep: Aztec 1200 with a threshold a site 39.9 -> 28.2, 1600 42.3 -> 32.5;
        // 900, 6,700 words a stripe, 18.5 as it is).  Rows of lozenges and faces are
        // denser, and their stripes hash themselves faster (hexagon 1100 27.1, 34.7
        // apart).
        if (!c->use_reg && c->res.slots > 0 && c->g.lattice == LAT_DOMINO && c->res.max_words > 9600) {
            for (uint64_t i = 0; i < k && rc == TL_OK; ++i) {
                rc = run_resident(c, 1, nullptr, stream);
                if (rc != TL_OK) break;
                const int eh = launch_hash(c->g, c->rows, reinterpret_cast<unsigned long long*>(dring + i), stream);
                c->launches += 1;
                if (eh) rc = fail(TL_ECUDA, "hash kernel: %s", cudaGetErrorString((cudaError_t)eh));
            }
        } else if (rc == TL_OK) {
            rc = run_resident(c, k, reinterpret_cast<unsigned long long*>(dring), stream);
        }
        k = rc == TL_OK ? k : 0;
        goto copy_back;
    }
    for (uint64_t i = 0; i < k && rc == TL_OK; ++i) {
        rc = tl_run_sweeps(c, 1, stream);
        if (rc == TL_OK) {
            const int e = launch_hash(c->g, c->rows, reinterpret_cast<unsigned long long*>(dring + i), stream);
            c->launches += 1;
            if (e) rc = fail(TL_ECUDA, "hash kernel: %s", cudaGetErrorString((cudaError_t)e));
        }
    }
copy_back:
    if (tmp) {
        if (rc == TL_OK) {
            cudaError_t e = cudaMemcpyAsync(ring, tmp, k * 8, cudaMemcpyDeviceToHost, SS(stream));
            if (e == cudaSuccess) e = cudaStreamSynchronize(SS(stream));
            if (e != cudaSuccess) rc = fail(TL_ECUDA, "hash ring copy: %s", cudaGetErrorString(e));
        } else {
            cudaStreamSynchronize(SS(stream));
        }
        cudaFree(tmp);
    }
    return rc;
}

TL_API int tl_read_state(tl_chain* c, uint8_t* canon, size_t cap, void* stream)
{
    if (!c || !canon) return fail(TL_EINVAL, "tl_read_state: NULL argument");
    const size_t n = (size_t)c->g.ntype * c->g.W * c->g.H;
    if (cap < n) return fail(TL_EINVAL, "tl_read_state: cap %zu < %zu", cap, n);
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(require_local(canon, c->ctx->device, "tl_read_state"));
    if (is_device_ptr(canon)) {
        CUDA_TRY(launch_unpack(c->g, c->rows, canon, stream));
        c->launches += 1;
        return TL_OK;
    }
    CUDA_TRY(launch_unpack(c->g, c->rows, c->canon, stream));
    c->launches += 1;
    CUDA_TRY(cudaMemcpyAsync(canon, c->canon, n, cudaMemcpyDeviceToHost, SS(stream)));
    CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    return TL_OK;
}

// Checks the canonical state `dcanon` (device memory) against the chain's
// domain on the device; the same checks, and an error naming the first
// failure, as the host validation.
static int validate_device(tl_chain* c, const uint8_t* dcanon, void* stream)
{
    const tl_domain& d = c->dom_copy;
    const Geom& g = c->g;
    if (!c->vaux_d) {
        std::vector<uint8_t> aux;
        if (g.lattice == LAT_SIXV) {
            const int N = g.N;
            aux.resize((size_t)4 * N);
            for (int k = 1; k <= N; ++k) {
                aux[k - 1] = d.init[(size_t)k * g.W];
                aux[N + k - 1] = d.init[(size_t)k * g.W + N];
                aux[2 * N + k - 1] = d.init[(size_t)g.W * g.H + k];
                aux[3 * N + k - 1] = d.init[(size_t)g.W * g.H + (size_t)N * g.W + k];
            }
        } else {
            aux = d.cover;
        }
        TL_TRY(dev_alloc(&c->vaux_d, aux.size(), "validation data"));
        CUDA_TRY(cudaMemcpy(c->vaux_d, aux.data(), aux.size(), cudaMemcpyHostToDevice));
    }
    if (!c->vfirst_d) TL_TRY(dev_alloc(&c->vfirst_d, 1, "validation result"));
    const int e = launch_validate(g, dcanon, c->vaux_d, c->vfirst_d, stream);
    if (e) return fail(TL_ECUDA, "validation kernels: %s", cudaGetErrorString((cudaError_t)e));
    c->launches += 2;
    unsigned long long first = 0;
    CUDA_TRY(cudaMemcpyAsync(&first, c->vfirst_d, sizeof(first), cudaMemcpyDeviceToHost, SS(stream)));
    CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    if (first == ~0ull) return TL_OK;
    const int kind = (int)(first >> 48);
    const long long pos = (long long)(first & ((1ull << 48) - 1));
    switch (kind) {
    case 1: return fail(TL_EINVAL, "state byte %lld is not 0 or 1", pos);
    case 2:
    case 3: return fail(TL_EINVAL, "domino: edge outside the box set");
    case 4:
        return fail(TL_EINVAL, "domino: face (%lld,%lld) not covered once", pos % (g.W - 1), pos / (g.W - 1));
    case 5:
        return fail(TL_EINVAL, "lozenge: triangles at (%lld,%lld) not covered once", pos % (g.W + 1) - 1,
                    pos / (g.W + 1) - 1);
    case 6: return fail(TL_EINVAL, "six-vertex: bit set off the lattice at (%lld,%lld)", pos % g.W, pos / g.W);
    case 7: return fail(TL_EINVAL, "six-vertex: external edges differ from the boundary");
    default: return fail(TL_EINVAL, "six-vertex: ice rule fails at (%lld,%lld)", pos % g.W, pos / g.W);
    }
}

TL_API int tl_write_state(tl_chain* c, const uint8_t* canon, size_t n, void* stream)
{
    if (!c || !canon) return fail(TL_EINVAL, "tl_write_state: NULL argument");
    const size_t want = (size_t)c->g.ntype * c->g.W * c->g.H;
    if (n != want) return fail(TL_EINVAL, "tl_write_state: n %zu != %zu", n, want);
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(require_local(canon, c->ctx->device, "tl_write_state"));
    const bool dev = is_device_ptr(canon);
    if (dev) {
        // checked where it is, then copied and packed
        TL_TRY(validate_device(c, canon, stream));
        return upload_state(c, canon, true, stream);
    }
    // host bytes: copied into the chain's unpacked scratch, checked there on
    // the device, packed only if valid (the chain's state is untouched
    // otherwise)
    CUDA_TRY(cudaMemcpyAsync(c->canon, canon, n, cudaMemcpyHostToDevice, SS(stream)));
    TL_TRY(validate_device(c, c->canon, stream));
    CUDA_TRY(launch_pack(c->g, c->canon, c->rows, stream));
    c->launches += 1;
    return TL_OK;
}

TL_API int tl_state_hash(tl_chain* c, uint64_t* out, void* stream)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_state_hash: NULL argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(require_local(out, c->ctx->device, "tl_state_hash"));
    if (is_device_ptr(out)) {
        CUDA_TRY(launch_hash(c->g, c->rows, reinterpret_cast<unsigned long long*>(out), stream));
        c->launches += 1;
        return TL_OK;
    }
    CUDA_TRY(launch_hash(c->g, c->rows, c->hash, stream));
    c->launches += 1;
    CUDA_TRY(cudaMemcpyAsync(out, c->hash, 8, cudaMemcpyDeviceToHost, SS(stream)));
    CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    return TL_OK;
}

// Stripes of a resident shuffling launch whose last step is K: bounds of the
// rows n - K .. n + K that balance the work of that step, or an empty vector
// if they do not fit the SMs' shared memory.
//
// A step costs a stripe about 4 warp instructions per word it looks at and
// 2.4 per block it fills (a quarter of the blocks inside the inscribed
// circle).  The stripe through the middle is the slowest at every step, so
// balancing the last step balances them all.  Stripes are added while they
// hold at least `kStripeWork` of it: below that a step is bound by its latency,
// and a seam only adds exchanges.
static std::vector<int> shuffle_stripes(const tl_ctx* ctx, int n, int K, int Kw, int h, int threads, size_t* smem)
{
    const int H = 2 * K + 1;
    const int cap = (int)(((size_t)ctx->smem_optin - shuffle_static_smem(threads)) / shuffle_smem_bytes(1, Kw));   // local rows that fit
    std::vector<double> pre(H + 1, 0.0);
    for (int y = 0; y < H; ++y) {
        const double d = std::abs(y - K), chord = 0.5 * K * K - d * d;
        pre[y + 1] = pre[y] + 4.0 * ((K - d) / 32 + 1) + 0.6 * std::sqrt(std::max(0.0, chord));
    }
    const double kStripeWork = 1000.0;
    const int want = std::min(ctx->sms, std::max(1, (int)(pre[H] / kStripeWork)));
    auto partition = [&](double T, std::vector<int>& lo) {
        lo.assign(1, 0);
        for (int a = 0; a < H;) {
            int b = std::min(H, a + h);
            auto local = [&](int e) { return (e < H ? e + h : H) - (a > 0 ? a - h : 0); };
            if (local(b) > cap) return false;
            while (b < H && pre[b + 1] - pre[a] <= T && local(b + 1) <= cap) ++b;
            if (b < H && H - b < h) {
                b = H - h;
                if (b - a < h) return false;
            }
            lo.push_back(b);
            a = b;
            if ((int)lo.size() - 1 > want) return false;
        }
        return true;
    };
    std::vector<int> best, tmp;
    if (cap < 1 || !partition(pre[H] + 1, best)) return {};
    double tlo = 0, thi = pre[H] + 1;
    for (int it = 0; it < 40; ++it) {
        const double mid = 0.5 * (tlo + thi);
        if (partition(mid, tmp)) {
            thi = mid;
            best = tmp;
        } else {
            tlo = mid;
        }
    }
    const int C = (int)best.size() - 1;
    int nloc = 0;
    for (int k = 0; k < C; ++k)
        nloc = std::max(nloc, (k < C - 1 ? best[k + 1] + h : H) - (k > 0 ? best[k] - h : 0));
    *smem = shuffle_smem_bytes(nloc, Kw);
    for (int& y : best) y += n - K;
    return best;
}

// Buffers and stripes of order n (rebuilt when n changes).
static int shuffle_prepare(tl_ctx* ctx, int n)
{
    ShuffleCache& sc = ctx->shuffle;
    if (sc.n == n) return TL_OK;
    CUDA_TRY(cudaDeviceSynchronize());
    sc.release();
    sc.g = make_geom(LAT_DOMINO, 2 * n + 1, 2 * n + 1, 0);
    const int h = 4;
    // launches: the last covers steps up to n; each one before it ends where
    // the work of a step is half as much (the middle stripe of a launch's
    // partition does up to its last step's share of it all the time)
    std::vector<int> last(1, n);
    while (last.back() > 560) last.push_back(last.back() * 5 / 7);
    std::reverse(last.begin(), last.end());
    std::vector<int> stripes;
    std::vector<size_t> first;
    for (int K : last) {
        ShufflePlan sp{};
        // more warps hide the lists and reads of a step's second and third
        // turn behind the draws of others once a stripe's step takes that many
        // (order 2048: 7.2 -> 6.7 ms; order 1024, one turn: 1.91 -> 2.04)
        sp.threads = K > 1100 ? 768 : 512;
        const std::vector<int> lo = shuffle_stripes(ctx, n, K, sc.g.K, h, sp.threads, &sp.smem_bytes);
        if (lo.empty()) break;
        int bps = 0;
        if (shuffle_prepare_kernel(sp.threads, sp.smem_bytes, &bps) != 0 || (int)lo.size() - 1 > bps * ctx->sms) break;
        sp.last = K;
        sp.ctas = (int)lo.size() - 1;
        sp.halo = h;
        sc.xbuf_words = std::max(sc.xbuf_words, (size_t)sp.ctas * 4 * h * (size_t)sc.g.row_words);
        first.push_back(stripes.size());
        stripes.insert(stripes.end(), lo.begin(), lo.end());
        sc.seg.push_back(sp);
    }
    const bool fits = sc.seg.size() == last.size();
    int rc;
    if ((rc = dev_alloc(&sc.rows, (size_t)sc.g.total_words, "shuffle rows")) ||
        (rc = dev_alloc(&sc.status, 1, "status"))) {
        sc.release();
        return rc;
    }
    if (!fits) {
        sc.seg.clear();
        rc = dev_alloc(&sc.alt, (size_t)sc.g.total_words, "shuffle rows");
    } else {
        if ((rc = dev_alloc(&sc.stripe, stripes.size(), "stripes")) == TL_OK)
            rc = dev_alloc(&sc.xbuf, sc.xbuf_words, "exchange buffer");
        if (rc == TL_OK &&
            cudaMemcpy(sc.stripe, stripes.data(), sizeof(int) * stripes.size(), cudaMemcpyHostToDevice) != cudaSuccess)
            rc = fail(TL_ECUDA, "tl_aztec_shuffle: stripes");
        for (size_t i = 0; i < sc.seg.size(); ++i) {
            sc.seg[i].stripe_lo = sc.stripe + first[i];
            sc.seg[i].xbuf = sc.xbuf;
            sc.seg[i].status = sc.status;
        }
    }
    if (rc == TL_OK && cudaMemset(sc.status, 0, sizeof(int)) != cudaSuccess) rc = fail(TL_ECUDA, "tl_aztec_shuffle: memset");
    if (rc != TL_OK) {
        sc.release();
        return rc;
    }
    sc.n = n;
    return TL_OK;
}

TL_API int tl_aztec_shuffle(tl_ctx* ctx, int n, uint64_t seed, uint32_t stream_id, uint8_t* canon, size_t cap,
                            void* stream)
{
    NvtxRange nvtx_("tl_aztec_shuffle");
    if (!ctx || !canon || n < 1 || n > 32767) return fail(TL_EINVAL, "tl_aztec_shuffle: bad argument");
    const size_t W = 2 * (size_t)n + 1, ncanon = 2 * W * W;
    if (cap < ncanon) return fail(TL_EINVAL, "tl_aztec_shuffle: cap %zu < %zu", cap, ncanon);
    CUDA_TRY(cudaSetDevice(ctx->device));
    TL_TRY(require_local(canon, ctx->device, "tl_aztec_shuffle"));
    std::lock_guard<std::mutex> lock(ctx->shuffle_mu);
    TL_TRY(shuffle_prepare(ctx, n));
    ShuffleCache& sc = ctx->shuffle;
    const DevRng rng{(uint32_t)seed, (uint32_t)(seed >> 32), stream_id};
    const bool dev = is_device_ptr(canon);
    if (!dev && !sc.canon) TL_TRY(dev_alloc(&sc.canon, ncanon, "shuffle output"));
    int hstatus = 0;
    cudaError_t e =
        (cudaError_t)(!sc.seg.empty()
                          ? launch_shuffle(sc.seg.data(), (int)sc.seg.size(), n, sc.g.K, (size_t)sc.g.total_words,
                                           sc.xbuf_words, sc.rows, rng, stream)
                          : launch_shuffle_global(n, sc.g.K, (size_t)sc.g.total_words, sc.rows, sc.alt, rng, stream));
    if (e == cudaSuccess)
        e = (cudaError_t)launch_unpack_diamond(sc.g, sc.rows, dev ? canon : sc.canon, n, sc.status, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hstatus, sc.status, sizeof(int), cudaMemcpyDeviceToHost, SS(stream));
    if (e == cudaSuccess && !dev) e = cudaMemcpyAsync(canon, sc.canon, ncanon, cudaMemcpyDeviceToHost, SS(stream));
    if (e == cudaSuccess) e = cudaStreamSynchronize(SS(stream));
    if (e != cudaSuccess) return fail(TL_ECUDA, "tl_aztec_shuffle: %s", cudaGetErrorString(e));
    if (hstatus) {
        CUDA_TRY(cudaMemset(sc.status, 0, sizeof(int)));
        if (hstatus == 2) return fail(TL_ECUDA, "tl_aztec_shuffle: the result is not a tiling");
        return fail(TL_ETIMEOUT, "tl_aztec_shuffle: a bounded wait gave up");
    }
    return TL_OK;
}

TL_API int tl_chain_set_order(tl_chain* c, int order)
{
    if (!c || (order != TL_ORDER_FIXED && order != TL_ORDER_RANDOM)) return fail(TL_EINVAL, "tl_chain_set_order: bad argument");
    // the colours of one resident launch's pass slots: at most 60,000
    // exchange cycles of at most 64 passes per launch, sized here once so
    // that tl_run_sweeps only enqueues
    if (order == TL_ORDER_RANDOM && c->colours_cap < kMaxLaunchSlots) {
        CUDA_TRY(cudaSetDevice(c->ctx->device));
        CUDA_TRY(cudaDeviceSynchronize());
        cudaFree(c->colours);
        c->colours = nullptr;
        c->colours_cap = 0;
        TL_TRY(dev_alloc(&c->colours, kMaxLaunchSlots, "pass colours"));
        c->colours_cap = kMaxLaunchSlots;
    }
    c->random_order = order == TL_ORDER_RANDOM;
    return TL_OK;
}

TL_API int tl_chain_count_flips(tl_chain* c, int on)
{
    if (!c) return fail(TL_EINVAL, "tl_chain_count_flips: NULL chain");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    if (on && !c->flips_d) TL_TRY(dev_alloc(&c->flips_d, 1, "flip counter"));
    if (on) {   // starting resets the count; stopping keeps it readable
        CUDA_TRY(cudaDeviceSynchronize());
        CUDA_TRY(cudaMemset(c->flips_d, 0, sizeof(unsigned long long)));
    }
    c->count_flips = on != 0;
    return TL_OK;
}

TL_API int tl_chain_flips(tl_chain* c, uint64_t* out)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_chain_flips: NULL argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    if (!c->flips_d) {
        *out = 0;
        return TL_OK;
    }
    CUDA_TRY(cudaDeviceSynchronize());
    unsigned long long v = 0;
    CUDA_TRY(cudaMemcpy(&v, c->flips_d, sizeof(v), cudaMemcpyDeviceToHost));
    *out = v;
    return TL_OK;
}

TL_API int tl_chain_seek(tl_chain* c, uint64_t sweep)
{
    if (!c || sweep > 0xFFFFFFFFull) return fail(TL_EINVAL, "tl_chain_seek: bad argument");
    c->sweep = sweep;
    return TL_OK;
}

// ---------------------------------------------------------------------------
// Checkpoints: the chain's inputs and position (RandomWalk's state carried
// between calls, Sec. 2.2) in one self-describing byte string.
// ---------------------------------------------------------------------------
namespace {
constexpr uint32_t kBlobMagic = 0x4B434C54u;   // "TLCK"
constexpr uint32_t kBlobVersion = 1;
struct BlobHead {
    uint32_t magic, version;
    int32_t lattice, W, H, N, kappa, random_order;
    uint64_t seed, sweep;
    uint32_t stream_id;
    int32_t thr_kind;
    uint32_t thr_scalar;
    uint32_t table16[16];
    uint64_t canon_bytes, site_words;
};
}  // namespace

TL_API int tl_checkpoint(tl_chain* c, tl_blob* out)
{
    NvtxRange nvtx_("tl_checkpoint");
    if (!c || !out) return fail(TL_EINVAL, "tl_checkpoint: NULL argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    CUDA_TRY(cudaDeviceSynchronize());
    const Geom& g = c->g;
    const size_t ncanon = (size_t)g.ntype * g.W * g.H;
    BlobHead hd{};
    hd.magic = kBlobMagic;
    hd.version = kBlobVersion;
    hd.lattice = g.lattice;
    hd.W = g.W;
    hd.H = g.H;
    hd.N = g.N;
    hd.kappa = c->kappa;
    hd.random_order = c->random_order;
    hd.seed = c->seed;
    hd.sweep = c->sweep;
    hd.stream_id = c->stream_id;
    hd.thr_kind = c->thr_api_kind;
    hd.thr_scalar = c->th.scalar;
    for (int i = 0; i < 16; ++i) hd.table16[i] = c->thr_table16[i];
    hd.canon_bytes = ncanon;
    hd.site_words = c->thr_site.size();
    const size_t size = sizeof(hd) + 2 * ncanon + 4 * hd.site_words;
    uint8_t* buf = static_cast<uint8_t*>(std::malloc(size));
    if (!buf) return fail(TL_ENOMEM, "tl_checkpoint: %zu bytes", size);
    std::memcpy(buf, &hd, sizeof(hd));
    uint8_t* start = buf + sizeof(hd);
    uint8_t* cur = start + ncanon;
    cudaError_t e = (cudaError_t)launch_unpack(g, c->rows0, c->canon, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(start, c->canon, ncanon, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = (cudaError_t)launch_unpack(g, c->rows, c->canon, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(cur, c->canon, ncanon, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        std::free(buf);
        return fail(TL_ECUDA, "tl_checkpoint: %s", cudaGetErrorString(e));
    }
    c->launches += 2;
    if (hd.site_words) std::memcpy(cur + ncanon, c->thr_site.data(), 4 * hd.site_words);
    out->data = buf;
    out->size = size;
    return TL_OK;
}

TL_API void tl_blob_free(tl_blob* b)
{
    if (!b) return;
    std::free(b->data);
    b->data = nullptr;
    b->size = 0;
}

TL_API int tl_restore(tl_ctx* ctx, const tl_blob* blob, tl_chain** out)
{
    NvtxRange nvtx_("tl_restore");
    if (!ctx || !blob || !blob->data || !out) return fail(TL_EINVAL, "tl_restore: NULL argument");
    BlobHead hd;
    if (blob->size < sizeof(hd)) return fail(TL_EINVAL, "tl_restore: blob too short");
    std::memcpy(&hd, blob->data, sizeof(hd));
    if (hd.magic != kBlobMagic || hd.version != kBlobVersion)
        return fail(TL_EINVAL, "tl_restore: not a checkpoint of this library version");
    if (hd.lattice < 0 || hd.lattice > 2 || !box_ok(hd.W, hd.H) || hd.thr_kind < 0 || hd.thr_kind > 2 ||
        hd.sweep > 0xFFFFFFFFull || (hd.random_order != 0 && hd.random_order != 1))
        return fail(TL_EINVAL, "tl_restore: corrupt header");
    const int ntype = hd.lattice == LAT_LOZENGE ? 3 : 2;
    const uint64_t ncanon = (uint64_t)ntype * hd.W * hd.H;
    const uint64_t want_sites = hd.thr_kind == TL_T_SITE ? (uint64_t)hd.W * hd.H : 0;
    if (hd.canon_bytes != ncanon || hd.site_words != want_sites ||
        blob->size != sizeof(hd) + 2 * ncanon + 4 * want_sites)
        return fail(TL_EINVAL, "tl_restore: sizes do not match the header");
    const uint8_t* start = static_cast<const uint8_t*>(blob->data) + sizeof(hd);
    const uint8_t* cur = start + ncanon;
    // the domain: the six-vertex square from its size, a domino or lozenge
    // domain from the faces its starting tiling covers
    tl_domain* d = nullptr;
    int rc;
    if (hd.lattice == LAT_SIXV) {
        if (hd.N < 1 || hd.W != hd.N + 2 || hd.H != hd.N + 2) return fail(TL_EINVAL, "tl_restore: corrupt header");
        rc = tl_domain_dwbc(hd.N, &d);
    } else {
        d = new (std::nothrow) tl_domain();
        if (!d) return fail(TL_ENOMEM, "tl_restore: host allocation");
        d->g = make_geom(hd.lattice, hd.W, hd.H, 0);
        d->init.assign(start, start + ncanon);
        rc = finish_domain(d, 0, &d);
        if (rc == TL_OK) d->kappa = hd.kappa;
    }
    if (rc != TL_OK) return rc;
    tl_thresholds th{};
    th.kind = hd.thr_kind;
    th.scalar = hd.thr_scalar;
    for (int i = 0; i < 16; ++i) th.table16[i] = hd.table16[i];
    std::vector<uint32_t> site;
    if (want_sites) {
        site.resize(want_sites);
        std::memcpy(site.data(), cur + ncanon, 4 * want_sites);
        th.site = site.data();
    }
    tl_chain* c = nullptr;
    rc = tl_chain_create(ctx, d, start, hd.seed, hd.stream_id, &th, &c);
    tl_domain_destroy(d);
    if (rc != TL_OK) return rc;
    c->kappa = hd.kappa;
    c->random_order = hd.random_order;
    c->sweep = hd.sweep;
    rc = tl_write_state(c, cur, ncanon, nullptr);
    if (rc != TL_OK) {
        tl_chain_destroy(c);
        return rc;
    }
    *out = c;
    return TL_OK;
}

// Coupling from the past (Sec. 1.1.4).  Both chains use the random numbers
// of the absolute sweeps 2^32 - T .. 2^32 - 1, so when T doubles the last T
// sweeps repeat exactly the moves of the previous attempt: the run from
// time -2T first takes T new sweeps and then the old ones.
TL_API int tl_cftp(tl_ctx* ctx, const tl_domain* d, uint64_t seed, uint32_t stream_id, const tl_thresholds* th,
                   uint64_t t0, uint64_t tmax, uint8_t* canon_out, size_t cap, uint64_t* t_used, void* stream)
{
    NvtxRange nvtx_("tl_cftp");
    if (!ctx || !d || !th || !canon_out || t0 < 1 || tmax < t0 || tmax > 0x80000000ull)
        return fail(TL_EINVAL, "tl_cftp: bad argument");
    const size_t n = d->init.size();
    if (cap < n) return fail(TL_EINVAL, "tl_cftp: cap %zu < %zu", cap, n);
    std::vector<uint8_t> top_cfg, bot_cfg;
    TL_TRY(extreme_config(d, true, top_cfg));
    TL_TRY(extreme_config(d, false, bot_cfg));
    tl_chain *top = nullptr, *bot = nullptr;
    int rc = tl_chain_create(ctx, d, top_cfg.data(), seed, stream_id, th, &top);
    if (rc == TL_OK) rc = tl_chain_create(ctx, d, bot_cfg.data(), seed, stream_id, th, &bot);
    std::vector<uint8_t> a, b;
    uint64_t T = t0;
    bool done = false;
    // the two chains share every random number and run at the same time: in
    // one launch of the one-block kernel where they take it, else on two streams
    // where their stripes fit the SMs together
    const bool res = rc == TL_OK && want_resident(top) && want_resident(bot);
    const bool pair = res && small_run(top) && small_run(bot);
    cudaStream_t side = nullptr;
    cudaEvent_t ready = nullptr;
    if (res && !pair && top->res.ctas + bot->res.ctas <= ctx->sms &&
        (cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking) != cudaSuccess ||
         cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess))
        rc = fail(TL_ECUDA, "tl_cftp: side stream");
    while (rc == TL_OK && !done) {
        for (tl_chain* c : {top, bot}) {
            if (rc == TL_OK) rc = tl_chain_reset(c, stream);
            if (rc == TL_OK) rc = tl_chain_seek(c, 0x100000000ull - T);
        }
        if (pair) {
            for (uint64_t done = 0; rc == TL_OK && done < T;) {
                const uint64_t n = std::min(T - done, max_launch_sweeps(top));
                const int e = launch_small(top->g, top->rows, bot->rows, top->small_threads, (uint32_t)top->sweep,
                                           (uint32_t)n, top->rng, top->grange, stream);
                if (e) rc = fail(TL_ECUDA, "tl_cftp: %s", cudaGetErrorString((cudaError_t)e));
                for (tl_chain* c : {top, bot}) {
                    c->sweep += n;
                    c->launches += 1;
                }
                done += n;
            }
        } else if (side) {
            cudaError_t e = cudaEventRecord(ready, SS(stream));   // the resets
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ready, 0);
            if (rc == TL_OK && e != cudaSuccess) rc = fail(TL_ECUDA, "tl_cftp: %s", cudaGetErrorString(e));
            if (rc == TL_OK) rc = tl_run_sweeps(top, T, stream);
            if (rc == TL_OK) rc = tl_run_sweeps(bot, T, side);
            const int rs = tl_chain_sync(bot, side);
            if (rc == TL_OK) rc = rs;
            if (rc == TL_OK) rc = tl_chain_sync(top, stream);
        } else {
            for (tl_chain* c : {top, bot}) {
                if (rc == TL_OK) rc = tl_run_sweeps(c, T, stream);
                if (rc == TL_OK) rc = tl_chain_sync(c, stream);
            }
        }
        uint64_t ht = 0, hb = 0;
        if (rc == TL_OK) rc = tl_state_hash(top, &ht, stream);
        if (rc == TL_OK) rc = tl_state_hash(bot, &hb, stream);
        if (rc != TL_OK) break;
        if (ht == hb) {
            a.resize(n);
            b.resize(n);
            rc = tl_read_state(top, a.data(), n, stream);
            if (rc == TL_OK) rc = tl_read_state(bot, b.data(), n, stream);
            if (rc == TL_OK && a == b) done = true;
        }
        if (!done && rc == TL_OK) {
            if (T * 2 > tmax) {
                rc = fail(TL_EBUDGET, "tl_cftp: top and bottom chains still differ after %llu sweeps",
                          (unsigned long long)T);
                break;
            }
            T *= 2;
        }
    }
    if (rc == TL_OK) {
        if (is_device_ptr(canon_out)) {
            cudaSetDevice(ctx->device);
            const cudaError_t e = cudaMemcpy(canon_out, a.data(), n, cudaMemcpyHostToDevice);
            if (e != cudaSuccess) rc = fail(TL_ECUDA, "tl_cftp: %s", cudaGetErrorString(e));
        } else {
            std::memcpy(canon_out, a.data(), n);
        }
        if (t_used) *t_used = T;
    }
    if (side) cudaStreamSynchronize(side);
    if (ready) cudaEventDestroy(ready);
    if (side) cudaStreamDestroy(side);
    tl_chain_destroy(top);
    tl_chain_destroy(bot);
    return rc;
}

TL_API int tl_read_height(tl_chain* c, int32_t* out, size_t cap, void* stream)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_read_height: NULL argument");
    const tl_domain& d = c->dom_copy;
    const size_t n = (size_t)d.hw * d.hh;
    if (cap < n) return fail(TL_EINVAL, "tl_read_height: cap %zu < %zu", cap, n);
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    int32_t* dst = out;
    TL_TRY(require_local(out, c->ctx->device, "tl_read_height"));
    const bool dev = is_device_ptr(out);
    if (!dev) {
        if (!c->hscratch) TL_TRY(dev_alloc(&c->hscratch, n, "height scratch"));
        dst = c->hscratch;
    }
    const int e = launch_height(c->g, c->rows, c->hseg, d.nseg, d.hw, d.hh, dst, c->hbase, stream);
    if (e) return fail(TL_ECUDA, "height kernels: %s", cudaGetErrorString((cudaError_t)e));
    c->launches += (uint64_t)height_launches(d.nseg, d.hw, d.hh);
    if (!dev) {
        CUDA_TRY(cudaMemcpyAsync(out, dst, n * sizeof(int32_t), cudaMemcpyDeviceToHost, SS(stream)));
        CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    }
    return TL_OK;
}

TL_API int tl_read_height_noalloc(tl_chain* c, int32_t* out, size_t cap, void* stream)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_read_height_noalloc: NULL argument");
    const tl_domain& d = c->dom_copy;
    const size_t n = (size_t)d.hw * d.hh;
    if (cap < n) return fail(TL_EINVAL, "tl_read_height_noalloc: cap %zu < %zu", cap, n);
    if (d.nseg > noalloc_height_max_segments())
        return fail(TL_EINVAL, "tl_read_height_noalloc: %d height segments exceed the static scratch limit of %d",
                    d.nseg, noalloc_height_max_segments());
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(require_local(out, c->ctx->device, "tl_read_height_noalloc"));
    if (!is_device_ptr(out))
        return fail(TL_EINVAL, "tl_read_height_noalloc: `out` must be device memory (a host buffer would "
                               "need a staging allocation)");
    const int e = launch_height_noalloc(c->g, c->rows, c->hseg, d.nseg, d.hw, d.hh, out, c->ctx->device, stream);
    if (e) return fail(TL_ECUDA, "tl_read_height_noalloc: %s", cudaGetErrorString((cudaError_t)e));
    c->launches += (uint64_t)height_launches(d.nseg, d.hw, d.hh);
    return TL_OK;
}

TL_API int tl_density_begin(tl_chain* c, uint32_t stride, uint64_t burn_in)
{
    if (!c || stride == 0) return fail(TL_EINVAL, "tl_density_begin: bad argument");
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    const size_t n = (size_t)c->g.ntype * c->g.W * c->g.H;
    if (!c->counts) TL_TRY(dev_alloc(&c->counts, n, "density counters"));
    if (!c->cplanes) TL_TRY(dev_alloc(&c->cplanes, (size_t)32 * c->g.H * c->g.row_words, "density counter planes"));
    c->counts_dirty = true;
    c->samples = 0;
    c->stride = stride;
    c->burn = burn_in;
    c->density_on = true;
    return TL_OK;
}

template <class F>
static int to_output(tl_chain* c, double* out, size_t n, void* stream, F launch)
{
    TL_TRY(require_local(out, c->ctx->device, "density readback"));
    if (is_device_ptr(out)) {
        const int e = launch(out);
        if (e) return fail(TL_ECUDA, "density kernel: %s", cudaGetErrorString((cudaError_t)e));
        c->launches += 1;
        return TL_OK;
    }
    if (c->dscratch_n < n) {
        CUDA_TRY(cudaStreamSynchronize(SS(stream)));
        cudaFree(c->dscratch);
        c->dscratch = nullptr;
        c->dscratch_n = 0;
        TL_TRY(dev_alloc(&c->dscratch, n, "density output"));
        c->dscratch_n = n;
    }
    int e = launch(c->dscratch);
    c->launches += 1;
    if (!e) e = cudaMemcpyAsync(out, c->dscratch, n * sizeof(double), cudaMemcpyDeviceToHost, SS(stream));
    if (!e) e = cudaStreamSynchronize(SS(stream));
    if (e) return fail(TL_ECUDA, "density readback: %s", cudaGetErrorString((cudaError_t)e));
    return TL_OK;
}

TL_API int tl_read_density(tl_chain* c, double* out, size_t cap, uint64_t* samples, void* stream)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_read_density: NULL argument");
    if (!c->counts) return fail(TL_EINVAL, "tl_read_density: tl_density_begin was not called");
    const size_t n = (size_t)c->g.ntype * c->g.W * c->g.H;
    if (cap < n) return fail(TL_EINVAL, "tl_read_density: cap %zu < %zu", cap, n);
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(zero_counts_if_needed(c, stream));
    if (samples) *samples = c->samples;
    const int ed = launch_density_decode(c->g, c->cplanes, c->samples, c->counts, stream);
    if (ed) return fail(TL_ECUDA, "density decode: %s", cudaGetErrorString((cudaError_t)ed));
    c->launches += 1;
    return to_output(c, out, n, stream, [&](double* o) {
        return launch_density_read(c->counts, n, c->samples, o, stream);
    });
}

TL_API int tl_read_domino_nsew(tl_chain* c, double* out, size_t cap, void* stream)
{
    if (!c || !out) return fail(TL_EINVAL, "tl_read_domino_nsew: NULL argument");
    if (c->g.lattice != LAT_DOMINO) return fail(TL_EINVAL, "tl_read_domino_nsew: not a domino chain");
    if (!c->counts) return fail(TL_EINVAL, "tl_read_domino_nsew: tl_density_begin was not called");
    const size_t n = (size_t)4 * (c->g.W - 1) * (c->g.H - 1);
    if (cap < n) return fail(TL_EINVAL, "tl_read_domino_nsew: cap %zu < %zu", cap, n);
    CUDA_TRY(cudaSetDevice(c->ctx->device));
    TL_TRY(zero_counts_if_needed(c, stream));
    int launches = 1;
    const int rc = to_output(c, out, n, stream, [&](double* o) {
        return launch_nsew(c->g, c->cplanes, c->counts, c->samples, c->kappa, c->ctx->smem_optin, o, &launches, stream);
    });
    if (rc == TL_OK) c->launches += (uint64_t)(launches - 1);
    return rc;
}

// ---------------------------------------------------------------------------
// Batched chains
// ---------------------------------------------------------------------------
struct tl_batch {
    tl_ctx* ctx = nullptr;
    std::vector<tl_chain*> chains;
    std::vector<BatchChain> hchains;
    BatchChain* d_chains = nullptr;
    std::vector<uint32_t*> alt;           // second state buffer of every chain
    uint32_t* d_sweep = nullptr;          // per-chain sweep counters on the device
    uint32_t* h_sweep = nullptr;          // pinned staging for the counters
    size_t cap = 0;                       // capacity of the descriptor arrays
    std::vector<BatchTile> tiles_lpt;     // largest first (batched launches)
    std::vector<BatchTile> tiles_chain;   // grouped by chain (per-chain launches)
    std::vector<int> chain_first;         // first tile of each chain in tiles_chain
    BatchTile* d_tiles_lpt = nullptr;
    BatchTile* d_tiles_chain = nullptr;
    unsigned int* d_cursor = nullptr;     // one cursor per launch slot
    int ncursor = 0;
    unsigned long long* d_hash = nullptr;
    int* d_status = nullptr;              // raised by a bounded wait that gave up
    int tile_rows = 64, R = 2, block = 100, grid = 0;
    int threads = 256;                    // threads per tile (faces per thread)
    int run_threads = 256;                // threads per tile of the launches: more where tiles are few
    int run_rows = 64, run_R = 2;         // rows per tile and sweeps per launch: fewer where tiles are few or wide
    size_t smem = 0;
    int ntiles = 0;
    int src = 0;                          // buffer holding the current state
    uint64_t launches = 0;
    cudaGraphExec_t graph = nullptr;
    int graph_block = 0, graph_R = 0, graph_launches = 0;
    bool no_graph = false;
};

static int batch_raise_status(tl_batch* b)
{
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    const int one = 1;
    CUDA_TRY(cudaMemcpy(b->d_status, &one, sizeof(int), cudaMemcpyHostToDevice));
    return TL_OK;
}


static void batch_free_plan(tl_batch* b)
{
    cudaFree(b->d_tiles_lpt);
    cudaFree(b->d_tiles_chain);
    b->d_tiles_lpt = b->d_tiles_chain = nullptr;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
}

static void batch_free(tl_batch* b)
{
    if (!b) return;
    batch_free_plan(b);
    for (auto* p : b->alt) cudaFree(p);
    cudaFree(b->d_chains);
    cudaFree(b->d_sweep);
    cudaFreeHost(b->h_sweep);
    cudaFree(b->d_cursor);
    cudaFree(b->d_hash);
    cudaFree(b->d_status);
    tl_ctx* ctx = b->ctx;
    delete b;
    ctx_release(ctx);
}

// Tiles of a batch cut into `rows` rows.
static size_t batch_tiles(const tl_batch* b, int rows)
{
    size_t n = 0;
    for (const tl_chain* c : b->chains) n += (size_t)((c->g.H + rows - 1) / rows);
    return n;
}

// A batch with fewer tiles than SMs takes lower tiles (down to 64 rows) and
// more threads per tile: a serving mix of 12 jobs in 62 tiles of 128 rows left
// 90 SMs idle (100 sweeps and read-out: 1.52 ms so, 1.19 in tiles of 64 rows,
// 1.26 in tiles of 32, whose halos are as high).
static int batch_rows(const tl_batch* b, int tile_rows)
{
    int rows = tile_rows;
    while (rows >= 128 && batch_tiles(b, rows) < (size_t)b->ctx->sms) rows = (rows + 3) / 4 * 2;
    return rows;
}
static int batch_threads(const tl_batch* b, size_t ntiles, int threads)
{
    const size_t sms = (size_t)b->ctx->sms;
    return ntiles <= sms ? 512 : ntiles <= 2 * sms ? 256 : threads;
}

// Tiles of height tile_rows for every chain; shared memory for tile + halo.
static int batch_plan(tl_batch* b, int tile_rows, int R, int threads)
{
    if (tile_rows < 1 || R < 1 || R > 64 || (threads != 128 && threads != 256))
        return fail(TL_EINVAL, "batch plan: tile_rows %d, R %d, threads %d", tile_rows, R, threads);
    std::vector<BatchTile> tiles;
    std::vector<double> work;
    std::vector<int> first;
    size_t smem = 0;
    int rows = batch_rows(b, tile_rows);
    // the rows of a tile and its halos alone
    size_t need = 0;
    for (const tl_chain* c : b->chains)
        need = std::max(need, (size_t)std::min(rows + 2 * c->g.passes * R, c->g.H + 2) * (size_t)c->g.row_words * 4);
    if ((long)need > (long)b->ctx->smem_optin) return fail(TL_EUNSUPPORTED, "batch plan: a tile needs %zu B of shared memory", need);
    int bps = 0, run_threads = threads, run_R = R;
    // where the rows fit and the item table beside them does not, lower tiles do
    // (and below one row, whose halo is then the tile, fewer sweeps a launch)
    for (const int asked = rows;; rows > 1 ? rows = (rows + 1) / 2 : (rows = asked, run_R = (run_R + 1) / 2)) {
        tiles.clear();
        work.clear();
        first.clear();
        smem = 0;
        for (size_t i = 0; i < b->chains.size(); ++i) {
            const tl_chain* c = b->chains[i];
            const Geom& g = c->g;
            const int halo = g.passes * run_R, step = g.lattice == LAT_SIXV ? 2 : 1;
            const std::vector<int2> unit = unit_groups(c->dom_copy);
            std::vector<int> pre(unit.size() + 1, 0);
            for (size_t r = 0; r < unit.size(); ++r) pre[r + 1] = pre[r] + std::max(0, unit[r].y - unit[r].x);
            first.push_back((int)tiles.size());
            for (int lo = 0; lo < g.H; lo += rows) {
                const int hi = std::min(g.H, lo + rows);
                tiles.push_back(BatchTile{(int)i, lo, hi});
                const int slo = std::max(lo - halo, -1), shi = std::min(hi + halo, g.H + 1);
                const int ra = std::max(slo, 0) / step, rb = (std::min(shi, g.H) + step - 1) / step;
                const int items = pre[rb] - pre[ra];
                // rows, then the item table
                smem = std::max(smem, (size_t)(shi - slo) * (size_t)g.row_words * 4 + 4 * (size_t)(rb - ra + 1 + items));
                work.push_back((0.1 * (rb - ra) + items) * run_R);
            }
        }
        first.push_back((int)tiles.size());
        run_threads = batch_threads(b, tiles.size(), threads);
        if ((long)smem <= (long)b->ctx->smem_optin) {
            if (batch_prepare(smem, run_threads, &bps) == 0 && bps > 0) break;
            run_threads = threads;
            if (batch_prepare(smem, run_threads, &bps) == 0 && bps > 0) break;
        }
        if (rows == 1 && run_R == 1) return fail(TL_EUNSUPPORTED, "batch plan: a tile needs %zu B of shared memory", smem);
    }
    std::vector<int> order(tiles.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) { return work[a] > work[c]; });
    std::vector<BatchTile> lpt(tiles.size());
    for (size_t i = 0; i < order.size(); ++i) lpt[i] = tiles[order[i]];
    batch_free_plan(b);
    TL_TRY(dev_alloc(&b->d_tiles_lpt, lpt.size(), "tiles"));
    TL_TRY(dev_alloc(&b->d_tiles_chain, tiles.size(), "tiles"));
    CUDA_TRY(cudaMemcpy(b->d_tiles_lpt, lpt.data(), sizeof(BatchTile) * lpt.size(), cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(b->d_tiles_chain, tiles.data(), sizeof(BatchTile) * tiles.size(), cudaMemcpyHostToDevice));
    b->tiles_lpt = lpt;
    b->tiles_chain = tiles;
    b->chain_first = first;
    b->ntiles = (int)tiles.size();
    b->tile_rows = tile_rows;
    b->R = R;
    b->threads = threads;
    b->run_threads = run_threads;
    b->run_rows = rows;
    b->run_R = run_R;
    b->smem = smem;
    b->grid = std::min(bps * b->ctx->sms, b->ntiles);
    return TL_OK;
}

// (Re)build the device descriptors of every chain in the batch.
static int batch_rebuild(tl_batch* b)
{
    const size_t n = b->chains.size();
    if (n > b->cap) {
        const size_t cap = std::max<size_t>(n, 2 * b->cap);
        cudaFree(b->d_chains);
        cudaFree(b->d_sweep);
        cudaFree(b->d_hash);
        cudaFreeHost(b->h_sweep);
        b->d_chains = nullptr;
        b->d_sweep = nullptr;
        b->d_hash = nullptr;
        b->h_sweep = nullptr;
        TL_TRY(dev_alloc(&b->d_chains, cap, "batch chains"));
        TL_TRY(dev_alloc(&b->d_sweep, cap, "sweeps"));
        TL_TRY(dev_alloc(&b->d_hash, cap, "hashes"));
        if (cudaMallocHost((void**)&b->h_sweep, cap * 4) != cudaSuccess) {
            cudaGetLastError();
            return fail(TL_ENOMEM, "batch: pinned host allocation");
        }
        b->cap = cap;
    }
    b->hchains.clear();
    for (size_t i = 0; i < n; ++i) {
        tl_chain* c = b->chains[i];
        BatchChain bc{};
        bc.g = c->g;
        bc.rows[0] = c->rows;
        bc.rows[1] = b->alt[i];
        bc.gpre = reinterpret_cast<const int*>(c->grange + c->g.H);
        bc.gfirst = bc.gpre + c->g.H + 2;
        bc.th = c->th;
        bc.rng = c->rng;
        bc.sweep_base = b->d_sweep + i;
        b->hchains.push_back(bc);
    }
    if (n) CUDA_TRY(cudaMemcpy(b->d_chains, b->hchains.data(), sizeof(BatchChain) * n, cudaMemcpyHostToDevice));
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    if (n) return batch_plan(b, b->tile_rows, b->R, b->threads);
    b->ntiles = 0;
    return TL_OK;
}

static int batch_attach(tl_batch* b, tl_chain* c)
{
    if (!c || c->ctx->device != b->ctx->device) return fail(TL_EINVAL, "batch: chain on another device");
    if (c->density_on) return fail(TL_EINVAL, "batch: chain samples densities");
    if (c->random_order) return fail(TL_EUNSUPPORTED, "batch: chain uses the random pass order");
    for (auto* x : b->chains)
        if (x == c) return fail(TL_EINVAL, "batch: chain already in the batch");
    uint32_t* a = nullptr;
    TL_TRY(dev_alloc(&a, (size_t)c->g.total_words, "second state buffer"));
    if (cudaMemset(a, 0, (size_t)c->g.total_words * 4) != cudaSuccess) {
        cudaFree(a);
        return fail(TL_ECUDA, "batch: memset");
    }
    b->chains.push_back(c);
    b->alt.push_back(a);
    return TL_OK;
}

TL_API int tl_batch_create(tl_ctx* ctx, tl_chain* const* chains, size_t n, tl_batch** out)
{
    if (!ctx || !out || (n && !chains)) return fail(TL_EINVAL, "tl_batch_create: bad argument");
    CUDA_TRY(cudaSetDevice(ctx->device));
    tl_batch* b = new (std::nothrow) tl_batch();
    if (!b) return fail(TL_ENOMEM, "tl_batch_create: host allocation");
    b->ctx = ctx;
    ctx->refs.fetch_add(1);
    b->ncursor = 1024;
    int rc = dev_alloc(&b->d_cursor, (size_t)b->ncursor, "cursors");
    if (rc == TL_OK) rc = dev_alloc(&b->d_status, 1, "status");
    if (rc == TL_OK && (cudaMemset(b->d_cursor, 0, sizeof(unsigned int) * b->ncursor) != cudaSuccess ||
                        cudaMemset(b->d_status, 0, sizeof(int)) != cudaSuccess))
        rc = fail(TL_ECUDA, "tl_batch_create: memset");
    for (size_t i = 0; i < n && rc == TL_OK; ++i) rc = batch_attach(b, chains[i]);
    if (rc == TL_OK) rc = batch_rebuild(b);
    if (rc != TL_OK) {
        batch_free(b);
        return rc;
    }
    *out = b;
    return TL_OK;
}

TL_API int tl_batch_add(tl_batch* b, tl_chain* c)
{
    if (!b) return fail(TL_EINVAL, "tl_batch_add: NULL batch");
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    TL_TRY(batch_attach(b, c));
    return batch_rebuild(b);
}

TL_API int tl_batch_remove(tl_batch* b, tl_chain* c)
{
    if (!b || !c) return fail(TL_EINVAL, "tl_batch_remove: NULL argument");
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    size_t i = 0;
    while (i < b->chains.size() && b->chains[i] != c) ++i;
    if (i == b->chains.size()) return fail(TL_EINVAL, "tl_batch_remove: chain not in the batch");
    CUDA_TRY(cudaDeviceSynchronize());   // no launch may still use its second buffer
    cudaFree(b->alt[i]);
    b->chains.erase(b->chains.begin() + (long)i);
    b->alt.erase(b->alt.begin() + (long)i);
    return batch_rebuild(b);
}

TL_API size_t tl_batch_size(const tl_batch* b) { return b ? b->chains.size() : 0; }

TL_API void tl_batch_destroy(tl_batch* b)
{
    if (b) cudaSetDevice(b->ctx->device);
    batch_free(b);
}

TL_API uint64_t tl_batch_launches(const tl_batch* b) { return b ? b->launches : 0; }

static int batch_upload_sweeps(tl_batch* b, uint64_t k, void* stream)
{
    // the pinned staging buffer may still feed the previous run's copy
    CUDA_TRY(cudaStreamSynchronize(SS(stream)));
    for (size_t i = 0; i < b->chains.size(); ++i) {
        if (b->chains[i]->sweep + k > 0xFFFFFFFFull) return fail(TL_EINVAL, "batch: sweep index beyond 2^32");
        if (b->chains[i]->random_order) return fail(TL_EUNSUPPORTED, "batch: chain uses the random pass order");
        b->h_sweep[i] = (uint32_t)b->chains[i]->sweep;
    }
    CUDA_TRY(cudaMemcpyAsync(b->d_sweep, b->h_sweep, 4 * b->chains.size(), cudaMemcpyHostToDevice, SS(stream)));
    return TL_OK;
}

// One batched launch of r sweeps starting `off` sweeps after the counters.
static int batch_launch(tl_batch* b, int r, uint32_t off, int slot, void* stream, bool per_chain)
{
    unsigned int* cur = b->d_cursor + (slot % b->ncursor);
    if (!per_chain) {
        // cursors of the launches to come, cleared together (a clear before each
        // launch cost 1 us and a gap each); a grid that covers
        // the tiles reads none
        if (slot % b->ncursor == 0 && b->grid < b->ntiles)
            CUDA_TRY(cudaMemsetAsync(b->d_cursor, 0, sizeof(unsigned int) * b->ncursor, SS(stream)));
        const int e = launch_batch(b->d_chains, b->d_tiles_lpt, b->ntiles, r, off, b->src, cur, b->grid, b->run_threads,
                                   b->smem, b->d_status, stream);
        if (e) return fail(TL_ECUDA, "batch kernel: %s", cudaGetErrorString((cudaError_t)e));
        b->launches += 1;
    } else {
        for (size_t i = 0; i < b->chains.size(); ++i) {
            const int t0 = b->chain_first[i], nt = b->chain_first[i + 1] - t0;
            unsigned int* ci = b->d_cursor + ((slot * (int)b->chains.size() + (int)i) % b->ncursor);
            CUDA_TRY(cudaMemsetAsync(ci, 0, 4, SS(stream)));
            const int e = launch_batch(b->d_chains, b->d_tiles_chain + t0, nt, r, off, b->src, ci,
                                       std::min(nt, b->grid), b->run_threads, b->smem, b->d_status, stream);
            if (e) return fail(TL_ECUDA, "batch kernel: %s", cudaGetErrorString((cudaError_t)e));
            b->launches += 1;
        }
    }
    b->src ^= 1;
    return TL_OK;
}

static int batch_finish(tl_batch* b, uint64_t k, void* stream)
{
    // state back in each chain's own buffer; counters advanced
    if (b->src) {
        const int e = launch_batch_copy(b->d_chains, b->d_tiles_chain, b->ntiles, 1, stream);
        if (e) return fail(TL_ECUDA, "batch copy: %s", cudaGetErrorString((cudaError_t)e));
        b->launches += 1;
        b->src = 0;
    }
    for (auto* c : b->chains) c->sweep += k;
    return TL_OK;
}

// Launch sizes covering `k` sweeps with at most R sweeps each and an even
// number of launches, so that the state ends in the buffer it started in.
static std::vector<int> batch_launch_sizes(uint64_t k, int R)
{
    std::vector<int> v;
    for (uint64_t d = 0; d < k; d += (uint64_t)R) v.push_back((int)std::min<uint64_t>((uint64_t)R, k - d));
    if (v.size() % 2) {
        // split the largest launch in two (a launch of one sweep cannot be split)
        size_t i = 0;
        for (size_t j = 0; j < v.size(); ++j)
            if (v[j] > v[i]) i = j;
        if (v[i] >= 2) {
            const int a = v[i] / 2;
            v[i] -= a;
            v.insert(v.begin() + (long)i + 1, a);
        }
    }
    return v;
}

// Graph of one block of `block` sweeps: the launches plus the counter advance.
static int batch_build_graph(tl_batch* b, void* stream)
{
    if (b->graph && b->graph_block == b->block && b->graph_R == b->run_R) return TL_OK;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    cudaStream_t s = SS(stream);
    if (!s) return TL_OK;   // the legacy stream cannot be captured: run without a graph
    const std::vector<int> sizes = batch_launch_sizes((uint64_t)b->block, b->run_R);
    if (sizes.size() % 2) return TL_OK;   // cannot keep the buffers aligned: no graph
    const int src0 = b->src;
    const uint64_t l0 = b->launches;
    CUDA_TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    int rc = TL_OK;
    uint32_t off = 0;
    for (size_t j = 0; j < sizes.size() && rc == TL_OK; ++j) {
        rc = batch_launch(b, sizes[j], off, (int)j, stream, false);
        off += (uint32_t)sizes[j];
    }
    if (rc == TL_OK) {
        const int e = launch_batch_advance(b->d_chains, (int)b->chains.size(), (uint32_t)b->block, b->d_cursor, 0, stream);
        if (e) rc = fail(TL_ECUDA, "batch advance: %s", cudaGetErrorString((cudaError_t)e));
    }
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(s, &graph);
    b->src = src0;
    b->launches = l0;
    if (rc != TL_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (ce != cudaSuccess) return fail(TL_ECUDA, "batch graph capture: %s", cudaGetErrorString(ce));
    const cudaError_t ie = cudaGraphInstantiate(&b->graph, graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess) return fail(TL_ECUDA, "batch graph instantiate: %s", cudaGetErrorString(ie));
    b->graph_block = b->block;
    b->graph_R = b->run_R;
    b->graph_launches = (int)sizes.size();
    return TL_OK;
}

static int batch_run(tl_batch* b, uint64_t k, void* stream, bool per_chain)
{
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    if (k == 0 || b->chains.empty()) return TL_OK;
    TL_TRY(batch_upload_sweeps(b, k, stream));
    uint64_t done = 0;
    if (!per_chain && !b->no_graph && k >= (uint64_t)b->block) TL_TRY(batch_build_graph(b, stream));
    while (!per_chain && !b->no_graph && b->graph && k - done >= (uint64_t)b->block) {
        CUDA_TRY(cudaGraphLaunch(b->graph, SS(stream)));
        b->launches += (uint64_t)b->graph_launches + 1;
        done += (uint64_t)b->block;
    }
    // the rest: offsets relative to the counters after the last advance
    const uint64_t rest_start = done;
    const std::vector<int> sizes = batch_launch_sizes(k - done, b->run_R);
    uint32_t off = 0;
    for (size_t j = 0; j < sizes.size(); ++j) {
        TL_TRY(batch_launch(b, sizes[j], off, (int)j, stream, per_chain));
        off += (uint32_t)sizes[j];
    }
    if (k > rest_start) {
        const int e = launch_batch_advance(b->d_chains, (int)b->chains.size(), (uint32_t)(k - rest_start), b->d_cursor,
                                           0, stream);
        if (e) return fail(TL_ECUDA, "batch advance: %s", cudaGetErrorString((cudaError_t)e));
        b->launches += 1;
    }
    return batch_finish(b, k, stream);
}

TL_API int tl_batch_run(tl_batch* b, uint64_t k, void* stream)
{
    NvtxRange nvtx_("tl_batch_run");
    if (!b) return fail(TL_EINVAL, "tl_batch_run: NULL batch");
    return batch_run(b, k, stream, false);
}

TL_API int tl_batch_run_per_chain(tl_batch* b, uint64_t k, void* stream)
{
    if (!b) return fail(TL_EINVAL, "tl_batch_run_per_chain: NULL batch");
    return batch_run(b, k, stream, true);
}

TL_API int tl_batch_hashes(tl_batch* b, uint64_t* out, size_t n, void* stream)
{
    if (!b || !out || n < b->chains.size()) return fail(TL_EINVAL, "tl_batch_hashes: bad argument");
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    CUDA_TRY(cudaMemsetAsync(b->d_hash, 0, 8 * b->chains.size(), SS(stream)));
    const int e = launch_batch_hash(b->d_chains, b->d_tiles_chain, b->ntiles, b->src, b->d_hash, stream);
    if (e) return fail(TL_ECUDA, "batch hash: %s", cudaGetErrorString((cudaError_t)e));
    b->launches += 1;
    TL_TRY(require_local(out, b->ctx->device, "tl_batch_hashes"));
    const bool dev = is_device_ptr(out);
    CUDA_TRY(cudaMemcpyAsync(out, b->d_hash, 8 * b->chains.size(), dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                             SS(stream)));
    if (!dev) {
        CUDA_TRY(cudaStreamSynchronize(SS(stream)));
        int st = 0;
        CUDA_TRY(cudaMemcpy(&st, b->d_status, sizeof(int), cudaMemcpyDeviceToHost));
        if (st) {
            CUDA_TRY(cudaMemset(b->d_status, 0, sizeof(int)));
            return fail(TL_ETIMEOUT, "batch: a bounded wait gave up; chain states are undefined");
        }
    }
    return TL_OK;
}

TL_API int tl_batch_set_plan(tl_batch* b, const tl_batch_plan* p)
{
    if (!b || !p) return fail(TL_EINVAL, "tl_batch_set_plan: NULL argument");
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    const int tr = p->tile_rows > 0 ? p->tile_rows : b->tile_rows;
    const int R = p->sweeps_per_launch > 0 ? p->sweeps_per_launch : b->R;
    const int nt = p->threads > 0 ? p->threads : b->threads;
    if (p->graph_block > 0) {
        b->block = p->graph_block;
        b->no_graph = false;
    } else if (p->graph_block < 0) {
        b->no_graph = true;
    }
    CUDA_TRY(cudaDeviceSynchronize());
    return batch_plan(b, tr, R, nt);
}

TL_API int tl_batch_get_plan(tl_batch* b, tl_batch_plan* p)
{
    if (!b || !p) return fail(TL_EINVAL, "tl_batch_get_plan: NULL argument");
    p->tile_rows = b->tile_rows;
    p->sweeps_per_launch = b->R;
    p->graph_block = b->no_graph ? -1 : b->block;
    p->grid = b->grid;
    p->smem_bytes = (int)b->smem;
    p->ntiles = b->ntiles;
    p->threads = b->threads;
    return TL_OK;
}

TL_API int tl_batch_get_launch(tl_batch* b, int* tile_rows, int* sweeps, int* threads)
{
    if (!b) return fail(TL_EINVAL, "tl_batch_get_launch: NULL batch");
    if (tile_rows) *tile_rows = b->run_rows;
    if (sweeps) *sweeps = b->run_R;
    if (threads) *threads = b->run_threads;
    return TL_OK;
}

// Try tile heights x sweeps per launch on the batch itself, keep the fastest.
// The chains' states and sweep counters are restored afterwards, so tuning
// does not change any result.
// Autotune results per (lattices present, threshold kinds present, rows of
// the batch rounded down to a power of two, SMs, what the trials' tile heights
// and threads come to for its number of tiles): a batch like one already tuned
// takes that plan without trials.
namespace {
using TuneKey = std::tuple<int, int, int, int, int>;
constexpr int kTuneRows[] = {32, 64, 128};
constexpr int kTuneR[] = {1, 2, 4, 8};
constexpr int kTuneThreads[] = {256, 128};
std::mutex g_tune_mu;
struct TunePlan {
    int tile_rows, R, threads;
};
std::map<TuneKey, TunePlan> g_tune_cache;   // -> the plan the trials chose
TuneKey tune_key(const tl_batch* b)
{
    int lat = 0, thr = 0;
    uint64_t rows = 0;
    for (const tl_chain* c : b->chains) {
        lat |= 1 << c->g.lattice;
        thr |= 1 << c->th.kind;
        rows += (uint64_t)c->g.H;
    }
    int bucket = 0;
    while (rows > 1) {
        rows >>= 1;
        ++bucket;
    }
    // two trials that launch the same thing for this batch need not for one of
    // more tiles, which must not take their pick
    int form = 0;
    for (int tr : kTuneRows) {
        const int r = batch_rows(b, tr);
        const size_t n = batch_tiles(b, r);
        form = form * 6 + (r != tr) * 3 + (n <= (size_t)b->ctx->sms ? 0 : n <= 2 * (size_t)b->ctx->sms ? 1 : 2);
    }
    return TuneKey(lat, thr, bucket, b->ctx->sms, form);
}
}  // namespace

TL_API void tl_autotune_cache_clear(void)
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache.clear();
}

TL_API int tl_batch_autotune(tl_batch* b, uint64_t trial_sweeps, void* stream, tl_batch_plan* out)
{
    NvtxRange nvtx_("tl_batch_autotune");
    if (!b || trial_sweeps == 0) return fail(TL_EINVAL, "tl_batch_autotune: bad argument");
    CUDA_TRY(cudaSetDevice(b->ctx->device));
    const TuneKey key = tune_key(b);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end() &&
            batch_plan(b, it->second.tile_rows, it->second.R, it->second.threads) == TL_OK) {
            if (out) TL_TRY(tl_batch_get_plan(b, out));
            return TL_OK;
        }
    }
    // snapshot every chain's state
    size_t total = 0;
    for (auto* c : b->chains) total += (size_t)c->g.total_words;
    uint32_t* snap = nullptr;
    TL_TRY(dev_alloc(&snap, total, "autotune snapshot"));
    size_t o = 0;
    for (auto* c : b->chains) {
        CUDA_TRY(cudaMemcpyAsync(snap + o, c->rows, (size_t)c->g.total_words * 4, cudaMemcpyDeviceToDevice, SS(stream)));
        o += (size_t)c->g.total_words;
    }
    std::vector<uint64_t> sweeps;
    for (auto* c : b->chains) sweeps.push_back(c->sweep);
    std::set<std::tuple<int, int, int>> tried;   // what the trials launched
    float best = 1e30f;
    int best_t = b->tile_rows, best_r = b->R, best_nt = b->threads;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int rc = TL_OK;
    for (int nt : kTuneThreads)
    for (int tr : kTuneRows)
        for (int R : kTuneR) {
            if (rc != TL_OK) break;
            if (batch_plan(b, tr, R, nt) != TL_OK) continue;   // does not fit: skip
            if (!tried.insert({b->run_rows, b->run_R, b->run_threads}).second) continue;
            const uint64_t k = ((trial_sweeps + R - 1) / R) * R;
            const int saved_block = b->block;
            b->block = 1 << 30;                            // no graph during trials
            // two timed runs of the same sweeps (the first also warms the
            // plan up); the faster counts
            float ms = 1e30f;
            for (int rep = 0; rep < 2 && rc == TL_OK; ++rep) {
                if (rep) {
                    size_t o2 = 0;
                    for (size_t i = 0; i < b->chains.size(); ++i) {
                        tl_chain* c = b->chains[i];
                        cudaMemcpyAsync(c->rows, snap + o2, (size_t)c->g.total_words * 4, cudaMemcpyDeviceToDevice,
                                        SS(stream));
                        o2 += (size_t)c->g.total_words;
                        c->sweep = sweeps[i];
                    }
                }
                cudaEventRecord(e0, SS(stream));
                rc = batch_run(b, k, stream, false);
                cudaEventRecord(e1, SS(stream));
                if (rc != TL_OK) break;
                cudaEventSynchronize(e1);
                float t = 0;
                cudaEventElapsedTime(&t, e0, e1);
                ms = std::min(ms, t);
            }
            b->block = saved_block;
            if (rc != TL_OK) break;
            if (ms / k < best) {
                best = ms / k;
                best_t = tr;
                best_r = R;
                best_nt = nt;
            }
            // restore
            o = 0;
            for (size_t i = 0; i < b->chains.size(); ++i) {
                tl_chain* c = b->chains[i];
                cudaMemcpyAsync(c->rows, snap + o, (size_t)c->g.total_words * 4, cudaMemcpyDeviceToDevice, SS(stream));
                o += (size_t)c->g.total_words;
                c->sweep = sweeps[i];
            }
        }
    cudaStreamSynchronize(SS(stream));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(snap);
    if (rc != TL_OK) return rc;
    TL_TRY(batch_plan(b, best_t, best_r, best_nt));
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tune_cache[key] = TunePlan{best_t, best_r, best_nt};
    }
    if (out) TL_TRY(tl_batch_get_plan(b, out));
    return TL_OK;
}
