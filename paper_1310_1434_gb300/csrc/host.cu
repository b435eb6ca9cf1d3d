// Host side of the AIR library: plans (geometry tables + workspace), argument
// checking, the stand-alone operator calls and the solver programs.
#include <cmath>
#include <algorithm>
#include <atomic>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "host_common.h"
#include "launch.h"
#include "orbit.h"
#include "ramp_tc.h"

using namespace air;

namespace air {

thread_local std::string g_err;

air_status fail(air_status s, const std::string &msg) {
    g_err = msg;
    return s;
}

double fan_pitch(const air_geometry &g) {
    if (g.dgamma > 0.0) return g.dgamma;
    return 2.0 * std::asin(g.n * g.pixel_mm / std::sqrt(2.0) / g.dso_mm) / g.n_bins;
}

air_status validate_geometry(const air_geometry *g) {
    if (!g) return fail(AIR_ERR_INVALID_ARG, "geometry is NULL");
    if (g->n < 1 || g->n > 4096) return fail(AIR_ERR_INVALID_ARG, "n must be in 1..4096");
    if (!(g->pixel_mm > 0.0) || !std::isfinite(g->pixel_mm))
        return fail(AIR_ERR_INVALID_ARG, "pixel_mm must be > 0");
    if (g->n_views < 1 || g->n_views > 65536) return fail(AIR_ERR_INVALID_ARG, "n_views must be in 1..65536");
    if (g->n_bins < 1 || g->n_bins > RAMP_MAX_BINS) return fail(AIR_ERR_INVALID_ARG, "n_bins must be in 1..8192");
    if ((long long)g->n_views * g->n_bins > (1ll << 26))
        return fail(AIR_ERR_INVALID_ARG, "n_views * n_bins must be <= 2^26");
    const double rc = g->n * g->pixel_mm / std::sqrt(2.0);
    if (!(g->dso_mm >= rc + 8.0 * g->pixel_mm) || !std::isfinite(g->dso_mm))
        return fail(AIR_ERR_INVALID_ARG,
                    "dso_mm must exceed the image's circumscribed radius n*dx/sqrt(2) by 8 pixels");
    if (!(g->dgamma >= 0.0) || !std::isfinite(g->dgamma)) return fail(AIR_ERR_INVALID_ARG, "dgamma must be >= 0");
    if (!std::isfinite(g->beta0) || !std::isfinite(g->arc) || g->arc == 0.0)
        return fail(AIR_ERR_INVALID_ARG, "beta0 must be finite and arc finite and nonzero");
    if (g->filter != AIR_FILTER_NONE && g->filter != AIR_FILTER_RAMLAK)
        return fail(AIR_ERR_INVALID_ARG, "filter must be AIR_FILTER_NONE or AIR_FILTER_RAMLAK");
    if (g->precision != AIR_PREC_FP32 && g->precision != AIR_PREC_BF16X3)
        return fail(AIR_ERR_INVALID_ARG, "precision must be AIR_PREC_FP32 or AIR_PREC_BF16X3");
    return AIR_OK;
}

// Device pointer check: non-NULL, 16-byte aligned, and device accessible
// (a host pointer handed to a kernel would fault the GPU).
air_status check_dev_ptr(const void *p, const char *what) {
    if (!p) return fail(AIR_ERR_INVALID_ARG, std::string(what) + " is NULL");
    if (reinterpret_cast<uintptr_t>(p) & 15u)
        return fail(AIR_ERR_INVALID_ARG, std::string(what) + " is not 16-byte aligned");
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(AIR_ERR_INVALID_ARG, std::string(what) + " is not a CUDA pointer");
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return fail(AIR_ERR_INVALID_ARG, std::string(what) + " is not device memory");
    return AIR_OK;
}

bool overlap(const void *a, size_t na, const void *b, size_t nb) {
    const char *pa = (const char *)a, *pb = (const char *)b;
    return pa < pb + nb && pb < pa + na;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace air

// -------------------------------------------------------------------- plan
namespace air {
// Backprojector view parts of a slice: enough (pixel tile, part) blocks for
// about 12 per SM (2.4 waves at 5 resident blocks), at most one part per
// view.  The autotuner starts from this and tries up to twice as many.
static int sm_count();
int choose_bwd_parts(const SliceDesc &s) {
    const int sms = sm_count();
    const int txy = tiles_bwd_xy(s), target = 2 * 6 * sms;
    const int S = (target + txy - 1) / txy;
    return S < 1 ? 1 : (S > s.V ? s.V : S);
}

cudaError_t launch_backprojection(const SliceDesc &s, int mode, bool packed, cudaStream_t st, bool overlap) {
    cudaError_t e = s.orb && !packed ? launch_op(OP_ORB_ZPACK, s, mode, st, overlap) : cudaSuccess;
    if (e == cudaSuccess) e = launch_op(s.orb ? OP_ORB_BWD : OP_BWD, s, mode, st, overlap);
    if (e == cudaSuccess && (mode != BWD_PLAIN || bwd_images(s) > 1)) e = launch_op(OP_BWD_FIN, s, mode, st, overlap);
    return e;
}

// Most splits of the orbit backprojector's segments: about two waves of three
// blocks per SM, at most 8 (each split adds eight images to the sum).
static int orb_splits_max(int n, int nf, int sms) {
    const int tiles = ((n + BWD_T - 1) / BWD_T) * ((n + BWD_T - 1) / BWD_T) * (nf == 8 ? 1 : 2);
    const int S = (2 * 3 * sms + tiles - 1) / tiles;
    return S < 1 ? 1 : (S > 8 ? 8 : S);
}

// Column parts of the orbit projector: as few as give the device about 24
// warps per SM (each part pays for the warp's set-up and the sum).
static int choose_orb_ks(int warps, int sms) {
    int ks = 1;
    while (ks < 8 && (long long)warps * ks < 2400ll * sms) ks *= 2;
    return ks;
}

// The FBP backprojection over orbits of views: split until the blocks fill
// the device about three times (five of 256 threads per SM), within what the
// part buffer holds of images and, behind them, the packed views; a multiple
// of eight images for their sum.
static void choose_fbp(SliceDesc &s, const FbpOrbits &F, float *bpart, int parts_max, int sms) {
    s.fbp_nf = 0;
    if (!F.nf) return;
    const size_t nn = (size_t)s.n * s.n, packed = F.base.size() * (size_t)(s.nb + 4) * F.nf;
    const int step = 8 / F.nf, most = std::min<int>(8, (int)F.base.size()) / step * step;
    int splits = std::min(most, (3 * 5 * sms + tiles_shr(s) - 1) / tiles_shr(s) / step * step);
    splits = std::max(splits, step);
    while (splits > step && align_up((size_t)splits * F.nf * nn, 4) + packed > (size_t)parts_max * nn) splits -= step;
    const size_t off = align_up((size_t)splits * F.nf * nn, 4);
    if (off + packed > (size_t)parts_max * nn) return;
    s.fbp_nf = F.nf;
    s.fbp_nbase = (int)F.base.size();
    s.fbp_splits = splits;
    for (int f = 0; f < 8; ++f) s.fbp_code[f] = F.code[f];
    s.fbp_q = reinterpret_cast<float4 *>(bpart + off);
}

static int sm_count() {
    int sms = 148, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    return sms;
}

// Device bytes of the tensor-core filter's buffers (ramp_tc_create).
static size_t filter_bytes(const air_geometry &g) {
    if (g.precision != AIR_PREC_BF16X3) return 0;
    const size_t kp = ((size_t)g.n_bins + 127) / 128 * 128;   // split Y; both parities' T_far pieces
    return (size_t)g.n_views * 3 * kp * 2 + 3 * kp * kp + 1024;
}

// Least device bytes a plan of this geometry can do with (the pieces of
// carve, without orbits, and the filter's), to within alignment; needs no
// tables.
size_t plan_bytes_estimate(const air_geometry &g) {
    SliceDesc s{};
    s.n = g.n;
    s.V = g.n_views;
    s.nb = g.n_bins;
    const size_t nn = (size_t)g.n * g.n, rays = (size_t)g.n_views * g.n_bins;
    // the part buffer holds the autotuner's largest split, as carve sizes it
    const size_t parts = (size_t)std::min(g.n_views, 2 * choose_bwd_parts(s));
    size_t b = rays * (sizeof(RayFx) + 4) + (size_t)g.n_views * tiles_bwd_xy(s) * 4 + (size_t)g.n_bins * 4;
    b += nn * 4 * (7 + parts + 18 + 1);          // x r p q rhs0 g g', parts, b b2, xbuf
    b += (size_t)g.n * (g.n + 1) * 8 * 2;        // xp xt (pairs)
    b += (size_t)g.n_views * 8 + (size_t)g.n_bins * 8;   // FBP tables
    b += rays * 4 * 3;                           // z zc ybuf
    b += sizeof(CgState) + ((size_t)max_reduce_tiles(s) + 64) * 8 + 24 * 256;
    return b + filter_bytes(g);
}
}  // namespace air

namespace {
long long floor_div(long long a, long long b) {   // b > 0
    long long q = a / b;
    return (a % b != 0 && a < 0) ? q - 1 : q;
}
long long ceil_div(long long a, long long b) {    // b > 0
    return -floor_div(-a, b);
}
}  // namespace

// The fixed-point form of the line through (px, py) with unit direction
// (ux, uy), pixel units with the origin at the image corner (see RayFx), and
// its walk word.
RayFx air::make_ray_fx(double px, double py, double ux, double uy, int n, unsigned *walk) {
    const double two32 = 4294967296.0;
    const bool cols = std::fabs(ux) >= std::fabs(uy);       // walk columns
    const double a = cols ? px : py, b = cols ? py : px;    // along / across the walk
    const double ua = cols ? ux : uy, ub = cols ? uy : ux;
    const double m = ub / ua;                               // |m| <= 1
    const double y0 = b - a * m;                            // across-coordinate at walk-coordinate 0
    long long M = std::llround(m * two32);
    const long long mmax = (1ll << 32) - 1;
    if (M > mmax) M = mmax;
    if (M < -mmax) M = -mmax;
    if (M == 0) M = 1;        // an exactly axis-parallel ray, tilted by 2^-32
    const long long Y0 = std::llround(y0 * two32);
    RayFx r{};
    r.Mlo = (unsigned)(M & 0xffffffffll);
    r.L0 = Y0 + (M < 0 ? M : 0);
    const unsigned Ma = (unsigned)(M < 0 ? -M : M);
    const float c = (float)((1.0 / std::fabs(ua)) / (double)Ma);
    r.cs = M < 0 ? -c : c;
    // walk range: columns k in [0, n) whose span [lo, lo + Ma] meets rows [0, n)
    const long long N2 = (long long)n << 32;
    long long ks, ke;
    if (M > 0) {
        ks = floor_div(-r.L0 - (long long)Ma, M) + 1;       // hi(k) > 0
        ke = ceil_div(N2 - r.L0, M);                        // lo(k) < N2
    } else {
        const long long Mp = -M;
        ks = floor_div(r.L0 - N2, Mp) + 1;                  // lo(k) < N2
        ke = ceil_div(r.L0 + (long long)Ma, Mp);            // hi(k) > 0
    }
    // clamp to [0, n] before packing: a ray that misses the image can give a
    // start column far outside it (the walk word holds 16 and 15 bits)
    ks = std::min<long long>(std::max<long long>(ks, 0), n);
    ke = std::min<long long>(std::max<long long>(ke, ks), n);
    auto meets = [&](long long k) {
        const long long lo = r.L0 + k * M;
        return lo + (long long)Ma > 0 && lo < N2;
    };
    while (ks < ke && !meets(ks)) ++ks;
    while (ke > ks && !meets(ke - 1)) --ke;
    *walk = ray_walk((int)ks, (int)ke, cols);
    return r;
}

// ------------------------------------------------------------ autotuner
// The projector's tile shape (views per block) and the backprojector's view
// split are timed on the plan's own workspace (the kernels' work does not
// depend on the data) and the fastest kept; results are cached per geometry
// for the life of the process, so every plan of a geometry uses the same
// configuration.  The general pair is timed without launch overlap, each kernel
// by itself; the orbit backprojector with it, as the solver runs it.
namespace {
struct TuneKey {
    int n, V, nb, orb;
    double dx, dso, dg, beta0, arc;
    bool operator<(const TuneKey &o) const {
        return std::memcmp(this, &o, sizeof(TuneKey)) < 0;
    }
};
struct Tuned {
    int vpb, parts, splits;   // general projector and backprojector; orbit backprojector
};
std::mutex g_tune_mu;
std::map<TuneKey, Tuned> g_tune_cache;
}  // namespace

namespace air {
air_status autotune(air_plan *P) {
    SliceDesc &s = P->desc;
    TuneKey key;
    std::memset(&key, 0, sizeof(key));
    key.n = s.n;
    key.V = s.V;
    key.nb = s.nb;
    key.orb = s.orb;
    key.dx = P->geom.pixel_mm;
    key.dso = P->geom.dso_mm;
    key.dg = fan_pitch(P->geom);
    key.beta0 = P->geom.beta0;
    key.arc = P->geom.arc;
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            s.fwd_vpb = it->second.vpb;
            s.bwd_parts = std::min(it->second.parts, P->bwd_parts_max);
            s.orb_splits = std::min(it->second.splits, std::max(1, P->bwd_parts_max / 8));
            return AIR_OK;
        }
    }
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.x, 0, (size_t)s.n * s.n * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s.z, 0, (size_t)s.V * s.nb * 4, st);
    auto timed = [&](auto &&launch) -> float {
        if (e != cudaSuccess) return 1e30f;
        launch();                                   // warm-up
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) launch();
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        float ms = 1e30f;
        if (e == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    // projector: views per block, from the most down; a smaller tile is
    // kept only if it is 2 % faster (within that, grouped batches run the
    // taller tiles a little faster)
    SliceDesc t = s;
    t.orb = 0;
    t.ext_in = s.x;
    t.ext_out = s.z;
    int best_vpb = 1;
    float best = 1e30f;
    for (int vpb : {8, 4, 2, 1}) {
        if (vpb > s.V) continue;
        t.fwd_vpb = vpb;
        const float ms = timed([&] {
            if (e == cudaSuccess) e = launch_op(OP_TRANSPOSE, t, SRC_EXT, st, false);
            if (e == cudaSuccess) e = launch_op(OP_FWD, t, SRC_EXT, st, false);
        });
        if (ms < best * 0.98f) {
            best = ms;
            best_vpb = vpb;
        }
    }
    // backprojector: view splits up to the part buffer's size, timed as the
    // solver runs them (the parts, then their sum, OP_BWD_FIN, which the CG
    // epilogue needs at any split); the heuristic's choice is tried first
    // and kept unless another is 2 % faster
    if (e == cudaSuccess) e = cudaMemsetAsync(s.zc, 0, (size_t)s.V * s.nb * 4, st);
    const int S0 = s.bwd_parts, most = std::min(s.V, 2 * S0);
    int best_S = S0;
    best = 1e30f;
    for (int S : {S0, 1, 2, 3, 4, 6, 8, 12, 16}) {
        if (S > most || (S == S0 && best < 1e30f)) continue;
        t.bwd_parts = S;
        const float ms = timed([&] {
            if (e == cudaSuccess) e = launch_backprojection(t, BWD_RHS0, true, st, false);
        });
        if (ms < best * 0.98f) {
            best = ms;
            best_S = S;
        }
    }
    // orbit backprojector: splits of its segments, the fewest first; one more
    // is kept if it is 1 % faster, with the launches overlapped as the solver's
    // are (without, 350^2 / 200 views often took one at 26.5 us for 24.3)
    int best_split = 1;
    best = 1e30f;
    t.orb = s.orb;
    for (int S : {1, 2, 3, 4, 6, 8, 12, 16}) {
        if (!s.orb || 8 * S > P->bwd_parts_max) continue;
        t.orb_splits = S;
        const float ms = timed([&] {
            if (e == cudaSuccess) e = launch_backprojection(t, BWD_RHS0, true, st, true);
        });
        if (ms < best * 0.99f) {
            best = ms;
            best_split = S;
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    if (e != cudaSuccess) return fail(AIR_ERR_CUDA, std::string("autotuning: ") + cudaGetErrorString(e));
    s.fwd_vpb = best_vpb;
    s.bwd_parts = best_S;
    s.orb_splits = best_split;
    std::lock_guard<std::mutex> lock(g_tune_mu);
    g_tune_cache[key] = {best_vpb, best_S, best_split};
    return AIR_OK;
}
}  // namespace air

// ------------------------------------------------------------ geometry tables
// The host-side tables of a geometry (FP64 arithmetic, stored as the device
// formats), cached per geometry for the process: plans of one geometry (a
// batch, the server's pool) share one computation.
namespace {
struct HostTables {
    std::vector<RayFx> ray;
    std::vector<unsigned> walk;
    std::vector<unsigned> vt;
    std::vector<float> taps, fbw, fbt;
    std::vector<float2> fview;
    float ramp_diag = 0.f, fbp_diag = 0.f;
    OrbitTables orb;
    FbpOrbits fbp;
    std::vector<float2> fbp_c;
    // the tables as a plan holds them, one behind the other, for one upload
    mutable std::once_flag packed;
    mutable std::vector<char> blob;
};

air_status build_tables(const air_geometry &g, double dg, int ntxy, HostTables &T) {
    const int n = g.n, V = g.n_views, nb = g.n_bins;
    const size_t rays = (size_t)V * nb;
    // geometry tables, computed in FP64: per view the source (pixel units,
    // centred) and the central-ray direction; per ray the fixed-point line
    std::vector<RayFx> &hray = T.ray;
    std::vector<unsigned> &hwalk = T.walk;
    hray.resize(rays);
    hwalk.resize(rays);
    struct ViewSrc { double x, y, z, w; };   // source (pixel units, centred), central direction
    std::vector<ViewSrc> hsrc(V);
    std::vector<float> &htaps = T.taps;
    htaps.resize(nb);
    const double inv_dx = 1.0 / g.pixel_mm;
    for (int v = 0; v < V; ++v) {
        const double beta = g.beta0 + g.arc * (double)v / (double)V;
        const double cb = std::cos(beta), sb = std::sin(beta);
        const double Sx = g.dso_mm * cb, Sy = g.dso_mm * sb;
        hsrc[v] = ViewSrc{Sx * inv_dx, Sy * inv_dx, -cb, -sb};
        for (int j = 0; j < nb; ++j) {
            const double gamma = ((double)j - 0.5 * (nb - 1)) * dg;
            const double th = beta + M_PI + gamma;
            const double ux = std::cos(th), uy = std::sin(th);
            const double su = Sx * ux + Sy * uy;
            // closest point to the image centre, pixel units, origin at the image corner
            const double px = (Sx - su * ux) * inv_dx + 0.5 * n, py = (Sy - su * uy) * inv_dx + 0.5 * n;
            hray[(size_t)v * nb + j] = make_ray_fx(px, py, ux, uy, n, &hwalk[(size_t)v * nb + j]);
        }
    }
    // the projector walks [k0, k1) without bounds checks (the image copies
    // it reads are padded by one entry per row end): every walked column must
    // lie in the image and its span start in rows [-1, n-1]
    for (size_t i = 0; i < rays; ++i) {
        const RayFx &r = hray[i];
        const int k0 = walk_k0(hwalk[i]), k1 = walk_k1(hwalk[i]);
        bool ok = 0 <= k0 && k0 <= k1 && k1 <= n;
        for (int k : {k0, k1 - 1}) {
            if (!ok || k0 == k1) break;
            const long long r0 = (r.L0 + (long long)k * ray_M(r)) >> 32;
            ok = r0 >= -1 && r0 <= n - 1;
        }
        if (!ok) return fail(AIR_ERR_INTERNAL, "ray table: a walk range leaves the image");
    }
    // backprojector ray ranges: per view and 32 x 32 pixel tile, the rays
    // whose fan angle lies between the extreme fan angles of the tile's
    // corners (the tile is convex and the source outside it, so exactly
    // these rays can meet it), widened by 0.02 bin; and whether they all walk
    // the same way with slopes of one sign.  Fan angles at the corner grid
    // are shared by neighbouring tiles.
    const int tpr = (n + BWD_T - 1) / BWD_T;
    std::vector<unsigned> &hvt = T.vt;
    hvt.assign((size_t)V * ntxy, 0u);
    {
        std::vector<double> gam((size_t)(tpr + 1) * (tpr + 1));
        std::vector<int> chg(nb);   // number of changes of orientation or slope sign among rays 0..j
        const double jm = 0.5 * (nb - 1);
        for (int v = 0; v < V; ++v) {
            const ViewSrc w = hsrc[v];
            for (int iy = 0; iy <= tpr; ++iy)
                for (int ix = 0; ix <= tpr; ++ix) {
                    const double px = std::min(ix * BWD_T, n) - 0.5 * n, py = std::min(iy * BWD_T, n) - 0.5 * n;
                    const double dxs = px - w.x, dys = py - w.y;
                    gam[(size_t)iy * (tpr + 1) + ix] = std::atan2(w.z * dys - w.w * dxs, w.z * dxs + w.w * dys);
                }
            const RayFx *rv = hray.data() + (size_t)v * nb;
            const unsigned *wv = hwalk.data() + (size_t)v * nb;
            chg[0] = 0;
            for (int j = 1; j < nb; ++j)
                chg[j] = chg[j - 1] +
                         (walk_cols(wv[j]) != walk_cols(wv[j - 1]) || (rv[j].cs < 0.f) != (rv[j - 1].cs < 0.f));
            for (int ty = 0; ty < tpr; ++ty)
                for (int tx = 0; tx < tpr; ++tx) {
                    double gmin = 1e30, gmax = -1e30;
                    for (int cy = 0; cy < 2; ++cy)
                        for (int cx = 0; cx < 2; ++cx) {
                            const double gc = gam[(size_t)(ty + cy) * (tpr + 1) + tx + cx];
                            gmin = std::min(gmin, gc);
                            gmax = std::max(gmax, gc);
                        }
                    const double f0 = std::ceil(gmin / dg + jm - 0.02), f1 = std::floor(gmax / dg + jm + 0.02);
                    const int j0 = (int)std::max(0.0, std::min(f0, (double)nb));
                    const int j1 = (int)std::max(-1.0, std::min(f1, (double)nb - 1));   // inclusive
                    unsigned ent = vt_pack(0, 0, 0, false, false);
                    if (j1 >= j0)
                        ent = vt_pack(j0, j1 + 1, walk_cols(wv[j0]), rv[j0].cs < 0.f, chg[j1] != chg[j0]);
                    hvt[(size_t)(ty * tpr + tx) * V + v] = ent;
                }
        }
    }
    const double c0 = M_PI / ((double)V * g.pixel_mm * g.pixel_mm);
    double diag = 0.0;   // h[0] + 2 sum_{odd m < nb} h[m]: the difference form's centre weight
    for (int k = nb - 1; k >= 0; --k) {
        const double h = k == 0 ? 0.25 : (k % 2 ? -1.0 / (M_PI * M_PI * (double)k * (double)k) : 0.0);
        htaps[k] = (float)(c0 * h);
        diag += k == 0 ? h : 2.0 * h;
    }
    T.ramp_diag = (float)(c0 * diag);
    // fan-beam FBP (full scans): per view the central direction; per bin the
    // pre-weight cos gamma_j and the fan ramp alpha D g(m alpha), g(0) =
    // 1/(8 alpha^2), g(odd m) = -1/(2 pi^2 sin^2(m alpha)), g(even m) = 0
    std::vector<float2> &hfview = T.fview;
    std::vector<float> &hfbw = T.fbw, &hfbt = T.fbt;
    hfview.resize(V);
    hfbw.resize(nb);
    hfbt.resize(nb);
    for (int v = 0; v < V; ++v) {
        const double beta = g.beta0 + g.arc * (double)v / (double)V;
        hfview[v] = make_float2((float)(-std::cos(beta)), (float)(-std::sin(beta)));
    }
    double fdiag = 0.0;
    for (int k = nb - 1; k >= 0; --k) {
        const double gm = k == 0 ? 1.0 / (8.0 * dg * dg)
                                 : (k % 2 ? -1.0 / (2.0 * M_PI * M_PI * std::sin(k * dg) * std::sin(k * dg)) : 0.0);
        const double t = dg * g.dso_mm * gm;
        hfbt[k] = (float)t;
        fdiag += k == 0 ? t : 2.0 * t;
        hfbw[k] = (float)std::cos(((double)k - 0.5 * (nb - 1)) * dg);
    }
    T.fbp_diag = (float)fdiag;
    build_orbits(g, dg, T.orb);
    build_fbp_orbits(g, T.fbp);
    for (int v : T.fbp.base) T.fbp_c.push_back(hfview[v]);
    return AIR_OK;
}

struct GeomKey {
    int n, V, nb;
    double dx, dso, dg, beta0, arc;
    bool operator<(const GeomKey &o) const { return std::memcmp(this, &o, sizeof(GeomKey)) < 0; }
};
std::mutex g_tables_mu;
std::map<GeomKey, std::shared_ptr<const HostTables>> g_tables;
constexpr size_t TABLE_CACHE_MAX = 16;

air_status geometry_tables(const air_geometry &g, double dg, int ntxy, std::shared_ptr<const HostTables> *out) {
    GeomKey key;
    std::memset(&key, 0, sizeof(key));
    key.n = g.n;
    key.V = g.n_views;
    key.nb = g.n_bins;
    key.dx = g.pixel_mm;
    key.dso = g.dso_mm;
    key.dg = dg;
    key.beta0 = g.beta0;
    key.arc = g.arc;
    {
        std::lock_guard<std::mutex> lock(g_tables_mu);
        auto it = g_tables.find(key);
        if (it != g_tables.end()) {
            *out = it->second;
            return AIR_OK;
        }
    }
    auto T = std::make_shared<HostTables>();
    air_status st = build_tables(g, dg, ntxy, *T);
    if (st != AIR_OK) return st;
    std::lock_guard<std::mutex> lock(g_tables_mu);
    if (g_tables.size() >= TABLE_CACHE_MAX) g_tables.erase(g_tables.begin());
    g_tables[key] = T;
    *out = T;
    return AIR_OK;
}
// A plan's one allocation: the pieces that its descriptor points to.
struct Piece { void **dst; size_t bytes; const void *src = nullptr; size_t off = 0; };
struct Carve {
    SliceDesc s{};
    float *ybuf = nullptr, *xbuf = nullptr;
    std::vector<Piece> pieces;          // dst: pointers in here, which is not copied
    size_t total = 0, tables_end = 0, zero_end = 0;
    int parts_max = 1;                  // images the part buffer holds

    // orbits: with the tables and buffers of the scan's orbits, where it has them
    Carve(const air_geometry &g, const HostTables &T, bool orbits);
    Carve(const Carve &) = delete;
};

Carve::Carve(const air_geometry &g, const HostTables &T, bool orbits) {
    const int n = g.n, V = g.n_views, nb = g.n_bins;
    const size_t nn = (size_t)n * n, rays = (size_t)V * nb;
    s.n = n;
    s.V = V;
    s.nb = nb;
    s.half_n = 0.5f * n;
    s.dx = (float)g.pixel_mm;
    s.filter = g.filter;
    s.fwd_vpb = 1;
    s.bwd_parts = choose_bwd_parts(s);
    static const OrbitTables none;
    const OrbitTables &O = orbits ? T.orb : none;
    const int sms = sm_count();
    // the autotuner may pick up to twice the heuristic's view split; the
    // orbit backprojector's splits write eight images each
    parts_max = std::min(V, 2 * s.bwd_parts);
    if (O.nf) parts_max = std::max(parts_max, 8 * orb_splits_max(n, O.nf, sms));
    s.orb = O.nf;
    s.orb_splits = 1;
    s.orb_ntask = (int)O.task.size();
    s.orb_nseg = (int)O.seg.size();
    s.orb_npad = (int)O.bray.size();
    s.orb_ks = choose_orb_ks(s.orb_ntask, sms);
    for (int p = 0; p < 8; ++p) s.orb_frame[p] = O.frame[p];
    const size_t npad = (size_t)n * (n + 1) * 2;   // pair copies of the projector's input (floats)
    const size_t nstack = O.nf ? (size_t)2 * n * orb_ld(n) : 0;
    const size_t nz = O.bray.size() * orb_planes(s);
    const size_t npart = (size_t)max_reduce_tiles(s) + 64;
    auto table = [](auto **dst, const auto &v) { return Piece{(void **)dst, v.size() * sizeof(v[0]), v.data()}; };
    pieces = {
        // the tables; the orbits' last, so that a plan without them takes the same blob's front
        table(&s.ray, T.ray), table(&s.walk, T.walk), table(&s.vt, T.vt), table(&s.taps, T.taps), table(&s.fview, T.fview),
        table(&s.fbp_w, T.fbw), table(&s.fbp_taps, T.fbt), table(&s.fbp_c, T.fbp_c), table(&s.fbp_view, T.fbp.view),
        table(&s.orb_seg, O.seg), table(&s.orb_ray, O.ray), table(&s.orb_info, O.info), table(&s.orb_ent, O.ent),
        table(&s.orb_task, O.task), table(&s.orb_tile0, O.tile0), table(&s.orb_bray, O.bray), table(&s.orb_zmap, O.zmap),
        // zeroed once: the image copies' pads and the empty rays' samples stay zero
        {(void **)&s.xp, npad * 4}, {(void **)&s.xt, npad * 4}, {(void **)&s.orb_stack, nstack * sizeof(float4)},
        {(void **)&s.orb_z, nz * sizeof(float4)}, {(void **)&s.cg, sizeof(CgState)},
        // workspace
        {(void **)&s.bwd_part, (size_t)parts_max * nn * 4},
        {(void **)&s.x, nn * 4}, {(void **)&s.r, nn * 4}, {(void **)&s.p, nn * 4}, {(void **)&s.q, nn * 4},
        {(void **)&s.rhs0, nn * 4}, {(void **)&s.g, nn * 4}, {(void **)&s.g2, nn * 4}, {(void **)&s.b, 9 * nn * 4},
        {(void **)&s.b2, 9 * nn * 4}, {(void **)&s.z, rays * 4}, {(void **)&s.zc, rays * 4}, {(void **)&ybuf, rays * 4},
        {(void **)&xbuf, nn * 4}, {(void **)&s.partial, npart * sizeof(double)}};
    for (auto &pc : pieces) {
        pc.off = align_up(total, 256);
        total = pc.off + pc.bytes;
        if (pc.src) tables_end = total;
        if (pc.dst == (void **)&s.cg) zero_end = total;
    }
    total = align_up(total, 256);
}
}  // namespace

// A plan with or without orbits, in at most `limit` device bytes.
static air_status plan_attempt(const air_geometry &g, const HostTables &T, bool orbits, size_t limit, air_plan *P) {
    const double dg = fan_pitch(g);
    Carve C(g, T, orbits);
    std::call_once(T.packed, [&] {
        const Carve F(g, T, true);
        T.blob.assign(F.tables_end, 0);
        for (auto &pc : F.pieces)
            if (pc.src && pc.bytes) std::memcpy(T.blob.data() + pc.off, pc.src, pc.bytes);
    });
    const size_t need = C.total + filter_bytes(g);
    if (C.s.orb && need > limit)
        return fail(AIR_ERR_OOM, "the plan needs " + std::to_string(need) + " bytes of " + std::to_string(limit));
    char *mem = nullptr;
    if (cudaMalloc(&mem, C.total) != cudaSuccess) {
        cudaGetLastError();
        return fail(AIR_ERR_OOM, "cudaMalloc of the plan workspace failed (" + std::to_string(C.total) + " bytes)");
    }
    for (auto &pc : C.pieces) *pc.dst = mem + pc.off;
    SliceDesc &s = C.s;

    s.ramp_diag = T.ramp_diag;
    s.fbp_diag = T.fbp_diag;
    s.dso_px = (float)(g.dso_mm / g.pixel_mm);
    s.inv_dg = (float)(1.0 / dg);
    s.inv_dg_lo = (float)(1.0 / dg - (double)s.inv_dg);
    s.jmid = 0.5f * (g.n_bins - 1);
    s.fbp_scale = (float)(g.arc / (double)g.n_views / (g.pixel_mm * g.pixel_mm));
    cudaError_t e = cudaMemcpy(mem, T.blob.data(), C.tables_end, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(mem + C.tables_end, 0, C.zero_end - C.tables_end);
    if (e != cudaSuccess) {
        cudaFree(mem);
        return fail(AIR_ERR_CUDA, std::string("plan table upload: ") + cudaGetErrorString(e));
    }
    choose_fbp(s, T.fbp, s.bwd_part, C.parts_max, sm_count());
    s.y = C.ybuf;
    s.mu = 1.f;
    s.tau = 0.f;
    P->geom = g;
    P->desc = s;
    P->mem = mem;
    P->bytes = C.total;
    P->bwd_parts_max = C.parts_max;
    P->ybuf = C.ybuf;
    P->xbuf = C.xbuf;
    cudaGetDevice(&P->device);
    if (g.precision == AIR_PREC_BF16X3) {
        air_status st = ramp_tc_create(P);
        if (st != AIR_OK) {
            cudaFree(mem);
            P->mem = nullptr;
            return st;
        }
    }
    // The clears above are asynchronous to the host, and the first call on the
    // plan may come on a stream that does not wait for theirs: its results
    // would be cleared from under it.
    e = cudaStreamSynchronize(nullptr);
    air_status st = e == cudaSuccess ? autotune(P)
                                     : fail(AIR_ERR_CUDA, std::string("plan table upload: ") + cudaGetErrorString(e));
    if (st == AIR_OK) st = noalloc_prepare();
    if (st != AIR_OK) {
        ramp_tc_destroy(P);
        cudaFree(mem);
        P->mem = nullptr;
        return st;
    }
    return AIR_OK;
}

// Orbits cost a plan memory (68 -> 104 MB at 512^2 / 800 views): one that does
// not fit the limit, or the device, with them is made without.
static air_status plan_build(const air_geometry &g, size_t limit, air_plan *P) {
    SliceDesc s{};
    s.n = g.n;
    std::shared_ptr<const HostTables> T;
    if (air_status st = geometry_tables(g, fan_pitch(g), tiles_bwd_xy(s), &T); st != AIR_OK) return st;
    const air_status st = plan_attempt(g, *T, true, limit, P);
    return st == AIR_ERR_OOM && T->orb.nf ? plan_attempt(g, *T, false, limit, P) : st;
}

// Device bytes of the plan that plan_create makes under this limit; builds the
// geometry's tables (which plan_create then finds).  0: they cannot be built.
size_t air::plan_bytes(const air_geometry &g, size_t limit) {
    SliceDesc s{};
    s.n = g.n;
    std::shared_ptr<const HostTables> T;
    if (geometry_tables(g, fan_pitch(g), tiles_bwd_xy(s), &T) != AIR_OK) return 0;
    const size_t b = Carve(g, *T, true).total + filter_bytes(g);
    return T->orb.nf && b > limit ? Carve(g, *T, false).total + filter_bytes(g) : b;
}

extern "C" const char *air_last_error(void) { return g_err.c_str(); }

extern "C" air_status air_plan_create(const air_geometry *geom, air_plan **out) {
    return plan_create(geom, SIZE_MAX, out);
}

air_status air::plan_create(const air_geometry *geom, size_t limit, air_plan **out) {
    if (!out) return fail(AIR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    air_status st = validate_geometry(geom);
    if (st != AIR_OK) return st;
    air_plan *P = new (std::nothrow) air_plan();
    if (!P) return fail(AIR_ERR_OOM, "host allocation failed");
    static std::atomic<uint64_t> ids{0};
    P->id = ++ids;
    st = plan_build(*geom, limit, P);
    if (st != AIR_OK) {
        delete P;
        return st;
    }
    *out = P;
    return AIR_OK;
}

extern "C" air_status air_plan_destroy(air_plan *P) {
    if (!P) return AIR_OK;
    batch_forget(P->id);
    ramp_tc_destroy(P);
    if (P->mem) cudaFree(P->mem);
    delete P;
    return AIR_OK;
}

extern "C" size_t air_plan_bytes(const air_plan *P) { return P ? P->bytes + P->tc_bytes : 0; }

extern "C" air_status air_plan_tune(air_plan *P, int fwd_views_per_block, int bwd_view_parts) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    const int v = fwd_views_per_block;
    if (v != 1 && v != 2 && v != 4 && v != 8) return fail(AIR_ERR_INVALID_ARG, "fwd_views_per_block must be 1, 2, 4 or 8");
    if (bwd_view_parts < 1 || bwd_view_parts > P->bwd_parts_max)
        return fail(AIR_ERR_INVALID_ARG, "bwd_view_parts must be in 1.." + std::to_string(P->bwd_parts_max));
    P->desc.fwd_vpb = v;
    // what air_plan_config reports of this plan; the general pair, which an
    // orbit plan's solves with history run, keeps its own split
    if (P->desc.orb) P->desc.orb_splits = std::max(1, bwd_view_parts / 8);
    else P->desc.bwd_parts = bwd_view_parts;
    return AIR_OK;
}

extern "C" air_status air_plan_config(const air_plan *P, int *fwd_views_per_block, int *bwd_view_parts,
                                      int *bwd_view_parts_max) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    if (fwd_views_per_block) *fwd_views_per_block = P->desc.fwd_vpb;
    if (bwd_view_parts) *bwd_view_parts = bwd_images(P->desc);
    if (bwd_view_parts_max) *bwd_view_parts_max = P->bwd_parts_max;
    return AIR_OK;
}

extern "C" air_status air_set_wait_budget(int64_t polls) {
    const long long v = polls < 0 ? -1ll : (long long)polls;
    cudaError_t e = set_barrier_budget(v);
    if (e == cudaSuccess) e = ramp_tc_set_wait_budget(v);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(AIR_ERR_CUDA, std::string("setting the wait budget: ") + cudaGetErrorString(e));
    }
    return AIR_OK;
}

extern "C" air_status air_plan_status(const air_plan *P) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    const int st = ramp_tc_status(P);
    if (st == (int)AIR_ERR_TIMEOUT) return fail(AIR_ERR_TIMEOUT, "a bounded wait in the tensor-core filter gave up");
    if (st != 0) return fail(AIR_ERR_CUDA, "reading the plan status failed");
    return AIR_OK;
}

// ------------------------------------------------------- stand-alone ops
#define TRY(expr)                                   \
    do {                                            \
        air_status st_ = (expr);                    \
        if (st_ != AIR_OK) return st_;              \
    } while (0)
#define CUDA_TRY(expr)                                                                           \
    do {                                                                                         \
        cudaError_t e_ = (expr);                                                                 \
        if (e_ != cudaSuccess) return fail(AIR_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// The FP32 filter puts its results where the orbit backprojector reads them;
// behind the tensor-core filter OP_ORB_ZPACK does (its epilogue's scattered
// stores took longer: 2.52 against 2.41 ms for two outer steps of five CG steps
// at 512^2 / 800 views).
static bool filter_packs(const air_plan *P, const SliceDesc &s) {
    return s.orb && !(P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK);
}
static size_t img_bytes(const air_plan *P) { return (size_t)P->geom.n * P->geom.n * 4; }
static size_t sino_bytes(const air_plan *P) { return (size_t)P->geom.n_views * P->geom.n_bins * 4; }

namespace air {
// Z = C Y into dst (plan precision), from src (device); pack: into the orbits'
// packed samples (FP32 filter; dst is not written).
air_status apply_filter(const air_plan *P, const SliceDesc &base, const float *src, float *dst, bool pack,
                        cudaStream_t st) {
    if (P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK)
        return ramp_tc_apply(P, src, nullptr, dst, base.cg, 0, st);
    SliceDesc s = base;
    s.ext_in = src;
    s.ext_out = dst;
    CUDA_TRY(launch_op(OP_RAMP, s, RSRC_EXT | (pack ? ARG_PACK : 0), st));
    return AIR_OK;
}
}  // namespace air

extern "C" air_status air_project(const air_plan *P, const float *X, float *Y, air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(X, "X"));
    TRY(check_dev_ptr(Y, "Y"));
    if (overlap(X, img_bytes(P), Y, sino_bytes(P))) return fail(AIR_ERR_INVALID_ARG, "X and Y overlap");
    SliceDesc s = P->desc;
    s.ext_in = X;
    s.ext_out = Y;
    CUDA_TRY(launch_op(s.orb ? OP_ORB_PACK : OP_TRANSPOSE, s, SRC_EXT, (cudaStream_t)stream));
    CUDA_TRY(launch_op(s.orb ? OP_ORB_FWD : OP_FWD, s, SRC_EXT, (cudaStream_t)stream));
    return AIR_OK;
}

extern "C" air_status air_filter(const air_plan *P, const float *Y, float *Z, air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(Z, "Z"));
    if (overlap(Y, sino_bytes(P), Z, sino_bytes(P))) return fail(AIR_ERR_INVALID_ARG, "Y and Z overlap");
    return apply_filter(P, P->desc, Y, Z, false, (cudaStream_t)stream);
}

extern "C" air_status air_backproject(const air_plan *P, const float *Y, float *X, air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    if (overlap(X, img_bytes(P), Y, sino_bytes(P))) return fail(AIR_ERR_INVALID_ARG, "X and Y overlap");
    SliceDesc s = P->desc;
    s.ext_in = Y;
    s.ext_out = X;
    CUDA_TRY(launch_backprojection(s, BWD_PLAIN, false, (cudaStream_t)stream));
    return AIR_OK;
}

extern "C" air_status air_filtered_backproject(const air_plan *P, const float *Y, float *X,
                                               air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    if (overlap(X, img_bytes(P), Y, sino_bytes(P))) return fail(AIR_ERR_INVALID_ARG, "X and Y overlap");
    const cudaStream_t st = (cudaStream_t)stream;
    const bool packed = filter_packs(P, P->desc);
    TRY(apply_filter(P, P->desc, Y, P->desc.zc, packed, st));
    SliceDesc s = P->desc;
    s.ext_in = P->desc.zc;
    s.ext_out = X;
    CUDA_TRY(launch_backprojection(s, BWD_PLAIN, packed, st));
    return AIR_OK;
}

extern "C" air_status air_framelet(const air_plan *P, const float *in, float *out, int adjoint,
                                   air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(in, "in"));
    TRY(check_dev_ptr(out, "out"));
    const size_t bi = adjoint ? 9 * img_bytes(P) : img_bytes(P);
    const size_t bo = adjoint ? img_bytes(P) : 9 * img_bytes(P);
    if (overlap(in, bi, out, bo)) return fail(AIR_ERR_INVALID_ARG, "in and out overlap");
    SliceDesc s = P->desc;
    s.ext_in = in;
    s.ext_out = out;
    CUDA_TRY(launch_op(adjoint ? OP_FRAMELET_T : OP_FRAMELET, s, 0, (cudaStream_t)stream));
    return AIR_OK;
}

extern "C" air_status air_shrink(const air_plan *P, const float *X, float *b, float *g, float thresh,
                                 double *resid, air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    TRY(check_dev_ptr(X, "X"));
    TRY(check_dev_ptr(b, "b"));
    TRY(check_dev_ptr(g, "g"));
    if (resid) TRY(check_dev_ptr(resid, "resid"));
    if (!(thresh >= 0.f) || !std::isfinite(thresh)) return fail(AIR_ERR_INVALID_ARG, "thresh must be >= 0");
    const size_t ib = img_bytes(P);
    if (overlap(X, ib, b, 9 * ib) || overlap(X, ib, g, ib) || overlap(b, 9 * ib, g, ib))
        return fail(AIR_ERR_INVALID_ARG, "X, b and g must not overlap");
    const cudaStream_t st = (cudaStream_t)stream;
    SliceDesc s = P->desc;
    s.ext_in = X;
    s.ext_out = b;
    s.ext_out2 = g;
    s.tau = thresh;
    s.ext_scalar = resid;
    s.resid_out = nullptr;
    CUDA_TRY(launch_op(OP_SHRINK, s, 2, st));
    CUDA_TRY(cudaMemcpyAsync(b, P->desc.b2, 9 * ib, cudaMemcpyDeviceToDevice, st));
    return AIR_OK;
}

// ------------------------------------------------------------------ solve
namespace air {

// The split-Bregman program of one slice (Methods, Eq. 5 and ref. [24]).
// Each outer step's CG restarts from the residual the previous CG left,
// corrected for the change of the right-hand side (OP_RESTART): CG keeps
// r = b - M X, and b changes between outer steps only by mu (g_new - g_old).
// zpack_slot, cg_b_slot: a program without OP_ORB_ZPACK or OP_CG_B keeps its
// place free (batch_programs).
std::vector<Phase> solve_program(int n_outer, int n_cg, bool tc_ramp, bool orb, bool zpack_slot, bool cg_b_slot) {
    std::vector<Phase> prog;
    const int ramp = tc_ramp ? OP_RAMP_TC : OP_RAMP, pack = orb && !tc_ramp ? ARG_PACK : 0;
    const int copies = orb ? OP_ORB_PACK : OP_TRANSPOSE, fwd = orb ? OP_ORB_FWD : OP_FWD;
    auto push_bwd = [&](int mode) {
        if (orb && tc_ramp) prog.push_back({OP_ORB_ZPACK, mode});
        else if (zpack_slot) prog.push_back({OP_NOP, 0});
        prog.push_back({orb ? OP_ORB_BWD : OP_BWD, mode});
    };
    prog.push_back({ramp, RSRC_Y | pack});   // zc = C y
    push_bwd(BWD_RHS0);                      // rhs0 = A^T zc
    prog.push_back({OP_BWD_FIN, BWD_RHS0});
    prog.push_back({OP_ZERO, 0});            // X = 0, b = 0, g = g' = 0
    prog.push_back({OP_RESTART, -1});        // r = p = rhs0 (X = 0, g = 0)
    for (int k = 0; k < n_outer; ++k) {
        for (int i = 0; i < n_cg; ++i) {
            const int swap = orb && (i & 1) ? ARG_SWAP : 0;                       // see ARG_SWAP
            prog.push_back({copies, (orb && i > 0 ? SRC_P_NEXT : SRC_P) | swap});   // q = M p
            prog.push_back({fwd, SRC_P});
            prog.push_back({ramp, RSRC_Z | pack});
            push_bwd(BWD_Q);
            prog.push_back({OP_BWD_FIN, BWD_Q | swap});
            prog.push_back({OP_CG_A, swap});
            if (!orb) prog.push_back({OP_CG_B, 0});
            else if (cg_b_slot) prog.push_back({OP_NOP, 0});
        }
        prog.push_back({OP_SHRINK, k & 1});
        if (k + 1 < n_outer) prog.push_back({OP_RESTART, k & 1});   // r += mu (g_k - g_{k-1})
    }
    return prog;
}

// The programs of a batch, phase for phase: slices on different paths or with
// different filters keep each other's extra phases free, so that they meet in
// the operators they share (30 x 8 steps, FP32 and BF16X3 slices with orbits:
// 1745 grouped launches; phase by phase as they come, 3008).
std::vector<std::vector<Phase>> batch_programs(const std::vector<SolveForm> &forms) {
    bool zpack = false, cg_b = false;
    for (const SolveForm &f : forms) {
        zpack |= f.orb && f.tc_ramp;
        cg_b |= !f.orb;
    }
    std::vector<std::vector<Phase>> out;
    for (const SolveForm &f : forms) out.push_back(solve_program(f.n_outer, f.n_cg, f.tc_ramp, f.orb, zpack, cg_b));
    return out;
}

// L2-regularised AIR, Eq. (5): (A'^T A + lambda I) X = A'^T Y by n_cg CG steps
// from X = 0 (the first L2 step of the split-Bregman program with g = 0 and
// mu = lambda, without the shrink).
std::vector<Phase> l2_program(int n_cg, bool tc_ramp, bool orb) {
    std::vector<Phase> prog = solve_program(1, n_cg, tc_ramp, orb);
    prog.pop_back();   // the SHRINK of the outer step
    return prog;
}

// Forward-backward splitting AIR: per iteration the forward step of Eq. (6),
// q = X + step A'^T (Y - A X) in the backprojection's epilogue, then the
// framelet proximal step.
std::vector<Phase> fbs_program(int n_iter, bool tc_ramp, bool orb) {
    std::vector<Phase> prog;
    const int ramp = tc_ramp ? OP_RAMP_TC : OP_RAMP, pack = orb && !tc_ramp ? ARG_PACK : 0;
    const int copies = orb ? OP_ORB_PACK : OP_TRANSPOSE, fwd = orb ? OP_ORB_FWD : OP_FWD;
    auto push_bwd = [&](int mode) {
        if (orb && tc_ramp) prog.push_back({OP_ORB_ZPACK, mode});
        prog.push_back({orb ? OP_ORB_BWD : OP_BWD, mode});
    };
    prog.push_back({ramp, RSRC_Y | pack});
    push_bwd(BWD_RHS0);
    prog.push_back({OP_BWD_FIN, BWD_RHS0});
    prog.push_back({OP_ZERO, 0});
    for (int k = 0; k < n_iter; ++k) {
        prog.push_back({copies, SRC_X});
        prog.push_back({fwd, SRC_X});
        prog.push_back({ramp, RSRC_Z | pack});
        push_bwd(BWD_STEP);
        prog.push_back({OP_BWD_FIN, BWD_STEP});
        prog.push_back({OP_PROX, 0});
    }
    return prog;
}

air_status run_program_single(const air_plan *P, const SliceDesc &s, const std::vector<Phase> &prog,
                              cudaStream_t st) {
    for (const Phase &ph : prog) {
        if (ph.op == OP_RAMP_TC) {
            const bool meas = ph.arg == RSRC_Y;
            TRY(ramp_tc_apply(P, meas ? s.y : s.z, nullptr, s.zc, s.cg, !meas, st));
        } else {
            CUDA_TRY(launch_op(ph.op, s, ph.arg, st));
        }
    }
    return AIR_OK;
}

air_status check_solve_args(const air_plan *P, const float *Y, float lambda, float mu, int n_outer,
                            int n_cg, const float *X) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    if (!(mu > 0.f) || !std::isfinite(mu)) return fail(AIR_ERR_INVALID_ARG, "mu must be > 0");
    if (!(lambda >= 0.f) || !std::isfinite(lambda)) return fail(AIR_ERR_INVALID_ARG, "lambda must be >= 0");
    if (n_outer < 0 || n_cg < 0 || n_outer > 100000 || n_cg > 100000)
        return fail(AIR_ERR_INVALID_ARG, "n_outer and n_cg must be in 0..100000");
    if (Y && X && overlap(X, img_bytes(P), Y, sino_bytes(P)))
        return fail(AIR_ERR_INVALID_ARG, "X and Y overlap");
    return AIR_OK;
}

SliceDesc solve_desc(const air_plan *P, const float *Y, float lambda, float mu, float *X, double *resid) {
    SliceDesc s = P->desc;
    s.y = Y;
    s.x = X;
    s.mu = mu;
    s.tau = lambda / mu;
    s.resid_out = resid;
    // The residual history keeps one summation order, that of the general pair:
    // the orbit pair would move its FP64 values by 1e-8, and takes half the time
    // (a 30 x 8 split-BF16 solve at 512^2 / 800 views: 96 ms with history, 49
    // without).
    if (resid) s.orb = 0;
    return s;
}

}  // namespace air

extern "C" air_status air_solve(const air_plan *P, const float *Y, float lambda, float mu, int n_outer,
                                int n_cg, float *X, double *resid, air_stream stream) {
    TRY(check_solve_args(P, Y, lambda, mu, n_outer, n_cg, X));
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    if (resid) TRY(check_dev_ptr(resid, "resid"));
    const bool tc = P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK;
    SliceDesc s = solve_desc(P, Y, lambda, mu, X, resid);
    return run_program_single(P, s, solve_program(n_outer, n_cg, tc, s.orb != 0), (cudaStream_t)stream);
}

extern "C" air_status air_solve_l2(const air_plan *P, const float *Y, float lambda, int n_cg, float *X,
                                   air_stream stream) {
    if (!(lambda > 0.f) || !std::isfinite(lambda)) return fail(AIR_ERR_INVALID_ARG, "lambda must be > 0");
    TRY(check_solve_args(P, Y, 0.f, lambda, 0, n_cg, X));
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    const bool tc = P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK;
    SliceDesc s = solve_desc(P, Y, 0.f, lambda, X, nullptr);
    return run_program_single(P, s, l2_program(n_cg, tc, P->desc.orb != 0), (cudaStream_t)stream);
}

extern "C" air_status air_solve_fbs(const air_plan *P, const float *Y, float lambda, float step, int n_iter,
                                    float *X, air_stream stream) {
    if (!(step > 0.f) || !std::isfinite(step)) return fail(AIR_ERR_INVALID_ARG, "step must be > 0");
    TRY(check_solve_args(P, Y, lambda, 1.f, n_iter, 0, X));
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    const bool tc = P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK;
    SliceDesc s = solve_desc(P, Y, 0.f, 1.f, X, nullptr);
    s.tau = step * lambda;      // the proximal threshold
    s.step = step;
    return run_program_single(P, s, fbs_program(n_iter, tc, P->desc.orb != 0), (cudaStream_t)stream);
}

extern "C" air_status air_fbp(const air_plan *P, const float *Y, float *X, air_stream stream) {
    if (!P) return fail(AIR_ERR_INVALID_ARG, "plan is NULL");
    if (std::fabs(P->geom.arc - 2.0 * M_PI) > 1e-9 * 2.0 * M_PI)
        return fail(AIR_ERR_INVALID_ARG, "FBP needs a full 2 pi scan");
    TRY(check_dev_ptr(Y, "Y"));
    TRY(check_dev_ptr(X, "X"));
    if (overlap(X, img_bytes(P), Y, sino_bytes(P))) return fail(AIR_ERR_INVALID_ARG, "X and Y overlap");
    const cudaStream_t st = (cudaStream_t)stream;
    SliceDesc f = P->desc;        // the filter: the ramp tile with the fan ramp and pre-weight
    f.filter = AIR_FILTER_RAMLAK;
    f.taps = f.fbp_taps;
    f.ramp_diag = f.fbp_diag;
    f.prew = f.fbp_w;
    f.ext_in = Y;
    f.ext_out = P->desc.zc;
    CUDA_TRY(launch_op(OP_RAMP, f, RSRC_EXT, st));
    SliceDesc b = P->desc;
    b.ext_out = X;
    if (!b.fbp_nf) {
        CUDA_TRY(launch_op(OP_FBP, b, 0, st));
        return AIR_OK;
    }
    CUDA_TRY(launch_op(OP_FBP_PACK, b, 0, st));
    CUDA_TRY(launch_op(OP_FBP_ORB, b, 0, st));
    b.orb = 0;                    // the sum of the orbits' images in a row, scaled
    b.bwd_parts = b.fbp_splits * b.fbp_nf;
    b.dx = b.fbp_scale;
    CUDA_TRY(launch_op(OP_BWD_FIN, b, BWD_PLAIN, st));
    return AIR_OK;
}

extern "C" air_status air_solve_host(const air_plan *P, const float *Y_host, float lambda, float mu,
                                     int n_outer, int n_cg, float *X_host, air_stream stream) {
    TRY(check_solve_args(P, nullptr, lambda, mu, n_outer, n_cg, nullptr));
    if (!Y_host || !X_host) return fail(AIR_ERR_INVALID_ARG, "Y_host and X_host must not be NULL");
    const cudaStream_t st = (cudaStream_t)stream;
    CUDA_TRY(cudaMemcpyAsync(P->ybuf, Y_host, sino_bytes(P), cudaMemcpyHostToDevice, st));
    const bool tc = P->geom.precision == AIR_PREC_BF16X3 && P->geom.filter == AIR_FILTER_RAMLAK;
    SliceDesc s = solve_desc(P, P->ybuf, lambda, mu, P->xbuf, nullptr);
    TRY(run_program_single(P, s, solve_program(n_outer, n_cg, tc, P->desc.orb != 0), st));
    CUDA_TRY(cudaMemcpyAsync(X_host, P->xbuf, img_bytes(P), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return tc ? air_plan_status(P) : AIR_OK;
}
