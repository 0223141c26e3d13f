// lb_engine.cu -- host-side engine shared by the single-lattice ABI and the
// lattice pool: parameter validation, device regions, TMA descriptors,
// model coefficients, lattice descriptors, the work partition and launch of
// the persistent step kernel, and the observe/initialise helpers.  Every
// step of the model runs in the kernels of lb_kernels.cu.
#include "lb_engine.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>

namespace lbgb {

constexpr size_t kAlign = 256;
size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Multi-range weights p(|d|^2) (8th-order isotropic, second moment 1/3) and
// the D2Q9 weights w(|d|^2), for the 12 pair representatives used by the
// kernels: (1,0) (0,1) (1,1) (-1,1) (2,0) (0,2) (2,1) (1,2) (-1,2) (-2,1)
// (2,2) (-2,2).
static double p_weight(int c2) {
    switch (c2) {
        case 1: return 4.0 / 63.0;
        case 2: return 4.0 / 135.0;
        case 4: return 1.0 / 180.0;
        case 5: return 2.0 / 945.0;
        case 8: return 1.0 / 15120.0;
    }
    return 0.0;
}
static double w_weight(int c2) { return c2 == 1 ? 1.0 / 9.0 : c2 == 2 ? 1.0 / 36.0 : 0.0; }

lb_status validate_params(const lb_params* p) {
    if (!p) return LB_ERR_INVALID;
    if (p->nx < 8 || p->ny < 8 || p->nx > (1 << 20) || p->ny > (1 << 19)) return LB_ERR_INVALID;
    if (p->boundary != LB_PERIODIC && p->boundary != LB_COUETTE) return LB_ERR_INVALID;
    if (p->precision < LB_FP64 || p->precision > LB_BF16_OFFSET) return LB_ERR_INVALID;
    if (p->psi_form != LB_PSI_SQRT_RHO0 && p->psi_form != LB_PSI_RHO0) return LB_ERR_INVALID;
    if (p->force_scheme != LB_FORCE_SHIFT && p->force_scheme != LB_FORCE_SOURCE) return LB_ERR_INVALID;
    if (!(p->tau_A > 0.5) || !(p->tau_B > 0.5) || !(p->rho0 > 0.0)) return LB_ERR_INVALID;
    if (p->stress_every < 1 || p->stress_t0 < 0) return LB_ERR_INVALID;
    if (p->rounding != LB_ROUND_NEAREST && p->rounding != LB_ROUND_STOCHASTIC) return LB_ERR_INVALID;
    if (p->tile_rows != 0 && p->tile_rows != 8 && p->tile_rows != 16) return LB_ERR_INVALID;
    if (p->tile_rows == 16 && p->precision == LB_FP64) return LB_ERR_INVALID;
    const double vals[] = {p->tau_A, p->tau_B, p->G_A1, p->G_A2, p->G_B1, p->G_B2, p->G_X,
                           p->rho0, p->u_wall, p->init_amp, p->rho_ref, p->g_x, p->kolmo_amp,
                           p->kolmo_k};
    for (double v : vals)
        if (!std::isfinite(v)) return LB_ERR_INVALID;
    if (p->init_amp < 0.0 || p->init_amp >= 1.0 || p->rho_ref < 0.0) return LB_ERR_INVALID;
    return LB_OK;
}

lb_status cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return LB_OK;
    cudaGetLastError();
    if (e == cudaErrorMemoryAllocation) return LB_ERR_NOMEM;
    return LB_ERR_CUDA;
}

int device_sms(int device) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
        sms = 1;
    return sms;
}

// L2 bytes of the current device (0 if unknown).
static long long device_l2_bytes() {
    int dev = 0, l2 = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) != cudaSuccess)
        return 0;
    return l2;
}

static Geom make_geom(const lb_params* p) {
    Geom g;
    const int prec = p->precision;
    const int es = kernel_elem_bytes(prec);
    const int gx = kernel_ghost_x(prec);
    // a row of pairs is 2 * pitch * es bytes: keep pitch * es a multiple of 16
    const int align_pairs = 16 / es;
    const int box_w = kernel_tile_x(prec) + 2 * gx;
    int pitch = (int)align_up((size_t)(p->nx + 2 * gx), (size_t)align_pairs);
    if (pitch < box_w) pitch = box_w;
    g.nx = p->nx;
    g.ny = p->ny;
    g.pitch = pitch;
    g.rows = p->ny + 2 * kGY;
    g.plane = (long long)g.rows * g.pitch;
    g.gx = gx;
    g.periodic = p->boundary == LB_PERIODIC ? 1 : 0;
    // the tile stores end at the last 16-byte boundary of a row's lattice part
    const int pair_bytes = 2 * es;
    g.x_tail = (p->nx + gx) * pair_bytes / 16 * 16 / pair_bytes - gx;
    return g;
}

// Device region of one lattice: stats, observe slots, wall columns, two
// buffers.
struct Region {
    size_t stats, slots, wallx, wsum, f0, f1, total, fbytes;
};
static Region region_layout(const lb_params* p) {
    Geom g = make_geom(p);
    const int tx = kernel_tile_x(p->precision), ty = kernel_tile_y(p->precision);
    const size_t ntiles = (size_t)((p->nx + tx - 1) / tx) * (size_t)((p->ny + ty - 1) / ty);
    Region r;
    size_t off = 0;
    r.stats = off;
    off = align_up(off + sizeof(DevStats), kAlign);
    r.slots = off;
    off = align_up(off + sizeof(double) * 4 * ntiles, kAlign);
    // the wall-momentum pair of every wall site (bottom row, then top row) of
    // two steps, in the compute precision
    r.wallx = off;
    off = align_up(off + (size_t)4 * (size_t)p->nx *
                             (p->precision == LB_FP64 ? sizeof(double2) : sizeof(float2)), kAlign);
    // their sums per strip (at most nx strips), bottom then top
    r.wsum = off;
    off = align_up(off + (size_t)2 * (size_t)p->nx * sizeof(double), kAlign);
    r.fbytes = align_up((size_t)18 * (size_t)g.plane * (size_t)kernel_elem_bytes(p->precision), kAlign);
    r.f0 = off;
    off += r.fbytes;
    r.f1 = off;
    off += r.fbytes;
    r.total = off;
    return r;
}

size_t lattice_bytes(const lb_params* p) { return region_layout(p).total; }

template <typename C>
static void fill_coef(Coef<C>& k, const lb_params* p) {
    const double Ga[2] = {p->G_A1, p->G_B1};
    const double Gr[2] = {p->G_A2, p->G_B2};
    // K(|d|^2) per species: attraction on the first belt (|d|^2 = 1, 2) with
    // the D2Q9 weights, repulsion on both belts with the weights p; the row
    // sums use K(1), K(2), K(5) and 2 K(4), 2 K(5), 2 K(8) (doubling is exact)
    const int c2s[6] = {1, 2, 5, 4, 5, 8};
    for (int r = 0; r < 6; ++r) {
        const int c2 = c2s[r];
        C K[2];
        for (int s = 0; s < 2; ++s)
            K[s] = (C)((c2 <= 2 ? Ga[s] * w_weight(c2) : 0.0) + Gr[s] * p_weight(c2));
        const C f = r < 3 ? C(1) : C(2);
        k.KC[r].x = K[0] * f;
        k.KC[r].y = K[1] * f;
    }
    const bool f64 = sizeof(C) == 8;
    k.WC[0].x = k.WC[0].y = f64 ? C(4) : (C)w_weight(1);
    k.WC[1].x = k.WC[1].y = f64 ? C(1) : (C)w_weight(2);
    // Offsets are taken from rho_ref rounded to the compute precision, so that
    // rho = rho_ref + sum_i h_i holds with the same rho_ref on every path.
    const double rref = (double)(C)(p->rho_ref > 0.0 ? p->rho_ref : p->rho0);
    const double pref = p->psi_form == LB_PSI_RHO0 ? p->rho0 : std::sqrt(p->rho0);
    k.gx_rho0 = (C)(p->G_X / p->rho0 * (f64 ? w_weight(2) : 1.0));
    k.rho_ref = (C)rref;
    k.psi_ref = (C)(pref * (1.0 - std::exp(-rref / p->rho0)));
    k.psi_scale = (C)(pref * std::exp(-rref / p->rho0));
    k.inv_rho0 = (C)(1.0 / p->rho0);
    k.exp_c = (C)(-64.0 / (M_LN2 * p->rho0));
    k.tau15[0] = (C)(1.5 * p->tau_A);
    k.tau15[1] = (C)(1.5 * p->tau_B);
    k.omega[0] = (C)(1.0 / p->tau_A);
    k.omega[1] = (C)(1.0 / p->tau_B);
    // omega w times the storage scale (a power of two: exact), per class of
    // |c_i|^2; the products are rounded once, in the compute precision
    const double sc = std::ldexp(1.0, kernel_scale_log2(p->precision));
    const double wc[3] = {4.0 / 9.0, 1.0 / 9.0, 1.0 / 36.0};
    for (int c = 0; c < 3; ++c) {
        k.omw[c].x = (C)(sc * wc[c] / p->tau_A);
        k.omw[c].y = (C)(sc * wc[c] / p->tau_B);
    }
    for (int c = 0; c < 2; ++c) {
        k.omw2[c].x = C(2) * k.omw[c + 1].x;
        k.omw2[c].y = C(2) * k.omw[c + 1].y;
    }
    k.omm.x = (C)(1.0 - 1.0 / p->tau_A);
    k.omm.y = (C)(1.0 - 1.0 / p->tau_B);
    k.u_wall = (C)p->u_wall;
    k.g_x = (C)p->g_x;
    k.kolmo_amp = (C)p->kolmo_amp;
    k.kolmo_w = (C)(2.0 * M_PI * p->kolmo_k / p->ny);
    k.sr = (p->rounding == LB_ROUND_STOCHASTIC &&
            (p->precision == LB_FP16_OFFSET || p->precision == LB_BF16_OFFSET)) ? 1 : 0;
    k.source = p->force_scheme == LB_FORCE_SOURCE ? 1 : 0;
    k.has_accel = (p->g_x != 0.0 || p->kolmo_amp != 0.0) ? 1 : 0;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// TMA descriptor of one population buffer: 9 direction planes of interleaved
// (A, B) pairs, a row holding 2 * pitch elements.  Box: cols pairs x rows x
// 9 planes.  The descriptor spans the first ext_pairs pairs of each of the
// first ext_rows rows (all of the padded plane when 0): a store clips what
// falls outside.
static lb_status make_tmap(CUtensorMap* m, int precision, const Geom& g, void* base, int cols,
                           int rows, int ext_pairs = 0, int ext_rows = 0) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return LB_ERR_CUDA;
    const int es = kernel_elem_bytes(precision);
    CUtensorMapDataType dt = precision == LB_FP64   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                             : precision == LB_FP32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                                    : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    cuuint64_t dims[3] = {(cuuint64_t)(2 * (ext_pairs > 0 ? ext_pairs : g.pitch)),
                          (cuuint64_t)(ext_rows > 0 ? ext_rows : g.rows), 9};
    cuuint64_t strides[2] = {(cuuint64_t)(2 * g.pitch) * es,
                             (cuuint64_t)g.rows * (cuuint64_t)(2 * g.pitch) * es};
    cuuint32_t box[3] = {(cuuint32_t)(2 * cols), (cuuint32_t)rows, 9};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(m, dt, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LB_OK : LB_ERR_CUDA;
}

lb_status lattice_setup(Lattice& L, const lb_params* p, char* region) {
    L.p = *p;
    L.g = make_geom(p);
    Region r = region_layout(p);
    L.region = region;
    L.st = reinterpret_cast<DevStats*>(region + r.stats);
    L.slots = reinterpret_cast<double*>(region + r.slots);
    L.wallx = region + r.wallx;
    L.wsum = reinterpret_cast<double*>(region + r.wsum);
    L.fbuf[0] = region + r.f0;
    L.fbuf[1] = region + r.f1;
    L.fbytes = r.fbytes;
    L.cur = 0;
    L.pull = 0;
    L.mom = false;
    L.inited = false;
    L.t = 0;
    L.err_latched = 0;
    const int tx = kernel_tile_x(p->precision), ty = kernel_tile_y(p->precision);
    L.nstrips = (p->nx + tx - 1) / tx;
    L.ntiles_y = (p->ny + ty - 1) / ty;
    L.seg = 1;
    fill_coef(L.kd, p);
    fill_coef(L.kf, p);
    const int bx = tx + 2 * L.g.gx;
    lb_status s = LB_OK;
    for (int b = 0; b < 2 && s == LB_OK; ++b) {
        s = make_tmap(&L.tblock[b], p->precision, L.g, L.fbuf[b], bx, kernel_block_rows(p->precision));
        // Tile stores end at the lattice's last row and at the last 16-byte
        // boundary of its rows (x_tail): a clipped bulk store writes up to a
        // 16-byte boundary, which would reach into the ghost column beside
        // an unaligned last lattice column and race with the plain stores
        // of the ghost copies.  Columns x_tail .. nx - 1 get plain stores.
        if (s == LB_OK)
            s = make_tmap(&L.ttile[b], p->precision, L.g, L.fbuf[b], tx, ty, L.g.x_tail + L.g.gx,
                          p->ny + kGY);
        if (s == LB_OK) s = make_tmap(&L.tobs[b], p->precision, L.g, L.fbuf[b], bx, ty + 2 * kGY);
    }
    return s;
}

// Load-balance model of the persistent step kernel: items are segments of
// `seg` tiles of the column strips; CTA b takes items b, b + G, ...  A CTA's
// cost is its tiles plus a quarter tile per item (the first tile of an item
// computes 12 rather than 8 deviation rows).  Returns the seg in [1, 64]
// minimising the most loaded CTA (ties: longer segments).
int choose_seg(const int* nstrips, const int* ntiles_y, int nlat, int G) {
    int best_seg = 1;
    double best = 1e300;
    std::vector<double> cost;
    for (int seg = 1; seg <= 64; ++seg) {
        long long items = 0;
        for (int l = 0; l < nlat; ++l) items += (long long)nstrips[l] * ((ntiles_y[l] + seg - 1) / seg);
        const int g = items < G ? (int)items : G;
        if (g <= 0) continue;
        // equal items go round the CTAs: whole rounds count once, for all
        cost.assign((size_t)g, 0.0);
        double all = 0.0;
        int at = 0;   // the CTA whose turn it is
        auto deal = [&](long long n, double c) {
            all += (double)(n / g) * c;
            for (int k = (int)(n % g); k > 0; --k) {
                cost[(size_t)at] += c;
                if (++at == g) at = 0;
            }
        };
        for (int l = 0; l < nlat; ++l) {
            deal((long long)nstrips[l] * (ntiles_y[l] / seg), seg + 0.25);
            if (ntiles_y[l] % seg) deal(nstrips[l], ntiles_y[l] % seg + 0.25);
        }
        double mx = 0.0;
        for (double c : cost) mx = c > mx ? c : mx;
        mx += all;
        if (mx <= best) {
            best = mx;
            best_seg = seg;
        }
    }
    return best_seg;
}

int tiles_y(const Lattice& L, int shape) {
    const int ty = shape_rows(shape);
    return (L.p.ny + ty - 1) / ty;
}
// The moment kernel: FP32, omega = 1 for both species in FP32, no source term.
bool moments_ok(const Lattice& L) {
    return L.p.precision == LB_FP32 && L.kf.omm.x == 0.0f && L.kf.omm.y == 0.0f && !L.kf.source;
}
// Default tile shape of a lattice set with `tiles8` 8-row tiles.
//  One tile per SM at most: the direct kernel, with the shortest chain (its
//  figures are there; with two tiles on a CTA it loses: 256^2 FP16, 160 tiles,
//  6.9 us a step against 6.3).
//  Up to 1.5 tiles per SM: one site per thread, which finishes a tile sooner
//  (256^2 FP16: 6.3 us with SHAPE_8, 6.9 with SHAPE_8X2; 512^2, 576 tiles: 11.0
//  and 9.7.  FP32: 6.5 us with 8 rows, 7.3 with 16; 512^2: 11.2 and 10.2).
//  Beyond: two sites per thread, two CTAs per SM where they fit.
int default_shape(int precision, bool moments, long long tiles8, int sms) {
    const bool few = 2 * tiles8 <= 3LL * sms;
    if (moments) return few ? SHAPE_M8 : SHAPE_M8X2;
    if (precision == LB_FP64) return SHAPE_8;
    if (tiles8 <= sms) return SHAPE_D8;
    if (few) return SHAPE_8;
    return has_shape(precision, SHAPE_8X2) ? SHAPE_8X2 : SHAPE_16;
}
int shape_of_rows(int precision, bool moments, int rows, long long tiles8, int sms) {
    if (rows == 0) return default_shape(precision, moments, tiles8, sms);
    if (rows == 16) return has_shape(precision, SHAPE_16) ? SHAPE_16 : 0;
    if (rows != 8) return 0;
    const int d = default_shape(precision, false, tiles8, sms);
    return d == SHAPE_16 ? SHAPE_8 : d;
}

template <typename C>
static void fill_desc(LatDesc<C>& d, const Lattice& L, const Coef<C>& k, int ntiles) {
    memset(&d, 0, sizeof(d));
    for (int b = 0; b < 2; ++b) {
        d.tin[b] = L.tblock[b];
        d.tout[b] = L.ttile[b];
        d.fbuf[b] = L.fbuf[b];
    }
    d.g = L.g;
    d.v = vals_of(k);
    d.st = L.st;
    d.wallx = L.wallx;
    d.wsum = L.wsum;
    d.nstrips = L.nstrips;
    d.ntiles_y = ntiles;
    d.stress_every = L.p.stress_every;
}

// Items (int4) | CTA offsets.  Segments and runs of tiles hold a tile at least
// each.  FP64 runs are cut by rows: a run per CTA (one CTA per SM), cut again
// where it enters a strip.  (84 x 152: 152 items, 57 tiles.)
size_t launch_area_doubles(int precision, size_t tiles, size_t strips, int sms) {
    const size_t items = precision == LB_FP64 ? std::max(tiles, (size_t)sms) + strips : tiles;
    return 2 * items + (2 * (size_t)sms + 2) / 2;   // at most two CTAs per SM
}

namespace {

struct Item {
    int lat, strip, ty_a, ty_b;
};

// seg > 0: segments of seg tiles, numbered lattice by lattice, segment row by
// segment row, strip by strip; CTA b takes items b, b + G, ...
// seg < 0: the tiles of all lattices in strip order (lattice, strip, tile
// row) cut into G contiguous runs of equal estimated cost, each run cut
// again at strip boundaries: every CTA walks one or two strips.
// rows > 0 (FP64 launches): the units cut and dealt are groups of `rows` rows in
// place of tiles, all of the same cost.
void partition(Lattice* const* lats, int nlat, int seg, int shape, int sms, std::vector<Item>& items,
               std::vector<int>& cta, int* grid, int rows = 0) {
    items.clear();
    cta.clear();
    std::vector<int> nty((size_t)nlat);
    long long tiles = 0;
    for (int l = 0; l < nlat; ++l) {
        nty[(size_t)l] = rows ? (lats[l]->p.ny + rows - 1) / rows : tiles_y(*lats[l], shape);
        tiles += (long long)lats[l]->nstrips * nty[(size_t)l];
    }
    // Tile costs relative to a full interior tile, fitted on GB300 to the
    // per-CTA times of single steps (5 x 512^2 sweeps, periodic and Couette,
    // FP32 and FP16, 16-row tiles): tiles writing periodic ghost columns
    // +0.21; ghost rows +0.25 where they leave through the staging tile, +0.02
    // where the threads store them directly; Couette tiles holding a wall row
    // (mirror, bounce-back, wall momentum) 1.38; ragged tiles 1.07; and an
    // item's start (its block ring fills, it computes four more deviation
    // rows) 0.8 of a tile.
    auto cost = [&](int l, int sx, int ty) {
        if (rows) return 1.0;
        const Lattice& L = *lats[l];
        const int tx = kernel_tile_x(L.p.precision), tyy = shape_rows(shape);
        const int x0 = sx * tx, y0 = ty * tyy;
        const bool full = x0 + tx <= L.p.nx && y0 + tyy <= L.p.ny;
        if (!full) return 1.07;
        const bool per = L.g.periodic != 0;
        if (!per && (y0 == 0 || y0 + tyy >= L.p.ny)) return 1.38;
        double c = 1.0;
        if (shape_moments(shape)) return c;   // no ghost copies
        if (x0 < 3 || x0 + tx > L.p.nx - 3) c += 0.21;
        if (per && (y0 < 3 || y0 + tyy > L.p.ny - 3)) c += kernel_staged(L.p.precision, shape) ? 0.25 : 0.02;
        return c;
    };
    // An FP64 item start is four more window rows at a quarter of a row's work
    // each, and the wait for its first blocks.
    const double kItemStart = rows ? 1.6 / rows : 0.8;
    if (seg > 0) {
        // Segments in band order (all strips of a segment row, row after row),
        // each given to the CTA with the least work so far (the lowest index
        // among equals): round-robin dealing when costs are equal, while the
        // CTAs that draw the costlier edge segments take fewer of them.
        long long nseg = 0;
        for (int l = 0; l < nlat; ++l) nseg += (long long)lats[l]->nstrips * ((nty[(size_t)l] + seg - 1) / seg);
        const int G = (int)std::min<long long>(nseg, sms);
        std::vector<std::vector<Item>> mine((size_t)G);
        for (auto& m : mine) m.reserve((size_t)(nseg / G + 2));
        typedef std::pair<double, int> Load;   // (work so far, CTA): a heap, smallest first
        std::vector<Load> heap((size_t)G);
        for (int b = 0; b < G; ++b) heap[(size_t)b] = {0.0, b};
        // the item to the heap's first CTA, whose load then sinks to its place
        auto deal = [&](const Item& it, double w) {
            const Load top = {heap[0].first + w, heap[0].second};
            mine[(size_t)top.second].push_back(it);
            size_t at = 0;
            for (size_t c = 1; c < heap.size(); c = 2 * at + 1) {
                if (c + 1 < heap.size() && heap[c + 1] < heap[c]) ++c;
                if (!(heap[c] < top)) break;
                heap[at] = heap[c];
                at = c;
            }
            heap[at] = top;
        };
        for (int l = 0; l < nlat; ++l) {
            const int ns = lats[l]->nstrips, nt = nty[(size_t)l];
            for (int a = 0; a < nt; a += seg) {
                const int b = std::min(a + seg, nt);
                auto work = [&](int sx) {
                    double w = kItemStart;
                    for (int ty = a; ty < b; ++ty) w += cost(l, sx, ty);
                    return w;
                };
                // (a strip between the first and the last two costs what its neighbours do)
                double w = 0.0;
                for (int sx = 0; sx < ns; ++sx) {
                    if (sx < 2 || sx >= ns - 2) w = work(sx);
                    deal({l, sx, a, b}, w);
                }
            }
        }
        for (int b = 0; b < G; ++b) {
            cta.push_back((int)items.size());
            items.insert(items.end(), mine[(size_t)b].begin(), mine[(size_t)b].end());
        }
        cta.push_back((int)items.size());
        *grid = G;
        return;
    }
    // Contiguous runs over the tiles in order (lattice, strip, tile row); a
    // run pays an item start where it begins and where it crosses into the
    // next strip.  The runs minimise the largest run cost: the smallest bound
    // B for which runs filled greedily (a run takes the next tile while its
    // cost stays within B) number at most sms, found by bisection -- at most
    // one tile above the mean, where cutting at equal cumulative cost lets
    // some runs overshoot by a whole tile.
    std::vector<double> tc, upto;   // tile costs; their sums with the strips' starts
    tc.reserve((size_t)tiles);
    upto.reserve((size_t)tiles + 1);
    upto.push_back(0.0);
    double cmax = 0.0;
    for (int l = 0; l < nlat; ++l)
        for (int sx = 0; sx < lats[l]->nstrips; ++sx)
            for (int ty = 0; ty < nty[(size_t)l]; ++ty) {
                const double c = cost(l, sx, ty);
                tc.push_back(c);
                upto.push_back(upto.back() + c + (ty == 0 ? kItemStart : 0.0));
                cmax = std::max(cmax, c);
            }
    const double sum = upto.back();
    // Runs needed under bound B; with starts, the first tile of each run.  A run
    // from tile k costs its first tile and a start, then what the sums grow by;
    // its end is found by bisection (costs are multiples of 0.01: sums closer
    // than 1e-6 are equal).
    auto runs_for = [&](double B, std::vector<long long>* starts) -> long long {
        long long n = 0;
        for (long long k = 0; k < tiles;) {
            ++n;
            if (starts) starts->push_back(k);
            const double most = upto[(size_t)k + 1] + (B - tc[(size_t)k] - kItemStart) + 1e-6;
            k = std::upper_bound(upto.begin() + (k + 2), upto.end(), most) - upto.begin() - 1;
        }
        return n;
    };
    // (from just above the mean run; costs are multiples of 0.01, so a bound
    // known to 0.002 gives the optimal runs)
    double lo = std::max(cmax + kItemStart, sum / sms), hi = lo;
    if (runs_for(lo, nullptr) > sms) {
        do {
            hi += cmax + 2.0 * kItemStart;
        } while (runs_for(hi, nullptr) > sms);
        while (hi - lo > 0.002) {
            const double mid = 0.5 * (lo + hi);
            if (runs_for(mid, nullptr) <= sms) hi = mid; else lo = mid;
        }
    }
    std::vector<long long> starts;
    runs_for(hi, &starts);
    const int G = (int)starts.size();
    starts.push_back(tiles);
    // tile k -> (lattice, strip, tile row), walking the same order
    int l = 0, sx = 0, ty = 0;
    for (int b = 0; b < G; ++b) {
        cta.push_back((int)items.size());
        long long k = starts[(size_t)b];
        while (k < starts[(size_t)b + 1]) {
            const int nt = nty[(size_t)l];
            const int take = (int)std::min<long long>(nt - ty, starts[(size_t)b + 1] - k);
            items.push_back({l, sx, ty, ty + take});
            k += take;
            ty += take;
            if (ty == nt) {
                ty = 0;
                if (++sx == lats[l]->nstrips) {
                    sx = 0;
                    ++l;
                }
            }
        }
    }
    cta.push_back((int)items.size());
    *grid = G;
}

}  // namespace

// Default partition: cost-balanced contiguous runs while each CTA has up to
// ~40 tiles of 8 rows (measured faster on 512^2-1024^2 lattices), the
// load-balance model's dealt segments beyond (their CTAs sweep a band of
// rows together, which keeps the halo columns in L2 on large lattices);
// `tiles` counts tiles of the shape, `ctas` the launch's CTAs.  The moment kernel
// moves a third of the bytes and takes contiguous runs at every size (4096^2:
// 304 us a step, the best dealt segments 310; 4 x 1024^2: 84 and 84).
// Contiguous runs also for more tiles where every lattice's buffer takes at most
// a third of L2 (`largest` bytes): neighbouring strips then find each other's
// halo columns there (4 x 1024^2 FP16: 78 us a step, dealt segments 83; one
// 2048^2, the same number of tiles: 101 and 78).
static int default_seg(long long tiles, int shape, const int* ns, const int* nt, int nlat, int sms,
                       int ctas, long long largest) {
    return shape_moments(shape) || tiles * shape_rows(shape) <= 8LL * 40 * sms ||
                   largest * 3 <= device_l2_bytes()
               ? -1
               : choose_seg(ns, nt, nlat, ctas);
}

// Host-only plan of a launch's work items (lb_plan_partition).
lb_status plan_partition(const lb_params* ps, int nlat, int seg, int tile_rows, int sms,
                         int32_t* items, int32_t* nitems, int32_t* cta, int32_t* grid,
                         int32_t* seg_used) {
    if (!ps || nlat < 1 || sms < 1 || !nitems || !grid || !seg_used) return LB_ERR_INVALID;
    std::vector<Lattice> lv((size_t)nlat);
    std::vector<Lattice*> lp((size_t)nlat);
    std::vector<int> ns((size_t)nlat), nt((size_t)nlat);
    if (validate_params(&ps[0]) != LB_OK) return LB_ERR_INVALID;
    if (tile_rows != 0 && tile_rows != 8 && tile_rows != 16) return LB_ERR_INVALID;
    const int shape = tile_rows == 16 ? SHAPE_16 : SHAPE_8;   // (any 8-row shape: one CTA per SM)
    if (shape == SHAPE_16 && !has_shape(ps[0].precision, shape)) return LB_ERR_INVALID;
    long long tiles = 0;
    for (int l = 0; l < nlat; ++l) {
        if (validate_params(&ps[l]) != LB_OK || ps[l].precision != ps[0].precision)
            return LB_ERR_INVALID;
        Lattice& L = lv[(size_t)l];
        L.p = ps[l];
        L.g = make_geom(&ps[l]);
        const int tx = kernel_tile_x(ps[l].precision);
        L.nstrips = (ps[l].nx + tx - 1) / tx;
        L.ntiles_y = tiles_y(L, SHAPE_8);
        lp[(size_t)l] = &L;
        ns[(size_t)l] = L.nstrips;
        nt[(size_t)l] = tiles_y(L, shape);
        tiles += (long long)L.nstrips * nt[(size_t)l];
    }
    const int s = seg != 0 ? seg : default_seg(tiles, shape, ns.data(), nt.data(), nlat, sms, sms,
                                            1LL << 60);
    std::vector<Item> it;
    std::vector<int> c;
    int G = 0;
    partition(lp.data(), nlat, s, shape, sms, it, c, &G);
    const int cap_items = *nitems, cap_cta = *grid;
    *nitems = (int32_t)it.size();
    *grid = G;
    *seg_used = s;
    if (cap_items < (int)it.size() || cap_cta < G + 1 || !items || !cta) return LB_ERR_INVALID;
    for (size_t k = 0; k < it.size(); ++k) {
        items[4 * k] = it[k].lat;
        items[4 * k + 1] = it[k].strip;
        items[4 * k + 2] = it[k].ty_a;
        items[4 * k + 3] = it[k].ty_b;
    }
    for (int b = 0; b <= G; ++b) cta[b] = c[(size_t)b];
    return LB_OK;
}

HostStage::~HostStage() {
    for (Buffer& b : buf_)
        if (b.done) {
            if (b.busy) cudaEventSynchronize(b.done);
            cudaEventDestroy(b.done);
        }
    for (char* m : blocks_) cudaFreeHost(m);
}

cudaError_t HostStage::reserve(size_t bytes) {
    cudaError_t e = cudaSuccess;
    for (Buffer& b : buf_)
        if (!b.done && (e = cudaEventCreateWithFlags(&b.done, cudaEventDisableTiming)) != cudaSuccess) {
            b.done = nullptr;
            return e;
        }
    if (bytes <= cap_) return e;
    const size_t cap = align_up(std::max(bytes, 2 * cap_), 64 << 10);
    char* m = nullptr;
    e = cudaHostAlloc(reinterpret_cast<void**>(&m), kBuffers * cap, cudaHostAllocDefault);
    if (e != cudaSuccess) return e;
    blocks_.push_back(m);
    cap_ = cap;
    // (copies out of the buffers before may be on their way: their memory stays)
    for (int k = 0; k < kBuffers; ++k) {
        buf_[k].mem = m + k * cap;
        buf_[k].busy = false;
    }
    return e;
}

char* HostStage::get(size_t bytes) {
    if (reserve(bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    last_ = (last_ + 1) % kBuffers;
    Buffer& b = buf_[last_];
    if (b.busy && cudaEventSynchronize(b.done) != cudaSuccess) return nullptr;
    b.busy = false;
    return b.mem;
}

cudaError_t HostStage::sent(cudaStream_t s) {
    Buffer& b = buf_[last_];
    const cudaError_t e = cudaEventRecord(b.done, s);
    b.busy = e == cudaSuccess;
    return e;
}

lb_status launch_build(Launch& Ln, Lattice* const* lats, int nlat, void* descs, double* slots,
                       size_t room, unsigned int* ticket, int sms, cudaStream_t stream, HostStage* stage,
                       int forced_seg, int shape) {
    if (nlat < 1) return LB_ERR_INVALID;
    const int prec = lats[0]->p.precision;
    if (!has_shape(prec, shape)) return LB_ERR_INVALID;
    std::vector<int> ns((size_t)nlat), nt((size_t)nlat);
    bool allper = true, gen = false, tau1 = true;
    long long tiles = 0, strips = 0;
    for (int l = 0; l < nlat; ++l) {
        ns[(size_t)l] = lats[l]->nstrips;
        nt[(size_t)l] = tiles_y(*lats[l], shape);
        allper = allper && lats[l]->g.periodic;
        gen = gen || lats[l]->kd.source || lats[l]->kd.has_accel;
        // 1 - omega rounds to zero in the compute precision for both species:
        // the collision does not read the populations (kernel variant bit 4)
        tau1 = tau1 && (prec == LB_FP64
                            ? (lats[l]->kd.omm.x == 0.0 && lats[l]->kd.omm.y == 0.0)
                            : (lats[l]->kf.omm.x == 0.0f && lats[l]->kf.omm.y == 0.0f));
        tiles += (long long)lats[l]->nstrips * nt[(size_t)l];
        strips += lats[l]->nstrips;
    }
    const int ctas = sms * shape_ctas(shape);
    long long largest = 0;
    for (int l = 0; l < nlat; ++l) largest = std::max(largest, (long long)lats[l]->fbytes);
    const int seg = forced_seg != 0 ? forced_seg
                                    : default_seg(tiles, shape, ns.data(), nt.data(), nlat, sms, ctas, largest);
    std::vector<Item> items;
    std::vector<int> cta;
    int grid = 0;
    if (prec == LB_FP64) {
        // Rows, in groups of 1, 2, 4 or 8, so that a CTA gets 16 to 32 of them;
        // a requested segment is in tiles.
        long long all = 0;
        for (int l = 0; l < nlat; ++l) all += (long long)lats[l]->nstrips * lats[l]->p.ny;
        int rows = seg > 0 ? shape_rows(shape) : 1;
        while (rows < shape_rows(shape) && all > 32LL * ctas * rows) rows *= 2;
        partition(lats, nlat, seg, shape, ctas, items, cta, &grid, rows);
        for (Item& it : items) {
            it.ty_a *= rows;
            it.ty_b = std::min(it.ty_b * rows, lats[it.lat]->p.ny);
        }
    } else {
        partition(lats, nlat, seg, shape, ctas, items, cta, &grid);
    }
    const int nitems = (int)items.size();
    const size_t dsz = prec == LB_FP64 ? sizeof(LatDesc<double>) : sizeof(LatDesc<float>);
    // descriptors | items | CTA offsets, as they go to the device
    const size_t at_items = align_up(dsz * (size_t)nlat, 128);
    const size_t at_cta = at_items + sizeof(Item) * (size_t)nitems;
    const size_t bytes = at_cta + sizeof(int) * cta.size();
    if (bytes - at_items > room * sizeof(double)) return LB_ERR_NOMEM;
    std::vector<char> own;
    char* hs = stage ? stage->get(bytes) : nullptr;
    if (!hs) {   // no stage, or no pinned memory to be had
        stage = nullptr;
        own.resize(bytes + 128);
        hs = own.data() + (128 - reinterpret_cast<uintptr_t>(own.data()) % 128) % 128;
    }
    memcpy(hs + at_items, items.data(), sizeof(Item) * (size_t)nitems);
    memcpy(hs + at_cta, cta.data(), sizeof(int) * cta.size());
    for (int l = 0; l < nlat; ++l) {
        lats[l]->seg = seg;
        if (prec == LB_FP64)
            fill_desc(*reinterpret_cast<LatDesc<double>*>(hs + l * dsz), *lats[l], lats[l]->kd,
                      lats[l]->p.ny);   // (items in rows)
        else
            fill_desc(*reinterpret_cast<LatDesc<float>*>(hs + l * dsz), *lats[l], lats[l]->kf,
                      nt[(size_t)l]);
    }
    // device tables: items (16-byte aligned), CTA offsets
    int4* d_items = reinterpret_cast<int4*>(slots);
    int* d_cta = reinterpret_cast<int*>(d_items + nitems);
    static_assert(sizeof(Item) == sizeof(int4), "item layout");
    cudaError_t e = cudaMemcpyAsync(descs, hs, dsz * nlat, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        // (the CTA offsets follow the items on both sides)
        e = cudaMemcpyAsync(d_items, hs + at_items, bytes - at_items, cudaMemcpyHostToDevice, stream);
    // (also after a copy that failed: the one before it may be on its way)
    const cudaError_t es = stage ? stage->sent(stream) : cudaStreamSynchronize(stream);
    if (e == cudaSuccess) e = es;
    if (e != cudaSuccess) return cuda_status(e);
    Ln.precision = prec;
    Ln.variant = (allper ? 1 : 0) | (gen ? 2 : 0) | (tau1 ? 4 : 0);
    Ln.shape = shape;
    Ln.grid = dim3((unsigned)grid, 1, 1);
    Ln.nitems = nitems;
    Ln.seg = seg;
    // One buffer of every lattice within 80 % of L2: the step's output can
    // stay in L2 for the next step, next to the input streaming through.
    long long buf = 0;
    for (int l = 0; l < nlat; ++l)
        buf += shape_moments(shape) ? 24LL * lats[l]->p.nx * lats[l]->p.ny : (long long)lats[l]->fbytes;
    const int l2_resident = buf * 5 <= device_l2_bytes() * 4 ? 1 : 0;
    // With the collision free of the populations (tau = 1), a tile's ring
    // slots can be refilled as soon as its density phase is done.  Measured
    // on GB300: that deeper prefetch pays where the step's input comes
    // largely from L2 (one buffer of every lattice within L2) and for the
    // 16-bit formats (issue-bound), but costs FP32 lattices streaming from
    // DRAM (4096^2, 16-row tiles: 39.2 against 42.3 GLUPS), which keep the
    // refill after the site phase.
    const int early_release = tau1 && (l2_resident || prec == LB_FP16_OFFSET || prec == LB_BF16_OFFSET) ? 1 : 0;
    if (prec == LB_FP64) {
        BatchArgs<double>& a = Ln.ad;
        a.k = lats[0]->kd;
        a.lat = reinterpret_cast<const LatDesc<double>*>(descs);
        a.nlat = nlat;
        a.nitems = nitems;
        a.items = d_items;
        a.cta_items = d_cta;
        a.ticket = ticket;
        a.l2_resident = l2_resident;
        a.early_release = early_release;
    } else {
        BatchArgs<float>& a = Ln.af;
        a.k = lats[0]->kf;
        a.lat = reinterpret_cast<const LatDesc<float>*>(descs);
        a.nlat = nlat;
        a.nitems = nitems;
        a.items = d_items;
        a.cta_items = d_cta;
        a.ticket = ticket;
        a.l2_resident = l2_resident;
        a.early_release = early_release;
    }
    return LB_OK;
}

lb_status launch_run(Launch& Ln, int step_k, int advance, cudaStream_t s) {
    Ln.ad.step_k = Ln.af.step_k = step_k;
    Ln.ad.advance = Ln.af.advance = advance;
    const void* args = Ln.precision == LB_FP64 ? (const void*)&Ln.ad : (const void*)&Ln.af;
    return cuda_status(launch_step(Ln.precision, args, Ln.variant, Ln.shape, Ln.grid, s));
}

lb_status launch_window(Launch& Ln, int n, cudaStream_t s, bool* broken) {
    *broken = false;
    for (int k = 0; k < n; ++k) {
        const lb_status st = launch_run(Ln, k, k == n - 1 ? n : 0, s);
        if (st != LB_OK) {
            *broken = k > 0;
            return st;
        }
    }
    return LB_OK;
}

static lb_status lattice_observe_pull(Lattice& L, int obs, double* const dst[4], int q0, int q1, int pull,
                                      cudaStream_t s);
lb_status lattice_observe(Lattice& L, int obs, double* const dst[4], int q0, int q1, cudaStream_t s) {
    return lattice_observe_pull(L, obs, dst, q0, q1, L.pull, s);
}

static lb_status lattice_observe_pull(Lattice& L, int obs, double* const dst[4], int q0, int q1, int pull,
                                      cudaStream_t s) {
    // CTAs take several tiles each once every SM of a GB300 is full (2048 threads
    // on each of 152; not the device's own count: the CTAs set the order in which
    // the totals are added, which is the same on every GPU)
    const long long tiles = (long long)L.nstrips * L.ntiles_y;
    const int threads = L.p.precision == LB_FP64 ? 256 : 512;
    const long long most = 152LL * (2048 / threads);
    dim3 grid((unsigned)std::min(tiles, most), 1, 1);
    cudaError_t e;
    if (L.p.precision == LB_FP64) {
        StepArgs<double> a;
        memset(&a, 0, sizeof(a));
        a.g = L.g;
        a.k = L.kd;
        a.st = L.st;
        a.slots = L.slots;
        a.pull = pull;
        a.obs = obs;
        for (int k = 0; k < 4; ++k) a.obs_dst[k] = dst ? dst[k] : nullptr;
        a.q0 = q0;
        a.q1 = q1;
        a.wsum = L.wsum;
        a.nstrips = L.nstrips;
        e = launch_observe(L.p.precision, &L.tobs[L.cur], &a, grid, s);
    } else {
        StepArgs<float> a;
        memset(&a, 0, sizeof(a));
        a.g = L.g;
        a.k = L.kf;
        a.st = L.st;
        a.slots = L.slots;
        a.pull = pull;
        a.obs = obs;
        for (int k = 0; k < 4; ++k) a.obs_dst[k] = dst ? dst[k] : nullptr;
        a.q0 = q0;
        a.q1 = q1;
        a.wsum = L.wsum;
        a.nstrips = L.nstrips;
        a.mom = L.mom ? reinterpret_cast<const float2*>(L.fbuf[L.cur]) : nullptr;
        e = launch_observe(L.p.precision, &L.tobs[L.cur], &a, grid, s);
    }
    return cuda_status(e);
}

lb_status lattice_read_stats(Lattice& L, DevStats* out, cudaStream_t s) {
    cudaError_t e = cudaMemcpyAsync(out, L.st, sizeof(DevStats), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    L.err_latched |= out->err;
    if (L.err_latched & ERR_TIMEOUT) return LB_ERR_TIMEOUT;
    if (L.err_latched & ERR_NONFINITE) return LB_ERR_NONFINITE;
    return LB_OK;
}

// The first step >= t at which the wall momentum is sampled:
// stress_t0 + k stress_every, k >= 0.
static long long first_sample(const lb_params& p, long long t) {
    if (t <= p.stress_t0) return p.stress_t0;
    const long long every = p.stress_every > 0 ? p.stress_every : 1;
    return p.stress_t0 + (t - p.stress_t0 + every - 1) / every * every;
}

// Host side of a restart at step t with the stored form `pull`, and what the
// initialising kernel is to leave on the device.
static StateInit lattice_reset(Lattice& L, long long t, int pull) {
    L.t = t;
    L.cur = 0;
    L.pull = pull;
    L.mom = false;
    L.inited = true;
    L.err_latched = 0;
    StateInit z;
    z.st = L.st;
    z.t = t;
    z.next_sample = first_sample(L.p, t);
    z.pull = pull;
    z.wsum = L.wsum;
    z.nwsum = L.g.periodic ? 0 : 2 * L.nstrips;
    return z;
}

// Whether [p, p + bytes) lies in one allocation or registration as the driver
// knows it (the two ends alone do not tell: they may be pinned apart, with
// pageable memory between them).
typedef CUresult (*PointerAttributeFn)(void*, CUpointer_attribute, CUdeviceptr);
static bool in_one_range(const void* p, size_t bytes) {
    static const PointerAttributeFn get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<PointerAttributeFn>(f);
    }();
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    CUdeviceptr start = 0;
    size_t size = 0;
    return get && get(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, at) == CUDA_SUCCESS &&
           get(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, at) == CUDA_SUCCESS && at >= start &&
           at - start <= size && bytes <= size - (at - start);
}

// The address under which the device reaches `bytes` of pinned host memory, or
// null where they do not lie in one pinned range (or are not aligned for doubles).
// Kernels read and write pinned arrays over the link themselves, at the rate of
// a copy (193 GB/s out, 211 GB/s in), which saves the staging pass, the copies
// and their launches: lb_fields of the densities of a 512^2 FP16 lattice 81 -> 64
// us, all four fields of 4096^2 3.9 -> 3.2 ms; lb_restore of 1024^2 910 -> 740 us.
static double* pinned_view(const double* host, size_t bytes) {
    cudaPointerAttributes a;
    if (reinterpret_cast<uintptr_t>(host) % sizeof(double) != 0) return nullptr;
    if (cudaPointerGetAttributes(&a, host) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer || !in_one_range(host, bytes)) return nullptr;
    return reinterpret_cast<double*>(a.devicePointer);
}

static void* coef_ptr(Lattice& L) {
    return L.p.precision == LB_FP64 ? (void*)&L.kd : (void*)&L.kf;
}

lb_status lattice_init_seeded(Lattice& L, uint64_t seed, cudaStream_t s) {
    const StateInit z = lattice_reset(L, 0, 0);
    return cuda_status(launch_init_seeded(L.p.precision, L.g, coef_ptr(L), L.fbuf[0], L.p.rho0,
                                          L.p.init_amp, L.p.u_wall, L.p.init_shear,
                                          (unsigned long long)seed, z, s));
}

lb_status lattice_init_fields(Lattice& L, const double* rho_A, const double* rho_B,
                              const double* ux, const double* uy, cudaStream_t s) {
    const StateInit z = lattice_reset(L, 0, 0);
    const size_t n = (size_t)L.p.nx * L.p.ny;
    // Pageable fields are staged in buffer 1 (its size, 18 planes of at least
    // 2 bytes per padded site, always exceeds 32 bytes per site).
    double* stage = reinterpret_cast<double*>(L.fbuf[1]);
    const double* src[4] = {rho_A, rho_B, ux, uy};
    const double* f[4] = {nullptr, nullptr, nullptr, nullptr};
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 4 && e == cudaSuccess; ++k) {
        if (!src[k]) continue;
        f[k] = pinned_view(src[k], n * 8);
        if (f[k]) continue;
        f[k] = stage + k * n;
        e = cudaMemcpyAsync(stage + k * n, src[k], n * 8, cudaMemcpyHostToDevice, s);
    }
    if (e == cudaSuccess) e = launch_init_fields(L.p.precision, L.g, coef_ptr(L), L.fbuf[0], f, z, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return cuda_status(e);
}

lb_status lattice_load_populations(Lattice& L, const double* f, long long t, int pulled,
                                   cudaStream_t s) {
    if (t < 0 || (pulled != 0 && pulled != 1) || (pulled && t < 1)) return LB_ERR_INVALID;
    const size_t n = (size_t)L.p.nx * L.p.ny;
    // Pageable populations: whole directions (both species, 16 bytes per site)
    // staged in buffer 1.
    const int per = (int)(L.fbytes / (n * 16));
    if (per < 1) return LB_ERR_UNSUPPORTED;
    const StateInit z = lattice_reset(L, t, pulled);
    StateInit none = {};
    cudaError_t e = cudaSuccess;
    if (const double* v = pinned_view(f, 18 * n * 8)) {
        e = launch_load_pops(L.p.precision, L.g, coef_ptr(L), L.fbuf[0], v, 9 * n, n, 0, 9, z, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        return cuda_status(e);
    }
    double* stage = reinterpret_cast<double*>(L.fbuf[1]);
    for (int i0 = 0; i0 < 9 && e == cudaSuccess; i0 += per) {
        const int i1 = i0 + per < 9 ? i0 + per : 9;
        for (int i = i0; i < i1 && e == cudaSuccess; ++i)
            for (int sp = 0; sp < 2 && e == cudaSuccess; ++sp)
                e = cudaMemcpyAsync(stage + ((size_t)(i - i0) * 2 + sp) * n,
                                    f + ((size_t)sp * 9 + i) * n, n * 8, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = launch_load_pops(L.p.precision, L.g, coef_ptr(L), L.fbuf[0], stage, n, 2 * n, i0, i1,
                                 i1 == 9 ? z : none, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the stage is reused
    }
    return cuda_status(e);
}

void lattice_advanced(Lattice& L, long long n, int shape) {
    if (n <= 0) return;
    L.t += n;
    L.cur ^= (int)(n & 1);
    L.pull = 1;
    L.mom = shape_moments(shape);
}

lb_status lattice_to_populations(Lattice& L, cudaStream_t s) {
    if (!L.mom) return LB_OK;
    cudaError_t e = launch_expand(L.g, L.kf, reinterpret_cast<const float2*>(L.fbuf[L.cur]),
                                  L.fbuf[1 - L.cur], s);
    L.cur ^= 1;
    L.mom = false;
    const int state[2] = {L.cur, 1};   // DevStats::cur, pull
    static_assert(offsetof(DevStats, pull) == offsetof(DevStats, cur) + sizeof(int), "cur, pull");
    if (e == cudaSuccess) e = cudaMemcpyAsync(&L.st->cur, state, sizeof(state), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // `state` is on this stack
    return cuda_status(e);
}

lb_status lattice_fields(Lattice& L, double* rho_A, double* rho_B, double* ux, double* uy,
                         cudaStream_t s) {
    const size_t n = (size_t)L.p.nx * L.p.ny;
    double* out = reinterpret_cast<double*>(L.fbuf[1 - L.cur]);
    double* dst[4] = {rho_A, rho_B, ux, uy};
    // Arrays that share memory keep the order of copies: the last one's values.
    bool apart = true;
    for (int k = 0; k < 4; ++k)
        for (int j = 0; j < k; ++j)
            apart = apart && (!dst[k] || !dst[j] || dst[k] >= dst[j] + n || dst[j] >= dst[k] + n);
    double* to[4] = {nullptr, nullptr, nullptr, nullptr};
    bool copy[4] = {false, false, false, false};
    for (int k = 0; k < 4; ++k) {
        if (!dst[k]) continue;
        if (apart) to[k] = pinned_view(dst[k], n * 8);
        copy[k] = !to[k];
        if (copy[k]) to[k] = out + k * n;
    }
    lb_status st = lattice_observe(L, OBS_FIELDS, to, 0, 0, s);
    if (st != LB_OK) return st;
    for (int k = 0; k < 4; ++k)
        if (copy[k]) {
            cudaError_t e = cudaMemcpyAsync(dst[k], to[k], n * 8, cudaMemcpyDeviceToHost, s);
            if (e != cudaSuccess) return cuda_status(e);
        }
    DevStats ds;
    return lattice_read_stats(L, &ds, s);
}

lb_status lattice_populations(Lattice& L, double* f, cudaStream_t s, int raw) {
    const size_t n = (size_t)L.p.nx * L.p.ny;
    double* out = reinterpret_cast<double*>(L.fbuf[1 - L.cur]);
    const int pull = raw ? 0 : L.pull;
    DevStats ds;
    if (double* v = pinned_view(f, 18 * n * 8)) {
        double* const to[4] = {v, nullptr, nullptr, nullptr};
        lb_status st = lattice_observe_pull(L, OBS_POPS, to, 0, 18, pull, s);
        return st != LB_OK ? st : lattice_read_stats(L, &ds, s);
    }
    int per = (int)(L.fbytes / (n * 8));
    if (per < 1) return LB_ERR_UNSUPPORTED;
    if (per > 18) per = 18;
    for (int q0 = 0; q0 < 18; q0 += per) {
        const int q1 = q0 + per < 18 ? q0 + per : 18;
        double* const to[4] = {out, nullptr, nullptr, nullptr};
        lb_status st = lattice_observe_pull(L, OBS_POPS, to, q0, q1, pull, s);
        if (st != LB_OK) return st;
        cudaError_t e = cudaMemcpyAsync(f + (size_t)q0 * n, out, (size_t)(q1 - q0) * n * 8,
                                        cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_status(e);
    }
    return lattice_read_stats(L, &ds, s);
}

lb_status lattice_stress(Lattice& L, lb_stress_out* out, cudaStream_t s) {
    lb_status st = lattice_observe(L, OBS_TOTALS, nullptr, 0, 0, s);
    if (st != LB_OK) return st;
    DevStats ds;
    st = lattice_read_stats(L, &ds, s);
    memset(out, 0, sizeof(*out));
    out->mass_A = ds.totals[0];
    out->mass_B = ds.totals[1];
    out->mom_x = ds.totals[2];
    out->mom_y = ds.totals[3];
    out->samples = ds.samples;
    out->step = L.t;
    if (ds.samples > 0) {
        out->sigma_bot = ds.sum_bot / (double)ds.samples;
        out->sigma_top = ds.sum_top / (double)ds.samples;
        out->sigma_mean = 0.5 * (out->sigma_bot - out->sigma_top);
    }
    const double rate = 2.0 * L.p.u_wall / L.p.ny;
    const double mass = ds.totals[0] + ds.totals[1];
    const double rho_mean = mass / ((double)L.p.nx * L.p.ny);
    if (L.p.boundary == LB_COUETTE && rate != 0.0 && rho_mean > 0.0 && ds.samples > 0) {
        out->nu_eff = out->sigma_mean / (rate * rho_mean);
        const double tau = mass > 0.0 ? (L.p.tau_A * ds.totals[0] + L.p.tau_B * ds.totals[1]) / mass
                                      : L.p.tau_A;
        const double nu0 = (tau - 0.5) / 3.0;
        out->response_R = out->nu_eff != 0.0 ? nu0 / out->nu_eff : 0.0;
    }
    return st;
}

}  // namespace lbgb
