// lb_internal.h -- structures shared by the host side of the C ABI
// (lb_api.cu) and the kernels (lb_kernels.cu).  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda.h>           // CUtensorMap (type only; the driver is reached via
#include <cuda_runtime.h>   // cudaGetDriverEntryPointByVersion)

#include "../../include/lb.h"

namespace lbgb {

// Device-resident counters and accumulators of one lattice.
struct DevStats {
    unsigned int err;       // bit 0: non-finite density, bit 1: TMA wait timeout
    unsigned int ticket;    // CTA arrival counter of the observe reductions
    long long t;            // completed time steps
    double sum_bot;         // sum of the bottom-wall samples, as of the last observe pass
    double sum_top;         // sum of the top-wall samples
    long long samples;      // number of samples in the sums
    double totals[4];       // last observe pass: mass_A, mass_B, mom_x, mom_y
    int cur;                // buffer holding the current state (0 or 1)
    int pull;               // what it holds, 0: f(t) in place; 1: post-collision f*(t-1);
                            // 2: the moments that f*(t-1) is the equilibrium of (k_step_m)
    long long next_sample;  // the next step whose wall momentum is sampled
                            // (stress_t0 + k stress_every >= t; set by the host
                            // with t, advanced by the kernel with t)
    double pad_[5];
};
static_assert(sizeof(DevStats) == 128, "DevStats is one 128-byte line");

enum : unsigned int { ERR_NONFINITE = 1u, ERR_TIMEOUT = 2u };

// The bounded-wait self-test kernel (lb_selftest_wait).
cudaError_t launch_wait_selftest(unsigned int* err, int limit, cudaStream_t s);
// The FP32 exp(x) - 1 / reciprocal probe (lb_selftest_math).
cudaError_t launch_math_probe(const float* x, float* out, long long n, cudaStream_t s);
// The FP64 functions (lb_selftest_math64).
cudaError_t launch_math64_probe(double rho0, const double* x, const double* y, double* out, long long n,
                                cudaStream_t s);

// Geometry of the ghost-padded population planes.  Plane i (i = 0..8, the
// D2Q9 direction) holds (ny + 2*kGY) rows of `pitch` interleaved (A, B)
// pairs; lattice site (x, y) sits at row y + kGY, pair column x + gx.  The
// kGY = 3 rows and gx >= 3 columns on each side hold periodic copies so that
// the tile loads never wrap.
constexpr int kGY = 3;

struct Geom {
    int nx, ny;
    int pitch;          // (A, B) pairs per padded row (row bytes a multiple of 16)
    int rows;           // ny + 2*kGY
    long long plane;    // pairs per direction plane = rows * pitch
    int gx;             // ghost columns on each side
    int periodic;       // 1: periodic in y; 0: Couette walls in y
    // Lattice columns x >= x_tail (at most 3) are written by plain stores,
    // not by the tile's bulk tensor store: a clipped bulk store ends on a
    // 16-byte boundary, so its descriptor stops at the last 16-byte
    // boundary of the lattice row and leaves the ghost column beside it alone.
    int x_tail;
};

// The (A, B) pair type of a compute precision.
template <typename C> struct PairOf;
template <> struct PairOf<float> { typedef float2 T; };
template <> struct PairOf<double> { typedef double2 T; };

// Per-launch model coefficients, in the compute precision C.  The stencil
// sums of Eq. (2) are taken row by row (see the step kernel): with
// K(|d|^2) = G^a w(|d|^2) + G^r p(|d|^2) per species, the like-species
// weights are the (A, B) pairs KC = {K(1), K(2), K(5), 2 K(4), 2 K(5),
// 2 K(8)} (the factors 2 are the stencil components |d_x| or |d_y| = 2,
// exact), and the cross-species ones WC = {w(1), w(2)} for both species.
// FP64 folds factors so that a site takes fewer FP64 operations: its window
// holds E = exp(-(rho - rho_ref)/rho0) - 1 in place of the Psi deviation
// -psi_scale E, its cross weights are {4, 1} = {w(1), w(2)} / w(2), and the
// site's -Psi (neg_psi) and gx_rho0 carry the factors.
template <typename C>
struct Coef {
    typedef typename PairOf<C>::T C2;
    C2 KC[6];          // like-species row weights, (A, B) pairs
    C2 WC[2];          // cross-species row weights, equal in both lanes
    C gx_rho0;         // G_X / rho0 (FP64: times w(2))
    C psi_ref;         // Psi(rho_ref)
    C psi_scale;       // P exp(-rho_ref / rho0)
    C inv_rho0;        // 1 / rho0
    C exp_c;           // FP64: -64 / (ln2 rho0), which picks the table entry (pexpm1_scaled)
    C rho_ref;         // reference density of the stored offsets
    // (16-byte aligned: the constants from here on are read in groups; a forced
    // 128^2 FP32 step took 3.635 us with them 8 bytes off, 3.608 so)
    alignas(16) C tau15[2];   // 1.5 tau_s (the velocity shift is taken for v = 1.5u)
    C omega[2];        // 1 / tau
    C2 omw[3];         // omega_s S w for the D2Q9 classes |c|^2 = 0, 1, 2 (S the storage scale)
    C2 omw2[2];        // 2 omega_s S w for the classes |c|^2 = 1, 2 (exact doubles of omw[1..2])
    C2 omm;            // 1 - omega_s
    C u_wall;          // Couette wall speed (top +, bottom -)
    C g_x;             // uniform body acceleration
    C kolmo_amp;       // Kolmogorov acceleration amplitude
    C kolmo_w;         // 2 pi kolmo_k / ny
    int sr;            // 1: half formats stored with stochastic rounding
    int source;        // 1: additive source term; 0: velocity shift
    int has_accel;     // 1 if g_x or kolmo_amp is nonzero
};

// Values that vary between the lattices of one step launch.
template <typename C>
struct LatVals {
    C rho_ref, psi_ref, psi_scale, inv_rho0, gx_rho0, u_wall;
    C kolmo_w;         // 2 pi kolmo_k / ny (ny is per lattice)
    C exp_c;           // (FP64)
};
template <typename C>
__host__ __device__ inline LatVals<C> vals_of(const Coef<C>& k) {
    LatVals<C> v;
    v.rho_ref = k.rho_ref;
    v.psi_ref = k.psi_ref;
    v.psi_scale = k.psi_scale;
    v.inv_rho0 = k.inv_rho0;
    v.gx_rho0 = k.gx_rho0;
    v.u_wall = k.u_wall;
    v.kolmo_w = k.kolmo_w;
    v.exp_c = k.exp_c;
    return v;
}

// One lattice of a step launch, in device memory (128-byte aligned for the
// tensor maps).  Both buffers are described; the device-side DevStats::cur
// says which one holds the current state.
template <typename C>
struct alignas(128) LatDesc {
    CUtensorMap tin[2];    // 8-row block loads of buffer b: box {2 BX, 8, 9}
    CUtensorMap tout[2];   // tile stores into buffer b: box {2 TX, 8, 9}, clipped at x = x_tail, y = ny
    Geom g;
    LatVals<C> v;
    void* fbuf[2];
    DevStats* st;
    void* wallx;           // [2][2][nx] compute-type pairs, by the parity of the window's
                           // step: x-momentum handed to the bottom (then top) wall by
                           // the links leaving site x in that step
    double* wsum;          // [2][nstrips]: those summed per strip (bottom, then top) and
                           // over the sampled steps
    int nstrips;           // ceil(nx / TX)
    int ntiles_y;          // tile rows of the launch's tile shape (FP64: ny)
    int stress_every;
};

// Arguments of the (multi-lattice) step kernel.
template <typename C>
struct BatchArgs {
    Coef<C> k;                  // coefficients shared by all lattices of the launch
    const LatDesc<C>* lat;      // nlat descriptors
    int nlat;
    int nitems;                 // total work items
    // Work items (lattice, strip, first tile row, end tile row; FP64: first row,
    // end row), grouped by CTA: CTA b takes items cta_items[b] .. cta_items[b + 1] - 1 in order.
    const int4* items;
    const int* cta_items;
    unsigned int* ticket;       // CTA arrival counter of the launch (zero between launches)
    // Launches come in windows of consecutive steps: this one takes step
    // DevStats::t + step_k, and the window's last one has advance = the
    // window's steps (else 0), by which it moves the lattices' counters.
    int step_k, advance;
    int l2_resident;            // one buffer of all lattices fits in L2: cache-policy hints
    int early_release;          // kernel variant bit 2 only: a tile's ring slots are refilled
                                // after its density phase (else after its site phase)
};

// The device-side state that an initialising kernel leaves with the
// populations: counters cleared but for these, wall momentum totals zero.
struct StateInit {
    DevStats* st;          // null: leave the state alone
    long long t, next_sample;
    int pull;
    double* wsum;          // nwsum totals (0: none)
    int nwsum;
};

// Observe-mode outputs (the kernel writes FP64 planes of nx*ny values).
enum ObsKind : int { OBS_NONE = 0, OBS_FIELDS = 1, OBS_POPS = 2, OBS_TOTALS = 3 };

template <typename C>
struct StepArgs {
    Geom g;
    Coef<C> k;
    void* fout;            // output population buffer (padded planes)
    DevStats* st;
    double* slots;         // per-CTA partial sums
    int pull;              // 1: input holds post-collision f*(t-1); 0: f(t) in place
    const float2* mom;     // FP32: the state's moments [3][ny][nx] where it is held by them, else null
    int obs;               // ObsKind; OBS_NONE = a time step
    // OBS_FIELDS: rho_A, rho_B, u_x, u_y (null: not wanted), OBS_POPS: the first
    // plane's address; device memory or pinned host memory
    double* obs_dst[4];
    int q0, q1;            // OBS_POPS: planes [q0, q1) written
    const double* wsum;    // Couette: the strips' wall momentum totals, [2][nstrips]
    int nstrips;
};

// Tile shapes of the step kernels (see Layout and MLayout).
//  SHAPE_8    8-row tiles, one site per thread, one CTA per SM;
//  SHAPE_16   16-row tiles, two sites per thread, one CTA per SM;
//  SHAPE_8X2  8-row tiles, two sites per thread, two CTAs of half the threads
//             per SM (16-bit formats: their shared memory holds two);
//  SHAPE_D8   8-row tiles, one site per thread, the tile loaded by plain loads
//             (FP32 and 16-bit populations, few tiles: see k_step_d);
//  SHAPE_M8, SHAPE_M8X2  8-row tiles with one site per thread, and with
//             two and two CTAs per SM, of the moment kernel (FP32,
//             tau = 1, velocity shift: see k_step_m).
enum Shape : int { SHAPE_8 = 1, SHAPE_16 = 2, SHAPE_8X2 = 3, SHAPE_D8 = 4, SHAPE_M8 = 5, SHAPE_M8X2 = 6 };
constexpr bool shape_moments(int shape) { return shape >= SHAPE_M8; }
constexpr bool has_shape(int precision, int shape) {
    return shape == SHAPE_8 || (shape == SHAPE_16 && precision != LB_FP64) ||
           (shape == SHAPE_8X2 && (precision == LB_FP16_OFFSET || precision == LB_BF16_OFFSET)) ||
           (shape == SHAPE_D8 && precision != LB_FP64) ||
           (shape_moments(shape) && precision == LB_FP32);
}
constexpr int shape_rows(int shape) { return shape == SHAPE_16 ? 16 : 8; }
constexpr int shape_ctas(int shape) {   // per SM
    return shape == SHAPE_8X2 || shape == SHAPE_M8X2 ? 2 : 1;
}

// Host-side launch helpers (lb_dispatch.cu).
int kernel_smem_bytes(int precision);
int kernel_tile_x(int precision);
int kernel_tile_y(int precision);
int kernel_ghost_x(int precision);
int kernel_elem_bytes(int precision);
int kernel_smem_obs_bytes(int precision);
int kernel_block_rows(int precision);
int kernel_scale_log2(int precision);
// 1 if the step kernel of a shape leaves through a staging tile (its periodic
// ghost copies are then separate stores after the tile)
int kernel_staged(int precision, int shape);

// Step: the persistent multi-lattice kernel (args: BatchArgs<C>), variant
// bit 0 = every lattice periodic, bit 1 = general forcing, bit 2 = 1 - omega
// rounds to zero for both species (the collision reads no populations), in one of the
// precision's tile shapes; without args the kernel is only made ready (call it so
// before capturing launches into a graph).  Observe: one lattice (args: StepArgs<C>, tin: tile-box
// load map), at most one CTA per 8-row tile.
cudaError_t launch_step(int precision, const void* args, int variant, int shape, dim3 grid,
                        cudaStream_t s);
cudaError_t launch_observe(int precision, const CUtensorMap* tin, const void* args, dim3 grid,
                           cudaStream_t s);
// Initial states (see k_init).  fields: rho_A, rho_B, u_x, u_y (velocities may
// be null: zero), in device memory or pinned host memory.
cudaError_t launch_init_seeded(int precision, const Geom& g, const void* coef, void* fout,
                               double rho0, double amp, double u_wall, int init_shear,
                               unsigned long long seed, const StateInit& state, cudaStream_t s);
cudaError_t launch_init_fields(int precision, const Geom& g, const void* coef, void* fout,
                               const double* const fields[4], const StateInit& state, cudaStream_t s);

// FP32: the populations f* of a state held by its moments, into a population
// buffer (with its ghost copies).
cudaError_t launch_expand(const Geom& g, const Coef<float>& k, const float2* mom, void* fout,
                          cudaStream_t s);

// Restore directions [i0, i1) from FP64 populations: species s of direction i at
// pops + s species + (i - i0) direction (device or pinned host memory).
cudaError_t launch_load_pops(int precision, const Geom& g, const void* coef, void* fout,
                             const double* pops, size_t species, size_t direction, int i0, int i1,
                             const StateInit& state, cudaStream_t s);

// Per-precision launchers, explicitly instantiated by the compilations of
// lb_kernels.cu (-DLB_PREC=P; launch_step_shape with -DLB_PART=SH).
template <int P, int SH>
cudaError_t launch_step_shape(const void* args, int variant, dim3 grid, cudaStream_t s);
template <int P>
cudaError_t launch_step_prec(const void* args, int variant, int shape, dim3 grid, cudaStream_t s);
template <int P>
cudaError_t launch_observe_prec(const CUtensorMap* tin, const void* args, dim3 grid,
                                cudaStream_t s);
template <int P>
cudaError_t launch_load_pops_prec(const Geom& g, const void* coef, void* fout, const double* pops,
                                  size_t species, size_t direction, int i0, int i1,
                                  const StateInit& state, cudaStream_t s);
template <int P>
cudaError_t launch_init_prec(const Geom& g, const void* coef, void* fout, const double* const* fields,
                             double rho0, double amp, double u_wall, int init_shear,
                             unsigned long long seed, const StateInit& state, cudaStream_t s);

}  // namespace lbgb
