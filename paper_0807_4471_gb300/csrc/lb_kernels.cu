// lb_kernels.cu -- sm_103a kernels of the two-species multi-range
// pseudo-potential lattice Boltzmann step (Benzi, Chibbaro & Succi,
// arXiv:0807.4471, Eqs. (1)-(2)).
//
// One launch of k_step advances every site of a set of lattices by one time
// step.  Layout in HBM: 9 direction planes, each a ghost-padded
// [ny + 6][pitch] array of interleaved (A, B) pairs of the storage type,
// holding offsets h_i = f_i - w_i rho_ref.  The buffer read by a step holds
// the post-collision populations f*(t-1) of the previous step; streaming is
// a pull, f_i(r, t) = f*_i(r - c_i, t - 1).
//
// k_step is persistent: one CTA per SM walks its work items (a lattice's
// strip of TX x TY tiles, one after the other).  Per tile:
//  1. TMA: 3-D box loads bring f* in 8-row blocks (both species, 9 planes,
//     the strip plus its ghost columns) into a ring of shared-memory slots,
//     several blocks ahead.  The ghost columns/rows of the padded planes
//     hold periodic copies, so a box never wraps.
//  2. density phase: density and pseudo-potential deviations on the tile
//     plus a 2-row halo (halfway bounce-back at Couette walls; mirrored
//     beyond a wall), and at tau = 1 the momenta of the tile's sites.
//  3. site phase, one or two sites per thread: the force of Eq. (2) from the
//     shared deviation window (row sums of the 24-neighbour stencil and of
//     the cross term), the forced BGK relaxation of Eq. (1), the write-back
//     (staging tile + TMA bulk tensor store, or direct stores) and the
//     periodic ghost copies.
//  4. Couette: the wall sites' momentum exchange, summed per strip in FP64
//     by the next launch (a window's last launch: at its end) and, at sampled
//     steps, added to the strip's total.
// Two more step kernels share its site arithmetic: k_step_d, for lattices with
// few tiles (a shorter chain of latencies), and k_step_m, for FP32 at tau = 1
// (the state held by its moments).  There is no dense contraction anywhere, so
// no tensor cores are used.
//
// Compiled once per storage precision and part (-DLB_PREC=0..3 -DLB_PART=k): part 0
// is the observe and initialising kernels and the launchers' dispatch, part k >= 1
// the step kernels of tile shape k (Shape; SHAPE_M8: both moment shapes).  A
// unit's kernels are one module to the driver, which loads it at the first use of
// one of them, at a cost that grows with all of them: with one module per
// precision the first initialisation of a process took 1.16 ms and its first step
// 0.68 ms (FP16), now 0.26 and 0.36.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <type_traits>
#include <utility>

#include "lb_internal.h"
#include "lb_layout.cuh"

#if !defined(LB_PREC) || !defined(LB_PART)
#error "compile lb_kernels.cu with -DLB_PREC=0..3 -DLB_PART=0..5"
#endif

namespace lbgb {

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void tma_prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y,
                                            int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
// The same box load, and the bulk tensor store of a shared-memory box to
// global memory (bulk group), with an L2 cache policy (createpolicy).
__device__ __forceinline__ void tma_load_3d_hint(void* dst, const CUtensorMap* map, int x, int y,
                                                 int z, uint64_t* bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)),
        "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_store_3d_hint(const CUtensorMap* map, const void* src, int x,
                                                  int y, int z, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group.L2::cache_hint"
        " [%0, {%2, %3, %4}], [%1], %5;" ::"l"(reinterpret_cast<uint64_t>(map)),
        "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "l"(policy)
        : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_normal() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until the committed bulk stores have finished reading shared memory.
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// Wait until the committed bulk stores have completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Programmatic dependent launch: wait for the grids this one depends on to
// complete (their writes visible), and let this grid's dependents be
// scheduled onto SMs as this grid's CTAs retire.  Both are no-ops when the
// launch carries no programmatic dependency.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Arrival at a launch's CTA counter: the old count, with release semantics
// for this CTA's writes (made ordered before by a CTA barrier) and acquire
// semantics for those of the CTAs that arrived before, at GPU scope.
__device__ __forceinline__ unsigned int ticket_arrive(unsigned int* ticket) {
    unsigned int old;
    asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(old) : "l"(ticket) : "memory");
    return old;
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: each try_wait suspends for a hardware-chosen interval, so the
// default bound is a few seconds at most.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  int limit = 1 << 22) {
    for (int it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// ---------------------------------------------------------- site helpers
// Pair (A, B) of plane i at site (x, y) in the padded global buffer, in
// units of pairs: row stride `pitch`, plane stride rows * pitch.
template <typename T2>
__device__ __forceinline__ void put2(T2* base, const Geom& g, int i, int x, int y, T2 v) {
    const long long pl = (long long)g.rows * g.pitch;
    T2* p = base + i * pl + (long long)(y + kGY) * g.pitch + (x + g.gx);
    const int dX = (x < 3) ? g.nx : ((x >= g.nx - 3) ? -g.nx : 0);
    long long dY = 0;
    if (g.periodic) dY = (y < 3) ? (long long)g.ny * g.pitch : ((y >= g.ny - 3) ? -(long long)g.ny * g.pitch : 0);
    p[0] = v;
    if (dX) p[dX] = v;
    if (dY) {
        p[dY] = v;
        if (dX) p[dY + dX] = v;
    }
}

// ((h0 + h1) + (h2 + h3)) + ((h4 + h5) + (h6 + h7)) + h8, per species.
template <typename C2>
__device__ __forceinline__ C2 sum9(const C2 h[9]) {
    return padd(padd(padd(padd(h[0], h[1]), padd(h[2], h[3])), padd(padd(h[4], h[5]), padd(h[6], h[7]))),
                h[8]);
}

// The offsets h_i(r, t) of both species at lattice row y, as (A, B) pairs,
// in the storage scale of precision P.
// bm, b0, bp point at the site's pair in the staged rows y-1, y, y+1 of
// plane 0 (plane i is PS pairs further).  pull = 1: streamed from
// h*(r - c_i, t - 1), with halfway bounce-back at the Couette walls:
// f_i = f*_opp(i)(r) + 6 w_i rho_w (c_i . u_w), rho_w the pre-streaming
// density of the boundary node, rho_ref + sum_j h*_j(r).  pull = 0: the
// state in place.
template <int P, int PS>
__device__ __forceinline__ void load_site(const typename Prec<P>::T2* bm,
                                          const typename Prec<P>::T2* b0,
                                          const typename Prec<P>::T2* bp, int y, bool per,
                                          int pull, const Geom& g,
                                          const LatVals<typename Prec<P>::C>& v,
                                          typename Prec<P>::C2 h[9]) {
    typedef typename Prec<P>::C C;
    typedef typename Prec<P>::C2 C2;
    if (pull) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const typename Prec<P>::T2* r = cy(i) == 1 ? bm : (cy(i) == -1 ? bp : b0);
            h[i] = dec2(r[i * PS - cx(i)]);
        }
        if (!per && (y == 0 || y == g.ny - 1)) {
            C2 sv[9];
#pragma unroll
            for (int j = 0; j < 9; ++j) sv[j] = dec2(b0[j * PS]);
            const C2 rw = pfma(sum9(sv), pset(inv_scale_of<P>()), pset(v.rho_ref));
            const int up = (y == 0);                 // links arriving upward
            const C uw = up ? -v.u_wall : v.u_wall;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if ((up && cy(i) == 1) || (!up && cy(i) == -1)) {
                    const C m = scale_of<P>() * C(6) * wgt<C>(i) * (C(cx(i)) * uw);
                    h[i] = pfma(pset(m), rw, sv[opp(i)]);
                }
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = dec2(b0[i * PS]);
    }
}

#if LB_PREC == 0
static __device__ const ExpTable g_exp_tab = {{LB_EXP_TABLE}, {LB_EXP_ARGS}};
#endif

// Deviation of the pseudo-potential from Psi(rho_ref), both species:
// Psi(rho_ref + d) - Psi(rho_ref) = -P exp(-rho_ref/rho0) expm1(-d/rho0).
// FP64: without the factor -P exp(-rho_ref/rho0), which neg_psi carries; tab:
// the exponential table.
__device__ __forceinline__ float2 dpsi_of(float2 d, const LatVals<float>& v, const ExpTable*) {
    return pmul(pset(-v.psi_scale), pexpm1(pmul(d, pset(-v.inv_rho0))));
}
__device__ __forceinline__ double2 dpsi_of(double2 d, const LatVals<double>& v, const ExpTable* tab) {
    return pexpm1_scaled(d, v.exp_c, v.inv_rho0, tab);
}
// -Psi_s(r) from the window value; FP64: times the factor that the stencil
// sums of the window values lack, -psi_scale.  (Not as psi_ref psi_scale -
// psi_scale^2 E, two operations less a site: psi_scale^2 leaves the normal numbers
// where rho_ref / rho0 is above 354.)
__device__ __forceinline__ float2 neg_psi(float2 dpsi, const LatVals<float>& v) {
    return psub(pset(-v.psi_ref), dpsi);
}
__device__ __forceinline__ double2 neg_psi(double2 E, const LatVals<double>& v) {
    return pmul(pset(-v.psi_scale), pfma(pset(v.psi_scale), E, pset(-v.psi_ref)));
}
// Adds 0 * rho to nf: NaN from the first inf or NaN density on, else zero.
// (FP64: by the exponent bits, without an FP64 operation.)
__device__ __forceinline__ void note_nonfinite(float2 rho, float2& nf) { nf = pfma(rho, pset(0.0f), nf); }
__device__ __forceinline__ void note_nonfinite(double2 rho, double2& nf) {
    const int a = __double2hiint(rho.x) & 0x7ff00000, b = __double2hiint(rho.y) & 0x7ff00000;
    if (max(a, b) == 0x7ff00000) nf.x = __hiloint2double(0x7ff80000, 0);
}

// Momentum j = sum_i c_i f_i of both species from the offsets (sum_i w_i c_i
// = 0, so the offsets carry all of j), in the compute scale.
// SCALED = false: left in the storage scale (the caller folds the scale,
// a power of two, into a later factor).
template <int P, bool SCALED = true>
__device__ __forceinline__ void moments(const typename Prec<P>::C2 h[9], typename Prec<P>::C2& jx,
                                        typename Prec<P>::C2& jy) {
    typedef typename Prec<P>::C2 C2;
    const C2 d57 = psub(h[5], h[7]), d68 = psub(h[6], h[8]);
    jx = padd(psub(h[1], h[3]), psub(d57, d68));
    jy = padd(psub(h[2], h[4]), padd(d57, d68));
    if constexpr (SCALED && Prec<P>::SCALE_LOG2 != 0) {
        jx = pmul(jx, pset(inv_scale_of<P>()));
        jy = pmul(jy, pset(inv_scale_of<P>()));
    }
}

// Density and pseudo-potential deviations (rho - rho_ref, Psi - Psi(rho_ref))
// of both species at one site; with J, also the site's momentum, in the
// storage scale.
template <int P, int PS, bool J = false>
__device__ __forceinline__ void cell_dev(const typename Prec<P>::T2* bm,
                                         const typename Prec<P>::T2* b0,
                                         const typename Prec<P>::T2* bp, int y, bool per, int pull,
                                         const Geom& g, const LatVals<typename Prec<P>::C>& v,
                                         typename Prec<P>::C2& r, typename Prec<P>::C2& q,
                                         const ExpTable* tab, typename Prec<P>::C2* j = nullptr) {
    typename Prec<P>::C2 h[9];
    load_site<P, PS>(bm, b0, bp, y, per, pull, g, v, h);
    r = sum9(h);
    if constexpr (Prec<P>::SCALE_LOG2 != 0) r = pmul(r, pset(inv_scale_of<P>()));
    q = dpsi_of(r, v, tab);
    if constexpr (J) moments<P, false>(h, j[0], j[1]);
}

// Post-collision offsets of both species (Eq. (1), BGK toward the
// equilibrium at velocity u, per species), written with z = 1.5u (half of
// 3u, so that the halves below are exact and take no operation):
//   h*_i = (1 - omega) h_i + omega heq_i [+ 3 w_i c_i . F for the source scheme],
//   heq_i = f^eq_i - w_i rho_ref = w_i [d_rho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u^2)]
//         = w_i [Q + (2 rho) (c.z) + (2 rho) (c.z)^2],  Q = d_rho - (2/3) rho z^2,
// evaluated per pair (i, opp(i)), whose c.z differ only in sign:
// heq = w (g +- 2 rho c.z) with g = Q + (2 rho c.z) (c.z).  h and out are in
// the storage scale SC (a power of two); k.omw holds omega SC w per class
// of |c|^2 and k.omm = 1 - omega.
//
// TAU1 (omega = 1): h*_i = heq_i, taken per class c of |c_i|^2 as
//   h*_{i, opp(i)} = E +- kv,  E = T_c + kv (c.z),  kv = K_c (c.z),
// with T_c = omega S w_c Q and K_c = 2 omega S w_c rho per site; h is not read.
template <typename C, typename C2, bool SRC, bool TAU1 = false>
__device__ __forceinline__ void collide(const C2 h[9], C2 out[9], C2 drho, C2 rho, C2 zx, C2 zy,
                                        const Coef<C>& k, C2 Fx, C2 Fy, C SC) {
    const C2 Q = pfma(pmul(rho, pset(C(-4) / C(6))), pfma(zx, zx, pmul(zy, zy)), drho);
    out[0] = TAU1 ? pmul(k.omw[0], Q) : pfma(k.omw[0], Q, pmul(k.omm, h[0]));
    C2 T[2], K[2], rho2;
    if (TAU1) {
        T[0] = pmul(k.omw[1], Q);
        T[1] = pmul(k.omw[2], Q);
        K[0] = pmul(k.omw2[0], rho);
        K[1] = pmul(k.omw2[1], rho);
    } else {
        rho2 = padd(rho, rho);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = q == 0 ? 1 : (q == 1 ? 2 : (q == 2 ? 5 : 6));   // c.z = zx, zy, zx+zy, zy-zx
        const int j = opp(i);
        const C2 cz = q == 0 ? zx : (q == 1 ? zy : (q == 2 ? padd(zx, zy) : psub(zy, zx)));
        if (TAU1) {
            const C2 kv = pmul(K[q >> 1], cz);
            const C2 E = pfma(kv, cz, T[q >> 1]);
            out[i] = padd(E, kv);
            out[j] = psub(E, kv);
        } else {
            const C2 ow = k.omw[q < 2 ? 1 : 2];
            const C2 rv = pmul(rho2, cz);
            const C2 g = pfma(rv, cz, Q);
            out[i] = pfma(ow, padd(g, rv), pmul(k.omm, h[i]));
            out[j] = pfma(ow, psub(g, rv), pmul(k.omm, h[j]));
        }
        if (SRC) {
            const C w3 = C(3) * SC * wgt<C>(i);
            const C2 S = pmul(pset(w3), pfma(pset(C(cx(i))), Fx, pmul(pset(C(cy(i))), Fy)));
            out[i] = padd(out[i], S);
            out[j] = psub(out[j], S);
        }
    }
}

// ------------------------------------------------------- force of Eq. (2)
// The stencil sums of Eq. (2) are taken row by row.  For the stencil row at
// vertical offset dy of a site, with the row's deviations q(dx), dx = -2..2
// (Psi for the like-species terms, rho for the cross term), and weights
// K(d) that depend on |d|^2 = dx^2 + dy^2 only:
//   sum_dx K(d) d_x q(dx) = K(1,|dy|) [q(1) - q(-1)] + 2 K(2,|dy|) [q(2) - q(-2)],
//   sum_dx K(d) d_y q(dx) = dy [K(0,|dy|) q(0) + K(1,|dy|) (q(1) + q(-1))
//                              + K(2,|dy|) (q(2) + q(-2))].
// (The reference values of Psi and rho drop out: sum_d K(d) d = 0.)  The
// differences and sums of a row are shared by every site whose stencil
// holds the row; each site adds its rows in a fixed order (x: dy = -2 .. 2;
// y: the rows above minus the rows below, each part in the order of dy), so
// a site's force is the same whether it shares rows with another or not.

// The shared quantities of one stencil row, p at the site's column.
template <typename C2>
struct Row5 {
    C2 d1, d2, s1, s2, q0;
};
template <typename C2>
__device__ __forceinline__ Row5<C2> row5(const C2* p) {
    const C2 m2 = p[-2], m1 = p[-1], q0 = p[0], p1 = p[1], p2 = p[2];
    Row5<C2> r;
    r.d1 = psub(p1, m1);
    r.d2 = psub(p2, m2);
    r.s1 = padd(p1, m1);
    r.s2 = padd(p2, m2);
    r.q0 = q0;
    return r;
}
template <typename C2>
struct Row3 {
    C2 e, t, q0;
};
template <typename C2>
__device__ __forceinline__ Row3<C2> row3(const C2* p) {
    const C2 m1 = p[-1], q0 = p[0], p1 = p[1];
    Row3<C2> r;
    r.e = psub(p1, m1);
    r.t = padd(p1, m1);
    r.q0 = q0;
    return r;
}

// Like-species row at offset dy (|dy| <= 2) into the x and y sums, with the
// weights KC = {K(1), K(2), K(5), 2K(4), 2K(5), 2K(8)}: x takes
// K(1,|dy|) = K(1), K(2), K(5) and 2K(2,|dy|) = 2K(4), 2K(5), 2K(8) for
// |dy| = 0, 1, 2; y takes {K(1), K(2), K(5)} for |dy| = 1 and
// {2K(4), 2K(5), 2K(8)} for |dy| = 2.  The y sum is kept as two chains,
// rows below the site (fyn: dy = -2, -1) and above it (fyp: dy = 1, 2),
// each started by its first row; fy = fyp - fyn.
template <typename C, typename C2>
__device__ __forceinline__ void like_row(int dy, const Row5<C2>& r, const Coef<C>& k, C2& fx,
                                         C2& fyp, C2& fyn) {
    const int a = dy < 0 ? -dy : dy;
    fx = pfma(a == 0 ? k.KC[0] : (a == 1 ? k.KC[1] : k.KC[2]), r.d1, fx);
    fx = pfma(a == 0 ? k.KC[3] : (a == 1 ? k.KC[4] : k.KC[5]), r.d2, fx);
    if (a != 0) {
        C2& t = dy > 0 ? fyp : fyn;
        const C2 K0 = a == 1 ? k.KC[0] : k.KC[3];
        t = (dy == -2 || dy == 1) ? pmul(K0, r.q0) : pfma(K0, r.q0, t);
        t = pfma(a == 1 ? k.KC[1] : k.KC[4], r.s1, t);
        t = pfma(a == 1 ? k.KC[2] : k.KC[5], r.s2, t);
    }
}
// Cross-species row at offset dy (|dy| <= 1), D2Q9 weights WC = {w(1), w(2)};
// qy is taken as qyp - qyn, the rows above and below.
template <typename C, typename C2>
__device__ __forceinline__ void cross_row(int dy, const Row3<C2>& r, const Coef<C>& k, C2& qx,
                                          C2& qyp, C2& qyn) {
    qx = pfma(dy == 0 ? k.WC[0] : k.WC[1], r.e, qx);
    if (dy != 0) {
        C2& u = dy > 0 ? qyp : qyn;
        u = pfma(k.WC[1], r.t, pmul(k.WC[0], r.q0));
    }
}

// Stencil sums of NS vertically adjacent sites.  ps, rr: the Psi and rho
// deviation rows (row stride RXS) at the sites' column, starting two rows
// above the first site.  Out, per site s: fx, fy = sum_d K_s(d) d Psi_s(r+d),
// qx, qy = sum_d w(d) d rho_s(r+d) (species not yet swapped), and the site's
// own Psi and rho deviations.
template <int NS, int RXS, typename C, typename C2>
__device__ __forceinline__ void force_sums(const C2* ps, const C2* rr, const Coef<C>& k, C2 fx[NS],
                                           C2 fy[NS], C2 qx[NS], C2 qy[NS], C2 dpsi[NS],
                                           C2 drho[NS]) {
    const C2 z = pset(C(0));
    C2 fyp[NS], fyn[NS], qyp[NS], qyn[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) fx[s] = qx[s] = z;
#pragma unroll
    for (int r = 0; r < NS + 4; ++r) {
        const Row5<C2> w = row5(ps + r * RXS);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int dy = r - 2 - s;
            if (dy >= -2 && dy <= 2) like_row(dy, w, k, fx[s], fyp[s], fyn[s]);
            if (dy == 0) dpsi[s] = w.q0;
        }
    }
#pragma unroll
    for (int r = 1; r < NS + 3; ++r) {
        const Row3<C2> w = row3(rr + r * RXS);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int dy = r - 2 - s;
            if (dy >= -1 && dy <= 1) cross_row(dy, w, k, qx[s], qyp[s], qyn[s]);
            if (dy == 0) drho[s] = w.q0;
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        fy[s] = psub(fyp[s], fyn[s]);
        qy[s] = psub(qyp[s], qyn[s]);
    }
}

// FP64: the stencil sums of a warp's row of sites, taken column by column.
// The FP64 step is bound by its FP64 operations (two lanes per SM and clock),
// while shuffles and shared-memory loads are nearly free beside them, so the
// sums over a window column are taken once, by a lane of the column's own, and
// shared along the row by shuffles: with v_k = q(+k) + q(-k) and
// w_k = q(+k) - q(-k) of a column (k rows above and below, v_0 = q) and
// D_k = v_k(+1) - v_k(-1) across the columns beside it,
//   sum_d K d_x q: A + B(+1) + B(-1),
//     A = K(1) D_0 + K(2) D_1 + K(5) D_2,  B = 2K(4) D_0 + 2K(5) D_1 + 2K(8) D_2,
//   sum_d K d_y q: C_0 + C_1(+1) + C_1(-1) + C_2(+2) + C_2(-2),
//     C_0 = K(1) w_1 + 2K(4) w_2,  C_1 = K(2) w_1 + 2K(5) w_2,  C_2 = K(5) w_1 + 2K(8) w_2
// (arguments: columns right or left), 26 FP64 operations per species against
// 41 row by row; the cross sums likewise in 7 against 13.  Differences come
// before weights in both directions, as row by row: the sums of a smooth field are
// small differences, and weighted columns subtracted afterwards (23 and 6
// operations; 50 steps of a 512^2 Couette lattice 6869 us against 7063) left the x
// force with 1.6 to 1.75 times the y force's error, now within 8 %.
// ps, rr: the Psi and rho window rows (row stride RXS) at window column
// `lane`, starting two rows above the sites; a lane's site is two columns to
// the right of its window column.  All lanes of the warp call it.
__device__ __forceinline__ double2 shfl_down2(double2 v, int n) {
    return make_double2(__shfl_down_sync(0xffffffffu, v.x, n), __shfl_down_sync(0xffffffffu, v.y, n));
}
template <int RXS>
__device__ __forceinline__ void force_sums_warp(const double2* ps, const double2* rr,
                                                const Coef<double>& k, double2& fx, double2& fy,
                                                double2& qx, double2& qy, double2& dpsi,
                                                double2& drho) {
    {
        const double2 q0 = ps[2 * RXS];
        const double2 v1 = padd(ps[3 * RXS], ps[RXS]), w1 = psub(ps[3 * RXS], ps[RXS]);
        const double2 v2 = padd(ps[4 * RXS], ps[0]), w2 = psub(ps[4 * RXS], ps[0]);
        dpsi = shfl_down2(q0, 2);
        // of the column to the right of the lane's own
        const double2 D0 = psub(dpsi, q0), D1 = psub(shfl_down2(v1, 2), v1), D2 = psub(shfl_down2(v2, 2), v2);
        const double2 A = pfma(k.KC[2], D2, pfma(k.KC[1], D1, pmul(k.KC[0], D0)));
        const double2 B = pfma(k.KC[5], D2, pfma(k.KC[4], D1, pmul(k.KC[3], D0)));
        fx = padd(shfl_down2(A, 1), padd(shfl_down2(B, 2), B));
        const double2 C0 = pfma(k.KC[3], w2, pmul(k.KC[0], w1));
        const double2 C1 = pfma(k.KC[4], w2, pmul(k.KC[1], w1));
        const double2 C2 = pfma(k.KC[5], w2, pmul(k.KC[2], w1));
        fy = padd(padd(shfl_down2(C0, 2), padd(shfl_down2(C1, 3), shfl_down2(C1, 1))),
                  padd(shfl_down2(C2, 4), C2));
    }
    {
        const double2 r0 = rr[2 * RXS];
        const double2 v = padd(rr[3 * RXS], rr[RXS]), w = psub(rr[3 * RXS], rr[RXS]);
        drho = shfl_down2(r0, 2);
        qx = shfl_down2(pfma(k.WC[0], psub(drho, r0), psub(shfl_down2(v, 2), v)), 1);   // weights 4, 1
        qy = pfma(k.WC[0], shfl_down2(w, 2), padd(shfl_down2(w, 3), shfl_down2(w, 1)));
    }
}

// Plain global stores of a stored pair, with an L2 cache policy.
__device__ __forceinline__ void st_pair(float2* p, float2 v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(v.x), "f"(v.y),
                 "l"(pol));
}
__device__ __forceinline__ void st_pair(double2* p, double2 v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v2.f64 [%0], {%1, %2}, %3;" ::"l"(p), "d"(v.x), "d"(v.y),
                 "l"(pol));
}
template <typename T2>
__device__ __forceinline__ void st_pair(T2* p, T2 v, uint64_t pol) {   // 16-bit pairs
    static_assert(sizeof(T2) == 4, "a pair of 16-bit values");
    asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(p),
                 "r"(*reinterpret_cast<const uint32_t*>(&v)), "l"(pol));
}

// Random word of site (x, y) for the stochastic rounding of its stored
// pairs, from key, the hash of the lattice's step: sites (x, 2m) and
// (x, 2m + 1) share one hash of (x, 2m) -- the second site takes it times an
// odd constant (a bijection, so each word is uniform) -- whichever thread
// updates them.
__device__ __forceinline__ uint32_t sr_hash(uint32_t key, int x, int y, int nx) {
    return hash32(key ^ (uint32_t)((y & ~1) * nx + x));
}
__device__ __forceinline__ uint32_t sr_word(uint32_t h, int y) {
    return (y & 1) ? h * 0x2c1b3c6du : h;
}

// Where a site update sends its result.
enum SiteSink : int { SINK_STAGE = 0, SINK_GLOBAL = 1 };
template <typename T2>
struct SiteOut {
    T2* stage;             // SINK_STAGE: staging tile slot of the site (plane 0)
    T2* gout;              // SINK_GLOBAL: the site's pair in plane 0 of the output buffer
    long long plane;       // SINK_GLOBAL: plane stride (pairs)
    long long gdy;         // SINK_GLOBAL: offset of the periodic image in y (0: none)
    int gdx;               // SINK_GLOBAL: offset of the periodic image in x (0: none)
    uint64_t pol;          // SINK_GLOBAL: L2 policy of the stores
    uint32_t rbits;        // stochastic rounding: the site's random word (sr_word)
    int valid;             // 0: a site beyond the lattice, computed only to keep
                           // the site updates of a thread free of branches:
                           // its global stores and non-finite flag are dropped
    void* wallx;           // the lattice's wall-momentum pairs, [2][nx] compute type
};

// Body acceleration along x at lattice row y.
template <typename C>
__device__ __forceinline__ C body_accel(const Coef<C>& k, const LatVals<C>& v, int y) {
    C acc = k.g_x;
    if (k.kolmo_amp != C(0)) acc += k.kolmo_amp * csin(v.kolmo_w * C(y));
    return acc;
}
// Eq. (2): F_s = -Psi_s(r) sum_d K_s(d) d Psi_s(r + d)
//               - (G_X/rho0) rho_s(r) sum_d w(d) d rho_s'(r + d);
// species A feels rho_B, so the cross sums are used swapped.
template <bool GEN, typename C, typename C2>
__device__ __forceinline__ void site_force(C2 fxl, C2 fyl, C2 qx, C2 qy, C2 dpsi, C2 rho, int y,
                                           const LatVals<C>& v, const Coef<C>& k, C2& Fx, C2& Fy) {
    const C2 npc = neg_psi(dpsi, v);                       // -Psi_s(r)
    const C2 ng = pmul(pset(-v.gx_rho0), rho);             // -(G_X/rho0) rho_s
    Fx = pfma(npc, fxl, pmul(ng, pair(qx.y, qx.x)));
    Fy = pfma(npc, fyl, pmul(ng, pair(qy.y, qy.x)));
    if (GEN && k.has_accel) Fx = pfma(rho, pset(body_accel(k, v, y)), Fx);
}
// Velocities of the forced BGK relaxation (Eq. (1)), as z = 1.5u: the common
// velocity u' = sum_s (j_s/tau_s) / sum_s (rho_s/tau_s) and, unless `source`,
// the shift u_s = u' + tau_s F_s/rho_s.  (Selects, not branches: an empty site
// has u' = 0 and no shift.)  TAU1: omega = 1 exactly, and the products are the
// values themselves; j is taken in the storage scale of precision P, whose
// inverse the factor 1.5 / den takes up (both exact powers of two apart).
template <int P, bool TAU1, typename C, typename C2>
__device__ __forceinline__ void site_velocity(C2 rho, C2 jx, C2 jy, C2 Fx, C2 Fy, bool source,
                                              const Coef<C>& k, C2& zx, C2& zy) {
    const C2 om = pair(k.omega[0], k.omega[1]);
    const C2 ro = TAU1 ? rho : pmul(rho, om), jxo = TAU1 ? jx : pmul(jx, om),
             jyo = TAU1 ? jy : pmul(jy, om);
    const C den = ro.x + ro.y;
    const C inv = den != C(0) ? (TAU1 ? C(1.5) * inv_scale_of<P>() : C(1.5)) * recip(den) : C(0);
    zx = pset((jxo.x + jxo.y) * inv);
    zy = pset((jyo.x + jyo.y) * inv);
    if (!source) {
        const C2 tr = pair(rho.x != C(0) ? k.tau15[0] * recip(rho.x) : C(0),
                           rho.y != C(0) ? k.tau15[1] * recip(rho.y) : C(0));
        zx = pfma(tr, Fx, zx);
        zy = pfma(tr, Fy, zy);
    }
}
// x-momentum handed to the wall by the links that will bounce back at the next
// streaming, from the stored (rounded) values sv (storage scale of P):
// sum_i c_ix (f*_i + f_opp), f_opp = f*_i - 6 w_i rho_w (c_i . u_w),
// over the three links i leaving through the wall, which is
// 2 (f*_a - f*_b) - 6 rho_w u_w (w_a + w_b) = 2 (f*_a - f*_b) - rho_w u_w / 3
// with (a, b) = (8, 7) at the bottom wall and (5, 6) at the top
// (c_ax = 1, c_bx = -1; w_a = w_b, so the offsets' difference is the
// populations').  One compute-type value per site and species, kept
// in the lattice's wall columns for the next launch's sums (wall_sums).
template <int P, typename C, typename C2>
__device__ __forceinline__ C2 wall_momentum(const C2 sv[9], bool down, const LatVals<C>& v) {
    const C uw = down ? -v.u_wall : v.u_wall;
    const C2 rw2 = pfma(sum9(sv), pset(inv_scale_of<P>()), pset(v.rho_ref));
    const C2 dd = pmul(down ? psub(sv[8], sv[7]) : psub(sv[5], sv[6]), pset(inv_scale_of<P>()));
    return psub(pmul(pset(C(2)), dd), pmul(rw2, pset(uw * (C(1) / C(3)))));
}

// One lattice site, given its force sums: moments from its pulled
// populations, the force of Eq. (2), the forced BGK collision and the
// write-back.  Both species are carried as (A, B) pairs throughout.  TAU1
// (omega = 1 for both species): the collision needs the populations only
// through j, which the caller passes in jg = {jx, jy} (in the storage scale);
// bm, b0 and bp are not read.  *nf accumulates 0 * rho, which turns NaN at an
// inf or NaN density and stays zero otherwise.
template <int P, bool GEN, int PS, int SINK, bool TAU1 = false>
__device__ __forceinline__ void site_update(
    const typename Prec<P>::T2* bm, const typename Prec<P>::T2* b0,
    const typename Prec<P>::T2* bp, typename Prec<P>::C2 fxl, typename Prec<P>::C2 fyl,
    typename Prec<P>::C2 qx, typename Prec<P>::C2 qy, typename Prec<P>::C2 dpsi,
    typename Prec<P>::C2 drho, int x, int y, bool per, int pull, const Geom& g,
    const LatVals<typename Prec<P>::C>& v, const Coef<typename Prec<P>::C>& k,
    const SiteOut<typename Prec<P>::T2>& o, typename Prec<P>::C2* nf,
    const typename Prec<P>::C2* jg = nullptr) {
    typedef typename Prec<P>::T2 T2;
    typedef typename Prec<P>::C C;
    typedef typename Prec<P>::C2 C2;
    C2 h[9];
    C2 jx, jy;
    if constexpr (TAU1) {
        jx = jg[0];
        jy = jg[1];
    } else {
        load_site<P, PS>(bm, b0, bp, y, per, pull, g, v, h);
        moments<P>(h, jx, jy);
    }
    const C2 rho = padd(pset(v.rho_ref), drho);
    if (o.valid) note_nonfinite(rho, *nf);   // stays zero unless a density is inf or NaN
    C2 Fx, Fy;
    site_force<GEN>(fxl, fyl, qx, qy, dpsi, rho, y, v, k, Fx, Fy);

    // Eq. (1): forced BGK relaxation.
    const bool source = GEN && k.source;
    C2 zx, zy;
    site_velocity<P, TAU1>(rho, jx, jy, Fx, Fy, source, k, zx, zy);
    C2 hs[9];
    if (source)
        collide<C, C2, true, TAU1>(h, hs, drho, rho, zx, zy, k, Fx, Fy, scale_of<P>());
    else
        collide<C, C2, false, TAU1>(h, hs, drho, rho, zx, zy, k, Fx, Fy, scale_of<P>());
    T2 e[9];
    if constexpr (sizeof(T2) == 4) {
        if (k.sr) {   // half formats: random bits from (site, step), one word per pair
            const uint32_t r = o.rbits;
#pragma unroll
            for (int i = 0; i < 9; ++i) e[i] = enc2_sr<T2>(hs[i], r * sr_mult(i));
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) e[i] = enc2<T2, C>(hs[i].x, hs[i].y);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) e[i] = enc2<T2, C>(hs[i].x, hs[i].y);
    }

    if constexpr (SINK == SINK_STAGE) {
        // The staging tile leaves by a bulk tensor store (clipped at the
        // lattice edge); the periodic ghost copies follow by the plain
        // stores of write_edges after the tile's barrier.
        constexpr int TX = Prec<P>::TX, TY = Prec<P>::TY;
#pragma unroll
        for (int i = 0; i < 9; ++i) o.stage[i * TY * TX] = e[i];
    } else {
        // Straight to the output buffer, and to the periodic images of a
        // site within three sites of an edge (ghost columns, and ghost rows
        // when periodic in y).
        if (o.valid) {
#pragma unroll
            for (int i = 0; i < 9; ++i) st_pair(o.gout + i * o.plane, e[i], o.pol);
        }
        if (o.valid && (o.gdx != 0 || o.gdy != 0)) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                T2* d = o.gout + i * o.plane;
                if (o.gdx) st_pair(d + o.gdx, e[i], o.pol);
                if (o.gdy) {
                    st_pair(d + o.gdy, e[i], o.pol);
                    if (o.gdx) st_pair(d + o.gdy + o.gdx, e[i], o.pol);
                }
            }
        }
    }
    if (!per && (y == 0 || y == g.ny - 1)) {
        const bool down = y == 0;
        C2 sv[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) sv[i] = dec2(e[i]);
        const C2 m = wall_momentum<P>(sv, down, v);
        if (o.valid) reinterpret_cast<C2*>(o.wallx)[(down ? 0 : g.nx) + x] = m;
    }
}

// A float widened to double.  The conversion instruction runs on the FP64
// pipe; a normal value's bits are moved by integer operations instead.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
    return m == 0u ? __hiloint2double((int)b, 0) : (double)x;
}
__device__ __forceinline__ double widen(double x) { return x; }

// The wall columns [2][nx] that a window's step `step` writes: two sets in turn.
template <typename C2>
__device__ __forceinline__ C2* wall_columns(void* wallx, int nx, int step) {
    return reinterpret_cast<C2*>(wallx) + (step & 1) * 2 * nx;
}

// Wall momentum of one CTA's items that hold a wall row, in FP64, at the
// lattices' sampled steps: the wall-site values the site phase left in the
// lattice's wall columns, summed over the item's strip in a fixed order (lane l
// takes columns l, l + 32, ..., then the butterfly), one warp per item, and
// added to the strip's running total -- so the totals do not depend on the
// partition or the tile shape, and no CTA has to wait for the others' sums.
// Sampled steps: stress_t0 + k stress_every; DevStats::next_sample is the
// first one from the window's start on (32-bit remainder: a window is short,
// and a 64-bit one would compile to a call).
// The chain of dependent loads and FP64 additions takes 1.5 us, as much as half a
// small lattice's step.  So a launch sums the previous launch's values (step
// `step` of the window, from the wall columns of that parity) while its own
// first loads are in flight, and only the window's last launch sums its own
// at its end: 300 x 211 FP32 with tau = 0.8 7.39 -> 6.31 us a step, tau = 1 6.45 -> 5.35,
// FP16 6.96 -> 5.80, 128^2 FP16 6.62 -> 5.74.  (The last warps: the first ones have the most to do.)
template <int P, class L>
__device__ __forceinline__ void wall_sums(const BatchArgs<typename Prec<P>::C>& a, int it0, int it_end,
                                       int tid, int step) {
    typedef typename L::C C;
    typedef typename L::C2 C2;
    const int lane = tid & 31, warp = tid >> 5;
    for (int it = it0 + (L::NT / 32 - 1 - warp); it < it_end; it += L::NT / 32) {
        const int4 w = a.items[it];
        const LatDesc<C>* d = &a.lat[w.x];
        const bool bot = w.z == 0, top = w.w == d->ntiles_y;
        if (d->g.periodic || !(bot || top)) continue;
        const long long since = d->st->t + step - d->st->next_sample;
        if (since < 0 || (unsigned)since % (unsigned)d->stress_every != 0u) continue;
        const int nx = d->g.nx;
        const int xe = min(w.y * L::TX + L::TX, nx);
        const C2* wx = wall_columns<C2>(d->wallx, nx, step);
        auto strip = [&](const C2* m, double* total) {
            double sum = 0.0;
            for (int x = w.y * L::TX + lane; x < xe; x += 32) sum += widen(m[x].x) + widen(m[x].y);
            sum = warp_sum(sum);
            if (lane == 0) *total += sum;
        };
        if (bot) strip(wx, d->wsum + w.y);
        if (top) strip(wx + nx, d->wsum + d->nstrips + w.y);
    }
}

// The last CTA of a window's last launch: every lattice's step counter, buffer
// parity, state form (DevStats::pull) and wall-sample schedule, one thread per
// lattice.
template <int NT, typename C>
__device__ __forceinline__ void advance_lattices(const BatchArgs<C>& a, int tid, int pull) {
    for (int l = tid; l < a.nlat; l += NT) {
        const LatDesc<C>* d = &a.lat[l];
        DevStats* st = d->st;
        const long long t = st->t + a.advance, next = st->next_sample;
        if (!d->g.periodic && t > next) {   // samples taken in the window
            const unsigned every = (unsigned)d->stress_every;
            const unsigned m = ((unsigned)(t - next) + every - 1u) / every;
            st->samples += m;
            st->next_sample = next + (long long)m * every;
        }
        st->t = t;
        st->cur ^= a.advance & 1;
        st->pull = pull;
    }
}

// Periodic images of one tile's edge sites, from the staging tile into the
// ghost columns (x within 3 of either edge) and, when the lattice is
// periodic in y, the ghost rows (y within 3 of either edge) and corners, and
// the sites themselves in the last lattice columns the bulk store leaves
// out (x >= x_tail, within 3 of the right edge); by
// all NT threads of the CTA, one (site, plane) copy each in turn, with
// consecutive threads on consecutive sites of a plane.  The first copies go
// to warps 2 and up: warps 0 and 1 have just issued the tile's loads and
// store, and every warp waits for the last one at the next barrier.  Kept
// out of the site update, whose register allocation it would otherwise
// burden.  L: the step kernel's layout (tile rows TY, staging layout).
template <int P, class L>
__device__ __forceinline__ void write_edges(const typename Prec<P>::T2* stage,
                                            typename Prec<P>::T2* fout, const Geom& g, int x0,
                                            int y0, bool per, int tid) {
    typedef typename Prec<P>::T2 T2;
    constexpr int TX = L::TX, TY = L::TY, NT = L::NT;
    const int w = min(TX, g.nx - x0), h = min(TY, g.ny - y0);   // valid part of the tile
    // source columns [0, nca) and [cb0, w), rows [0, na) and [rb0, h); the
    // two ranges of each never meet since nx, ny >= 8
    const int nca = max(0, min(3 - x0, w)), cb0 = max(g.nx - 3 - x0, 0), ncb = max(w - cb0, 0);
    const int na = per ? max(0, min(3 - y0, h)) : 0;
    const int rb0 = max(g.ny - 3 - y0, 0), nb = per ? max(h - rb0, 0) : 0;
    const int nrow = na + nb;                 // ghost-source rows: every column
    const int mid0 = na, mid1 = nb > 0 ? rb0 : h;   // other rows: the edge columns only
    const int ncol = nca + ncb;
    const int nA = nrow * w, nB = max(mid1 - mid0, 0) * ncol, n = nA + nB;
    if (n == 0) return;
    const long long PL = (long long)g.rows * g.pitch;
    const long long SY = (long long)g.ny * g.pitch;
    for (int u = tid >= 64 ? tid - 64 : tid + NT - 64; u < 9 * n; u += NT) {
        const int i = u / n, k = u - i * n;
        int lx, ly;
        if (k < nA) {
            const int r = k / w;
            lx = k - r * w;
            ly = r < na ? r : rb0 + (r - na);
        } else {
            const int kb = k - nA, r = kb / ncol, c = kb - r * ncol;
            ly = mid0 + r;
            lx = c < nca ? c : cb0 + (c - nca);
        }
        const int dX = lx < nca ? g.nx : (ncb > 0 && lx >= cb0 ? -g.nx : 0);
        const long long dY = ly < na ? SY : (nb > 0 && ly >= rb0 ? -SY : 0);
        const T2 e = stage[L::stage_off(ly, lx) + i * L::TYB * TX];
        T2* d = fout + i * PL + (long long)(y0 + ly + kGY) * g.pitch + (x0 + lx + g.gx);
        if (x0 + lx >= g.x_tail) d[0] = e;
        if (dX) d[dX] = e;
        if (dY) {
            d[dY] = e;
            if (dX) d[dY + dX] = e;
        }
    }
}

// FP64 block sums of red[0..3] over all threads; sum k is the result of thread
// 8 k.  The four sums share the butterfly: its first two steps hand half of the
// lanes' values over, so a warp takes 6 FP64 additions instead of 20.
template <int NT>
__device__ __forceinline__ double block_sum4(const double red[4], double (*s_red)[4]) {
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool h16 = lane & 16, h8 = lane & 8;
    double a = (h16 ? red[2] : red[0]) + __shfl_xor_sync(full, h16 ? red[0] : red[2], 16);
    double b = (h16 ? red[3] : red[1]) + __shfl_xor_sync(full, h16 ? red[1] : red[3], 16);
    a = (h8 ? b : a) + __shfl_xor_sync(full, h8 ? a : b, 8);
    a += __shfl_xor_sync(full, a, 4);
    a += __shfl_xor_sync(full, a, 2);
    a += __shfl_xor_sync(full, a, 1);
    __syncthreads();
    if ((lane & 7) == 0) s_red[warp][lane >> 3] = a;
    __syncthreads();
    if (warp == 0) {
        a = 0.0;
        for (int w = lane & 7; w < NT / 32; w += 8) a += s_red[w][lane >> 3];
        a += __shfl_xor_sync(full, a, 4);
        a += __shfl_xor_sync(full, a, 2);
        a += __shfl_xor_sync(full, a, 1);
    }
    return a;
}

// ------------------------------------------------------------ step kernel
// Persistent and multi-lattice.  The work items of a launch are runs of
// tiles (TY = 8 SPT rows each) down TX-wide column strips, over all
// lattices; CTA b takes the items a.items[a.cta_items[b] .. a.cta_items[b + 1])
// of a table the host builds (segments dealt by estimated work in band
// order, or one contiguous run per CTA).  Walking down a strip, a CTA keeps
// the 8-row blocks of f* (TMA-loaded into a ring of NB slots, ahead of use
// and across item boundaries) and a window of the density/Psi deviation rows
// y0 - 2 .. y0 + TY + 1 of the current tile, whose last four rows are
// carried forward as the next tile's first four; so each block is loaded
// and each deviation row computed once per strip, and only the x halo (4 of
// 64 columns) is redundant.  Every thread keeps one column and SPT rows of
// the window (its own sites' cells, see t_m and t_w), so all its
// shared-memory addresses within a slot are fixed.  SPT = 2: each thread
// updates two vertically adjacent
// sites, which share four of their six stencil rows.  Tiles leave through a
// staging tile by TMA bulk tensor stores (one per 8 rows), clipped at the
// lattice edge, and tiles near an edge then write the periodic ghost
// copies; where the staging tile does not fit beside the ring (FP32 with
// 16-row tiles) the threads store their sites and ghost copies to global
// memory themselves.  The last CTA of a window's last launch advances every
// lattice's step counter and buffer parity.
// V: bit 0 = every lattice periodic (no wall code); bit 1 = general forcing;
// bit 2 = omega = 1 for both species (the site phase reads no populations).
template <int P, int V, int SH>
__global__ void __launch_bounds__(Layout<P, SH>::NT, Layout<P, SH>::CTAS)
    k_step(const __grid_constant__ BatchArgs<typename Prec<P>::C> a) {
    typedef Layout<P, SH> L;
    constexpr int SPT = L::SPT, ADV = L::ADV, NBT = L::NBT;
    // FP64: items are runs of rows (y_a, y_b) in place of runs of tiles, cut
    // into tiles of 8 rows from their own first row on, the last one partial.
    // Its time is the number of rows a CTA sums (the FP64 pipe), so a lattice
    // is spread over the SMs row by row (128^2: 80 CTAs of one 8-row tile, 20.5 us
    // a step; 130 CTAs of 5 rows, 16.4.  512^2: 142 -> 128 us.  With the exacter
    // functions and force sums since, 16.9 and 135).
    constexpr bool ROWS = P == LB_FP64;
    typedef typename L::T2 T2;
    typedef typename L::C C;
    typedef typename L::C2 C2;
    constexpr bool ALLPER = (V & 1) != 0;
    constexpr bool GEN = (V & 2) != 0;
    // omega = 1 for both species: the site phase needs the populations only
    // through j, which the density phase computes beside rho and Psi
    constexpr bool TAU1 = (V & 4) != 0;
    constexpr bool STAGED = L::STAGED;   // output through the staging tile
    constexpr int PS = L::TYB * L::BX;   // plane stride in a block slot (pairs)
    extern __shared__ unsigned char smem_raw[];
    // 128-byte aligned base, derived from the shared array by indexing so
    // that every access below compiles to shared-memory instructions.
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    C2* win_r = reinterpret_cast<C2*>(smem + L::WIN_OFF);     // [WIN][RX]
    C2* win_p = win_r + L::WIN * L::RX;                       // [WIN][RX]
    T2* stage = reinterpret_cast<T2*>(smem + L::STAGE_OFF);   // staging tile (STAGED)
    __shared__ __align__(8) uint64_t bars[L::NB];
    __shared__ int s_fail, s_last;
    __shared__ uint64_t s_pol[2];   // L2 policies of the block loads and the tile stores

    const int tid = threadIdx.x;
    const int G = gridDim.x;
    // thread 0 issues the block loads; this thread (warp 1) the bulk stores
    // of the staging tile and the waits on them (STAGED)
    constexpr int kStoreThread = 32;
    // When one buffer of every lattice of the launch fits in L2 together, the
    // step's output stays there for the next step (evict last) and the input,
    // dead once read, goes first; otherwise both keep the normal priority.
    // The two policies are made once, by thread 0, and kept in shared memory
    // (held in registers through the tile loop, or made at each issue, they
    // cost the large lattices 1-3 %).
    // window column and block row of this thread (both phases)
    const int t_lx = tid % L::RX, t_j = tid / L::RX;
    static_assert(L::NT == L::RX * L::TR && L::TY >= 4, "one window column per thread and block row");
    static_assert(P != LB_FP64 || (L::RX == 32 && SPT == 1), "FP64: a warp is a row of a tile");
    // Rows of the density phase: thread row t_j computes the new window rows
    // 4 + SPT t_m + c, c < SPT, which hold its own sites (window rows
    // 2 + SPT t_j + c) for t_j >= 2 / SPT; the first 2 / SPT thread rows,
    // whose sites sit in the two rows carried over from the previous tile,
    // compute the last two rows -- the next tile's first sites, theirs again.
    // So every thread's sites were computed by the thread itself, in this
    // tile or (first thread rows) in the previous one, and their momenta stay
    // with it (TAU1): in registers, and for the first thread rows across the
    // tile boundary in a small shared buffer of their own.
    constexpr int kCarry = 2 / SPT;   // thread rows whose sites are carried rows
    static_assert(2 % SPT == 0, "two carried rows per tile");
    const int t_m = (t_j + L::TR - kCarry) % L::TR;
    const bool t_carry = t_j < kCarry;
    // Columns likewise: window column w holds lattice column x0 - 2 + w and
    // site column lx is window column lx + 2, so thread t_lx computes window
    // column (t_lx + 2) mod RX -- its own site column, and for the RX - TX
    // threads without a site the halo columns.
    const int t_w = (t_lx + 2) % L::RX;
    // TAU1: momenta (jx, jy) of the first thread rows' new cells, kept for
    // the next tile, whose first sites they are; jc: this thread's entries
    // FP64: the exponential table, copied while the previous step drains
    ExpTable* s_tab = reinterpret_cast<ExpTable*>(smem + L::TAB_OFF);
#if LB_PREC == 0
    static_assert(sizeof(ExpTable) % sizeof(double2) == 0, "copied in pairs");
    for (int i = tid; i < (int)(sizeof(ExpTable) / sizeof(double2)); i += L::NT)
        reinterpret_cast<double2*>(s_tab)[i] = reinterpret_cast<const double2*>(&g_exp_tab)[i];
#endif
    __shared__ __align__(16) C2 s_jcarry[kCarry * L::RX * SPT * 2];
    C2* const jc = s_jcarry + ((t_carry ? t_j : 0) * L::RX + t_lx) * (SPT * 2);
    auto slot = [&](int pos) { return reinterpret_cast<T2*>(smem + (pos % L::NB) * L::SLOT_BYTES); };
    const int it_end = a.cta_items[blockIdx.x + 1];

    if (tid == 0) {
        s_fail = 0;
        for (int b = 0; b < L::NB; ++b) mbar_init(&bars[b], 1);
        fence_mbar_init();
        s_pol[0] = a.l2_resident ? policy_evict_first() : policy_evict_normal();
        s_pol[1] = a.l2_resident ? policy_evict_last() : policy_evict_normal();
    }
    __syncthreads();
    // Before the wait only shared memory, the host-built tables and, after a
    // window's first launch, the lattices' counters are read: the previous
    // launch of the window leaves the counters alone, and the launch before it
    // has completed.  Everything else of the lattice state is read after the
    // wait.  The next step's CTAs may then take each SM as soon as this CTA
    // leaves it (one CTA fills an SM).
    const int step_k = a.step_k;
    if (step_k == 0) griddep_wait();

    // Producer (thread 0): the blocks of this CTA's items, in order.  Item
    // tiles [ty_a, ty_b) need blocks SPT ty_a .. SPT ty_b (block j = padded
    // rows [8j, 8j + 8)); consecutive items' blocks follow each other.
    int p_item = a.cta_items[blockIdx.x], p_j = 0, p_pos = 0;
    // cached geometry of the producer's current item
    const CUtensorMap* p_map = nullptr;
    int p_x0 = 0, p_y = 0, p_nblk = 0;
    auto p_load = [&]() {
        if (p_item >= it_end) return;
        const int4 w = a.items[p_item];
        const LatDesc<C>* d = &a.lat[w.x];
        p_x0 = w.y * L::TX;
        p_y = ROWS ? w.z : L::TY * w.z;   // padded row of the first block
        p_nblk = ADV * (ROWS ? (w.w - w.z + L::TY - 1) / L::TY : w.w - w.z) + 1;
        p_map = &d->tin[*((volatile int*)&d->st->cur) ^ (step_k & 1)];
        tma_prefetch_map(p_map);
    };
    auto issue_next = [&]() -> bool {
        if (p_item >= it_end) return false;
        uint64_t* bar = &bars[p_pos % L::NB];
        mbar_expect_tx(bar, (uint32_t)L::SLOT_BYTES);
        // box origin: pair column x0 (= x0 - gx + gx) -> element 2 x0; padded row 8j
        tma_load_3d_hint(slot(p_pos), p_map, 2 * p_x0, p_y + L::TYB * p_j, 0, bar,
                         s_pol[0]);
        ++p_pos;
        if (++p_j == p_nblk) {
            p_j = 0;
            ++p_item;
            p_load();
        }
        return true;
    };
    if (tid == 0) p_load();
    if (step_k != 0) griddep_wait();
    griddep_launch_dependents();
    if (tid == 0)
        while (p_pos < L::NB && issue_next()) {}
    if constexpr (!ALLPER)
        if (step_k != 0) wall_sums<P, L>(a, a.cta_items[blockIdx.x], it_end, tid, step_k - 1);
    int ty_b = 0, ty = 0;   // the consumer's item end and tile (read by release)
    // Producer: the tile whose first block is at position q is done with
    // its blocks before the next tile's first one (all of them at an item's
    // last tile): refill those slots.
    auto release = [&](int q) {
        const int released = (ty + 1 < ty_b) ? q + ADV : q + NBT;
        fence_proxy_async();   // generic reads of freed slots before async writes
        while (p_pos < released + L::NB && issue_next()) {}
    };

    int c_pos = 0;   // ring position of the current item's first block
    for (int it = a.cta_items[blockIdx.x]; it < it_end && !s_fail; ++it) {
        const int4 w = a.items[it];
        const LatDesc<C>* d = &a.lat[w.x];
        const int x0 = w.y * L::TX;
        const int ty_a = ROWS ? 0 : w.z;
        ty_b = ROWS ? (w.w - w.z + L::TY - 1) / L::TY : w.w;
        const int y_first = ROWS ? w.z : 0;   // lattice row of tile 0
        const Geom g = d->g;
        const LatVals<C> v = d->v;
        const bool per_lat = ALLPER || g.periodic;
        // the counters advance only after every CTA of a window's last launch is done
        const int cur = *((volatile int*)&d->st->cur) ^ (step_k & 1);
        const int pull = step_k != 0 ? 1 : *((volatile int*)&d->st->pull);
        const uint32_t key =
            hash32(((uint32_t)*((volatile long long*)&d->st->t) + (uint32_t)step_k) * 0x9e3779b9u);
        T2* fout = reinterpret_cast<T2*>(d->fbuf[cur ^ 1]);
        C2 nf = pset(C(0));   // 0 * rho over the item's sites: NaN at a non-finite density
        // ring slot and phase parity of the tile's first block, kept as the
        // tiles advance
        int qm = c_pos % L::NB, qph = (c_pos / L::NB) & 1;
        for (ty = ty_a; ty < ty_b; ++ty) {
            const int q = c_pos + ADV * (ty - ty_a);   // this tile uses blocks q .. q + ADV
            // Each thread sees the blocks land itself (the first block of a
            // tile after an item's first was seen as the previous tile's
            // last); a timeout is acted on after the next barrier (garbage
            // read meanwhile is harmless).
            int sl[NBT];
#pragma unroll
            for (int b = 0; b < NBT; ++b) {
                int sb = qm + b, ph = qph;
                if (sb >= L::NB) {
                    sb -= L::NB;
                    ph ^= 1;
                }
                sl[b] = sb;
                if ((b > 0 || ty == ty_a) && !mbar_wait_bounded(&bars[sb], ph)) s_fail = 1;
            }
            const int y0 = y_first + ty * L::TY;
            const int y_end = ROWS ? w.w : g.ny;   // end of the rows this item updates
            // The tile's padded rows [y0, y0 + 8 (SPT + 1)) are blocks q ..
            // q + SPT; brow(r, c): padded row y0 + r, pair column c, plane 0.
            const T2* s0 = reinterpret_cast<const T2*>(smem + sl[0] * L::SLOT_BYTES);
            const T2* s1 = reinterpret_cast<const T2*>(smem + sl[1] * L::SLOT_BYTES);
            const T2* s2 = reinterpret_cast<const T2*>(smem + sl[ADV] * L::SLOT_BYTES);
            auto brow = [&](int r, int c) {
                const T2* base = r < L::TYB ? s0 : (ADV == 1 || r < 2 * L::TYB ? s1 : s2);
                return base + (r & (L::TYB - 1)) * L::BX + c;
            };

            // The tile's two phases, with or without the wall code: a tile
            // whose deviation window (rows y0 - 2 .. y0 + TY + 1) keeps clear
            // of the walls and of the periodic ghost rows runs the periodic
            // code, which is exact there, so only the tiles at a wall pay for
            // the wall logic.  Returns false when a block wait gave up.
            auto tile_body = [&](auto wall_tag) -> bool {
                constexpr bool W = decltype(wall_tag)::value;
                const bool per = !W || per_lat;
                C2 jn[SPT][2];   // TAU1: momenta of this thread's new rows
                // Phase 2: window row k holds lattice row y0 - 2 + k (padded row
                // y0 + 1 + k).  Rows 4 .. TY + 3 are new: thread (t_lx, t_j)
                // computes rows 4 + SPT t_m + c, c < SPT, of window column t_w
                // (the thread's own sites, see t_m).  Rows 0 .. 3 are the previous
                // tile's rows TY .. TY + 3, carried forward by the threads that
                // own those before they overwrite them, or at an item's first
                // tile computed from block q.  No other thread touches these
                // cells in this phase.
                {
                    const int bc = t_w - 2 + L::GX;   // pair column in the block
                    // rows 0 .. 3: carried forward, or computed at an item's first
                    // tile, before this thread's new rows overwrite their sources
                    // (rows 2 and 3, at an item's first tile, by the thread rows
                    // whose sites they are: their momenta start the carry)
    #pragma unroll
                    for (int c = 0; c < SPT; ++c) {
                        const int k = 4 + SPT * t_m + c;
                        const int kk = k - L::TY;
                        if (kk >= 0) {
                            if (ty == ty_a) {
                                C2 r, p, jt[2];
                                cell_dev<P, PS, TAU1>(brow(kk, bc), brow(kk + 1, bc), brow(kk + 2, bc),
                                                      y0 - 2 + kk, per, pull, g, v, r, p, s_tab, jt);
                                win_r[kk * L::RX + t_w] = r;
                                win_p[kk * L::RX + t_w] = p;
                                if (TAU1 && t_carry) {   // rows 2 and 3: this thread's sites
                                    jc[2 * c] = jt[0];
                                    jc[2 * c + 1] = jt[1];
                                }
                            } else {
                                win_r[kk * L::RX + t_w] = win_r[k * L::RX + t_w];
                                win_p[kk * L::RX + t_w] = win_p[k * L::RX + t_w];
                            }
                        }
                    }
                    // The new rows, without a branch between the cells.  Rows
                    // outside the lattice (beyond a wall, or below a ragged last
                    // tile) are computed from whatever the slots hold there (the
                    // TMA fill or ghost rows): no site reads them -- the wall
                    // mirror below overwrites the two rows past each wall.
    #pragma unroll
                    for (int c = 0; c < SPT; ++c) {
                        const int k = 4 + SPT * t_m + c;
                        if (ROWS && k >= y_end - y0 + 4) break;   // (a warp is a row)
                        C2 r, p;
                        cell_dev<P, PS, TAU1>(brow(k, bc), brow(k + 1, bc), brow(k + 2, bc), y0 - 2 + k,
                                              per, pull, g, v, r, p, s_tab, jn[c]);
                        win_r[k * L::RX + t_w] = r;
                        win_p[k * L::RX + t_w] = p;
                    }
                    // The first thread rows (whole warps) swap their new cells'
                    // momenta, the next tile's, for their sites', kept from the
                    // previous tile; jn then holds every thread's sites'.
                    if (TAU1 && t_carry) {
    #pragma unroll
                        for (int c = 0; c < SPT; ++c) {
                            const C2 px = jc[2 * c], py = jc[2 * c + 1];
                            jc[2 * c] = jn[c][0];
                            jc[2 * c + 1] = jn[c][1];
                            jn[c][0] = px;
                            jn[c][1] = py;
                        }
                    }
                }
                // mirror the deviations about the halfway walls, in the tiles whose
                // window rows y0 - 2 .. y0 + TY + 1 reach past a wall (uniform)
                if (!per && (y0 < 2 || y0 + L::TY + 1 >= g.ny)) {
                    __syncthreads();
                    for (int c = tid; c < L::WIN * L::RX; c += L::NT) {
                        const int k = c / L::RX, lx = c - k * L::RX;
                        const int y = y0 - 2 + k;
                        int ym;
                        if (y < 0) ym = -1 - y;
                        else if (y >= g.ny && y <= g.ny + 1) ym = 2 * g.ny - 1 - y;
                        else continue;
                        const int km = ym - (y0 - 2);   // in [0, WIN): see the wall cases
                        win_r[k * L::RX + lx] = win_r[km * L::RX + lx];
                        win_p[k * L::RX + lx] = win_p[km * L::RX + lx];
                    }
                }
                if (STAGED && tid == kStoreThread) bulk_wait_read();   // previous bulk store has read the staging tile
                __syncthreads();
                if (s_fail) return false;
                if constexpr (TAU1) {
                    // The site phase reads no populations: the tile's blocks
                    // before the next tile's first one are free already.
                    if (a.early_release && tid == 0) release(q);
                }

                // Phase 3: SPT sites per thread (lx < TX): sites (x0 + t_lx,
                // y0 + SPT t_j + s), whose stencil rows y - 2 .. y + 2 are window
                // rows SPT t_j + s .. SPT t_j + s + 4 and whose populations sit in
                // padded rows y0 + SPT t_j + s + 2 .. + 4.
                {
                    const int lx = t_lx, ly = SPT * t_j;
                    const int x = x0 + lx, y = y0 + ly;
                    C2 fx[SPT], fy[SPT], qx[SPT], qy[SPT], dp[SPT], dr[SPT];
                    if constexpr (P == LB_FP64) {   // a warp is a row (RX = 32)
                        if (y < y_end)
                            force_sums_warp<L::RX>(win_p + ly * L::RX + lx, win_r + ly * L::RX + lx, a.k,
                                                   fx[0], fy[0], qx[0], qy[0], dp[0], dr[0]);
                    }
                    if (lx < L::TX && x < g.nx && y < y_end) {
                        if constexpr (P != LB_FP64)
                            force_sums<SPT, L::RX>(win_p + ly * L::RX + lx + 2,
                                                   win_r + ly * L::RX + lx + 2, a.k, fx, fy, qx, qy, dp, dr);
                        SiteOut<T2> o;
                        o.rbits = 0u;
                        [[maybe_unused]] uint32_t srh = 0u;   // the shared hash of this thread's sites
                        if constexpr (sizeof(T2) == 4) srh = sr_hash(key, x, y, g.nx);
                        o.valid = 1;
                        o.wallx = wall_columns<C2>(d->wallx, g.nx, step_k);
                        if constexpr (!STAGED) {
                            o.plane = g.plane;
                            o.gdx = x < 3 ? g.nx : (x >= g.nx - 3 ? -g.nx : 0);
                            o.pol = s_pol[1];
                        }
                        // Both sites are updated without a branch between them (a
                        // site below the lattice's last row, in a ragged tile, is
                        // computed and dropped), so their work can interleave.
    #pragma unroll
                        for (int s = 0; s < SPT; ++s) {
                            const int ys = y + s;
                            o.valid = s == 0 || ys < g.ny;
                            if constexpr (sizeof(T2) == 4) {
                                // SPT = 2: y is even (tile rows are multiples of 16)
                                o.rbits = sr_word(SPT == 2 ? srh : sr_hash(key, x, ys, g.nx), ys);
                            }
                            if constexpr (STAGED) {
                                o.stage = stage + L::stage_off(ly + s, lx);
                            } else {
                                o.gout = fout + (long long)(ys + kGY) * g.pitch + (x + g.gx);
                                o.gdy = !per ? 0
                                        : ys < 3 ? (long long)g.ny * g.pitch
                                        : (ys >= g.ny - 3 ? -(long long)g.ny * g.pitch : 0);
                            }
                            if constexpr (TAU1) {
                                site_update<P, GEN, PS, STAGED ? SINK_STAGE : SINK_GLOBAL, true>(
                                    nullptr, nullptr, nullptr, fx[s], fy[s], qx[s], qy[s], dp[s], dr[s],
                                    x, ys, per, pull, g, v, a.k, o, &nf, jn[s]);
                            } else {
                                const int bc = lx + L::GX;
                                site_update<P, GEN, PS, STAGED ? SINK_STAGE : SINK_GLOBAL>(
                                    brow(ly + s + 2, bc), brow(ly + s + 3, bc), brow(ly + s + 4, bc),
                                    fx[s], fy[s], qx[s], qy[s], dp[s], dr[s], x, ys, per, pull, g, v,
                                    a.k, o, &nf);
                            }
                        }
                        if constexpr (STAGED) fence_proxy_async();   // staging writes before the bulk store
                    }
                }
                return true;
            };
            bool ok;
            if constexpr (ALLPER)
                ok = tile_body(std::false_type{});
            else if (per_lat || (y0 >= 3 && y0 + L::TY + 3 <= g.ny))
                ok = tile_body(std::false_type{});
            else
                ok = tile_body(std::true_type{});
            if (!ok) break;
            __syncthreads();
            if constexpr (STAGED) {
                // The bulk stores and the next loads are issued by two threads
                // of different warps, side by side.
                if (tid == kStoreThread) {
                    // site (x0, y0 + 8h) in padded coordinates: pair column
                    // x0 + gx, row y0 + 8h + kGY; a ragged tile's store is
                    // clipped at x = nx, y = ny (no box starts below the lattice)
#pragma unroll
                    for (int h = 0; h < ADV; ++h)
                        if (h == 0 || y0 + h * L::TYB < g.ny)
                            tma_store_3d_hint(&d->tout[cur ^ 1], stage + L::stage_off(h * L::TYB, 0),
                                              2 * (x0 + L::GX), y0 + h * L::TYB + kGY, 0, s_pol[1]);
                    bulk_commit();
                }
            }
            if (!(TAU1 && a.early_release) && tid == 0) release(q);
            if constexpr (STAGED) {
                // only tiles within 3 sites of an edge write periodic ghost copies
                const bool edge = x0 < 3 || x0 + L::TX > g.nx - 3 ||
                                  (per_lat && (y0 < 3 || y0 + L::TY > g.ny - 3));
                if (edge) write_edges<P, L>(stage, fout, g, x0, y0, per_lat, tid);
            }
            qm += ADV;
            if (qm >= L::NB) {
                qm -= L::NB;
                qph ^= 1;
            }
        }
        if (!(nf.x == C(0) && nf.y == C(0)))   // a density of this lattice went non-finite
            atomicOr(&d->st->err, ERR_NONFINITE);
        if (s_fail) break;
        c_pos += ADV * (ty_b - ty_a) + 1;
    }
    // The wall momentum of a window's last step (see wall_sums).  Kept out of
    // the tile loop: a per-item reduction there (barriers, FP64 shuffles) cost
    // the generic variant 1-4 % even on periodic lattices, which skip it.
    if constexpr (!ALLPER)
        if (a.advance) {
            __syncthreads();   // this CTA's wall-site values are written
            if (!s_fail) wall_sums<P, L>(a, a.cta_items[blockIdx.x], it_end, tid, step_k);
        }
    if (STAGED && tid == kStoreThread) bulk_wait_all();
    if (s_fail && tid == 0) {
        // Let copies in flight land before the CTA exits.  No slot is
        // re-armed once a wait has failed, so the last NB positions issued
        // are each slot's latest arm, and every earlier one has landed; wait
        // on each of those once, with its own phase parity (a position that
        // has landed returns at once).
        for (int pos = p_pos > L::NB ? p_pos - L::NB : 0; pos < p_pos; ++pos)
            mbar_wait_bounded(&bars[pos % L::NB], (pos / L::NB) & 1);
    }
    if (s_fail && tid == 0)   // report on every lattice of the launch
        for (int l = 0; l < a.nlat; ++l) atomicOr(&a.lat[l].st->err, ERR_TIMEOUT);

    // A window's last launch advances the lattices, by its last CTA; the other
    // launches need no arrival counter.  That and the set-up ahead of the wait
    // took a step of one 128^2 FP32 lattice from 8.2 to 6.1 us (its counter's
    // round trip, the last CTA's work and four dependent loads before the first
    // block load), 300 x 211 Couette from 11.8 to 9.0, the 5 x 512^2 sweep from
    // 35.0 to 33.3.
    if (!a.advance) return;
    __syncthreads();   // this CTA's writes (wall sums, timeout flags) precede its arrival
    if (tid == 0) s_last = ticket_arrive(a.ticket) == (unsigned int)(G - 1);
    __syncthreads();
    if (!s_last) return;
    advance_lattices<L::NT>(a, tid, 1);
    // no other CTA of the launch touches the ticket again; the next launch
    // reads it after this one has completed
    if (tid == 0) *a.ticket = 0u;
}

// ------------------------------------- direct kernel (few tiles, not FP64)
// The step for lattices whose tiles do not fill the SMs: a step then is one
// chain of latencies, and k_step's ring, descriptors, staging tile and bulk
// stores only lengthen it.  A CTA loads a tile's populations by plain loads (all
// of a thread's at once) into shared memory, takes the tile's whole deviation
// window (no rows are carried), updates one site per thread and stores it from
// registers.  One CTA per SM; the site arithmetic is k_step's.  Measured, k_step
// -> this: 300 x 211 FP32 Couette with tau 0.8 (135 tiles) 8.3 -> 7.4 us a step,
// 128^2 FP16 5.25 -> 4.67, 64^2 FP16 5.18 -> 4.61.
#if LB_PART == 4
template <int P, int V>
__global__ void __launch_bounds__(DLayout<P>::NT, 1)
    k_step_d(const __grid_constant__ BatchArgs<float> a) {
    typedef DLayout<P> L;
    typedef typename L::T2 T2;
    constexpr bool ALLPER = (V & 1) != 0;
    constexpr bool GEN = (V & 2) != 0;
    constexpr bool TAU1 = (V & 4) != 0;
    constexpr int TY = L::TY, TX = L::TX, RX = L::RX, NR = L::NR, BX = L::BX, PS = L::PS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    T2* const box = reinterpret_cast<T2*>(smem);                     // [9][NR][BX]
    float2* const win_r = reinterpret_cast<float2*>(smem + L::WIN_OFF);   // [WIN][RX]
    float2* const win_p = win_r + L::WIN * RX;                            // [WIN][RX]
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const int t_lx = tid % RX, t_j = tid / RX;
    const int t_w = (t_lx + 2) % RX;   // window column, the site's own for t_lx < TX
    const int it0 = a.cta_items[blockIdx.x], it_end = a.cta_items[blockIdx.x + 1];
    const int step_k = a.step_k;
    // tables and counters are read ahead of the wait, as in k_step
    int4 w = make_int4(0, 0, 0, 0);
    const LatDesc<float>* d = nullptr;
    Geom g = {};
    LatVals<float> v = {};
    int cur = 0, pull = 1;
    uint32_t key = 0;
    auto load_item = [&](int it) {
        w = a.items[it];
        d = &a.lat[w.x];
        g = d->g;
        v = d->v;
    };
    auto load_state = [&]() {
        cur = *((volatile int*)&d->st->cur) ^ (step_k & 1);
        if (step_k == 0) pull = *((volatile int*)&d->st->pull);
        key = hash32(((uint32_t)*((volatile long long*)&d->st->t) + (uint32_t)step_k) * 0x9e3779b9u);
    };
    if (it0 < it_end) {
        load_item(it0);
        if (step_k != 0) load_state();
    }
    griddep_wait();
    griddep_launch_dependents();
    if (it0 < it_end && step_k == 0) load_state();
    const uint64_t pol = a.l2_resident ? policy_evict_last() : policy_evict_normal();
    for (int it = it0; it < it_end; ++it) {
        if (it != it0) {
            load_item(it);
            load_state();
        }
        const int x0 = w.y * TX;
        const bool per_lat = ALLPER || g.periodic;
        const T2* const fin = reinterpret_cast<const T2*>(d->fbuf[cur]);
        T2* const fout = reinterpret_cast<T2*>(d->fbuf[cur ^ 1]);
        float2 nf = pset(0.0f);
        for (int ty = w.z; ty < w.w; ++ty) {
            const int y0 = ty * TY;
            // box row r: lattice row y0 - 3 + r (the padded planes hold rows up to
            // ny + 2 and columns up to nx + 2; beyond them no site reads)
            auto cell = [&](int r, int c, T2 h[9]) {
                const int y = min(y0 - 3 + r, g.ny + 2), x = min(x0 - 3 + c, g.nx + 2);
                const T2* f = fin + (long long)(y + kGY) * g.pitch + (x + g.gx);
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = __ldcg(f + i * g.plane);
            };
            auto put = [&](int r, int c, const T2 h[9]) {
#pragma unroll
                for (int i = 0; i < 9; ++i) box[i * PS + r * BX + c] = h[i];
            };
            {
                T2 h0[9], h1[9], he[9];
                cell(t_j, t_w + 1, h0);
                if (t_j + 8 < NR) cell(t_j + 8, t_w + 1, h1);
                const int r = tid >> 1, c = tid & 1 ? BX - 1 : 0;   // outermost columns
                if (tid < 2 * NR) cell(r, c, he);
                if constexpr (!ALLPER)   // (the loads are on their way)
                    if (step_k != 0 && it == it0 && ty == w.z) wall_sums<P, L>(a, it0, it_end, tid, step_k - 1);
                put(t_j, t_w + 1, h0);
                if (t_j + 8 < NR) put(t_j + 8, t_w + 1, h1);
                if (tid < 2 * NR) put(r, c, he);
            }
            __syncthreads();
            auto tile_body = [&](auto wall_tag) {
                constexpr bool W = decltype(wall_tag)::value;
                const bool per = !W || per_lat;
                // Density phase: window row k holds lattice row y0 - 2 + k, box row
                // k + 1; the thread's own site row k = t_j + 2, and the rows 0, 1,
                // 10, 11 by the first four thread rows.
                float2 jn[2];
                const T2* bc = box + t_w + 1;
                auto window = [&](int k, float2* j) {
                    float2 r, q;
                    cell_dev<P, PS, TAU1>(bc + k * BX, bc + (k + 1) * BX, bc + (k + 2) * BX, y0 - 2 + k, per,
                                          pull, g, v, r, q, nullptr, j);
                    win_r[k * RX + t_w] = r;
                    win_p[k * RX + t_w] = q;
                };
                window(t_j + 2, jn);
                if (t_j < 4) {
                    float2 unused[2];
                    window(t_j < 2 ? t_j : t_j + 8, unused);
                }
                if (!per && (y0 < 2 || y0 + TY + 1 >= g.ny)) {   // mirror about the halfway walls
                    __syncthreads();
                    for (int c = tid; c < L::WIN * RX; c += L::NT) {
                        const int k = c / RX, lx = c - k * RX;
                        const int y = y0 - 2 + k;
                        int ym;
                        if (y < 0) ym = -1 - y;
                        else if (y >= g.ny && y <= g.ny + 1) ym = 2 * g.ny - 1 - y;
                        else continue;
                        const int km = ym - (y0 - 2);
                        win_r[k * RX + lx] = win_r[km * RX + lx];
                        win_p[k * RX + lx] = win_p[km * RX + lx];
                    }
                }
                __syncthreads();
                const int x = x0 + t_lx, y = y0 + t_j;
                if (t_lx < TX && x < g.nx && y < g.ny) {
                    float2 fx[1], fy[1], qx[1], qy[1], dp[1], dr[1];
                    force_sums<1, RX>(win_p + t_j * RX + t_lx + 2, win_r + t_j * RX + t_lx + 2, a.k, fx, fy, qx,
                                      qy, dp, dr);
                    SiteOut<T2> o;
                    o.valid = 1;
                    o.wallx = wall_columns<float2>(d->wallx, g.nx, step_k);
                    o.plane = g.plane;
                    o.pol = pol;
                    o.gout = fout + (long long)(y + kGY) * g.pitch + (x + g.gx);
                    o.gdx = x < 3 ? g.nx : (x >= g.nx - 3 ? -g.nx : 0);
                    o.gdy = !per_lat ? 0
                            : y < 3 ? (long long)g.ny * g.pitch
                            : (y >= g.ny - 3 ? -(long long)g.ny * g.pitch : 0);
                    o.rbits = 0u;
                    if constexpr (sizeof(T2) == 4) o.rbits = sr_word(sr_hash(key, x, y, g.nx), y);
                    const T2* b0 = bc + (t_j + 3) * BX;   // (t_w is the site's column here)
                    site_update<P, GEN, PS, SINK_GLOBAL, TAU1>(b0 - BX, b0, b0 + BX, fx[0], fy[0], qx[0], qy[0],
                                                               dp[0], dr[0], x, y, per, pull, g, v, a.k, o, &nf,
                                                               jn);
                }
            };
            if constexpr (ALLPER)
                tile_body(std::false_type{});
            else if (per_lat || (y0 >= 3 && y0 + TY + 3 <= g.ny))
                tile_body(std::false_type{});
            else
                tile_body(std::true_type{});
            __syncthreads();   // the box and the windows have been read
        }
        if (!(nf.x == 0.0f && nf.y == 0.0f)) atomicOr(&d->st->err, ERR_NONFINITE);
    }
    if (!a.advance) return;
    if constexpr (!ALLPER) wall_sums<P, L>(a, it0, it_end, tid, step_k);   // (behind the tiles' last barrier)
    __syncthreads();
    if (tid == 0) s_last = ticket_arrive(a.ticket) == (unsigned int)(gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    advance_lattices<L::NT>(a, tid, 1);
    if (tid == 0) *a.ticket = 0u;
}
#endif

// ------------------------------------------------- moment kernel (FP32)
// The step of FP32 lattices with tau = 1 for both species and the velocity
// shift.  There the post-collision populations are the equilibrium of six
// numbers per site -- (drho, z_x, z_y) per species, see collide -- so a step
// stores those instead of 18 populations: 24 bytes a site written and read
// instead of 72, and the next step evaluates the populations where it needs
// them, by the same operations on the same values (the results are the same
// to the bit; the first step reads the initial populations themselves).
// Bound: the population form ran at 90 % of the DRAM copy rate on 4096^2; this
// one moves 57 bytes a site through DRAM there and is bound by instruction
// issue (44 % busy, two barriers a tile) and the shared-memory pipe (62 %), as
// the 16-bit kernels are.  Measured, populations -> moments: 4096^2 391 -> 304
// us a step, 2048^2 107 -> 83, 1024^2 26.1 -> 22.1, 5 x 512^2 33.3 -> 27.3 (both
// buffers of all five lattices now fit in L2), 128^2 5.0 -> 3.9, 512^2 Couette
// 12.5 -> 10.1.
//
// The moments of a lattice are three unpadded planes [ny][nx] of (A, B) pairs;
// loads wrap around the lattice, so no ghost copies are written.  Per tile:
//  1. expand: the tile's 8 new rows of moments (loaded into registers during
//     the previous tile) become populations in the ring, columns x0 - 3 ..
//     x0 + 62 (thread column t_lx takes window column t_w; 16 threads of the
//     first warp the two outermost columns),
//  2. density phase and 3. site phase as in k_step, the ring in place of the
//     block slots; the site's moments go straight to global memory.
// Two barriers per tile: after the expansion, and before the site phase.  The
// site phase reads no populations, so the next tile's expansion follows it
// without one.
#if LB_PART == 5
template <int V, int SH>
__global__ void __launch_bounds__(MLayout<SH>::NT, MLayout<SH>::CTAS)
    k_step_m(const __grid_constant__ BatchArgs<float> a) {
    typedef MLayout<SH> L;
    constexpr int P = LB_FP32;
    constexpr bool ALLPER = (V & 1) != 0;
    constexpr bool GEN = (V & 2) != 0;
    constexpr int SPT = L::SPT, TY = L::TY, TX = L::TX, RX = L::RX, NR = L::NR, BX = L::BX, PS = L::PS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float2* ring = reinterpret_cast<float2*>(smem);                  // [9][NR][BX]
    float2* const win_r0 = reinterpret_cast<float2*>(smem + L::WIN_OFF);   // [WROWS][RX]
    float2* const win_p0 = win_r0 + L::WROWS * RX;                         // [WROWS][RX]
    constexpr int kCarry = 2 / SPT;
    __shared__ __align__(16) float2 s_jcarry[kCarry * RX * SPT * 2];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const int t_lx = tid % RX, t_j = tid / RX;
    // window rows and column of this thread, as in k_step
    const int t_m = (t_j + L::TR - kCarry) % L::TR;
    const bool t_carry = t_j < kCarry;
    const int t_w = (t_lx + 2) % RX;
    float2* const jc = s_jcarry + ((t_carry ? t_j : 0) * RX + t_lx) * (SPT * 2);
    const int it0 = a.cta_items[blockIdx.x], it_end = a.cta_items[blockIdx.x + 1];
    const int step_k = a.step_k;
    // The first item's tables are read ahead of the wait (as in k_step).
    int4 w = make_int4(0, 0, 0, 0);
    const LatDesc<float>* d = nullptr;
    Geom g = {};
    LatVals<float> v = {};
    auto load_item = [&](int it) {
        w = a.items[it];
        d = &a.lat[w.x];
        g = d->g;
        v = d->v;
    };
    int cur = 0, form = 2;
    auto load_state = [&]() {
        cur = *((volatile int*)&d->st->cur) ^ (step_k & 1);
        if (step_k == 0) form = *((volatile int*)&d->st->pull);
    };
    if (it0 < it_end) {
        load_item(it0);
        if (step_k != 0) load_state();
    }
    griddep_wait();
    griddep_launch_dependents();
    if (it0 < it_end && step_k == 0) load_state();
    const uint64_t pol = a.l2_resident ? policy_evict_last() : policy_evict_normal();

    for (int it = it0; it < it_end; ++it) {
        if (it != it0) {
            load_item(it);
            load_state();
        }
        const int x0 = w.y * TX, nx = g.nx, ny = g.ny;
        const bool per_lat = ALLPER || g.periodic;
        const bool mom = form == 2;
        const int pull = form != 0;
        const size_t N = (size_t)nx * ny;
        const float2* const m_in = reinterpret_cast<const float2*>(d->fbuf[cur]);
        float2* const m_out = reinterpret_cast<float2*>(d->fbuf[cur ^ 1]);
        float2 nf = pset(0.0f);
        // The lattice column of ring column c (0 .. BX - 1), wrapped around the
        // lattice, and the row of y, wrapped (periodic) or clamped to the
        // lattice (walls: no site reads what lies beyond).
        auto column = [&](int c) {
            const int x = (x0 - 3 + c) % nx;
            return x < 0 ? x + nx : x;
        };
        auto row = [&](int y) {
            if (!per_lat) return min(max(y, 0), ny - 1);
            y = y < 0 ? y + ny : y;
            y = y >= ny ? y - ny : y;
            return y >= ny ? y - ny : y;   // (ny = 8, 9 below a ragged tile)
        };
        const int xw = column(t_w + 1);
        const int xe = column(tid & 1 ? BX - 1 : 0);   // outermost columns
        struct Mom {
            float2 r, zx, zy;
        };
        auto load_mom = [&](int y, int x) {
            const size_t o = (size_t)row(y) * nx + x;
            Mom m;
            m.r = __ldcg(m_in + o);
            m.zx = __ldcg(m_in + N + o);
            m.zy = __ldcg(m_in + 2 * N + o);
            return m;
        };
        // Populations of a cell into ring slot row s, ring column c; edge: one of
        // the two outermost columns, of which only the three directions that
        // point into the window are pulled.
        auto put = [&](const float2 h[9], int s, int c, bool edge) {
            float2* o = ring + s * BX + c;
            if (edge) {
                o[(c ? 3 : 1) * PS] = c ? h[3] : h[1];
                o[(c ? 6 : 5) * PS] = c ? h[6] : h[5];
                o[(c ? 7 : 8) * PS] = c ? h[7] : h[8];
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) o[i * PS] = h[i];
            }
        };
        auto put_mom = [&](const Mom& m, int s, int c, bool edge) {
            float2 h[9];
            collide<float, float2, false, true>(nullptr, h, m.r, padd(pset(v.rho_ref), m.r), m.zx, m.zy, a.k,
                                                m.r, m.r, 1.0f);
            put(h, s, c, edge);
        };
        // the same from the population planes (the state before the first step)
        auto put_pops = [&](int y, int x, int s, int c) {
            const float2* f = m_in + (size_t)(row(y) + kGY) * g.pitch + (x + g.gx);
            float2 h[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = __ldcg(f + i * g.plane);
            put(h, s, c, false);
        };
        const int ty_a = w.z, ty_b = w.w;
        const int ya = ty_a * TY;
        // The item's first NR rows, y = ya - 3 .. ya + 10; all loads are issued
        // before the first row is expanded (an item's start waits for one memory
        // latency instead of two to four: 128^2 3.9 -> 3.6 us a step, 5 x 512^2
        // 27.3 -> 26.0).
        if (mom) {
            constexpr int R = (NR + L::TR - 1) / L::TR;
            Mom hd[R], he;
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (t_j + q * L::TR < NR) hd[q] = load_mom(ya - 3 + t_j + q * L::TR, xw);
            if (tid < 2 * NR) he = load_mom(ya - 3 + (tid >> 1), xe);
            if constexpr (!ALLPER)   // (the loads are on their way)
                if (step_k != 0 && it == it0) wall_sums<P, L>(a, it0, it_end, tid, step_k - 1);
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (t_j + q * L::TR < NR) put_mom(hd[q], t_j + q * L::TR, t_w + 1, false);
            if (tid < 2 * NR) put_mom(he, tid >> 1, tid & 1 ? BX - 1 : 0, true);
        } else {
            for (int r = t_j; r < NR; r += L::TR) put_pops(ya - 3 + r, xw, r, t_w + 1);
            if (tid < 2 * NR) put_pops(ya - 3 + (tid >> 1), xe, tid >> 1, tid & 1 ? BX - 1 : 0);
        }
        Mom pf[SPT], pfe;   // the next tile's new rows (and outermost columns)
        int base = 0;       // ring slot of row y0 - 3
        int wm = 0;         // the tile's window starts at row wm TY
        auto slot_of = [&](int r) { return base + r >= NR ? base + r - NR : base + r; };
        for (int ty = ty_a; ty < ty_b; ++ty) {
            const int y0 = ty * TY;
            if (ty > ty_a) {   // expand rows y0 + 3 .. y0 + 10
#pragma unroll
                for (int c = 0; c < SPT; ++c) {
                    const int m = SPT * t_j + c;
                    if (mom) put_mom(pf[c], slot_of(6 + m), t_w + 1, false);
                    else put_pops(y0 + 3 + m, xw, slot_of(6 + m), t_w + 1);
                }
                if (tid < 2 * TY) {
                    const int m = tid >> 1, c = tid & 1 ? BX - 1 : 0;
                    if (mom) put_mom(pfe, slot_of(6 + m), c, true);
                    else put_pops(y0 + 3 + m, xe, slot_of(6 + m), c);
                }
            }
            if (mom && ty + 1 < ty_b) {
#pragma unroll
                for (int c = 0; c < SPT; ++c) pf[c] = load_mom(y0 + TY + 3 + SPT * t_j + c, xw);
                if (tid < 2 * TY) pfe = load_mom(y0 + TY + 3 + (tid >> 1), xe);
            }
            float2* const win_r = win_r0 + wm * (TY * RX);
            float2* const win_p = win_p0 + wm * (TY * RX);
            __syncthreads();   // the ring's rows are there; the previous site phase is over
            auto tile_body = [&](auto wall_tag) {
                constexpr bool W = decltype(wall_tag)::value;
                const bool per = !W || per_lat;
                float2 jn[SPT][2];
                // Density phase: window rows as in k_step; row k pulls from the
                // ring rows k, k + 1, k + 2 above y0 - 3.
                {
                    const float2* rc = ring + t_w + 1;
                    auto cell = [&](int k, float2& r, float2& q, float2* j) {
                        cell_dev<P, PS, true>(rc + slot_of(k) * BX, rc + slot_of(k + 1) * BX,
                                              rc + slot_of(k + 2) * BX, y0 - 2 + k, per, pull, g, v, r, q,
                                              nullptr, j);
                    };
#pragma unroll
                    for (int c = 0; c < SPT; ++c) {
                        const int k = 4 + SPT * t_m + c;
                        const int kk = k - TY;
                        if (kk >= 0) {
                            if (ty == ty_a) {
                                float2 r, q, jt[2];
                                cell(kk, r, q, jt);
                                win_r[kk * RX + t_w] = r;
                                win_p[kk * RX + t_w] = q;
                                if (t_carry) {
                                    jc[2 * c] = jt[0];
                                    jc[2 * c + 1] = jt[1];
                                }
                            } else if (wm == 0) {   // from the previous tile's window
                                constexpr int back = (L::WM - 1) * TY;
                                win_r[kk * RX + t_w] = win_r[(back + k) * RX + t_w];
                                win_p[kk * RX + t_w] = win_p[(back + k) * RX + t_w];
                            }
                        }
                    }
#pragma unroll
                    for (int c = 0; c < SPT; ++c) {
                        const int k = 4 + SPT * t_m + c;
                        float2 r, q;
                        cell(k, r, q, jn[c]);
                        win_r[k * RX + t_w] = r;
                        win_p[k * RX + t_w] = q;
                    }
                    if (t_carry) {
#pragma unroll
                        for (int c = 0; c < SPT; ++c) {
                            const float2 px = jc[2 * c], py = jc[2 * c + 1];
                            jc[2 * c] = jn[c][0];
                            jc[2 * c + 1] = jn[c][1];
                            jn[c][0] = px;
                            jn[c][1] = py;
                        }
                    }
                }
                if (!per && (y0 < 2 || y0 + TY + 1 >= ny)) {   // mirror about the halfway walls
                    __syncthreads();
                    for (int c = tid; c < L::WIN * RX; c += L::NT) {
                        const int k = c / RX, lx = c - k * RX;
                        const int y = y0 - 2 + k;
                        int ym;
                        if (y < 0) ym = -1 - y;
                        else if (y >= ny && y <= ny + 1) ym = 2 * ny - 1 - y;
                        else continue;
                        const int km = ym - (y0 - 2);
                        win_r[k * RX + lx] = win_r[km * RX + lx];
                        win_p[k * RX + lx] = win_p[km * RX + lx];
                    }
                }
                __syncthreads();
                // Site phase.
                const int lx = t_lx, ly = SPT * t_j;
                const int x = x0 + lx, y = y0 + ly;
                if (lx < TX && x < nx && y < ny) {
                    float2 fx[SPT], fy[SPT], qx[SPT], qy[SPT], dp[SPT], dr[SPT];
                    force_sums<SPT, RX>(win_p + ly * RX + lx + 2, win_r + ly * RX + lx + 2, a.k, fx, fy, qx,
                                        qy, dp, dr);
                    float2* const o = m_out + (size_t)y * nx + x;
#pragma unroll
                    for (int s = 0; s < SPT; ++s) {
                        const int ys = y + s;
                        const bool valid = s == 0 || ys < ny;
                        const float2 rho = padd(pset(v.rho_ref), dr[s]);
                        if (valid) note_nonfinite(rho, nf);
                        float2 Fx, Fy, zx, zy;
                        site_force<GEN>(fx[s], fy[s], qx[s], qy[s], dp[s], rho, ys, v, a.k, Fx, Fy);
                        site_velocity<P, true>(rho, jn[s][0], jn[s][1], Fx, Fy, false, a.k, zx, zy);
                        if (valid) {
                            float2* const os = o + s * nx;
                            st_pair(os, dr[s], pol);
                            st_pair(os + N, zx, pol);
                            st_pair(os + 2 * N, zy, pol);
                        }
                        if (!per && valid && (ys == 0 || ys == ny - 1)) {
                            float2 h[9];
                            collide<float, float2, false, true>(nullptr, h, dr[s], rho, zx, zy, a.k, Fx, Fy,
                                                                1.0f);
                            // h[0] = omega w_0 Q as the next step's expansion rounds it: here it
                            // has no use but the density's sum, into which the compiler fuses
                            // the packed product; a scalar one it does not
                            const float2 Q = pfma(pmul(rho, pset(-4.0f / 6.0f)), pfma(zx, zx, pmul(zy, zy)), dr[s]);
                            h[0] = make_float2(__fmul_rn(a.k.omw[0].x, Q.x), __fmul_rn(a.k.omw[0].y, Q.y));
                            wall_columns<float2>(d->wallx, nx, step_k)[(ys == 0 ? 0 : nx) + x] =
                                wall_momentum<P>(h, ys == 0, v);
                        }
                    }
                }
            };
            if constexpr (ALLPER)
                tile_body(std::false_type{});
            else if (per_lat || (y0 >= 3 && y0 + TY + 3 <= ny))
                tile_body(std::false_type{});
            else
                tile_body(std::true_type{});
            base = slot_of(TY);
            wm = wm + 1 == L::WM ? 0 : wm + 1;
        }
        if (!(nf.x == 0.0f && nf.y == 0.0f)) atomicOr(&d->st->err, ERR_NONFINITE);
    }
    if (!a.advance) return;
    if constexpr (!ALLPER) {
        __syncthreads();   // this CTA's wall-site values are written
        wall_sums<P, L>(a, it0, it_end, tid, step_k);
    }
    __syncthreads();
    if (tid == 0) s_last = ticket_arrive(a.ticket) == (unsigned int)(gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    advance_lattices<L::NT>(a, tid, 2);
    if (tid == 0) *a.ticket = 0u;
}

#endif

#if LB_PART == 0
#if LB_PREC == 1
// The populations of a state held by its moments, into population planes with
// their ghost copies.
__global__ void k_expand(Geom g, const __grid_constant__ Coef<float> k, const float2* mom, float2* fout) {
    const size_t N = (size_t)g.nx * g.ny;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < N;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(idx % g.nx), y = (int)(idx / g.nx);
        const float2 r = mom[idx];
        float2 h[9];
        collide<float, float2, false, true>(nullptr, h, r, padd(pset(k.rho_ref), r), mom[N + idx],
                                            mom[2 * N + idx], k, r, r, 1.0f);
#pragma unroll
        for (int i = 0; i < 9; ++i) put2<float2>(fout, g, i, x, y, h[i]);
    }
}
#endif

// m / t, given r = recip(t): m r and one correction by the remainder, which is
// rounded as the division where r is the rounded reciprocal (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", IBM
// J. Res. Dev. 34, 1990) and nothing leaves the normal range; else the division.
// Three FP64 operations (m r alone is up to 1.45 ulp off: one in four velocities
// differed from the division's).
static __device__ __noinline__ double over_slow(double m, double t) { return m / t; }
__device__ __forceinline__ double over(double m, double t, double r) {
    const unsigned hm = (unsigned)__double2hiint(m), ht = (unsigned)__double2hiint(t);
    if (((ht >> 20) & 0x7ffu) - 823u < 400u) {   // |t| within 2^+-200
        const double q = m * r;
        if (((hm >> 20) & 0x7ffu) - 323u < 1400u) return fma(fma(-q, t, m), r, q);   // |m| within 2^+-700
        if (((hm << 1) | (unsigned)__double2loint(m)) == 0u) return q;               // a zero
    }
    return over_slow(m, t);
}

// --------------------------------------------------------- observe kernel
// Fields, totals or populations of one lattice's current state, with the same
// site arithmetic as the step; CTAs take tiles b, b + G, ...  GB300 has two FP64
// lanes per SM and clock, and the observables' FP64 work bounded this kernel
// (2048^2 FP16: 51 FP64-pipe operations a site for the totals, 504 us; 71 for
// the fields, 638 us): floats are widened by integer operations, the sums are
// reduced once per CTA instead of once per tile, one reciprocal serves both
// velocity components, and populations take no force and no totals (2048^2 FP16:
// 15 operations, 154 us, and 21, 222 us; FP32 from the moments about the same).

template <int P, int V, bool POPS>
__global__ void __launch_bounds__(Layout<P>::NT, P == LB_FP64 ? 1 : 2)
    k_observe(const __grid_constant__ CUtensorMap tin,
              const __grid_constant__ StepArgs<typename Prec<P>::C> a) {
    typedef Layout<P> L;
    typedef typename L::T2 T2;
    typedef typename L::C C;
    typedef typename L::C2 C2;
    constexpr bool GEN = (V & 2) != 0;
    constexpr int PS = L::BY * L::BX;    // plane stride in the tile box (pairs)
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    T2* box = reinterpret_cast<T2*>(smem);                    // [9][BY][BX]
    C2* srho = reinterpret_cast<C2*>(smem + L::BOX_STRIDE);   // [RY][RX]
    C2* spsi = srho + L::RX * L::RY;
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_fail, s_last;
    __shared__ double s_red[L::NT / 32][4];
    const int tid = threadIdx.x;
    const Geom& g = a.g;
    const bool per = g.periodic != 0;
    const LatVals<C> v = vals_of(a.k);
    const ExpTable* tab = nullptr;
#if LB_PREC == 0
    tab = &g_exp_tab;
#endif
    bool from_mom = false;
#if LB_PREC == 1
    from_mom = a.mom != nullptr;
#endif
    if (tid == 0) {
        s_fail = 0;
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int ntx = (g.nx + L::TX - 1) / L::TX, ntiles = ntx * ((g.ny + L::TY - 1) / L::TY);
    const size_t N = (size_t)g.nx * g.ny;
    double red[4] = {0.0, 0.0, 0.0, 0.0};
    bool bad = false;
    int phase = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1) {
        const int x0 = (tile % ntx) * L::TX, y0 = (tile / ntx) * L::TY;
#if LB_PREC == 1
        if (from_mom) {   // the box's populations from the state's moments, wrapped (or clamped at walls)
            for (int c = tid; c < L::BY * L::BX; c += L::NT) {
                const int by = c / L::BX, bx = c - by * L::BX;
                int x = (x0 - L::GX + bx) % g.nx, y = y0 - kGY + by;
                x = x < 0 ? x + g.nx : x;
                if (per) {
                    y %= g.ny;
                    y = y < 0 ? y + g.ny : y;
                } else {
                    y = min(max(y, 0), g.ny - 1);
                }
                const float2* m = a.mom + (size_t)y * g.nx + x;
                const float2 r = m[0];
                float2 h[9];
                collide<float, float2, false, true>(nullptr, h, r, padd(pset(a.k.rho_ref), r), m[N], m[2 * N],
                                                    a.k, r, r, 1.0f);
#pragma unroll
                for (int i = 0; i < 9; ++i) box[i * PS + c] = h[i];
            }
        }
#endif
        if (!from_mom) {
            if (tid == 0) {
                fence_proxy_async();   // generic reads of the previous tile's box before async writes
                mbar_expect_tx(&bar, (uint32_t)L::BOX_BYTES);
                tma_load_3d(box, &tin, 2 * x0, y0, 0, &bar);
            }
            if (!mbar_wait_bounded(&bar, phase)) s_fail = 1;
        }
        __syncthreads();
        if (s_fail) break;
        const int lx = tid % L::RX, ly = tid / L::RX;
        const int x = x0 + lx, y = y0 + ly;
        const bool site = lx < L::TX && x < g.nx && y < g.ny;
        const T2* b0 = box + (ly + kGY) * L::BX + lx + L::GX;
        const size_t idx = (size_t)y * g.nx + x;
        C2 h[9];
        if constexpr (POPS) {
            if (site) {
                load_site<P, PS>(b0 - L::BX, b0, b0 + L::BX, y, per, a.pull, g, v, h);
                const C2 r = sum9(h);
                if (!(isfinite(r.x) && isfinite(r.y))) bad = true;
                const double is = (double)inv_scale_of<P>(), rref = (double)v.rho_ref;
#pragma unroll
                for (int q = 0; q < 18; ++q)
                    if (q >= a.q0 && q < a.q1)
                        a.obs_dst[0][(size_t)(q - a.q0) * N + idx] =
                            widen(q < 9 ? h[q % 9].x : h[q % 9].y) * is + wgt<double>(q % 9) * rref;
            }
        } else {
            // box row of lattice row y: y - y0 + kGY; deviation tile row: y - y0 + 2
            for (int c = tid; c < L::RX * L::RY; c += L::NT) {
                const int cy = c / L::RX, cx = c - cy * L::RX;
                const int yc = y0 - 2 + cy;
                if (!per && (yc < 0 || yc >= g.ny)) continue;
                const T2* c0 = box + (cy + 1) * L::BX + cx - 2 + L::GX;
                C2 r, p;
                cell_dev<P, PS>(c0 - L::BX, c0, c0 + L::BX, yc, per, a.pull, g, v, r, p, tab);
                srho[cy * L::RX + cx] = r;
                spsi[cy * L::RX + cx] = p;
            }
            if (!per) {
                __syncthreads();
                for (int c = tid; c < L::RX * L::RY; c += L::NT) {
                    const int cy = c / L::RX, cx = c - cy * L::RX;
                    const int yc = y0 - 2 + cy;
                    int ym;
                    if (yc < 0) ym = -1 - yc;
                    else if (yc >= g.ny) ym = 2 * g.ny - 1 - yc;
                    else continue;
                    const int lm = ym - (y0 - 2);
                    if (lm < 0 || lm >= L::RY) continue;
                    srho[cy * L::RX + cx] = srho[lm * L::RX + cx];
                    spsi[cy * L::RX + cx] = spsi[lm * L::RX + cx];
                }
            }
            __syncthreads();
            C2 fx[1], fy[1], qx[1], qy[1], dp[1], dr[1];
            if constexpr (P == LB_FP64)   // a warp is a row (RX = 32)
                force_sums_warp<L::RX>(spsi + ly * L::RX + lx, srho + ly * L::RX + lx, a.k, fx[0], fy[0], qx[0],
                                       qy[0], dp[0], dr[0]);
            if (site) {
                if constexpr (P != LB_FP64)
                    force_sums<1, L::RX>(spsi + ly * L::RX + lx + 2, srho + ly * L::RX + lx + 2, a.k, fx, fy,
                                         qx, qy, dp, dr);
                load_site<P, PS>(b0 - L::BX, b0, b0 + L::BX, y, per, a.pull, g, v, h);
                C2 jx, jy, Fx, Fy;
                moments<P>(h, jx, jy);
                const C2 rho = padd(pset(v.rho_ref), dr[0]);
                if (!(isfinite(rho.x) && isfinite(rho.y))) bad = true;
                site_force<GEN>(fx[0], fy[0], qx[0], qy[0], dp[0], rho, y, v, a.k, Fx, Fy);
                const double rref = (double)v.rho_ref;
                const double rA = rref + widen(dr[0].x), rB = rref + widen(dr[0].y);
                const double mx = widen(jx.x) + widen(jx.y) + 0.5 * (widen(Fx.x) + widen(Fx.y));
                const double my = widen(jy.x) + widen(jy.y) + 0.5 * (widen(Fy.x) + widen(Fy.y));
                if (a.obs_dst[0]) a.obs_dst[0][idx] = rA;
                if (a.obs_dst[1]) a.obs_dst[1][idx] = rB;
                if (a.obs_dst[2] || a.obs_dst[3]) {
                    const double tot = rA + rB;
                    const unsigned e = ((unsigned)__double2hiint(tot) >> 20) & 0x7ffu;
                    double ux, uy;
                    if (e - 64u < 1920u) {   // well inside the normal range
                        const double r = recip(tot);
                        ux = over(mx, tot, r);
                        uy = over(my, tot, r);
                    } else {
                        ux = tot != 0.0 ? mx / tot : 0.0;
                        uy = tot != 0.0 ? my / tot : 0.0;
                    }
                    if (a.obs_dst[2]) a.obs_dst[2][idx] = ux;
                    if (a.obs_dst[3]) a.obs_dst[3][idx] = uy;
                }
                red[0] += rA;
                red[1] += rB;
                red[2] += mx;
                red[3] += my;
            }
        }
        __syncthreads();   // the box and the window have been read
    }
    if (s_fail && tid == 0) {
        atomicOr(&a.st->err, ERR_TIMEOUT);
        mbar_wait_bounded(&bar, phase);
    }
    if (bad) atomicOr(&a.st->err, ERR_NONFINITE);
    if constexpr (POPS) return;
    const double part = block_sum4<L::NT>(red, s_red);
    if (tid < 32 && (tid & 7) == 0) a.slots[4 * blockIdx.x + (tid >> 3)] = part;
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&a.st->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const volatile double* vs = a.slots;
#pragma unroll
    for (int q = 0; q < 4; ++q) red[q] = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += L::NT)
#pragma unroll
        for (int q = 0; q < 4; ++q) red[q] += vs[4 * b + q];
    const double total = block_sum4<L::NT>(red, s_red);
    if (tid < 32 && (tid & 7) == 0) a.st->totals[tid >> 3] = total;
    // the wall momentum totals: the strips' running totals, in a fixed order
    // (lane l adds strips l, l + 32, ..., then the butterfly)
    if (tid < 32 && !a.g.periodic) {
        double sb = 0.0, st = 0.0;
        for (int i = tid; i < a.nstrips; i += 32) {
            sb += a.wsum[i];
            st += a.wsum[a.nstrips + i];
        }
        sb = warp_sum(sb);
        st = warp_sum(st);
        if (tid == 0) {
            a.st->sum_bot = sb * (1.0 / a.g.nx);
            a.st->sum_top = st * (1.0 / a.g.nx);
        }
    }
    if (tid == 0) {
        a.st->ticket = 0u;
        __threadfence();
    }
}

// ------------------------------------------------------------ init kernels
// f(r, 0) = f^eq(rho_s, u) in place (the first step reads it unshifted).
// rho_s from the counter generator (rA null), or from FP64 fields (ux, uy null:
// zero).  The lattice's counters and wall totals are set along with it, so that
// an initialisation is one launch.
__device__ __forceinline__ void init_state(const StateInit& z) {
    if (!z.st || blockIdx.x != 0 || blockIdx.y != 0) return;
    if (threadIdx.x == 0) {
        DevStats st = {};
        st.t = z.t;
        st.next_sample = z.next_sample;
        st.pull = z.pull;
        *z.st = st;
    }
    for (int i = threadIdx.x; i < z.nwsum; i += blockDim.x) z.wsum[i] = 0.0;
}
template <int P>
__global__ void k_init(Geom g, Coef<typename Prec<P>::C> k, typename Prec<P>::T2* fout,
                       const double* rA, const double* rB, const double* fux, const double* fuy,
                       double rho0, double amp, double u_wall, int init_shear, unsigned long long seed,
                       StateInit state) {
    typedef typename Prec<P>::T2 T2;
    init_state(state);
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    for (int y = blockIdx.y; y < g.ny; y += gridDim.y) {
        const size_t idx = (size_t)y * g.nx + x;
        double r[2], ux, uy;
        if (!rA) {
            for (int s = 0; s < 2; ++s) {
                const uint64_t ctr = ((uint64_t)s * g.ny + y) * g.nx + x;
                const uint64_t z = mix64(seed ^ mix64(ctr + 0x9E3779B97F4A7C15ULL));
                // x = z >> 11 as a double: its low 52 bits as the fraction of
                // 2^52 + (x mod 2^52), less 2^52 unless bit 52 is set (exact)
                const double f = __hiloint2double((int)((unsigned)(z >> 43) & 0xfffffu | 0x43300000u), (int)(z >> 11));
                const double u = ((long long)z < 0 ? f : f - 4503599627370496.0) * (1.0 / 9007199254740992.0);
                r[s] = rho0 * (1.0 + amp * (2.0 * u - 1.0));
            }
            ux = init_shear ? u_wall * (2.0 * y + 1.0 - g.ny) / (double)g.ny : 0.0;
            uy = 0.0;
        } else {
            r[0] = rA[idx];
            r[1] = rB[idx];
            ux = fux ? fux[idx] : 0.0;
            uy = fuy ? fuy[idx] : 0.0;
        }
        const double usq = ux * ux + uy * uy;
        const double rref = (double)k.rho_ref;
        if (ux == 0.0 && uy == 0.0) {
            // at rest: sc w_i (rho - rho_ref), three values per species (the
            // terms below, which are exact zeros, bound this kernel by their
            // FP64 operations)
            const double sc = (double)scale_of<P>();
            const double dA = r[0] - rref, dB = r[1] - rref;
#pragma unroll
            for (int i = 0; i < 9; ++i)
                put2<T2>(fout, g, i, x, y, encd2<T2>(sc * wgt<double>(i) * dA, sc * wgt<double>(i) * dB));
            continue;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double cu = cx(i) * ux + cy(i) * uy;
            const double e = 3.0 * cu + 4.5 * cu * cu - 1.5 * usq;
            // f^eq_i - w_i rho_ref for both species
            const double sc = (double)scale_of<P>();
            const double hA = sc * wgt<double>(i) * ((r[0] - rref) + r[0] * e);
            const double hB = sc * wgt<double>(i) * ((r[1] - rref) + r[1] * e);
            put2<T2>(fout, g, i, x, y, encd2<T2>(hA, hB));
        }
    }
}

// Restore directions [i0, i1) of a saved state: pops holds FP64 populations
// f_is(r), species s of direction i at s species + (i - i0) direction; the
// offsets f - w_i rho_ref are encoded to the storage format (plus ghost copies).
template <int P>
__global__ void k_load_pops(Geom g, typename Prec<P>::C rho_ref, typename Prec<P>::T2* fout,
                            const double* pops, size_t species, size_t direction, int i0, int i1,
                            StateInit state) {
    typedef typename Prec<P>::T2 T2;
    init_state(state);
    const double rref = (double)rho_ref;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    for (int y = blockIdx.y; y < g.ny; y += gridDim.y) {
        const double* src = pops + (size_t)y * g.nx + x;
        double f[9][2];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (i >= i0 && i < i1) {
                f[i][0] = src[(size_t)(i - i0) * direction];
                f[i][1] = src[(size_t)(i - i0) * direction + species];
            }
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (i >= i0 && i < i1) {
                const double off = wgt<double>(i) * rref, sc = (double)scale_of<P>();
                put2<T2>(fout, g, i, x, y, encd2<T2>(sc * (f[i][0] - off), sc * (f[i][1] - off)));
            }
    }
}

// ------------------------------------------------------ wait self-test
// One CTA arms an mbarrier that no copy will ever complete and waits on it
// with the step kernel's bounded wait (bound `limit`); the wait gives up, the
// kernel latches ERR_TIMEOUT in *err and returns, leaving the context usable.
// (Compiled in the FP32 translation unit only.)
#if LB_PREC == 1
// ------------------------------------------------------ FP32 math probe
// The step kernel's FP32 exp(x) - 1 and reciprocal on caller values, next
// to the CUDA library's expm1f: out[3k] = pexpm1(x[k]), out[3k + 1] =
// expm1f(x[k]), out[3k + 2] = recip(x[k]) (x[k] taken in pairs, as the
// kernel does; an odd tail element is paired with itself).
__global__ void k_math_probe(const float* __restrict__ x, float* __restrict__ out, long long n) {
    for (long long k = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); k < n;
         k += 2LL * gridDim.x * blockDim.x) {
        const float a = x[k], b = k + 1 < n ? x[k + 1] : a;
        const float2 e = pexpm1(make_float2(a, b));
        out[3 * k] = e.x;
        out[3 * k + 1] = expm1f(a);
        out[3 * k + 2] = recip(a);
        if (k + 1 < n) {
            out[3 * k + 3] = e.y;
            out[3 * k + 4] = expm1f(b);
            out[3 * k + 5] = recip(b);
        }
    }
}

__global__ void k_wait_selftest(unsigned int* err, int limit) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0, limit)) atomicOr(err, ERR_TIMEOUT);
}
#endif

#if LB_PREC == 0
// The FP64 functions of the step and observe kernels on caller values, next to
// CUDA's: see lb_selftest_math64.
__global__ void k_math64_probe(double rho0, const double* __restrict__ x, const double* __restrict__ y,
                               double* __restrict__ out, long long n) {
    const double inv_rho0 = 1.0 / rho0, c = -64.0 / (0.693147180559945309417 * rho0);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const double a = x[k], b = y[k];
        out[6 * k] = pexpm1_scaled(make_double2(a, b), c, inv_rho0, &g_exp_tab).x;
        out[6 * k + 1] = expm1(-a * inv_rho0);
        out[6 * k + 2] = recip(a);
        out[6 * k + 3] = 1.0 / a;
        out[6 * k + 4] = over(b, a, recip(a));
        out[6 * k + 5] = b / a;
    }
}
#endif
#endif   // LB_PART == 0

// ------------------------------------------------------------- launchers
// A kernel's opt-in to its dynamic shared memory and to room for its resident
// CTAs: at its first launch on each device.
struct OptIn {
    std::atomic<unsigned long long> devices{0};
};
template <typename K>
static cudaError_t opt_in(OptIn& done, K kernel, int bytes) {
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
    if (done.devices.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) done.devices.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

#if LB_PART != 0
// LB_PDL=0 in the environment turns the programmatic launches off (A/B
// timing); read once per process.
static bool pdl_enabled() {
    static const bool on = [] {
        const char* v = getenv("LB_PDL");
        return !(v && v[0] == '0');
    }();
    return on;
}

// Consecutive steps on a stream overlap the next launch's set-up with the
// previous launch's last CTAs (programmatic stream serialization); the kernels
// wait for the previous grid before they read the lattice state.
template <typename K, typename A>
static cudaError_t launch_pdl(K kernel, const A& a, int threads, int smem, dim3 grid, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

#if LB_PART == 4
constexpr int kVariants = 8;
template <int P, int SH> using StepLayout = DLayout<P>;
template <int P, int SH, int V> static constexpr auto step_kernel() { return &k_step_d<P, V>; }
#elif LB_PART == 5   // (omega = 1 throughout: no variant bit 2)
constexpr int kVariants = 4;
template <int P, int SH> using StepLayout = MLayout<SH>;
template <int P, int SH, int V> static constexpr auto step_kernel() { return &k_step_m<V, SH>; }
#else
constexpr int kVariants = 8;
template <int P, int SH> using StepLayout = Layout<P, SH>;
template <int P, int SH, int V> static constexpr auto step_kernel() { return &k_step<P, V, SH>; }
#endif

template <int P, int SH, int V>
static cudaError_t launch_variant(const void* args, dim3 grid, cudaStream_t s) {
    typedef StepLayout<P, SH> L;
    static OptIn done;
    const cudaError_t e = opt_in(done, step_kernel<P, SH, V>(), L::SMEM);
    if (e != cudaSuccess || !args) return e;
    return launch_pdl(step_kernel<P, SH, V>(), *reinterpret_cast<const BatchArgs<typename Prec<P>::C>*>(args), L::NT,
                      L::SMEM, grid, s);
}
template <int P, int SH, int... V>
static cudaError_t launch_one_of(const void* args, int variant, dim3 grid, cudaStream_t s,
                                 std::integer_sequence<int, V...>) {
    cudaError_t e = cudaErrorInvalidValue;
    (void)((variant == V && ((e = launch_variant<P, SH, V>(args, grid, s)), true)) || ...);
    return e;
}
template <int P, int SH>
cudaError_t launch_step_shape(const void* args, int variant, dim3 grid, cudaStream_t s) {
    return launch_one_of<P, SH>(args, variant & (kVariants - 1), grid, s, std::make_integer_sequence<int, kVariants>{});
}
template cudaError_t launch_step_shape<LB_PREC, LB_PART>(const void*, int, dim3, cudaStream_t);
#if LB_PART == 5
template cudaError_t launch_step_shape<LB_PREC, SHAPE_M8X2>(const void*, int, dim3, cudaStream_t);
#endif

#else   // LB_PART == 0
#if LB_PREC == 1
cudaError_t launch_expand(const Geom& g, const Coef<float>& k, const float2* mom, void* fout,
                          cudaStream_t s) {
    const long long N = (long long)g.nx * g.ny;
    const long long blocks = (N + 255) / 256;
    k_expand<<<(unsigned)(blocks < 152 * 32 ? blocks : 152 * 32), 256, 0, s>>>(
        g, k, mom, reinterpret_cast<float2*>(fout));
    return cudaGetLastError();
}
#endif

template <int P>
cudaError_t launch_step_prec(const void* args, int variant, int shape, dim3 grid, cudaStream_t s) {
    switch (shape) {
        case SHAPE_8: return launch_step_shape<P, SHAPE_8>(args, variant, grid, s);
        case SHAPE_16:
            if constexpr (has_shape(P, SHAPE_16)) return launch_step_shape<P, SHAPE_16>(args, variant, grid, s);
            break;
        case SHAPE_8X2:
            if constexpr (has_shape(P, SHAPE_8X2)) return launch_step_shape<P, SHAPE_8X2>(args, variant, grid, s);
            break;
        case SHAPE_D8:
            if constexpr (has_shape(P, SHAPE_D8)) return launch_step_shape<P, SHAPE_D8>(args, variant, grid, s);
            break;
        case SHAPE_M8:
            if constexpr (has_shape(P, SHAPE_M8)) return launch_step_shape<P, SHAPE_M8>(args, variant, grid, s);
            break;
        case SHAPE_M8X2:
            if constexpr (has_shape(P, SHAPE_M8X2)) return launch_step_shape<P, SHAPE_M8X2>(args, variant, grid, s);
            break;
    }
    return cudaErrorInvalidValue;
}

template <int P, int V, bool POPS>
static cudaError_t observe(const CUtensorMap* tin, const void* args, dim3 grid, cudaStream_t s) {
    typedef Layout<P> L;
    static OptIn done;
    const cudaError_t e = opt_in(done, k_observe<P, V, POPS>, L::SMEM_OBS);
    if (e != cudaSuccess) return e;
    k_observe<P, V, POPS><<<grid, L::NT, L::SMEM_OBS, s>>>(
        *tin, *reinterpret_cast<const StepArgs<typename L::C>*>(args));
    return cudaGetLastError();
}
template <int P>
cudaError_t launch_observe_prec(const CUtensorMap* tin, const void* args, dim3 grid,
                                cudaStream_t s) {
    const auto& a = *reinterpret_cast<const StepArgs<typename Prec<P>::C>*>(args);
    if (a.obs == OBS_POPS)
        return a.g.periodic ? observe<P, 3, true>(tin, args, grid, s) : observe<P, 2, true>(tin, args, grid, s);
    return a.g.periodic ? observe<P, 3, false>(tin, args, grid, s) : observe<P, 2, false>(tin, args, grid, s);
}

// One thread per column, rows dealt over the grid: no index is divided.
static dim3 site_grid(const Geom& g) {
    const unsigned gx = (unsigned)((g.nx + 127) / 128);
    const unsigned gy = gx < 152 * 128 ? 152 * 128 / gx : 1;
    return dim3(gx, (unsigned)g.ny < gy ? (unsigned)g.ny : gy, 1);
}
template <int P>
cudaError_t launch_init_prec(const Geom& g, const void* coef, void* fout, const double* const* fields,
                             double rho0, double amp, double u_wall, int init_shear,
                             unsigned long long seed, const StateInit& state, cudaStream_t s) {
    typedef typename Prec<P>::C C;
    typedef typename Prec<P>::T2 T2;
    const double* const none[4] = {nullptr, nullptr, nullptr, nullptr};
    const double* const* f = fields ? fields : none;
    k_init<P><<<site_grid(g), 128, 0, s>>>(g, *reinterpret_cast<const Coef<C>*>(coef),
                                           reinterpret_cast<T2*>(fout), f[0], f[1], f[2], f[3], rho0, amp,
                                           u_wall, init_shear, seed, state);
    return cudaGetLastError();
}
template <int P>
cudaError_t launch_load_pops_prec(const Geom& g, const void* coef, void* fout, const double* pops,
                                  size_t species, size_t direction, int i0, int i1,
                                  const StateInit& state, cudaStream_t s) {
    typedef typename Prec<P>::C C;
    typedef typename Prec<P>::T2 T2;
    k_load_pops<P><<<site_grid(g), 128, 0, s>>>(g, reinterpret_cast<const Coef<C>*>(coef)->rho_ref,
                                                reinterpret_cast<T2*>(fout), pops, species, direction, i0, i1,
                                                state);
    return cudaGetLastError();
}

template cudaError_t launch_step_prec<LB_PREC>(const void*, int, int, dim3, cudaStream_t);
template cudaError_t launch_observe_prec<LB_PREC>(const CUtensorMap*, const void*, dim3,
                                                  cudaStream_t);
template cudaError_t launch_load_pops_prec<LB_PREC>(const Geom&, const void*, void*, const double*,
                                                    size_t, size_t, int, int, const StateInit&,
                                                    cudaStream_t);
template cudaError_t launch_init_prec<LB_PREC>(const Geom&, const void*, void*, const double* const*,
                                               double, double, double, int, unsigned long long,
                                               const StateInit&, cudaStream_t);

#if LB_PREC == 0
cudaError_t launch_math64_probe(double rho0, const double* x, const double* y, double* out, long long n,
                                cudaStream_t s) {
    long long blocks = (n + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_math64_probe<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, s>>>(rho0, x, y, out, n);
    return cudaGetLastError();
}
#elif LB_PREC == 1
cudaError_t launch_wait_selftest(unsigned int* err, int limit, cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(err, limit);
    return cudaGetLastError();
}
cudaError_t launch_math_probe(const float* x, float* out, long long n, cudaStream_t s) {
    long long blocks = (n + 511) / 512;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_math_probe<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, s>>>(x, out, n);
    return cudaGetLastError();
}
#endif
#endif   // LB_PART == 0

}  // namespace lbgb
