// lb_noalloc.cu -- lb_totals_noalloc: the FP64 mass/momentum reduction of
// the observe pass, for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: code that runs inside a fixed device
// arena it may not grow, or inside a framework that forbids allocation on its
// hot path.  lb_create allocates, and lb_create_in still needs a workspace for
// the reduction slots.  This entry point takes the caller's device fields and
// output and keeps its scratch -- one FP64 partial-sum slot per CTA -- in a
// file-scope device array of fixed size, which every GPU that loads the library
// holds until the process exits.
#include <mutex>

#include "lb_internal.h"

namespace lbgb {
namespace {

constexpr int kThreads = 256;
constexpr int kGroup = 4;                                   // sites of one thread at a time
constexpr long long kChunk = (long long)kThreads * kGroup;  // sites of a CTA at a time
// CTAs of a large reduction: four per SM of a 152-SM GPU (each thread has 16
// loaded values in flight, 128 KB on an SM -- three times what the memory
// latency needs at full bandwidth -- and while one CTA waits for its loads
// the others keep the FP64 pipe busy).
constexpr int kMaxBlocks = 608;
// Up to this many sites one CTA writes the totals itself: it needs no second
// kernel, whose launch costs more than the turns.
constexpr long long kOneBlockSites = 8 * kChunk;

// Scratch: one slot of four FP64 partial sums per CTA.
struct NoAllocScratch {
    double slots[kMaxBlocks][4];
};
constexpr size_t kScratchDoubles = sizeof(NoAllocScratch) / sizeof(double);

static __device__ __align__(256) double g_noalloc_scratch[kScratchDoubles];

// Running sum of doubles.  GB300 has two FP64 lanes per SM and clock, and the
// masses' plain FP64 additions would be two of a site's five FP64 operations,
// so densities are summed as 64-bit integers instead, on the integer pipe:
// mantissas (53 bits) shifted by 5 and aligned to a reference exponent `eref`,
// set two above the largest of the first group.  A term is below 2^58; up to
// 32 of them are added before the sum is rounded to FP64 (flush).  Terms down
// to 2^-3 of the first group's largest stay exact, smaller ones lose less than
// 2^-55 of it -- less than an FP64 addition rounds off.  Groups that do not
// fit the reference start a new one; values that are not positive, normal and
// finite, or lie 2^29 or more apart, take FP64 additions.
struct MassSum {
    unsigned long long acc = 0;
    int eref = 0, terms = 0;
    double sum = 0.0;

    __device__ __forceinline__ void flush() {
        // times 2^(eref - 1075 - 5), a normal number (eref >= 66)
        if (terms) sum = fma((double)acc, __hiloint2double((eref - 57) << 20, 0), sum);
        acc = 0;
        terms = 0;
    }
    __device__ __forceinline__ void add(const double v[kGroup]) {
        int hi[kGroup], mx = __double2hiint(v[0]), mn = mx;
#pragma unroll
        for (int k = 0; k < kGroup; ++k) {
            hi[k] = __double2hiint(v[k]);
            mx = max(mx, hi[k]);
            mn = min(mn, hi[k]);
        }
        const int emax = mx >> 20, emin = mn >> 20;
        if (!(terms && terms <= 32 - kGroup && emax <= eref && eref - emin <= 31)) {
            flush();
            eref = emax + 2;
            // 64 <= emin: also excludes zero, subnormal and negative values;
            // eref <= 2046: excludes non-finite ones
            if (!(emin >= 64 && eref <= 2046 && eref - emin <= 31)) {
#pragma unroll
                for (int k = 0; k < kGroup; ++k) sum += v[k];
                return;
            }
        }
#pragma unroll
        for (int k = 0; k < kGroup; ++k) {
            const unsigned int lo = (unsigned int)__double2loint(v[k]);
            const unsigned int mh = ((unsigned int)hi[k] & 0xfffffu) | 0x100000u;
            const unsigned int d = (unsigned int)(eref - (hi[k] >> 20));   // 0 .. 31
            const unsigned int h5 = __funnelshift_l(lo, mh, 5), l5 = lo << 5;
            acc += ((unsigned long long)(h5 >> d) << 32) | __funnelshift_r(l5, h5, d);
        }
        terms += kGroup;
    }
};

// Block sum of v[0..3] in a fixed order; sum k is thread 8 k's result.
// The four sums share the butterfly: its first two steps hand half of the
// lanes' values over instead of adding all four everywhere, so a warp takes
// 6 FP64 additions instead of 20.
__device__ __forceinline__ double block_sum4d(const double v[4], double (*s_red)[4]) {
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool h16 = lane & 16, h8 = lane & 8;
    double a = (h16 ? v[2] : v[0]) + __shfl_xor_sync(full, h16 ? v[0] : v[2], 16);
    double b = (h16 ? v[3] : v[1]) + __shfl_xor_sync(full, h16 ? v[1] : v[3], 16);
    a = (h8 ? b : a) + __shfl_xor_sync(full, h8 ? a : b, 8);
    a += __shfl_xor_sync(full, a, 4);
    a += __shfl_xor_sync(full, a, 2);
    a += __shfl_xor_sync(full, a, 1);
    if ((lane & 7) == 0) s_red[warp][lane >> 3] = a;   // value 2 (lane >> 4) + (lane >> 3 & 1)
    __syncthreads();
    static_assert(kThreads == 256, "8 warps x 4 sums in one warp");
    if (warp == 0) {
        a = s_red[lane & 7][lane >> 3];
        a += __shfl_xor_sync(full, a, 4);
        a += __shfl_xor_sync(full, a, 2);
        a += __shfl_xor_sync(full, a, 1);
    }
    return a;   // lanes 8 k of warp 0: sum k
}

// Partial sums: CTA b sums chunks b, b + G, ... of kChunk sites into its slot
// (a single CTA straight into `out`).  VEC: 16-byte loads (all four arrays
// 16-byte aligned); every thread issues the group's loads of all four arrays
// before it uses one.  Bound by the FP64 pipe (three operations a site, 1.5
// clocks of an SM against 1.4 for the 32 bytes): 2048^2 takes 39 us a call
// (with one FP64 addition per mass, a counter cleared before each call and
// 8-byte loads 65 us), 4096^2 121 us (217), 4.4 TB/s.
template <bool VEC>
__global__ void __launch_bounds__(kThreads, 4)
    k_totals(NoAllocScratch* sc, long long n, const double* __restrict__ rA,
             const double* __restrict__ rB, const double* __restrict__ ux,
             const double* __restrict__ uy, double* __restrict__ out) {
    __shared__ double s_red[kThreads / 32][4];
    const int tid = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    MassSum mA, mB;
    for (long long base = (long long)blockIdx.x * kChunk; base < n; base += (long long)gridDim.x * kChunk) {
        if (base + kChunk <= n) {
            double a[kGroup], b[kGroup], x[kGroup], y[kGroup];
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                if (VEC) {
                    if (k & 1) continue;
                    const long long i = base + (long long)(k / 2) * (2 * kThreads) + 2 * tid;
                    const double2 da = *reinterpret_cast<const double2*>(rA + i);
                    const double2 db = *reinterpret_cast<const double2*>(rB + i);
                    const double2 dx = *reinterpret_cast<const double2*>(ux + i);
                    const double2 dy = *reinterpret_cast<const double2*>(uy + i);
                    a[k] = da.x, a[k + 1] = da.y;
                    b[k] = db.x, b[k + 1] = db.y;
                    x[k] = dx.x, x[k + 1] = dx.y;
                    y[k] = dy.x, y[k + 1] = dy.y;
                } else {
                    const long long i = base + (long long)k * kThreads + tid;
                    a[k] = rA[i];
                    b[k] = rB[i];
                    x[k] = ux[i];
                    y[k] = uy[i];
                }
            }
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                const double tot = a[k] + b[k];
                v[2] = fma(tot, x[k], v[2]);
                v[3] = fma(tot, y[k], v[3]);
            }
            mA.add(a);
            mB.add(b);
        } else {
            for (long long i = base + tid; i < n; i += kThreads) {
                const double a = rA[i], b = rB[i], tot = a + b;
                v[0] += a;
                v[1] += b;
                v[2] = fma(tot, ux[i], v[2]);
                v[3] = fma(tot, uy[i], v[3]);
            }
        }
    }
    mA.flush();
    mB.flush();
    v[0] += mA.sum;
    v[1] += mB.sum;
    const double r = block_sum4d(v, s_red);
    if (tid < 32 && (tid & 7) == 0) (gridDim.x == 1 ? out : sc->slots[blockIdx.x])[tid >> 3] = r;
}

// Sum of the slots, in a fixed order.  Launched with programmatic stream
// serialization: its launch overlaps the partial sums, and it waits for them
// (no arrival counter, and so no clearing of one before every call).
__global__ void __launch_bounds__(kThreads)
    k_totals_final(const NoAllocScratch* sc, int nslots, double* __restrict__ out) {
    __shared__ double s_red[kThreads / 32][4];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nslots; b += kThreads)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += sc->slots[b][k];
    const double r = block_sum4d(v, s_red);
    if (threadIdx.x < 32 && (threadIdx.x & 7) == 0) out[threadIdx.x >> 3] = r;
}

// Unique id of the calling thread's current context (cuCtxGetId: unique over
// the life of the process, unlike the CUcontext handle, which a context
// created after a device reset may reuse).  False when there is no current
// context yet or the driver does not offer the call.
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

bool current_context_id(unsigned long long* id) {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static bool looked_up = false;
    if (!looked_up) {
        void* a = nullptr;
        void* b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa) ==
                cudaSuccess && qa == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) ==
                cudaSuccess && qb == cudaDriverEntryPointSuccess) {
            get_current = reinterpret_cast<CtxGetCurrentFn>(a);
            get_id = reinterpret_cast<CtxGetIdFn>(b);
        }
        cudaGetLastError();
        looked_up = true;
    }
    CUcontext ctx = nullptr;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return get_id(ctx, id) == CUDA_SUCCESS;
}

// Device address of the scratch array, looked up once per device and
// context: a context created after a device reset loads the module again,
// possibly elsewhere, so its address is looked up afresh.
std::mutex g_mu;
void* g_addr[64] = {nullptr};
unsigned long long g_ctx[64] = {0};

lb_status scratch_address(NoAllocScratch** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LB_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_mu);
    unsigned long long id = 0;
    bool have_id = current_context_id(&id);
    if (!g_addr[dev] || !have_id || g_ctx[dev] != id) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return LB_ERR_CUDA;
        }
        // the lookup made the device's primary context current if it was not
        if (!have_id) have_id = current_context_id(&id);
        g_addr[dev] = p;
        g_ctx[dev] = have_id ? id : 0;
        if (!have_id) {   // no context id to key on: look up again next call
            *out = reinterpret_cast<NoAllocScratch*>(p);
            g_addr[dev] = nullptr;
            return LB_OK;
        }
    }
    *out = reinterpret_cast<NoAllocScratch*>(g_addr[dev]);
    return LB_OK;
}

}  // namespace
}  // namespace lbgb

extern "C" lb_status lb_totals_noalloc(int32_t nx, int32_t ny, const double* rho_A,
                                        const double* rho_B, const double* ux, const double* uy,
                                        double* totals, void* stream) {
    using namespace lbgb;
    if (nx < 1 || ny < 1 || !rho_A || !rho_B || !ux || !uy || !totals) return LB_ERR_INVALID;
    const long long n = (long long)nx * ny;
    if (n > LB_NOALLOC_MAX_SITES) return LB_ERR_INVALID;
    NoAllocScratch* sc = nullptr;
    lb_status s = scratch_address(&sc);
    if (s != LB_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bool vec = ((reinterpret_cast<uintptr_t>(rho_A) | reinterpret_cast<uintptr_t>(rho_B) |
                       reinterpret_cast<uintptr_t>(ux) | reinterpret_cast<uintptr_t>(uy)) & 15) == 0;
    long long blocks = n <= kOneBlockSites ? 1 : (n + kChunk - 1) / kChunk;
    if (blocks > kMaxBlocks) blocks = kMaxBlocks;
    if (vec)
        k_totals<true><<<(unsigned)blocks, kThreads, 0, st>>>(sc, n, rho_A, rho_B, ux, uy, totals);
    else
        k_totals<false><<<(unsigned)blocks, kThreads, 0, st>>>(sc, n, rho_A, rho_B, ux, uy, totals);
    if (blocks > 1) {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, k_totals_final, (const NoAllocScratch*)sc, (int)blocks, totals) !=
            cudaSuccess) {
            cudaGetLastError();
            return LB_ERR_CUDA;
        }
    }
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}
