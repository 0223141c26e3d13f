// A stand-in for the CUDA runtime, for tests of the library's host code on a
// machine without a GPU.  "Device" memory is host memory with every allocation
// on record; copies run at once and are checked against the records; kernels do
// not run, their launches are recorded, and a step launch's tables are checked:
// descriptors, work items and CTA offsets lie in live allocations, and the
// items lie in their lattices.  A call can be made to fail (fk_fail).
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../paper_0807_4471_gb300/csrc/lb_internal.h"

#undef cudaEventElapsedTime
#undef cudaGetDriverEntryPointByVersion

namespace {

struct Range {
    size_t bytes;
    int type;   // cudaMemoryTypeDevice or cudaMemoryTypeHost
    bool live;
    bool owned;
};
struct LaunchRec {
    std::string name;
    unsigned grid, block;
    std::string items;   // step launches: the item table and CTA offsets, as text
    std::vector<double*> dst;   // observe launches: the outputs
};
std::map<char*, Range> ranges;
std::map<std::string, int> calls;
struct Fault {
    int nth, err;
};
std::map<std::string, Fault> faults;
std::map<const void*, std::string> kernels;
std::map<std::string, int> module_of;   // kernel name -> the module (compilation unit) it is in
int modules = 0;
std::vector<LaunchRec> launches;
std::string errors;
int sms = 152;
cudaError_t last = cudaSuccess;

void complain(const std::string& s) { errors += s + "\n"; }

// Counts a call; the error it is to fail with, or success.
cudaError_t call(const char* name) {
    ++calls[name];
    auto it = faults.find(name);
    if (it != faults.end() && --it->second.nth == 0) {
        last = (cudaError_t)it->second.err;
        faults.erase(it);
        return last;
    }
    return cudaSuccess;
}

Range* find(const void* p, char** start = nullptr) {
    auto it = ranges.upper_bound((char*)p);
    if (it == ranges.begin()) return nullptr;
    --it;
    if ((char*)p >= it->first + it->second.bytes) return nullptr;
    if (start) *start = it->first;
    return &it->second;
}
// [p, p + bytes) lies in one live allocation of the type
bool inside(const void* p, size_t bytes, int type) {
    char* s;
    Range* r = find(p, &s);
    return r && r->live && r->type == type && (char*)p + bytes <= s + r->bytes;
}

char* take(size_t bytes, int type) {
    char* p = (char*)aligned_alloc(256, (bytes + 255) / 256 * 256);
    memset(p, 0, (bytes + 255) / 256 * 256);
    ranges[p] = Range{bytes, type, true, true};
    return p;
}
void drop(void* p, int type, const char* what) {
    if (!p) return;
    auto it = ranges.find((char*)p);
    if (it == ranges.end() || !it->second.live || it->second.type != type)
        complain(std::string(what) + " of memory that is not allocated");
    else
        it->second.live = false;   // kept: a later use is reported, not a crash
}

template <typename C>
void check_step(const lbgb::BatchArgs<C>& a, bool rows, int tile_rows, unsigned grid, LaunchRec& rec) {
    const int dev = cudaMemoryTypeDevice;
    if (!inside(a.lat, sizeof(lbgb::LatDesc<C>) * (size_t)a.nlat, dev)) return complain("step: descriptors not in live memory");
    if (!inside(a.items, sizeof(int4) * (size_t)a.nitems, dev)) return complain("step: items not in live memory");
    if (!inside(a.cta_items, sizeof(int) * (grid + 1), dev)) return complain("step: CTA offsets not in live memory");
    if (!inside(a.ticket, 4, dev)) return complain("step: ticket not in live memory");
    if (a.cta_items[0] != 0 || a.cta_items[grid] != a.nitems) complain("step: CTA offsets do not span the items");
    for (unsigned b = 0; b < grid; ++b)
        if (a.cta_items[b] > a.cta_items[b + 1]) complain("step: CTA offsets not ascending");
    for (int l = 0; l < a.nlat; ++l)
        for (int b = 0; b < 2; ++b)
            if (!inside(a.lat[l].fbuf[b], 1, dev)) complain("step: a lattice's buffer is not in live memory");
    for (int k = 0; k < a.nitems; ++k) {
        const int4 w = a.items[k];
        if (w.x < 0 || w.x >= a.nlat) {
            complain("step: item of no lattice");
            continue;
        }
        const lbgb::LatDesc<C>& d = a.lat[w.x];
        const int end = rows ? d.g.ny : (d.g.ny + tile_rows - 1) / tile_rows;
        if (w.y < 0 || w.y >= d.nstrips || w.z < 0 || w.z >= w.w || w.w > end || d.ntiles_y != end)
            complain("step: item outside its lattice");
    }
    char line[96];
    for (unsigned b = 0; b < grid; ++b)
        for (int k = a.cta_items[b]; k < a.cta_items[b + 1]; ++k) {
            snprintf(line, sizeof line, "%u %d %d %d %d\n", b, a.items[k].x, a.items[k].y, a.items[k].z, a.items[k].w);
            rec.items += line;
        }
}

cudaError_t launch(const void* func, dim3 grid, dim3 block, void** args, const char* api) {
    const cudaError_t e = call(api);
    if (e != cudaSuccess) return e;
    LaunchRec rec{kernels.count(func) ? kernels[func] : "?", grid.x, block.x, "", {}};
    const std::string& n = rec.name;
    // k_step<P, V, SHAPE>, k_step_d<P, V>, k_step_m<V, SHAPE>, mangled
    size_t at;
    int p = 0, v = 0, sh = 0;
    if ((at = n.find("k_stepILi")) != std::string::npos && sscanf(n.c_str() + at, "k_stepILi%dELi%dELi%dE", &p, &v, &sh) == 3) {
        if (p == LB_FP64) check_step(*(const lbgb::BatchArgs<double>*)args[0], true, 8, grid.x, rec);
        else check_step(*(const lbgb::BatchArgs<float>*)args[0], false, lbgb::shape_rows(sh), grid.x, rec);
    } else if (n.find("k_step_d") != std::string::npos || n.find("k_step_m") != std::string::npos) {
        check_step(*(const lbgb::BatchArgs<float>*)args[0], false, 8, grid.x, rec);
    } else if ((at = n.find("k_observeILi")) != std::string::npos) {
        double* const* d = n[at + 12] == '0' ? ((const lbgb::StepArgs<double>*)args[1])->obs_dst
                                             : ((const lbgb::StepArgs<float>*)args[1])->obs_dst;
        rec.dst.assign(d, d + 4);
    }
    launches.push_back(rec);
    return cudaSuccess;
}

struct Config {
    dim3 grid, block;
    size_t shmem;
    void* stream;
} pushed;

CUresult encode(...) { return CUDA_SUCCESS; }
CUresult ctx_current(CUcontext* c) {
    *c = (CUcontext)8;
    return CUDA_SUCCESS;
}
CUresult ctx_id(CUcontext, unsigned long long* id) {
    *id = 1;
    return CUDA_SUCCESS;
}
CUresult pointer_attribute(void* data, CUpointer_attribute a, CUdeviceptr p) {
    char* s;
    Range* r = find((void*)p, &s);
    if (!r || !r->live) return CUDA_ERROR_INVALID_VALUE;
    if (a == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr*)data = (CUdeviceptr)s;
    else if (a == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t*)data = r->bytes;
    else return CUDA_ERROR_INVALID_VALUE;
    return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---------------------------------------------------------------- controls
int fk_count(const char* name) { return calls.count(name) ? calls[name] : 0; }
void fk_reset() {
    calls.clear();
    launches.clear();
}
// The nth call from now of a function (1: the next) returns err.
void fk_fail(const char* name, int nth, int err) { faults[name] = Fault{nth, err}; }
void fk_sms(int n) { sms = n; }
// Memory that counts as pinned from now on.
void fk_pin(void* p, size_t bytes) { ranges[(char*)p] = Range{bytes, cudaMemoryTypeHost, true, false}; }
const char* fk_errors() { return errors.c_str(); }
int fk_launches() { return (int)launches.size(); }
const char* fk_launch_name(int k) { return launches[(size_t)k].name.c_str(); }
int fk_launch_grid(int k) { return (int)launches[(size_t)k].grid; }
const char* fk_launch_items(int k) { return launches[(size_t)k].items.c_str(); }
void* fk_launch_dst(int k, int q) {
    return launches[(size_t)k].dst.size() ? launches[(size_t)k].dst[(size_t)q] : nullptr;
}
// An allocation of the library's kind, for a caller's workspace.
void* fk_device(size_t bytes) { return take(bytes, cudaMemoryTypeDevice); }

int fk_module(const char* kernel) { return module_of.count(kernel) ? module_of[kernel] : -1; }
// Kernels in a module whose names hold `part`.
int fk_module_kernels(int m, const char* part) {
    int n = 0;
    for (auto& k : module_of) n += k.second == m && k.first.find(part) != std::string::npos;
    return n;
}

// ----------------------------------------------------------- registration
void** __cudaRegisterFatBinary(void*) { return (void**)(intptr_t)(8 * ++modules); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void** module, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*,
                            dim3*, int*) {
    kernels[host] = name;
    module_of[name] = (int)((intptr_t)module / 8);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shmem, void* stream) {
    pushed = Config{grid, block, shmem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shmem, void* stream) {
    *grid = pushed.grid;
    *block = pushed.block;
    *shmem = pushed.shmem;
    *(void**)stream = pushed.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* func) {
    *k = (cudaKernel_t)func;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t, cudaStream_t) {
    return launch((const void*)k, grid, block, args, "launch");
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void** args) {
    return launch(func, c->gridDim, c->blockDim, args, "launch");
}

// ----------------------------------------------------------------- runtime
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrL2CacheSize ? 135266304 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
    const cudaError_t e = call("cudaMalloc");
    *p = e == cudaSuccess ? take(bytes, cudaMemoryTypeDevice) : nullptr;
    return e;
}
cudaError_t cudaFree(void* p) {
    call("cudaFree");
    drop(p, cudaMemoryTypeDevice, "cudaFree");
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
    const cudaError_t e = call("cudaHostAlloc");
    *p = e == cudaSuccess ? take(bytes, cudaMemoryTypeHost) : nullptr;
    return e;
}
cudaError_t cudaFreeHost(void* p) {
    call("cudaFreeHost");
    drop(p, cudaMemoryTypeHost, "cudaFreeHost");
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t bytes, cudaMemcpyKind kind, cudaStream_t) {
    const cudaError_t e = call("cudaMemcpyAsync");
    if (e != cudaSuccess) return e;
    const void* dev = kind == cudaMemcpyHostToDevice ? dst : src;
    if (!inside(dev, bytes, cudaMemoryTypeDevice)) {
        complain("cudaMemcpyAsync past the end of an allocation");
        return cudaSuccess;
    }
    memmove(dst, src, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* dst, int v, size_t bytes, cudaStream_t) {
    const cudaError_t e = call("cudaMemsetAsync");
    if (e != cudaSuccess) return e;
    if (!inside(dst, bytes, cudaMemoryTypeDevice)) complain("cudaMemsetAsync past the end of an allocation");
    else memset(dst, v, bytes);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* func, cudaFuncAttribute, int) {
    calls[std::string("attribute ") + (kernels.count(func) ? kernels[func] : "?")]++;
    return call("cudaFuncSetAttribute");
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static void* m = take(1 << 20, cudaMemoryTypeDevice);
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    memset(a, 0, sizeof *a);
    Range* r = find(p);
    a->type = r && r->live ? (cudaMemoryType)r->type : cudaMemoryTypeUnregistered;
    if (r && r->live) a->devicePointer = const_cast<void*>(p);
    if (a->type == cudaMemoryTypeHost) a->hostPointer = const_cast<void*>(p);
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *q = cudaDriverEntryPointSuccess;
    if (!strcmp(name, "cuTensorMapEncodeTiled")) *p = (void*)encode;
    else if (!strcmp(name, "cuCtxGetCurrent")) *p = (void*)ctx_current;
    else if (!strcmp(name, "cuCtxGetId")) *p = (void*)ctx_id;
    else if (!strcmp(name, "cuPointerGetAttribute")) *p = (void*)pointer_attribute;
    else *q = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)16;
    return call("cudaStreamCreateWithFlags");
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return call("cudaStreamSynchronize"); }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return call("cudaStreamBeginCapture"); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)24;
    return call("cudaStreamEndCapture");
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* g, cudaGraph_t, unsigned long long) {
    *g = (cudaGraphExec_t)32;
    return call("cudaGraphInstantiate");
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return call("cudaGraphLaunch"); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)40;
    return call("cudaEventCreate");
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = (cudaEvent_t)40;
    return call("cudaEventCreate");
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return call("cudaEventRecord"); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return call("cudaEventSynchronize"); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}

}  // extern "C"
