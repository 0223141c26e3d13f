// lb_engine.h -- host-side engine shared by the single-lattice ABI
// (lb_api.cu) and the lattice pool (lb_pool.cu): device regions of lattices,
// their TMA descriptors and coefficients, the work partition and launch of
// the persistent step kernel, and the observe/initialise helpers.
#pragma once

#include <vector>

#include "lb_internal.h"

namespace lbgb {

// Host-side state of one resident lattice.
struct Lattice {
    lb_params p;
    Geom g;
    char* region;            // device region: stats | observe slots | wall columns | wall sums |
                             // buffer 0 | buffer 1
    DevStats* st;
    double* slots;           // observe partial sums, 4 per tile
    char* wallx;             // two steps' wall-momentum pairs: [2][2][nx] (bottom, top), compute type
    double* wsum;            // their sums per strip and over the sampled steps: [2][nstrips]
    char* fbuf[2];
    size_t fbytes;
    CUtensorMap tblock[2];   // step kernel: 8-row block loads of buffer b
    CUtensorMap ttile[2];    // step kernel: tile stores into buffer b, clipped at the lattice edge
    CUtensorMap tobs[2];     // observe kernel: tile + halo loads of buffer b
    Coef<double> kd;
    Coef<float> kf;
    int nstrips, ntiles_y, seg;
    int cur, pull;           // host mirror of DevStats::cur, and of pull != 0
    bool mom;                // host mirror of DevStats::pull == 2: held by its moments
    bool inited;
    long long t;             // host mirror of the step count
    unsigned int err_latched;
};

// One launch of the persistent step kernel over a set of lattices.
struct Launch {
    int precision;
    int variant;             // bit 0: all periodic; bit 1: general forcing; bit 2: 1 - omega = 0
    int shape;               // tile shape (Shape)
    dim3 grid;
    int nitems, seg;
    BatchArgs<double> ad;
    BatchArgs<float> af;
};

size_t align_up(size_t v, size_t a);
lb_status validate_params(const lb_params* p);
lb_status cuda_status(cudaError_t e);
int device_sms(int device);

// Bytes of a lattice's device region, and binding a lattice to one.
size_t lattice_bytes(const lb_params* p);
lb_status lattice_setup(Lattice& L, const lb_params* p, char* region);

// Host-only plan of one launch's work items (the lb_plan_partition entry).
lb_status plan_partition(const lb_params* ps, int nlat, int seg, int tile_rows, int sms,
                         int32_t* items, int32_t* nitems, int32_t* cta, int32_t* grid,
                         int32_t* seg_used);

// Segment length (tiles per work item) minimising the most loaded CTA.
int choose_seg(const int* nstrips, const int* ntiles_y, int nlat, int G);

// Tile rows of a lattice in a shape; whether its steps may take the moment
// kernel; the library's default shape for a set of lattices with tiles8 8-row
// tiles in all; and the shape for a requested tile height (0: the default;
// 8 or 16: a population kernel; result 0: the precision has no such tile).
int tiles_y(const Lattice& L, int shape);
bool moments_ok(const Lattice& L);
int default_shape(int precision, bool moments, long long tiles8, int sms);
int shape_of_rows(int precision, bool moments, int rows, long long tiles8, int sms);

// Pinned host buffers for tables on their way to the device: a few, used in
// turn, so that a launch can be built while the device still works on the
// steps before it.  A buffer is handed out again once its copies are done.
// Allocating and freeing pinned memory may wait for the device: reserve() takes
// them where a set is put together, larger ones at least double the size, and all
// are freed together at the end (the first run of a fresh pool: 90 us with
// pageable tables, 240 with buffers allocated in it).
class HostStage {
public:
    ~HostStage();
    // room for `bytes` in every buffer
    cudaError_t reserve(size_t bytes);
    // `bytes` of pinned memory (128-byte aligned), or null
    char* get(size_t bytes);
    // the copies out of the last buffer handed out are enqueued on s
    cudaError_t sent(cudaStream_t s);

private:
    static constexpr int kBuffers = 4;
    struct Buffer {
        char* mem = nullptr;
        cudaEvent_t done = nullptr;
        bool busy = false;
    } buf_[kBuffers];
    size_t cap_ = 0;              // bytes of a buffer
    std::vector<char*> blocks_;   // each allocation: kBuffers buffers
    int last_ = 0;
};

// Write the lattices' descriptors to `descs` (device, 128-byte aligned, room
// for nlat LatDesc<double>) and the item tables to `slots`, and fill the
// launch.  With a stage the copies are only enqueued; without one they go
// through pageable memory and the stream is synchronised.  All lattices share the precision
// and the coefficients of lats[0] (couplings, tau, forcing).  seg > 0 forces
// the segment length; seg = 0 takes choose_seg's; seg < 0 cuts the tiles
// into one contiguous run per CTA.  `slots` holds `room` doubles for the item
// tables, launch_area_doubles of the lattices' total 8-row tiles and strips;
// LB_ERR_NOMEM where they do not fit.
lb_status launch_build(Launch& Ln, Lattice* const* lats, int nlat, void* descs, double* slots,
                       size_t room, unsigned int* ticket, int sms, cudaStream_t stream, HostStage* stage,
                       int seg = 0, int shape = SHAPE_8);
size_t launch_area_doubles(int precision, size_t tiles, size_t strips, int sms);
// Enqueue step step_k of a window of consecutive steps (0-based); advance: the
// window's steps on its last launch, else 0.  The device's step counters move
// with the window's last launch only.
lb_status launch_run(Launch& Ln, int step_k, int advance, cudaStream_t s);
// Enqueue n steps as one window (n < 2^30).  *broken: a launch failed with
// earlier ones of the window enqueued, which no launch's counters follow.
lb_status launch_window(Launch& Ln, int n, cudaStream_t s, bool* broken);

lb_status lattice_init_seeded(Lattice& L, uint64_t seed, cudaStream_t s);
lb_status lattice_init_fields(Lattice& L, const double* rho_A, const double* rho_B,
                              const double* ux, const double* uy, cudaStream_t s);
// Resume from populations [2][9][ny][nx] (host FP64, as lattice_populations
// writes them) at step t; stress averages restart.
// pulled = 1: f holds the stored post-collision state f*(t-1) (a raw
// checkpoint); 0: the populations f(t) before collision.
lb_status lattice_load_populations(Lattice& L, const double* f, long long t, int pulled,
                                   cudaStream_t s);
// n steps of a launch with tile shape `shape` were enqueued.
void lattice_advanced(Lattice& L, long long n, int shape);
// Make a state that is held by its moments a population state (f*).
lb_status lattice_to_populations(Lattice& L, cudaStream_t s);
// dst: the outputs of the kind (see StepArgs::obs_dst), or null.
lb_status lattice_observe(Lattice& L, int obs, double* const dst[4], int q0, int q1, cudaStream_t s);
lb_status lattice_fields(Lattice& L, double* rho_A, double* rho_B, double* ux, double* uy,
                         cudaStream_t s);
// raw = 0: f(t) after streaming; raw = 1: the stored state as it is (f*(t-1)
// when L.pull, else f(t)), for an exact checkpoint.
lb_status lattice_populations(Lattice& L, double* f, cudaStream_t s, int raw = 0);
lb_status lattice_stress(Lattice& L, lb_stress_out* out, cudaStream_t s);
lb_status lattice_read_stats(Lattice& L, DevStats* out, cudaStream_t s);

}  // namespace lbgb
