// Host-side simulation handle shared by the C-ABI translation units.
#pragma once

#include <cuda_runtime.h>

#include <string>

#include "../../include/pic.h"
#include "sff_common.cuh"
#include "sff_kernels.h"

using sff::Group;
using sff::SimDev;
using sff::Work;

// bump allocator over one device allocation (256-byte aligned pieces)
struct Arena {
    char* base = nullptr;
    size_t size = 0, used = 0;
    void* take(size_t bytes)
    {
        size_t off = (used + 255) & ~size_t(255);
        if (off + bytes > size) return nullptr;
        used = off + bytes;
        return base + off;
    }
};

struct GraphBundle {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

struct pic_sim {
    pic_config cfg;
    pic_params prm;
    int device = 0;
    int es = 4;                  // element size
    SimDev h;                    // host copy of the descriptor
    SimDev* d = nullptr;         // device descriptor
    pic_allocator alloc{};
    bool use_cuda_malloc = true;
    Arena arena;
    // single-simulation launch group
    Group grp{};
    Work* d_ywork = nullptr;
    int nywork = 0;              // field-solver work items (yee_tile_active)
    int* d_gprefix = nullptr;    // chunk numbering of the single-simulation group
    int* d_counters = nullptr;
    double* d_acc = nullptr;     // 8 doubles
    unsigned long long* d_bits = nullptr;
    GraphBundle step_graph;
    GraphBundle many_graph;      // MANY_STEPS steps (captured when a call first asks for a few times that)
    bool many_failed = false;    // ... could not be
    // id of the launch group whose chunk numbering and work counters are set for this sim's
    // current particle layout (each step ends by setting them for its own group; any other
    // change of the layout clears it, and the next step of a group starts with k_prefix)
    long long prefix_group = 0;
    long long own_group_id = 0;  // id of the single-simulation group
    GraphBundle sort_graph;      // the step whose re-sort orders the tiles by cell
    int sort_every = 0;          // steps between cell sorts (0: none)
    int since_sort = 0;          // steps through pic_step / pic_profile_step since the last one
    cudaStream_t cap_stream = nullptr;
    cudaStream_t cap_stream2 = nullptr;   // the field-solve branch of the captured step
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::string err;
    long long nalloc_tot = 0;    // na_x*na_y*na_z
    size_t stage_bytes = 0;      // staging memory of the state's conversions (h.scratch)
    long long pcap = 0;          // particle capacity (the buffer sets hold h.cap slots)
};


// Particles per push work item when the configuration leaves it open, for n particles: about four
// items for every block that the GPU holds at once (152 SMs; blocks per SM by registers and, in FP32,
// shared memory; 3D FP64 counts two, of which its box lets one run at a time), a multiple of a block's round (256; FP64 128), at most ITEM_MAX.  With fewer items than
// that the last ones of a launch leave most SMs idle, below that the per-item set-up (the box load,
// the clearing and the flush of the current) shows.  Push at the focus, items of 256 / 512 / 1024 /
// 2048: 2D 14 k electrons 0.018 / 0.025 / 0.028 / 0.034 ms, 2D FP64 131 k 0.34 / 0.36 / 0.40 /
// 0.65 ms, 3D 89 k 0.039 / 0.040 / 0.048 / - ms, 2D 2.1 M - / 0.127 / 0.124 / 0.146 ms, 3D 2.0 M
// - / 0.368 / 0.337 / 0.327 ms, 2D 4.5 M - / 0.204 / 0.181 / 0.180 ms.
constexpr int ITEM_MAX = 2048;
int default_item(long long n, int dim, bool fp64);
// ... and with the configuration's limit.  An FP64 item never gets larger than the default: one that
// spans a dense tile leaves its block's four warps the last at work (1D plane wave at step 1800,
// 32 768 electrons in tiles of 16 cells, limit 2048: step 0.0472 -> 0.0276 ms).
int work_item(const pic_config* c, long long n);

// a fresh launch-group id (never 0; never reused in the process)
long long new_group_id();

// drop cached batch graphs that contain `s` (called by pic_destroy)
void batch_forget(pic_sim* s);
