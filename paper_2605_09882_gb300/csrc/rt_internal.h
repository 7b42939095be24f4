// Internal types of the tracer library (host and device).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/rt_api.h"

namespace rt {

constexpr int kDepth = 21;          // anchor depth of the Morton lattice
constexpr int kMaxSpecies = 8;
constexpr int kBaseTableLevel = 7;  // coarse table level for every tree (8^7 = 2M entries at most)
constexpr int kMaxTableLevel = 10;  // deepest coarse table (the lookup's cell index holds 30 bits)
// Coarse-table entries: the first leaf and a code for what is there: log2 of the
// leaf's size for a cell inside one leaf, kCellLeaves more than that for a cell
// whose leaves all have one finer level, or one of the two codes after it.
// An octree of fewer than 2^26 leaves packs them into 32 bits, leaf << 6 | code:
// at level 8 the table then takes 67 MB, beside the leaves' densities in a 129
// MB L2, and not 134.  A larger one keeps the leaf in the low half of 64 bits and
// the code in the high half.
constexpr uint32_t kCellLeaves = 32;
constexpr uint32_t kCellMixed = 62;  // leaves of several levels
constexpr uint32_t kCellHole = 63;   // outside the domain box
constexpr int64_t kNarrowLeaves = 1ll << 26;
constexpr uint64_t table_entry(uint64_t first, uint32_t code) { return first | (uint64_t)code << 32; }

// Device view of an octree handle.
struct DevTree {
    const uint64_t* keys;
    const uint8_t* levels;
    const void* table;       // [8^T] entries, uint32 or (wide) uint64
    int64_t n;
    uint32_t ext[3];
    int T;                   // coarse table level
    int wide;                // 64-bit table entries
    int uniform_level;       // >= 0: full cube of leaves all at this level (O(1) index)
    int lmax;
    int64_t step_cap;
};

// Per-direction constants, computed on the host from the HEALPix table.
struct DirConst {
    double m[3];
    double inv[3];   // 1 / m_b (0 where m_b == 0)
    float m32[3];    // m_b rounded to float
    float ih[3];     // inv_b = ih + il (float-float split)
    float il[3];
    int flags;       // bit b: m_b != 0; bit 3+b: m_b > 0; bits 6,7,8: |inv| equal for (0,1),(0,2),(1,2)
    int pad;
};

// Statistics block in device memory (one per octree handle).
struct DevStats {
    unsigned long long queue;      // work-queue counter (reset before every launch)
    unsigned long long rays;
    unsigned long long segments;
    unsigned long long exit_fb;
    unsigned long long lookup_fb;
    int status;
    int gather_off;                // nonzero when the shared-offset form (columns, epilogue, adjoint) did not apply
    long long fault_ray;
    int gathered;                  // set when a leaf-gather adjoint ran
    int pad;
};

struct TraceArgs {
    DevTree t;
    const DirConst* dirs;
    int nd;
    const double* src;
    int64_t n_src;
    int64_t n_src_pad;       // n_src rounded up to a multiple of 32
    const void* dens;        // forward: densities; adjoint: unused
    int dens_f64;
    int S;
    void* out;               // forward: columns; adjoint: grad_dens (double)
    const void* gin;         // adjoint: d_grad_out
    uint32_t* nseg;          // path fingerprints (optional)
    uint64_t* hash;
    DevStats* st;
    int batch;               // ray groups per queue pop
    int gw;                  // rays a group: 32, or fewer to spread a call of few rays over the warps
    int layout;              // ray order: 0 direction-major (sources padded to 32), 1 source-major
    int dgroup;              // layout 0: directions per group (a divisor of nd; <= 1: one)
    int pair;                // forward on a uniform cube: two rays per lane (k_trace_pair; n_src_pad % 64 == 0)
    // path recording (KIND 3): per 32-ray group, segment k of lane i is entry
    // rec_off[g] + 32 k + i of rec_leaf / rec_ds
    const long long* rec_off;
    uint32_t* rec_leaf;
    void* rec_ds;
    // fused epilogue (KIND 4): combined column N = sum_k epi_w[k] I_k per ray
    int epi_kind;
    double epi_w[kMaxSpecies];
    double epi_a, epi_gamma;
    const double* epi_coef;
    // runs only if *gate is nonzero (the shared-offset form launched before it
    // did not apply to this call); NULL: always runs
    const int* gate;
    // forward and epilogue: the sources the shared-offset form left out, walked
    // when *gate is zero (NULL: none)
    const uint32_t* rest;
    const unsigned int* n_rest;
};

// Ray order of a trace: direction-major (32 neighbouring sources share a
// direction in a warp) unless there are too few sources to fill a warp, then
// source-major (a warp walks 32 directions of the same source).
inline int ray_layout(int64_t n_src) { return n_src < 32 ? 1 : 0; }

// Launch helpers (defined in the .cu files).
cudaError_t launch_forward(const TraceArgs& a, int mode, int block, int grid, cudaStream_t s);
cudaError_t launch_paths(const TraceArgs& a, int mode, int block, int grid, cudaStream_t s);
cudaError_t launch_adjoint(const TraceArgs& a, int mode, int block, int grid, cudaStream_t s);
cudaError_t launch_epilogue(const TraceArgs& a, int mode, int block, int grid, cudaStream_t s);
int occupancy_epi(int mode, int S, bool uniform, int block);
int occupancy_fwd(int kind, int mode, int S, bool uniform, int block);
int occupancy_pair(int S, int block);
int occupancy_adj(int mode, int S, bool uniform, int block);

}  // namespace rt

// Host-side octree handle.
struct rt_octree {
    rt::DevTree dev;
    rt::DevStats* st;        // device
    void* table;             // device, owned
    int device;
    int uniform_allowed;     // 0: use the coarse table even for a uniform grid
    int64_t default_cap;
    void* adj_tab;           // device, owned: step tables of the leaf-gather adjoint (grown on demand)
    size_t adj_tab_bytes;
    void* fwd_tab;           // device: step tables of the shared-offset trace
    size_t fwd_tab_bytes;
    int fwd_pool;            // a user of its pool
    int fwd_tab_lent;        // fwd_tab belongs to the caller that built the handle
    unsigned long long gen;  // build number, unique in the process (a reused address is another tree)
};
