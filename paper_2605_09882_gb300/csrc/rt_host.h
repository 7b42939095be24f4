// Host-side helpers shared by the library's translation units.
#pragma once

#include <string.h>

#include <algorithm>

#include "rt_internal.h"

namespace rt {
int set_error(int code, const char* msg);
int cuda_error(const char* where);
void clear_error();
// current launch shape (threads per block, blocks per SM cap, groups per pop)
void launch_shape(int* block, int* blocks_per_sm, int* groups_per_pop);
// device direction table of nside on device dev (uploaded on first use)
const DirConst* direction_table(int dev, int nside, int* status);
int sm_count_of(int dev);
// spreads a call of few rays over the warps of its launch (groups per pop, rays
// per group)
void spread_rays(TraceArgs& a, long long warps);
// deepest coarse-table level rt_build_octree may choose (-1: no cap)
int table_level_cap();
// enqueues the density check (RT_ERR_NONFINITE into st for a NaN, infinite or
// negative value; leaf index base + i / S as the fault position)
int check_densities(const void* dens, long long n_leaves, int S, int f64, long long base, DevStats* st,
                    cudaStream_t s);
// rt_trace_columns with the density check optional (the host-buffer call
// checks the whole array once, not per source chunk)
int trace_columns_impl(const rt_octree* t, const double* d_src, int64_t n_src, int nside, const void* d_dens,
                       int n_species, int dens_dtype, int mode, void* d_out, void* stream, bool check);
// argument checks and TraceArgs of the single-octree trace entry points
int prepare_trace(const rt_octree* t, const double* d_src, int64_t n_src, int nside, int S, int mode,
                  TraceArgs& a, const char* who);
// shared-offset trace of a cube (rt_beam.cu): the tables it keeps (bytes; 0: the
// shape does not admit it), the memory of one call (p null: the form did not
// run; given back to the pool, in the order of s, when destroyed) and its launch,
// with the density check if asked.
// kBeamVotes: sources of 32 at the commonest offset below which a form that may leave out a
// sixteenth is not tried.  With a sixteenth elsewhere at random, fewer than 24
// agree once in 9,000 calls (and the walk then does what the form would have);
// with half elsewhere, more than 23 once in 280.
constexpr int kBeamVotes = 24;
size_t beam_bytes(const rt_octree* t, int64_t n_src, int nd, int S, int mode);
struct BeamCall {
    void* p = nullptr;
    cudaStream_t s = nullptr;
    ~BeamCall();
};
int launch_beam(rt_octree* t, TraceArgs& a, int mode, bool epilogue, bool check, cudaStream_t s, BeamCall& call);
// a user of the pool that memory comes from (a handle, the host call's buffers)
// comes and goes
bool beam_pool_join(int dev);
void beam_pool_leave(int dev);
// leaf-gather adjoint (rt_beam.cu): whether the call's shape admits it, and
// its launch (source check, step tables, gather) on stream s
bool gather_applies(const rt_octree* t, const TraceArgs& a);
int launch_adjoint_gather(rt_octree* t, const TraceArgs& a, int mode, cudaStream_t s);
}  // namespace rt
