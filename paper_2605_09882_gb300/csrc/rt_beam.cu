// Columns and adjoint on a cube whose sources share one offset: a full cube of
// equal-level leaves, sources in consecutive leaves (source s in leaf j0 + s),
// all at the same offset inside their leaf (every run of leaf centres is one).
// The slab exits of the definition, t_b = (F_b - Q_b) / m_b, then depend only on
// F_b - Q_b, which is the same list of distances for every source, so along
// direction q every ray takes the same exit-axis sets E_i and the same segment
// lengths ds_i in the same order; only the step at which it leaves the cube
// depends on the source.  The ray from source s visits leaf s + o_i at step i
// (o_i the summed steps), so with the steps in a table
//   I[s,q,k]  = sum_i [s + o_qi in the cube] n[s + o_qi, k] ds_qi,
//   grad[j,k] = sum_q sum_i [j - o_qi in the cube] g[j - o_qi, q, k] ds_qi:
// two sums of shifted copies of a field, computed by the same kernel
// (k_beam), without a walk, without atomics, the same bits on every run.
//
// The tables come from the walk itself, run once per direction from the corner
// the direction starts from (the longest path), so every ds is bitwise the one
// the walk uses, and the columns add the same products in the same order with
// the same operations: they are bit for bit those of the walk.  A device check
// lists the sources that are elsewhere in their leaf (a centre rounded in its
// last place, say); the walk launched after this form traces those, or every
// source if there are many.
//
// Layout: the field (densities, or one direction's slice of the column
// gradient) is first copied from Morton order into rows along an axis, so that
// the 32 lanes of a warp, which take 32 neighbouring leaves of one row, read
// one contiguous run at every step.
//
// Tables per direction.  The dominant axis of the direction is its run axis;
// the steps are cut into runs: consecutive steps along the run axis alone, at
// most kRun of them.  A run holds the row-layout offset of its first cell, the
// run-axis cells passed before it, and its segment lengths.  For every axis b
// and every r, P_b[r] is the first step that is more than r cells from the
// start on b, and C_b[r] the same in runs for the two other axes.
#include <mutex>

#include "rt_host.h"
#include "rt_kernels.cuh"

namespace rt {

// 10-bit coordinate of axis 0 of a 30-bit Morton index (inverse of spread10).
__device__ __forceinline__ uint32_t compact10(uint32_t v)
{
    v &= 0x09249249u;
    v = (v | (v >> 2)) & 0x030c30c3u;
    v = (v | (v >> 4)) & 0x0300f00fu;
    v = (v | (v >> 8)) & 0x030000ffu;
    v = (v | (v >> 16)) & 0x3ffu;
    return v;
}

constexpr int kRun = 4;  // steps of a run at most

// A run of k steps along the run axis.
template <class T>
struct alignas(16) BeamRun {
    int off;      // row-layout offset of its first cell from the source's leaf
    int at;       // cells passed along the run axis before it
    int k;        // its steps
    int pad;
    T ds[kRun];   // their lengths
};

// A direction's axes: run (dominant), lane (the fastest of the row layout) and
// the third.  Rows lie along x, except for directions that run along x.
struct BeamAxes {
    int run, lane, third;
};

__device__ __forceinline__ BeamAxes beam_axes(const DirConst* __restrict__ d)
{
    const double x = fabs(__ldg(&d->m[0])), y = fabs(__ldg(&d->m[1])), z = fabs(__ldg(&d->m[2]));
    BeamAxes a;
    if (x > y && x > z) { a.run = 0; a.lane = 1; a.third = 2; }
    else if (y > z) { a.run = 1; a.lane = 0; a.third = 2; }
    else { a.run = 2; a.lane = 0; a.third = 1; }
    return a;
}

// Row-layout stride of axis b when rows lie along axis `lane` (0 or 1).
__device__ __forceinline__ int beam_stride(int b, int lane, int L)
{
    return b == lane ? 1 : (b == 2 ? 1 << (2 * L) : 1 << L);
}

// Per-direction tables, one row of each per direction.
struct BeamTables {
    int4* info;      // [nd] runs, steps
    void* run;       // [nd][lcap] BeamRun<float or double>
    int* fb;         // [nd][lcap] exit fall-backs up to and including step i
    int* P;          // [nd][3][pcap] first step beyond r cells on axis b
    int* C;          // [nd][3][pcap] first run beyond r cells on axis b (not the run axis)
    int* D;          // [nd][lcap] row-layout offset of step i's cell from the source's leaf (NULL: not kept)
    void* ds;        // [nd][lcap] length of step i (float or double)
    int lcap, pcap;
};

// Visitor that writes a direction's tables while the walk runs.  Leaf indices
// are level-L Morton indices; an axis stepped when its bits of the index
// changed.  dstep[b] is the row-layout index change of one cell along the ray
// on axis b.
template <class T>
struct RunTable {
    BeamRun<T>* run;
    int *fb, *P, *C, *D;
    T* ds;
    const WalkCounters* wc;
    int n, nr, k, cap, pcap, raxis;
    uint32_t prev;
    int cnt[3], dstep[3], off;
    __device__ __forceinline__ void pre(uint32_t j)
    {
        bool cut = n == 0 || k == kRun;
        if (n > 0) {
#pragma unroll
            for (int b = 0; b < 3; b++)
                if (b != raxis && ((prev ^ j) & (kDilX << b))) cut = true;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                if ((prev ^ j) & (kDilX << b)) {
                    if (cnt[b] < pcap) {
                        P[b * pcap + cnt[b]] = n;
                        C[b * pcap + cnt[b]] = nr;  // the run about to start, if b is not the run axis
                    }
                    cnt[b]++;
                    off += dstep[b];
                }
            }
        }
        if (cut) {
            if (nr < cap) {
                run[nr].off = off;
                run[nr].at = raxis == 0 ? cnt[0] : (raxis == 1 ? cnt[1] : cnt[2]);
            }
            nr++;
            k = 0;
        }
        prev = j;
    }
    template <class F>
    __device__ __forceinline__ void acc(F d)
    {
        if (nr <= cap) {
            run[nr - 1].ds[k] = (T)d;
            run[nr - 1].k = k + 1;
        }
        if (n < cap) {
            fb[n] = (int)wc->exit_fb;
            if (D) {
                D[n] = off;
                ds[n] = (T)d;
            }
        }
        k++;
        n++;
    }
    template <class F>
    __device__ __forceinline__ void seg(uint32_t j, F d) { pre(j); acc(d); }
};

// The offset most sources share, and the leaf source 0 would lie in with it.
struct BeamRef {
    long long f[3];      // offset inside the leaf (2^-53 lattice)
    long long j0;        // level-L Morton index of source 0's leaf
    unsigned int n_rest; // sources left out
    unsigned int key;    // level, mode and directions of the tables
    unsigned int done;   // directions whose tables are written
    unsigned int stale;  // the tables are to be written
    unsigned int pad[4];
};

// One warp: the most common offset (and leaf minus index) among 32 sources
// spread over the list, and the reset of the check's results and of the queues.
// Fewer than `need` of the 32 at that offset settle it: st->gather_off is set
// and nothing more is prepared for a form that cannot apply (scattered points).
// The tables
// depend on the level, the mode, the directions and the offset alone: those of
// an earlier call on this scratch with the same values stand (a walk of a few
// hundred steps by one thread a direction: 26 us at 32^3, 48 us at 128^3, which
// a trace in source chunks would pay for each chunk).
__global__ void k_beam_ref(const double* __restrict__ src, long long n, int L, unsigned int key, int nd, int need,
                           BeamRef* ref, unsigned long long* queue, int queues, DevStats* st)
{
    const int lane = threadIdx.x;
    const long long s = (n - 1) * lane / 31;
    const int sh = kDepth - L;
    long long f[3];
    uint32_t j = 0;
#pragma unroll
    for (int b = 0; b < 3; b++) {
        long long q = 0;
        fixed_source(__ldg(src + 3 * s + b), q);
        f[b] = q & ((1ll << (sh + 32)) - 1);
        j |= spread10((uint32_t)(q >> (sh + 32))) << b;
    }
    const long long j0 = (long long)j - s;
    int votes = 0;
    for (int o = 0; o < 32; o++) {
        // every lane takes part in every exchange: no short circuit
        const long long a = __shfl_sync(RT_FULL, f[0], o), b = __shfl_sync(RT_FULL, f[1], o);
        const long long c = __shfl_sync(RT_FULL, f[2], o), d = __shfl_sync(RT_FULL, j0, o);
        votes += (a == f[0]) & (b == f[1]) & (c == f[2]) & (d == j0);
    }
    const int most = __reduce_max_sync(RT_FULL, votes);
    const unsigned who = __ballot_sync(RT_FULL, votes == most);
    for (int i = lane; i < queues; i += 32) queue[i] = 0ull;
    if (lane == __ffs(who) - 1) {
        st->queue = 0ull;  // the walk's, launched after this form
        if (ref->key != key || ref->done != (unsigned int)nd || ref->f[0] != f[0] || ref->f[1] != f[1] || ref->f[2] != f[2]) {
            ref->key = key;
            ref->done = 0u;
            ref->stale = 1u;
#pragma unroll
            for (int b = 0; b < 3; b++) ref->f[b] = f[b];
        } else {
            ref->stale = 0u;
        }
        ref->j0 = j0;
        ref->n_rest = 0u;
        st->gather_off = (votes < need || j0 < 0 || j0 + n > (1ll << (3 * L))) ? 1 : 0;
    }
}

// Blocks 0 .. nd - 1: direction q's tables, by one thread that walks the ray
// from the corner leaf the direction starts from, at the shared offset.
// False, with st->gather_off set, if the walk did not end as every walk does.
template <int MODE>
__device__ __forceinline__ bool beam_table(const DevTree& t, const DirConst* __restrict__ dirs, int q,
                                           const BeamRef* __restrict__ ref, const BeamTables& tab, DevStats* st)
{
    using T = typename std::conditional<MODE == RT_MODE_FP64, double, float>::type;
    const int L = t.uniform_level;
    const int sh = kDepth - L;
    const int N = 1 << L;
    const int flags = __ldg(&dirs[q].flags);
    const BeamAxes ax = beam_axes(dirs + q);
    double x[3];
    WalkCounters wc = {0u, 0u, 0u};
    RunTable<T> rec;
    rec.run = (BeamRun<T>*)tab.run + (size_t)q * tab.lcap;
    rec.fb = tab.fb + (size_t)q * tab.lcap;
    rec.P = tab.P + (size_t)q * 3 * tab.pcap;
    rec.C = tab.C + (size_t)q * 3 * tab.pcap;
    rec.D = tab.D ? tab.D + (size_t)q * tab.lcap : nullptr;
    rec.ds = (T*)tab.ds + (size_t)q * tab.lcap;
    rec.wc = &wc;
    rec.n = rec.nr = rec.k = 0;
    rec.cap = tab.lcap;
    rec.pcap = tab.pcap;
    rec.raxis = ax.run;
    rec.prev = 0u;
    rec.off = 0;
#pragma unroll
    for (int b = 0; b < 3; b++) {
        const bool moving = flags & (1 << b), up = (flags >> (3 + b)) & 1;
        const long long cell = (moving && !up) ? N - 1 : 0;
        x[b] = __dmul_rn(__ll2double_rn((cell << (sh + 32)) | ref->f[b]), 0x1p-53);  // exact
        const int stride = beam_stride(b, ax.lane, L);
        rec.dstep[b] = up ? stride : -stride;
        rec.cnt[b] = 0;
    }
    const int status = walk<MODE, true>(t, dirs + q, x, t.step_cap, rec, wc);
    const bool ok = status == RT_OK && rec.n <= tab.lcap;
    if (!ok) atomicOr(&st->gather_off, 2);
    const int n = min(rec.n, tab.lcap), nr = min(rec.nr, tab.lcap);
    tab.info[q] = make_int4(nr, n, 0, 0);
    // steps an axis never reaches within the walk end every range at its end
#pragma unroll
    for (int b = 0; b < 3; b++)
        for (int r = min(rec.cnt[b], tab.pcap); r < tab.pcap; r++) {
            rec.P[b * tab.pcap + r] = n;
            rec.C[b * tab.pcap + r] = nr;
        }
    return ok;
}

// Tables (the first nd blocks, one thread each) and source check (the other
// blocks, 32 sources a warp): source s belongs in leaf j0 + s at the shared
// offset.  Those that are not there are marked in `out` and listed in `rest`;
// more than `most` of them set st->gather_off.
template <int MODE>
__global__ void __launch_bounds__(256) k_beam_setup(const DevTree t, const DirConst* __restrict__ dirs, int nd,
                                                    const double* __restrict__ src, long long n, BeamRef* ref,
                                                    BeamTables tab, uint32_t* out, uint32_t* rest, unsigned int most,
                                                    DevStats* st)
{
    if (*(volatile int*)&st->gather_off) return;
    if (blockIdx.x < nd) {
        if (threadIdx.x == 0 && ref->stale && beam_table<MODE>(t, dirs, blockIdx.x, ref, tab, st))
            atomicAdd(&ref->done, 1u);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int L = t.uniform_level;
    const int sh = kDepth - L;
    const long long fmask = (1ll << (sh + 32)) - 1;
    const long long j0 = ref->j0;
    const long long f0[3] = {ref->f[0], ref->f[1], ref->f[2]};
    const long long warps = (long long)(gridDim.x - nd) * (blockDim.x >> 5);
    for (long long base = (((blockIdx.x - nd) * (long long)blockDim.x + threadIdx.x) >> 5) * 32; base < n;
         base += warps * 32) {
        const int off = *(volatile int*)&st->gather_off;
        if (__any_sync(RT_FULL, off != 0)) return;  // already decided
        const long long s = base + lane;
        bool bad = false;
        if (s < n) {
#pragma unroll
            for (int b = 0; b < 3; b++) {
                long long q;
                if (!fixed_source(__ldg(src + 3 * s + b), q)) {
                    bad = true;
                } else {
                    const uint32_t cell = compact10((uint32_t)(j0 + s) >> b);
                    bad |= (q >> (sh + 32)) != (long long)cell || (q & fmask) != f0[b];
                }
            }
        }
        const unsigned bads = __ballot_sync(RT_FULL, bad);
        if (lane == 0) out[base >> 5] = bads;
        if (bads) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&ref->n_rest, (unsigned)__popc(bads));
            at = __shfl_sync(RT_FULL, at, 0);
            if (at + __popc(bads) > most) {
                if (lane == 0) atomicOr(&st->gather_off, 1);
                return;
            }
            if (bad) rest[at + __popc(bads & ((1u << lane) - 1u))] = (uint32_t)s;
        }
    }
}

// Stores SM values, as vectors.
template <class T, int SM>
__device__ __forceinline__ void store_row(T* __restrict__ dst, const T v[SM])
{
    if (sizeof(T) == 4 && SM % 4 == 0) {
#pragma unroll
        for (int h = 0; h < SM / 4; h++)
            ((float4*)dst)[h] = make_float4((float)v[4 * h], (float)v[4 * h + 1], (float)v[4 * h + 2], (float)v[4 * h + 3]);
    } else if (sizeof(T) == 4 && SM == 2) {
        *(float2*)dst = make_float2((float)v[0], (float)v[1]);
    } else if (sizeof(T) == 8 && SM % 2 == 0) {
#pragma unroll
        for (int h = 0; h < SM / 2; h++) ((double2*)dst)[h] = make_double2((double)v[2 * h], (double)v[2 * h + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < SM; k++) dst[k] = v[k];
    }
}

// Loads SM values, as vectors.
template <class T, int SM>
__device__ __forceinline__ void load_row(const T* __restrict__ p, T v[SM])
{
    if (sizeof(T) == 4 && SM % 4 == 0) {
#pragma unroll
        for (int h = 0; h < SM / 4; h++) {
            const float4 w = __ldg((const float4*)p + h);
            v[4 * h] = (T)w.x; v[4 * h + 1] = (T)w.y; v[4 * h + 2] = (T)w.z; v[4 * h + 3] = (T)w.w;
        }
    } else if (sizeof(T) == 4 && SM == 2) {
        const float2 w = __ldg((const float2*)p);
        v[0] = (T)w.x; v[1] = (T)w.y;
    } else if (sizeof(T) == 8 && SM % 2 == 0) {
#pragma unroll
        for (int h = 0; h < SM / 2; h++) {
            const double2 w = __ldg((const double2*)p + h);
            v[2 * h] = (T)w.x; v[2 * h + 1] = (T)w.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < SM; k++) v[k] = __ldg(p + k);
    }
}

// Leaf (Morton index) of row-layout index i, rows along `lane` (0: x, 1: y).
__device__ __forceinline__ uint32_t row_leaf(unsigned long long i, int L, int lane)
{
    const uint32_t M = (1u << L) - 1u;
    const uint32_t u = (uint32_t)i & M, v = (uint32_t)(i >> L) & M, z = (uint32_t)(i >> (2 * L));
    const uint32_t x = lane ? v : u, y = lane ? u : v;
    return spread10(x) | (spread10(y) << 1) | (spread10(z) << 2);
}

// The densities of leaf j, SM values (zeros past S), in the type the columns are
// summed in (the conversion the walk makes on each load); with check, checked as
// k_check_dens does.
template <class T, int SM>
__device__ __forceinline__ void beam_dens(const void* __restrict__ dens, int f64, int S, uint32_t j, T v[SM], bool check,
                                          DevStats* st)
{
    if (S == SM && !f64) load_dens<SM, T>(dens, 0, SM, j, v);
    else load_dens<SM, T>(dens, f64, S, j, v);
    if (!check) return;
    bool bad = false;
    if (f64) {
        for (int k = 0; k < S; k++) {
            const double w = __ldg((const double*)dens + (size_t)j * S + k);
            bad |= !(w >= 0.0 && w <= 1.7976931348623157e308);
        }
    } else {
#pragma unroll
        for (int k = 0; k < SM; k++) bad |= !(v[k] >= (T)0 && v[k] <= (T)3.402823466e38f);
    }
    if (bad) report_fault(st, RT_ERR_NONFINITE, (long long)j);
}

// The densities in row layout along x, then along y.  The check runs whether or
// not the sources have the shared offset.
template <class T, int SM>
__global__ void k_beam_dens(const void* __restrict__ dens, int f64, int S, int L, T* __restrict__ along_x,
                            T* __restrict__ along_y, int check, DevStats* st)
{
    const bool off = *(volatile const int*)&st->gather_off != 0;
    const unsigned long long n = 1ull << (3 * L), end = off ? (check ? n : 0ull) : 2ull * n;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < end;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const bool y = i >= n;
        const unsigned long long r = y ? i - n : i;
        T v[SM];
        beam_dens<T, SM>(dens, f64, S, off ? (uint32_t)r : row_leaf(r, L, y), v, check && !y, st);
        if (!off) store_row<T, SM>((y ? along_y : along_x) + (size_t)r * SM, v);
    }
}

// Direction q's slice of the column gradient in the row layout of the
// direction: gl[i][k] = g[(leaf(i) nd + q) SM + k].
template <class T, int SM>
__global__ void k_beam_slice(const T* __restrict__ g, const DirConst* __restrict__ dirs, int q, int nd, int L,
                             T* __restrict__ gl, const DevStats* st)
{
    if (*(volatile const int*)&st->gather_off) return;
    const int lane = beam_axes(dirs + q).lane;
    const unsigned long long n = 1ull << (3 * L);
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        T v[SM];
        load_row<T, SM>(g + ((size_t)row_leaf(i, L, lane) * nd + q) * SM, v);
        store_row<T, SM>(gl + (size_t)i * SM, v);
    }
}

// ------------------------------------------------------------ the kernel

enum { kBeamColumns = 0, kBeamEpilogue = 1, kBeamAdjoint = 2 };

struct BeamArgs {
    TraceArgs t;            // octree, directions, sources, output, epilogue, statistics
    BeamTables tab;
    const void* field[2];   // row layouts along x and along y (adjoint: the slice, in either)
    const BeamRef* ref;
    const uint32_t* out;    // a bit per source: left out
    unsigned long long* queue;  // units handed out so far (adjoint: one a direction)
    int q0, nq, dgroup;     // directions [q0, q0 + nq), dgroup at a time
    long long blocks;       // 32^3-leaf blocks the sources can touch
};

// Sums of one leaf's terms: F32-Kahan columns and gradients add every product
// with one Kahan step, species two at a time; FP64 columns add the rounded
// product, FP64 gradients a fused one.
template <int MODE, int SM, int OP>
struct BeamSum {
    float s[SM], c[SM];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int k = 0; k < SM; k++) s[k] = c[k] = 0.f;
    }
    __device__ __forceinline__ void add(const float n[SM], float ds)
    {
        unsigned long long d2 = 0ull;
        if (SM > 1) asm("mov.b64 %0, {%1, %1};" : "=l"(d2) : "f"(ds));
#pragma unroll
        for (int k = 0; k + 1 < SM; k += 2) kahan2(s[k], s[k + 1], c[k], c[k + 1], n[k], n[k + 1], d2);
        if (SM & 1) {
            const float y = __fmaf_rn(n[SM - 1], ds, c[SM - 1]);
            const float tt = __fadd_rn(s[SM - 1], y);
            c[SM - 1] = __fsub_rn(y, __fsub_rn(tt, s[SM - 1]));
            s[SM - 1] = tt;
        }
    }
    __device__ __forceinline__ double total(int k) const { return __dadd_rn((double)s[k], (double)c[k]); }
};
template <int SM, int OP>
struct BeamSum<RT_MODE_FP64, SM, OP> {
    double s[SM];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int k = 0; k < SM; k++) s[k] = 0.0;
    }
    __device__ __forceinline__ void add(const double n[SM], double ds)
    {
#pragma unroll
        for (int k = 0; k < SM; k++)
            s[k] = OP == kBeamAdjoint ? __fma_rn(n[k], ds, s[k]) : __dadd_rn(s[k], __dmul_rn(n[k], ds));
    }
    __device__ __forceinline__ double total(int k) const { return s[k]; }
};

// Adds a whole run of K steps for R leaves in a row along the run axis: leaf r
// takes the cells r .. r + K - 1 of the R + K - 1 the leaves share, so each cell
// is loaded once for up to K leaves.
template <int MODE, int SM, int R, int OP, int K, class T>
__device__ __forceinline__ void whole_run(BeamSum<MODE, SM, OP> sum[R], const T* __restrict__ p, long long rs,
                                          const T ds[kRun])
{
    T v[R + K - 1][SM];
#pragma unroll
    for (int z = 0; z < R + K - 1; z++) load_row<T, SM>(p + z * rs, v[z]);
#pragma unroll
    for (int z = 0; z < R + K - 1; z++) {
#pragma unroll
        for (int r = 0; r < R; r++) {
            if (z - r >= 0 && z - r < K) sum[r].add(v[z], ds[z - r < 0 || z - r >= K ? 0 : z - r]);
        }
    }
}

// A run near the cube's face: only its first lim cells exist.
template <int MODE, int SM, int R, int OP, class T>
__device__ __forceinline__ void cut_run(BeamSum<MODE, SM, OP> sum[R], const T* __restrict__ p, long long rs, int k,
                                        int lim, const T ds[kRun])
{
#pragma unroll
    for (int z = 0; z < R + kRun - 1; z++) {
        if (z < lim && z < R + k - 1) {
            T v[SM];
            load_row<T, SM>(p + z * rs, v);
#pragma unroll
            for (int r = 0; r < R; r++)
                if (z - r >= 0 && z - r < kRun && z - r < k) sum[r].add(v, ds[z - r < 0 || z - r >= kRun ? 0 : z - r]);
        }
    }
}

template <class T>
__device__ __forceinline__ void load_run(const BeamRun<T>* __restrict__ e, int4& h, T ds[kRun])
{
    h = __ldg((const int4*)e);
    load_row<T, kRun>((const T*)((const char*)e + 16), ds);
}

// Leaves a thread takes along the run axis (R), and blocks of kBeamWarps warps
// an SM holds.  A longer row shares each loaded cell among more leaves and
// spreads a run's fixed cost (its table entry, its branch, the wait for its
// cells) over more sums; it takes registers from the warps in flight.
// Columns of every leaf, Nside 1, R = 2 / 4 / 8:
//   F32-Kahan, 256^3, ms, at 4 blocks (1 species 16.5 / 14.7 / 9.6, 2: 21.0 / 19.2 / 13.1, 4: 29.1 /
//   21.4 / 18.9, 8: 49.3 / 38.5 / 80.5, spilling), 5 blocks (16.2 / 14.7 / 9.6, 21.0 / 16.1 / 12.0, 29.8
//   / 21.4 / 22.9) and 3 blocks (8 species 59.7 / 43.8 / 50.7; 4 species at R = 8 21.0);
//   FP64, 128^3, ms (1 species 7.76 / 7.12 / 7.27, 2: 14.4 / 14.1 / 14.4, 4: 27.8 / 28.0 / 28.6, 8: 55.3 /
//   55.4 / 55.9; 3 or 5 blocks within 1 %) and 32^3, us (90 / 96 / 118, 134 / 143 / 219, 203 / 255 / 381, 351 /
//   415 / 567).
// 8 or 16 warps a block in place of 4: 23.8 and 25.3 against 23.2 ms (256^3, 4 species,
// R = 4, 128 registers).  Loading the next run's cells while the current one is
// added, into a second register set: 26.3 to 28.6.
constexpr int kBeamWarps = 4;
template <int MODE, int SM>
__host__ __device__ constexpr int beam_r()
{
    return MODE == RT_MODE_FP64 ? (SM >= 4 ? 2 : 4) : (SM >= 8 ? 4 : 8);
}
template <int MODE, int SM, int R>
__host__ __device__ constexpr int beam_blocks()
{
    if (R == 1) return MODE == RT_MODE_FP64 ? (SM >= 8 ? 3 : SM >= 4 ? 4 : SM >= 2 ? 6 : 8) : (SM >= 8 ? 6 : 8);
    if (MODE == RT_MODE_F32_KAHAN && SM == 4 && R == 4) return 5;
    return MODE == RT_MODE_FP64 ? (SM >= 8 ? 2 : 4) : (SM == 2 ? 5 : 4);
}

// Leaves a thread takes in the adjoint.  It is launched one direction at a time,
// so a launch has a twelfth (Nside 1) of the columns' units, and on a small cube
// a long row leaves the chip short of warps: there a thread takes one leaf and
// four steps' cells at once (add_steps).  Adjoint of a 64^3 cube, all directions,
// us, one leaf against beam_r: F32-Kahan 1 species 293 / 437, 4 397 / 599, 8 650
// / 719; FP64 472 / 702, 1240 / 1405, 2231 / 2368.  Of a 128^3 cube: F32-Kahan
// 1497 / 1313, 2867 / 2844, 5431 / 4837; FP64 1 species 3931 / 4146, 2 7186 /
// 7370, 4 13436 / 13268, 8 25758 / 26132 (more registers; at 256^3 FP64 1
// species 51.0 / 50.6 ms).  F32-Kahan, 4 species: 4 leaves at 96 registers against
// 8, 128^3 2760 / 2844, 256^3 27.9 / 26.0 ms.
template <int MODE, int SM>
__host__ __device__ constexpr int beam_adjoint_r(int level)
{
    return level <= (MODE == RT_MODE_FP64 && SM <= 2 ? 7 : 6) ? 1
         : MODE == RT_MODE_F32_KAHAN && SM == 4 && level == 7 ? 4 : beam_r<MODE, SM>();
}

// The runs [0, nr) of a direction's n_run for R leaves in a row (ahead: cells of the cube from
// the first leaf on, itself among them).  The next run's entry is read ahead of
// its use.
template <int MODE, int SM, int R, int OP, class T>
__device__ __forceinline__ void add_runs(BeamSum<MODE, SM, OP> sum[R], const BeamRun<T>* __restrict__ run, int nr,
                                         int n_run, int ahead, const T* __restrict__ base, long long rs)
{
    int4 h;
    T ds[kRun];
    load_run(run, h, ds);
    for (int e = 0; e < nr; e++) {
        int4 hn;
        T dn[kRun];
        load_run(run + min(e + 1, n_run - 1), hn, dn);
        const int lim = ahead - h.y;
        if (lim <= 0) break;
        const T* p = base + (long long)(OP == kBeamAdjoint ? -h.x : h.x) * SM;
        if (lim >= R + h.z - 1) {
            switch (h.z) {
            case 1: whole_run<MODE, SM, R, OP, 1>(sum, p, rs, ds); break;
            case 2: whole_run<MODE, SM, R, OP, 2>(sum, p, rs, ds); break;
            case 3: whole_run<MODE, SM, R, OP, 3>(sum, p, rs, ds); break;
            default: whole_run<MODE, SM, R, OP, 4>(sum, p, rs, ds); break;
            }
        } else {
            cut_run<MODE, SM, R, OP>(sum, p, rs, h.z, lim, ds);
        }
        h = hn;
#pragma unroll
        for (int k = 0; k < kRun; k++) ds[k] = dn[k];
    }
}

// The steps [0, n) of direction q for one leaf of the adjoint, kSteps cells
// loaded before the first is added: with one leaf a thread and few warps in
// flight it is the wait for the cells that counts, and a run holds as few as one.
constexpr int kSteps = 4;
template <int MODE, int SM, int OP, class T>
__device__ __forceinline__ void add_steps(BeamSum<MODE, SM, OP>& sum, const BeamTables& tab, int q, int n,
                                          const T* __restrict__ base)
{
    const int* __restrict__ D = tab.D + (size_t)q * tab.lcap;
    const T* __restrict__ ds = (const T*)tab.ds + (size_t)q * tab.lcap;
    int i = 0;
    for (; i + kSteps <= n; i += kSteps) {
        const int4 at = __ldg((const int4*)(D + i));
        T d[kSteps], v[kSteps][SM];
        load_row<T, kSteps>(ds + i, d);
        load_row<T, SM>(base - (long long)at.x * SM, v[0]);
        load_row<T, SM>(base - (long long)at.y * SM, v[1]);
        load_row<T, SM>(base - (long long)at.z * SM, v[2]);
        load_row<T, SM>(base - (long long)at.w * SM, v[3]);
#pragma unroll
        for (int u = 0; u < kSteps; u++) sum.add(v[u], d[u]);
    }
    for (; i < n; i++) {
        T v[SM];
        load_row<T, SM>(base - (long long)__ldg(D + i) * SM, v);
        sum.add(v, __ldg(ds + i));
    }
}

// Units of a leaf block of edge B and one direction: R leaves a warp along the
// run axis, W warps.
__host__ __device__ __forceinline__ int beam_units(int B, int R, int W)
{
    return B == 32 ? 32 * 32 / (R * W) : ((B + W - 1) / W) * ((B + R - 1) / R);
}

// A block takes units of 32 (lane axis) x wt (third axis) x R wr (run axis)
// leaves, wt wr warps, and one direction.  A unit moving with the rays enters
// 32 (m_run wt + m_third R wr) new cells a step through those faces, least at
// R wr^2 = W m_run / m_third.  Units are handed out 32^3-leaf block by
// block in Morton order, dgroup directions of each in turn, so the units in
// flight lie close together (their cells stay in L2) and a leaf's outputs for
// dgroup directions are written close in time (they meet in L2).
template <int MODE, int SM, int R, int OP>
__global__ void __launch_bounds__(32 * kBeamWarps, beam_blocks<MODE, SM, R>()) k_beam(const BeamArgs a)
{
    using T = typename std::conditional<MODE == RT_MODE_FP64, double, float>::type;
    if (*(volatile const int*)&a.t.st->gather_off) return;
    if (OP == kBeamAdjoint && a.q0 == 0 && blockIdx.x == 0 && threadIdx.x == 0) a.t.st->gathered = 1;
    __shared__ unsigned long long s_unit;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = a.t.t.uniform_level;
    const int N = 1 << L;
    const int B = min(32, N);                            // edge of a leaf block
    constexpr int W = kBeamWarps;
    const int U = beam_units(B, R, W);
    const uint32_t j0 = OP == kBeamAdjoint ? 0u : (uint32_t)a.ref->j0;
    const long long total = a.blocks * a.nq * U;
    unsigned long long n_segs = 0, n_rays = 0, n_efb = 0;
    const bool once = R == 1 && total <= gridDim.x;  // a block a unit needs no queue (32^3, 1 species: 178 -> 166 us)
    for (bool first_unit = true;; first_unit = false) {
        long long u = blockIdx.x;
        if (!once) {
            __syncthreads();
            if (threadIdx.x == 0) s_unit = atomicAdd(a.queue, 1ull);
            __syncthreads();
            u = (long long)s_unit;
        }
        if (u >= total || (once && !first_unit)) break;
        const int ut = (int)(u % U);
        const long long v = u / U;
        const int qd = (int)(v % a.dgroup);
        const long long w = v / a.dgroup;
        const uint32_t blk = (uint32_t)(w % a.blocks) + (B == 32 ? j0 >> 15 : 0u);
        const int q = a.q0 + (int)(w / a.blocks) * a.dgroup + qd;
        const DirConst* d = a.t.dirs + q;
        const int flags = __ldg(&d->flags);
        const BeamAxes ax = beam_axes(d);
        int wr = 1;
        if (B == 32) {
            const float mr = fabsf(sel3(d->m32, ax.run)), mt = fabsf(sel3(d->m32, ax.third));
            while (2 * wr <= W && 2 * wr * R <= 32 && 2 * wr * wr * R * mt < W * mr) wr *= 2;
        }
        const int wt = W / wr, U3 = (B + wt - 1) / wt;
        const int3 org = make_int3(32 * (int)compact10(blk), 32 * (int)compact10(blk >> 1), 32 * (int)compact10(blk >> 2));
        const int oL = ax.lane == 0 ? org.x : org.y;
        const int oR = ax.run == 0 ? org.x : (ax.run == 1 ? org.y : org.z);
        const int oT = ax.third == 1 ? org.y : org.z;
        const int cl = oL + lane, ct = oT + wt * (ut % U3) + warp / wr;
        const int cr = oR + R * (wr * (ut / U3) + warp % wr);
        if (cl >= N || ct >= N || cr >= N) continue;  // cubes below 32^3, or past the last block
        // the ray's cells lie ahead of the source; the adjoint's sources behind the leaf
        const int sgn = OP == kBeamAdjoint ? ~flags : flags;
        const bool upL = (sgn >> (3 + ax.lane)) & 1, upR = (sgn >> (3 + ax.run)) & 1, upT = (sgn >> (3 + ax.third)) & 1;
        const int4 info = __ldg(a.tab.info + q);
        const int* __restrict__ Pq = a.tab.P + (size_t)q * 3 * a.tab.pcap;
        const int* __restrict__ Cq = a.tab.C + (size_t)q * 3 * a.tab.pcap;
        int nr = info.x, steps = info.y;
        if (flags & (1 << ax.lane)) {
            const int room = upL ? N - 1 - cl : cl;
            nr = min(nr, __ldg(Cq + ax.lane * a.tab.pcap + room));
            steps = min(steps, __ldg(Pq + ax.lane * a.tab.pcap + room));
        }
        if (flags & (1 << ax.third)) {
            const int room = upT ? N - 1 - ct : ct;
            nr = min(nr, __ldg(Cq + ax.third * a.tab.pcap + room));
            steps = min(steps, __ldg(Pq + ax.third * a.tab.pcap + room));
        }
        const int st_r = beam_stride(ax.run, ax.lane, L), st_t = beam_stride(ax.third, ax.lane, L);
        const int first = upR ? cr : cr + R - 1;      // the leaf with the most cells ahead
        const int ahead = upR ? N - first : first + 1;  // itself among them
        const long long rs = (long long)(upR ? st_r : -st_r) * SM;
        const T* __restrict__ base = (const T*)a.field[ax.lane] + ((long long)cl + (long long)ct * st_t + (long long)first * st_r) * SM;
        BeamSum<MODE, SM, OP> sum[R];  // sum[r]: leaf `first` + r steps forward
#pragma unroll
        for (int r = 0; r < R; r++) sum[r].init();
        if constexpr (R == 1)
            add_steps(sum[0], a.tab, q, min(steps, __ldg(Pq + ax.run * a.tab.pcap + ahead - 1)), base);
        else
            add_runs<MODE, SM, R, OP>(sum, (const BeamRun<T>*)a.tab.run + (size_t)q * a.tab.lcap, nr, info.x, ahead, base, rs);
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int c = upR ? first + r : first - r;
            if (c < N) {
                const int x = ax.run == 0 ? c : cl, y = ax.run == 1 ? c : (ax.lane == 1 ? cl : ct);
                const int z = ax.run == 2 ? c : ct;
                const uint32_t j = spread10((uint32_t)x) | (spread10((uint32_t)y) << 1) | (spread10((uint32_t)z) << 2);
                const long long s = (long long)j - (long long)j0;
                if (OP == kBeamAdjoint || (s >= 0 && s < a.t.n_src && !((__ldg(a.out + (s >> 5)) >> (s & 31)) & 1u))) {
                    const long long ray = s * a.t.nd + q;
                    if (OP == kBeamAdjoint) {
                        double* gp = (double*)a.t.out + (size_t)j * SM;
#pragma unroll
                        for (int k = 0; k < SM; k++) gp[k] = __dadd_rn(gp[k], sum[r].total(k));
                    } else if (OP == kBeamEpilogue) {
                        double comb = 0.0;
#pragma unroll
                        for (int k = 0; k < SM; k++)
                            if (k < a.t.S) comb = __dadd_rn(comb, __dmul_rn(a.t.epi_w[k], (double)sum[r].s[k]));
                        ray_epilogue(a.t, s, ray, comb);
                    } else {
                        T* o = (T*)a.t.out + (size_t)ray * a.t.S;
                        if (a.t.S == SM) {
                            T col[SM];
#pragma unroll
                            for (int k = 0; k < SM; k++) col[k] = sum[r].s[k];
                            store_row<T, SM>(o, col);
                        } else {
#pragma unroll
                            for (int k = 0; k < SM; k++)
                                if (k < a.t.S) o[k] = sum[r].s[k];
                        }
                    }
                    // statistics of the rays as the walk counts them
                    int len = steps;
                    const int room = upR ? N - 1 - c : c;
                    len = min(len, __ldg(Pq + ax.run * a.tab.pcap + room));
                    n_segs += (unsigned)len;
                    n_rays += 1;
                    if (OP != kBeamAdjoint && MODE == RT_MODE_F32_KAHAN)
                        n_efb += (unsigned)__ldg(a.tab.fb + (size_t)q * a.tab.lcap + (len - 1));
                }
            }
        }
    }
    if constexpr (R > 1) {
        __syncwarp();
        flush_counters(a.t.st, n_rays, n_segs, n_efb, 0ull);
    } else {
        // the adjoint of a small cube is a launch of some microseconds a direction, and
        // additions to one address follow one another at about 2 ns each: one a
        // block and not one a warp (64^3, 1 species, 309 -> 293 us)
        __shared__ unsigned long long s_sum[2];
        __syncthreads();
        if (threadIdx.x < 2) s_sum[threadIdx.x] = 0ull;
        __syncthreads();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n_rays += __shfl_down_sync(RT_FULL, n_rays, o);
            n_segs += __shfl_down_sync(RT_FULL, n_segs, o);
        }
        if (lane == 0) {
            atomicAdd(s_sum, n_rays);
            atomicAdd(s_sum + 1, n_segs);
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_sum[0]) {
            atomicAdd(&a.t.st->rays, s_sum[0]);
            atomicAdd(&a.t.st->segments, s_sum[1]);
        }
    }
}

// Launches k_beam for the directions [g.q0, g.q0 + g.nq), units handed out over g.queue.
template <int MODE, int SM, int R, int OP>
static cudaError_t go_beam(const BeamArgs& g, cudaStream_t s)
{
    constexpr int W = kBeamWarps;
    int dev = 0, fit = 0;
    cudaGetDevice(&dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, k_beam<MODE, SM, R, OP>, 32 * W, 0);
    const int B = std::min(32, 1 << g.t.t.uniform_level);
    const long long units = g.blocks * g.nq * beam_units(B, R, W);
    const int grid = (int)std::min<long long>(units, (long long)sm_count_of(dev) * std::max(1, fit));
    if (OP != kBeamAdjoint) {
        k_beam<MODE, SM, R, OP><<<grid, 32 * W, 0, s>>>(g);
        return cudaGetLastError();
    }
    // one direction after another
    using T = typename std::conditional<MODE == RT_MODE_FP64, double, float>::type;
    const int sgrid = (int)std::min<long long>((g.t.n_src + 255) / 256, (long long)sm_count_of(dev) * 16);
    BeamArgs d = g;
    for (int q = 0; q < g.t.nd; q++) {
        k_beam_slice<T, SM><<<sgrid, 256, 0, s>>>((const T*)g.t.gin, g.t.dirs, q, g.t.nd, g.t.t.uniform_level, (T*)g.field[0], g.t.st);
        d.q0 = q;
        d.queue = g.queue + q;
        k_beam<MODE, SM, R, OP><<<grid, 32 * W, 0, s>>>(d);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int MODE, int SM>
static cudaError_t go_beam_op(const BeamArgs& g, int op, cudaStream_t s)
{
    constexpr int R = beam_r<MODE, SM>();
    if (op == kBeamAdjoint) {
        const int r = beam_adjoint_r<MODE, SM>(g.t.t.uniform_level);
        if (r == 1) return go_beam<MODE, SM, 1, kBeamAdjoint>(g, s);
        if constexpr (beam_adjoint_r<MODE, SM>(7) == 4 && R != 4)
            if (r == 4) return go_beam<MODE, SM, 4, kBeamAdjoint>(g, s);
        return go_beam<MODE, SM, R, kBeamAdjoint>(g, s);
    }
    if (op == kBeamEpilogue) return go_beam<MODE, SM, R, kBeamEpilogue>(g, s);
    return go_beam<MODE, SM, R, kBeamColumns>(g, s);
}

// ------------------------------------------------------------- host side

static size_t round256(size_t v) { return (v + 255) / 256 * 256; }

static int padded_species(int S) { return S <= 1 ? 1 : S <= 2 ? 2 : S <= 4 ? 4 : 8; }

// Scratch of a call in two parts, laid out from p (the tables, which a later
// call finds there, so at places that do not depend on n_src) and from v (the
// check's results); sizes only if p is null.  A sixteenth of the sources may be left
// out (the form gains beyond that: 4 species, F32-Kahan, of a 64^3 cube a 16th 270 us against
// 1744 walked, a quarter 438 / 1870; FP64 2455 / 5067, 3442 / 5591.  The line
// keeps the list a quarter byte a source, and is what the vote of 32 can tell
// from scattered points).
struct BeamScratch {
    BeamTables tab;
    BeamRef* ref;
    uint32_t *out, *rest;
    unsigned long long* queue;
    unsigned int most;
    size_t kept, call;  // bytes of the two parts
};

static BeamScratch beam_scratch(char* p, char* v, int nd, int L, int64_t n_src, int mode, bool adjoint)
{
    BeamScratch b;
    memset(&b, 0, sizeof b);
    const int N = 1 << L;
    const int lcap = (3 * N + 3 + 15) / 16 * 16, pcap = (N + 1 + 3) / 4 * 4;
    const size_t rsz = mode == RT_MODE_FP64 ? sizeof(BeamRun<double>) : sizeof(BeamRun<float>);
    const size_t steps = adjoint ? (size_t)nd * lcap : 0;
    const size_t bytes[] = {sizeof(BeamRef), (size_t)nd * sizeof(int4), (size_t)nd * lcap * rsz, (size_t)nd * lcap * 4,
                            (size_t)nd * 3 * pcap * 4, (size_t)nd * 3 * pcap * 4, steps * 4,
                            steps * (mode == RT_MODE_FP64 ? 8 : 4), (size_t)(adjoint ? nd : 1) * 8};
    size_t at[10] = {0};
    for (int i = 0; i < 9; i++) at[i + 1] = at[i] + round256(bytes[i]);
    b.most = (unsigned int)(n_src / 16);
    const size_t list = round256((size_t)((n_src + 31) / 32) * 4);
    b.kept = at[9];
    b.call = list + round256((size_t)b.most * 4);
    b.tab.lcap = lcap;
    b.tab.pcap = pcap;
    if (p) {
        b.ref = (BeamRef*)(p + at[0]);
        b.tab.info = (int4*)(p + at[1]);
        b.tab.run = p + at[2];
        b.tab.fb = (int*)(p + at[3]);
        b.tab.P = (int*)(p + at[4]);
        b.tab.C = (int*)(p + at[5]);
        b.tab.D = adjoint ? (int*)(p + at[6]) : nullptr;
        b.tab.ds = adjoint ? p + at[7] : nullptr;
        b.queue = (unsigned long long*)(p + at[8]);
        b.out = (uint32_t*)v;
        b.rest = (uint32_t*)(v + list);
    }
    return b;
}

// Enqueues the source check (most: sources that may be left out) and the tables,
// and resets the queues.
static cudaError_t beam_setup(const TraceArgs& a, int mode, const BeamScratch& b, unsigned int most, int queues, cudaStream_t s)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const int grid = a.nd + (int)std::max<long long>(1, std::min<long long>((a.n_src + 255) / 256, (long long)sm_count_of(dev) * 8));
    const unsigned int key = 1u | (unsigned)a.t.uniform_level << 1 | (unsigned)mode << 6 | (unsigned)a.nd << 7;
    k_beam_ref<<<1, 32, 0, s>>>(a.src, a.n_src, a.t.uniform_level, key, a.nd, most ? kBeamVotes : 32, b.ref, b.queue, queues, a.st);
    if (mode == RT_MODE_FP64)
        k_beam_setup<RT_MODE_FP64><<<grid, 256, 0, s>>>(a.t, a.dirs, a.nd, a.src, a.n_src, b.ref, b.tab, b.out, b.rest, most, a.st);
    else
        k_beam_setup<RT_MODE_F32_KAHAN><<<grid, 256, 0, s>>>(a.t, a.dirs, a.nd, a.src, a.n_src, b.ref, b.tab, b.out, b.rest, most, a.st);
    return cudaGetLastError();
}

// True when the call's shape admits the adjoint as a gather (the sources are
// checked on the device): a full cube of equal-level leaves under its O(1)
// index, one source per leaf, the default step cap and a species count
// gathered as one vector.
bool gather_applies(const rt_octree* t, const TraceArgs& a)
{
    return a.t.uniform_level >= 0 && a.n_src == t->dev.n && t->dev.step_cap >= t->default_cap &&
           (a.S == 1 || a.S == 2 || a.S == 4 || a.S == 8);
}

// Enqueues the source check, the tables and the gather on `s`: one direction
// after another (the stream orders them, so each leaf's gradient takes its
// directions in a fixed order and no two threads update it at once).  The
// scatter launched after it must carry gate = &st->gather_off.
int launch_adjoint_gather(rt_octree* t, const TraceArgs& a, int mode, cudaStream_t s)
{
    const size_t tsz = mode == RT_MODE_FP64 ? 8 : 4;
    const BeamScratch sz = beam_scratch(nullptr, nullptr, a.nd, a.t.uniform_level, a.n_src, mode, true);
    const size_t need = sz.kept + sz.call + (size_t)a.n_src * a.S * tsz;
    if (t->adj_tab_bytes < need) {
        if (t->adj_tab) {
            cudaStreamSynchronize(s);
            cudaFree(t->adj_tab);
            t->adj_tab = nullptr;
            t->adj_tab_bytes = 0;
        }
        if (cudaMalloc(&t->adj_tab, need) != cudaSuccess) {
            t->adj_tab = nullptr;
            return cuda_error("rt_trace_columns_adjoint: gather scratch allocation");
        }
        t->adj_tab_bytes = need;
        cudaMemsetAsync(t->adj_tab, 0, sizeof(BeamRef), s);  // no tables yet
    }
    BeamArgs g;
    memset(&g, 0, sizeof g);
    g.t = a;
    const BeamScratch b = beam_scratch((char*)t->adj_tab, (char*)t->adj_tab + sz.kept, a.nd, a.t.uniform_level, a.n_src, mode, true);
    g.tab = b.tab;
    g.queue = b.queue;
    char* gl = (char*)t->adj_tab + sz.kept + sz.call;
    g.field[0] = g.field[1] = gl;
    g.nq = g.dgroup = 1;
    const int L = a.t.uniform_level;
    g.blocks = L >= 5 ? 1ll << (3 * (L - 5)) : 1;
    cudaError_t e = beam_setup(a, mode, b, 0, a.nd, s);  // a source left out: no gather
    if (e == cudaSuccess) {
        if (mode == RT_MODE_FP64)
            e = a.S == 1 ? go_beam_op<RT_MODE_FP64, 1>(g, kBeamAdjoint, s) : a.S == 2 ? go_beam_op<RT_MODE_FP64, 2>(g, kBeamAdjoint, s)
              : a.S == 4 ? go_beam_op<RT_MODE_FP64, 4>(g, kBeamAdjoint, s) : go_beam_op<RT_MODE_FP64, 8>(g, kBeamAdjoint, s);
        else
            e = a.S == 1 ? go_beam_op<RT_MODE_F32_KAHAN, 1>(g, kBeamAdjoint, s) : a.S == 2 ? go_beam_op<RT_MODE_F32_KAHAN, 2>(g, kBeamAdjoint, s)
              : a.S == 4 ? go_beam_op<RT_MODE_F32_KAHAN, 4>(g, kBeamAdjoint, s) : go_beam_op<RT_MODE_F32_KAHAN, 8>(g, kBeamAdjoint, s);
    }
    if (e != cudaSuccess) return cuda_error("rt_trace_columns_adjoint: gather launch");
    return RT_OK;
}

// Blocks of 32^3 leaves n_src consecutive leaves of a cube of level L may touch.
static long long beam_blocks_of(int L, int64_t n_src)
{
    return std::min<long long>(1ll << (3 * (L - 5)), (n_src + 32767) / 32768 + 1);
}

// True where the form pays, us of it and of the walk (one ray a lane), sources at leaf
// centres.  It computes whole 32^3 blocks: at most 1.5 leaves computed a source
// (FP64, bound by its operations: 1 species 2, 5 to 8 species 1.2), and 2^18 rays to
// fill the chip.
//
// F32-Kahan, 64^3 at 1.25, 1.5 and 2 leaves a source: 1 species 97 / 153, 81 / 100, 69 /
// 60; 4 species 130 / 186, 95 / 111, 88 / 65; 8 species 172 / 294, 124 / 168, 97 / 93.
// Every leaf of 32^3 (3.9e5 rays) 54 / 41, 58 / 49, 63 / 67, half of it 53 / 34, 57 / 40, 63 / 47.
// FP64, the same: 381 / 731, 246 / 404, 190 / 235; 1252 / 1445, 782 / 827, 544 / 528;
// 2430 / 2393, 1501 / 1261, 1041 / 1041.  32^3, 1 species: 92 / 88 on densities in
// L2, 95 / 122 on new ones, half of it (2.0e5) 92 / 72, at Nside 2 203 / 280.
//
// Sources in a sixteenth of the leaves or more: of 128^3, 4 species, F32-Kahan, 191 / 266, of
// 256^3 1408 / 3086.  It gains below that too (256^3, a 32nd 813 / 1512), but scattered
// points pay for the vote (12 us), of which a smaller call is a larger part.
static bool beam_pays(int L, int64_t n_src, int nd, int S, int mode, int64_t n_leaves)
{
    const long long done = beam_blocks_of(L, n_src) * 32768;
    if (n_src * 16 < n_leaves || n_src * nd < (1ll << 18)) return false;
    if (mode != RT_MODE_FP64 || (S > 1 && S <= 4)) return done * 2 <= n_src * 3;
    return S == 1 ? done <= n_src * 2 : done * 5 <= n_src * 6;
}

// Bytes of tables the shared-offset trace keeps on this octree, 0 when its
// shape does not admit it: a cube of at least 32^3 leaves (its rows fill a
// warp), a call that it is worth for, the default step cap and tables of at most
// 256 MB.
size_t beam_bytes(const rt_octree* t, int64_t n_src, int nd, int S, int mode)
{
    const int L = t->uniform_allowed ? t->dev.uniform_level : -1;
    if (L < 5 || n_src < 32 || n_src > t->dev.n || !beam_pays(L, n_src, nd, S, mode, t->dev.n) || t->dev.step_cap < t->default_cap)
        return 0;
    const size_t kept = beam_scratch(nullptr, nullptr, nd, L, n_src, mode, false).kept;
    return kept > (256ull << 20) ? 0 : kept;
}

// Memory of the shared-offset trace comes from a pool of the device, in the order
// of the stream: a call takes what it needs (two row copies of the
// densities, the check's results) and gives it back behind its last kernel, so
// no call waits for the device, and between calls a handle holds its tables
// alone.  The pool keeps what is given back for the next call (a 4.3 GB block: 1.5
// us, against 2.5 ms from the device and 4.3 to return it) while a handle or
// the host call's buffers use it, and returns all of it with the last of them;
// an allocation by cudaMalloc that does not fit takes it from the pool before that.
// It is never used by way of another stream's unfinished work (no stream
// waits for another on account of memory).
namespace {
struct Pool {
    cudaMemPool_t pool = nullptr;
    int users = 0;
};
std::mutex g_pool_mu;
Pool g_pool[64];
}  // namespace

// An allocation here is safe beside another stream's capture, but the runtime
// refuses it, and breaks that capture, unless this thread asks for relaxed checks.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

bool beam_pool_join(int dev)
{
    if (dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    Pool& p = g_pool[dev];
    if (!p.pool) {
        RelaxedCapture relaxed;
        cudaMemPoolProps props;
        memset(&props, 0, sizeof props);
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        unsigned long long keep = ~0ull;
        int no = 0;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess ||
            cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &no) != cudaSuccess) {
            cudaGetLastError();
            if (pool) cudaMemPoolDestroy(pool);
            return false;
        }
        p.pool = pool;
    }
    p.users++;
    return true;
}

void beam_pool_leave(int dev)
{
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (--g_pool[dev].users == 0) cudaMemPoolTrimTo(g_pool[dev].pool, 0);
}

// `bytes` of the device's pool on `s`, null if there is no room.
static void* beam_alloc(int dev, size_t bytes, cudaStream_t s)
{
    RelaxedCapture relaxed;
    void* p = nullptr;
    if (cudaMallocFromPoolAsync(&p, bytes, g_pool[dev].pool, s) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

BeamCall::~BeamCall()
{
    if (!p) return;
    RelaxedCapture relaxed;
    cudaFreeAsync(p, s);
}

template <int MODE, int SM>
static cudaError_t go_trace(const BeamArgs& g, void* const rows[2], bool check, int op, cudaStream_t s)
{
    using T = typename std::conditional<MODE == RT_MODE_FP64, double, float>::type;
    int dev = 0;
    cudaGetDevice(&dev);
    const int L = g.t.t.uniform_level;
    const int grid = (int)std::min<long long>(1ll << (3 * L - 7), (long long)sm_count_of(dev) * 16);
    k_beam_dens<T, SM><<<grid, 256, 0, s>>>(g.t.dens, g.t.dens_f64, g.t.S, L, (T*)rows[0], (T*)rows[1], check, g.t.st);
    return go_beam_op<MODE, SM>(g, op, s);
}

// Enqueues the shared-offset forward trace (with the density check) or
// epilogue on `s`, if the call's shape admits it; call.p tells whether it did.
// It sets a's gate and list of left-out sources for the walk launched after
// it (call holds what that walk reads, until it is destroyed), and resets that
// walk's queue.  A captured stream, or no memory, leaves the call to the walk.
int launch_beam(rt_octree* t, TraceArgs& a, int mode, bool epilogue, bool check, cudaStream_t s, BeamCall& call)
{
    const size_t kept = beam_bytes(t, a.n_src, a.nd, a.S, mode);
    if (!kept || a.t.uniform_level < 0) return RT_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return RT_OK;
    }
    if (!t->fwd_pool && !(t->fwd_pool = beam_pool_join(t->device))) return RT_OK;
    const int L = a.t.uniform_level, SM = padded_species(a.S);
    const size_t row_bytes = round256((size_t)t->dev.n * SM * (mode == RT_MODE_FP64 ? 8 : 4));
    const BeamScratch sz = beam_scratch(nullptr, nullptr, a.nd, L, a.n_src, mode, false);
    if (t->fwd_tab_bytes < kept) {
        if (t->fwd_tab_lent) return RT_OK;
        BeamCall old{t->fwd_tab, s};
        t->fwd_tab_bytes = 0;
        if (!(t->fwd_tab = beam_alloc(t->device, kept, s))) return RT_OK;
        t->fwd_tab_bytes = kept;
        cudaMemsetAsync(t->fwd_tab, 0, sizeof(BeamRef), s);  // no tables yet
    }
    char* v = (char*)beam_alloc(t->device, sz.call + 2 * row_bytes, s);
    if (!v) return RT_OK;
    call.p = v;
    call.s = s;
    BeamArgs g;
    memset(&g, 0, sizeof g);
    g.t = a;
    const BeamScratch b = beam_scratch((char*)t->fwd_tab, v, a.nd, L, a.n_src, mode, false);
    g.tab = b.tab;
    g.queue = b.queue;
    g.ref = b.ref;
    g.out = b.out;
    void* rows[2] = {v + sz.call, v + sz.call + row_bytes};
    g.field[0] = rows[0];
    g.field[1] = rows[1];
    g.nq = a.nd;
    g.dgroup = a.dgroup > 1 ? a.dgroup : 1;
    g.blocks = beam_blocks_of(L, a.n_src);
    const int op = epilogue ? kBeamEpilogue : kBeamColumns;
    cudaError_t e = beam_setup(a, mode, b, b.most, 1, s);
    if (e == cudaSuccess) {
        if (mode == RT_MODE_FP64)
            e = SM == 1 ? go_trace<RT_MODE_FP64, 1>(g, rows, check, op, s) : SM == 2 ? go_trace<RT_MODE_FP64, 2>(g, rows, check, op, s)
              : SM == 4 ? go_trace<RT_MODE_FP64, 4>(g, rows, check, op, s) : go_trace<RT_MODE_FP64, 8>(g, rows, check, op, s);
        else
            e = SM == 1 ? go_trace<RT_MODE_F32_KAHAN, 1>(g, rows, check, op, s) : SM == 2 ? go_trace<RT_MODE_F32_KAHAN, 2>(g, rows, check, op, s)
              : SM == 4 ? go_trace<RT_MODE_F32_KAHAN, 4>(g, rows, check, op, s) : go_trace<RT_MODE_F32_KAHAN, 8>(g, rows, check, op, s);
    }
    if (e != cudaSuccess) return cuda_error("shared-offset trace: launch");
    a.gate = &t->st->gather_off;
    a.rest = b.rest;
    a.n_rest = &b.ref->n_rest;
    return RT_OK;
}

}  // namespace rt
