// Device-side definitions shared by the CS and FD kernels.
//
// Work model: a "group" is a set of lattices with the same model, velocity
// set and storage type. Every kernel is persistent over a flat list of work
// items (one item = one tile of one lattice); item -> lattice by binary
// search of the lattices' first items. A single lattice is a group of one.
//
// Per-lattice dynamic state (which CS buffer is current, steps done, steps
// left) lives in the device descriptor and is advanced on the device at the
// end of every chunk of steps, so a captured chunk can be replayed as a CUDA
// graph any number of times.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lbm.h"

namespace lbm {

// Rows of partial sums one block adds up (obs_add_group).
constexpr int OBS_GROUP = 256;
__host__ __device__ constexpr long long obs_groups(long long items) { return (items + OBS_GROUP - 1) / OBS_GROUP; }

constexpr int NOBS = 4;  // sum rho (minus the storage offset), sum j_x, sum j_y, probe sum

struct alignas(16) LatDesc {   // copied in 16-byte chunks
    void* buf[3];           // CS: buf[0]/buf[1] ping-pong; FD: f^n, f^(1), f^(2)
    int nx, ny;
    int pitch;              // row pitch in elements (multiple of 32)
    int tiles_x;            // tiles along x for the group's tile shape
    long long plane;        // elements per population plane
    int item_begin;         // first work item of this lattice in its group
    int items;              // number of work items
    int cur;                // CS: index (0/1) of the buffer holding the state; in place: the phase
    int inplace;            // CS: one buffer updated in place (AA pattern)
    int obs_every;          // record observables when (step - obs_base) % obs_every == 0 (0: off)
    long long obs_base;     // step at which recording started
    long long step0;        // steps completed
    long long remaining;    // steps still to run (skipped when exhausted)
    double omega;           // CS: dt / tau_LU
    double cdx;             // FD: dt / dx
    double dt_tau;          // FD: dt / tau_FD
    double rho0;            // storage offset: populations stored as f - w_k rho0 (0 for FP64)
    double eps;             // FD: WENO epsilon
    double dt;              // time step, for time stamps
    int probe_comp;         // 0: u_x, 1: u_y, -1: no probe
    int obs_cap;            // capacity of the series
    double probe_norm;
    const double* probe_px;   // [nx]
    const double* probe_py;   // [ny]
    const float* probe_pxf;   // float copies for FP32 kernels
    const float* probe_pyf;
    double* partials;       // [items][NOBS], this lattice's slice (rows of a launch's blocks)
    double* group_partials; // [obs_groups][NOBS]: sums of OBS_GROUP rows each
    unsigned* obs_count;    // [obs_groups + 1]: rows done of each group, groups done (0 between launches)
    lbm_obs* series;        // [obs_cap]
    double* snap;           // [NOBS] result of a one-off observables reduction
    // float copies of omega, cdx, dt_tau, rho0, eps for the FP32 kernels (a
    // conversion from double would run on the narrow FP64 pipe every tile)
    float omega_f, cdx_f, dt_tau_f, rho0_f, eps_f;
    int* err;               // the group's error word (header word 2)
};

// State buffers: element (0, 0) of a buffer sits STATE_HEAD elements into its
// slot of the lattice's allocation and every slot ends with STATE_TAIL spare
// elements (row segments of bulk copies may reach into them).
constexpr long long STATE_HEAD = 4, STATE_TAIL = 1024;

// Error bits of the group error word: an access outside a state buffer caught
// by the bounds-checked build; an input value rejected by the state
// initialisation kernels (rho <= 0 or a non-finite value).
constexpr int ERR_BOUNDS = 2;
constexpr int ERR_INPUT = 4;

// Bounds-checked build (-DLBM_BOUNDS_CHECK; compute-sanitizer stand-in): a
// single-element access to a state buffer must hit a node of the lattice
// (population < K, row < ny, column < nx), a bulk row copy must stay inside
// the buffer's slot of the allocation. A failing check skips the access and
// sets ERR_BOUNDS; nothing traps. Without the flag the checks compile away.
#ifdef LBM_BOUNDS_CHECK
__device__ __forceinline__ bool bc_report(const LatDesc* d) {
    atomicOr(d->err, ERR_BOUNDS);
    return false;
}
__device__ __forceinline__ bool bc_node(const LatDesc* d, int K, long long off) {
    bool ok = off >= 0 && off < (long long)K * d->plane;
    if (ok) {
        const long long r = off % d->plane;
        ok = (r % d->pitch) < d->nx && (r / d->pitch) < d->ny;
    }
    return ok || bc_report(d);
}
__device__ __forceinline__ bool bc_span(const LatDesc* d, int K, long long off, long long n) {
    return (off >= -STATE_HEAD && off + n <= (long long)K * d->plane + STATE_TAIL) || bc_report(d);
}
#define LBM_BC_NODE(d, K, off) bc_node((d), (K), (off))
#define LBM_BC_SPAN(d, K, off, n) bc_span((d), (K), (off), (n))
#else
#define LBM_BC_NODE(d, K, off) true
#define LBM_BC_SPAN(d, K, off, n) true
#endif

// A per-lattice constant in the kernel's precision.
template <typename T>
__device__ __forceinline__ T lat_val(double d, float f);
template <>
__device__ __forceinline__ double lat_val<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float lat_val<float>(double, float f) { return f; }

// ---------------------------------------------------------------------------
// Gauss-Hermite nodes and weights (probabilists', weights summing to 1):
//   3 nodes: 0, +-sqrt(3); w = 2/3, 1/6 (the D2Q9 set of Sec. 2)
//   4 nodes: +-sqrt(3 -+ sqrt 6); w = (3 +- sqrt 6)/12
//   5 nodes: 0, +-sqrt(5 -+ sqrt 10); w = 8/15, (7 +- 2 sqrt 10)/60
// Values are the closed forms evaluated to 21 digits. Index i runs over the
// nodes in ascending order. All functions fold to immediates when i is a
// compile-time constant (fully unrolled population loops).
// ---------------------------------------------------------------------------
template <int Q1>
struct GH;

template <>
struct GH<3> {
    static __host__ __device__ constexpr double v(int i) {
        return i == 0 ? -1.73205080756887729353 : (i == 1 ? 0.0 : 1.73205080756887729353);
    }
    static __host__ __device__ constexpr double w(int i) { return i == 1 ? 2.0 / 3.0 : 1.0 / 6.0; }
    static __host__ __device__ constexpr double vmax() { return 1.73205080756887729353; }
};

template <>
struct GH<4> {
    static __host__ __device__ constexpr double v(int i) {
        return i == 0 ? -2.33441421833897723932
                      : (i == 1 ? -0.741963784302725857649
                                : (i == 2 ? 0.741963784302725857649 : 2.33441421833897723932));
    }
    static __host__ __device__ constexpr double w(int i) {
        return (i == 0 || i == 3) ? 0.0458758547680684918169 : 0.454124145231931508183;
    }
    static __host__ __device__ constexpr double vmax() { return 2.33441421833897723932; }
};

template <>
struct GH<5> {
    static __host__ __device__ constexpr double v(int i) {
        return i == 0 ? -2.85697001387280565416
                      : (i == 1 ? -1.35562617997426586583
                                : (i == 2 ? 0.0
                                          : (i == 3 ? 1.35562617997426586583 : 2.85697001387280565416)));
    }
    static __host__ __device__ constexpr double w(int i) {
        return (i == 0 || i == 4) ? 0.0112574113277206889334
                                  : ((i == 1 || i == 3) ? 0.2220759220056126444 : 0.533333333333333333333);
    }
    static __host__ __device__ constexpr double vmax() { return 2.85697001387280565416; }
};

// Population k = ix + Q1*iy of the product set.
template <int Q1>
__host__ __device__ constexpr double vx_of(int k) { return GH<Q1>::v(k % Q1); }
template <int Q1>
__host__ __device__ constexpr double vy_of(int k) { return GH<Q1>::v(k / Q1); }
template <int Q1>
__host__ __device__ constexpr double w_of(int k) { return GH<Q1>::w(k % Q1) * GH<Q1>::w(k / Q1); }
// D2Q9 lattice vector c_k = v_k dt/dx in {-1, 0, 1}.
__host__ __device__ constexpr int c3_of(int i) { return i - 1; }

// ---------------------------------------------------------------------------
// Work-item lookup: the lattice whose item range holds `item`.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_lattice(const int* __restrict__ item_begin, int n, int item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(item_begin + mid) <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Last i in 0 .. n - 1 with at_most(i), which holds for 0 and up to that i, by a
// warp (all lanes): 32 positions per round, so that a set of thousands of
// lattices takes two or three loads in turn, not a dozen (FD 9-velocity, 2000
// lattices of 32 x 32: 461 -> 421 us per step).
template <typename Fn>
__device__ __forceinline__ int last_at_most(int n, int lane, Fn at_most) {
    int lo = 0;
    while (n > 1) {   // it is one of lo .. lo + n - 1
        const int step = (n + 31) / 32, at = lane * step;
        const unsigned below = __ballot_sync(0xffffffffu, at < n && at_most(lo + at));
        const int c = max(__popc(below) - 1, 0);
        lo += c * step;
        n = min(step, n - c * step);
    }
    return lo;
}
__device__ __forceinline__ int find_lattice_warp(const int* __restrict__ item_begin, int n, int item, int lane) {
    return last_at_most(n, lane, [&](int i) { return __ldg(item_begin + i) <= item; });
}

// Last item of this block's sequence (first item `item`, stride gridDim.x)
// that still belongs to lattice d. A lattice that sits out a step (its step
// budget is spent) is passed over in one jump: the item loop continues from
// there, so its tiles cost nothing however many there are.
__device__ __forceinline__ int last_item_of(const LatDesc& d, int item) {
    const int stride = (int)gridDim.x;
    return item + (d.item_begin + d.items - 1 - item) / stride * stride;
}

// Observe the state at sub-step j of this chunk?
__device__ __forceinline__ bool observe_now(const LatDesc& d, int j) {
    if (d.obs_every <= 0) return false;
    const long long s = d.step0 + j - d.obs_base;
    return s >= 0 && (s % d.obs_every) == 0 && (s / d.obs_every) < d.obs_cap;
}


// 1 / x to within an ulp or two for a normal x far from the range limits:
// the hardware's approximate reciprocal; double: refined by one third-order
// Householder step r (1 + e + e^2), e = 1 - x r (three FP64 operations; the
// FP64 pipe bounds the FP64 kernels, a division takes over twice as many).
__device__ __forceinline__ float fast_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double fast_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = ::fma(-x, r, 1.0);
    return ::fma(::fma(e, e, e), r, r);
}

// The sums of NOBS values per lane over a warp, one of them in each lane (number
// obs_of_lane): 6 shuffles and additions, each quantity added up in a tree of 32
// values (with a butterfly for each of the four there are 20).
__device__ __forceinline__ int obs_of_lane(int lane) { return (lane & 1) * 2 + (lane >> 1 & 1); }
template <typename T>
__device__ __forceinline__ T warp_obs_sums(const T (&v)[NOBS], int lane) {
    static_assert(NOBS == 4, "two halvings");
    const bool b0 = lane & 1, b1 = lane & 2;
    const T a0 = (b0 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b0 ? v[0] : v[2], 1);
    const T a1 = (b0 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, b0 ? v[1] : v[3], 1);
    T a = (b1 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, b1 ? a0 : a1, 2);
#pragma unroll
    for (int o = 4; o <= 16; o *= 2) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// Block reduction of NOBS per-thread partial sums into out[NOBS], in a fixed
// order. Must be called by all threads of the block.
template <int NT>
__device__ __forceinline__ void block_reduce_obs(const double (&v)[NOBS], double* out, double* smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double x = warp_obs_sums(v, lane);
    if (lane < NOBS) smem[warp * NOBS + obs_of_lane(lane)] = x;
    __syncthreads();
    if (threadIdx.x < NOBS) {
        double s = 0.0;
        for (int w = 0; w < NT / 32; ++w) s += smem[w * NOBS + threadIdx.x];
        out[threadIdx.x] = s;
    }
    __syncthreads();
}

// The observables record of a state from its NOBS global sums.
__device__ __forceinline__ lbm_obs make_obs(long long step, double dt, int nx, int ny, double rho0, int probe_comp,
                                            double probe_norm, const double* tot) {
    lbm_obs o;
    o.step = step;
    o.time = (double)step * dt;
    o.mass = (double)nx * (double)ny * rho0 + tot[0];
    o.mom_x = tot[1];
    o.mom_y = tot[2];
    o.amp = probe_comp >= 0 ? probe_norm * tot[3] : 0.0;
    o.nonfinite = (isfinite(o.mass) && isfinite(o.amp) && isfinite(o.mom_x) && isfinite(o.mom_y)) ? 0 : 1;
    o.reserved = 0;
    return o;
}

// Sum of n rows of NOBS doubles by NT threads (fixed order): per-warp sums in
// red[warp][NOBS] after a barrier.
template <int NT, typename Sync>
__device__ __forceinline__ void sum_partials(const double* p, int n, int tid, double* red, Sync sync) {
    double a[NOBS] = {0.0, 0.0, 0.0, 0.0};
    for (int i = tid; i < n; i += NT) {
        const double2 u = __ldcg(reinterpret_cast<const double2*>(p + (long long)i * NOBS));
        const double2 v = __ldcg(reinterpret_cast<const double2*>(p + (long long)i * NOBS) + 1);
        a[0] += u.x;
        a[1] += u.y;
        a[2] += v.x;
        a[3] += v.y;
    }
#pragma unroll
    for (int q = 0; q < NOBS; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a[q] += __shfl_xor_sync(0xffffffffu, a[q], o);
        if ((tid & 31) == 0) red[(tid >> 5) * NOBS + q] = a[q];
    }
    sync();
}

// The sums of a lattice observed at `step`, from rows of partial sums: block b
// of a launch adds up the tiles it does (obs_tile below) and stores them as
// row `its first tile of the lattice`; the first min(grid, items) tiles belong
// to as many blocks, so those are the rows. All functions are called by NT
// threads (tid 0 .. NT - 1, `sync` a barrier of theirs); red: NT / 32 * NOBS
// doubles, flag: one int of shared memory.

// Did this block count last of `of`? Its earlier stores (by threads below
// NOBS) are visible to the block that does.
template <typename Sync>
__device__ __forceinline__ bool obs_last(unsigned* count, int of, int tid, int* flag, Sync sync) {
    if (tid < NOBS) __threadfence();
    sync();
    if (tid == 0) {
        *flag = atomicAdd(count, 1u) == (unsigned)of - 1u;
        __threadfence();
    }
    sync();
    return *flag != 0;
}
// Add up group g (OBS_GROUP rows) of the lattice's rows; the block that adds
// up the last group adds the groups up and writes the record: in a fixed
// order, whichever block it is.
template <int NT, typename Sync>
__device__ __forceinline__ void obs_add_group(const LatDesc& d, int g, int rows, long long step, int tid, double* red,
                                              int* flag, Sync sync) {
    const int groups = (int)obs_groups(rows);
    sum_partials<NT>(d.partials + (long long)g * OBS_GROUP * NOBS, min(OBS_GROUP, rows - g * OBS_GROUP), tid, red, sync);
    if (groups > 1) {
        if (tid < NOBS) {
            double t = 0.0;
            for (int w = 0; w < NT / 32; ++w) t += red[w * NOBS + tid];
            d.group_partials[(long long)g * NOBS + tid] = t;
        }
        if (!obs_last(d.obs_count + groups, groups, tid, flag, sync)) return;
        sum_partials<NT>(d.group_partials, groups, tid, red, sync);
        if (tid == 0) d.obs_count[groups] = 0;
    }
    if (tid == 0) {
        double tot[NOBS];
        for (int q = 0; q < NOBS; ++q) {
            tot[q] = 0.0;
            for (int w = 0; w < NT / 32; ++w) tot[q] += red[w * NOBS + q];
        }
        d.series[(step - d.obs_base) / d.obs_every] =
            make_obs(step, d.dt, d.nx, d.ny, d.rho0, d.probe_comp, d.probe_norm, tot);
    }
}
// A block's tile `local` of an observed lattice, its warps' sums in red[warp]
// [NOBS]: they are added up (across warps and tiles in double, in threads below
// NOBS) and the block's last tile of the lattice stores its row. With `finish` the block that completes OBS_GROUP
// rows goes on as above: no launch after the step (two such launches took 5 us
// of every recorded step of a small lattice). Without it a launch of
// obs_finish_kernel does: where a launch has thousands of blocks, a fence and
// a count in each of them cost more (CS 8192^2: 0.767 ms per step against
// 0.745).
template <int NT, typename Sync>
__device__ __forceinline__ void obs_warp_sums(const LatDesc& d, int local, long long step, int tid, double& run,
                                              double* red, int* flag, Sync sync, bool finish) {
    sync();
    const int grid = (int)gridDim.x;
    if (tid < NOBS) {
        double s = 0.0;
        for (int w = 0; w < NT / 32; ++w) s += red[w * NOBS + tid];
        run = local < grid ? s : run + s;
    }
    if (local + grid >= d.items) {
        const int row = local % grid, rows = min(grid, d.items), g = row / OBS_GROUP;
        if (tid < NOBS) d.partials[(long long)row * NOBS + tid] = run;
        if (finish && obs_last(d.obs_count + g, min(OBS_GROUP, rows - g * OBS_GROUP), tid, flag, sync)) {
            if (tid == 0) d.obs_count[g] = 0;
            obs_add_group<NT>(d, g, rows, step, tid, red, flag, sync);
        }
    }
    sync();   // red and flag are free again
}
// The same from the threads' sums v, added up per warp in T: 32 of them in
// float, each of them a float sum over the thread's nodes (CS: 1 to 4, bulk
// tiles up to 32; temporally blocked FD step: 1).
template <typename T, int NT, typename Sync>
__device__ __forceinline__ void obs_tile(const T (&v)[NOBS], const LatDesc& d, int local, long long step, int tid,
                                         double& run, double* red, int* flag, Sync sync, bool finish) {
    // (warp_obs_sums would take fewer shuffles, and CS 128 x 1 from 64 registers to
    // 72: 2048^2, not recorded, 60.5 -> 64.1 us per step)
#pragma unroll
    for (int q = 0; q < NOBS; ++q) {
        T x = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((tid & 31) == 0) red[(tid >> 5) * NOBS + q] = (double)x;
    }
    obs_warp_sums<NT>(d, local, step, tid, run, red, flag, sync, finish);
}

}  // namespace lbm
