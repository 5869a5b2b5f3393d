// Finite-difference LB update (Sec. 2): Eq. (evolution) in conservative form
//     d f_k/dt = L(f)_k = -v_kx D_x f_k - v_ky D_y f_k - (f_k - f^eq_k) / tau,
// advected with WENO-5 (Jiang-Shu) and advanced with the three-stage TVD
// (SSP) Runge-Kutta scheme in Shu-Osher form:
//     f1 = f + dt L(f);  f2 = 3/4 f + 1/4 (f1 + dt L(f1));
//     f^{n+1} = 1/3 f + 2/3 (f2 + dt L(f2)).
// One launch = one stage for every lattice of the group. The moments (rho, u)
// and so f^eq are taken from that stage's input, as the BGK term belongs to L.
//
// Per tile (TX x TY nodes), two kinds of warps of a block:
//   preparing warps, one tile ahead of the others: copy every population of
//   the stage input with a periodic halo of 3 nodes (the WENO-5 stencil reach)
//   to shared memory and form the moments of the tile's nodes,
//   march warps: each takes one population up the rows of the tile. Along y
//   the stencil slides in registers (an interface value is computed once, as
//   the face above a row and then the face below the next); along x a lane
//   computes the faces on the upwind side of its nodes and takes the others
//   from the neighbouring lane. Both sides of an interface use the same value,
//   so the flux form is conservative. The node then adds the BGK term and
//   combines with f^n for the stage.
// The WENO-5 face value is upwinded by the sign of the (constant) velocity
// component: for v > 0 the face i+1/2 is reconstructed from f_{i-2..i+2},
// for v < 0 from f_{i+3..i-1} (mirror image). Components equal to 0 (the
// 3- and 5-node sets) do not advect along that axis.
//
// Buffers: buf[0] = f^n (updated in place by stage 3: it is read only at the
// node being written, by the thread writing it), buf[1] = f^(1),
// buf[2] = f^(2). Storage offset as in the CS kernel (deviation form for
// FP32, full f for FP64): WENO differences and the stage combination are
// unchanged by the constant offset w_k rho0.
#include <atomic>

#include "fd_common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace lbm {

// Column sums cs[ix] = sum_iy g(ix + Q1 iy) and row sums rs[iy] =
// sum_ix g(ix + Q1 iy) of a quantity over the product set, then its zeroth
// and first moments sum g, sum g v_x, sum g v_y (v_x depends on ix only, v_y
// on iy only): fewer operations than K products per component.
template <typename T, int Q1, typename Fn>
__device__ __forceinline__ void set_moments(Fn g, typename Lanes<T>::V& m0, typename Lanes<T>::V& mx,
                                            typename Lanes<T>::V& my) {
    using P = Lanes<T>;
    using V = typename P::V;
    V cs[Q1], rs[Q1];
#pragma unroll
    for (int iy = 0; iy < Q1; ++iy)
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) {
            const V v = g(ix + Q1 * iy);
            cs[ix] = iy == 0 ? v : P::add(cs[ix], v);
            rs[iy] = ix == 0 ? v : P::add(rs[iy], v);
        }
    m0 = cs[0];
#pragma unroll
    for (int i = 1; i < Q1; ++i) m0 = P::add(m0, cs[i]);
    mx = P::mulc(cs[0], (T)GH<Q1>::v(0));
    my = P::mulc(rs[0], (T)GH<Q1>::v(0));
#pragma unroll
    for (int i = 1; i < Q1; ++i) {
        if (GH<Q1>::v(i) != 0.0) {
            mx = P::fmac(cs[i], (T)GH<Q1>::v(i), mx);
            my = P::fmac(rs[i], (T)GH<Q1>::v(i), my);
        }
    }
}

// The equilibrium at a node as five numbers, p = u / 2, j = rho u and e0 =
// dr - j . p: stored f^eq_k / w_k = (v_k . p)(v_k . j) + v_k . j + e0, i.e. Eq.
// (herfeq) minus w_k rho0. FP32 takes (1 + v_k . p)(v_k . j) + e0: five
// operations, as many as the square of one product with p = j / sqrt(2 rho)
// takes, and like Eq. (herfeq) defined for every density but zero.
template <typename T>
struct Equil {
    using P = Lanes<T>;
    using V = typename P::V;
    V px, py, jx, jy, e0;
    __device__ __forceinline__ void set(V rho, V dr, V jx_, V jy_) {
        jx = jx_;
        jy = jy_;
        const V h = P::mulc(P::rcp_node(rho), T(0.5));
        px = P::mul(jx, h);
        py = P::mul(jy, h);
        e0 = P::fma(P::neg(jy), py, P::fma(P::neg(jx), px, dr));
    }
    // (f^eq_k) / w_k; vx, vy: the population's velocity, broadcast
    __device__ __forceinline__ V over_w(V vx, V vy) const {
        const V xj = P::fma(vx, jx, P::mul(vy, jy));
        if constexpr (sizeof(T) == 4) {
            return P::fma(P::fma(vx, px, P::fma(vy, py, P::sp(T(1)))), xj, e0);
        } else {
            const V xi = P::fma(vx, px, P::mul(vy, py));
            return P::add(P::fma(xi, xj, xj), e0);
        }
    }
};

// The same for all populations of a set in turn (compile-time k), with the
// terms in v_y formed once per row of the product set. The operations and
// their order are Equil::over_w's: the residual moments below have to be those
// of the equilibrium the update uses, to the last bit (with products and sums
// rounded apart here, the FP32 decay rate of an IMEX run is off by 2.6e-4).
template <typename T, int Q1>
struct EquilAll {
    using P = Lanes<T>;
    using V = typename P::V;
    V px, jx, yp[Q1], yj[Q1], e0;
    __device__ __forceinline__ explicit EquilAll(const Equil<T>& e) : px(e.px), jx(e.jx), e0(e.e0) {
#pragma unroll
        for (int i = 0; i < Q1; ++i) {
            const T v = (T)GH<Q1>::v(i);
            yp[i] = sizeof(T) == 4 ? P::fmac(e.py, v, P::sp(T(1))) : P::mulc(e.py, v);
            yj[i] = P::mulc(e.jy, v);
        }
    }
    // f^eq_k / w_k
    __device__ __forceinline__ V over_w(int k) const {
        const int ix = k % Q1, iy = k / Q1;
        const T v = (T)GH<Q1>::v(ix);
        const V xi = P::fmac(px, v, yp[iy]), vj = P::fmac(jx, v, yj[iy]);
        if constexpr (sizeof(T) == 4) return P::fma(xi, vj, e0);
        else return P::add(P::fma(xi, vj, vj), e0);
    }
};

// Velocity tables of a product set for run-time population indices; the
// values are those the unrolled loops fold to immediates.
template <typename T, int Q1>
struct SetTable {
    T vx[Q1 * Q1], vy[Q1 * Q1], w[Q1 * Q1];
    constexpr SetTable() : vx{}, vy{}, w{} {
        for (int k = 0; k < Q1 * Q1; ++k) {
            vx[k] = (T)vx_of<Q1>(k);
            vy[k] = (T)vy_of<Q1>(k);
            w[k] = (T)w_of<Q1>(k);
        }
    }
};
template <typename T, int Q1>
__constant__ SetTable<T, Q1> c_set{};

// Geometry of a tile: TX = 32 nodes along x by TY rows. A lane holds N
// neighbouring nodes of a row (Lanes<T>::V: a pair for FP32, so that every
// packed FP32x2 instruction does the same arithmetic for two nodes; one for
// FP64); a row takes LC = 32 / N lanes and the N row groups of a warp lie H =
// TY / N rows apart. A population's staged tile has RT = TY + 6 rows of HXP =
// 40 columns, x0 - 4 .. x0 + 35 (16-byte aligned; the stencils need x0 - 3 ..
// x0 + 34). Rows are marched in the direction of v_y by a run-time row stride,
// so the code differs only by the sign of v_x and stays in the instruction
// cache.
constexpr int FD_TX = 32;
constexpr int FD_HXP = 40;

template <typename T, int Q1, int TY, bool IMEX>
struct FdGeo {
    static constexpr int N = Lanes<T>::N;
    static constexpr int K = Q1 * Q1;
    static constexpr int H = TY / N;
    static constexpr int RT = TY + 6;
    static constexpr int PL = RT * FD_HXP;
    // A march is one population and S-th of the tile's rows (9 velocities:
    // halves, for more warps; tiles of 4 rows too: 88 x 152, 15.3 -> 11.7 us
    // per step). Warps per block: NM march warps, NA preparing.
    static constexpr int S = Q1 == 3 && sizeof(T) == 4 && H >= 2 ? 2 : 1;
    static constexpr int HS = H / S;
    static constexpr int NM = Q1 == 5 ? 13 : K * S;
    // IMEX prepares more: with four preparing warps 9 velocities take 575 us
    // per step of 2048^2, with eight 494.
    static constexpr int NA = Q1 == 4 || S == 2 ? (IMEX ? 8 : 4) : 7;
    static constexpr int NT = (NM + NA) * 32;
    static constexpr size_t n_mom = (size_t)5 * TY * FD_TX;
    static constexpr size_t n_edge = ((size_t)K * TY + 3) / 4 * 4;
    static constexpr size_t buf = (size_t)K * PL + n_mom + n_edge;   // values of a tile buffer
    // two tile buffers (the next item is prepared while one is marched) where
    // they fit the device's 227 KiB next to 3 KiB of static shared memory
    static constexpr int NB = sizeof(T) * 2 * buf + sizeof(double) * NA * NOBS <= 224 * 1024 ? 2 : 1;
    static constexpr size_t bytes = sizeof(T) * NB * buf + sizeof(double) * NA * NOBS;
};

// N neighbouring values from shared or global memory (aligned to the pair).
__device__ __forceinline__ float2 ldv(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ double ldv(const double* p) { return *p; }
__device__ __forceinline__ void stv(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ void stv(double* p, double v) { *p = v; }
__device__ __forceinline__ void ldv2(const float* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ldv2(const double* p, double& a, double& b) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    a = v.x;
    b = v.y;
}
__device__ __forceinline__ void stv2(float* p, float2 a, float2 b) {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void stv2(double* p, double a, double b) { *reinterpret_cast<double2*>(p) = make_double2(a, b); }
// Read again instead of kept in registers since the last read.
__device__ __forceinline__ float2 ldv_again(const float* p) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(smem_addr(p)));
    return v;
}
__device__ __forceinline__ double ldv_again(const double* p) { return *p; }
// The same through global addresses (the state pointers come from memory, so
// the compiler takes them for generic ones).
__device__ __forceinline__ float2 ldg_v(const float* p) {
    float2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(__cvta_generic_to_global(p)));
    return v;
}
__device__ __forceinline__ double ldg_v(const double* p) {
    double v;
    asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(__cvta_generic_to_global(p)));
    return v;
}
__device__ __forceinline__ void stg_v(float* p, float2 v) {
    asm volatile("st.global.v2.f32 [%0], {%1, %2};" ::"l"(__cvta_generic_to_global(p)), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void stg_v(double* p, double v) {
    asm volatile("st.global.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "d"(v) : "memory");
}
__device__ __forceinline__ void stg_1(float* p, float v) {
    asm volatile("st.global.f32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "f"(v) : "memory");
}
__device__ __forceinline__ void stg_1(double* p, double v) { stg_v(p, v); }

// The node differences d1 .. d4 (weno5_diff) of the x-face on the upwind side
// of a lane's nodes, from row pointer t (column -4 of the lane's first node);
// SX: sign of v_x. Returns the nodes' own values.
template <int SX>
__device__ __forceinline__ float2 x_diffs(const float* t, float2& d1, float2& d2, float2& d3, float2& d4) {
    const float2 B = ldv(t + 2), C = ldv(t + 4), E = ldv(t + 6);
    if constexpr (SX > 0) {
        const float2 A = ldv(t);
        d1 = make_float2(A.y - B.x, B.x - B.y);
        d2 = make_float2(B.x - B.y, B.y - C.x);
        d3 = make_float2(B.y - C.x, C.x - C.y);
        d4 = make_float2(C.x - C.y, C.y - E.x);
    } else {
        const float2 G = ldv(t + 8);
        d1 = make_float2(E.y - E.x, G.x - E.y);
        d2 = make_float2(E.x - C.y, E.y - E.x);
        d3 = make_float2(C.y - C.x, E.x - C.y);
        d4 = make_float2(C.x - B.y, C.y - C.x);
    }
    return C;
}
template <int SX>
__device__ __forceinline__ double x_diffs(const double* t, double& d1, double& d2, double& d3, double& d4) {
    const double a = t[4 - 3 * SX], b = t[4 - 2 * SX], c = t[4 - SX], d = t[4], e = t[4 + SX];
    d1 = a - b;
    d2 = b - c;
    d3 = c - d;
    d4 = d - e;
    return d;
}
// The faces on the downwind side of a lane's nodes: those on the upwind side
// of the next nodes in the direction of v_x, the outermost lane's from `edge`.
template <int SX>
__device__ __forceinline__ float2 x_next(float2 f, float edge, bool outer) {
    if constexpr (SX > 0) {
        const float n = __shfl_down_sync(0xffffffffu, f.x, 1);
        return make_float2(f.y, outer ? edge : n);
    } else {
        const float n = __shfl_up_sync(0xffffffffu, f.y, 1);
        return make_float2(outer ? edge : n, f.x);
    }
}
template <int SX>
__device__ __forceinline__ double x_next(double f, double edge, bool outer) {
    const double n = SX > 0 ? __shfl_down_sync(0xffffffffu, f, 1) : __shfl_up_sync(0xffffffffu, f, 1);
    return outer ? edge : n;
}

template <int S>
struct Const {
    static constexpr int value = S;
};

// IMEX-SSP2(2,2,2) (LBM_TS_IMEX): gamma of the implicit tableau, 1 - 1/sqrt 2.
constexpr double IMEX_GAMMA = 0.29289321881345247560;

// What bounds it. FP32: the register file and the FP32 pipe. A packed FP32x2
// multiply-add with three distinct operand pairs issues every 3.2 cycles, with
// two every 2.2 (measured), so operands count as much as operations: literals
// go into scalar instructions as immediates, products that share a term are
// folded. FP64: the FP64 pipe (1/64 of the FP32 rate).
// Why this split. With every warp doing all parts of a tile in turn, copies,
// barriers and the moments left the pipe idle for half of the time (1.19 ms
// per stage of FD 16-velocity 4096^2 FP32 however the tile was cut). Here the
// preparing warps' work overlaps the march, which never waits for memory: f^n
// is loaded a march ahead, the rest is in shared memory. Stages of that lattice:
// 1.19 / 1.13 / 1.13 -> 0.98 / 0.98 / 0.99 ms; FP64 256^2: 275 -> 198 us per stage
// (fewer operations per face and node, one reciprocal instead of a division).
// Named barriers hand the buffers over: waiting warps take no issue slots
// (polling an mbarrier took 10% of them).
//
// One stage of the FD update. IMEX = false: SSP-RK3 stage `stage` (1..3).
// IMEX = true: stage 1 or 2 of IMEX-SSP2(2,2,2) with explicit WENO-5
// advection A and implicit BGK C. With Y_i the stage values (below), the
// scheme's
//   Y_2 = f^n + dt A(Y_1) + (1 - 2g) dt C(Y_1) + g dt C(Y_2),
//   f^{n+1} = f^n + dt/2 (A(Y_1) + A(Y_2) + C(Y_1) + C(Y_2))
// are evaluated as: stage 1 stages f^n, maps it to Y_1, and writes
//   Z = f^n + dt A(Y_1) + (1 - 2g) dt C(Y_1)      (buffer 1)
//   P = f^n + 2g dt C(Y_1)                          (buffer 2);
// stage 2 stages Z, maps it to Y_2, and writes
//   f^{n+1} = P + ((Z - P) + dt A(Y_2) + dt C(Y_2)) / 2   (buffer 0),
// with dt C(Y_i) = -(dt/tau) (u_i - f^eq(u_i)) / (1 + lam), u_i the stage's
// input (f^n or Z): no difference of nearly equal values is multiplied by
// dt/tau, so the rounding stays small however stiff the collision is.
template <typename T, int Q1, int TY, bool IMEX>
__global__ void __launch_bounds__(FdGeo<T, Q1, TY, IMEX>::NT, 1) fd_stage_kernel(GroupDev g, int j, int stage) {
    using Ge = FdGeo<T, Q1, TY, IMEX>;
    using P = Lanes<T>;
    using V = typename P::V;
    constexpr int K = Ge::K, N = Ge::N, H = Ge::H, RT = Ge::RT, PL = Ge::PL, NM = Ge::NM, NA = Ge::NA, NB = Ge::NB, S = Ge::S,
                  HS = Ge::HS;
    constexpr int TX = FD_TX, HXP = FD_HXP, LC = TX / N;
    constexpr int VEC = 16 / (int)sizeof(T);   // values per 16-byte copy
    constexpr int CH = HXP / VEC;              // 16-byte chunks per staged row
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // NB tile buffers: [K][RT][HXP] staged values; per node the corrected
    // moments, [TY][TX / N][2] (px, py), the same (jx, jy), [TY][TX] e0; [K][TY]
    // faces beyond the outermost lane. Named barriers hand them over (2, 3:
    // prepared; 4, 5: marched)
    T* bufs = reinterpret_cast<T*>(smem_raw);
    double* red = reinterpret_cast<double*>(bufs + NB * Ge::buf);
    // the lattices' first items and whether they sit this step out (up to
    // LATS of them; more are looked up in global memory), and the block's items
    // in turn with their lattices' descriptors and tile origins
    constexpr int LATS = 256;
    __shared__ int s_begin[LATS];
    __shared__ unsigned char s_dead[LATS];
    __shared__ __align__(16) LatDesc s_desc[4];
    __shared__ int s_item[4];
    __shared__ int s_last;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int grp = lane / LC, c0 = (lane % LC) * N;   // row group and first column of the lane's nodes
    constexpr int DCH = sizeof(LatDesc) / 16;          // 16-byte chunks of a descriptor
    static_assert(sizeof(LatDesc) % 16 == 0 && DCH <= 32, "descriptors are copied in 16-byte chunks by one warp");
    wait_for_previous_launch();
    // a lone lattice's descriptor is read while the group's header is on its way
    if (tid < DCH) reinterpret_cast<uint4*>(s_desc)[tid] = reinterpret_cast<const uint4*>(g.desc)[tid];
    const int n_lat = g.hdr[0];
    const int total = g.hdr[1];
    if (n_lat > 1 && n_lat <= LATS)
        for (int i = tid; i < n_lat; i += Ge::NT) {
            s_begin[i] = g.item_begin[i];
            s_dead[i] = (long long)j >= g.desc[i].remaining;
        }
    __syncthreads();
    const int in_idx = IMEX ? (stage == 1 ? 0 : 1) : (stage == 1 ? 0 : (stage == 2 ? 1 : 2));
    const int out_idx = IMEX ? (stage == 1 ? 1 : 0) : (stage == 1 ? 1 : (stage == 2 ? 2 : 0));
    // the stage reads its input at its own node from global memory too (IMEX:
    // the staged tile holds the stage values Y instead), and f^n (RK3 stages 2, 3)
    const bool node_in = IMEX || stage != 1;

    if (warp >= NM) {
        // ---- preparing warps: look up the block's items, copy their tiles,
        //      form their moments and outer faces, one item ahead of the march
        const int aw = warp - NM, atid = tid - NM * 32;
        auto live_item = [&](int item, int& li) {
            // first item from `item` on whose lattice still has steps to run
            // (`total` or beyond: none), and that lattice
            for (; item < total; item += gridDim.x) {
                li = 0;
                int end = total;
                bool dead;
                if (n_lat == 1) {
                    dead = (long long)j >= s_desc[0].remaining;
                } else if (n_lat <= LATS) {
                    int hi = n_lat - 1;
                    while (li < hi) {
                        const int mid = (li + hi + 1) >> 1;
                        if (s_begin[mid] <= item) li = mid;
                        else hi = mid - 1;
                    }
                    if (li + 1 < n_lat) end = s_begin[li + 1];
                    dead = s_dead[li];
                } else {
                    li = find_lattice_warp(g.item_begin, n_lat, item, lane);
                    dead = (long long)j >= g.desc[li].remaining;
                    if (dead) end = g.desc[li].item_begin + g.desc[li].items;
                }
                if (!dead) break;
                item += (end - 1 - item) / (int)gridDim.x * (int)gridDim.x;   // passed over in one jump
            }
            return item;
        };
        // the item at or after `item` into slot s (one warp, asynchronous copy;
        // a lone lattice's descriptor is in slot 0 already)
        auto look_up = [&](int item, int s) {
            int li = 0;
            item = live_item(item, li);
            if (lane == 0) s_item[s] = item;
            if (item < total && lane < DCH && (n_lat > 1 || s != 0))
                cp_async16(reinterpret_cast<uint4*>(s_desc + s) + lane, reinterpret_cast<const uint4*>(g.desc + li) + lane);
        };
        constexpr int NIT = (RT * CH + 31) / 32;   // chunks of a population's tile per lane
        if (aw == 0) look_up(blockIdx.x, 0);
        cp_async_wait_all();
        named_sync(1, NA * 32);
        double run = 0.0;   // observables of this block's tiles so far
        for (unsigned n = 0;; ++n) {
            const int slot = n & 3;
            const int b = NB == 2 ? n & 1 : 0;
            T* const buf = bufs + b * Ge::buf;
            T* const mo = buf + (size_t)K * PL;
            T* const edges = mo + Ge::n_mom;
            if (n >= NB) named_sync(4 + b, Ge::NT);
            const int item = s_item[slot];
            if (item >= total) {   // the march warps stop too
                // a block takes its SM whole, so the next launch's blocks have
                // no place before this one ends: let in at the start, they only
                // kept SMs that were free from other streams (and 1 to 3% slower)
                allow_next_launch();
                named_arrive(2 + b, Ge::NT);
                if (NB == 2 && n >= 1) named_sync(4 + (1 - b), Ge::NT);
                break;
            }
            const LatDesc* const cp = s_desc + slot;
            const int local = item - cp->item_begin;
            const int x0 = local % cp->tiles_x * TX, y0 = local / cp->tiles_x * TY;
            const int nx = cp->nx, ny = cp->ny, pitch = cp->pitch;
            const long long plane = cp->plane;
            // 1. the K halo tiles of the stage input: 16-byte asynchronous
            //    copies (rows are 16-byte aligned: x0 - 4 is a multiple of 4, the
            //    pitch of 32). At the periodic edge a chunk wraps as a whole when
            //    nx is a multiple of VEC; otherwise the few columns of the chunks
            //    that cross it (before x = 0, and from the last chunk's start to
            //    nx + 2) go value by value, spread over all preparing lanes, each
            //    with one column's offset for all populations (wrapping every
            //    value of every such chunk in the lane of its copy took half as
            //    long again as the next width that is a multiple of 4: FD
            //    16-velocity 750 x 322 FP32, 112 -> 74 us per step; 9-velocity
            //    IMEX 68 -> 51). Columns that no node of the lattice reaches
            //    (beyond nx + 2) are left out.
            //    Offsets are below 2^32: a plane's elements times the three
            //    buffers fit the device.
            const T* const U0 = static_cast<const T*>(cp->buf[in_idx]);
            const bool interior = x0 >= 4 && x0 + TX + 4 <= nx && y0 >= 3 && y0 + TY + 3 <= ny;
            unsigned so[NIT], whole = 0;   // one bit per chunk of the lane
#pragma unroll
            for (int i = 0; i < NIT; ++i) {
                const int q = lane + 32 * i, r = q / CH, c = (q - r * CH) * VEC;
                const int y = y0 - 3 + r, x = x0 - 4 + c;
                if (((i + 1) * 32 <= RT * CH || q < RT * CH) &&
                    (interior || (x < nx + 3 && (nx % VEC == 0 || (x >= 0 && x + VEC <= nx)))))
                    whole |= 1u << i;
                so[i] = interior ? (unsigned)y * (unsigned)pitch + (unsigned)x
                                 : (unsigned)wrap_near(y, ny) * (unsigned)pitch + (unsigned)wrap_near(x, nx);
            }
            for (int k = aw; k < K; k += NA) {
                const T* U = U0 + k * plane;
                T* t = buf + k * PL + lane * VEC;
#pragma unroll
                for (int i = 0; i < NIT; ++i) {
                    if ((whole >> i) & 1u) {
                        const T* s = U + so[i];
                        if (LBM_BC_NODE(cp, K, s - U0) && LBM_BC_NODE(cp, K, s - U0 + VEC - 1)) cp_async16(t + 32 * VEC * i, s);
                    }
                }
            }
            if (nx % VEC != 0 && (x0 == 0 || x0 + TX + 3 > nx - nx % VEC)) {
                const int xr = nx - nx % VEC;   // first column of the chunk across nx
                const int nl = x0 == 0 ? 3 : 0, nr = max(min(nx + 3, x0 + TX + 3) - xr, 0);
                for (int p = atid; p < RT * (nl + nr); p += NA * 32) {
                    const int r = p / (nl + nr), e = p - r * (nl + nr);
                    const int x = e < nl ? e - 3 : xr + e - nl;
                    const T* s = U0 + ((unsigned)wrap_near(y0 - 3 + r, ny) * (unsigned)pitch + (unsigned)wrap_near(x, nx));
                    T* t = buf + r * HXP + (x - x0 + 4);
#pragma unroll 1
                    for (int k = 0; k < K; ++k, s += plane, t += PL)
                        if (LBM_BC_NODE(cp, K, s - U0)) cp_async_small<sizeof(T)>(t, s);
                }
            }
            // the next item's descriptor travels with the copies
            if (aw == 0) look_up(item + gridDim.x, (n + 1) & 3);
            const T r0 = lat_val<T>(cp->rho0, cp->rho0_f);
            const V eps = P::sp(lat_val<T>(cp->eps, cp->eps_f) * T(0.75));
            const bool obs = stage == 1 && observe_now(*cp, j);
            cp_async_wait_all();
            named_sync(1, NA * 32);
            // population k at tile row r, column c (halo: negative and beyond
            // TY, TX)
            auto at = [&](int k, int r, int c) {
                return buf + k * PL + (r + 3) * HXP + c + 4;
            };
            // FP32: the map below sums the moments of Y, kept for the tile's own nodes (a
            // pass of their own took 1 to 3% of a step); FP64, whose pipe is the
            // bound, sums them for the tile's nodes only (map: 2 to 7% slower)
            constexpr bool SUM_Y = IMEX && sizeof(T) == 4;
            if constexpr (IMEX) {
                // the implicit BGK part of the stage in closed form, at every
                // staged node: the stage value Y solves Y = u + dt g C(Y), C(Y) =
                // -(Y - f^eq(Y)) / tau; the collision conserves rho and rho u
                // (Eq. herfeq has the moments of Eq. f_moments_discrete), so
                // f^eq(Y) = f^eq(u) and Y = (u + lam f^eq(u)) / (1 + lam). Values
                // in the storage form: the map is linear, the offsets carry over.
                // lam = g dt/tau, il = 1/(1 + lam)
                const V vlam = P::mulc(P::sp(lat_val<T>(cp->dt_tau, cp->dt_tau_f)), T(IMEX_GAMMA));
                const V vil = P::sp(T(1) / P::get(P::add(P::sp(T(1)), vlam), 0));
                for (int pos = atid; pos < RT * (HXP / N); pos += NA * 32) {
                    const int r = pos / (HXP / N) - 3, c = pos % (HXP / N) * N - 4;
                    V dr, jx, jy;
                    set_moments<T, Q1>([&](int k) { return ldv(at(k, r, c)); }, dr, jx, jy);
                    Equil<T> e;
                    e.set(P::add(P::sp(r0), dr), dr, jx, jy);
                    const EquilAll<T, Q1> ea(e);
                    auto map = [&](int k) {
                        const V geq = P::mulc(ea.over_w(k), (T)w_of<Q1>(k));
                        T* u = at(k, r, c);
                        const V y = P::mul(P::fma(vlam, geq, ldv_again(u)), vil);
                        stv(u, y);
                        return y;
                    };
                    if constexpr (SUM_Y) {
                        set_moments<T, Q1>(map, dr, jx, jy);
                        if (r >= 0 && r < TY && c >= 0 && c < TX) {
                            e.set(P::add(P::sp(r0), dr), dr, jx, jy);
                            T* m = mo + 2 * (r * TX + c);
                            stv2(m, e.px, e.py);
                            stv2(m + 2 * TY * TX, e.jx, e.jy);
                            stv(mo + 4 * TY * TX + r * TX + c, e.e0);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < K; ++k) map(k);
                    }
                }
                named_sync(1, NA * 32);
            }

            // 2. per warp, one of: the moments of a row of each group (Eq.
            //    f_moments_discrete) with the observables of the state; the
            //    faces beyond the outermost lane, one (population, rows) per lane
            double sum = 0.0;   // of observable obs_of_lane(lane) over the warp's nodes
            constexpr int KX = Q1 * (Q1 - Q1 % 2);   // populations with faces along x
            constexpr int NE = (KX * H + 31) / 32;
            for (int task = aw; task < H + NE; task += NA) {
                if (task < H) {
                    const int r = task + grp * H;   // tile row
                    T* m = mo + 2 * (r * TX + c0);
                    Equil<T> e;
                    if (!SUM_Y || obs) {
                        V dr, jx, jy;
                        set_moments<T, Q1>([&](int k) { return ldv(at(k, r, c0)); }, dr, jx, jy);
                        const V rho = P::add(P::sp(r0), dr);
                        if (obs) {
                            // one node of each lane is added up per warp in T (32
                            // float values, as with a node per thread), the rest
                            // in double
                            const int pc = cp->probe_comp, y = y0 + r;
#pragma unroll 1
                            for (int h = 0; h < N; ++h) {
                                const int x = x0 + c0 + h;
                                T v[NOBS] = {T(0), T(0), T(0), T(0)};
                                if (x < nx && y < ny) {
                                    v[0] = P::get(dr, h);
                                    v[1] = P::get(jx, h);
                                    v[2] = P::get(jy, h);
                                    if (pc >= 0) {
                                        T pxv, pyv;
                                        if constexpr (sizeof(T) == 4) {
                                            pxv = cp->probe_pxf[x];
                                            pyv = cp->probe_pyf[y];
                                        } else {
                                            pxv = cp->probe_px[x];
                                            pyv = cp->probe_py[y];
                                        }
                                        v[3] = (pc == 0 ? P::get(jx, h) : P::get(jy, h)) / P::get(rho, h) * pxv * pyv;
                                    }
                                }
                                sum += (double)warp_obs_sums(v, lane);
                            }
                        }
                        if constexpr (!SUM_Y) e.set(rho, dr, jx, jy);
                    }
                    if constexpr (SUM_Y) {
                        ldv2(m, e.px, e.py);
                        ldv2(m + 2 * TY * TX, e.jx, e.jy);
                        e.e0 = ldv(mo + 4 * TY * TX + r * TX + c0);
                    }
                    // FP32: residual moments of the collision term. In exact
                    // arithmetic sum_k (u_k - geq_k) (1, v_k) = 0; in float32 the
                    // rounding of the moments and of geq leaves a residual of
                    // ~1e-7 of the momentum per stage, which is not small next to
                    // the viscous decay per stage of a slowly decaying flow. It is
                    // computed from the differences u_k - geq_k (accurate) and
                    // removed with w_k (R0 + v_k . R1), which has exactly these
                    // moments (quadrature identities of the set): the equilibrium
                    // takes the shifted moments dr + R0, j + R1 (p . R1, which the
                    // shifted j adds to its zeroth moment, is taken off e0).
                    if constexpr (sizeof(T) == 4) {
                        const T* U = static_cast<const T*>(cp->buf[in_idx]) + ((long long)(y0 + r) * pitch + x0 + c0);
                        const bool in = y0 + r < ny && x0 + c0 < nx;
                        const EquilAll<T, Q1> ea(e);
                        V R0, R1x, R1y;
                        set_moments<T, Q1>(
                            [&](int k) {
                                const V ew = ea.over_w(k);
                                V u;
                                if constexpr (IMEX)   // the stage input (the tile holds the stage values)
                                    u = in && LBM_BC_NODE(cp, K, U - static_cast<const T*>(cp->buf[in_idx]) + k * plane)
                                            ? ldv(U + k * plane) : P::sp(T(0));
                                else
                                    u = ldv_again(at(k, r, c0));
                                return P::fmac(ew, -(T)w_of<Q1>(k), u);
                            },
                            R0, R1x, R1y);
                        e.e0 = P::add(e.e0, P::fma(P::neg(e.py), R1y, P::fma(P::neg(e.px), R1x, R0)));
                        e.jx = P::add(e.jx, R1x);
                        e.jy = P::add(e.jy, R1y);
                    }
                    stv2(m, e.px, e.py);
                    stv2(m + 2 * TY * TX, e.jx, e.jy);
                    stv(mo + 4 * TY * TX + r * TX + c0, e.e0);
                } else {
                    const int q = (task - H) * 32 + lane;
                    const int i = q / H, r = q - i * H;   // march row (of each group)
                    // the i-th population whose v_x is not 0
                    const int k = Q1 % 2 == 0 ? i : i + (i + Q1 / 2) / (Q1 - 1);
                    if (i < KX) {
                        const bool mx = 2 * (k % Q1) + 1 < Q1;
                        const int st = mx ? -1 : 1;
                        const bool my = 2 * (k / Q1) + 1 < Q1;
                        const T* a = buf + k * PL + (my ? RT - 4 - r : r + 3) * HXP + (mx ? 6 : TX + 1);
                        const T* b = a + (my ? 1 - N : N - 1) * H * HXP;
                        const V f = weno5_vals<P, T>(P::mk(a[0], b[0]), P::mk(a[st], b[st]), P::mk(a[2 * st], b[2 * st]),
                                                     P::mk(a[3 * st], b[3 * st]), P::mk(a[4 * st], b[4 * st]), eps);
                        edges[k * TY + r] = P::get(f, 0);
                        edges[k * TY + r + (N - 1) * H] = P::get(f, N - 1);
                    }
                }
            }
            if (obs) {
                if (lane < NOBS) red[aw * NOBS + obs_of_lane(lane)] = sum;
                obs_warp_sums<NA * 32>(*cp, local, cp->step0 + j, atid, run, red, &s_last,
                                       [] { named_sync(1, NA * 32); }, g.finish_obs != 0);
            }
            named_arrive(2 + b, Ge::NT);
        }
        return;
    }

    // ---- march warps
    // stage weights: f^(s) = f^n + cb ((u - f^n) + dt L(u)), i.e. the Shu-Osher
    // combinations 3/4 f^n + 1/4 (u + dt L(u)) and 1/3 f^n + 2/3 (u + dt L(u))
    const V cb = P::sp(stage == 1 ? T(1) : (stage == 2 ? T(0.25) : T(2.0 / 3.0)));
    for (unsigned n = 0;; ++n) {
        const int slot = n & 3;
        const int b = NB == 2 ? n & 1 : 0;
        T* const buf = bufs + b * Ge::buf;
        const T* const mom = buf + (size_t)K * PL;
        const T* const edges = mom + Ge::n_mom;
        named_sync(2 + b, Ge::NT);
        const int item = s_item[slot];
        if (item >= total) break;
        const LatDesc* const cp = s_desc + slot;
        const int local = item - cp->item_begin;
        const int x0 = local % cp->tiles_x * TX, y0 = local / cp->tiles_x * TY;
        const int nx = cp->nx, ny = cp->ny, pitch = cp->pitch;
        const long long plane = cp->plane;
        const T cdx = lat_val<T>(cp->cdx, cp->cdx_f);
        const T dtt = lat_val<T>(cp->dt_tau, cp->dt_tau_f);
        const V eps = P::sp(lat_val<T>(cp->eps, cp->eps_f) * T(0.75));
        // IMEX: (dt/tau) / (1 + lam)
        [[maybe_unused]] const T c1 = dtt / P::get(P::add(P::sp(T(1)), P::mulc(P::sp(dtt), T(IMEX_GAMMA))), 0);

        auto march = [&](auto sx_, auto full_, int k, int seg, const T* tk) {
            constexpr int SX = decltype(sx_)::value;
            constexpr bool FULL = decltype(full_)::value;   // every node of the tile is inside the lattice
            const T svx = c_set<T, Q1>.vx[k], svy = c_set<T, Q1>.vy[k];
            const bool my = svy < T(0);
            const bool movy = Q1 % 2 == 0 || svy != T(0);
            const V vx = P::sp(svx), vy = P::sp(svy), w = P::sp(c_set<T, Q1>.w[k]);
            const V cvx = P::sp((SX < 0 ? -svx : svx) * cdx), cvy = P::sp((my ? -svy : svy) * cdx);
            const V vdtt = P::sp(IMEX ? c1 : dtt);
            const bool outer = lane % LC == (SX > 0 ? LC - 1 : 0);
            const int rs = my ? -HXP : HXP;           // row stride of the march
            const int t0 = grp * H + seg * HS;        // rows before the march's first, in its direction
            tk += (my ? RT - 1 - t0 : t0) * HXP + c0;   // march row -3, column -4 of the lane's nodes
            const T* ek = edges + k * TY + t0;
            const int yt = my ? TY - 1 - t0 : t0;     // tile row of march row 0
            const T* mp = mom + 2 * (yt * TX + c0);
            const T* mp0 = mom + 4 * TY * TX + yt * TX + c0;
            const int ms = my ? -TX : TX;
            const int x = x0 + c0;
            const long long off = k * plane + (long long)(y0 + yt) * pitch + x;
            const long long os = my ? -pitch : pitch;
            // node pointers, stepped row by row: f^n (RK3) or the stage input
            // (IMEX), the output, IMEX P
            const T* fp = static_cast<const T*>(cp->buf[IMEX ? in_idx : 0]) + off;
            T* op = static_cast<T*>(cp->buf[out_idx]) + off;
            [[maybe_unused]] T* pp = static_cast<T*>(cp->buf[2]) + off;
            [[maybe_unused]] const T* pp_in = pp;
            // march rows inside the lattice, one bit each (none beyond nx)
            unsigned rows;
            {
                const int n = my ? TY - (ny - y0) - t0 : ny - y0 - t0;   // first row / row count
                const int m = n < 0 ? 0 : (n > HS ? HS : n);
                rows = x < nx ? (my ? ~((1u << m) - 1u) : (1u << m) - 1u) : 0u;
            }
            const bool two = N == 2 && x + 1 < nx;
            auto load_nodes = [&](const T* p, int r) {
                if ((FULL || ((rows >> r) & 1u)) && LBM_BC_NODE(cp, K, off + r * os)) return ldg_v(p);   // beyond nx: row padding, not used
                return P::sp(T(0));
            };
            auto store_nodes = [&](T* p, int r, V v) {
                if ((FULL || ((rows >> r) & 1u)) && LBM_BC_NODE(cp, K, off + r * os)) {
                    if (FULL || N == 1 || two) stg_v(p, v);
                    else stg_1(p, P::get(v, 0));
                }
            };
            // rows unrolled: all of them, or two where the copies for the signs
            // of v_x (three with an odd set) would outgrow the instruction cache
            // (IMEX: or the registers)
            constexpr int UN = IMEX || Q1 == 3 ? (HS < 2 ? HS : 2) : (Q1 == 5 && HS > 4 ? 2 : HS);
            // the node values are loaded AH rows ahead of their use
            constexpr int AH = Q1 == 4 && !IMEX ? HS : UN;
            V fq[AH];
            [[maybe_unused]] V pq[IMEX ? AH : 1];
#pragma unroll
            for (int r = 0; r < AH; ++r) {
                fq[r] = node_in ? load_nodes(fp, r) : P::sp(T(0));
                if constexpr (IMEX) pq[r] = stage == 2 ? load_nodes(pp_in, r) : P::sp(T(0));
                fp += os;
                if constexpr (IMEX) pp_in += os;
            }
            // face below march row 0
            V dy1 = P::sp(T(0)), dy2 = dy1, dy3 = dy1, fy2 = dy1, top = dy1, last = dy1;
            if (movy) {
                const V a = ldv(tk + 4), b = ldv(tk + rs + 4), c = ldv(tk + 2 * rs + 4), d = ldv(tk + 3 * rs + 4);
                last = ldv(tk + 4 * rs + 4);
                const V d1 = P::sub(a, b);
                dy1 = P::sub(b, c);
                dy2 = P::sub(c, d);
                dy3 = P::sub(d, last);
                fy2 = weno5_f<P, T>(dy2, eps);
                top = weno5_diff<P, T>(d1, dy1, dy2, dy3, weno5_f<P, T>(dy1, eps), fy2);
            }
            const T *tr = tk + 3 * rs, *ty = tk + 5 * rs + 4;   // the node's row; two rows ahead, the lane's column
#pragma unroll (UN)
            for (int r = 0; r < HS; ++r, mp += 2 * ms, mp0 += ms, op += os, tr += rs, ty += rs) {
                const V fcur = fq[r % AH];
                [[maybe_unused]] V pcur = P::sp(T(0));
                if constexpr (IMEX) pcur = pq[r % AH];
                if (r + AH < HS) {
                    if (node_in) fq[r % AH] = load_nodes(fp, r + AH);
                    fp += os;
                    if constexpr (IMEX) {
                        if (stage == 2) pq[r % AH] = load_nodes(pp_in, r + AH);
                        pp_in += os;
                    }
                }
                V uk, fl, dcx;
                if constexpr (SX != 0) {
                    V d1, d2, d4;
                    uk = x_diffs<SX>(tr, d1, d2, dcx, d4);
                    fl = weno5_diff<P, T>(d1, d2, dcx, d4, weno5_f<P, T>(d2, eps), weno5_f<P, T>(dcx, eps));
                } else {
                    uk = ldv(tr + 4);
                }
                Equil<T> e;
                ldv2(mp, e.px, e.py);
                ldv2(mp + 2 * TY * TX, e.jx, e.jy);
                e.e0 = ldv(mp0);
                const V ew = e.over_w(vx, vy);
                // dt L(u)_k = -(dt/dx) v . dF - (u - geq) dt/tau; IMEX: dt C(Y)
                // of the stage input u at the node
                const V dtc = P::mulr(P::fma(w, ew, P::neg(IMEX ? fcur : uk)), vdtt);
                V inc = IMEX ? P::sp(T(0)) : dtc;
                if (movy) {
                    const V nw = ldv(ty);
                    const V dy4 = P::sub(last, nw);
                    last = nw;
                    const V fy3 = weno5_f<P, T>(dy3, eps);
                    const V up = weno5_diff<P, T>(dy1, dy2, dy3, dy4, fy2, fy3);
                    // flux difference (f_i - f_{i-1}) + (d_{i+1/2} - d_{i-1/2})/3
                    // (negated): the upwind node values differ by one node
                    // (exact for close values), the corrections d are small
                    inc = P::fma(cvy, P::fmac(P::sub(top, up), T(1.0 / 3.0), dy2), inc);
                    top = up;
                    dy1 = dy2;
                    dy2 = dy3;
                    dy3 = dy4;
                    fy2 = fy3;
                }
                if constexpr (SX != 0) {
                    const V fh = x_next<SX>(fl, ek[r], outer);
                    inc = P::fma(cvx, P::fmac(P::sub(fl, fh), T(1.0 / 3.0), dcx), inc);
                }
                if constexpr (!IMEX) {
                    // stage combination in increment form: one rounding of the
                    // stored value per stage (u - f^n is exact for close values);
                    // stage 1: u + dt L(u) (fcur is 0, cb 1)
                    store_nodes(op, r, P::fma(cb, P::add(P::sub(uk, fcur), inc), fcur));
                } else if (stage == 1) {
                    store_nodes(op, r, P::add(fcur, P::fmac(dtc, T(1.0 - 2.0 * IMEX_GAMMA), inc)));   // Z
                    store_nodes(pp, r, P::fmac(dtc, T(2.0 * IMEX_GAMMA), fcur));                       // P
                    pp += os;
                } else {
                    store_nodes(op, r, P::fmac(P::add(P::sub(fcur, pcur), P::add(inc, dtc)), T(0.5), pcur));
                }
            }
        };
        const bool full_tile = x0 + TX <= nx && y0 + TY <= ny;
#pragma unroll 1
        for (int m = warp; m < K * S; m += NM) {
            const int k = S == 1 ? m : m % K, seg = S == 1 ? 0 : m / K;
            const T* tk = buf + k * PL;
            auto by_sign = [&](auto full_) {
                if (Q1 % 2 == 1 && 2 * (k % Q1) + 1 == Q1) march(Const<0>{}, full_, k, seg, tk);
                else if (2 * (k % Q1) + 1 < Q1) march(Const<-1>{}, full_, k, seg, tk);
                else march(Const<1>{}, full_, k, seg, tk);
            };
            if (full_tile) by_sign(Const<1>{});
            else by_sign(Const<0>{});
        }
        named_arrive(4 + b, Ge::NT);
    }
}

int fd_tile_tx(int v) { return (v >= 0 && v < FD_NALL) ? FD_TX : 0; }
int fd_tile_ty(int v) {
    switch (v) {
        case FD_T32x8: return 8;
        case FD_T32x4: return 4;
        case FD_T32x16: return 16;
        case FD_T32x2: return 2;
        case FD_T32x1: return 1;
    }
    return 0;
}

// A kernel variant: its entry, block size and dynamic shared memory.
struct FdVariant {
    const void* fn = nullptr;
    int threads = 0;
    size_t bytes = 0;
};
template <typename T, int Q1, int TY, bool IMEX>
static FdVariant fd_variant_of() {
    using Ge = FdGeo<T, Q1, TY, IMEX>;
    return FdVariant{(const void*)fd_stage_kernel<T, Q1, TY, IMEX>, Ge::NT, Ge::bytes};
}
template <typename T, int Q1, bool IMEX>
static FdVariant fd_variant_q(int tile) {
    switch (tile) {
        case FD_T32x8: return fd_variant_of<T, Q1, 8, IMEX>();
        case FD_T32x4: return fd_variant_of<T, Q1, 4, IMEX>();
        case FD_T32x16: return fd_variant_of<T, Q1, 16, IMEX>();
        case FD_T32x2: return fd_variant_of<T, Q1, 2, IMEX>();
        case FD_T32x1:
            if constexpr (sizeof(T) == 8) return fd_variant_of<T, Q1, 1, IMEX>();
    }
    return FdVariant{};
}
template <typename T, bool IMEX>
static FdVariant fd_variant_t(int tile, int q1) {
    switch (q1) {
        case 3: return fd_variant_q<T, 3, IMEX>(tile);
        case 4: return fd_variant_q<T, 4, IMEX>(tile);
        case 5: return fd_variant_q<T, 5, IMEX>(tile);
    }
    return FdVariant{};
}
static FdVariant fd_variant(int precision, int tile, int q1, int scheme) {
    if (scheme == LBM_TS_IMEX)
        return precision == LBM_FP64 ? fd_variant_t<double, true>(tile, q1) : fd_variant_t<float, true>(tile, q1);
    return precision == LBM_FP64 ? fd_variant_t<double, false>(tile, q1) : fd_variant_t<float, false>(tile, q1);
}

// Opt each variant (both schemes' kernels) into the dynamic shared memory it
// needs; once per process. A variant that cannot fit on this device is
// refused (and the CUDA error state cleared).
static cudaError_t fd_prepare(int precision, int tile, int q1) {
    // 0 unknown, 1 ready, 2 does not fit; atomic: the two lanes of a server
    // may prepare the same variant at once (both then make the same calls)
    static std::atomic<int> state[2][FD_NALL][3] = {};
    const int p = precision == LBM_FP64 ? 0 : 1;
    std::atomic<int>& st = state[p][tile][q1 - 3];
    if (st == 1) return cudaSuccess;
    if (st == 2) return cudaErrorInvalidConfiguration;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorInvalidConfiguration;
    }
    for (int scheme : {LBM_TS_RK3, LBM_TS_IMEX}) {
        const FdVariant v = fd_variant(precision, tile, q1, scheme);
        if (!v.fn || v.bytes > (size_t)optin ||
            cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.bytes) != cudaSuccess) {
            cudaGetLastError();
            st = 2;
            return cudaErrorInvalidConfiguration;
        }
    }
    st = 1;
    return cudaSuccess;
}

cudaError_t launch_fd_stage(int precision, int q1, int scheme, int tile, int grid, const GroupDev& g, int j,
                            int stage, cudaStream_t s) {
    if (tile < 0 || tile >= FD_NALL || grid <= 0 || q1 < 3 || q1 > 5 ||
        (scheme != LBM_TS_RK3 && scheme != LBM_TS_IMEX && scheme != LBM_TS_RK3_FUSED) || stage < 1 ||
        stage > fd_stages(scheme))
        return cudaErrorInvalidValue;
    if (scheme == LBM_TS_RK3_FUSED) return launch_fd_fused(precision, q1, tile, grid, g, j, s);
    cudaError_t e = fd_prepare(precision, tile, q1);
    if (e != cudaSuccess) return e;
    const FdVariant v = fd_variant(precision, tile, q1, scheme);
    GroupDev gg = g;
    int jj = j, ss = stage;
    void* args[] = {&gg, &jj, &ss};
    return launch_overlapped(v.fn, grid, v.threads, args, v.bytes, s, g.overlap != 0);
}

bool fd_variant_fits(int precision, int q1, int tile, int scheme) {
    if (scheme == LBM_TS_RK3_FUSED) return fd_fused_fits(precision, q1, tile);
    return tile >= 0 && tile < FD_NALL && q1 >= 3 && q1 <= 5 && fd_prepare(precision, tile, q1) == cudaSuccess;
}

int fd_blocks_per_sm(int precision, int q1, int tile, int scheme) {
    if (scheme == LBM_TS_RK3_FUSED) return fd_fused_blocks_per_sm(precision, q1, tile);
    if (!fd_variant_fits(precision, q1, tile, scheme)) return 1;
    const FdVariant v = fd_variant(precision, tile, q1, scheme);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, v.fn, v.threads, v.bytes) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

}  // namespace lbm
