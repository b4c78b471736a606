// lbm_kernels.cuh -- CUDA kernels of the lattice Boltzmann hot path
// (arXiv 2512.12213) and their launchers, templated on the lattice (Q), the
// population storage format (S) and EXT (Lorentz force, Maxwell equilibrium
// or LES present).  Instantiated per storage format in inst_*.cu.
#pragma once

#include <algorithm>
#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "lbm_staged.cuh"

namespace lbm {

constexpr int STEP_THREADS = 128;
constexpr int NODE_THREADS = 256;
// blocks of NODE_THREADS per SM for the coupled field step: FP32 compute 3
// (85 registers, no spill), FP64 2
template <class S> struct MhdOcc {
    static constexpr int value = sizeof(typename S::R) == 8 ? 2 : 3;
};
constexpr int RED_THREADS = 256;

// ------------------------------------------------------------ warp helpers
template <class T> union Bits16 {
    T t;
    unsigned short s;
};
template <class T> __device__ __forceinline__ T shfl_up1(T v)
{
    if constexpr (sizeof(T) == 2) {
        Bits16<T> b;
        b.t = v;
        b.s = (unsigned short)__shfl_up_sync(0xffffffffu, (unsigned)b.s, 1);
        return b.t;
    } else {
        return __shfl_up_sync(0xffffffffu, v, 1);
    }
}
template <class T> __device__ __forceinline__ T shfl_down1(T v)
{
    if constexpr (sizeof(T) == 2) {
        Bits16<T> b;
        b.t = v;
        b.s = (unsigned short)__shfl_down_sync(0xffffffffu, (unsigned)b.s, 1);
        return b.t;
    } else {
        return __shfl_down_sync(0xffffffffu, v, 1);
    }
}

// sum W doubles over the block; thread 0 gets the totals in v[].  The FP64
// pipe takes a warp addition in ~19 cycles, so the values are reduced
// together: the first steps halve the values a lane carries along with the
// lanes that carry them (9 additions a warp for 8 values, not 40).
template <int W>
__device__ __forceinline__ void block_sum(double (&v)[W], double* smem /* >= W * 32 */)
{
    constexpr int P = W <= 2 ? 2 : (W <= 4 ? 4 : 8), G = 32 / P;
    static_assert(W <= 8, "at most 8 values");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    double t[P];
#pragma unroll
    for (int k = 0; k < P; ++k) t[k] = k < W ? v[k] : 0.0;
#pragma unroll
    for (int n = P / 2; n >= 1; n /= 2) {
        const int o = n * G;                     // 16, 8, ...
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double keep = up ? t[i + n] : t[i], send = up ? t[i] : t[i + n];
            t[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o /= 2) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
    const int k = lane / G, sub = lane % G;      // this lane's value
    if (sub == 0 && k < W) smem[k * 32 + wid] = t[0];
    __syncthreads();
    if (wid == 0) {
        double s = 0.0;
        for (int j = sub; j < nw; j += G) s += k < W ? smem[k * 32 + j] : 0.0;
#pragma unroll
        for (int o = G / 2; o > 0; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] = __shfl_sync(0xffffffffu, s, i * G);
    }
}

// The end of a reduction: thread 0 holds the block's sums in v; they become
// the block's partial row, and the block that finishes last (a ticket, zero
// between launches) adds the rows in the order of k_reduce_rows -- lane l of
// a column's warp takes rows l, l+32, ..., then a fixed shuffle tree -- so
// the result does not depend on timing and no second launch is needed
// (a wall force of 10^4 links 12.8 -> 10.7 us).  out[W] = out[0] / out[1]
// with RATIO.  ticket null: the rows alone.
template <int W, bool RATIO = false>
__device__ __forceinline__ void finish_rows(const double (&v)[W], double* __restrict__ partials, const RedOut& ro)
{
    __shared__ int last;
    __shared__ double col[W];
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < W; ++k) partials[(long long)blockIdx.x * W + k] = v[k];
        last = 0;
        if (ro.ticket) {
            __threadfence();
            last = atomicAdd(ro.ticket, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < W; k += (int)(blockDim.x >> 5)) {
        double s = 0.0;
        for (int r = lane; r < (int)gridDim.x; r += 32) s += __ldcg(partials + (long long)r * W + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) col[k] = ro.out[k] = (ro.accumulate ? ro.out[k] : 0.0) + ro.weight * s;
    }
    if (threadIdx.x == 0) *ro.ticket = 0u;
    if constexpr (RATIO) {
        __syncthreads();
        if (threadIdx.x == 0 && ro.ratio) ro.out[W] = col[1] > 0.0 ? col[0] / col[1] : 0.0;
    }
}

// ------------------------------------------------- fused collide-stream step
// One thread owns V consecutive nodes of a row (one 16-byte vector per
// direction).  For every direction it loads the aligned vector of the pull
// source row; the x-shifted directions take their edge element from the
// neighbouring lane (warp shuffle), or from one scalar load at a row edge or
// warp edge.  16-bit formats stay packed two to a register (the x shift is a
// byte permute) and are relaxed two nodes at a time.  A chunk that holds a
// boundary, solid or padding node is recomputed node by node with explicit
// bounce-back, the warp's such nodes spread over its lanes: one lane walking
// its chunk held the warp for up to four round trips, and a box of ragged
// rows has such a chunk in every row (sphere 250 x 121 x 99 in FP32: 141 ->
// 92 us).  Chunks of padding alone are not touched unless zero_pad asks for it
// (a destination that is not the context's own, whose padding is zero
// already).  FP32 and 16-bit storage (lbm_step64.cuh: FP64).  Populations are in storage units (kernel
// parameters scaled to match).
// blocks of 128 threads per SM the register allocation must allow: 4 (128
// registers; for 16-bit storage measured faster than 5 blocks at 96, which
// spill with the FP32x2 node pairs)
// (the EXT node code in FP32x2 node pairs, 32-bit storage with closed faces:
// 3, where it needs 158 registers without spill)
template <class S, bool EXT, bool FACES = false, bool FULL = false, bool LP = false> struct StepOcc {
    static constexpr bool PAIRX = EXT && !FULL && !LP && FACES && sizeof(typename S::T) == 4;
    static constexpr int value = PAIRX ? 3 : 4;
};

// FULL: the boundary path interpolates at walls off the half-grid and the
// EXT node code reads the Lorentz coefficient of insulating walls from the
// device and sums the flow velocity (contexts with a wall distance or
// insulating walls).  Kept out of the other instantiations: even as one
// out-of-line call the interpolation cost the fused step ~3% (inlined ~5%),
// and the insulating-wall code cost the LES cavity 8%.
// LP: the LES-only contexts with 16-bit storage (Smagorinsky with a uniform
// body force and no other EXT term) relax their all-fluid chunks with the
// FP32x2 pair code specialised for LES; chunks with a wall keep the scalar
// EXT node code.
template <int Q, class S, bool EXT, bool FACES, bool SR, bool FULL = false, bool LP = false>
__global__ void __launch_bounds__(STEP_THREADS, StepOcc<S, EXT, FACES, FULL, LP>::value)
k_step(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
       const uint8_t* __restrict__ cls, const Geo g, const KP<typename S::R> p, uint32_t seed, int zero_pad)
{
    pdl_trigger();
    using T = typename S::T;
    using R = typename S::R;
    constexpr int V = S::V;
    constexpr bool PACKED = sizeof(T) == 2;
    static_assert(V == 4, "FP64 has its own step");
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int ncx = g.nxp / V;
    const long long nch = (long long)ncx * g.ny * g.nz;
    const bool active = tid < nch;
    const long long ch = active ? tid : nch - 1;
    const int cx = (int)(ch % ncx);
    const long long row = ch / ncx;
    const int y = (int)(row % g.ny);
    const int z = (int)(row / g.ny);
    const int x0 = cx * V;

    // class bytes of the chunk: fast path if all are bulk (or, with FACES, face)
    bool special, face_chunk = false;
    const bool pad = x0 >= g.nx;
    const int xl = pad ? (g.nx - 1) / V * V : x0;     // a padding chunk repeats the row's last loads
    {
        const uint8_t* cp = cls + row * g.nxp + x0;
        const uint32_t cb = *reinterpret_cast<const uint32_t*>(cp);
        if (FACES) {
            special = (cb & ~0x02020202u) != 0u;
            face_chunk = (cb & 0x02020202u) != 0u;
        } else {
            special = cb != 0u;
        }
    }
    FaceInfo fi;
    if (FACES) {
        fi.closed_x = !g.periodic[0];
        fi.yo_lo = !g.periodic[1] && y == 0;
        fi.yo_hi = !g.periodic[1] && y == g.ny - 1;
        fi.zo_lo = (Q == 19) && !g.periodic[2] && z == 0;
        fi.zo_hi = (Q == 19) && !g.periodic[2] && z == g.nz - 1;
        fi.wx_lo = g.face_wall[0]; fi.wx_hi = g.face_wall[1];
        fi.wy_lo = g.face_wall[2]; fi.wy_hi = g.face_wall[3];
        fi.wz_lo = g.face_wall[4]; fi.wz_hi = g.face_wall[5];
    }
    // row offsets of the pull sources, by (E_y, E_z)
    long long roff[3][3];
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dz = -1; dz <= 1; ++dz) {
            const int ys = wrapi(y - dy, g.ny);
            const int zs = (Q == 19) ? wrapi(z - dz, g.nz) : 0;
            roff[dy + 1][dz + 1] = ((long long)zs * g.ny + ys) * g.nxp;
        }
    const long long own = row * g.nxp;
    pdl_wait(src);

    using RawT = typename RawVec<sizeof(T) * V>::type;
    // shifted source values: packed words for 16-bit formats, else elements
    uint32_t w[Q][PACKED ? V / 2 : 1];
    T f[Q][PACKED ? 1 : V];
    if constexpr (!FACES) {
        // periodic box: per direction, vector load, shuffle, and a scalar load
        // at the warp or row edge (measured faster here than the split order
        // of the closed-face variant)
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const T* rp = src + (long long)a * g.sq + roff[EY<Q>(a) + 1][EZ<Q>(a) + 1];
            VecN<T, V> raw;
            raw.raw = *reinterpret_cast<const RawT*>(rp + xl);
            const int ex = EX<Q>(a);
            T edge = raw.e[0];
            // periodic x: the wrap of a row edge and the warp edge are plain loads
            if (EX<Q>(a) == 1) {
                edge = shfl_up1(raw.e[V - 1]);
                if (lane == 0 || cx == 0) edge = rp[cx == 0 ? g.nx - 1 : x0 - 1];
            } else if (EX<Q>(a) == -1) {
                edge = shfl_down1(raw.e[0]);
                if (lane == 31 || x0 + V >= g.nx) edge = rp[x0 + V >= g.nx ? 0 : x0 + V];
            }
            if constexpr (PACKED) {
                const uint32_t* rw = raw.u;
                Bits16<T> eb;
                eb.t = edge;
                const uint32_t ew = (uint32_t)eb.s;
                if (ex == 0) {
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) w[a][i] = rw[i];
                } else if (ex == 1) {             // value k <- raw k-1
                    w[a][0] = __byte_perm(ew, rw[0], 0x5410);
#pragma unroll
                    for (int i = 1; i < V / 2; ++i) w[a][i] = __byte_perm(rw[i - 1], rw[i], 0x5432);
                } else {                           // value k <- raw k+1
#pragma unroll
                    for (int i = 0; i < V / 2 - 1; ++i) w[a][i] = __byte_perm(rw[i], rw[i + 1], 0x5432);
                    w[a][V / 2 - 1] = __byte_perm(rw[V / 2 - 1], ew, 0x5432);
                }
            } else {
                if (ex == 0) {
#pragma unroll
                    for (int k = 0; k < V; ++k) f[a][k] = raw.e[k];
                } else if (ex == 1) {
                    f[a][0] = edge;
#pragma unroll
                    for (int k = 1; k < V; ++k) f[a][k] = raw.e[k - 1];
                } else {
#pragma unroll
                    for (int k = 0; k < V - 1; ++k) f[a][k] = raw.e[k + 1];
                    f[a][V - 1] = edge;
                }
            }
        }
    } else {
        // closed faces: all vector loads first, then the edge-element loads,
        // and only then the shuffles that wait for them (one memory round trip)
        auto row_ptr = [&](int a, bool rout) -> const T* {
            // bounced rows read the node's own value of the opposite direction
            return rout ? src + (long long)OPP<Q>(a) * g.sq + own
                        : src + (long long)a * g.sq + roff[EY<Q>(a) + 1][EZ<Q>(a) + 1];
        };
        VecN<T, V> raw[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            int rwall = 0;
            const bool rout = row_out<Q>(fi, a, rwall);
            raw[a].raw = *reinterpret_cast<const RawT*>(row_ptr(a, rout) + xl);
        }
        // lanes at a warp edge or a row edge load the element the shuffle
        // cannot give them: the left neighbour of x0 (E_x = +1) or the right
        // neighbour of x0 + V - 1 (E_x = -1), wrapped on a periodic x axis, or
        // the node's own opposite population at a closed x face
        const bool needL = (lane == 0 || cx == 0), needR = (lane == 31 || x0 + V >= g.nx);
        T eload[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            eload[a] = raw[a].e[0];
            int rwall = 0;
            const bool rout = row_out<Q>(fi, a, rwall);
            const T* rp = row_ptr(a, rout);
            if (EX<Q>(a) == 1 && !rout && needL) {
                if (cx == 0 && fi.closed_x) eload[a] = src[(long long)OPP<Q>(a) * g.sq + own];
                else eload[a] = rp[cx == 0 ? g.nx - 1 : x0 - 1];
            } else if (EX<Q>(a) == -1 && !rout && needR) {
                if (x0 + V >= g.nx && fi.closed_x) eload[a] = src[(long long)OPP<Q>(a) * g.sq + own + g.nx - 1];
                else eload[a] = rp[x0 + V >= g.nx ? 0 : x0 + V];
            }
        }
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            int rwall = 0;
            const bool rout = row_out<Q>(fi, a, rwall);
            const int ex = rout ? 0 : EX<Q>(a);
            T edge = raw[a].e[0];
            if (EX<Q>(a) == 1) {
                edge = shfl_up1(raw[a].e[V - 1]);
                if (needL) edge = eload[a];
            } else if (EX<Q>(a) == -1) {
                edge = shfl_down1(raw[a].e[0]);
                if (needR) edge = eload[a];
            }
            if constexpr (PACKED) {
                const uint32_t* rw = raw[a].u;
                Bits16<T> eb;
                eb.t = edge;
                const uint32_t ew = (uint32_t)eb.s;
                if (ex == 0) {
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) w[a][i] = rw[i];
                } else if (ex == 1) {             // value k <- raw k-1
                    w[a][0] = __byte_perm(ew, rw[0], 0x5410);
#pragma unroll
                    for (int i = 1; i < V / 2; ++i) w[a][i] = __byte_perm(rw[i - 1], rw[i], 0x5432);
                } else {                           // value k <- raw k+1
#pragma unroll
                    for (int i = 0; i < V / 2 - 1; ++i) w[a][i] = __byte_perm(rw[i], rw[i + 1], 0x5432);
                    w[a][V / 2 - 1] = __byte_perm(rw[V / 2 - 1], ew, 0x5432);
                }
            } else {
                if (ex == 0) {
#pragma unroll
                    for (int k = 0; k < V; ++k) f[a][k] = raw[a].e[k];
                } else if (ex == 1) {
                    f[a][0] = edge;
#pragma unroll
                    for (int k = 1; k < V; ++k) f[a][k] = raw[a].e[k - 1];
                } else {
#pragma unroll
                    for (int k = 0; k < V - 1; ++k) f[a][k] = raw[a].e[k + 1];
                    f[a][V - 1] = edge;
                }
            }
        }
    }
    // insulating walls: this thread's sum of the flow velocity v over the
    // fluid nodes it relaxes, summed over the warp by a fixed shuffle tree in
    // FP64 (every thread of the block reaches it, inactive ones with zero),
    // one row per warp for the fixed-order reduction of the field
    R vs[3] = {R(0), R(0), R(0)};
    auto add_v = [&](const NodeM<R>& m) {
        if constexpr (EXT && FULL) {
            vs[0] += m.v[0];
            vs[1] += m.v[1];
            vs[2] += m.v[2];
        }
    };
    auto put_v = [&]() {
        if constexpr (EXT && FULL) {
            if (p.ins_rows) {
                double t[3] = {(double)vs[0], (double)vs[1], (double)vs[2]};
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int k = 0; k < 3; ++k) t[k] += __shfl_down_sync(0xffffffffu, t[k], o);
                if (lane == 0)
#pragma unroll
                    for (int k = 0; k < 3; ++k) p.ins_rows[(tid >> 5) * 3 + k] = t[k];
            }
        }
    };
    if (active && !special) {

        // Ladd terms of moving face walls, added after unpacking (face chunks only)
        const bool ladd = FACES && face_chunk && p.face_ladd;
        auto add_ladd = [&](R (&d)[Q], int k) {
#pragma unroll
            for (int a = 1; a < Q; ++a) {
                int wall = 0;
                bool hit = row_out<Q>(fi, a, wall);
                if (fi.closed_x) {
                    if (EX<Q>(a) == 1 && x0 + k == 0) { hit = true; wall = fi.wx_lo; }
                    if (EX<Q>(a) == -1 && x0 + k == g.nx - 1) { hit = true; wall = fi.wx_hi; }
                }
                if (hit) d[a] = ladd_on<Q, R>(d[a], p, a, wall);
            }
        };

        // the same for two consecutive nodes k, k+1 held as pairs
        auto add_ladd2 = [&](F2 (&d)[Q], int k) {
#pragma unroll
            for (int a = 1; a < Q; ++a) {
                int wall = 0;
                const bool hit = row_out<Q>(fi, a, wall);
                int w0 = wall, w1 = wall;
                bool h0 = hit, h1 = hit;
                if (fi.closed_x) {
                    if (EX<Q>(a) == 1 && x0 + k == 0) { h0 = true; w0 = fi.wx_lo; }
                    if (EX<Q>(a) == -1 && x0 + k == g.nx - 1) { h0 = true; w0 = fi.wx_hi; }
                    if (EX<Q>(a) == -1 && x0 + k + 1 == g.nx - 1) { h1 = true; w1 = fi.wx_hi; }
                }
                if (h0) d[a].v.x = ladd_on<Q, R>(d[a].v.x, p, a, w0);
                if (h1) d[a].v.y = ladd_on<Q, R>(d[a].v.y, p, a, w1);
            }
        };
        // two nodes at a time in packed FP32x2 arithmetic (FP32 compute without
        // the Lorentz force, Maxwell term or LES)
        constexpr bool PAIR2 = (!EXT || LP) && sizeof(R) == 4;
    // the EXT node code in node pairs too: FP32 storage with closed faces (the
    // LES cavity 24.7k -> 26.6k MLUPS); measured slower for 16-bit storage
    // (-3.7%) and periodic FP32 boxes (-2.5%, spills), which keep the scalar code
    constexpr bool PAIRX = StepOcc<S, EXT, FACES, FULL, LP>::PAIRX;

        const long long base = row * g.nxp + x0;
        {
            if constexpr (PACKED && PAIR2) {
#pragma unroll
                for (int i = 0; i < V / 2; ++i) {
                    F2 dd[Q];
#pragma unroll
                    for (int a = 0; a < Q; ++a) dd[a] = F2{S::unpack2(w[a][i])};
                    if (ladd) add_ladd2(dd, 2 * i);
                    pair_collide<Q, LP, true>(dd, p);
                    if constexpr (SR) {
                        NodeRng rp((uint32_t)(base + 2 * i), seed);     // the pair's first node
#pragma unroll
                        for (int a = 0; a < Q; ++a) w[a][i] = S::pack2_sr(dd[a].v.x, dd[a].v.y, rp.word());
                    } else {
#pragma unroll
                        for (int a = 0; a < Q; ++a) w[a][i] = S::pack2(dd[a].v.x, dd[a].v.y);
                    }
                }
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    VecN<T, V> o;
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) o.u[i] = w[a][i];
                    *reinterpret_cast<typename RawVec<sizeof(T) * V>::type*>(dst + (long long)a * g.sq + base) = o.raw;
                }
            } else if constexpr (PACKED) {
                // two nodes per packed word: unpack both, relax them, pack both
                // with one conversion
#pragma unroll
                for (int i = 0; i < V / 2; ++i) {
                    R d0[Q], d1[Q];
#pragma unroll
                    for (int a = 0; a < Q; ++a) {
                        const float2 v = S::unpack2(w[a][i]);
                        d0[a] = v.x;
                        d1[a] = v.y;
                    }
                    if (ladd) {
                        add_ladd(d0, 2 * i);
                        add_ladd(d1, 2 * i + 1);
                    }
                    {
                        NodeM<R> m;
                        node_macro<R, Q, EXT, FULL>(d0, p, m);
                        node_relax<R, Q, EXT>(d0, p, m);
                        add_v(m);
                    }
                    {
                        NodeM<R> m;
                        node_macro<R, Q, EXT, FULL>(d1, p, m);
                        node_relax<R, Q, EXT>(d1, p, m);
                        add_v(m);
                    }
                    if constexpr (SR) {
                        NodeRng rp((uint32_t)(base + 2 * i), seed);     // the pair's first node
#pragma unroll
                        for (int a = 0; a < Q; ++a) w[a][i] = S::pack2_sr(d0[a], d1[a], rp.word());
                    } else {
#pragma unroll
                        for (int a = 0; a < Q; ++a) w[a][i] = S::pack2(d0[a], d1[a]);
                    }
                }
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    VecN<T, V> o;
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) o.u[i] = w[a][i];
                    *reinterpret_cast<typename RawVec<sizeof(T) * V>::type*>(dst + (long long)a * g.sq + base) = o.raw;
                }
            } else {
                if constexpr (PAIRX) {
                    // the EXT node code in node pairs, as a rolled queue of pairs
#pragma unroll 1
                    for (int k = 0; k < V / 2; ++k) {
                        F2 dd[Q];
#pragma unroll
                        for (int a = 0; a < Q; ++a) dd[a] = F2{make_float2(S::to_raw(f[a][0]), S::to_raw(f[a][1]))};
                        if (ladd) add_ladd2(dd, 2 * k);
                        pair_collide_ext<Q>(dd, p);
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
#pragma unroll
                            for (int j = 0; j < V - 2; ++j) f[a][j] = f[a][j + 2];
                            f[a][V - 2] = S::from_raw(dd[a].v.x);
                            f[a][V - 1] = S::from_raw(dd[a].v.y);
                        }
                    }
                } else if constexpr (EXT && !LP) {
                    // larger node code (Lorentz / Maxwell / LES): the same rolled queue
#pragma unroll 1
                    for (int k = 0; k < V; ++k) {
                        R d[Q];
#pragma unroll
                        for (int a = 0; a < Q; ++a) d[a] = S::to_raw(f[a][0]);
                        if (ladd) add_ladd(d, k);
                        NodeM<R> m;
                        node_macro<R, Q, EXT, FULL>(d, p, m);
                        node_relax<R, Q, EXT>(d, p, m);
                        add_v(m);
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
#pragma unroll
                            for (int j = 0; j < V - 1; ++j) f[a][j] = f[a][j + 1];
                            f[a][V - 1] = S::from_raw(d[a]);
                        }
                    }
                } else if constexpr (PAIR2) {
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) {
                        F2 dd[Q];
#pragma unroll
                        for (int a = 0; a < Q; ++a) dd[a] = F2{make_float2(S::to_raw(f[a][2 * i]), S::to_raw(f[a][2 * i + 1]))};
                        if (ladd) add_ladd2(dd, 2 * i);
                        pair_collide<Q, LP>(dd, p);
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            f[a][2 * i] = S::from_raw(dd[a].v.x);
                            f[a][2 * i + 1] = S::from_raw(dd[a].v.y);
                        }
                    }
                }
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    VecN<T, V> o;
#pragma unroll
                    for (int k = 0; k < V; ++k) o.e[k] = f[a][k];
                    *reinterpret_cast<typename RawVec<sizeof(T) * V>::type*>(dst + (long long)a * g.sq + base) = o.raw;
                }
            }
        }
    }
    // the warp's chunks with a solid neighbour or padding, one node per lane
    const unsigned todo = __ballot_sync(0xffffffffu, active && special && !pad);
    for (int i = lane; i < V * __popc(todo); i += 32) {
        unsigned rest = todo;
        for (int k = i / V; k > 0; --k) rest &= rest - 1;      // the (i / V)-th special chunk
        const unsigned sch = (unsigned)(tid - lane) + (unsigned)__ffs(rest) - 1u;
        const unsigned sr = sch / (unsigned)ncx;
        const int sx = (int)(sch - sr * (unsigned)ncx) * V + i % V;
        const int sz = (int)(sr / (unsigned)g.ny), sy = (int)(sr - (unsigned)sz * (unsigned)g.ny);
        const long long n = (long long)sr * g.nxp + sx;
        const uint8_t c = cls[n];
        if (nc_solid(c) || c == NC_PAD) {
#pragma unroll
            for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw(R(0));
            continue;
        }
        R d[Q];
        if (FULL && g.phi && c == NC_BOUND) gather_node<Q, S, true, true>(src, cls, g, p, sx, sy, sz, d);
        else pull_walls<Q, S, true>(src, cls, g, p, Around<Q>(g, sx, sy, sz), d);
        NodeM<R> m;
        node_macro<R, Q, EXT, FULL>(d, p, m);
        node_relax<R, Q, EXT>(d, p, m);
        add_v(m);
        if constexpr (SR) {
            NodeRng rng((uint32_t)n, seed);
#pragma unroll
            for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw_sr(d[a], rng.bits(a));
        } else {
#pragma unroll
            for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw(d[a]);
        }
    }
    if (zero_pad && active && pad)
        for (int a = 0; a < Q; ++a)
            *reinterpret_cast<RawT*>(dst + (long long)a * g.sq + row * g.nxp + x0) = RawT{};
    __syncwarp();
    put_v();
}

// ------------------------------------------------- deviations and populations
// w rho0 of the speed classes (rest, axis, diagonal) in FP64 and as an
// unevaluated FP32 sum hi + lo + lo2 of the same value
struct WRho {
    double c[3];
    float hi[3], lo[3], lo2[3];
};
template <int Q> inline WRho wrho_of(double rho0)
{
    WRho w;
    constexpr int a[3] = {0, 1, Q == 9 ? 5 : 7};
    for (int k = 0; k < 3; ++k) {
        w.c[k] = WD<Q>(a[k]) * rho0;
        w.hi[k] = (float)w.c[k];
        w.lo[k] = (float)(w.c[k] - (double)w.hi[k]);
        w.lo2[k] = (float)(w.c[k] - (double)w.hi[k] - (double)w.lo[k]);
    }
    return w;
}
// x + y = s + e without error (Knuth's two-sum), for two values together
__device__ __forceinline__ F2 two_sum(F2 x, F2 y, F2& e)
{
    const F2 s = f2add(x, y), b = f2sub(s, x);
    e = f2add(f2sub(x, f2sub(s, b)), f2sub(y, b));
    return s;
}
// the node's d_a + sign w_a rho0 rounded once to FP32, two opposite directions
// together: s + e = d + hi and r + f = s + lo without error, and what is left,
// e + lo2 + f, is rounded to 2^-24 of itself before it decides the rounding of
// r.  (With lo2 left out and e + lo rounded first, 7 us less of the 108 of an
// export of 256 x 128 x 128 FP32 nodes, a value beside rest was off by 0.66
// units in the last place: s is then a unit of hi, and lo is as large as it.)
// An FP64 addition holds an SM's FP64 pipe ~20 cycles a warp, 19 of them a
// node 0.17 ms of that box.
template <int Q>
__device__ __forceinline__ void add_wrho(float (&d)[Q], const WRho& wr, float sign)
{
    auto add = [&](F2 v, int k) {
        F2 e, f;
        const F2 s = two_sum(v, f2s(sign * wr.hi[k]), e), r = two_sum(s, f2s(sign * wr.lo[k]), f);
        v = f2add(r, f2add(f, f2add(e, f2s(sign * wr.lo2[k]))));
        // an infinite or undefined sum has no error term
        if (!(fabsf(s.v.x) <= 3.402823466e38f)) v.v.x = s.v.x;
        if (!(fabsf(s.v.y) <= 3.402823466e38f)) v.v.y = s.v.y;
        return v;
    };
    d[0] = add(F2{make_float2(d[0], 0.0f)}, 0).v.x;
#pragma unroll
    for (int k = 0; k < LatDim<Q>::NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const F2 v = add(F2{make_float2(d[a], d[b])}, SPEED2<Q>(a));
        d[a] = v.v.x;
        d[b] = v.v.y;
    }
}

// ------------------------------------------ inverse propagation (import/init)
// Stored state P with gather(P) = the given canonical f: every node stores its
// own populations where its pulls read them (push_node), so a node's values
// are formed once.  The sources give one value (src_value, for walls off the
// half-grid) or all of a node's (node_values).
struct SrcCanonD { const double* f; long long N; };
struct SrcCanonF { const float* f; long long N; };
struct SrcFields { const double* rho; const double* u; const double* xi; long long N; double ic; };   // ic = 1 / c

// the deviations f_a - w_a rho0 of node n
template <int Q, typename R, class Src>
__device__ __forceinline__ void node_values(const Src& s, const KP<R>&, const WRho& wr, long long n, R (&d)[Q])
{
    std::remove_cv_t<std::remove_pointer_t<decltype(s.f)>> f[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) f[a] = s.f[(long long)a * s.N + n];
    if constexpr (sizeof(R) == 4 && sizeof(f[0]) == 4) {
#pragma unroll
        for (int a = 0; a < Q; ++a) d[a] = f[a];
        add_wrho<Q>(d, wr, -1.0f);
    } else {
#pragma unroll
        for (int a = 0; a < Q; ++a) d[a] = R((double)f[a] - wr.c[SPEED2<Q>(a)]);
    }
}
// Eq. (1) (+ Eq. 10) in FP64, times 1 + xi.  The FP64 pipe bounds it (1.7
// lanes per cycle and SM), so the node's terms are shared: with m = 3 rho W
// and q_k = m_k W_k, an opposite pair is w (even +- odd), odd = E.m and
// even = rho - rho0 - sum q / 2 + 3/2 (E.m)(E.W), the last product
// q_i + q_j +- 2 m_i W_j for a diagonal pair: 67 operations a node.
template <int Q, typename R>
__device__ __forceinline__ void fields_values64(const SrcFields& s, const KP<R>& p, const WRho& wr, long long n,
                                                double rho, const double (&W)[3], R (&d)[Q])
{
    constexpr int D = LatDim<Q>::D;
    double m[3], q[3], sq = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        m[k] = 3.0 * rho * W[k];
        q[k] = m[k] * W[k];
        sq += q[k];
    }
    const double h = p.stokes ? 0.0 : 1.5;       // the linear equilibrium drops the quadratic terms
    const double base = fma(-h / 3.0, sq, rho - (double)p.rho0);
    auto put = [&](int a, double v) {
        if (p.maxwell) v += (double)p.mx[a];
        if (s.xi) v = fma(v + wr.c[SPEED2<Q>(a)], s.xi[(long long)a * s.N + n], v);
        d[a] = R(v);
    };
    put(0, WD<Q>(0) * base);
#pragma unroll
    for (int k = 0; k < LatDim<Q>::NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const double w = WD<Q>(a);
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
        double em = 0.0, eq = 0.0, mw = 0.0;     // E.m, the q_k of its axes, m_i W_j signed
        int first = -1;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            if (!e[c]) continue;
            if (first < 0) {
                em = e[c] > 0 ? m[c] : -m[c];
                eq = q[c];
                first = c;
            } else {
                em = e[c] > 0 ? em + m[c] : em - m[c];
                eq += q[c];
                mw = e[first] * e[c] > 0 ? m[first] * W[c] : -(m[first] * W[c]);
            }
        }
        double even = fma(h * w, eq, w * base);
        if (SPEED2<Q>(a) == 2) even = fma(2.0 * h * w, mw, even);
        put(a, fma(w, em, even));
        put(b, fma(-w, em, even));
    }
}

__device__ __forceinline__ FF ff_mul(FF x, FF y)
{
    const float p = __fmul_rn(x.h, y.h);
    return FF{p, __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmaf_rn(x.h, y.h, -p)))};
}
__device__ __forceinline__ FF ff_neg(FF x) { return FF{-x.h, -x.l}; }
__device__ __forceinline__ FF ff_scale(FF x, float c) { return FF{x.h * c, x.l * c}; }      // c a power of two
__host__ __device__ constexpr FF ff_const(double c) { return FF{(float)c, (float)(c - (double)(float)c)}; }
// x as h + l by its bits (the FP64 pipe converts as slowly as it adds): h the
// leading 24 bits, l the other 29 rounded to 24; ok = false outside
// 2^-73 .. 2^60 (zero is in)
__device__ __forceinline__ FF ff_split(double x, bool& ok)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7FFu, sign = hi & 0x80000000u;
    if (((hi << 1) | lo) == 0u) return FF{0.0f, 0.0f};
    if (e - 950u > 1083u - 950u) ok = false;
    const float h = __uint_as_float(sign | ((((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | (lo >> 29)));
    // 2^(exponent - 52), signed; e - 1023 - 52 + 127 = e - 948
    const float u = __uint_as_float(sign | ((e - 948u) << 23));
    return FF{h, __fmul_rn((float)(lo & 0x1FFFFFFFu), u)};
}

// the deviations of the equilibrium (without xi), for FP32 compute: as
// fields_values64, in unevaluated FP32 sums, whose ~480 FP32 operations a node
// cost a sixth of 67 FP64 ones.  With J = rho W, K_k = J_k W_k, X = J_i W_j
// and Z = rho - rho0 - 3/2 sum K, the pairs are  w1 Z + 9/2 w1 K_k +- 3 w1 J_k
// and  w2 Z + 9/2 w2 (K_i + K_j +- 2 X) +- 3 w2 (J_i +- J_j); 9/2 w is a power
// of two.  Rounded to FP32 at the end, as the FP64 values were: the stored values'
// error against 64 bits is the rounding's, 2.7e-8, at deviations of 1e-2 to
// 1e-8 alike.  256 x 128 x 128: 1,335 us in FP64 -> 168 us.  A value that lies within the two evaluations' errors of the
// middle of two FP32 numbers (about one of 1e5) takes the FP64 formula, so
// that the rounding is that of the FP64 evaluation; not in a flow whose
// deviations are below 1e-8, where the sums here are the more exact.  false (d
// not set): an input outside the range of ff_split.
template <int Q>
__device__ __forceinline__ bool fields_values32(const KP<float>& p, const WRho& wr, double rho, const double (&Wd)[3],
                                                float (&d)[Q])
{
    constexpr int D = LatDim<Q>::D;
    constexpr double w1 = WD<Q>(1), w2 = WD<Q>(Q == 9 ? 5 : 7);
    bool ok = true;
    const FF dr = ff_split(rho - (double)p.rho0, ok);
    const FF rh = ff_add(FF{p.rho0, 0.0f}, dr);
    FF W[3], J[3], O[3], K[3], Z = dr;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        W[k] = ff_split(Wd[k], ok);
        J[k] = ff_mul(rh, W[k]);
        O[k] = ff_mul(J[k], ff_const(3.0 * w1));
    }
    if (!ok) return false;
    const bool quad = !p.stokes;                 // the linear equilibrium drops the quadratic terms
    if (quad) {
        FF sum{0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < D; ++k) {
            K[k] = ff_mul(J[k], W[k]);
            sum = k ? ff_add(sum, K[k]) : K[k];
        }
        Z = ff_add(ff_add(Z, ff_neg(sum)), ff_scale(sum, -0.5f));
    }
    // errors, over w: 2^-43 of the terms here, 2^-50 of w rho in FP64
    float tol = fabsf(dr.h);
#pragma unroll
    for (int k = 0; k < D; ++k) tol = fmaf(4.0f, fabsf(W[k].h), tol);
    tol = fmaf(1.1368684e-13f, tol, 8.8817842e-16f * p.rho0);
    unsigned redo = 0;
    auto put = [&](int a, FF v) {
        if (p.maxwell) v = ff_add(v, FF{p.mx[a], 0.0f});
        const float r = __fadd_rn(v.h, v.l), t = tol * (float)WD<Q>(a);
        d[a] = r;
        // |v - r| near half a unit in the last place of r, or a quarter (the
        // half below a power of two)
        const float e = fabsf(__fadd_rn(__fsub_rn(v.h, r), v.l));
        const float half = __uint_as_float(__float_as_uint(r) & 0x7F800000u) * 5.9604645e-8f;
        if (t <= 0.0625f * half && (fabsf(e - half) <= t || fabsf(e - 0.5f * half) <= t)) redo |= 1u << a;
    };
    put(0, ff_mul(Z, ff_const(WD<Q>(0))));
    const FF Z1 = ff_mul(Z, ff_const(w1)), Z2 = ff_scale(Z1, (float)(w2 / w1));
#pragma unroll
    for (int k = 0; k < LatDim<Q>::NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
        const int i = e[0] ? 0 : (e[1] ? 1 : 2);
        FF even, odd;
        if (SPEED2<Q>(a) == 1) {
            even = quad ? ff_add(Z1, ff_scale(K[i], (float)(4.5 * w1))) : Z1;
            odd = O[i];
        } else {
            const int j = e[2] ? 2 : 1;
            const FF oi = ff_scale(O[i], (float)(e[i] * w2 / w1)), oj = ff_scale(O[j], (float)(e[j] * w2 / w1));
            odd = ff_add(oi, oj);
            even = Z2;
            if (quad) {
                even = ff_add(Z2, ff_scale(ff_add(K[i], K[j]), (float)(4.5 * w2)));
                even = ff_add(even, ff_scale(ff_mul(J[i], W[j]), (float)(9.0 * w2 * e[i] * e[j])));
            }
        }
        put(a, ff_add(even, odd));
        put(b, ff_add(even, ff_neg(odd)));
    }
    if (redo) {
        const double ww = Wd[0] * Wd[0] + Wd[1] * Wd[1] + Wd[2] * Wd[2];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            if (!(redo >> a & 1u)) continue;
            const double eu = EX<Q>(a) * Wd[0] + EY<Q>(a) * Wd[1] + EZ<Q>(a) * Wd[2];
            double fe = p.stokes ? rho * WD<Q>(a) * (1.0 + 3.0 * eu)
                                 : rho * WD<Q>(a) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * ww);
            if (p.maxwell) fe += (double)p.mx[a];
            d[a] = (float)(fe - wr.c[SPEED2<Q>(a)]);
        }
    }
    return true;
}

template <int Q, typename R>
__device__ __forceinline__ void node_values(const SrcFields& s, const KP<R>& p, const WRho& wr, long long n, R (&d)[Q])
{
    double W[3] = {0.0, 0.0, 0.0};
    const double rho = s.rho[n];
#pragma unroll
    for (int k = 0; k < LatDim<Q>::D; ++k) {
        W[k] = s.u[(long long)k * s.N + n];
        if (s.ic != 1.0) W[k] *= s.ic;
    }
    if constexpr (sizeof(R) == 4) {
        if (!s.xi && fields_values32<Q>(p, wr, rho, W, d)) return;
    }
    fields_values64<Q, R>(s, p, wr, n, rho, W, d);
}

// one of them (a is a constant: the others' terms are dropped)
template <int Q, typename R, class Src>
__device__ __forceinline__ R src_value(const Src& s, const KP<R>& p, const WRho& wr, int a, long long n)
{
    R d[Q];
    node_values<Q, R>(s, p, wr, n, d);
    return d[a];
}

// canonical index of a fluid node given by its padded index
__device__ __forceinline__ long long canon_of(const Geo& g, long long padded)
{
    const int xs = (int)(padded % g.nxp);
    return (padded / g.nxp) * g.nx + xs;
}

// The stored value P_a(x) of a link a that leaves fluid node x (padded own)
// into a wall, such that the bounced population of b = opp(a) at x (see
// bounced) is the given fb = f_b(x), fa = f_a(x): the inverse of the halfway or
// interpolated rule.  Every case is explicit except both opposite links of
// x hitting solids with q >= 1/2, a 2 x 2 solve.
template <int Q, typename R, class Src>
__device__ R unbounced(const Src& s, const KP<R>& p, const WRho& wr, const Geo& g, const uint8_t* __restrict__ cls, int x, int y, int z,
                       long long own, R fa, R fb, int a, int wall)
{
    const int b = OPP<Q>(a);
    const R half = ladd_off<Q, R>(fb, p, b, wall);
    if (!g.phi) return half;
    const long long sa = link_target(g, x, y, z, EX<Q>(a), EY<Q>(a), EZ<Q>(a));
    if (sa < 0 || !nc_solid(cls[sa])) return half;               // a closed box face
    const R qa = R(g.phi[own]) / (R(g.phi[own]) - R(g.phi[sa]));
    long long nb;
    int wb;
    const bool b_fluid = pull_source(g, cls, x, y, z, EX<Q>(a), EY<Q>(a), EZ<Q>(a), nb, wb);   // x + E_b = x - E_a
    if (qa < R(0.5)) {
        if (!b_fluid) return half;
        return (half - (R(1) - R(2) * qa) * fa) / (R(2) * qa);       // fa = P_a(x - E_a)
    }
    R Pb;
    if (b_fluid) {
        Pb = src_value<Q, R>(s, p, wr, b, canon_of(g, nb));           // node x + E_b pulls b from x
        return ladd_off<Q, R>(R(2) * qa * fb - (R(2) * qa - R(1)) * Pb, p, b, wall);
    }
    // the link b of x hits a wall too (wall id wb)
    const long long sb = link_target(g, x, y, z, EX<Q>(b), EY<Q>(b), EZ<Q>(b));
    const R qb = (sb >= 0 && nc_solid(cls[sb])) ? R(g.phi[own]) / (R(g.phi[own]) - R(g.phi[sb])) : R(0.5);
    if (qb < R(0.5) || !(sb >= 0 && nc_solid(cls[sb]))) {
        // b bounces halfway (its second node x + E_a is the solid, or a face)
        Pb = ladd_off<Q, R>(fa, p, a, wb);
        return ladd_off<Q, R>(R(2) * qa * fb - (R(2) * qa - R(1)) * Pb, p, b, wall);
    }
    const R A1 = ladd_off<Q, R>(R(2) * qa * fb, p, b, wall), k1 = R(2) * qa - R(1);
    const R A2 = ladd_off<Q, R>(R(2) * qb * fa, p, a, wb), k2 = R(2) * qb - R(1);
    return (A1 - k1 * A2) / (R(1) - k1 * k2);
}

// one padded node per thread.  Before (each node pulling its 18 neighbours'
// values, with their equilibria in FP64) a 192^3 binary16 box took 12.2 ms
// from fields and 1.04 ms from FP32 populations; so 0.44 ms and
// 0.23 ms (0.53 of the copy bandwidth).
template <int Q, class S, class Src, bool CURVED>
__global__ void __launch_bounds__(NODE_THREADS, CURVED ? 1 : 4)
k_inverse_stream(typename S::T* __restrict__ P, const uint8_t* __restrict__ cls, const Geo g,
                 const KP<typename S::R> p, const WRho wr, const Src s)
{
    pdl_wait();
    using R = typename S::R;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= g.sq) return;
    const unsigned r = (unsigned)n / (unsigned)g.nxp;
    const int x = (int)((unsigned)n - r * (unsigned)g.nxp);
    const int z = (int)(r / (unsigned)g.ny), y = (int)(r - (unsigned)z * (unsigned)g.ny);
    const uint8_t c = cls[n];
    if (x >= g.nx || nc_solid(c) || c == NC_PAD) {
#pragma unroll
        for (int a = 0; a < Q; ++a) P[(long long)a * g.sq + n] = S::from_r(R(0));
        return;
    }
    const long long nd = (long long)r * g.nx + x;
    R d[Q];
    node_values<Q, R>(s, p, wr, nd, d);
    if constexpr (CURVED) {
        if (c == NC_BOUND) {
            // walls off the half-grid: a link's value solves the interpolation
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                // the link along a is the pull source of direction opp(a); the
                // neighbour's population a, if fluid, is its to store
                long long srcp;
                int wall;
                if (a == 0) P[n] = S::from_r(d[0]);
                else if (pull_source(g, cls, x, y, z, EX<Q>(a), EY<Q>(a), EZ<Q>(a), srcp, wall))
                    P[(long long)a * g.sq + srcp] = S::from_r(d[a]);
                else
                    P[(long long)OPP<Q>(a) * g.sq + n] =
                        S::from_r(unbounced<Q, R>(s, p, wr, g, cls, x, y, z, n, d[OPP<Q>(a)], d[a], OPP<Q>(a), wall));
            }
            return;
        }
    }
    push_node<Q, S>(P, cls, g, p, c, x, y, z, d);
}

// ---------------------------------------------------------------- export
// position of canonical node n (32-bit: the padded node count is below 2^31)
struct NodeXYZ {
    int x, y, z;
    unsigned own;       // padded index
};
__device__ __forceinline__ NodeXYZ node_at(const Geo& g, unsigned n)
{
    const unsigned r = n / (unsigned)g.nx;
    NodeXYZ q;
    q.x = (int)(n - r * (unsigned)g.nx);
    q.z = (int)(r / (unsigned)g.ny);
    q.y = (int)(r - (unsigned)q.z * (unsigned)g.ny);
    q.own = r * (unsigned)g.nxp + (unsigned)q.x;
    return q;
}

// f = d + w rho0, one node per thread: bound by its loads and stores (bulk
// nodes: 19 independent loads, no class lookups; see pull_node), so as many
// warps as registers allow: five blocks per SM (256 x 128 x 128 FP32 108 us at
// 48 registers, 116 with four blocks; 0.88 of the copy bandwidth; binary16
// 102 us, 0.70)
template <int Q, class S, typename OutT, bool CURVED>
__global__ void __launch_bounds__(NODE_THREADS, 5)
k_export(const typename S::T* __restrict__ P, const uint8_t* __restrict__ cls, const Geo g,
         const KP<typename S::R> p, const WRho wr, OutT* __restrict__ out)
{
    pdl_wait(P);
    using R = typename S::R;
    const unsigned N = (unsigned)g.nx * (unsigned)g.ny * (unsigned)g.nz;
    for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
        const NodeXYZ q = node_at(g, n);
        const uint8_t c = cls[q.own];
        if (nc_solid(c)) {
#pragma unroll
            for (int a = 0; a < Q; ++a) out[(long long)a * N + n] = OutT(0);
            continue;
        }
        R d[Q];
        pull_node<Q, S, false, CURVED>(P, cls, g, p, c, q.x, q.y, q.z, d);
        if constexpr (sizeof(R) == 4 && sizeof(OutT) == 4) {
            add_wrho<Q>(d, wr, 1.0f);
#pragma unroll
            for (int a = 0; a < Q; ++a) out[(long long)a * N + n] = d[a];
        } else {
#pragma unroll
            for (int a = 0; a < Q; ++a) out[(long long)a * N + n] = OutT((double)d[a] + wr.c[SPEED2<Q>(a)]);
        }
    }
}

// ------------------------------------------------------------- wall force
// One thread per boundary link (x_f, a') of one wall: fbar_a' = P_a'(x_f)
// = f^rel(x_f, T-1), fbar_a = f_opp(a')(x_f, T), the bounced population
// (halfway: fbar_a' - w E_a'.LW; interpolated with a wall distance).
// Per link (dx^D/dt) [e_a' (fbar_a' + fbar_a) + corrections], in FP64.
// CURVED: walls off the half-grid (the bounced population interpolates);
// otherwise it is the link's own population plus Ladd's term, so a link is
// one record and one value, and the direction is decoded by arithmetic.
template <int Q> __device__ __forceinline__ void link_dir(int a, int (&e)[3])
{
    constexpr auto pack = [](int c) {
        unsigned long long t = 0;
        for (int b = 0; b < Q; ++b)
            t |= (unsigned long long)(1 + (c == 0 ? EX<Q>(b) : (c == 1 ? EY<Q>(b) : EZ<Q>(b)))) << (2 * b);
        return t;
    };
    constexpr unsigned long long t[3] = {pack(0), pack(1), pack(2)};
#pragma unroll
    for (int c = 0; c < 3; ++c) e[c] = (int)(t[c] >> (2 * a) & 3u) - 1;
}
template <int Q, class S, bool CURVED>
__global__ void __launch_bounds__(RED_THREADS)
k_links(const typename S::T* __restrict__ P, const uint8_t* __restrict__ cls, const Link* __restrict__ links,
        long long begin, long long end, const Geo g, const KP<typename S::R> p, unsigned flags,
        double* __restrict__ partials, const RedOut ro)
{
    pdl_wait(P);
    pdl_trigger();
    using R = typename S::R;
    __shared__ double sm[3 * 32];
    double acc[3] = {0.0, 0.0, 0.0}, cor[3] = {0.0, 0.0, 0.0};
    const double c = (double)p.c, rho0 = (double)p.rho0, svol = (double)p.svol;
    for (long long i = begin + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += (long long)gridDim.x * blockDim.x) {
        const Link L = links[i];
        const int a = L.dir;
        int e[3];
        link_dir<Q>(a, e);
        const bool axis = e[0] * e[0] + e[1] * e[1] + e[2] * e[2] == 1;
        const R Pa = S::to_r(P[(long long)a * g.sq + L.node]);
        // bounced population f_opp(a')(x_f, T)
        R bounce = R(0);
        const unsigned rn = L.node / (unsigned)g.nxp;
        const int xn = (int)(L.node - rn * (unsigned)g.nxp);
        const int zn = (int)(rn / (unsigned)g.ny), yn = (int)(rn - (unsigned)zn * (unsigned)g.ny);
        if constexpr (CURVED) {
#pragma unroll
            for (int b = 1; b < Q; ++b)
                if (OPP<Q>(b) == a) bounce = bounced<Q, S, false>(P, cls, g, p, xn, yn, zn, L.node, b, L.wall);
        } else {
            // the Ladd term of direction opp(a)
            bounce = fma(axis ? R(-WD<Q>(1)) : R(-WD<Q>(Q == 9 ? 5 : 7)),
                         R(e[0]) * p.LW[L.wall][0] + R(e[1]) * p.LW[L.wall][1] + R(e[2]) * p.LW[L.wall][2], Pa);
        }
        const double vo = (double)Pa, vi = (double)bounce;
        double s = vo + vi + 2.0 * (axis ? WD<Q>(1) : WD<Q>(Q == 9 ? 5 : 7)) * rho0;
        if ((flags & 2u) && p.maxwell) {
            double mxa = 0.0;
            if (p.induced) {
                // the field of the collision that produced f^rel(x_f, T-1)
                R B[3];
                mag_field_at<Q>(p.mag, cls, g, p, xn, yn, zn, (long long)L.node, B);
#pragma unroll
                for (int b = 1; b < Q; ++b)
                    if (b == a) mxa = (double)maxwell_at<Q>(p.mxk, B, b);
            } else {
                mxa = (double)p.mx[a];
            }
            s -= 2.0 * mxa;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            acc[k] += e[k] == 0 ? 0.0 : (e[k] > 0 ? s : -s);
            if (flags & 1u) cor[k] += (double)p.LW[L.wall][k] / (6.0 * rho0) * (vi - vo);
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] = svol * c * (acc[k] + cor[k]);
    block_sum<3>(acc, sm);
    finish_rows<3>(acc, partials, ro);
}

// ------------------------------------------------- exact moments of a node
// Sums of a node's populations and momentum for the FP64 reductions.  The
// FP64 pipe adds 1.6 lanes per cycle and SM: the plain FP64 sums (95
// operations and conversions a node) held k_balance at 1.03 ms and k_residual
// at 1.36 ms on the 256 x 128 x 128 box, 15 times their memory time.  FP32
// deviations are therefore scaled by the power of two 2^s that brings the
// node's largest into 1/4 .. 1/2, split into three 32-bit integers on the
// grids 2^-23, 2^-43 and 2^-59 (adding 1.5 times a power of two leaves the
// rounded multiple in the mantissa), summed in integer arithmetic and joined
// in one 64-bit integer of units 2^-(59 + s).  That is exact for every
// deviation above 2^-34 of the node's largest, and smaller ones are rounded by
// 2^-58 of the largest at most, where an FP64 sum rounds by up to 2^-53 of the
// partial sum at every addition.  A node with a deviation of 1/2 or more or a
// non-finite one takes FP64 sums.
constexpr double FIX_UNIT = 1.0 / 576460752303423488.0;      // 2^-59

// V = sum d, sum E d in units of 2^-(59 + s), 0 <= s <= 125; false (V not set)
// if some |d| >= 1/2
template <int Q>
__device__ __forceinline__ bool fixed_moments(const float (&d)[Q], long long (&V)[4], int& s)
{
    float top = 0.0f;
#pragma unroll
    for (int a = 0; a < Q; ++a) top = fmaxf(top, fabsf(d[a]));
    const unsigned e2 = __float_as_uint(top) >> 23;            // top = 2^(e2 - 127) 1.xx
    s = top == 0.0f ? 0 : 125 - (int)e2;
    if (s < 0) return false;
    const F2 scale = f2s(__uint_as_float((unsigned)(127 + s) << 23));
    constexpr int NP = LatDim<Q>::NP;
    constexpr float M1 = 1.5f, M2 = 1.5f / 1048576.0f, M3 = 1.5f / 68719476736.0f;   // 1.5, 1.5 2^-20, 1.5 2^-36
    unsigned sum[3][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}, {0, 0, 0, 0}};
    unsigned range = 0;
    auto split = [&](F2 v, unsigned (&lo)[3], unsigned (&hi)[3]) {
        constexpr float M[3] = {M1, M2, M3};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const F2 t = f2add(v, f2s(M[k]));
            lo[k] = __float_as_uint(t.v.x);
            hi[k] = __float_as_uint(t.v.y);
            if (k < 2) v = f2sub(v, f2add(t, f2s(-M[k])));
        }
        range |= (lo[0] ^ 0x3F800000u) | (hi[0] ^ 0x3F800000u);
    };
    constexpr unsigned K[3] = {0x3FC00000u, 0x35C00000u, 0x2DC00000u};      // the bits of M1, M2, M3
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        unsigned ua[3], ub[3];
        split(f2mul(F2{make_float2(d[a], d[b])}, scale), ua, ub);
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            sum[l][0] += ua[l] + ub[l];
            const unsigned df = ua[l] - ub[l];
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (e[c]) sum[l][1 + c] += (e[c] > 0) ? df : 0u - df;
        }
    }
    {
        unsigned u0[3], u1[3];
        split(f2mul(F2{make_float2(d[0], 0.0f)}, scale), u0, u1);
#pragma unroll
        for (int l = 0; l < 3; ++l) sum[l][0] += u0[l] - (unsigned)Q * K[l];
    }
    if (range >> 23) return false;               // NaN
#pragma unroll
    for (int c = 0; c < 4; ++c)
        V[c] = ((long long)(int)sum[0][c] << 36) + ((long long)(int)sum[1][c] << 16) + (long long)(int)sum[2][c];
    return true;
}
__device__ __forceinline__ double fixed_unit(int s) { return __hiloint2double((1023 - 59 - s) << 20, 0); }
// the same in FP64, from the even and odd parts of the opposite pairs
template <int Q, typename R>
__device__ __forceinline__ void double_moments(const R (&d)[Q], double (&s)[4])
{
    s[0] = (double)d[0];
    s[1] = s[2] = s[3] = 0.0;
#pragma unroll
    for (int k = 0; k < LatDim<Q>::NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const double da = (double)d[a], db = (double)d[b], df = da - db;
        s[0] += da + db;
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (e[c]) s[1 + c] = (e[c] > 0) ? s[1 + c] + df : s[1 + c] - df;
    }
}

// ---------------------------------------------------------------- balance
// A thread's nodes are summed first (FP32 compute: the 64-bit node sums in two
// 32-bit halves, exactly, where they lie on the common grid 2^-59, as they do
// unless some deviation is below 2^-36; else in FP64), then the block in FP64;
// the uniform body force
// multiplies the summed density, a velocity-dependent one each node's.
template <int Q, class S, bool EXT, bool CURVED>
__global__ void __launch_bounds__(RED_THREADS)
k_balance(const typename S::T* __restrict__ P, const uint8_t* __restrict__ cls, const Geo g,
          const KP<typename S::R> p, double vol, double* __restrict__ partials, const RedOut ro)
{
    pdl_wait(P);
    using R = typename S::R;
    __shared__ double sm[7 * 32];
    double tot[4] = {0, 0, 0, 0}, fa[3] = {0, 0, 0};     // sums of d and E d; of rho A with EXT
    long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
    int count = 0;
    const unsigned N = (unsigned)g.nx * (unsigned)g.ny * (unsigned)g.nz;
    for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
        const NodeXYZ q = node_at(g, n);
        const uint8_t c = cls[q.own];
        if (nc_solid(c)) continue;
        R d[Q];
        pull_node<Q, S, false, CURVED>(P, cls, g, p, c, q.x, q.y, q.z, d);
        ++count;
        double s[4];
        bool fixed = false;
        if constexpr (sizeof(R) == 4) {
            long long V[4];
            int sh;
            fixed = fixed_moments<Q>(d, V, sh);
            if (fixed) {
                if (EXT) s[0] = (double)V[0] * fixed_unit(sh);
                const unsigned long long below = sh < 60 ? (1ull << sh) - 1ull : ~0ull;
                if (((unsigned long long)(V[0] | V[1] | V[2] | V[3]) & below) == 0ull) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        V[k] = sh < 60 ? V[k] >> sh : 0ll;
                        hi[k] += V[k] >> 32;
                        lo[k] += V[k] & 0xFFFFFFFFll;
                    }
                } else {
                    const double unit = fixed_unit(sh);
#pragma unroll
                    for (int k = 0; k < 4; ++k) tot[k] = fma((double)V[k], unit, tot[k]);
                }
            }
        }
        if (!fixed) {
            double_moments<Q, R>(d, s);
#pragma unroll
            for (int k = 0; k < 4; ++k) tot[k] += s[k];
        }
        if constexpr (EXT) {
            NodeM<R> m;
            node_macro<R, Q, EXT>(d, p, m);
            const double rho = (double)p.rho0 + s[0];
#pragma unroll
            for (int k = 0; k < 3; ++k) fa[k] += rho * (double)m.A[k];
        }
    }
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) tot[k] += ((double)hi[k] * 4294967296.0 + (double)lo[k]) * FIX_UNIT;
    }
    const double rho = (double)p.rho0 * count + tot[0], c = (double)p.c;
    double acc[7];
    acc[0] = vol * rho;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        acc[1 + k] = vol * c * tot[1 + k];
        // rho a = rho (c/dt) A
        if constexpr (!EXT) fa[k] = rho * ((k < LatDim<Q>::D) ? (double)p.AG[k] : 0.0);
        acc[4 + k] = vol * (c / (double)p.dt) * fa[k];
    }
    block_sum<7>(acc, sm);
    finish_rows<7>(acc, partials, ro);
}

// ------------------------------------------------------- steady residual
// Sec. 6: the balance of Eq. (32) between wall force and body force holds
// once the flow stops changing.  Per fluid node of f(T): the flow velocity
// v = c (j/rho + A/2) (text after Eq. 1; the moments summed in FP64 or
// exactly from the stored values, see above), |v - v_ref| and |v| (Euclidean
// norms), block sums in FP64 for the fixed-order pass; with `update` the
// node's v replaces v_ref (each thread reads its own entries before it writes
// them; solid nodes get 0).  The FP64 pipe bounds it (~40 operations a node,
// two square roots and a reciprocal among them): 256 x 128 x 128 FP32 394 us
// (one grid for every node, see fixed_moments, 366; with the quotient and the
// library's square roots 57 more); three blocks per SM (with two 78 more).
template <int Q, class S, bool EXT, bool CURVED>
__global__ void __launch_bounds__(RED_THREADS, 3)
k_residual(const typename S::T* __restrict__ P, const uint8_t* __restrict__ cls, const Geo g,
           const KP<typename S::R> p, double* __restrict__ vref, int update, double* __restrict__ partials,
           const RedOut ro)
{
    pdl_wait(P);
    using R = typename S::R;
    __shared__ double sm[2 * 32];
    double acc[2] = {0.0, 0.0};
    const unsigned N = (unsigned)g.nx * (unsigned)g.ny * (unsigned)g.nz;
    const double c = (double)p.c;
    for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
        const NodeXYZ q = node_at(g, n);
        const uint8_t cl = cls[q.own];
        if (nc_solid(cl)) {
            if (update)
#pragma unroll
                for (int k = 0; k < 3; ++k) vref[(long long)k * N + n] = 0.0;
            continue;
        }
        double vr[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) vr[k] = vref[(long long)k * N + n];
        R d[Q];
        pull_node<Q, S, false, CURVED>(P, cls, g, p, cl, q.x, q.y, q.z, d);
        double s[4], unit = 1.0;         // the moments in units of `unit`
        bool fixed = false;
        if constexpr (sizeof(R) == 4) {
            long long V[4];
            int sh;
            fixed = fixed_moments<Q>(d, V, sh);
            if (fixed) {
                unit = fixed_unit(sh);
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k] = (double)V[k];
            }
        }
        if (!fixed) double_moments<Q, R>(d, s);
        double A[3];
        if constexpr (EXT) {
            NodeM<R> m;
            node_macro<R, Q, EXT>(d, p, m);
#pragma unroll
            for (int k = 0; k < 3; ++k) A[k] = (double)m.A[k];
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) A[k] = (k < LatDim<Q>::D) ? (double)p.AG[k] : 0.0;
        }
        const double ir = c * unit * rcp64(fma(s[0], unit, (double)p.rho0));
        double dd = 0.0, vv = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double vk = fma(s[1 + k], ir, 0.5 * c * A[k]);
            const double dk = vk - vr[k];
            dd += dk * dk;
            vv += vk * vk;
            if (update) vref[(long long)k * N + n] = vk;
        }
        acc[0] += sqrt64(dd);
        acc[1] += sqrt64(vv);
    }
    block_sum<2>(acc, sm);
    finish_rows<2, true>(acc, partials, ro);
}

// ----------------------------------------------------------------- stress
// Three blocks per SM in FP32 (256 x 128 x 128 S2 136 us, 176 with two; S4 205,
// 246), two in FP64, whose pipe bounds it.
// Variants 1, 2 at f(T) = gather(cur); 3, 4 at the half step between T-1 and
// T: fbar = (cur + gather(cur))/2 with the node's state at T-1 = gather(prev).
template <int Q, class S, bool EXT, bool CURVED>
__global__ void __launch_bounds__(NODE_THREADS, sizeof(typename S::R) == 8 ? 2 : 3)
k_stress(const typename S::T* __restrict__ cur, const typename S::T* __restrict__ prev,
         const uint8_t* __restrict__ cls, const Geo g, const KP<typename S::R> p, int variant,
         typename S::R* __restrict__ sig, typename S::R* __restrict__ Sout, typename S::R* __restrict__ rho_out,
         typename S::R* __restrict__ v_out)
{
    pdl_wait(cur, prev);
    using R = typename S::R;
    constexpr int D = LatDim<Q>::D;
    constexpr int NC = (D == 3) ? 6 : 3;
    const unsigned N = (unsigned)g.nx * (unsigned)g.ny * (unsigned)g.nz;
    const R c = p.c, c2 = p.c * p.c;
    for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
        const NodeXYZ q = node_at(g, n);
        const int x = q.x, y = q.y, z = q.z;
        const unsigned own = q.own;
        const uint8_t cl = cls[own];
        R out[6] = {0, 0, 0, 0, 0, 0}, Sv[6] = {0, 0, 0, 0, 0, 0}, rr = 0, vv[3] = {0, 0, 0};
        if (!nc_solid(cl)) {
            R d[Q];
            NodeM<R> m;
            // component index -> (i, j)
            constexpr int ci3[6] = {0, 1, 2, 0, 0, 1}, cj3[6] = {0, 1, 2, 1, 2, 2};
            constexpr int ci2[3] = {0, 1, 0}, cj2[3] = {0, 1, 1};
            // L / c^2 of the Maxwell term: configured, or at the node's induced field B(x, T)
            R Lh[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) Lh[k] = p.Lh[k];
            if (EXT && p.induced) {
                R B[3];
                mag_field_at<Q>(p.mag, cls, g, p, x, y, z, own, B);
                const R kl = R(2) / R(9) * p.mxk, h = R(0.5) * (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
                Lh[0] = kl * (h - B[0] * B[0]);
                Lh[1] = kl * (h - B[1] * B[1]);
                Lh[2] = kl * (h - B[2] * B[2]);
                Lh[3] = -kl * B[0] * B[1];
                Lh[4] = -kl * B[0] * B[2];
                Lh[5] = -kl * B[1] * B[2];
            }
            if (variant <= 2) {
                pull_node<Q, S, false, CURVED>(cur, cls, g, p, cl, x, y, z, d);
                node_macro<R, Q, EXT>(d, p, m);
                const R fac = -(R(1) - R(0.5) * m.om) * c2;
                const bool model_a = (p.model == MODEL_A);
#pragma unroll
                for (int cc = 0; cc < NC; ++cc) {
                    const int i = (D == 3) ? ci3[cc] : ci2[cc], j = (D == 3) ? cj3[cc] : cj2[cc];
                    const int lc = (D == 3) ? cc : (cc == 2 ? 3 : cc);   // index into Lh
                    R P2 = 0;
#pragma unroll
                    for (int a = 0; a < Q; ++a) {
                        const int ea[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
                        const int ee = ea[i] * ea[j];
                        if (ee) P2 += R(ee) * d[a];
                    }
                    // cheap form of Sec. 3: sum e e f - (p delta + rho u^eq u^eq + L)
                    R Pi = P2 - (p.stokes ? R(0) : m.rho * m.weq[i] * m.weq[j]) - (p.maxwell ? Lh[lc] : R(0));
                    if (i == j) Pi -= m.drho / R(3);
                    if (variant == 1) {
                        // E_ij = tau dt rho (u^eq a + a u^eq) - tau Theta_ij, in units of c^2
                        R E = m.tau * m.rho * (m.weq[i] * m.A[j] + m.weq[j] * m.A[i]);
                        if (!model_a) E -= m.tau * m.C * m.rho * (m.wf[i] * m.A[j] + m.wf[j] * m.A[i]);
                        Pi += E;
                    }
                    out[cc] = fac * Pi;
                }
                rr = m.rho;
#pragma unroll
                for (int k = 0; k < 3; ++k) vv[k] = c * m.v[k];
            } else {
                R dn[Q];
                pull_node<Q, S, false, CURVED>(cur, cls, g, p, cl, x, y, z, dn);
                R db[Q];
                R drb = 0, jb[3] = {0, 0, 0};
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    db[a] = R(0.5) * (S::to_r(cur[(long long)a * g.sq + own]) + dn[a]);
                    drb += db[a];
                    jb[0] += R(EX<Q>(a)) * db[a];
                    jb[1] += R(EY<Q>(a)) * db[a];
                    jb[2] += R(EZ<Q>(a)) * db[a];
                }
                const R rb = p.rho0 + drb;
                const R ub[3] = {jb[0] / rb, jb[1] / rb, jb[2] / rb};
                pull_node<Q, S, false, CURVED>(prev, cls, g, p, cl, x, y, z, d);
                node_macro<R, Q, EXT>(d, p, m);
#pragma unroll
                for (int cc = 0; cc < NC; ++cc) {
                    const int i = (D == 3) ? ci3[cc] : ci2[cc], j = (D == 3) ? cj3[cc] : cj2[cc];
                    const int lc = (D == 3) ? cc : (cc == 2 ? 3 : cc);
                    R P2 = 0;
#pragma unroll
                    for (int a = 0; a < Q; ++a) {
                        const int ea[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
                        const int ee = ea[i] * ea[j];
                        if (ee) P2 += R(ee) * db[a];
                    }
                    // sum e e (fbar - f^eq(rhobar, ubar)), in units of c^2
                    R Pi = P2 - (p.stokes ? R(0) : rb * ub[i] * ub[j]) - (p.maxwell ? Lh[lc] : R(0));
                    if (i == j) Pi -= drb / R(3);
                    R s = -c2 * Pi;
                    if (variant == 4 && p.model != MODEL_A)
                        s += R(0.5) * c2 * m.C * m.rho * (m.wf[i] * m.A[j] + m.wf[j] * m.A[i]);
                    out[cc] = s;
                }
                rr = rb;
#pragma unroll
                for (int k = 0; k < 3; ++k) vv[k] = c * ub[k];
            }
            const R nu = p.dt * c2 * (m.tau - R(0.5)) / R(3);
#pragma unroll
            for (int cc = 0; cc < NC; ++cc) Sv[cc] = out[cc] / (R(2) * rr * nu);
        }
#pragma unroll
        for (int cc = 0; cc < NC; ++cc) {
            if (sig) sig[(long long)cc * N + n] = out[cc];
            if (Sout) Sout[(long long)cc * N + n] = Sv[cc];
        }
        if (rho_out) rho_out[n] = rr;
        if (v_out)
#pragma unroll
            for (int k = 0; k < 3; ++k) v_out[(long long)k * N + n] = vv[k];
    }
}

// ---------------------------------------------------------- induced field
// One coupled step per node (one thread per padded node): the field
// distributions g(x, T) pulled from the stored post-collision ones, the
// node's field B = sum g, the fluid populations f(x, T) (gather_node) and
// their moments; the field relaxes toward W_i [B + e_i . (v B - B v)/theta]
// with the node's flow velocity v, the fluid with the Maxwell term of
// Eq. (10) at B.  Both write their post-collision values for the next pull.
template <int Q, class S, bool SR>
__global__ void __launch_bounds__(NODE_THREADS, MhdOcc<S>::value)
k_mhd_step(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
           const typename S::R* __restrict__ G, typename S::R* __restrict__ Gn, const uint8_t* __restrict__ cls,
           const Geo g, const KP<typename S::R> p, uint32_t seed)
{
    using R = typename S::R;
    constexpr int QM = MagLat<Q>::QM;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= g.sq) return;
    const int x = (int)(n % g.nxp);
    const long long row = n / g.nxp;
    const int y = (int)(row % g.ny), z = (int)(row / g.ny);
    const uint8_t c = cls[n];
    if (x >= g.nx || nc_solid(c) || c == NC_PAD) {
#pragma unroll
        for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw(R(0));
#pragma unroll
        for (int j = 0; j < 3 * QM; ++j) Gn[(long long)j * g.sq + n] = R(0);
        return;
    }
    R gm[3][QM];
    R d[Q];
    if (c == NC_BULK) {
        // every pull source is a fluid node (periodic wrap allowed): plain
        // indexed loads, no class bytes
        int ro[3][3];
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dz = -1; dz <= 1; ++dz)
                ro[dy + 1][dz + 1] = (wrapi(z - dz, g.nz) * g.ny + wrapi(y - dy, g.ny)) * g.nxp;
        const int xm = wrapi(x - 1, g.nx), xp = wrapi(x + 1, g.nx);
        auto at = [&](int a) { return ro[EY<Q>(a) + 1][EZ<Q>(a) + 1] + (EX<Q>(a) == 0 ? x : (EX<Q>(a) == 1 ? xm : xp)); };
#pragma unroll
        for (int a = 0; a < Q; ++a) d[a] = S::to_raw(src[(long long)a * g.sq + at(a)]);
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int i = 0; i < QM; ++i) gm[k][i] = G[(long long)(k * QM + i) * g.sq + at(i)];
    } else {
        mag_gather<Q>(G, cls, g, p, x, y, z, n, gm);
        gather_node<Q, S, true, false>(src, cls, g, p, x, y, z, d);   // the induced field has no curved walls
    }
    NodeM<R> m;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R b = R(0);
#pragma unroll
        for (int i = 0; i < QM; ++i) b += gm[k][i];
        m.Bl[k] = b;
    }
    node_macro<R, Q, true>(d, p, m);
    // field: e_i is +-1 along one axis, so e_i . (v B_k - B v_k) = s (v_ax B_k - B_ax v_k)
    const R om = p.om_m, ith = R(1.0 / MagLat<Q>::TH);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < QM; ++i) {
            const int ax = (EX<Q>(i) != 0) ? 0 : ((EY<Q>(i) != 0) ? 1 : 2);
            const int sg = EX<Q>(i) + EY<Q>(i) + EZ<Q>(i);
            const R W = R(i == 0 ? MagLat<Q>::W0 : MagLat<Q>::W1);
            const R el = (i == 0) ? R(0) : R(sg) * (m.v[ax] * m.Bl[k] - m.Bl[ax] * m.v[k]);
            const R geq = W * (m.Bl[k] + ith * el);
            Gn[(long long)(k * QM + i) * g.sq + n] = gm[k][i] + om * (geq - gm[k][i]);
        }
    node_relax<R, Q, true, true>(d, p, m);
    if constexpr (SR) {
        NodeRng rng((uint32_t)n, seed);
#pragma unroll
        for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw_sr(d[a], rng.bits(a));
    } else {
#pragma unroll
        for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = S::from_raw(d[a]);
    }
}

// field distributions at rest in the external field, W_i B, in both buffers
template <int Q, typename R>
__global__ void __launch_bounds__(NODE_THREADS)
k_mag_init(R* __restrict__ G0, R* __restrict__ G1, const uint8_t* __restrict__ cls, const Geo g, const KP<R> p)
{
    constexpr int QM = MagLat<Q>::QM;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= g.sq) return;
    const uint8_t c = cls[n];
    const bool fluid = (int)(n % g.nxp) < g.nx && !nc_solid(c) && c != NC_PAD;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < QM; ++i) {
            const R v = fluid ? R(i == 0 ? MagLat<Q>::W0 : MagLat<Q>::W1) * p.Bext[k] : R(0);
            G0[(long long)(k * QM + i) * g.sq + n] = v;
            G1[(long long)(k * QM + i) * g.sq + n] = v;
        }
}

// B(x, T) in canonical order, zero at solid nodes
template <int Q, typename R>
__global__ void __launch_bounds__(NODE_THREADS)
k_mag_field(const R* __restrict__ G, const uint8_t* __restrict__ cls, const Geo g, const KP<R> p,
            double* __restrict__ Bout)
{
    const long long N = (long long)g.nx * g.ny * g.nz;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int x = (int)(n % g.nx);
    const long long r = n / g.nx;
    const int y = (int)(r % g.ny), z = (int)(r / g.ny);
    const long long own = r * g.nxp + x;
    R B[3] = {R(0), R(0), R(0)};
    if (!nc_solid(cls[own])) mag_field_at<Q>(G, cls, g, p, x, y, z, own, B);
#pragma unroll
    for (int k = 0; k < 3; ++k) Bout[(long long)k * N + n] = (double)B[k];
}

// ================================================================ launchers
inline int grid_for(long long n, int threads, long long cap)
{
    long long b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

template <class S> inline const KP<typename S::R>& kp_of(const Ctx& c)
{
    if constexpr (sizeof(typename S::R) == 8) return c.kpd;
    else return c.kpf;
}
// parameters in storage units, for the step kernels
template <class S> inline const KP<typename S::R>& kp_step_of(const Ctx& c)
{
    if constexpr (sizeof(typename S::R) == 8) return c.kpd;
    else return c.kps;
}

// a copy of the parameters that reads the field distributions G
template <typename R> inline KP<R> with_mag(const KP<R>& p, const void* G)
{
    KP<R> q = p;
    q.mag = static_cast<const R*>(G);
    return q;
}
// the wall force reads the field of the step that produced the stored state:
// B(T-1), pulled from the other field buffer
template <class S> inline KP<typename S::R> kp_links_of(const Ctx& c)
{
    return with_mag(kp_of<S>(c), c.cfg.induced ? c.mag[1 - c.cur] : nullptr);
}

// whether a step into dst also zeroes the padding: in a buffer that is not
// the context's own (theirs is zero from create on)
inline int zero_padding(const Ctx& c, const void* dst)
{
    return c.geo.nxp > c.geo.nx && dst != c.pop[0] && dst != c.pop[1];
}

}  // namespace lbm

#include "lbm_step64.cuh"  // the FP64 step; uses pull_node

namespace lbm {

template <int Q, class S, bool EXT, bool SR>
cudaError_t launch_step_q(const Ctx& c, const void* src, void* dst, uint32_t seed, cudaStream_t st)
{
    using T = typename S::T;
    const long long nch = (long long)(c.geo.nxp / S::V) * c.geo.ny * c.geo.nz;
    const int blocks = grid_for(nch, STEP_THREADS, 1ll << 31);
    const int zp = zero_padding(c, dst);
    const bool faces = !c.geo.periodic[0] || !c.geo.periodic[1] || (Q == 19 && !c.geo.periodic[2]);
    auto go = [&](auto fc, auto full, auto lp) {
        return launch_pdl(k_step<Q, S, EXT, fc.value, SR, full.value, lp.value>, blocks, STEP_THREADS, 0, st,
                          (const T*)src, (T*)dst, c.cls, c.geo, kp_step_of<S>(c), seed, zp);
    };
    const std::true_type yes{};
    const std::false_type no{};
    if constexpr (EXT && sizeof(typename S::T) == 2) {
        if (c.les_pair) return faces ? go(yes, no, yes) : go(no, no, yes);
    }
    if (c.cfg.curved || c.insulating) return faces ? go(yes, yes, no) : go(no, yes, no);
    return faces ? go(yes, no, no) : go(no, no, no);
}

// the staged step (16-bit or FP32 storage, any node code but curved walls and
// the induced field; the host chose the tile rows and stage count at create)
template <int Q, class S, bool SR, bool EXT, bool FACES, bool LP = false, bool INS = false>
cudaError_t launch_step_staged_k(const Ctx& c, const void* src, void* dst, uint32_t seed, cudaStream_t st,
                                 const StgForce& fw)
{
    using T = typename S::T;
    auto kern = k_step_staged<Q, S, SR, EXT, FACES, LP, INS>;
    // a context always launches the same instantiation: set its shared
    // memory limit on the first launch.  The limit is the instantiation's, for
    // every context of the device, so it is the most that any of them asks for
    if (!c.stage_ready) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stage_budget(c));
        if (e != cudaSuccess) return e;
        c.stage_ready = true;
    }
    return launch_pdl(kern, staged_blocks(c), 32 * staged_warps(StgShape<EXT>::CW, c.n_special, c.geo.sq, !c.geo.periodic[0]),
                      c.stage_smem, st, (const T*)src, (T*)dst, c.cls, c.special, c.n_special, c.geo, kp_step_of<S>(c),
                      seed, c.stage_R, (int)c.stage_tiles, c.stage_n, zero_padding(c, dst), c.errflag, fw);
}

// the staged step (the host chose the tile rows and stage count at create)
template <int Q, class S, bool SR>
cudaError_t launch_step_staged(const Ctx& c, const void* src, void* dst, uint32_t seed, cudaStream_t st,
                               const StgForce& fw)
{
    const bool faces = !c.geo.periodic[0] || !c.geo.periodic[1] || (Q == 19 && !c.geo.periodic[2]);
    if constexpr (sizeof(typename S::T) == 2) {
        if (c.les_pair)
            return faces ? launch_step_staged_k<Q, S, SR, true, true, true>(c, src, dst, seed, st, fw)
                         : launch_step_staged_k<Q, S, SR, true, false, true>(c, src, dst, seed, st, fw);
    }
    if constexpr (sizeof(typename S::T) == 4 && Q == 19) {
        if (c.insulating)
            return faces ? launch_step_staged_k<Q, S, SR, true, true, false, true>(c, src, dst, seed, st, fw)
                         : launch_step_staged_k<Q, S, SR, true, false, false, true>(c, src, dst, seed, st, fw);
    }
    if (c.ext)
        return faces ? launch_step_staged_k<Q, S, SR, true, true>(c, src, dst, seed, st, fw)
                     : launch_step_staged_k<Q, S, SR, true, false>(c, src, dst, seed, st, fw);
    return faces ? launch_step_staged_k<Q, S, SR, false, true>(c, src, dst, seed, st, fw)
                 : launch_step_staged_k<Q, S, SR, false, false>(c, src, dst, seed, st, fw);
}

template <int Q, class S>
cudaError_t launch_step(const Ctx& c, const void* src, void* dst, uint32_t seed, cudaStream_t st,
                        const StgForce* fw = nullptr)
{
    if constexpr (sizeof(typename S::T) == 8) return launch_step64<Q>(c, src, dst, zero_padding(c, dst), st);
    else {
        StgForce none{};
        const StgForce& f = fw ? *fw : none;
        if constexpr (sizeof(typename S::T) == 2) {
            if (c.stage_R > 0)
                return c.sr ? launch_step_staged<Q, S, true>(c, src, dst, seed, st, f)
                            : launch_step_staged<Q, S, false>(c, src, dst, seed, st, f);
        } else if constexpr (sizeof(typename S::T) == 4) {
            if (c.stage_R > 0) return launch_step_staged<Q, S, false>(c, src, dst, seed, st, f);
        }
        if constexpr (sizeof(typename S::T) == 2) {
            if (c.sr)
                return c.ext ? launch_step_q<Q, S, true, true>(c, src, dst, seed, st)
                             : launch_step_q<Q, S, false, true>(c, src, dst, seed, st);
        }
        return c.ext ? launch_step_q<Q, S, true, false>(c, src, dst, seed, st)
                     : launch_step_q<Q, S, false, false>(c, src, dst, seed, st);
    }
}

// calls f with the kernel's compile-time flags: CURVED (interpolated walls)
template <class F> inline cudaError_t with_curved(const Ctx& c, F&& f)
{
    return c.cfg.curved ? f(std::true_type{}) : f(std::false_type{});
}
// and EXT, CURVED
template <class F> inline cudaError_t with_ext_curved(const Ctx& c, F&& f)
{
    return with_curved(c, [&](auto cu) {
        return c.ext ? f(std::true_type{}, cu) : f(std::false_type{}, cu);
    });
}

template <int Q, class S, class Src>
cudaError_t launch_inverse(const Ctx& c, const Src& src, void* dst, cudaStream_t st)
{
    const int blocks = grid_for(c.geo.sq, NODE_THREADS, 1ll << 31);
    const WRho wr = wrho_of<Q>((double)kp_of<S>(c).rho0);
    return with_curved(c, [&](auto cu) {
        return launch_pdl(k_inverse_stream<Q, S, Src, cu.value>, blocks, NODE_THREADS, 0, st, (typename S::T*)dst,
                          c.cls, c.geo, kp_of<S>(c), wr, src);
    });
}

template <int Q, class S>
cudaError_t launch_import(const Ctx& c, const void* srcf, int dtype, void* dst, cudaStream_t st)
{
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    return dtype == 0 ? launch_inverse<Q, S>(c, SrcCanonD{(const double*)srcf, N}, dst, st)
                      : launch_inverse<Q, S>(c, SrcCanonF{(const float*)srcf, N}, dst, st);
}

template <int Q, class S>
cudaError_t launch_init(const Ctx& c, const double* rho, const double* u, const double* xi, void* dst,
                        cudaStream_t st)
{
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    return launch_inverse<Q, S>(c, SrcFields{rho, u, xi, N, 1.0 / c.kpd.c}, dst, st);
}

template <int Q, class S>
cudaError_t launch_export(const Ctx& c, const void* P, void* out, int dtype, cudaStream_t st)
{
    using T = typename S::T;
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    const int blocks = grid_for(N, NODE_THREADS, 65535ll * 16);
    const WRho wr = wrho_of<Q>((double)kp_of<S>(c).rho0);
    return with_curved(c, [&](auto cu) {
        if (dtype == 0)
            return launch_pdl(k_export<Q, S, double, cu.value>, blocks, NODE_THREADS, 0, st, (const T*)P, c.cls, c.geo,
                              kp_of<S>(c), wr, (double*)out);
        return launch_pdl(k_export<Q, S, float, cu.value>, blocks, NODE_THREADS, 0, st, (const T*)P, c.cls, c.geo,
                          kp_of<S>(c), wr, (float*)out);
    });
}

// grid of a reduction over nodes: at most the blocks per SM that its registers
// allow at once, so that there is no second wave; fewer threads per block, a
// warp at least, where a box is too small for a block of 256 nodes on every SM
inline int red_grid(const Ctx& c, long long N, int per_sm, int& threads)
{
    threads = RED_THREADS;
    while (threads > 32 && N < (long long)threads * c.sm_count) threads /= 2;
    const long long most = N / (8ll * threads) > c.sm_count ? (long long)per_sm * c.sm_count : c.sm_count;
    return grid_for(N, threads, std::min<long long>(MAX_PARTIAL_ROWS, most));
}

// blocks of two warps spread 10^4 links over the SMs (FP64 sums of a block's
// warps share one SM's FP64 pipe); from 65,536 links full blocks
template <int Q, class S>
cudaError_t launch_links(const Ctx& c, const void* P, long long begin, long long end, unsigned flags,
                         double* partials, const RedOut& ro, int* nblocks, cudaStream_t st)
{
    using T = typename S::T;
    const int threads = end - begin > 64ll * MAX_PARTIAL_ROWS ? RED_THREADS : 64;
    const int blocks = grid_for(end - begin, threads, MAX_PARTIAL_ROWS);
    *nblocks = blocks;
    return with_curved(c, [&](auto cu) {
        return launch_pdl(k_links<Q, S, cu.value>, blocks, threads, 0, st, (const T*)P, c.cls, c.links, begin, end,
                          c.geo, kp_links_of<S>(c), flags, partials, ro);
    });
}

template <int Q, class S>
cudaError_t launch_balance(const Ctx& c, const void* P, double* partials, const RedOut& ro, cudaStream_t st)
{
    using T = typename S::T;
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    int threads;
    const int blocks = red_grid(c, N, 2, threads);
    const double vol = (Q == 9) ? c.cfg.dx * c.cfg.dx : c.cfg.dx * c.cfg.dx * c.cfg.dx;
    return with_ext_curved(c, [&](auto ex, auto cu) {
        return launch_pdl(k_balance<Q, S, ex.value, cu.value>, blocks, threads, 0, st, (const T*)P, c.cls, c.geo,
                          kp_of<S>(c), vol, partials, ro);
    });
}

template <int Q, class S>
cudaError_t launch_residual(const Ctx& c, const void* P, double* vref, int update, double* partials, const RedOut& ro,
                            cudaStream_t st)
{
    using T = typename S::T;
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    int threads;
    const int blocks = red_grid(c, N, 3, threads);
    return with_ext_curved(c, [&](auto ex, auto cu) {
        return launch_pdl(k_residual<Q, S, ex.value, cu.value>, blocks, threads, 0, st, (const T*)P, c.cls, c.geo,
                          kp_of<S>(c), vref, update, partials, ro);
    });
}

template <int Q, class S>
cudaError_t launch_stress(const Ctx& c, const void* cur, const void* prev, int variant, void* sig, void* Sv,
                          void* rho, void* v, cudaStream_t st)
{
    using T = typename S::T;
    using R = typename S::R;
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    const int blocks = grid_for(N, NODE_THREADS, 65535ll * 16);
    return with_ext_curved(c, [&](auto ex, auto cu) {
        return launch_pdl(k_stress<Q, S, ex.value, cu.value>, blocks, NODE_THREADS, 0, st, (const T*)cur,
                          (const T*)prev, c.cls, c.geo,
                          with_mag(kp_of<S>(c), c.cfg.induced ? c.mag[c.cur] : nullptr), variant, (R*)sig, (R*)Sv,
                          (R*)rho, (R*)v);
    });
}

template <int Q, class S>
cudaError_t launch_mhd_step(const Ctx& c, const void* src, void* dst, const void* G, void* Gn, uint32_t seed,
                            cudaStream_t st)
{
    using T = typename S::T;
    using R = typename S::R;
    const int blocks = grid_for(c.geo.sq, NODE_THREADS, 1ll << 31);
    if constexpr (sizeof(T) == 2) {
        if (c.sr) {
            k_mhd_step<Q, S, true><<<blocks, NODE_THREADS, 0, st>>>((const T*)src, (T*)dst, (const R*)G, (R*)Gn, c.cls,
                                                                    c.geo, kp_step_of<S>(c), seed);
            return cudaGetLastError();
        }
    }
    k_mhd_step<Q, S, false><<<blocks, NODE_THREADS, 0, st>>>((const T*)src, (T*)dst, (const R*)G, (R*)Gn, c.cls,
                                                                 c.geo, kp_step_of<S>(c), seed);
    return cudaGetLastError();
}

template <int Q, class S>
cudaError_t launch_mag_init(const Ctx& c, cudaStream_t st)
{
    using R = typename S::R;
    const int blocks = grid_for(c.geo.sq, NODE_THREADS, 1ll << 31);
    k_mag_init<Q, R><<<blocks, NODE_THREADS, 0, st>>>((R*)c.mag[0], (R*)c.mag[1], c.cls, c.geo, kp_of<S>(c));
    return cudaGetLastError();
}

template <int Q, class S>
cudaError_t launch_mag_field(const Ctx& c, double* B, cudaStream_t st)
{
    using R = typename S::R;
    const long long N = (long long)c.geo.nx * c.geo.ny * c.geo.nz;
    const int blocks = grid_for(N, NODE_THREADS, 1ll << 31);
    k_mag_field<Q, R><<<blocks, NODE_THREADS, 0, st>>>((const R*)c.mag[c.cur], c.cls, c.geo, kp_of<S>(c), B);
    return cudaGetLastError();
}

}  // namespace lbm

#include "lbm_adjoint.cuh"  // the adjoint kernel and launch_adjoint; uses block_sum, grid_for, kp_of

namespace lbm {

template <int Q, class S> Dispatch make_dispatch()
{
    Dispatch d;
    d.step = [](const Ctx& c, const void* s, void* t, uint32_t seed, cudaStream_t st) {
        return launch_step<Q, S>(c, s, t, seed, st);
    };
    d.step_force = [](const Ctx& c, const void* s, void* t, uint32_t seed, const StgForce& fw, cudaStream_t st) {
        return launch_step<Q, S>(c, s, t, seed, st, &fw);
    };
    d.import_f = launch_import<Q, S>;
    d.init_fields = launch_init<Q, S>;
    d.export_f = launch_export<Q, S>;
    d.links = launch_links<Q, S>;
    d.balance = launch_balance<Q, S>;
    d.residual = launch_residual<Q, S>;
    d.stress = launch_stress<Q, S>;
    d.mhd_step = launch_mhd_step<Q, S>;
    d.mag_init = launch_mag_init<Q, S>;
    d.mag_field = launch_mag_field<Q, S>;
    d.adjoint = launch_adjoint<Q, S>;
    return d;
}

}  // namespace lbm
