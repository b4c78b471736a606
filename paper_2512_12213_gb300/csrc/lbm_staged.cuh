// lbm_staged.cuh -- the fused collide-stream step (Eq. 2 with Eqs. 1 and 3,
// and Eq. 10 with the Maxwell term) as a persistent kernel whose input rows
// are staged in shared memory by the bulk asynchronous copies of the tensor
// memory accelerator, for 16-bit or FP32 storage with halfway walls, closed
// or periodic box faces and every node code but the induced field; insulating
// walls in FP32 on D3Q19 (the INS instantiation).
//
// Pull scheme: a tile is R consecutive rows (y0 .. y0+R-1) of one z plane;
// for direction a the tile reads the R source rows shifted by (E_y, E_z),
// which lie contiguously in that direction's plane, so one bulk copy per
// direction (two where the rows wrap around the periodic y axis) brings them
// in, and every stored population is read from HBM once per step.  The x
// shift of the pull is an offset inside the staged row (the periodic x wrap
// an index at the row ends): no shuffles, and no register holds a load in
// flight.  A bulk copy costs the copy engine of an SM a fixed time (measured
// ~33 ns on GB300 whether it moves 512 B or 1 KB), so R is chosen for copies
// of at least 2 KB per direction (R nxp = 1024 nodes for 16-bit storage, 512
// for FP32), and the relaxed populations leave with ordinary coalesced
// stores, which cost the copy engine nothing.
//
// One producer warp keeps up to 8 stages in flight (lane a copies direction
// a): it refills a stage as soon as the consumer warps have released it (full
// / empty mbarriers, the full one with the copies' transaction bytes).  The
// consumer warps form groups that take alternate tiles, a group's warps its
// 64-node tasks in turn.  The number of stages is a multiple of the number of
// groups, so every stage belongs to one group, and every warp of a group
// waits for and releases each of its tiles, with a task in it or not: a warp
// can then only wait on the use of a stage whose predecessor it has released
// itself, and a parity wait cannot mistake a phase two uses old for the
// current one.  A thread relaxes one pair
// of nodes of a 64-node warp task at a time (one 32-bit word per direction
// for 16-bit storage, one float2 for FP32) with k_step's node code for the
// configuration.  Closed faces follow k_step: a source row outside a closed
// y or z face is the node's own row of the opposite direction (the producer
// copies that row instead), the element outside a closed x face is the
// node's own opposite population (the producer stages these face values),
// and moving faces add Ladd's term.  The 4-node chunks that touch a solid
// node, a wall or the end of a ragged row are not the pipeline's: the
// boundary warps take their share of their list (built on the host) and
// compute them node by node from global memory with explicit bounce-back,
// exactly as k_step does, beside the pipeline -- inline, one such chunk held up its
// stage and with it the in-order producer (the sphere box ran at half the
// rate of the same box without the sphere).  The arithmetic and the
// stochastic rounding stream are those of k_step, so the two kernels store
// the same bits.
//
// Every mbarrier wait is bounded (about a second of the global timer); on
// expiry a warp records a flag for lbm_device_status and stops, and the
// producer waits (again bounded) for the copies it issued before it returns.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// Consumer warps, in G groups of W that take alternate tiles.  Without the EXT
// terms two groups of 8: with the producer and up to three others that is
// five warps on each of the SM's four sub-partitions, 96 registers, which the
// plain node code fits, and while one group starts a tile the other is in the
// middle of one (binary16 sphere 256 x 128 x 128 54.5 us; one group of 16
// 58.1, of 12 55.0; bfloat16 250 x 121 x 99 54.1, 62.8, 61.1).  The LES and
// EXT node codes spill at 96: one group of 12, four warps a sub-partition,
// 128 registers (cavity 256^3: binary16 327 us against 334 for two groups of
// 8, FP32 427 against 441; Brinkman box FP32 100 against 106).
template <bool EXT> struct StgShape {
    static constexpr int G = EXT ? 1 : 2, W = EXT ? 12 : 8;
    static constexpr int CW = G * W;
    static constexpr int MAXW = CW + 4;          // warps of a block at most
};
// boundary warps: one, or as many as the block may hold where more than 0.5%
// of the chunks are special (a ragged row has one in every row).  The kernel
// takes the number from its block size.
inline int staged_warps(int cw, long long n_special, long long nodes, bool closed_x)
{
    return n_special * 200 > nodes / 4 ? cw + 4 : cw + 2 + (closed_x ? 1 : 0);
}
constexpr int STG_COPY_BYTES = 2048;                  // least bytes per direction and tile
constexpr int STG_TASK_NODES = 64;                    // nodes per warp task (32 pairs)
constexpr int STG_MAX_STAGES = 8;
constexpr unsigned long long STG_WAIT_NS = 1000000000ull;   // bounded waits: 1 s
constexpr unsigned STG_ERR_TIMEOUT = 1u;
constexpr unsigned STG_ERR_CONFIG = 2u;                     // a launch with a stage count out of range

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// true once the phase of this parity has completed; false after ~1 s
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > STG_WAIT_NS) return false;
    return true;
}
// bulk copy global -> shared, completing on the mbarrier's transaction count;
// both addresses 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

__host__ __device__ inline size_t stg_round128(size_t b) { return (b + 127) / 128 * 128; }

// layout of one stage: Q directions x R rows x nxp values; R x nxp class
// bytes; at a 16-byte boundary the face values, [2][Q][R] values (the
// node's own opposite population at x = 0 and x = nx - 1, for boxes closed
// in x)
__host__ __device__ inline size_t stg_cls_off(int Q, int R, int nxp, int elem) { return (size_t)Q * R * nxp * elem; }
__host__ __device__ inline size_t stg_face_off(int Q, int R, int nxp, int elem)
{
    return (stg_cls_off(Q, R, nxp, elem) + (size_t)R * nxp + 15) / 16 * 16;
}
__host__ __device__ inline size_t stg_stage_bytes(int Q, int R, int nxp, int elem)
{
    return stg_round128(stg_face_off(Q, R, nxp, elem) + (size_t)2 * Q * R * elem);
}

// producer warp: stage the source rows of tile t (plane z, rows y0 .. y0+nr-1).
// Lane 0 arms the full barrier with the tile's copy bytes (its arrival); lane
// a < Q copies direction a's rows and lane Q the class bytes, so the copies
// of a tile are issued in parallel.  A source row outside a closed y or z
// face is replaced by the node's own row of the opposite direction (the
// bounced population, k_step's rule).
template <int Q, class S, bool FACES>
__device__ __forceinline__ void stg_issue(const typename S::T* __restrict__ src, const uint8_t* __restrict__ cls,
                                          const Geo& g, int R, int nty, int t, unsigned char* stage, uint64_t* bar,
                                          int lane, int ey, int ez, int oa)
{
    using T = typename S::T;
    const int z = t / nty, y0 = (t - z * nty) * R;
    const int nr = min(R, g.ny - y0);
    const uint32_t rowb = (uint32_t)g.nxp * (uint32_t)sizeof(T);
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)Q * nr * rowb + (uint32_t)nr * g.nxp);
    __syncwarp();
    if (lane < Q) {
        T* d = reinterpret_cast<T*>(stage) + (size_t)lane * R * g.nxp;
        // the node's own rows of the opposite direction (closed faces)
        const T* so = src + (long long)oa * g.sq + (long long)z * g.ny * g.nxp;
        const int zr = z - ez;
        if (FACES && !g.periodic[2] && (zr < 0 || zr >= g.nz)) {
            bulk_g2s(d, so + (long long)y0 * g.nxp, (uint32_t)nr * rowb, bar);
        } else {
            const T* s = src + (long long)lane * g.sq + (long long)wrapi(zr, g.nz) * g.ny * g.nxp;
            const int ys0 = y0 - ey;
            const bool cy = FACES && !g.periodic[1];
            if (ys0 < 0) {                       // row -1: row ny-1, or out of a closed face
                bulk_g2s(d, cy ? so + (long long)y0 * g.nxp : s + (long long)(g.ny - 1) * g.nxp, rowb, bar);
                if (nr > 1) bulk_g2s(d + g.nxp, s, (uint32_t)(nr - 1) * rowb, bar);
            } else if (ys0 + nr > g.ny) {        // row ny: row 0, or out of a closed face
                const int n1 = g.ny - ys0;
                if (n1 > 0) bulk_g2s(d, s + (long long)ys0 * g.nxp, (uint32_t)n1 * rowb, bar);
                bulk_g2s(d + (size_t)n1 * g.nxp, cy ? so + (long long)(y0 + n1) * g.nxp : s,
                         (uint32_t)(nr - n1) * rowb, bar);
            } else {
                bulk_g2s(d, s + (long long)ys0 * g.nxp, (uint32_t)nr * rowb, bar);
            }
        }
    } else if (lane == Q) {
        bulk_g2s(stage + stg_cls_off(Q, R, g.nxp, sizeof(T)), cls + ((long long)z * g.ny + y0) * g.nxp,
                 (uint32_t)nr * g.nxp, bar);
    }
}

// face warp (boxes closed in x): the face values of tile t, the node's own
// opposite populations at x = 0 for the directions that enter there (E_x = 1)
// and at x = nx - 1 (E_x = -1), by plain loads issued together.  In the
// producer warp their round trip stood before every further copy (binary16
// cavity, stochastic rounding, 256^3: 511 -> 335 us).
template <int Q, class S>
__device__ __forceinline__ void stg_faces(const typename S::T* __restrict__ src, const Geo& g, int R, int nty, int t,
                                          unsigned char* stage, int lane)
{
    using T = typename S::T;
    constexpr int NF = Q == 9 ? 6 : 10;           // entering directions of both faces
    const int z = t / nty, y0 = (t - z * nty) * R;
    const int nr = min(R, g.ny - y0);
    T* fa = reinterpret_cast<T*>(stage + stg_face_off(Q, R, g.nxp, sizeof(T)));
    const T* rows = src + ((long long)z * g.ny + y0) * g.nxp;
    for (int i0 = 0; i0 < NF * nr; i0 += 64) {
        T v[2];
        int at[2] = {-1, -1};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = i0 + 32 * k + lane;
            if (i < NF * nr) {
                const int f = i / nr, r = i - f * nr;
                int a = 0, oa = 0, side = 0, n = 0;
#pragma unroll
                for (int b = 1; b < Q; ++b)
                    if (EX<Q>(b) != 0) {
                        if (n == f) {
                            a = b;
                            oa = OPP<Q>(b);
                            side = EX<Q>(b) < 0;
                        }
                        ++n;
                    }
                v[k] = rows[(long long)oa * g.sq + (long long)r * g.nxp + (side ? g.nx - 1 : 0)];
                at[k] = (side * Q + a) * R + r;
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (at[k] >= 0) fa[at[k]] = v[k];
    }
}

// the pair (x0, x0+1) of a direction from a staged row: the pull sources
// x0 - ex and x0 + 1 - ex.  `e` is the element beside the pair, x0 - 1
// (ex = 1) or x0 + 2 (ex = -1), wrapped at the row ends of a periodic x axis,
// or at a closed x face the node's own opposite population; `own` says that
// the row holds the node's own opposite populations instead (a source row
// outside a closed y or z face), which are not shifted.
template <class S, int EX>
__device__ __forceinline__ float2 stg_pair(const typename S::T* __restrict__ row, int x0,
                                           const typename S::T* __restrict__ e, bool own)
{
    using T = typename S::T;
    if constexpr (sizeof(T) == 2) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(row + x0);
        if (EX == 0) return S::unpack2(w);
        const uint32_t b = *reinterpret_cast<const unsigned short*>(e);
        // bytes 0-3 of the permute are the element's, 4-7 the word's
        return S::unpack2(EX == 1 ? __byte_perm(b, w, own ? 0x7654 : 0x5410) : __byte_perm(b, w, own ? 0x7654 : 0x1076));
    } else {
        const float2 v = *reinterpret_cast<const float2*>(row + x0);
        if (EX == 0) return v;
        const float b = *e;
        if (EX == 1) return make_float2(own ? v.x : b, own ? v.y : v.x);
        return make_float2(own ? v.x : v.y, own ? v.y : b);
    }
}

// all directions' pairs; row0: the row of direction 0, pitch: elements between
// directions; el, er and their pitches: the elements beside the pair, one
// load each (loading the row's and both face values and selecting spent 38
// shared loads a pair in closed boxes; with the division of the task index
// gone too, sphere 256 x 128 x 128 58.3 -> 56.2 us, cavity 256^3 519 -> 511)
template <int Q, class S, bool FACES, int A = 0>
__device__ __forceinline__ void stg_load_pairs(F2 (&dd)[Q], const typename S::T* __restrict__ row0, int pitch, int x0,
                                               const typename S::T* __restrict__ el, int pl,
                                               const typename S::T* __restrict__ er, int pr, const FaceInfo& fi)
{
    if constexpr (A < Q) {
        int wall = 0;
        const bool own = FACES && row_out<Q>(fi, A, wall);
        dd[A] = F2{stg_pair<S, EX<Q>(A)>(row0 + A * pitch, x0, EX<Q>(A) == 1 ? el + A * pl : er + A * pr, own)};
        stg_load_pairs<Q, S, FACES, A + 1>(dd, row0, pitch, x0, el, pl, er, pr, fi);
    }
}

// the wall force fused into the staged step: the momentum exchange of Eq.
// (25) of the step that produced the stored state, summed over the links of
// one wall (wall < 0: every wall) in FP64; null `out`: not asked for
struct StgForce {
    double* out;          // one row of 3 doubles per boundary warp, or null
    int wall;
    unsigned flags;       // LBM_MOVING_CORR
    double c, rho0, svol; // physical units
    float lw[MAXW + 1][3];  // 6 rho0 u_w / c per wall id (physical units)
    // the last warp to write its row sums the rows (ticket: zero between
    // launches) into result: result = (accumulate ? result : 0) + weight sum
    unsigned* ticket;
    double* result;
    double weight;
    int accumulate;
};

// the canonical post-propagation deviations d_b(x) (storage units) of a node
// of a box periodic on every axis with halfway walls, as gather_node: the
// pull source P_b(x - E_b), or through a link into a solid node the bounced
// P_opp(b)(x) plus Ladd's term of the solid's wall.  Every load is issued
// before any is used (one memory round trip for the boundary warps).  With
// a force asked for, each link (x, a' = opp(b)) into a solid adds
// [e_a' (fbar_a' + fbar_b) (+ u_w (fbar_b - fbar_a'))] / c to acc (the FP64
// pipe takes a warp instruction in ~19 cycles: the common factor c dx^D/dt
// waits for the warp's sum), with
// fbar_a' = f^rel_a'(x, T-1) and fbar_b = f_b(x, T) its bounced population,
// as the link kernel of lbm_wall_force does.
template <int Q, class S>
__device__ __forceinline__ void gather_periodic(const typename S::T* __restrict__ P, const uint8_t* __restrict__ cls,
                                                const Geo& g, const KP<typename S::R>& p, int x, int y, int z,
                                                long long own, typename S::R (&d)[Q], const StgForce& fw,
                                                double (&acc)[3])
{
    using T = typename S::T;
    using R = typename S::R;
    uint8_t cs[Q];
    T pv[Q], bv[Q];
#pragma unroll
    for (int b = 1; b < Q; ++b) {
        const int xs = wrapi(x - EX<Q>(b), g.nx), ys = wrapi(y - EY<Q>(b), g.ny), zs = wrapi(z - EZ<Q>(b), g.nz);
        const long long src = ((long long)zs * g.ny + ys) * g.nxp + xs;
        cs[b] = cls[src];
        pv[b] = P[(long long)b * g.sq + src];
        bv[b] = P[(long long)OPP<Q>(b) * g.sq + own];
    }
    d[0] = S::to_raw(P[own]);
#pragma unroll
    for (int b = 1; b < Q; ++b) {
        if (nc_solid(cs[b])) {
            const int wall = nc_wall(cs[b]);
            d[b] = ladd_on<Q, R>(S::to_raw(bv[b]), p, b, wall);
            if (fw.out && (fw.wall < 0 || fw.wall == wall)) {
                // e_a' (fbar_a' + fbar_b) in lattice units, scaled by the caller
                const float* lw = fw.lw[wall];
                const double w = WD<Q>(b);
                const float Pa = S::to_r(bv[b]);
                const double vo = (double)Pa;           // rounded as ladd_on, in physical units
                const double vi = (double)fmaf((float)w, (float)EX<Q>(b) * lw[0] + (float)EY<Q>(b) * lw[1] +
                                                             (float)EZ<Q>(b) * lw[2], Pa);
                const double s = vo + vi + 2.0 * w * fw.rho0;
                const int e[3] = {-EX<Q>(b), -EY<Q>(b), -EZ<Q>(b)};     // e_a', a' = opp(b)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if (e[k]) acc[k] = e[k] > 0 ? acc[k] + s : acc[k] - s;
                    if (fw.flags & 1u) acc[k] += (double)lw[k] / (6.0 * fw.rho0) * (vi - vo);
                }
            }
        } else {
            d[b] = S::to_raw(pv[b]);
        }
    }
}

// EXT: the node code with the Lorentz force, Maxwell term, LES, linear
// equilibrium or Darcy resistance; FACES: some box axis is closed.  The node
// code of each configuration is k_step's: the FP32x2 pair code without EXT,
// the FP32x2 EXT pair code for FP32 storage with closed faces, else the
// scalar EXT code node by node; LP: the FP32x2 pair code specialised for
// LES (LES-only contexts); INS: insulating walls (the scalar code at the
// device's force coefficient, and the warps' sums of the flow velocity).
template <int Q, class S, bool SR, bool EXT = false, bool FACES = false, bool LP = false, bool INS = false>
__global__ void __launch_bounds__(32 * StgShape<EXT>::MAXW, 1)
k_step_staged(const typename S::T* __restrict__ src, typename S::T* __restrict__ dst,
              const uint8_t* __restrict__ cls, const uint32_t* __restrict__ special, long long nspecial, const Geo g,
              const KP<float> p, uint32_t seed, int R, int ntiles, int nstages, int zero_pad,
              unsigned* __restrict__ errflag, const StgForce fw)
{
    using T = typename S::T;
    using Rt = typename S::R;
    static_assert(sizeof(Rt) == 4, "the staged step computes in FP32");
    constexpr bool PAIRX = EXT && !LP && !INS && FACES && sizeof(T) == 4;
    constexpr int G = StgShape<EXT>::G, W = StgShape<EXT>::W, CW = StgShape<EXT>::CW;
    pdl_trigger();
    extern __shared__ __align__(128) unsigned char smem[];
    const size_t stage_bytes = stg_stage_bytes(Q, R, g.nxp, sizeof(T));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)nstages * stage_bytes);
    uint64_t* empty = full + nstages;
    const int nty = (g.ny + R - 1) / R;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (nstages < 2 || nstages % G || nstages > STG_MAX_STAGES) {    // every stage belongs to one group
        pdl_wait();
        if (threadIdx.x == 0) atomicOr(errflag, STG_ERR_CONFIG);
        return;
    }

    const bool face_warp = FACES && !g.periodic[0];
    if (threadIdx.x == 0) {
        for (int s = 0; s < nstages; ++s) {
            mbar_init(&full[s], face_warp ? 2 : 1);      // copies armed, and face values in
            mbar_init(&empty[s], W);
        }
        mbar_fence_init();
    }
    __syncthreads();
    pdl_wait(src);
    // insulating walls: the current force coefficient, and this lane's sum of
    // the flow velocity over its nodes (48 bits: a lane takes dozens)
    Rt aeb[3] = {Rt(0), Rt(0), Rt(0)};
    FF vs[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
    auto add_v = [&](const NodeM<Rt>& m) {
#pragma unroll
        for (int k = 0; k < 3; ++k) vs[k] = ff_add(vs[k], FF{m.v[k], 0.0f});
    };
    // one row per warp of the block, by a fixed shuffle tree
    auto put_v = [&]() {
        const long long row = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double t = (double)vs[k].h + (double)vs[k].l;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) p.ins_rows[row * 3 + k] = t;
        }
    };
    if constexpr (INS) {
#pragma unroll
        for (int k = 0; k < 3; ++k) aeb[k] = p.aeb_dev[k];
    }
    const Rt* const ins = INS ? aeb : nullptr;
    const int my_tiles = ((int)blockIdx.x < ntiles) ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    if (warp == CW) {
        // producer warp: refill a stage once every consumer warp released it
        int ey = 0, ez = 0, oa = 0;          // the pull shift and opposite of this lane's direction
#pragma unroll
        for (int b = 0; b < Q; ++b)
            if (b == lane) {
                ey = EY<Q>(b);
                ez = EZ<Q>(b);
                oa = OPP<Q>(b);
            }
        int k = 0;
        for (; k < my_tiles; ++k) {
            const int s = k % nstages, use = k / nstages;
            if (use > 0) {
                int ok = 0;
                if (lane == 0) ok = mbar_wait_bounded(&empty[s], (uint32_t)(use - 1) & 1u) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    if (lane == 0) atomicOr(errflag, STG_ERR_TIMEOUT);
                    break;
                }
            }
            stg_issue<Q, S, FACES>(src, cls, g, R, nty, (int)blockIdx.x + k * (int)gridDim.x,
                                   smem + (size_t)s * stage_bytes, &full[s], lane, ey, ez, oa);
        }
        if (k < my_tiles && lane == 0) {
            // stopped early: let the copies already issued land before leaving
            for (int j = (k > nstages ? k - nstages : 0); j < k; ++j)
                mbar_wait_bounded(&full[j % nstages], (uint32_t)(j / nstages) & 1u);
        }
        __syncwarp();
        if constexpr (INS) put_v();
        return;
    }

    if (face_warp && warp == CW + 1) {
        // the face warp refills a stage's face values as the producer does its rows
        for (int k = 0; k < my_tiles; ++k) {
            const int s = k % nstages, use = k / nstages;
            if (use > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)(use - 1) & 1u)) {
                if (lane == 0) atomicOr(errflag, STG_ERR_TIMEOUT);
                return;
            }
            stg_faces<Q, S>(src, g, R, nty, (int)blockIdx.x + k * (int)gridDim.x, smem + (size_t)s * stage_bytes, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s]);
        }
        if constexpr (INS) put_v();
        return;
    }

    if (warp > CW) {
        // boundary warps: the listed chunks, node by node (lane per node), and
        // the wall force of their links when asked for (each lane sums its
        // nodes in a fixed order, then a fixed shuffle tree, one row per warp)
        double acc[3] = {0.0, 0.0, 0.0};
        const long long nn = 4 * nspecial;
        const int first = CW + 1 + (face_warp ? 1 : 0);
        const int per = (int)(blockDim.x >> 5) - first;                   // boundary warps of a block
        const int bw = (int)blockIdx.x * per + warp - first, nbw = (int)gridDim.x * per;
        if (zero_pad) {
            // a destination that is not the context's own: zero its padding
            // (the special chunks cover the rest of a row's last chunk), at
            // most 15 chunks of 4 nodes a row, half a warp to a row, four rows
            // in flight (one value a store and a row a lane held up the
            // boundary warps: closed 96 x 64 x 64 bfloat16 29.4 -> 15.2 us,
            // sphere 130 x 96 x 96 112 -> 28)
            const int xp = ((g.nx + 3) & ~3) + 4 * (lane & 15);
            const long long rows = xp < g.nxp ? (long long)Q * g.ny * g.nz : 0;
            using Chunk = typename RawVec<4 * sizeof(T)>::type;
#pragma unroll 4
            for (long long r = (long long)bw * 2 + (lane >> 4); r < rows; r += (long long)nbw * 2)
                *reinterpret_cast<Chunk*>(dst + r * g.nxp + xp) = Chunk{};
        }
        for (long long j = (long long)bw * 32 + lane; j < nn; j += (long long)nbw * 32) {
            const long long node = (long long)special[j >> 2] + (j & 3);
            const int x = (int)(node % g.nxp);
            const long long row = node / g.nxp;
            const int y = (int)(row % g.ny), z = (int)(row / g.ny);
            const uint8_t c = cls[node];
            if (x >= g.nx || nc_solid(c) || c == NC_PAD) {
#pragma unroll
                for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + node] = S::from_raw(Rt(0));
                continue;
            }
            Rt d[Q];
            if constexpr (FACES) pull_walls<Q, S, true>(src, cls, g, p, Around<Q>(g, x, y, z), d);
            else gather_periodic<Q, S>(src, cls, g, p, x, y, z, node, d, fw, acc);
            NodeM<Rt> m;
            node_macro<Rt, Q, EXT, INS>(d, p, m, ins);
            node_relax<Rt, Q, EXT>(d, p, m);
            if constexpr (INS) add_v(m);
            if constexpr (SR) {
                NodeRng rng((uint32_t)node, seed);
#pragma unroll
                for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + node] = S::from_raw_sr(d[a], rng.bits(a));
            } else {
#pragma unroll
                for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + node] = S::from_raw(d[a]);
            }
        }
        if constexpr (INS) {
            __syncwarp();
            put_v();
        }
        if (!FACES && fw.out) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                acc[k] *= fw.svol * fw.c;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
                if (lane == 0) fw.out[(long long)bw * 3 + k] = acc[k];
            }
            // the last boundary warp sums the rows: lane l takes rows
            // l, l+32, ..., then a fixed shuffle tree (the order of the
            // library's fixed-order pass), and clears the ticket
            __threadfence();
            unsigned last = 0;
            if (lane == 0) last = (atomicAdd(fw.ticket, 1u) == (unsigned)nbw - 1u) ? 1u : 0u;
            last = __shfl_sync(0xffffffffu, last, 0);
            if (last) {
                __threadfence();
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    double sum = 0.0;
                    for (int r = lane; r < nbw; r += 32) sum += __ldcg(fw.out + (long long)r * 3 + k);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
                    if (lane == 0) fw.result[k] = (fw.accumulate ? fw.result[k] : 0.0) + fw.weight * sum;
                }
                if (lane == 0) *fw.ticket = 0u;
            }
        }
        return;
    }

    // a consumer warp's tasks: every W-th of its group's, R x tasks_per_row to
    // a tile (row and task of the row, carried over the tiles)
    const int group = warp / W, gw = warp % W;
    const int tasks_per_row = g.nxp / STG_TASK_NODES;
    const int r_step = W / tasks_per_row, xt_step = W % tasks_per_row;
    int r = gw / tasks_per_row, xt = gw % tasks_per_row;
    const long long sq = g.sq;
    const bool closed_x = FACES && !g.periodic[0];
    auto advance = [&]() {
        r += r_step;
        xt += xt_step;
        if (xt >= tasks_per_row) {
            xt -= tasks_per_row;
            ++r;
        }
    };
    int s = group;
    uint32_t phase = 0;
    // plane and tile of the plane, stepped without divisions
    const int t0 = (int)blockIdx.x + group * (int)gridDim.x;
    int z = t0 / nty, ty = t0 - z * nty;
    const int z_step = G * (int)gridDim.x / nty, ty_step = G * (int)gridDim.x - z_step * nty;
    const size_t cls_off = stg_cls_off(Q, R, g.nxp, sizeof(T)), face_off = stg_face_off(Q, R, g.nxp, sizeof(T));
    for (int k = group; k < my_tiles; k += G) {
        if (!mbar_wait_bounded(&full[s], phase)) {
            if (lane == 0) atomicOr(errflag, STG_ERR_TIMEOUT);
            return;
        }
        const int y0 = ty * R;
        const int nr = min(R, g.ny - y0);
        const unsigned char* st = smem + (size_t)s * stage_bytes;
        const T* sp = reinterpret_cast<const T*>(st);
        const uint8_t* sc = st + cls_off;
        const T* fa = reinterpret_cast<const T*>(st + face_off);
        for (; r < R; advance()) {
            if (r >= nr) continue;               // a ragged last tile
            const int x0 = xt * STG_TASK_NODES + 2 * lane;
            const int y = y0 + r;
            const long long base = ((long long)z * g.ny + y) * g.nxp + x0;
            // the pair path serves pairs whose aligned 4-node chunk holds only
            // bulk (and, with closed faces, face) nodes, as in k_step, whose
            // vector chunks are 4 nodes: both kernels run the same code on
            // every node
            const uint32_t cb = *reinterpret_cast<const uint32_t*>(sc + (size_t)r * g.nxp + (x0 & ~3));
            if ((cb & (FACES ? ~0x02020202u : ~0u)) != 0u) continue;   // the boundary warps' (listed on the host)
            FaceInfo fi;
            if constexpr (FACES) {
                fi.closed_x = closed_x;
                fi.yo_lo = !g.periodic[1] && y == 0;
                fi.yo_hi = !g.periodic[1] && y == g.ny - 1;
                fi.zo_lo = (Q == 19) && !g.periodic[2] && z == 0;
                fi.zo_hi = (Q == 19) && !g.periodic[2] && z == g.nz - 1;
                fi.wx_lo = g.face_wall[0]; fi.wx_hi = g.face_wall[1];
                fi.wy_lo = g.face_wall[2]; fi.wy_hi = g.face_wall[3];
                fi.wz_lo = g.face_wall[4]; fi.wz_hi = g.face_wall[5];
            }
            // the element beside the pair on either side: in the row, wrapped
            // at a periodic row end, or (closed x) among the face values, which
            // then replace the row's base and pitch for this lane
            const bool le = x0 == 0, re = x0 + 2 >= g.nx;
            const bool lf = closed_x && le, rf = closed_x && re;
            const T* el = lf ? fa + r : sp + (size_t)r * g.nxp + (le ? g.nx - 1 : x0 - 1);
            const T* er = rf ? fa + Q * R + r : sp + (size_t)r * g.nxp + (re ? x0 + 2 - g.nx : x0 + 2);
            const int pl = lf ? R : R * g.nxp, pr = rf ? R : R * g.nxp;
            const T* row0 = sp + (size_t)r * g.nxp;
            F2 dd[Q];
            // (a fold over the directions: the shift is a template argument)
            stg_load_pairs<Q, S, FACES>(dd, row0, R * g.nxp, x0, el, pl, er, pr, fi);
            if (FACES && p.face_ladd && (cb & 0x02020202u)) {
                // Ladd terms of moving face walls (k_step's add_ladd2)
#pragma unroll
                for (int a = 1; a < Q; ++a) {
                    int wall = 0;
                    const bool hit = row_out<Q>(fi, a, wall);
                    int w0 = wall, w1 = wall;
                    bool h0 = hit, h1 = hit;
                    if (fi.closed_x) {
                        if (EX<Q>(a) == 1 && x0 == 0) { h0 = true; w0 = fi.wx_lo; }
                        if (EX<Q>(a) == -1 && x0 == g.nx - 1) { h0 = true; w0 = fi.wx_hi; }
                        if (EX<Q>(a) == -1 && x0 + 1 == g.nx - 1) { h1 = true; w1 = fi.wx_hi; }
                    }
                    if (h0) dd[a].v.x = ladd_on<Q, float>(dd[a].v.x, p, a, w0);
                    if (h1) dd[a].v.y = ladd_on<Q, float>(dd[a].v.y, p, a, w1);
                }
            }
            if constexpr (!EXT || LP || PAIRX) {
                if constexpr (PAIRX) pair_collide_ext<Q>(dd, p);
                else pair_collide<Q, LP, sizeof(T) == 2>(dd, p);
            } else {
                // the scalar EXT node code, node by node
                Rt d0[Q], d1[Q];
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    d0[a] = dd[a].v.x;
                    d1[a] = dd[a].v.y;
                }
                {
                    NodeM<Rt> m;
                    node_macro<Rt, Q, true, INS>(d0, p, m, ins);
                    node_relax<Rt, Q, true>(d0, p, m);
                    if constexpr (INS) add_v(m);
                }
                {
                    NodeM<Rt> m;
                    node_macro<Rt, Q, true, INS>(d1, p, m, ins);
                    node_relax<Rt, Q, true>(d1, p, m);
                    if constexpr (INS) add_v(m);
                }
#pragma unroll
                for (int a = 0; a < Q; ++a) dd[a].v = make_float2(d0[a], d1[a]);
            }
            if constexpr (sizeof(T) == 2) {
                if constexpr (SR) {
                    NodeRng rp((uint32_t)base, seed);
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        *reinterpret_cast<uint32_t*>(dst + (long long)a * sq + base) =
                            S::pack2_sr(dd[a].v.x, dd[a].v.y, rp.word());
                } else {
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        *reinterpret_cast<uint32_t*>(dst + (long long)a * sq + base) = S::pack2(dd[a].v.x, dd[a].v.y);
                }
            } else {
#pragma unroll
                for (int a = 0; a < Q; ++a) *reinterpret_cast<float2*>(dst + (long long)a * sq + base) = dd[a].v;
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);     // this warp is done with stage s
        r -= R;
        z += z_step;
        ty += ty_step;
        if (ty >= nty) {
            ty -= nty;
            ++z;
        }
        s += G;
        if (s >= nstages) {
            s = group;
            phase ^= 1u;
        }
    }
    if constexpr (INS) put_v();
}

}  // namespace lbm
