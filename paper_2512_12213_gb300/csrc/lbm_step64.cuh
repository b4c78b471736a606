// lbm_step64.cuh -- the fused collide-stream step (Eq. 2 with Eqs. 1 and 3,
// and Eq. 10 with the Maxwell term) for FP64 storage.
//
// The FP64 pipe bounds it: it takes 1.7 lanes per cycle and SM (measured), so
// a warp's FP64 instruction holds it ~19 cycles and a D3Q19 node update of
// 218 of them took 0.42 ns of the whole chip against 0.046 ns for its 305
// bytes.  Two things follow.
//   * The node code counts operations.  With J = rho u^eq and rho u^F = J (or
//     J plus a multiple of rho A), the even part of an opposite pair is
//     w (om drho + 9/2 E.S.E - 3/2 tr S) with one symmetric tensor
//     S_ij = (J_i G_j + J_j G_i)/2 [+ rho K_ij], G = om J / rho + 2 C A, that
//     holds the quadratic equilibrium and the quadratic force term of every
//     model at once, and the odd part 3 w E.(om j + rho A): 137 operations a
//     D3Q19 node.  1/rho is Halley's iteration on the FP32 reciprocal (three
//     operations), range changes are integer work.
//   * One node per thread, in blocks of one warp while the box has few of
//     them: the work then spreads evenly over the SMs' FP64 pipes (64 x 32
//     nodes in two-node threads and blocks of 128 sat on 8 of 152 SMs).
// Step before -> now: D2Q9 64 x 32 12.4 -> 3.9 us, 256 x 128 with the Lorentz
// force 18.5 -> 8.9 us; D3Q19 128^3 890 -> 537 us.
#pragma once

namespace lbm {

// Eq. (2) for the FP64 deviations d of a node; v returns the flow velocity
// with EXT.  AEB: the Lorentz coefficient (configured, or insulating walls').
template <int Q, bool EXT>
__device__ __forceinline__ void node_update64(double (&d)[Q], const KP<double>& p, const double* AEB, double (&v)[3])
{
    constexpr int D = LatDim<Q>::D, NP = LatDim<Q>::NP;
    constexpr double w0 = WD<Q>(0), w1 = WD<Q>(1), w2 = WD<Q>(Q == 19 ? 7 : 5);
    double drho = d[0], j[3] = {0.0, 0.0, 0.0}, P[6] = {0, 0, 0, 0, 0, 0};
    const bool les = EXT && p.les;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const double sm = d[a] + d[b], df = d[a] - d[b];
        drho += sm;
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (e[c]) j[c] = (e[c] > 0) ? j[c] + df : j[c] - df;
        if (les) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (e[c]) P[c] += sm;
            if (e[0] * e[1]) P[3] = (e[0] * e[1] > 0) ? P[3] + sm : P[3] - sm;
            if (e[0] * e[2]) P[4] = (e[0] * e[2] > 0) ? P[4] + sm : P[4] - sm;
            if (e[1] * e[2]) P[5] = (e[1] * e[2] > 0) ? P[5] + sm : P[5] - sm;
        }
    }
    const double rho = p.rho0 + drho, ir = rcp64(rho);
    double A[3], J[3], om = p.om0, om1 = p.om1j, cA[3], tau = p.tau0, C = p.Cf;
    bool quad = !(EXT && p.stokes);
    if constexpr (!EXT) {
#pragma unroll
        for (int k = 0; k < D; ++k) {
            A[k] = p.AG[k];
            J[k] = fma(rho, p.ueq_c[k], j[k]);
            cA[k] = p.cA[k];
        }
    } else {
        double u[3];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            u[k] = j[k] * ir;
            A[k] = p.AG[k];
        }
        if (p.lorentz || p.darcy_h != 0.0) {
            // the implicit flow velocity, as in macro_from_moments
            double Ag[3], Bw = 0.0;
#pragma unroll
            for (int k = 0; k < D; ++k) {
                Ag[k] = fma(AEB[k], ir, p.AG[k]);
                Bw = fma(p.B[k], fma(0.5, Ag[k], u[k]), Bw);
            }
            const double kk = 0.5 * p.kappa * ir;
            const double hk = fma(kk, p.B2, p.darcy_h), den2 = 2.0 * rcp64(1.0 + hk);
            double s = kk * Bw;
            if (p.darcy_h != 0.0 || p.B2 != p.Bp2) s *= rcp64(fma(kk, p.B2 - p.Bp2, 1.0 + p.darcy_h));
#pragma unroll
            for (int k = 0; k < D; ++k) A[k] = den2 * fma(-hk, u[k], fma(s, p.B[k], 0.5 * Ag[k]));
        }
        const bool ve = p.model == MODEL_E;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            v[k] = fma(0.5, A[k], u[k]);
            J[k] = ve ? rho * v[k] : j[k];
        }
        if (les) {
            double PP = 0.0;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const int a = (c < 3) ? c : (c == 5 ? 1 : 0);
                const int b = (c < 3) ? c : (c == 3 ? 1 : 2);
                if (D == 2 && (a == 2 || b == 2)) continue;
                double Pc = P[c];
                if (quad) Pc = fma(-J[a] * ir, J[b], Pc);
                if (p.maxwell) Pc -= p.Lh[c];
                if (a == b) Pc = fma(drho, -1.0 / 3.0, Pc);
                PP = fma((a == b ? 1.0 : 2.0) * Pc, Pc, PP);
            }
            tau = 0.5 * (p.tau0 + sqrt(fma(p.lesc * ir, sqrt(2.0 * PP), p.tau0 * p.tau0)));
            om = 1.0 / tau;
            om1 = 1.0 - om;
            C = ve ? fma(-0.5, om, 1.0) : 1.0;
        }
        const double c2 = p.model == MODEL_A ? 0.0 : 2.0 * C;
#pragma unroll
        for (int k = 0; k < D; ++k) cA[k] = c2 * A[k];
    }
    // S: diagonal xx yy zz, and twice the off-diagonals xy xz yz
    double G[3], S[6];
    const double o = quad ? om * ir : 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) G[k] = fma(o, J[k], cA[k]);
#pragma unroll
    for (int k = 0; k < D; ++k) S[k] = J[k] * G[k];
#pragma unroll
    for (int c = 3; c < (D == 3 ? 6 : 4); ++c) {
        const int a = c == 5 ? 1 : 0, b = c == 3 ? 1 : 2;
        S[c] = fma(J[a], G[b], J[b] * G[a]);
    }
    if (p.model == MODEL_C || p.model == MODEL_D) {
        // rho u^F exceeds J by rho A/2 ([d]) or rho tau A/2 ([c])
        const double h = rho * (p.model == MODEL_C ? C * tau : C);
#pragma unroll
        for (int k = 0; k < D; ++k) S[k] = fma(h * A[k], A[k], S[k]);
#pragma unroll
        for (int c = 3; c < (D == 3 ? 6 : 4); ++c) {
            const int a = c == 5 ? 1 : 0, b = c == 3 ? 1 : 2;
            S[c] = fma(2.0 * h * A[a], A[b], S[c]);
        }
    }
    double tr = S[0] + S[1];
    if (D == 3) tr += S[2];
    const double base = fma(-1.5, tr, om * drho);
    const double b1 = w1 * base, b2 = w2 * base;
    // odd part 3 w (om j + rho A) per axis and speed class
    double o1[3], o2[3];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const double t = fma(rho, A[k], om * j[k]);
        o1[k] = (3.0 * w1) * t;
        o2[k] = (3.0 * w2) * t;
    }
    const bool mxw = EXT && p.maxwell;
    d[0] = fma(om1, d[0], w0 * base);
    if (mxw) d[0] = fma(om, p.mx[0], d[0]);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int a = PAIR<Q>(k), b = OPP<Q>(a);
        const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
        double even, odd;
        if (SPEED2<Q>(a) == 1) {
            const int c = e[0] ? 0 : (e[1] ? 1 : 2);
            even = fma(4.5 * w1, S[c], b1);
            odd = o1[c];
        } else {
            const int c = e[0] ? 0 : 1, f = e[2] ? 2 : 1, x = (c == 1) ? 5 : (f == 1 ? 3 : 4);
            even = fma(4.5 * w2, S[c] + S[f], b2);
            even = fma(e[c] * e[f] > 0 ? 4.5 * w2 : -4.5 * w2, S[x], even);
            odd = e[c] > 0 ? (e[f] > 0 ? o2[c] + o2[f] : o2[c] - o2[f]) : (e[f] > 0 ? o2[f] - o2[c] : -o2[c] - o2[f]);
        }
        if (mxw) even = fma(om, p.mx[a], even);
        d[a] = fma(om1, d[a], even + odd);
        d[b] = fma(om1, d[b], even - odd);
    }
}

constexpr int STEP64_THREADS = 128;

// one padded node per thread; FULL: curved or insulating walls
template <int Q, bool EXT, bool FULL>
__global__ void __launch_bounds__(STEP64_THREADS, 4)
k_step64(const double* __restrict__ src, double* __restrict__ dst, const uint8_t* __restrict__ cls, const Geo g,
         const KP<double> p, int zero_pad)
{
    const unsigned n = blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = n < (unsigned)g.sq;      // the same for 64 threads: the padded node count is a multiple of 64
    const unsigned r = n / (unsigned)g.nxp;
    const int x = (int)(n - r * (unsigned)g.nxp);
    const int z = (int)(r / (unsigned)g.ny), y = (int)(r - (unsigned)z * (unsigned)g.ny);
    const uint8_t c = active ? cls[n] : (uint8_t)NC_PAD;
    double v[3] = {0.0, 0.0, 0.0};
    pdl_wait(src);
    if (c == NC_PAD || nc_solid(c)) {
        if (active && (c != NC_PAD || zero_pad))
#pragma unroll
            for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = 0.0;
    } else {
        double d[Q];
        pull_node<Q, StoreF64, true, FULL>(src, cls, g, p, c, x, y, z, d);
        double aeb[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) aeb[k] = (FULL && p.aeb_dev) ? p.aeb_dev[k] : p.AEB[k];
        node_update64<Q, EXT>(d, p, aeb, v);
        // not earlier: blocks of the next step that are placed while this one
        // computes crowd some SMs' FP64 pipes (Hartmann 256 x 128: 27 us a
        // step with the trigger at entry, 8.9 here, 11.0 without)
        pdl_trigger();
#pragma unroll
        for (int a = 0; a < Q; ++a) dst[(long long)a * g.sq + n] = d[a];
    }
    if constexpr (EXT && FULL) {
        // insulating walls: the sum of v over 64 nodes, by a fixed shuffle
        // tree and then the two warps, is one row
        if (p.ins_rows) {
            __shared__ double half[STEP64_THREADS / 64][3];
            const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
#pragma unroll
                for (int k = 0; k < 3; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], s);
            if (lane == 0 && (w & 1))
#pragma unroll
                for (int k = 0; k < 3; ++k) half[w >> 1][k] = v[k];
            __syncthreads();
            if (active && lane == 0 && !(w & 1))
#pragma unroll
                for (int k = 0; k < 3; ++k) p.ins_rows[(long long)(n >> 6) * 3 + k] = v[k] + half[w >> 1][k];
        }
    }
}

// blocks of one warp (insulating walls: two) until every SM has the 20 warps
// that its registers hold
template <int Q>
cudaError_t launch_step64(const Ctx& c, const void* src, void* dst, int zero_pad, cudaStream_t st)
{
    const bool full = c.cfg.curved || c.insulating;
    const int threads = c.geo.sq < 640ll * c.sm_count ? (full ? 64 : 32) : STEP64_THREADS;
    const unsigned blocks = (unsigned)((c.geo.sq + threads - 1) / threads);
    auto go = [&](auto ex, auto fu) {
        return launch_pdl(k_step64<Q, ex.value, fu.value>, blocks, threads, 0, st, (const double*)src, (double*)dst,
                          c.cls, c.geo, c.kpd, zero_pad);
    };
    const std::true_type yes{};
    const std::false_type no{};
    if (c.ext) return full ? go(yes, yes) : go(yes, no);
    return full ? go(no, yes) : go(no, no);
}

}  // namespace lbm
