// lbm_adjoint.cuh -- the reverse step of the discrete adjoint of the
// collide-stream step and the momentum-exchange drag (arXiv 2512.12213,
// Eqs. 1-3 and 25), for gradients of time-averaged drag with respect to the
// body force and a wall velocity, and its launcher.  Included by
// lbm_kernels.cuh after the other launchers.
#pragma once

namespace lbm {

// per-launch constants of a reverse step, per direction a of a link into the
// target wall: the drag seed 2 w_J svol c (d . E_a) that the link adds to
// psi_a, and -6 w_a rho0 / c, the derivative of the Ladd term with respect
// to E_a . u_w
template <typename R> struct AdjConst {
    R seed[19];
    R gl[19];
};

// ---------------------------------------------------------------- adjoint
// One reverse step of the drag adjoint (uniform body force, any model).
// psi_a(x) = phi_next_a(x + E_a) through a fluid link, or phi_next_opp(a)(x)
// plus the drag seed through a link into the target wall; then
// phi_b = (1 - om) psi_b + A_rho + E_b . B_j, where A_rho and B_j collect the
// derivatives of G = f^eq/tau + F with respect to rho and j, formed from the
// weighted moments s0 = sum w psi, s1 = sum w psi E, s2 = sum w psi E E, which
// like the state's moments come from the sums and differences of the opposite
// pairs, each speed class weighted once.  One node per thread, psi in
// registers.  Bulk nodes (every link to a fluid node, periodic wrap allowed)
// address their neighbours without branches; nodes next to a wall or a closed
// face load their sources' class bytes together and then the values.  Bound by
// memory: 128^3 FP32 117 us a step before the pairs (940 instructions a node)
// -> 76, of 71 for its bytes.  Gradient terms are summed per thread
// in the compute precision and per block in FP64.
// blocks of RED_THREADS per SM: FP64 1; FP32 compute D3Q19 3 (80 registers;
// 18% faster than 2 blocks at 126 registers on the 128^3 sphere), D2Q9 2 (the
// 512 x 256 cylinder ran 23% slower at 3)
template <int Q, class S>
__global__ void __launch_bounds__(RED_THREADS, sizeof(typename S::R) == 8 ? 1 : (Q == 19 ? 3 : 2))
k_adjoint(const typename S::T* __restrict__ Pprev, const typename S::R* __restrict__ phin,
          typename S::R* __restrict__ phio, const uint8_t* __restrict__ cls, const Geo g,
          const KP<typename S::R> p, int target, const AdjConst<typename S::R> ac, double gscale,
          double* __restrict__ partials)
{
    using R = typename S::R;
    // FP64: not before the sums, as in k_step64 (D2Q9 channel
    // 256 x 128: 28.1 us with the trigger at entry, 17.3 here)
    if constexpr (sizeof(R) == 4) pdl_trigger();
    pdl_wait(Pprev, phin);
    using T = typename S::T;
    constexpr int D = LatDim<Q>::D, NP = LatDim<Q>::NP;
    __shared__ double sm[6 * 32];
    R accg[3] = {0, 0, 0}, accw[3] = {0, 0, 0};
    // node indices fit in 32 bits (the padded node count is below 2^31)
    const unsigned nxp = (unsigned)g.nxp, ny = (unsigned)g.ny;
    for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < (unsigned)g.sq; n += gridDim.x * blockDim.x) {
        const unsigned ur = n / nxp;
        const int x = (int)(n - ur * nxp);
        const int z = (int)(ur / ny), y = (int)(ur - (unsigned)z * ny);
        const uint8_t cl = cls[n];
        if (nc_solid(cl) || cl == NC_PAD) {
#pragma unroll
            for (int a = 0; a < Q; ++a) phio[(long long)a * g.sq + n] = R(0);
            continue;
        }
        R psi[Q], d[Q];
        const Around<Q> ar(g, x, y, z);          // x + E_a is the source of opp(a)
        if (cl == NC_BULK) {
            T v[Q];
#pragma unroll
            for (int a = 0; a < Q; ++a) v[a] = Pprev[(long long)a * g.sq + ar.at(a)];
#pragma unroll
            for (int a = 0; a < Q; ++a) psi[a] = phin ? phin[(long long)a * g.sq + ar.at(OPP<Q>(a))] : R(0);
#pragma unroll
            for (int a = 0; a < Q; ++a) d[a] = S::to_r(v[a]);
        } else {
            uint8_t cs[Q];
#pragma unroll
            for (int b = 1; b < Q; ++b) cs[b] = ar.out(b) ? nc_make_solid(ar.face(g, b)) : cls[ar.at(b)];
            d[0] = S::to_r(Pprev[n]);
            psi[0] = phin ? phin[n] : R(0);
#pragma unroll
            for (int b = 1; b < Q; ++b) {
                const int a = OPP<Q>(b);
                const bool hit = nc_solid(cs[b]);
                d[b] = S::to_r(Pprev[hit ? (long long)a * g.sq + n : (long long)b * g.sq + ar.at(b)]);
                psi[a] = phin ? phin[hit ? (long long)b * g.sq + n : (long long)a * g.sq + ar.at(b)] : R(0);
            }
#pragma unroll
            for (int b = 1; b < Q; ++b) {
                const int a = OPP<Q>(b);
                if (!nc_solid(cs[b])) continue;
                const int wall = nc_wall(cs[b]);
                d[b] = ladd_on<Q, R>(d[b], p, b, wall);
                if (wall == target) {
                    // u_w enters f(t+1) and F_t through the Ladd term
                    const R gl = ac.gl[a] * (psi[a] + R(0.5) * ac.seed[a]);
                    psi[a] += ac.seed[a];
                    accw[0] += gl * R(EX<Q>(a));
                    accw[1] += gl * R(EY<Q>(a));
                    accw[2] += gl * R(EZ<Q>(a));
                }
            }
        }
        NodeM<R> m;
        {
            Mom<R> mo;
            mom_zero(mo);
            mo.drho = d[0];
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int a = PAIR<Q>(k), b = OPP<Q>(a);
                const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
                const R df = d[a] - d[b];
                mo.drho += d[a] + d[b];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    if (e[c]) mo.j[c] = e[c] > 0 ? mo.j[c] + df : mo.j[c] - df;
            }
            macro_from_moments<R, Q, false>(mo, p, m);
        }
        // weighted moments of psi: per speed class, then w_axis and w_diag
        R s0, s1[3], s2[3][3];
        {
            constexpr R wa = R(WD<Q>(1)), wd = R(WD<Q>(Q == 9 ? 5 : 7));
            R ax = R(0), dg = R(0), j2[3] = {R(0), R(0), R(0)}, p2[3] = {R(0), R(0), R(0)}, x2[3] = {R(0), R(0), R(0)};
            R j1[3] = {R(0), R(0), R(0)}, p1[3] = {R(0), R(0), R(0)};
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int a = PAIR<Q>(k), b = OPP<Q>(a);
                const int e[3] = {EX<Q>(a), EY<Q>(a), EZ<Q>(a)};
                const R sp = psi[a] + psi[b], df = psi[a] - psi[b];
                if (SPEED2<Q>(a) == 1) {
                    const int c = e[0] ? 0 : (e[1] ? 1 : 2);
                    ax += sp;
                    p1[c] = sp;
                    j1[c] = e[c] > 0 ? df : -df;
                } else {
                    const int i = e[0] ? 0 : 1, j = e[2] ? 2 : 1, q = i == 1 ? 2 : (j == 2 ? 1 : 0);   // xy xz yz
                    dg += sp;
                    p2[i] += sp;
                    p2[j] += sp;
                    x2[q] = e[i] * e[j] > 0 ? x2[q] + sp : x2[q] - sp;
                    j2[i] = e[i] > 0 ? j2[i] + df : j2[i] - df;
                    j2[j] = e[j] > 0 ? j2[j] + df : j2[j] - df;
                }
            }
            s0 = R(WD<Q>(0)) * psi[0] + wa * ax + wd * dg;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                s1[c] = wa * j1[c] + wd * j2[c];
                s2[c][c] = wa * p1[c] + wd * p2[c];
            }
            s2[0][1] = s2[1][0] = wd * x2[0];
            s2[0][2] = s2[2][0] = wd * x2[1];
            s2[1][2] = s2[2][1] = wd * x2[2];
        }
        // sum psi f^eq(rho, W) = rho Psi_e(W); grad_W = rho (3 s1 + 9 s2 W - 3 s0 W)
        // sum psi F = C rho Psi_f; grad_Wf = C rho (9 s2 A - 3 s0 A); grad_A = C rho (3 s1 - 3 s0 Wf + 9 s2 Wf)
        const R* W = m.weq;
        const R* Wf = m.wf;
        const R* A = m.A;
        R s2W[3] = {0, 0, 0}, s2A[3] = {0, 0, 0}, s2F[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                s2W[i] += s2[i][j] * W[j];
                s2A[i] += s2[i][j] * A[j];
                s2F[i] += s2[i][j] * Wf[j];
            }
        R WW = 0, s1W = 0, WsW = 0, s1A = 0, FA = 0, FsA = 0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            WW += W[i] * W[i];
            s1W += s1[i] * W[i];
            WsW += W[i] * s2W[i];
            s1A += s1[i] * A[i];
            FA += Wf[i] * A[i];
            FsA += Wf[i] * s2A[i];
        }
        const bool ma = (p.model == MODEL_A);
        const R Psi_e = s0 + R(3) * s1W + R(4.5) * WsW - R(1.5) * WW * s0;
        const R Psi_f = ma ? R(3) * s1A : (R(3) * s1A - R(3) * FA * s0 + R(9) * FsA);
        R Ge[3], Gf[3], GA[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Ge[i] = (i < D) ? m.om * m.rho * (R(3) * s1[i] + R(9) * s2W[i] - R(3) * s0 * W[i]) : R(0);
            Gf[i] = (i < D && !ma) ? m.C * m.rho * (R(9) * s2A[i] - R(3) * s0 * A[i]) : R(0);
            GA[i] = (i < D) ? (ma ? m.C * m.rho * R(3) * s1[i]
                                  : m.C * m.rho * (R(3) * s1[i] - R(3) * s0 * Wf[i] + R(9) * s2F[i]))
                            : R(0);
        }
        // W and Wf move with u = j/rho: d/dj = I/rho, d/drho = -u/rho
        const R ir = R(1) / m.rho;
        R Arho = m.om * Psi_e + m.C * Psi_f;
        R Bj[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Arho -= (Ge[i] + Gf[i]) * m.u[i] * ir;
            Bj[i] = (Ge[i] + Gf[i]) * ir;
        }
        const R om1 = R(1) - m.om;
        phio[n] = fma(om1, psi[0], Arho);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int a = PAIR<Q>(k), b = OPP<Q>(a);
            R t = R(0);
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const int e = c == 0 ? EX<Q>(a) : (c == 1 ? EY<Q>(a) : EZ<Q>(a));
                if (e) t = e > 0 ? t + Bj[c] : t - Bj[c];
            }
            phio[(long long)a * g.sq + n] = fma(om1, psi[a], Arho + t);
            phio[(long long)b * g.sq + n] = fma(om1, psi[b], Arho - t);
        }
        // dJ/dg: A = dt g / c; W^eq moves with A/2 for [e]; W^F with tau/2 ([c]) or 1/2 ([d], [e])
        const R keq = (p.model == MODEL_E) ? R(0.5) : R(0);
        const R kf = (p.model == MODEL_C) ? R(0.5) * m.tau : ((p.model == MODEL_D || p.model == MODEL_E) ? R(0.5) : R(0));
#pragma unroll
        for (int i = 0; i < D; ++i) accg[i] += GA[i] + keq * Ge[i] + kf * Gf[i];
    }
    if constexpr (sizeof(R) == 8) pdl_trigger();
    double acc[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        acc[k] = gscale * (double)accg[k];
        acc[3 + k] = (double)accw[k];
    }
    block_sum<6>(acc, sm);
    if (threadIdx.x == 0)
        for (int k = 0; k < 6; ++k) partials[(long long)blockIdx.x * 6 + k] += acc[k];
}

// ---------------------------------------------------------------- launcher
template <int Q, class S>
cudaError_t launch_adjoint(const Ctx& c, const void* Pprev, const void* phin, void* phio, int wall,
                           const double* dir, double seedw, double* partials, cudaStream_t st)
{
    using T = typename S::T;
    using R = typename S::R;
    // a fixed grid per context, so every block owns the same partial row each
    // step: the blocks resident at once (SMs x occupancy), each walking the
    // nodes with the grid stride, so no partly filled last wave
    const long long NP = (long long)c.geo.nxp * c.geo.ny * c.geo.nz;
    if (c.adj_blocks == 0) {
        int occ = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_adjoint<Q, S>, RED_THREADS, 0);
        if (e != cudaSuccess) return e;
        c.adj_blocks = (int)std::min<long long>(grid_for(NP, RED_THREADS, ADJ_BLOCKS),
                                                 (long long)std::max(occ, 1) * c.sm_count);
    }
    const int blocks = std::min(c.adj_blocks, ADJ_BLOCKS);
    const KP<R>& p = kp_of<S>(c);
    const KP<double>& pd = c.kpd;
    AdjConst<R> ac;
    for (int a = 0; a < 19; ++a) {
        ac.seed[a] = R(0);
        ac.gl[a] = R(0);
    }
    for (int a = 0; a < Q; ++a) {
        const double de = pd.c * (dir[0] * EX<Q>(a) + dir[1] * EY<Q>(a) + dir[2] * EZ<Q>(a));
        ac.seed[a] = R(seedw * 2.0 * pd.svol * de);
        ac.gl[a] = R(-6.0 * WD<Q>(a) * pd.rho0 / pd.c);
    }
    return launch_pdl(k_adjoint<Q, S>, blocks, RED_THREADS, 0, st, (const T*)Pprev, (const R*)phin, (R*)phio, c.cls,
                      c.geo, p, wall, ac, pd.dt / pd.c, partials);
}

}  // namespace lbm
