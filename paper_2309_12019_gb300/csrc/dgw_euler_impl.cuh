// Stage kernel of the 1D Euler system (Sec. 5.6), included by the 1D stage translation
// units after the scalar kernel (it shares the tables, the launch scalars and the math
// helpers of dgw_stage_impl.cuh).
//
// State U = (rho, rho v, rho E) with p = (gamma - 1)(rho E - rho v^2 / 2); coefficient k
// of component comp of cell e at row comp (p+1) + k, i.e. U[(comp (p+1) + k) E + e].
// One CTA of TX threads owns TX consecutive cells, one per thread:
//   0. each thread loads its cell (one coalesced row per coefficient) and puts its
//      density coefficients and its six end-point values in shared memory; two threads
//      fetch the cells on either side of the tile's cells (the periodic image, or none
//      beyond a wall or an outflow side)
//   1. the sensor of Sec. 4 applied to the density (Sec. 5.6), the volume term at the
//      p+2 Gauss points, and lambda_e = max (|v| + c) over those points and the ends
//   2. every face of the tile once: the LLF flux with s+ the larger |v| + c of the two
//      states; beyond a wall the ghost state mirrors the momentum, beyond an outflow
//      side it copies the inner state
//   3. face terms, the stabilization of every component with the density's gamma,
//      M^{-1} and the Runge-Kutta combination Uout = cn Un + ck Uk + cl L(Uk)
// The operator constants are folded as in the scalar kernel:
//   L_k = (2/h) minv(k) [acc_k - gamma lambda / p (K_ref c)_k].

template <int P>
struct EulerSmem {
    static constexpr int N1 = P + 1;
    Real rho[N1][TX + 2];     // density coefficients, column lx + 1; halo cells 0 and nt + 1
    Real tr[2][3][TX + 2];    // values at xi = -1 (0) and xi = +1 (1), same columns
    Real hf[3][TX + 1];       // LLF flux of face f, between columns f and f + 1
    Real sp[2][TX + 1];       // |v| + c of the left (0) and right (1) state of face f
    int has[2];               // the halo cell on the left / right exists
};

struct EulerState {
    Real v, pr, inv_rho;
};

__device__ __forceinline__ EulerState euler_prim(const KParams& A, Real rho, Real m, Real en)
{
    EulerState s;
    s.inv_rho = rcp_e(rho);
    s.v = m * s.inv_rho;
    s.pr = A.gm1 * (en - Real(0.5) * m * s.v);
    return s;
}

__device__ __forceinline__ Real euler_speed(const KParams& A, const EulerState& s)
{
    return fabs(s.v) + sqrt_e(A.gam * s.pr * s.inv_rho);
}

// F(U) = (rho v, rho v^2 + p, (rho E + p) v)
__device__ __forceinline__ void euler_flux(const EulerState& s, Real m, Real en, Real F[3])
{
    F[0] = m;
    F[1] = fma(m, s.v, s.pr);
    F[2] = (en + s.pr) * s.v;
}

// Sensor of Sec. 4 (or the comparison sensor of Zhao et al., stab = ZHAO) of a 1D cell
// with coefficients c from its face neighbours cn[0] (left) and cn[1] (right), where
// they exist.  TILE: with the operations of process_tile from the weights on (roots and quotients
// of full precision, the ratio itself against b), so that a scalar cell gets the same bits.
template <int P, bool TILE = false>
__device__ __forceinline__ Real sensor_1d(const KParams& A, const Tab<P>& T, const Real* c, const Real (*cn)[P + 1],
                                          const bool* has)
{
    constexpr int N1 = P + 1;
    const int me = (has[0] ? 1 : 0) + (has[1] ? 1 : 0);
    const Real beta0 = qform<P>(T, c);
    const Real d0 = A.eps_w + beta0;
    Real own = Real(1) - Real(me) * A.w_nbr, nbr = A.w_nbr;     // numerators of the weights
    if (TILE) scale_weights(d0, own, nbr);
    const Real w0 = div_w(own, d0 * d0);
    Real wsum = w0;
    Real wnb[2] = {Real(0), Real(0)};
    Real dacc[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) dacc[k] = Real(0);
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        if (!has[f]) continue;
        // Hermite candidate: the neighbour's polynomial continued into this cell, mean
        // dropped (it does not enter the seminorms)
        Real cl[N1];
        cl[0] = Real(0);
#pragma unroll
        for (int k = 1; k < N1; ++k) {
            Real s = Real(0);
#pragma unroll
            for (int m = k; m < N1; ++m) s = fma(T.T[f][k][m], cn[f][m], s);
            cl[k] = s;
        }
        const Real dl = A.eps_w + qform<P>(T, cl);
        const Real wl = div_w(nbr, dl * dl);
        wsum += wl;
        wnb[f] = wl;
#pragma unroll
        for (int k = 1; k < N1; ++k) dacc[k] = fma(wl, c[k] - cl[k], dacc[k]);
    }
    const Real inv = (TILE && !kF32 && A.stab != STAB_ZHAO) ? Real(1) : div_w(Real(1), wsum);
    if (A.stab == STAB_ZHAO) {
        if (me == 0) return Real(0);
        const Real lin0 = Real(1) - Real(me) * A.w_nbr;
        Real dev = zpow(A, fabs(w0 * inv / lin0 - Real(1)));
#pragma unroll
        for (int f = 0; f < 2; ++f)
            if (has[f]) dev += zpow(A, fabs(wnb[f] * inv / A.w_nbr - Real(1)));
        const Real minlin = lin0 < A.w_nbr ? lin0 : A.w_nbr;
        if (TILE) return dev / (zpow(A, fabs(Real(1) / minlin - Real(1))) + Real(me));
        return dev * rcp_e(zpow(A, fabs(rcp_e(minlin) - Real(1))) + Real(me));
    }
    dacc[0] = Real(0);
    if constexpr (TILE) {
        Real r, g;
        if constexpr (kF32) {
#pragma unroll
            for (int k = 1; k < N1; ++k) dacc[k] *= inv;
            const Real num = sqrt_r(fmax(qform<P>(T, dacc), Real(0)));
            if (num <= A.eps_s) return Real(0);
            if (beta0 <= Real(0)) return Real(1);
            r = num / sqrt_r(beta0);
            g = r < Real(1) ? r : Real(1);
        } else {
            g = sensor_ratio(qform<P>(T, dacc), beta0, wsum, A.eps_s, &r);
        }
        if (!A.q_one) g = pow(g, A.q);
        return less_pos(r, A.b) ? Real(0) : g;
    }
    // U - U* = sum_l w_l (c - c_l); the ratio r = ||U - U*|| / ||U|| is taken through
    // its square: r <= 1 iff qd <= beta0, r < b iff r^2 < b^2, ||U - U*|| <= eps_s iff
    // qd <= eps_s^2
#pragma unroll
    for (int k = 1; k < N1; ++k) dacc[k] *= inv;
    const Real qd = fmax(qform<P>(T, dacc), Real(0));
    if (qd <= A.eps_s * A.eps_s) return Real(0);
    if (beta0 <= Real(0)) return Real(1);
    const Real r2 = qd * rcp_e(beta0);
    Real g = r2 < Real(1) ? sqrt_e(r2) : Real(1);
    if (!A.q_one) g = pow(g, A.q);
    if (r2 < A.b * A.b) g = Real(0);
    return g;
}

// Volume term acc_i = sum_q W_q P_i'(g_q) F(U_h(g_q)) (acc_0 = 0) and lambda_e = max (|v| + c) over
// the points, on the symmetric nodes.  Float with two node pairs (p = 2, 3): the pairs travel as
// the lanes of packed FP32 instructions, which the issue-bound kernel needs fewer of.  With the
// update of (rho, m) in pairs: Sod train of 2^22 cells, p = 2, 91.8 -> 86.8 us a stage (the 403 MB it
// moves would take 60).
template <int P>
__device__ __forceinline__ void euler_volume(const KParams& A, const Tab<P>& T, const Real (&c)[3][P + 1], bool need_lam,
                                             Real (&acc)[3][P + 1], Real& lam)
{
    constexpr int N1 = P + 1, NQ = P + 2;
    if constexpr (kF32 && P >= 2) {
        auto two = [](Real x) { return make_float2((float)x, (float)x); };
        // table entry i of the two positive nodes, outermost first
        auto pairB = [&](int i) { return make_float2((float)T.B[NQ - 1][i], (float)T.B[NQ - 2][i]); };
        float2 up[3], um[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float2 e = __ffma2_rn(pairB(2), two(c[q][2]), two(c[q][0]));
            float2 o = __fmul2_rn(pairB(1), two(c[q][1]));
            if constexpr (P == 3) o = __ffma2_rn(pairB(3), two(c[q][3]), o);
            up[q] = __fadd2_rn(e, o);
            um[q] = vsub(e, o);
        }
        // F_2, F_3 and |v| + c at both lanes of (rho, m, rho E)
        auto point = [&](const float2 (&u)[3], float2 (&F)[3]) {
            const float2 inv = make_float2(rcp_e(u[0].x), rcp_e(u[0].y));
            const float2 v = __fmul2_rn(u[1], inv);
            const float2 pr = __fmul2_rn(two(A.gm1), __ffma2_rn(__fmul2_rn(two(Real(-0.5)), u[1]), v, u[2]));
            F[0] = u[1];
            F[1] = __ffma2_rn(u[1], v, pr);
            F[2] = __fmul2_rn(__fadd2_rn(u[2], pr), v);
            if (need_lam) {
                const float2 s = __fmul2_rn(__fmul2_rn(two(A.gam), pr), inv);
                lam = max_nan(lam, max_nan(fabsf(v.x) + sqrt_e(s.x), fabsf(v.y) + sqrt_e(s.y)));
            }
        };
        float2 Fp[3], Fm[3];
        point(up, Fp);
        point(um, Fm);
        Real Fc[3] = {Real(0), Real(0), Real(0)};
        if constexpr (P == 3) {       // the centre node
            constexpr int qc = NQ / 2;
            Real u[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) u[q] = fma(T.B[qc][2], c[q][2], c[q][0]);
            const EulerState st = euler_prim(A, u[0], u[1], u[2]);
            euler_flux(st, u[1], u[2], Fc);
            if (need_lam) lam = max_nan(lam, euler_speed(A, st));
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float2 S = __fadd2_rn(Fp[q], Fm[q]), D = vsub(Fp[q], Fm[q]);
            acc[q][0] = Real(0);
#pragma unroll
            for (int i = 1; i < N1; ++i) {
                const float2 f = (i & 1) ? S : D;        // P_i' is even for odd i
                Real t = fma(T.WD[NQ - 2][i], f.y, T.WD[NQ - 1][i] * f.x);
                if (P == 3 && (i & 1)) t = fma(T.WD[NQ / 2][i], Fc[q], t);
                acc[q][i] = t;
            }
        }
    } else {
        Real u[3][NQ], F[3][NQ];
#pragma unroll
        for (int q = 0; q < 3; ++q) interp_sym<N1, NQ>(T.B, c[q], u[q]);
#pragma unroll
        for (int g = 0; g < NQ; ++g) {
            const EulerState st = euler_prim(A, u[0][g], u[1][g], u[2][g]);
            Real f[3];
            euler_flux(st, u[1][g], u[2][g], f);
            if (need_lam) lam = max_nan(lam, euler_speed(A, st));
#pragma unroll
            for (int q = 0; q < 3; ++q) F[q][g] = f[q];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            project_sym<true, N1, NQ>(T.WD, F[q], acc[q]);
            acc[q][0] = Real(0);
        }
    }
}

// MODE 0: stage / residual; MODE 1: sensor only (writes gamma_out).
template <int P, int MODE>
__global__ void __launch_bounds__(TX, kF32 ? 8 : 4) euler_kernel(const __grid_constant__ KParams A)
{
    constexpr int N1 = P + 1;
    __shared__ EulerSmem<P> S;
    pdl_begin();
    const Tab<P>& T = tab<P>();
    const int tid = threadIdx.x;
    const int64_t E = A.E;
    const int tx0 = blockIdx.x * TX;
    const int nt = A.nx - tx0 < TX ? A.nx - tx0 : TX;     // cells of this tile
    const int gx = tx0 + tid;
    const bool in = tid < nt;

    // ---- 0. own cell, halo cells ----
    Real c[3][N1];
#pragma unroll
    for (int comp = 0; comp < 3; ++comp)
#pragma unroll
        for (int k = 0; k < N1; ++k) c[comp][k] = Real(0);
    auto put = [&](const Real (&q)[3][N1], int col) {
#pragma unroll
        for (int k = 0; k < N1; ++k) S.rho[k][col] = q[0][k];
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            Real xm = Real(0), xp = Real(0);
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                xp += q[comp][k];
                xm = (k & 1) ? xm - q[comp][k] : xm + q[comp][k];
            }
            S.tr[0][comp][col] = xm;
            S.tr[1][comp][col] = xp;
        }
    };
    // Un is read only by the final combination: its loads are issued here, so that their
    // latency hides behind the sensor, volume and face work
    Real un[3][N1];
    if (in) {
        const Real* src = A.Uk + gx;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
#pragma unroll
            for (int k = 0; k < N1; ++k) c[comp][k] = src[(int64_t)(comp * N1 + k) * E];
        if (MODE == 0 && A.has_un) {
            const Real* usrc = A.Un + gx;
#pragma unroll
            for (int comp = 0; comp < 3; ++comp)
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    const Real* a = usrc + (int64_t)(comp * N1 + k) * E;
                    un[comp][k] = *a;
                }
        }
        put(c, tid + 1);
    }
    if (tid < 2) {
        const int hx = wrap_x(A, tid == 0 ? tx0 - 1 : tx0 + nt);
        S.has[tid] = hx >= 0;
        if (hx >= 0) {
            Real q[3][N1];
            const Real* src = A.Uk + hx;
#pragma unroll
            for (int comp = 0; comp < 3; ++comp)
#pragma unroll
                for (int k = 0; k < N1; ++k) q[comp][k] = src[(int64_t)(comp * N1 + k) * E];
            put(q, tid == 0 ? 0 : nt + 1);
        }
    }
    __syncthreads();

    // ---- 1. sensor of the density ----
    Real gamma = (MODE == 0 && A.stab == STAB_LO) ? Real(1) : Real(0);
    if (in && (MODE == 1 || A.stab >= STAB_WENO)) {
        const bool has[2] = {tid > 0 || S.has[0] != 0, tid < nt - 1 || S.has[1] != 0};
        Real cn[2][N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            cn[0][k] = has[0] ? S.rho[k][tid] : Real(0);
            cn[1][k] = has[1] ? S.rho[k][tid + 2] : Real(0);
        }
        gamma = sensor_1d<P>(A, T, c[0], cn, has);
        if (MODE == 1) A.gamma_out[gx] = (double)gamma;
    }
    if (MODE == 1) return;

    // ---- 1b. volume term: acc_i = sum_q W_q P_i'(g_q) F(U_h(g_q)); lambda_e ----
    Real acc[3][N1];
    Real lam = Real(0);
    const bool need_lam = A.stab != STAB_DG && !A.lam_fixed;
    if (in) euler_volume<P>(A, T, c, need_lam, acc, lam);

    // ---- 2. faces f = 0 .. nt of the tile ----
    for (int f = tid; f <= nt; f += TX) {
        Real uL[3], uR[3];
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            uL[comp] = S.tr[1][comp][f];
            uR[comp] = S.tr[0][comp][f + 1];
        }
        const bool wall_l = f == 0 && !S.has[0];
        const bool wall_r = f == nt && !S.has[1];
        if (wall_l) {
            const bool refl = A.bc[0] == BC_REFLECT;
            uL[0] = uR[0]; uL[1] = refl ? -uR[1] : uR[1]; uL[2] = uR[2];
        } else if (wall_r) {
            const bool refl = A.bc[1] == BC_REFLECT;
            uR[0] = uL[0]; uR[1] = refl ? -uL[1] : uL[1]; uR[2] = uL[2];
        }
        const EulerState sl = euler_prim(A, uL[0], uL[1], uL[2]);
        const EulerState sr = euler_prim(A, uR[0], uR[1], uR[2]);
        Real FL[3], FR[3];
        euler_flux(sl, uL[1], uL[2], FL);
        euler_flux(sr, uR[1], uR[2], FR);
        const Real spl = euler_speed(A, sl), spr = euler_speed(A, sr);
        S.sp[0][f] = spl;
        S.sp[1][f] = spr;
        const Real s = max_nan(spl, spr);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
            S.hf[comp][f] = Real(0.5) * ((FL[comp] + FR[comp]) - s * (uR[comp] - uL[comp]));
    }
    __syncthreads();
    if (!in) return;

    // ---- 3. face terms, stabilization, M^{-1}, Runge-Kutta combination ----
    // lambda_e: also |v| + c at the cell's two ends, its own states at faces tid, tid + 1
    if (need_lam) lam = max_nan(lam, max_nan(S.sp[1][tid], S.sp[0][tid + 1]));
    const Real ngs = A.stab == STAB_DG ? Real(0) : -(gamma * (A.lam_fixed ? A.lambda_nu : lam) * Real(1.0 / P));
    // (rho, m) of a mode as a pair (packed in float), rho E by itself
    using E2 = std::conditional_t<kF32, float2, double2>;
    auto pair = [](Real x, Real y) { E2 v; v.x = x; v.y = y; return v; };
    auto update = [&](auto hm, auto hp, auto acc_k, int k, const auto* cc, auto un_k) {
        // -P_k(+1) H_right + P_k(-1) H_left
        auto r = (k & 1) ? vsub(acc_k, vadd(hm, hp)) : vadd(acc_k, vsub(hm, hp));
        if (k > 0) {
            auto kc = vmul(T.A1[k][k], cc[k]);
#pragma unroll
            for (int m = 1; m < N1; ++m)
                if (m != k && ((k + m) & 1) == 0) kc = vfma(vbc<decltype(kc)>(T.A1[k][m]), cc[m], kc);
            r = vfma(vbc<decltype(r)>(ngs), kc, r);
        }
        auto out = vfma(vbc<decltype(r)>(A.cl), vmul(A.two_h * T.minv[k], r), vmul(A.ck, cc[k]));
        if (A.has_un) out = vfma(vbc<decltype(r)>(A.cn), un_k, out);
        return out;
    };
    E2 c2[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) c2[k] = pair(c[0][k], c[1][k]);
    const E2 hm2 = pair(S.hf[0][tid], S.hf[1][tid]), hp2 = pair(S.hf[0][tid + 1], S.hf[1][tid + 1]);
    const Real hm3 = S.hf[2][tid], hp3 = S.hf[2][tid + 1];
    E2 chk2 = pair(Real(0), Real(0));
    Real chk = Real(0);
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        const E2 o2 = update(hm2, hp2, pair(acc[0][k], acc[1][k]), k, c2, pair(un[0][k], un[1][k]));
        const Real o3 = update(hm3, hp3, acc[2][k], k, c[2], un[2][k]);
        chk2 = vfma(o2, pair(Real(0), Real(0)), chk2);
        chk = fma(o3, Real(0), chk);
        A.Uout[(int64_t)k * E + gx] = o2.x;
        A.Uout[(int64_t)(N1 + k) * E + gx] = o2.y;
        A.Uout[(int64_t)(2 * N1 + k) * E + gx] = o3;
    }
    chk += chk2.x + chk2.y;
    if (chk != chk) atomicOr(A.flag, 1u);
}

template <int P>
static cudaError_t launch_euler_p(const StageArgs& s, int mode, cudaStream_t st)
{
    const KParams a = make_params(s);
    const unsigned grid = (unsigned)((s.nx + TX - 1) / TX);
    if (grid == 0) return cudaSuccess;
    return mode == 0 ? launch_k<euler_kernel<P, 0>>(grid, TX, 0, s.pdl, st, a) : launch_k<euler_kernel<P, 1>>(grid, TX, 0, s.pdl, st, a);
}

static cudaError_t launch_euler(const StageArgs& s, int p, int mode, cudaStream_t st)
{
    switch (p) {
    case 1: return launch_euler_p<1>(s, mode, st);
    case 2: return launch_euler_p<2>(s, mode, st);
    case 3: return launch_euler_p<3>(s, mode, st);
    default: return cudaErrorInvalidValue;
    }
}
