// All steps of a small 1D mesh in one launch (included by the 1D stage translation units after
// the Euler kernel).
//
// A 1D mesh of the paper's sizes (16 to 2048 cells) fits in the registers of a few CTAs, and a
// stage of it is a chain of dependent operations: launched stage by stage it costs a launch, a
// round trip to memory and, in double, the arithmetic of 128 cells on one SM whose FP64 pipe has
// two lanes.  Here one thread-block cluster holds the mesh, one cell per thread, for all nsteps
// steps: the state and the step's start state stay in registers, and a stage exchanges only what
// neighbours read, through (distributed) shared memory and one cluster barrier.  The exchange is
// double-buffered, so the barrier of the next stage is also the one that frees a buffer; the
// volume term, which needs no neighbour, runs between the barrier's arrive and wait.
//
// CTAs are as small as the cluster limit lets them be, which spreads the FP64 work over the most
// SMs.  The scheme is that of process_tile and euler_kernel; a scalar cell on one lane also takes
// their operations in their order, the sensor's included, and so their bits.  (Euler cells and cells
// on eight lanes agree with the stage kernels to rounding.)  Each face is evaluated by both of its
// cells from the same values in the same way.
//
// Double, up to kWideMax cells: eight lanes per cell.  A warp's FP64 instruction occupies its
// scheduler's share of the FP64 pipe for 64 cycles however many lanes are active and however many
// are independent (measured; 76 with all four schedulers of an SM busy), so a stage costs its
// number of FP64 instructions times 64 cycles: about 190 (scalar, p = 2) or 480 (Euler) with one
// cell per lane.  With eight lanes each point, each face, each candidate of the sensor and each
// mode has a lane of its own, and the same instructions serve all of them: about 60 and 95.
//
// Measured (p = 2, us per stage; stage by stage / one lane per cell / eight):
//   FP64 advection,  128 cells: 11.6 / 5.9 / 2.7;   512: 12 / 6.0 / 4.9;   2048: 12 / 7.0 / -
//   FP64 Sod,        128 cells: 22.5 / 14.8 / 4.1;  512: 23 / 14.8 / 7.4;  2048: 23 / 16.5 / -
//   FP32 advection, 4096 cells:  6.1 / 1.0 / -
// so eight lanes serve up to 512 cells in double, one lane up to the largest cluster.  In float
// an instruction's latency is what counts, and one lane per cell has it lowest.

constexpr int kLineCluster = 16;                           // CTAs of a cluster (beyond 8: opt-in)
constexpr int kLineThreads = kF32 ? 256 : 128;             // largest CTA, one cell per thread
constexpr int kWideCells = 32;                             // largest CTA's cells, eight lanes per cell
constexpr int kWideMax = kF32 ? 0 : kLineCluster * kWideCells;

// Runge-Kutta coefficients of one launch.  order 2, 3: `stages` combinations
// cn Un + ck U + cl L(U); order 4 (ten stages): combination 0 nine times, with the register
// recombination after the fifth, then combination 1.
struct LineSteps {
    const Real* Uin;
    const Real* Un;                        // start state of the step, if not Uin (a single later stage; else null)
    Real* U;                               // the result (may be Uin or Un)
    int nsteps, order, stages, cells;      // cells: per CTA (all but the last are full)
    Real cn[3], ck[3], cl[3];
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Stores v to the word at `p` of this CTA's shared memory in the CTA of rank `rank`.
__device__ __forceinline__ void st_cluster(const Real* p, uint32_t rank, Real v)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
    if constexpr (kF32) asm volatile("st.shared::cluster.f32 [%0], %1;" :: "r"(d), "f"((float)v) : "memory");
    else asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(d), "d"((double)v) : "memory");
}

// Place of a thread's cell on the line and in the exchange buffers (columns 1 .. cells; halo
// columns 0 and, right of the CTA's last cell, its number of cells + 1).
struct LinePlace {
    int gx, col;
    bool in, has_l, has_r;
    bool edge_l, edge_r;           // the cell's values also go to a neighbouring CTA's halo column
    uint32_t rank_l, rank_r;
    int col_l, col_r;
    // tid: the cell's number in the CTA
    __device__ __forceinline__ LinePlace(const KParams& A, const LineSteps& L, int tid)
    {
        const int rank = (int)cluster_rank();
        const int last = (A.nx - 1) / L.cells;
        const int tx0 = rank * L.cells;
        const int nt = A.nx - tx0 < L.cells ? A.nx - tx0 : L.cells;
        gx = tx0 + tid;
        col = tid + 1;
        in = tid < nt;
        const bool per = A.bc[0] == BC_PERIODIC;
        has_l = in && (gx > 0 || per);
        has_r = in && (gx < A.nx - 1 || per);
        edge_l = tid == 0 && has_l;
        edge_r = tid == nt - 1 && has_r;
        // the first cell is the right halo of the CTA before, the last one the left halo of the next
        rank_l = rank > 0 ? rank - 1 : last;
        col_l = (rank > 0 ? L.cells : A.nx - last * L.cells) + 1;
        rank_r = rank < last ? rank + 1 : 0;
        col_r = 0;
    }
};

// The volume term of a scalar cell: acc_i = sum_q w_q P_i'(g_q) F(u_q) (acc_0 = 0), and the
// largest speed key of the points.
template <int P, int FLUX>
__device__ __forceinline__ void line_volume(const KParams& A, const Tab<P>& T, const Real (&c)[P + 1], const Real xc,
                                            Real (&acc)[P + 1], Real& key)
{
    constexpr int N1 = P + 1, NQ = P + 2;
    Real u[NQ], fx[NQ];
    interp_sym<N1, NQ>(T.B, c, u);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        Real fy, k;
        vol_flux_v<FLUX>(A, u[q], fma_x(A.hh, T.g[q], xc), Real(0), fx[q], fy, k);
        key = fmax(key, k);
    }
    project_sym<true, N1, NQ>(T.WD, fx, acc);
    acc[0] = Real(0);
}

// Values of a polynomial at xi = -1 and +1
template <int N1>
__device__ __forceinline__ void line_ends(const Real (&c)[N1], Real& lo, Real& hi)
{
    lo = hi = Real(0);
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        hi += c[k];
        lo = (k & 1) ? lo - c[k] : lo + c[k];
    }
}

// One coefficient of the update: r + (-gamma nu) (K c)_k, M^{-1}, Runge-Kutta combination.
template <int P>
__device__ __forceinline__ Real line_update(const KParams& A, const Tab<P>& T, int k, Real r, Real ngs,
                                            const Real (&c)[P + 1], Real un, Real cn, Real ck, Real cl)
{
    if (k > 0) {
        Real kc = Real(0);
#pragma unroll
        for (int m = 1; m <= P; ++m)
            if (((k + m) & 1) == 0) kc = fma(T.A1[k][m], c[m], kc);
        r = fma(ngs, kc, r);
    }
    const Real Lk = (A.two_h * T.minv[k]) * r;
    return fma(cn, un, fma(cl, Lk, ck * c[k]));
}

// Runs the stages of nsteps steps: stage(cn, ck, cl) advances c in place.
template <int NC, class Stage>
__device__ __forceinline__ void line_run(const LineSteps& L, Real (&c)[NC], Real (&un)[NC], Stage&& stage)
{
    for (int n = 0; n < L.nsteps; ++n) {
        if (!L.Un) {
#pragma unroll
            for (int k = 0; k < NC; ++k) un[k] = c[k];
        }
#pragma unroll 1
        for (int r = 0; r < L.stages; ++r) {
            const int i = L.order == 4 ? (r == 9) : r;
            stage(L.cn[i], L.ck[i], L.cl[i]);
            if (L.order == 4 && r == 4) {
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    un[k] = un[k] / Real(25) + Real(9) / Real(25) * c[k];
                    c[k] = Real(15) * un[k] - Real(5) * c[k];
                }
            }
        }
    }
}

template <int P, int FLUX>
__global__ void __launch_bounds__(kLineThreads) line_kernel(const __grid_constant__ KParams A, const __grid_constant__ LineSteps L)
{
    constexpr int N1 = P + 1;
    __shared__ Real sc[2][N1][kLineThreads + 2];      // coefficients, double-buffered
    const Tab<P>& T = tab<P>();
    const LinePlace w(A, L, threadIdx.x);
    Real c[N1], un[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        c[k] = w.in ? L.Uin[k * A.E + w.gx] : Real(0);
        un[k] = w.in && L.Un ? L.Un[k * A.E + w.gx] : c[k];
    }
    const bool find_lam = A.stab != STAB_DG && !A.lam_fixed;
    const Real xl = fma_x(Real(w.gx), A.h, A.x0), xr = fma_x(Real(w.gx + 1), A.h, A.x0);
    const Real xc = fma_x(Real(w.gx) + Real(0.5), A.h, A.x0);
    const bool has[2] = {w.has_l, w.has_r};
    Real chk = Real(0);
    int buf = 0;
    cluster_arrive();      // no CTA writes into another before all have started
    cluster_wait();
    line_run(L, c, un, [&](Real cn, Real ck, Real cl) {
        if (w.in) {
#pragma unroll
            for (int k = 0; k < N1; ++k) sc[buf][k][w.col] = c[k];
        }
        if (w.edge_l) {
#pragma unroll
            for (int k = 0; k < N1; ++k) st_cluster(&sc[buf][k][w.col_l], w.rank_l, c[k]);
        }
        if (w.edge_r) {
#pragma unroll
            for (int k = 0; k < N1; ++k) st_cluster(&sc[buf][k][w.col_r], w.rank_r, c[k]);
        }
        cluster_arrive();
        Real acc[N1], key = Real(0), lo, hi;
        line_volume<P, FLUX>(A, T, c, xc, acc, key);
        line_ends(c, lo, hi);
        cluster_wait();
        if (w.in) {
            Real nb[2][N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                nb[0][k] = w.has_l ? sc[buf][k][w.col - 1] : Real(0);
                nb[1][k] = w.has_r ? sc[buf][k][w.col + 1] : Real(0);
            }
            Real gamma = A.stab == STAB_LO ? Real(1) : Real(0);
            if (A.stab >= STAB_WENO) gamma = sensor_1d<P, true>(A, T, c, nb, has);
            // fluxes of the left and right face; beyond a side the ghost of the boundary
            Real ul, ur, t, h[2];
            line_ends(nb[0], t, ul);
            if (!w.has_l) ul = (A.bc[0] == BC_INFLOW_ZERO && -dflux_axis<FLUX>(A, 0, lo, xl, Real(0)) < Real(0)) ? Real(0) : lo;
            line_ends(nb[1], ur, t);
            if (!w.has_r) ur = (A.bc[1] == BC_INFLOW_ZERO && dflux_axis<FLUX>(A, 0, hi, xr, Real(0)) < Real(0)) ? Real(0) : hi;
            if constexpr (FLUX == FLUX_KPP) {
                h[0] = llf_kpp(ul, lo);
                h[1] = llf_kpp(hi, ur);
            } else {
                h[0] = llf<FLUX>(A, 0, ul, lo, xl, Real(0));
                h[1] = llf<FLUX>(A, 0, hi, ur, xr, Real(0));
            }
            Real lam = Real(0);
            if (find_lam)
                lam = speed_of_key<FLUX>(A, fmax(key, fmax(speed_key<FLUX>(A, lo, xl, Real(0)), speed_key<FLUX>(A, hi, xr, Real(0)))));
            const Real ngs = A.stab == STAB_DG ? Real(0) : -(gamma * (A.lam_fixed ? A.lambda_nu : lam) * Real(1.0 / P));
            const Real de = h[0] - h[1], dd = h[0] + h[1];
            Real out[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                out[k] = line_update<P>(A, T, k, (k & 1) ? acc[k] - dd : acc[k] + de, ngs, c, un[k], cn, ck, cl);
                chk = fma(out[k], Real(0), chk);
            }
#pragma unroll
            for (int k = 0; k < N1; ++k) c[k] = out[k];
        }
        buf ^= 1;
    });
    if (!w.in) return;
#pragma unroll
    for (int k = 0; k < N1; ++k) L.U[k * A.E + w.gx] = c[k];
    if (chk != chk) atomicOr(A.flag, 1u);
}

// The Euler system: a cell publishes its density coefficients and, for each of its ends, the
// state, the two flux components that differ from it and |v| + c, so that no state is
// converted to primitive variables twice.
template <int P>
__global__ void __launch_bounds__(kLineThreads) line_euler_kernel(const __grid_constant__ KParams A, const __grid_constant__ LineSteps L)
{
    constexpr int N1 = P + 1, NQ = P + 2, NS = N1 + 12;
    // rows 0 .. P: density; N1 + 6 s + {0, 1, 2, 3, 4, 5}: rho, m, rho E, F_1, F_2, |v| + c at end s
    extern __shared__ __align__(16) unsigned char smem_line[];
    Real (*sv)[NS][kLineThreads + 2] = reinterpret_cast<Real (*)[NS][kLineThreads + 2]>(smem_line);
    const Tab<P>& T = tab<P>();
    const LinePlace w(A, L, threadIdx.x);
    Real c[3 * N1], un[3 * N1];
#pragma unroll
    for (int k = 0; k < 3 * N1; ++k) {
        c[k] = w.in ? L.Uin[k * A.E + w.gx] : Real(k % N1 == 0 ? (k == N1 ? 0 : 1) : 0);
        un[k] = w.in && L.Un ? L.Un[k * A.E + w.gx] : c[k];
    }
    const bool find_lam = A.stab != STAB_DG && !A.lam_fixed;
    const bool has[2] = {w.has_l, w.has_r};
    Real chk = Real(0);
    int buf = 0;
    cluster_arrive();      // no CTA writes into another before all have started
    cluster_wait();
    line_run(L, c, un, [&](Real cn, Real ck, Real cl) {
        Real comp[3][N1], e[2][6];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int k = 0; k < N1; ++k) comp[q][k] = c[q * N1 + k];
#pragma unroll
        for (int q = 0; q < 3; ++q) line_ends(comp[q], e[0][q], e[1][q]);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const EulerState st = euler_prim(A, e[s][0], e[s][1], e[s][2]);
            Real F[3];
            euler_flux(st, e[s][1], e[s][2], F);
            e[s][3] = F[1];
            e[s][4] = F[2];
            e[s][5] = euler_speed(A, st);
        }
        if (w.in) {
#pragma unroll
            for (int k = 0; k < N1; ++k) sv[buf][k][w.col] = comp[0][k];
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < 6; ++i) sv[buf][N1 + 6 * s + i][w.col] = e[s][i];
        }
        if (w.edge_l) {        // the CTA before reads this cell's left end
#pragma unroll
            for (int k = 0; k < N1; ++k) st_cluster(&sv[buf][k][w.col_l], w.rank_l, comp[0][k]);
#pragma unroll
            for (int i = 0; i < 6; ++i) st_cluster(&sv[buf][N1 + i][w.col_l], w.rank_l, e[0][i]);
        }
        if (w.edge_r) {
#pragma unroll
            for (int k = 0; k < N1; ++k) st_cluster(&sv[buf][k][w.col_r], w.rank_r, comp[0][k]);
#pragma unroll
            for (int i = 0; i < 6; ++i) st_cluster(&sv[buf][N1 + 6 + i][w.col_r], w.rank_r, e[1][i]);
        }
        cluster_arrive();
        // volume term and lambda_e over its points
        Real acc[3][N1], lam = Real(0);
        {
            Real u[3][NQ], F[3][NQ];
#pragma unroll
            for (int q = 0; q < 3; ++q) interp_sym<N1, NQ>(T.B, comp[q], u[q]);
#pragma unroll
            for (int g = 0; g < NQ; ++g) {
                const EulerState st = euler_prim(A, u[0][g], u[1][g], u[2][g]);
                Real f[3];
                euler_flux(st, u[1][g], u[2][g], f);
                if (find_lam) lam = max_nan(lam, euler_speed(A, st));
#pragma unroll
                for (int q = 0; q < 3; ++q) F[q][g] = f[q];
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                project_sym<true, N1, NQ>(T.WD, F[q], acc[q]);
                acc[q][0] = Real(0);
            }
        }
        if (find_lam) lam = max_nan(lam, max_nan(e[0][5], e[1][5]));
        cluster_wait();
        if (w.in) {
            Real nb[2][N1], o[2][6];
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                nb[0][k] = w.has_l ? sv[buf][k][w.col - 1] : Real(0);
                nb[1][k] = w.has_r ? sv[buf][k][w.col + 1] : Real(0);
            }
            // the state across each face: the neighbour's end, or the boundary's ghost (a wall
            // mirrors the momentum, which keeps F_1 and |v| + c and mirrors F_2)
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    Real v = e[s][i];
                    if (A.bc[s] == BC_REFLECT && (i == 1 || i == 4)) v = -v;
                    o[s][i] = has[s] ? sv[buf][N1 + 6 * (1 - s) + i][w.col + (s ? 1 : -1)] : v;
                }
            Real gamma = A.stab == STAB_LO ? Real(1) : Real(0);
            if (A.stab >= STAB_WENO) gamma = sensor_1d<P>(A, T, comp[0], nb, has);
            const Real ngs = A.stab == STAB_DG ? Real(0) : -(gamma * (A.lam_fixed ? A.lambda_nu : lam) * Real(1.0 / P));
            Real h[2][3];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const Real (&uL)[6] = s ? e[1] : o[0];
                const Real (&uR)[6] = s ? o[1] : e[0];
                const Real sp = max_nan(uL[5], uR[5]);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const Real fl = q == 0 ? uL[1] : uL[2 + q], fr = q == 0 ? uR[1] : uR[2 + q];
                    h[s][q] = Real(0.5) * ((fl + fr) - sp * (uR[q] - uL[q]));
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    const Real r = acc[q][k] + ((k & 1) ? -(h[0][q] + h[1][q]) : (h[0][q] - h[1][q]));
                    const Real out = line_update<P>(A, T, k, r, ngs, comp[q], un[q * N1 + k], cn, ck, cl);
                    chk = fma(out, Real(0), chk);
                    c[q * N1 + k] = out;
                }
        }
        buf ^= 1;
    });
    if (!w.in) return;
#pragma unroll
    for (int k = 0; k < 3 * N1; ++k) L.U[k * A.E + w.gx] = c[k];
    if (chk != chk) atomicOr(A.flag, 1u);
}

// ------------------------------------------------------------------------------------
// Eight lanes per cell (double)
// ------------------------------------------------------------------------------------
__device__ __forceinline__ Real group_get(Real v, int src) { return __shfl_sync(0xffffffffu, v, src, 8); }
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }
__device__ __forceinline__ bool not_finite(float v) { return (__float_as_int(v) & 0x7f800000) == 0x7f800000; }
// largest v >= 0 of the cell's lanes
__device__ __forceinline__ Real group_max(Real v)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v = max_pos(v, __shfl_xor_sync(0xffffffffu, v, o, 8));
    return v;
}

// v^T G v in 1D (G_mn = 0 for odd m + n)
template <int P>
__device__ __forceinline__ Real qform_1d(const Tab<P>& T, const Real (&v)[P + 1])
{
    Real t = T.Gu[1][1] * v[1];
    if constexpr (P == 3) t = fma(T.Gu[1][3], v[3], t);
    Real s = t * v[1];
#pragma unroll
    for (int k = 2; k <= P; ++k) s = fma(T.Gu[k][k] * v[k], v[k], s);
    return s;
}

// What a lane keeps of the tables: lane `sub` of a cell evaluates point sub, candidate sub & 3
// (own, left, right, own), face sub & 1 and mode min(sub, P).
template <int P>
struct WideLane {
    static constexpr int N1 = P + 1, NQ = P + 2;
    int sub, role, side;
    Real shift[3];         // candidate: T(1,2), T(1,3), T(2,3); zero for the cell's own
    Real end;              // xi at the lane's face: -1 or +1
    Real lin;              // the candidate's linear weight; 0 for a neighbour that is missing
    __device__ __forceinline__ WideLane(const KParams& A, const Tab<P>& T, const LinePlace& w, int sub_)
        : sub(sub_), role(sub_ & 3), side(sub_ & 1)
    {
        const int me = (w.has_l ? 1 : 0) + (w.has_r ? 1 : 0);
        lin = role == 1 ? (w.has_l ? A.w_nbr : Real(0)) : (role == 2 ? (w.has_r ? A.w_nbr : Real(0)) : Real(1) - Real(me) * A.w_nbr);
        const int t = role == 2 ? 1 : 0;
        const bool nb = role == 1 || role == 2;
        shift[0] = nb && P >= 2 ? T.T[t][1][P >= 2 ? 2 : 0] : Real(0);
        shift[1] = nb && P >= 3 ? T.T[t][1][P >= 3 ? 3 : 0] : Real(0);
        shift[2] = nb && P >= 3 ? T.T[t][P >= 3 ? 2 : 0][P >= 3 ? 3 : 0] : Real(0);
        end = side ? Real(1) : Real(-1);
    }
    // sum_k x^k c_k for x = -1 or +1: the polynomial's value at that end
    __device__ __forceinline__ static Real at_end(const Real (&c)[N1], Real x)
    {
        Real v = c[0];
#pragma unroll
        for (int k = 1; k < N1; ++k) v = (k & 1) ? fma(x, c[k], v) : v + c[k];
        return v;
    }
};

// The sensor of sensor_1d with a candidate per lane.  Only ratios of the weights lin / (eps_w +
// beta)^2 matter, so they are scaled by all the (eps_w + beta)^2: no division but the last, and
// that one with its square root as one reciprocal square root: gamma = ||D|| / (W ||U||) for
// D = sum_l w_l (c - c_l), W = sum_l w_l.  States whose products could leave the range of double
// take sensor_1d.
template <int P, bool TILE>
__device__ __forceinline__ Real wide_sensor(const KParams& A, const Tab<P>& T, const WideLane<P>& w, const Real (&c)[P + 1],
                                            const Real (&nb)[2][P + 1], const bool (&has)[2])
{
    constexpr int N1 = P + 1;
    if (A.stab == STAB_ZHAO) return sensor_1d<P, TILE>(A, T, c, nb, has);
    Real cl[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) cl[k] = w.role == 1 ? nb[0][k] : (w.role == 2 ? nb[1][k] : c[k]);
    if constexpr (P >= 3) {
        cl[1] = fma(w.shift[0], cl[2], fma(w.shift[1], cl[3], cl[1]));
        cl[2] = fma(w.shift[2], cl[3], cl[2]);
    } else if constexpr (P == 2) {
        cl[1] = fma(w.shift[0], cl[2], cl[1]);
    }
    const Real beta = qform_1d<P>(T, cl);
    const Real beta0 = group_get(beta, 0);
    const Real d = A.eps_w + beta;
    const Real d2 = d * d;
    const Real one = Real(1);
    // (every lane takes part in the exchanges; a missing neighbour's value is then replaced)
    const Real d20 = group_get(d2, 0), g1 = group_get(d2, 1), g2 = group_get(d2, 2);
    const Real d21 = has[0] ? g1 : one, d22 = has[1] ? g2 : one;
    const bool nbr = w.role == 1 || w.role == 2;
    const Real wt = w.lin * ((nbr ? d20 : d21) * (w.role == 2 ? d21 : d22));
    const Real wl = group_get(wt, 1), wr = group_get(wt, 2);
    const Real W = (group_get(wt, 0) + wl) + wr;
    Real D[N1];
    D[0] = Real(0);
#pragma unroll
    for (int k = 1; k < N1; ++k) {
        const Real e = wt * (c[k] - cl[k]);
        D[k] = group_get(e, 1) + group_get(e, 2);
    }
    const Real qd = qform_1d<P>(T, D);
    const Real W2 = W * W, den = W2 * beta0, pr = qd * den;
    // every product above stays in range for 1e-16 <= (eps_w + beta)^2 <= 1e24
    const Real hi = max_pos(d20, max_pos(d21, d22)), lo = less_pos(d21, d22) ? d21 : d22;
    const bool flat = !less_pos(Real(0), qd) || !less_pos(Real(0), beta0);
    if (!less_pos(hi, Real(1e24)) || !less_pos(Real(1e-16), lo) || !less_pos(Real(1e-16), d20) ||
        !(flat || less_pos(Real(1e-280), pr)))
        return sensor_1d<P, TILE>(A, T, c, nb, has);
    if (!less_pos((A.eps_s * A.eps_s) * W2, qd)) return Real(0);
    if (flat) return Real(1);
    Real r = Real(1);
    if (less_pos(qd, den)) r = qd * rsqrt(pr);
    Real g = less_pos(r, Real(1)) ? r : Real(1);
    if (!A.q_one) g = pow(g, A.q);
    if (less_pos(r, A.b)) g = Real(0);
    return g;
}

template <int P, int FLUX>
__global__ void __launch_bounds__(8 * kWideCells) line_wide_kernel(const __grid_constant__ KParams A, const __grid_constant__ LineSteps L)
{
    constexpr int N1 = P + 1, NQ = P + 2;
    __shared__ Real sc[2][N1][kWideCells + 2];
    const Tab<P>& T = tab<P>();
    const LinePlace w(A, L, threadIdx.x >> 3);
    const WideLane<P> g(A, T, w, threadIdx.x & 7);
    const int q = g.sub < NQ ? g.sub : NQ - 1, km = g.sub < N1 ? g.sub : P;
    const bool owner = w.in && g.sub < N1;
    Real b[N1], wd[NQ], a1[N1], c[N1], v[1], un[1];
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        b[k] = T.B[q][k];
        a1[k] = k > 0 && km > 0 && ((km + k) & 1) == 0 ? T.A1[km][k] : Real(0);
        c[k] = w.in ? L.Uin[k * A.E + w.gx] : Real(0);
    }
#pragma unroll
    for (int i = 0; i < NQ; ++i) wd[i] = km > 0 ? T.WD[i][km] : Real(0);
    v[0] = c[0];
#pragma unroll
    for (int k = 1; k < N1; ++k)
        if (km == k) v[0] = c[k];
    un[0] = owner && L.Un ? L.Un[km * A.E + w.gx] : v[0];
    const Real sgk = (km & 1) ? Real(-1) : Real(1), mk = A.two_h * T.minv[km];
    const bool find_lam = A.stab != STAB_DG && !A.lam_fixed;
    const Real xq = fma_x(A.hh, T.g[q], fma_x(Real(w.gx) + Real(0.5), A.h, A.x0));
    const Real xf = fma_x(Real(w.gx + g.side), A.h, A.x0);
    const bool has[2] = {w.has_l, w.has_r};
    bool bad = false;
    int buf = 0;
    cluster_arrive();      // no CTA writes into another before all have started
    cluster_wait();
    line_run(L, v, un, [&](Real cn, Real ck, Real cl) {
        if (owner) {
            sc[buf][km][w.col] = v[0];
            if (w.edge_l) st_cluster(&sc[buf][km][w.col_l], w.rank_l, v[0]);
            if (w.edge_r) st_cluster(&sc[buf][km][w.col_r], w.rank_r, v[0]);
        }
        cluster_arrive();
        if (L.order == 4) {    // the recombination changed the modes in their own lanes only
#pragma unroll
            for (int k = 0; k < N1; ++k) c[k] = group_get(v[0], k);
        }
        // volume term: point q in lane q, mode k in lane k
        Real u = c[0], f, fy, key;
#pragma unroll
        for (int k = 1; k < N1; ++k) u = fma(b[k], c[k], u);
        vol_flux<FLUX>(A, u, xq, Real(0), f, fy, key);
        Real acc = wd[0] * group_get(f, 0);
#pragma unroll
        for (int i = 1; i < NQ; ++i) acc = fma(wd[i], group_get(f, i), acc);
        const Real own = WideLane<P>::at_end(c, g.end);
        cluster_wait();
        Real nb[2][N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            nb[0][k] = w.has_l ? sc[buf][k][w.col - 1] : Real(0);
            nb[1][k] = w.has_r ? sc[buf][k][w.col + 1] : Real(0);
        }
        Real gamma = A.stab == STAB_LO ? Real(1) : Real(0);
        if (A.stab >= STAB_WENO) gamma = wide_sensor<P, true>(A, T, g, c, nb, has);
        // the flux of the lane's face
        Real other;
        {
            Real o[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) o[k] = g.side ? nb[1][k] : nb[0][k];
            other = WideLane<P>::at_end(o, -g.end);
        }
        if (!(g.side ? w.has_r : w.has_l))
            other = (A.bc[g.side] == BC_INFLOW_ZERO && g.end * dflux_axis<FLUX>(A, 0, own, xf, Real(0)) < Real(0)) ? Real(0) : own;
        const Real ul = g.side ? own : other, ur = g.side ? other : own;
        Real h;
        if constexpr (FLUX == FLUX_KPP) h = llf_kpp(ul, ur);
        else h = llf<FLUX>(A, 0, ul, ur, xf, Real(0));
        const Real h0 = group_get(h, 0), h1 = group_get(h, 1);
        Real lam = Real(0);
        if (find_lam) lam = speed_of_key<FLUX>(A, group_max(max_pos(key, speed_key<FLUX>(A, own, xf, Real(0)))));
        const Real ngs = A.stab == STAB_DG ? Real(0) : -(gamma * (A.lam_fixed ? A.lambda_nu : lam) * Real(1.0 / P));
        // the lane's mode
        Real r = acc + fma(sgk, h0, -h1), kc = a1[1] * c[1];
#pragma unroll
        for (int k = 2; k < N1; ++k) kc = fma(a1[k], c[k], kc);
        r = fma(ngs, kc, r);
        v[0] = fma(cn, un[0], fma(cl, mk * r, ck * v[0]));
        bad = bad || not_finite(v[0]);
#pragma unroll
        for (int k = 0; k < N1; ++k) c[k] = group_get(v[0], k);
        buf ^= 1;
    });
    if (!owner) return;
    L.U[km * A.E + w.gx] = v[0];
    if (bad) atomicOr(A.flag, 1u);
}

// The Euler system, eight lanes per cell: a Gauss point or an end of the cell per lane, a
// component of a face per lane, a mode per lane in two rounds (mode i = 3 (P - k) + component, so
// that the round left over holds the simplest ones).
template <int P>
struct WideEulerSmem {
    static constexpr int N1 = P + 1, NQ = P + 2;
    // exchanged, double-buffered: density modes, then rho, m, rho E, F_1, F_2, |v| + c per end
    Real sv[2][N1 + 12][kWideCells + 2];
    Real f[kWideCells][3][NQ + 1];         // fluxes at the points (padded)
    Real h[kWideCells][3][2];              // fluxes of the faces
    Real c[kWideCells][3 * N1 + 1];        // modes
};

template <int P>
__global__ void __launch_bounds__(8 * kWideCells) line_wide_euler_kernel(const __grid_constant__ KParams A, const __grid_constant__ LineSteps L)
{
    constexpr int N1 = P + 1, NQ = P + 2, NM = 3 * N1, R = (NM + 7) / 8;
    constexpr bool kMeansOnly = P == 2;    // the last round holds one mode, the mean of rho E
    __shared__ WideEulerSmem<P> S;
    const Tab<P>& T = tab<P>();
    const int ci = threadIdx.x >> 3;
    const LinePlace w(A, L, ci);
    const WideLane<P> g(A, T, w, threadIdx.x & 7);
    // lanes 0 .. NQ-1: the points; NQ, NQ + 1: the ends
    const int pt = g.sub;
    Real b[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k)
        b[k] = pt < NQ ? T.B[pt < NQ ? pt : 0][k] : ((k & 1) && pt == NQ ? Real(-1) : Real(1));
    Real c[3][N1], v[R], un[R], mk[R], wd[R][NQ], a1[R][N1];
    int mode[R], mcomp[R], mdeg[R];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int k = 0; k < N1; ++k) c[q][k] = w.in ? L.Uin[(q * N1 + k) * A.E + w.gx] : Real(k == 0 && q != 1 ? 1 : 0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = g.sub + 8 * r < NM ? g.sub + 8 * r : NM - 1;
        mcomp[r] = i % 3;
        mdeg[r] = P - i / 3;
        mode[r] = mcomp[r] * N1 + mdeg[r];
        mk[r] = A.two_h * T.minv[mdeg[r]];
#pragma unroll
        for (int i = 0; i < NQ; ++i) wd[r][i] = T.WD[i][mdeg[r]];          // zero for the mean
#pragma unroll
        for (int m = 0; m < N1; ++m) a1[r][m] = m > 0 && mdeg[r] > 0 && ((mdeg[r] + m) & 1) == 0 ? T.A1[mdeg[r]][m] : Real(0);
        // (lanes without a cell keep a state at rest: no divisions by zero, which are slow)
        v[r] = w.in ? L.Uin[mode[r] * A.E + w.gx] : Real(mdeg[r] == 0 && mcomp[r] != 1 ? 1 : 0);
        un[r] = w.in && L.Un ? L.Un[mode[r] * A.E + w.gx] : v[r];
    }
    const bool find_lam = A.stab != STAB_DG && !A.lam_fixed;
    const bool has[2] = {w.has_l, w.has_r};
    const unsigned group = 0xffu << (threadIdx.x & 24);
    bool bad = false;
    int buf = 0;
    cluster_arrive();      // no CTA writes into another before all have started
    cluster_wait();
    line_run(L, v, un, [&](Real cn, Real ck, Real cl) {
        // all modes of the cell in every lane
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (g.sub + 8 * r < NM) S.c[ci][mode[r]] = v[r];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int k = 0; k < N1; ++k) c[q][k] = S.c[ci][q * N1 + k];
        // the lane's point or end
        Real u[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            u[q] = c[q][0];
#pragma unroll
            for (int k = 1; k < N1; ++k) u[q] = fma(b[k], c[q][k], u[q]);
        }
        const EulerState st = euler_prim(A, u[0], u[1], u[2]);
        Real F[3];
        euler_flux(st, u[1], u[2], F);
        const Real sp = euler_speed(A, st);
        if (pt < NQ) {
#pragma unroll
            for (int q = 0; q < 3; ++q) S.f[ci][q][pt] = F[q];
        } else if (pt < NQ + 2 && w.in) {
            const int s = pt - NQ;
            const Real e[6] = {u[0], u[1], u[2], F[1], F[2], sp};
            const bool edge = s ? w.edge_r : w.edge_l;
            const uint32_t rank = s ? w.rank_r : w.rank_l;
            const int col = s ? w.col_r : w.col_l;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                S.sv[buf][N1 + 6 * s + i][w.col] = e[i];
                if (edge) st_cluster(&S.sv[buf][N1 + 6 * s + i][col], rank, e[i]);
            }
        }
        if (g.sub < N1 && w.in) {
            Real rho = c[0][0];
#pragma unroll
            for (int k = 1; k < N1; ++k)
                if (g.sub == k) rho = c[0][k];
            S.sv[buf][g.sub][w.col] = rho;
            if (w.edge_l) st_cluster(&S.sv[buf][g.sub][w.col_l], w.rank_l, rho);
            if (w.edge_r) st_cluster(&S.sv[buf][g.sub][w.col_r], w.rank_r, rho);
        }
        cluster_arrive();
        // lambda_e over the points and the ends (a NaN speed stays one); the volume term
        Real lam = Real(0);
        if (find_lam) {
            const bool used = pt < NQ + 2;
            lam = group_max(used ? sp : Real(0));
            if (__ballot_sync(0xffffffffu, used && not_finite(sp)) & group) lam = Real(NAN);
        }
        __syncwarp();
        Real acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            acc[r] = Real(0);
            if (kMeansOnly && r == R - 1) continue;
#pragma unroll
            for (int i = 0; i < NQ; ++i) acc[r] = fma(wd[r][i], S.f[ci][mcomp[r]][i], acc[r]);
        }
        cluster_wait();
        Real nb[2][N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) {
            nb[0][k] = w.has_l ? S.sv[buf][k][w.col - 1] : Real(0);
            nb[1][k] = w.has_r ? S.sv[buf][k][w.col + 1] : Real(0);
        }
        Real gamma = A.stab == STAB_LO ? Real(1) : Real(0);
        if (A.stab >= STAB_WENO) gamma = wide_sensor<P, false>(A, T, g, c[0], nb, has);
        // lane sub < 6: component sub >> 1 of face sub & 1, between columns col - 1 + side and
        // col + side; beyond a side the ghost: the inner end, its momentum mirrored at a wall
        {
            const int q = g.sub < 6 ? g.sub >> 1 : 0, fr = N1 + (q == 0 ? 1 : 2 + q);   // row of F_q at end 0
            const bool gl = !w.has_l && g.side == 0, gr = !w.has_r && g.side == 1;
            const int colL = gl ? w.col : w.col - 1 + g.side, colR = gr ? w.col : w.col + g.side;
            const int eL = gl ? 0 : 6, eR = gr ? 6 : 0;
            Real uL = Real(0), uR = Real(0), fL = Real(0), fR = Real(0), sL = Real(0), sR = Real(0);
            if (w.in) {
                uL = S.sv[buf][N1 + eL + q][colL]; uR = S.sv[buf][N1 + eR + q][colR];
                fL = S.sv[buf][fr + eL][colL];     fR = S.sv[buf][fr + eR][colR];
                sL = S.sv[buf][N1 + eL + 5][colL]; sR = S.sv[buf][N1 + eR + 5][colR];
            }
            const bool wall = A.bc[g.side] == BC_REFLECT;
            if (gl && wall) { if (q == 1) uL = -uL; if (q != 1) fL = -fL; }
            if (gr && wall) { if (q == 1) uR = -uR; if (q != 1) fR = -fR; }
            Real s = max_pos(sL, sR);
            if (not_finite(sL)) s = sL;        // a state without a sound speed: NaN
            if (not_finite(sR)) s = sR;
            const Real h = Real(0.5) * ((fL + fR) - s * (uR - uL));
            if (g.sub < 6) S.h[ci][q][g.side] = h;
        }
        __syncwarp();
        const Real ngs = A.stab == STAB_DG ? Real(0) : -(gamma * (A.lam_fixed ? A.lambda_nu : lam) * Real(1.0 / P));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = mdeg[r];
            const Real h0 = S.h[ci][mcomp[r]][0], h1 = S.h[ci][mcomp[r]][1];
            Real x = acc[r] + ((k & 1) ? -(h0 + h1) : h0 - h1);
            if (!(kMeansOnly && r == R - 1)) {
                Real kc = Real(0);
#pragma unroll
                for (int m = 1; m < N1; ++m) kc = fma(a1[r][m], S.c[ci][mcomp[r] * N1 + m], kc);
                x = fma(ngs, kc, x);
            }
            if (w.in) v[r] = fma(cn, un[r], fma(cl, mk[r] * x, ck * v[r]));
            bad = bad || not_finite(v[r]);
        }
        __syncwarp();          // the next stage's modes replace those that other lanes read above
        buf ^= 1;
    });
    if (!w.in) return;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (g.sub + 8 * r < NM) L.U[mode[r] * A.E + w.gx] = v[r];
    if (bad) atomicOr(A.flag, 1u);
}

// Largest cluster of `fn` on the current device with `threads` threads a CTA: 16, 8, or 0 if
// neither can run.
static int line_max_cluster(const void* fn, int threads, size_t smem)
{
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
    if (smem > 48 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    for (int n = kLineCluster; n >= 8; n /= 2) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = n;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(n);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) == cudaSuccess && nc >= 1) return n;
        cudaGetLastError();
    }
    return 0;
}

// Launches fn (lanes threads per cell) on the smallest CTAs, from `smallest` cells up to
// `largest`, with which the mesh fits one cluster.
template <class Kernel>
static cudaError_t launch_line_k(Kernel fn, int lanes, int smallest, int largest, size_t smem, int (&limit)[64],
                                 const KParams& a, LineSteps& L, bool query, cudaStream_t st)
{
    const int dev = cur_device();
    int lim = __atomic_load_n(&limit[dev], __ATOMIC_RELAXED);
    if (lim == 0) {
        lim = line_max_cluster((const void*)fn, largest * lanes, smem);
        if (lim == 0) lim = -1;
        __atomic_store_n(&limit[dev], lim, __ATOMIC_RELAXED);
    }
    if (lim < 0) return cudaErrorNotSupported;
    int cells = smallest;
    while (cells <= largest && (a.nx + cells - 1) / cells > lim) cells *= 2;
    if (cells > largest) return cudaErrorNotSupported;
    if (query) return cudaSuccess;
    L.cells = cells;
    int n = 1;
    while (n * cells < a.nx) n *= 2;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(cells * lanes);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, a, L);
}

// Double: eight lanes per cell up to kWideMax cells (if clusters of 16 can run; with clusters of
// 8 up to half as many), one lane per cell beyond.
template <int P, int FLUX>
static cudaError_t launch_line_pf(const KParams& a, LineSteps& L, bool query, cudaStream_t st)
{
    if constexpr (!kF32) {
        static int wide[64] = {0};
        if (a.nx <= kWideMax) {
            const cudaError_t e = launch_line_k(line_wide_kernel<P, FLUX>, 8, 4, kWideCells, 0, wide, a, L, query, st);
            if (e != cudaErrorNotSupported) return e;
        }
    }
    static int limit[64] = {0};
    return launch_line_k(line_kernel<P, FLUX>, 1, 32, kLineThreads, 0, limit, a, L, query, st);
}

template <int P>
static cudaError_t launch_line_euler(const KParams& a, LineSteps& L, bool query, cudaStream_t st)
{
    if constexpr (!kF32) {
        static int wide[64] = {0};
        if (a.nx <= kWideMax) {
            const cudaError_t e = launch_line_k(line_wide_euler_kernel<P>, 8, 4, kWideCells, 0, wide, a, L, query, st);
            if (e != cudaErrorNotSupported) return e;
        }
    }
    static int limit[64] = {0};
    return launch_line_k(line_euler_kernel<P>, 1, 32, kLineThreads, sizeof(Real) * 2 * (P + 13) * (kLineThreads + 2), limit,
                         a, L, query, st);
}

template <int P>
static cudaError_t launch_line_p(const KParams& a, LineSteps& L, int flux, bool query, cudaStream_t st)
{
    switch (flux) {
    case FLUX_ADVECT: return launch_line_pf<P, FLUX_ADVECT>(a, L, query, st);
    case FLUX_ROTATION: return launch_line_pf<P, FLUX_ROTATION>(a, L, query, st);
    case FLUX_BURGERS: return launch_line_pf<P, FLUX_BURGERS>(a, L, query, st);
    case FLUX_KPP: return launch_line_pf<P, FLUX_KPP>(a, L, query, st);
    case FLUX_EULER: return launch_line_euler<P>(a, L, query, st);
    default: return cudaErrorInvalidValue;
    }
}

// Launches L, whose nsteps may be 0 to ask whether the mesh fits.
static cudaError_t launch_line_any(const KParams& a, LineSteps& L, int p, int flux, cudaStream_t st)
{
    const bool query = L.nsteps == 0;
    if (a.nx > kLineCluster * kLineThreads) return cudaErrorNotSupported;
    if (p == 1) return launch_line_p<1>(a, L, flux, query, st);
    if (p == 2) return launch_line_p<2>(a, L, flux, query, st);
    if (p == 3) return launch_line_p<3>(a, L, flux, query, st);
    return cudaErrorInvalidValue;
}

// The stage Uout = cn Un + ck Uk + cl L(Uk) of s alone.  cudaErrorNotSupported: the mesh does not
// fit one cluster, nothing was launched.
static cudaError_t launch_line_stage(const StageArgs& s, int p, int flux, cudaStream_t st)
{
    const KParams a = make_params(s);
    LineSteps L;
    memset(&L, 0, sizeof L);
    L.Uin = a.Uk;
    L.Un = a.has_un ? a.Un : nullptr;
    L.U = a.Uout;
    L.nsteps = L.stages = 1;
    L.cn[0] = a.cn;
    L.ck[0] = a.ck;
    L.cl[0] = a.cl;
    return launch_line_any(a, L, p, flux, st);
}

// nsteps steps of the mesh of s in place on U, or (nsteps = 0) only whether the mesh fits.
// cudaErrorNotSupported: it does not fit one cluster, nothing was launched.
static cudaError_t launch_line(const StageArgs& s, int p, int flux, void* U, double dt, int nsteps, int order, cudaStream_t st)
{
    const KParams a = make_params(s);
    LineSteps L;
    memset(&L, 0, sizeof L);
    L.Uin = L.U = static_cast<Real*>(U);
    L.order = order;
    L.stages = order == 4 ? 10 : order;
    const double t3[3][3] = {{0.0, 1.0, 1.0}, {0.75, 0.25, 0.25}, {1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0}};
    const double t2[2][3] = {{0.0, 1.0, 1.0}, {0.5, 0.5, 0.5}};
    const double t4[2][3] = {{0.0, 1.0, 1.0 / 6.0}, {1.0, 3.0 / 5.0, 1.0 / 10.0}};
    for (int i = 0; i < (order == 3 ? 3 : 2); ++i) {
        const double* t = order == 3 ? t3[i] : (order == 2 ? t2[i] : t4[i]);
        L.cn[i] = (Real)t[0];
        L.ck[i] = (Real)t[1];
        L.cl[i] = (Real)(t[2] * dt);
    }
    // launches of at most 1024 steps (a few milliseconds each)
    const int kChunk = 1024;
    int left = nsteps;
    do {
        L.nsteps = left < kChunk ? left : kChunk;
        const cudaError_t e = launch_line_any(a, L, p, flux, st);
        if (e != cudaSuccess) return e;
        left -= L.nsteps;
    } while (left > 0);
    return cudaSuccess;
}
