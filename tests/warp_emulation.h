// The eight-lane line kernels on the CPU: every lane is a coroutine that runs until it reaches a
// warp or cluster synchronisation and is taken up again only when all lanes it waits for have
// reached theirs.  Between synchronisations the lanes run one after the other, upwards or
// downwards, so a result that depends on the order misses one.  One CTA (a cluster of one); the
// arithmetic around the exchanges is a stand-in.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>
#include <ucontext.h>

#define __device__
#define __global__
#define __forceinline__ inline
#define __grid_constant__
#define __shared__ static
#define __align__(n)
#define __launch_bounds__(...)
using Real = double;
constexpr bool kF32 = false;
enum { FLUX_BURGERS = 2, FLUX_KPP = 3 };
enum { BC_PERIODIC, BC_INFLOW_ZERO, BC_OUTFLOW, BC_REFLECT };
enum { STAB_DG, STAB_LO, STAB_WENO, STAB_ZHAO };

// ---- lanes ----
struct Lane { ucontext_t ctx; std::vector<char> stack; bool done = false; int waits = 0, at = 0; };
struct Dim { int x; };
static std::vector<Lane> lanes;
static ucontext_t main_ctx;
static int cur;
static std::function<void()> body;
static Dim threadIdx;
static double slot[1024];
static bool flag_slot[1024];
static void entry() { body(); lanes[cur].done = true; swapcontext(&lanes[cur].ctx, &main_ctx); }
// wait until all lanes of the warp (1) or the CTA (2) have come as far
static void meet(int scope)
{
    Lane& l = lanes[cur];
    l.waits = scope;
    ++l.at;
    swapcontext(&l.ctx, &main_ctx);
}
static void run_lanes(int n, bool up, std::function<void()> f)
{
    lanes.assign(n, Lane());
    body = f;
    for (int i = 0; i < n; ++i) {
        lanes[i].stack.resize(256 << 10);
        getcontext(&lanes[i].ctx);
        lanes[i].ctx.uc_stack.ss_sp = lanes[i].stack.data();
        lanes[i].ctx.uc_stack.ss_size = lanes[i].stack.size();
        lanes[i].ctx.uc_link = &main_ctx;
        makecontext(&lanes[i].ctx, entry, 0);
    }
    for (bool any = true; any;) {
        any = false;
        // release the warps (and the CTA) whose lanes have all arrived
        auto release = [&](int lo, int hi, int scope) {
            for (int i = lo; i < hi; ++i) if (lanes[i].done || lanes[i].waits != scope || lanes[i].at != lanes[lo].at) return;
            for (int i = lo; i < hi; ++i) lanes[i].waits = 0;
        };
        for (int w = 0; w < n; w += 32) release(w, w + 32, 1);
        release(0, n, 2);
        for (int j = 0; j < n; ++j) {
            const int i = up ? j : n - 1 - j;
            if (lanes[i].done || lanes[i].waits) continue;
            cur = i;
            threadIdx.x = i;
            swapcontext(&main_ctx, &lanes[i].ctx);
            any = true;
        }
    }
    for (auto& l : lanes) if (!l.done) { std::puts("a lane never met its partners"); std::exit(2); }
}
static void resume() { threadIdx.x = cur; }
static void __syncwarp() { meet(1); resume(); }
static double exchange(double v, int src)
{
    const int me = threadIdx.x;
    slot[me] = v;
    __syncwarp();
    const double r = slot[src];
    __syncwarp();
    return r;
}
static double __shfl_sync(unsigned, double v, int src, int w) { return exchange(v, threadIdx.x / w * w + src % w); }
static double __shfl_xor_sync(unsigned, double v, int o, int) { return exchange(v, threadIdx.x ^ o); }
static unsigned __ballot_sync(unsigned, bool b)
{
    const int me = threadIdx.x, w0 = me & ~31;
    flag_slot[me] = b;
    __syncwarp();
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r |= (flag_slot[w0 + i] ? 1u : 0u) << i;
    __syncwarp();
    return r;
}
static uint32_t cluster_rank() { return 0; }
static void cluster_arrive() {}
static void cluster_wait() { meet(2); resume(); }
static void st_cluster(const Real* p, uint32_t, Real v) { *const_cast<Real*>(p) = v; }
static void atomicOr(unsigned* f, unsigned v) { *f |= v; }
static int __double2hiint(double v) { int64_t b; std::memcpy(&b, &v, 8); return (int)(b >> 32); }
static int __float_as_int(float v) { int b; std::memcpy(&b, &v, 4); return b; }

// ---- stand-ins for what the kernels call ----
struct KParams {
    Real h, hh, x0, two_h, w_nbr, eps_w, eps_s, b, q, lambda_nu;
    int stab, lam_fixed, q_one, nx, bc[4];
    int64_t E;
    unsigned* flag;
};
template <int P> struct Tab {
    Real g[P + 2], B[P + 2][P + 1], WD[P + 2][P + 1], T[2][P + 1][P + 1], Gu[P + 1][P + 1], A1[P + 1][P + 1], minv[P + 1];
};
template <int P> const Tab<P>& tab()
{
    static Tab<P> t;
    Real* v = reinterpret_cast<Real*>(&t);
    for (size_t i = 0; i < sizeof t / sizeof(Real); ++i) v[i] = 0.1 + 0.8 * std::fmod(0.618 * (i + 1), 1.0);
    return t;
}
struct EulerState { Real v, pr; };
static EulerState euler_prim(const KParams&, Real r, Real m, Real e) { return {m / r, e - m * m / r}; }
static void euler_flux(const EulerState& s, Real m, Real e, Real* F) { F[0] = m; F[1] = m * s.v + s.pr; F[2] = (e + s.pr) * s.v; }
static Real euler_speed(const KParams&, const EulerState& s) { return std::fabs(s.v) + std::sqrt(std::fabs(s.pr)); }
static bool less_pos(Real a, Real b) { return a < b; }
static Real max_pos(Real a, Real b) { return a < b ? b : a; }
static Real max_nan(Real a, Real b) { return a < b ? b : a; }
static Real rsqrt(Real x) { return 1 / std::sqrt(x); }
static Real fma_x(Real a, Real b, Real c) { return std::fma(a, b, c); }
using std::fabs; using std::fma; using std::pow;
template <int P, bool TILE = false> Real sensor_1d(const KParams&, const Tab<P>&, const Real* c, const Real (*n)[P + 1], const bool*) { return 0.5 + 0.1 * std::tanh(c[1] + n[0][1] - n[1][1]); }
template <int N1, int NQ> void interp_sym(const Real (&)[NQ][N1], const Real (&r)[N1], Real (&u)[NQ]) { for (auto& x : u) x = r[0]; }
template <bool, int N1, int NQ> void project_sym(const Real (&)[NQ][N1], const Real (&f)[NQ], Real (&o)[N1]) { for (auto& x : o) x = f[0]; }
template <int F> void vol_flux(const KParams&, Real u, Real, Real, Real& f, Real& fy, Real& k) { f = 0.5 * u * u; fy = 0; k = std::fabs(u); }
template <int F> void vol_flux_v(const KParams& A, Real u, Real x, Real y, Real& f, Real& fy, Real& k) { vol_flux<F>(A, u, x, y, f, fy, k); }
template <int F> Real speed_key(const KParams&, Real u, Real, Real) { return std::fabs(u); }
template <int F> Real speed_of_key(const KParams&, Real k) { return k; }
template <int F> Real dflux_axis(const KParams&, int, Real u, Real, Real) { return u; }
template <int F> Real llf(const KParams&, int, Real l, Real r, Real, Real) { return 0.25 * (l * l + r * r) - 0.1 * (r - l); }
static Real llf_kpp(Real l, Real r) { return 0.5 * (l + r); }
