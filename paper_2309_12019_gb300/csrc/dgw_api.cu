// C ABI of libdgw: contexts, argument checks, launch sequences, CUDA-graph replay of
// the SSP-RK3 loop, projection and the mass diagnostic.  See include/dgw.h.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>
#include <algorithm>
#include <vector>
#include <algorithm>
#include <numeric>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include "../../include/dgw.h"
#include "dgw_internal.h"
#include "dgw_math.cuh"

using namespace dgw;

static thread_local std::string g_err;

static dgw_status fail(dgw_status s, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
static dgw_status fail(dgw_status s, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

#define DGW_CUDA(call)                                                                    \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return fail(DGW_ECUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                        __FILE__, __LINE__);                                              \
    } while (0)

using GraphKey = std::tuple<void*, double, int, cudaStream_t>;
// (U_in, U_out, dt, stream, copy flags) of a pipelined host step
using BandKey = std::tuple<const void*, void*, double, cudaStream_t, int>;

struct dgw_ctx {
    int device = 0;
    dgw_mesh mesh{};
    int p = 0;
    dgw_flux flux{};
    dgw_params params{};
    int K = 0;
    int64_t E = 0;
    int eb = 8;
    double h = 0.0;
    void* S1 = nullptr;
    void* S2 = nullptr;
    void* Uhost_dev = nullptr;   // device copy for dgw_rk_step_host
    double* partial = nullptr;   // mass partial sums
    double* mass_dev = nullptr;
    unsigned* flag = nullptr;
    double* t_dev = nullptr;     // the context's time (DGW_BC_STATE sides), advanced per step
    bool state_sides = false;
    int wait_limit = 0;          // bounded TMA waits: 0 the kernels' default limit (dgw_debug)
    int stage_kernel = 0;        // dgw_set_stage_kernel
    std::map<GraphKey, cudaGraphExec_t> graphs;
    std::map<std::pair<const void*, int>, CUtensorMap> tmaps;   // TMA descriptors (2D): (array, box kind)
    void* adj_ws = nullptr;      // adjoint: per-cell partials (own), K*E
    void* adj_wn = nullptr;      // adjoint: per-cell partials (one block per face), 2*dim*K*E
    void* adj_b1 = nullptr;      // adjoint: lambda of stage 2
    void* adj_b2 = nullptr;      // adjoint: lambda of stage 1
    std::map<std::pair<const void*, int>, bool> no_tmap;
    // dgw_rk_step_host pipeline: streams for input copies, output copies and each stage; one
    // event per (input copy or stage, band); the join events
    cudaStream_t band_st[2 + 3] = {};
    cudaEvent_t band_ev[4][16] = {};
    cudaEvent_t band_join[2] = {};
    std::map<BandKey, cudaGraphExec_t> band_graphs;   // null: replay not possible (direct launches)
};

static const int kBands = 16;
static const int kBandStreams = 2 + 3;

static const int kMassBlocks = 1024;
static const int kMassThreads = 256;

extern "C" void dgw_defaults(dgw_mesh* m, dgw_flux* f, dgw_params* s)
{
    if (m) {
        std::memset(m, 0, sizeof *m);
        m->dim = 1; m->nx = 16; m->ny = 1;
        m->x0 = 0.0; m->x1 = 1.0; m->y0 = 0.0; m->y1 = 1.0;
        for (int i = 0; i < 4; ++i) m->bc[i] = DGW_BC_PERIODIC;
    }
    if (f) {
        std::memset(f, 0, sizeof *f);
        f->kind = DGW_FLUX_ADVECT; f->a[0] = 1.0; f->a[1] = 0.0;
        f->center[0] = f->center[1] = 0.5; f->omega = 1.0; f->lambda_nu = 0.0; f->gas_gamma = 1.4;
    }
    if (s) {
        std::memset(s, 0, sizeof *s);
        s->stab = DGW_STAB_WENO; s->q = 1.0; s->b = 0.1; s->w_nbr = 1e-2;
        s->eps_w = 1e-6; s->eps_s = 1e-12; s->prec = DGW_FP64; s->theta = 1.0; s->rk_order = 3;
    }
}

static dgw_status check_params(const dgw_params* s, int dim)
{
    if (!s) return fail(DGW_EINVAL, "params is NULL");
    if (s->stab < DGW_STAB_DG || s->stab > DGW_STAB_ZHAO) return fail(DGW_EINVAL, "bad stab %d", s->stab);
    if (s->prec != DGW_FP64 && s->prec != DGW_FP32) return fail(DGW_EINVAL, "bad prec %d", s->prec);
    if (!(s->q > 0.0) || !std::isfinite(s->q)) return fail(DGW_EINVAL, "q must be > 0");
    if (!(s->b >= 0.0 && s->b <= 1.0)) return fail(DGW_EINVAL, "b must lie in [0, 1]");
    if (!(s->w_nbr >= 0.0 && s->w_nbr * 2 * dim < 1.0))
        return fail(DGW_EINVAL, "w_nbr must lie in [0, 1/(2 dim))");
    if (!(s->eps_w > 0.0) || !(s->eps_s >= 0.0)) return fail(DGW_EINVAL, "eps_w > 0 and eps_s >= 0 required");
    if (s->stab == DGW_STAB_ZHAO && !(s->w_nbr > 0.0 && s->theta > 0.0 && std::isfinite(s->theta)))
        return fail(DGW_EINVAL, "the ZHAO sensor needs w_nbr > 0 and a finite theta > 0");
    if (s->rk_order < 2 || s->rk_order > 4) return fail(DGW_EINVAL, "rk_order must be 2, 3 or 4");
    return DGW_OK;
}

extern "C" dgw_status dgw_create(const dgw_mesh* mesh, int p, const dgw_flux* flux,
                                 const dgw_params* params, dgw_ctx** out)
{
    if (!mesh || !flux || !params || !out) return fail(DGW_EINVAL, "NULL argument to dgw_create");
    *out = nullptr;
    const dgw_mesh& m = *mesh;
    if (m.dim != 1 && m.dim != 2) return fail(DGW_EINVAL, "dim must be 1 or 2");
    if (m.nx < 1 || (m.dim == 2 && m.ny < 1)) return fail(DGW_EINVAL, "nx, ny must be >= 1");
    if (!(m.x1 > m.x0) || (m.dim == 2 && !(m.y1 > m.y0))) return fail(DGW_EINVAL, "empty box");
    for (int f = 0; f < 2 * m.dim; ++f)
        if (m.bc[f] < DGW_BC_PERIODIC || m.bc[f] > DGW_BC_STATE) return fail(DGW_EINVAL, "bad bc[%d]", f);
    for (int a = 0; a < m.dim; ++a)
        if ((m.bc[2 * a] == DGW_BC_PERIODIC) != (m.bc[2 * a + 1] == DGW_BC_PERIODIC))
            return fail(DGW_EINVAL, "periodic sides must come in pairs");
    const double hx = (m.x1 - m.x0) / m.nx;
    if (m.dim == 2) {
        const double hy = (m.y1 - m.y0) / m.ny;
        if (std::fabs(hx - hy) > 1e-12 * hx) return fail(DGW_EUNSUPPORTED, "2D cells must be square");
    }
    if (p < 1 || p > kMaxP) return fail(DGW_EUNSUPPORTED, "degree p=%d not built (1..3)", p);
    if (flux->kind < DGW_FLUX_ADVECT || flux->kind > DGW_FLUX_EULER) return fail(DGW_EINVAL, "bad flux kind");
    if (!(flux->lambda_nu >= 0.0)) return fail(DGW_EINVAL, "lambda_nu must be >= 0");
    const bool euler = flux->kind == DGW_FLUX_EULER;
    bool state_sides = false;
    for (int f = 0; f < 2 * m.dim; ++f) {
        if (m.bc[f] == DGW_BC_REFLECT && !euler) return fail(DGW_EINVAL, "bc[%d]: reflecting walls are for the Euler system", f);
        if (m.bc[f] == DGW_BC_INFLOW_ZERO && euler) return fail(DGW_EINVAL, "bc[%d]: inflow_zero is for scalar laws", f);
        if (m.bc[f] == DGW_BC_STATE) {
            if (!euler || m.dim != 2) return fail(DGW_EUNSUPPORTED, "bc[%d]: prescribed states are built for the 2D Euler system", f);
            if (flux->bbelow[f] < 0 || flux->bbelow[f] > 2 || flux->babove[f] < 0 || flux->babove[f] > 2)
                return fail(DGW_EINVAL, "bc[%d]: bbelow / babove must be 0, 1 (a state) or 2 (a wall)", f);
            if (!std::isfinite(flux->bsplit[f]) || !std::isfinite(flux->bspeed[f]))
                return fail(DGW_EINVAL, "bc[%d]: bsplit and bspeed must be finite", f);
            state_sides = true;
        }
    }
    if (state_sides && params->rk_order == 4)
        return fail(DGW_EUNSUPPORTED, "prescribed states with rk_order 4: the stage times are built for orders 2 and 3");
    if (euler && !(flux->gas_gamma > 1.0 && std::isfinite(flux->gas_gamma)))
        return fail(DGW_EINVAL, "gas_gamma must be a finite number > 1");
    dgw_status st = check_params(params, m.dim);
    if (st != DGW_OK) return st;
    const int64_t E = m.dim == 1 ? (int64_t)m.nx : (int64_t)m.nx * m.ny;
    if (E > ((int64_t)1 << 36)) return fail(DGW_EINVAL, "mesh too large");

    dgw_ctx* c = new dgw_ctx();
    c->mesh = m;
    if (m.dim == 1) { c->mesh.ny = 1; }
    c->p = p;
    c->flux = *flux;
    c->params = *params;
    c->K = (m.dim == 1 ? p + 1 : (p + 1) * (p + 1)) * (euler ? m.dim + 2 : 1);
    c->E = E;
    c->eb = params->prec == DGW_FP64 ? 8 : 4;
    c->h = hx;
    cudaError_t ce = cudaGetDevice(&c->device);
    HostTables t;
    build_tables(p, &t);
    if (ce == cudaSuccess) {
        if (params->prec == DGW_FP64) ce = m.dim == 1 ? upload_tables_f64_d1(t) : upload_tables_f64_d2(t);
        else ce = m.dim == 1 ? upload_tables_f32_d1(t) : upload_tables_f32_d2(t);
    }
    const size_t bytes = (size_t)c->K * E * c->eb;
    if (ce == cudaSuccess) ce = cudaMalloc(&c->S1, bytes);
    if (ce == cudaSuccess) ce = cudaMalloc(&c->S2, bytes);
    if (ce == cudaSuccess) ce = cudaMalloc(&c->partial, sizeof(double) * (kMassBlocks + 2));
    if (ce == cudaSuccess) ce = cudaMemset(c->partial + kMassBlocks + 1, 0, sizeof(double));   // t = 0
    if (ce == cudaSuccess) ce = cudaMalloc(&c->flag, sizeof(unsigned));
    if (ce == cudaSuccess) ce = cudaMemset(c->flag, 0, sizeof(unsigned));
    if (ce != cudaSuccess) {
        dgw_status s = fail(ce == cudaErrorMemoryAllocation ? DGW_ENOMEM : DGW_ECUDA,
                            "dgw_create: %s", cudaGetErrorString(ce));
        dgw_destroy(c);
        return s;
    }
    c->mass_dev = c->partial + kMassBlocks;
    c->t_dev = c->partial + kMassBlocks + 1;
    c->state_sides = state_sides;
    *out = c;
    return DGW_OK;
}

static void drop_graphs(dgw_ctx* c)
{
    for (auto& kv : c->graphs) cudaGraphExecDestroy(kv.second);
    c->graphs.clear();
    for (auto& kv : c->band_graphs)
        if (kv.second) cudaGraphExecDestroy(kv.second);
    c->band_graphs.clear();
}

extern "C" dgw_status dgw_destroy(dgw_ctx* c)
{
    if (!c) return DGW_OK;
    cudaDeviceSynchronize();
    drop_graphs(c);
    cudaFree(c->S1);
    cudaFree(c->S2);
    cudaFree(c->Uhost_dev);
    cudaFree(c->adj_ws);
    cudaFree(c->adj_wn);
    cudaFree(c->adj_b1);
    cudaFree(c->adj_b2);
    cudaFree(c->partial);
    cudaFree(c->flag);
    for (int i = 0; i < kBandStreams; ++i)
        if (c->band_st[i]) cudaStreamDestroy(c->band_st[i]);
    for (int i = 0; i < 4; ++i)
        for (int b = 0; b < kBands; ++b)
            if (c->band_ev[i][b]) cudaEventDestroy(c->band_ev[i][b]);
    for (int i = 0; i < 2; ++i)
        if (c->band_join[i]) cudaEventDestroy(c->band_join[i]);
    delete c;
    return DGW_OK;
}

extern "C" dgw_status dgw_sizes(const dgw_ctx* c, int64_t* E, int* K, int* eb)
{
    if (!c) return fail(DGW_EINVAL, "NULL context");
    if (E) *E = c->E;
    if (K) *K = c->K;
    if (eb) *eb = c->eb;
    return DGW_OK;
}

extern "C" dgw_status dgw_set_params(dgw_ctx* c, const dgw_params* s)
{
    if (!c) return fail(DGW_EINVAL, "NULL context");
    dgw_status st = check_params(s, c->mesh.dim);
    if (st != DGW_OK) return st;
    if (s->prec != c->params.prec) return fail(DGW_EINVAL, "precision is fixed at dgw_create");
    if (c->state_sides && s->rk_order == 4)
        return fail(DGW_EUNSUPPORTED, "prescribed states with rk_order 4: the stage times are built for orders 2 and 3");
    c->params = *s;
    drop_graphs(c);
    return DGW_OK;
}

// TMA descriptor of a state array viewed as a 3D tensor (x: nx, y: ny, k: K) with a
// stage-tile box.  Null when TMA does not apply: 1D meshes, or row / plane strides that
// are not multiples of 16 bytes.
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// box kind 0: tile plus halo (kBoxX2 x (rows + 2) x K); 1: tile (kTileX2 x rows x K),
// rows = stage_rows() of the context's precision; kinds 2 and 3: the same with rows =
// kPRows (the persistent float kernel).  True and the descriptor in *out if TMA applies.  The descriptor is copied out: the cache evicts all its entries when it grows
// past 64 arrays, so a pointer into it would not outlive the next lookup.
static bool tensor_map(const dgw_ctx* cc, const void* U, int kind, CUtensorMap* out)
{
    dgw_ctx* c = const_cast<dgw_ctx*>(cc);
    if (c->mesh.dim != 2 || !U || c->flux.kind == DGW_FLUX_EULER) return false;   // the Euler kernel stages by plain loads
    const auto key = std::make_pair(U, kind);
    auto it = c->tmaps.find(key);
    if (it != c->tmaps.end()) {
        *out = it->second;
        return true;
    }
    if (c->no_tmap.count(key)) return false;
    if (c->tmaps.size() + c->no_tmap.size() > 64) {
        c->tmaps.clear();
        c->no_tmap.clear();
    }
    const uint64_t eb = (uint64_t)c->eb, nx = (uint64_t)c->mesh.nx, ny = (uint64_t)c->mesh.ny;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc || (nx * eb) % 16 || (nx * ny * eb) % 16 || ((uintptr_t)U & 15u)) {
        c->no_tmap[key] = true;
        return false;
    }
    cuuint64_t dims[3] = {nx, ny, (cuuint64_t)c->K};
    cuuint64_t strides[2] = {nx * eb, nx * ny * eb};
    const int rows = kind >= 2 ? kPRows : stage_rows(eb == 8);
    const bool halo = kind == 0 || kind == 2;
    cuuint32_t box[3] = {(cuuint32_t)(halo ? kBoxX2 : kTileX2), (cuuint32_t)(halo ? rows + 2 : rows),
                         (cuuint32_t)c->K};
    cuuint32_t estr[3] = {1, 1, 1};
    CUtensorMap m;
    CUresult r = enc(&m, eb == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                     const_cast<void*>(U), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        c->no_tmap[key] = true;
        return false;
    }
    c->tmaps[key] = m;
    *out = m;
    return true;
}

static StageArgs base_args(const dgw_ctx* c)
{
    StageArgs a;
    std::memset(&a, 0, sizeof a);
    a.E = c->E;
    a.nx = c->mesh.nx;
    a.ny = c->mesh.dim == 2 ? c->mesh.ny : 1;
    a.x0 = c->mesh.x0;
    a.y0 = c->mesh.y0;
    a.h = c->h;
    for (int f = 0; f < 4; ++f) a.bc[f] = c->mesh.bc[f];
    a.a0 = c->flux.a[0];
    a.a1 = c->flux.a[1];
    a.cx = c->flux.center[0];
    a.cy = c->flux.center[1];
    a.omega = c->flux.omega;
    a.lambda_nu = c->flux.lambda_nu;
    a.stab = c->params.stab;
    a.q = c->params.q;
    a.b = c->params.b;
    a.w_nbr = c->params.w_nbr;
    a.eps_w = c->params.eps_w;
    a.eps_s = c->params.eps_s;
    a.theta = c->params.theta;
    a.gas_gamma = c->flux.gas_gamma;
    a.flag = c->flag;
    a.wait_limit = c->wait_limit;
    a.kernel_choice = c->stage_kernel;
    a.t_dev = c->t_dev;
    a.t_off = 0.0;
    for (int i = 0; i < 2; ++i)
        for (int k = 0; k < 4; ++k) a.bstate[i][k] = c->flux.bstate[i][k];
    for (int f = 0; f < 4; ++f) {
        a.bsplit[f] = c->flux.bsplit[f];
        a.bspeed[f] = c->flux.bspeed[f];
        a.bbelow[f] = c->flux.bbelow[f];
        a.babove[f] = c->flux.babove[f];
    }
    return a;
}

// How a sequence of stages on s may overlap its launches (StageArgs.pdl)
static int pdl_mode(cudaStream_t s)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (s == nullptr || cudaStreamIsCapturing(s, &cap) != cudaSuccess) return kPdlDirect;
    return cap == cudaStreamCaptureStatusNone ? kPdlDirect : kPdlCaptured;
}

// t += dt on the device, after each step of a context with prescribed-state sides
__global__ void advance_time_kernel(double* t, double dt) { *t += dt; }

static cudaError_t launch(const dgw_ctx* c, const StageArgs& a0, int mode, cudaStream_t s)
{
    StageArgs a = a0;
    CUtensorMap m_k, m_n, m_pk, m_pn;      // copies: the launch parameters take them by value
    a.tmap = tensor_map(c, a.Uk, 0, &m_k) ? &m_k : nullptr;
    a.tmap_un = (a.cn != 0.0 && a.Un && tensor_map(c, a.Un, 1, &m_n)) ? &m_n : nullptr;
    const bool f64 = c->params.prec == DGW_FP64;
    a.tmap_p = a.tmap_un_p = nullptr;
    // whole-mesh float stage launches run the persistent kernel when its boxes apply
    // (the Un box too, where the stage reads Un)
    if (!f64 && c->mesh.dim == 2 && mode == 0 && a.kernel_choice != 1 && a.tile_row0 == 0 && a.tile_rows == 0 &&
        a.tmap && tensor_map(c, a.Uk, 2, &m_pk)) {
        const bool need_un = a.cn != 0.0 && a.Un;
        if (!need_un || (a.tmap_un && tensor_map(c, a.Un, 3, &m_pn))) {
            a.tmap_p = &m_pk;
            a.tmap_un_p = need_un ? &m_pn : nullptr;
        }
    }
    if (c->mesh.dim == 1)
        return f64 ? launch_stage_f64_d1(a, c->p, c->flux.kind, mode, s)
                   : launch_stage_f32_d1(a, c->p, c->flux.kind, mode, s);
    return f64 ? launch_stage_f64_d2(a, c->p, c->flux.kind, mode, s)
               : launch_stage_f32_d2(a, c->p, c->flux.kind, mode, s);
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

static dgw_status check_ctx(const dgw_ctx* c)
{
    if (!c) return fail(DGW_EINVAL, "NULL context");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != c->device)
        return fail(DGW_EINVAL, "context belongs to device %d, current device is %d", c->device, dev);
    return DGW_OK;
}

extern "C" dgw_status dgw_residual(dgw_ctx* c, const void* U, void* L, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !L) return fail(DGW_EINVAL, "NULL array");
    if (!aligned16(U) || !aligned16(L)) return fail(DGW_EINVAL, "arrays must be 16-byte aligned");
    if (U == L) return fail(DGW_EINVAL, "U and L must not overlap");
    StageArgs a = base_args(c);
    a.Uk = U;
    a.Uout = L;
    a.cn = 0.0; a.ck = 0.0; a.cl = 1.0;
    DGW_CUDA(launch(c, a, 0, (cudaStream_t)stream));
    return DGW_OK;
}

extern "C" dgw_status dgw_sensor(dgw_ctx* c, const void* U, double* gamma, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !gamma) return fail(DGW_EINVAL, "NULL array");
    if (!aligned16(U)) return fail(DGW_EINVAL, "U must be 16-byte aligned");
    StageArgs a = base_args(c);
    a.Uk = U;
    a.gamma_out = gamma;
    DGW_CUDA(launch(c, a, 1, (cudaStream_t)stream));
    return DGW_OK;
}

// The register recombination of the ten-stage SSP method of order 4:
// q2 <- q2/25 + 9/25 q1, then q1 <- 15 q2 - 5 q1 (with the new q2).
template <typename Real>
__global__ void rk4_mix_kernel(Real* __restrict__ q2, Real* __restrict__ q1, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const Real b = q2[i] / Real(25) + Real(9) / Real(25) * q1[i];
        q2[i] = b;
        q1[i] = Real(15) * b - Real(5) * q1[i];
    }
}

// SSP Runge-Kutta of order 2 and 4 (c->params.rk_order; Sec. 5 integrates with order
// p + 1).  Order 2: S1 = U + dt L(U); U <- 1/2 U + 1/2 (S1 + dt L(S1)).  Order 4 (the
// ten-stage method of Ketcheson): q2 lives in U, q1 alternates between S1 and S2;
// five stages q1 <- q1 + dt/6 L(q1), the recombination, four more, and
// U <- q2 + 3/5 q1 + dt/10 L(q1).  Final stages write U in place (own-element reads).
static cudaError_t enqueue_steps_rk24(const dgw_ctx* c, void* U, double dt, int nsteps, cudaStream_t s)
{
    StageArgs a = base_args(c);
    a.pdl = pdl_mode(s);
    for (int n = 0; n < nsteps; ++n) {
        if (c->params.rk_order == 2) {
            a.Uk = U; a.Un = nullptr; a.Uout = c->S1;
            a.cn = 0.0; a.ck = 1.0; a.cl = dt; a.t_off = 0.0;
            cudaError_t e = launch(c, a, 0, s);
            if (e != cudaSuccess) return e;
            a.Uk = c->S1; a.Un = U; a.Uout = U;
            a.cn = 0.5; a.ck = 0.5; a.cl = 0.5 * dt; a.t_off = dt;
            e = launch(c, a, 0, s);
            if (e != cudaSuccess) return e;
            if (c->state_sides) {
                advance_time_kernel<<<1, 1, 0, s>>>(c->t_dev, dt);
                e = cudaGetLastError();
                if (e != cudaSuccess) return e;
            }
            continue;
        }
        void* q[2] = {c->S1, c->S2};
        int cur = 0;                       // q1 is q[cur]
        a.Un = nullptr; a.cn = 0.0; a.ck = 1.0; a.cl = dt / 6.0;
        for (int k = 0; k < 9; ++k) {
            a.Uk = k == 0 ? U : q[cur];
            a.Uout = k == 0 ? q[0] : q[cur ^ 1];
            cudaError_t e = launch(c, a, 0, s);
            if (e != cudaSuccess) return e;
            if (k > 0) cur ^= 1;
            if (k == 4) {
                const int64_t N = (int64_t)c->K * c->E;
                const unsigned blocks = (unsigned)std::min<int64_t>((N + 255) / 256, 152 * 16);
                if (c->eb == 8) rk4_mix_kernel<double><<<blocks, 256, 0, s>>>((double*)U, (double*)q[cur], N);
                else rk4_mix_kernel<float><<<blocks, 256, 0, s>>>((float*)U, (float*)q[cur], N);
                e = cudaGetLastError();
                if (e != cudaSuccess) return e;
            }
        }
        a.Uk = q[cur]; a.Un = U; a.Uout = U;
        a.cn = 1.0; a.ck = 3.0 / 5.0; a.cl = dt / 10.0;
        cudaError_t e = launch(c, a, 0, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// 1D meshes that fit one thread-block cluster take all their steps in one launch
// (dgw_line_impl.cuh); nsteps = 0 asks whether c's does.
static cudaError_t line_steps(const dgw_ctx* c, void* U, double dt, int nsteps, cudaStream_t s)
{
    if (c->mesh.dim != 1) return cudaErrorNotSupported;
    const StageArgs a = base_args(c);
    return c->eb == 8 ? launch_line_f64_d1(a, c->p, c->flux.kind, U, dt, nsteps, c->params.rk_order, s)
                      : launch_line_f32_d1(a, c->p, c->flux.kind, U, dt, nsteps, c->params.rk_order, s);
}

// One SSP-RK3 step (Eq. ssp): U1 = U + dt L(U); U2 = 3/4 U + 1/4 (U1 + dt L(U1));
// U <- 1/3 U + 2/3 (U2 + dt L(U2)).  The third stage writes U in place: each thread
// reads U only at its own element there.  Other orders: enqueue_steps_rk24.
static cudaError_t enqueue_steps(const dgw_ctx* c, void* U, double dt, int nsteps, cudaStream_t s)
{
    const cudaError_t le = line_steps(c, U, dt, nsteps, s);
    if (le != cudaErrorNotSupported) return le;
    if (c->params.rk_order != 3) return enqueue_steps_rk24(c, U, dt, nsteps, s);
    StageArgs a = base_args(c);
    a.pdl = pdl_mode(s);
    for (int n = 0; n < nsteps; ++n) {
        a.Uk = U; a.Un = nullptr; a.Uout = c->S1;
        a.cn = 0.0; a.ck = 1.0; a.cl = dt; a.t_off = 0.0;
        cudaError_t e = launch(c, a, 0, s);
        if (e != cudaSuccess) return e;
        a.Uk = c->S1; a.Un = U; a.Uout = c->S2;
        a.cn = 0.75; a.ck = 0.25; a.cl = 0.25 * dt; a.t_off = dt;
        e = launch(c, a, 0, s);
        if (e != cudaSuccess) return e;
        a.Uk = c->S2; a.Un = U; a.Uout = U;
        a.cn = 1.0 / 3.0; a.ck = 2.0 / 3.0; a.cl = 2.0 / 3.0 * dt; a.t_off = 0.5 * dt;
        e = launch(c, a, 0, s);
        if (e != cudaSuccess) return e;
        if (c->state_sides) {
            advance_time_kernel<<<1, 1, 0, s>>>(c->t_dev, dt);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// One SSP-RK3 step from U that keeps its stage states; without U_next the third stage is left out.
// By the kernels of enqueue_steps, so the states have dgw_rk_step's bits.
static cudaError_t enqueue_stages(const dgw_ctx* c, const void* U, double dt, void* U1, void* U2, void* U_next, cudaStream_t s)
{
    StageArgs a = base_args(c);
    a.pdl = pdl_mode(s);
    auto stage = [&](const void* Uk, const void* Un, void* Uout, double cn, double ck, double cl) {
        a.Uk = Uk; a.Un = Un; a.Uout = Uout;
        a.cn = cn; a.ck = ck; a.cl = cl;
        if (c->mesh.dim == 1) {
            const cudaError_t e = c->eb == 8 ? launch_line_stage_f64_d1(a, c->p, c->flux.kind, s)
                                             : launch_line_stage_f32_d1(a, c->p, c->flux.kind, s);
            if (e != cudaErrorNotSupported) return e;
        }
        return launch(c, a, 0, s);
    };
    cudaError_t e = stage(U, nullptr, U1, 0.0, 1.0, dt);
    if (e == cudaSuccess) e = stage(U1, U, U2, 0.75, 0.25, 0.25 * dt);
    if (e == cudaSuccess && U_next) e = stage(U2, U, U_next, 1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0 * dt);
    return e;
}

static const int kGraphChunk = 16;

static dgw_status run_graph(dgw_ctx* c, void* U, double dt, int n, cudaStream_t s)
{
    GraphKey key{U, dt, n, s};
    auto it = c->graphs.find(key);
    cudaGraphExec_t exec = nullptr;
    if (it == c->graphs.end()) {
        if (c->graphs.size() >= 8) drop_graphs(c);
        cudaGraph_t g = nullptr;
        DGW_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
        cudaError_t e = enqueue_steps(c, U, dt, n, s);
        cudaError_t e2 = cudaStreamEndCapture(s, &g);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return fail(DGW_ECUDA, "graph capture failed: %s",
                        cudaGetErrorString(e != cudaSuccess ? e : e2));
        }
        e = cudaGraphInstantiate(&exec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return fail(DGW_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
        c->graphs[key] = exec;
    } else {
        exec = it->second;
    }
    DGW_CUDA(cudaGraphLaunch(exec, s));
    return DGW_OK;
}

extern "C" dgw_status dgw_rk_step(dgw_ctx* c, void* U, double dt, int nsteps, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U) return fail(DGW_EINVAL, "NULL state");
    if (!aligned16(U)) return fail(DGW_EINVAL, "U must be 16-byte aligned");
    if (nsteps < 0) return fail(DGW_EINVAL, "nsteps < 0");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    if (nsteps == 0) return DGW_OK;
    cudaStream_t s = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (s != nullptr) DGW_CUDA(cudaStreamIsCapturing(s, &cap));
    if (s == nullptr || cap != cudaStreamCaptureStatusNone || line_steps(c, U, dt, 0, s) == cudaSuccess) {
        DGW_CUDA(enqueue_steps(c, U, dt, nsteps, s));
        return DGW_OK;
    }
    const int full = nsteps / kGraphChunk, rest = nsteps % kGraphChunk;
    for (int i = 0; i < full; ++i) {
        st = run_graph(c, U, dt, kGraphChunk, s);
        if (st != DGW_OK) return st;
    }
    if (rest) return run_graph(c, U, dt, rest, s);
    return DGW_OK;
}

// One SSP-RK3 step of a 2D mesh that is not periodic in y, as a wavefront over bands of
// tile rows: stage r of band b reads stage r - 1 only on bands b - 1 .. b + 1.  So the input
// copy of a band, the three stages and the output copy of a finished band overlap.  Streams,
// each in the order of the bands: input copies, output copies, one per stage; one event per
// (input copy or stage, band); all joined to the caller's stream s at both ends.  As a stream
// keeps its order, a stage waits for the highest band that it reads alone.  (A pool of four
// streams per stage, each kernel waiting for three bands, was as fast replayed from a graph, 0.64
// ms for 1024^2 Q3; launched directly, as on the default stream, its 276 calls took 0.80 ms, these
// 0.67.)  copy_in: U_in (host) is copied to c->Uhost_dev band by band first; copy_out:
// the result is copied to U_out band by band.  Stage 3 writes U in place; the old U of band b is
// still read by stage 1 of bands b - 1 and b + 1 (halo rows) and by stages 2, 3 of band b (own
// rows): stage 3 of band b waits for stage 2 of the bands up to b + 1, which waited for stage 1
// of the bands up to b + 2.
static dgw_status banded_step(dgw_ctx* c, const void* U_in, void* U_out, double dt, bool copy_in,
                              bool copy_out, cudaStream_t s)
{
    const int rows = stage_rows(c->eb == 8);
    const int trows = (c->mesh.ny + rows - 1) / rows;
    // bands of 64 tiles or more: smaller ones leave the GPU idle and only queue behind each other
    // (187^2 Q1 FP32, three steps: 12 bands of 6 tiles 0.38 ms, one band 0.11)
    const int64_t tiles = (int64_t)trows * ((c->mesh.nx + kTileX2 - 1) / kTileX2);
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(tiles / 64, trows < kBands ? trows : kBands));
    cudaStream_t* st = c->band_st;
    cudaStream_t in_st = st[0], out_st = st[1];
    auto& ev = c->band_ev;
    DGW_CUDA(cudaEventRecord(c->band_join[0], s));
    for (int i = 0; i < kBandStreams; ++i) DGW_CUDA(cudaStreamWaitEvent(st[i], c->band_join[0], 0));

    int t0[kBands + 1];                 // band b: tile rows [t0[b], t0[b + 1])
    for (int b = 0; b <= nb; ++b) t0[b] = (int)((int64_t)trows * b / nb);
    const size_t eb = (size_t)c->eb, nx = (size_t)c->mesh.nx, pitch = (size_t)c->E * eb;
    auto row_span = [&](int b, size_t* off, size_t* width) {
        const int r0 = t0[b] * rows;
        const int r1 = t0[b + 1] * rows < c->mesh.ny ? t0[b + 1] * rows : c->mesh.ny;
        *off = (size_t)r0 * nx * eb;
        *width = (size_t)(r1 - r0) * nx * eb;
    };
    char* U = static_cast<char*>(c->Uhost_dev);
    if (copy_in)
        for (int b = 0; b < nb; ++b) {
            size_t off, width;
            row_span(b, &off, &width);
            DGW_CUDA(cudaMemcpy2DAsync(U + off, pitch, static_cast<const char*>(U_in) + off, pitch, width,
                                       (size_t)c->K, cudaMemcpyHostToDevice, in_st));
            DGW_CUDA(cudaEventRecord(ev[0][b], in_st));
        }
    StageArgs a = base_args(c);
    for (int r = 0; r < 3; ++r) {
        if (r == 0) { a.Uk = U; a.Un = nullptr; a.Uout = c->S1; a.cn = 0.0; a.ck = 1.0; a.cl = dt; }
        if (r == 1) { a.Uk = c->S1; a.Un = U; a.Uout = c->S2; a.cn = 0.75; a.ck = 0.25; a.cl = 0.25 * dt; }
        if (r == 2) { a.Uk = c->S2; a.Un = U; a.Uout = U; a.cn = 1.0 / 3.0; a.ck = 2.0 / 3.0; a.cl = 2.0 / 3.0 * dt; }
        for (int b = 0; b < nb; ++b) {
            cudaStream_t ks = st[2 + r];
            if (r > 0 || copy_in) DGW_CUDA(cudaStreamWaitEvent(ks, ev[r][b + 1 < nb ? b + 1 : nb - 1], 0));
            a.tile_row0 = t0[b];
            a.tile_rows = t0[b + 1] - t0[b];
            DGW_CUDA(launch(c, a, 0, ks));
            DGW_CUDA(cudaEventRecord(ev[1 + r][b], ks));
        }
    }
    if (copy_out) {
        for (int b = 0; b < nb; ++b) {
            size_t off, width;
            row_span(b, &off, &width);
            DGW_CUDA(cudaStreamWaitEvent(out_st, ev[3][b], 0));
            DGW_CUDA(cudaMemcpy2DAsync(static_cast<char*>(U_out) + off, pitch, U + off, pitch, width,
                                       (size_t)c->K, cudaMemcpyDeviceToHost, out_st));
        }
        // the last output copy comes after every other operation (each copy waited for its
        // band's stage 3, which waited for everything before it)
        DGW_CUDA(cudaEventRecord(c->band_join[1], out_st));
        DGW_CUDA(cudaStreamWaitEvent(s, c->band_join[1], 0));
    } else {
        DGW_CUDA(cudaStreamWaitEvent(s, ev[3][nb - 1], 0));
    }
    return DGW_OK;
}

static dgw_status band_resources(dgw_ctx* c)
{
    for (int i = 0; i < kBandStreams; ++i)
        if (!c->band_st[i]) DGW_CUDA(cudaStreamCreateWithFlags(&c->band_st[i], cudaStreamNonBlocking));
    for (int i = 0; i < 4; ++i)
        for (int b = 0; b < kBands; ++b)
            if (!c->band_ev[i][b]) DGW_CUDA(cudaEventCreateWithFlags(&c->band_ev[i][b], cudaEventDisableTiming));
    for (int i = 0; i < 2; ++i)
        if (!c->band_join[i]) DGW_CUDA(cudaEventCreateWithFlags(&c->band_join[i], cudaEventDisableTiming));
    return DGW_OK;
}

// banded_step, replayed from a graph cached per (U_in, U_out, dt, stream, copies) when the
// stream can be captured; launched directly otherwise (the legacy stream, a stream that is
// itself being captured, or host memory that a graph cannot copy from).
static dgw_status banded(dgw_ctx* c, const void* U_in, void* U_out, double dt, bool copy_in, bool copy_out,
                         cudaStream_t s)
{
    dgw_status st = band_resources(c);
    if (st != DGW_OK) return st;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (s != nullptr) DGW_CUDA(cudaStreamIsCapturing(s, &cap));
    if (s == nullptr || cap != cudaStreamCaptureStatusNone) return banded_step(c, U_in, U_out, dt, copy_in, copy_out, s);
    const BandKey key{U_in, U_out, dt, s, (copy_in ? 1 : 0) | (copy_out ? 2 : 0)};
    auto it = c->band_graphs.find(key);
    if (it == c->band_graphs.end()) {
        if (c->band_graphs.size() >= 8) {
            for (auto& kv : c->band_graphs)
                if (kv.second) cudaGraphExecDestroy(kv.second);
            c->band_graphs.clear();
        }
        cudaGraphExec_t exec = nullptr;
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            const dgw_status sc = banded_step(c, U_in, U_out, dt, copy_in, copy_out, s);
            const cudaError_t e = cudaStreamEndCapture(s, &g);
            if (sc == DGW_OK && e == cudaSuccess && g && cudaGraphInstantiate(&exec, g, 0) != cudaSuccess) exec = nullptr;
            if (g) cudaGraphDestroy(g);
        }
        cudaGetLastError();    // a refused capture leaves no error behind for later calls
        it = c->band_graphs.emplace(key, exec).first;
    }
    if (!it->second) return banded_step(c, U_in, U_out, dt, copy_in, copy_out, s);
    DGW_CUDA(cudaGraphLaunch(it->second, s));
    return DGW_OK;
}

extern "C" dgw_status dgw_rk_step_host(dgw_ctx* c, const void* U_in, void* U_out, double dt,
                                       int nsteps, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U_in || !U_out) return fail(DGW_EINVAL, "NULL host array");
    if (nsteps < 1) return fail(DGW_EINVAL, "nsteps < 1");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    const size_t bytes = (size_t)c->K * c->E * c->eb;
    if (!c->Uhost_dev) {
        cudaError_t e = cudaMalloc(&c->Uhost_dev, bytes);
        if (e != cudaSuccess) return fail(DGW_ENOMEM, "dgw_rk_step_host: %s", cudaGetErrorString(e));
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int rows = stage_rows(c->eb == 8);
    const bool pipelined = c->mesh.dim == 2 && c->mesh.bc[2] != DGW_BC_PERIODIC && c->mesh.ny >= 2 * rows &&
                           c->params.rk_order == 3 && c->flux.kind != DGW_FLUX_EULER;
    if (!pipelined) {
        DGW_CUDA(cudaMemcpyAsync(c->Uhost_dev, U_in, bytes, cudaMemcpyHostToDevice, s));
        st = dgw_rk_step(c, c->Uhost_dev, dt, nsteps, stream);
        if (st != DGW_OK) return st;
        DGW_CUDA(cudaMemcpyAsync(U_out, c->Uhost_dev, bytes, cudaMemcpyDeviceToHost, s));
    } else if (nsteps == 1) {
        st = banded(c, U_in, U_out, dt, true, true, s);
        if (st != DGW_OK) return st;
    } else {
        st = banded(c, U_in, nullptr, dt, true, false, s);
        if (st == DGW_OK && nsteps > 2) st = dgw_rk_step(c, c->Uhost_dev, dt, nsteps - 2, stream);
        if (st == DGW_OK) st = banded(c, nullptr, U_out, dt, false, true, s);
        if (st != DGW_OK) return st;
    }
    DGW_CUDA(cudaStreamSynchronize(s));
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// projection
// ------------------------------------------------------------------------------------
// L2 projection, one thread per cell: c_ij = minv_i minv_j sum_ab w_a w_b P_i(g_a) P_j(g_b) f_ab
// by sum factorisation, two sample rows (+-g_b) at a time, each sample read once.  On the
// symmetric Gauss nodes P_i(-g) = +-P_i(g), so sums over +-pairs halve the multiplications.
// Double states and 1D: the sums in double, 288 operations a cell at 8 x 8 samples and p = 3; the
// FP64 pipe (2 lanes per SM) bounds them, not memory.  Float states in 2D: project_fixed_kernel.
struct ProjArgs {
    const double* f;
    void* U;
    int64_t E;
    int f64;
    int vec;                        // sample rows start on 16-byte boundaries
    double WB[8][kMaxN1];           // w_q P_i(g_q)
    double minv[kMaxN1];
    int mh[8][kMaxN1], ml[8][kMaxN1];   // minv_i w_q P_i(g_q) 2^60 = mh 2^31 + ml
};

// out[i] = sum_q WB[q][i] f[q] on symmetric nodes
template <int NQ, int N1>
__device__ __forceinline__ void proj_sum(const double (&WB)[8][kMaxN1], const double (&f)[NQ], double (&out)[N1])
{
    constexpr int NP = NQ / 2;
    double S[NP > 0 ? NP : 1], D[NP > 0 ? NP : 1];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        S[m] = f[NQ - 1 - m] + f[m];
        D[m] = f[NQ - 1 - m] - f[m];
    }
#pragma unroll
    for (int i = 0; i < N1; ++i) {
        double a = 0.0;
        if ((NQ & 1) != 0 && (i & 1) == 0) a = WB[NQ / 2][i] * f[NQ / 2];
#pragma unroll
        for (int m = 0; m < NP; ++m) a = fma(WB[NQ - 1 - m][i], (i & 1) ? D[m] : S[m], a);
        out[i] = a;
    }
}

// Sample row b of a cell's NPT samples f
template <int NQ>
__device__ __forceinline__ void proj_row(const double* f, int b, bool vec, double (&r)[NQ])
{
    const double* src = f + b * NQ;
    if ((NQ & 1) == 0 && vec) {
#pragma unroll
        for (int q = 0; q + 1 < NQ; q += 2) {
            const double2 v = *reinterpret_cast<const double2*>(src + q);
            r[q] = v.x;
            r[q + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < NQ; ++q) r[q] = src[q];
    }
}

// The modes of cell e in double, stored in the state's precision
template <int DIM, int N1, int NQ>
__device__ void project_cell(const ProjArgs& a, const int64_t e)
{
    constexpr int NPT = DIM == 1 ? NQ : NQ * NQ, NP = NQ / 2, K = DIM == 1 ? N1 : N1 * N1;
    const double* f = a.f + e * NPT;
    double c[K];
    if constexpr (DIM == 1) {
        double r[NQ];
        proj_row<NQ>(f, 0, a.vec, r);
        proj_sum<NQ, N1>(a.WB, r, c);
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) c[k] = 0.0;
        if constexpr ((NQ & 1) != 0) {
            double r[NQ], s[N1];
            proj_row<NQ>(f, NQ / 2, a.vec, r);
            proj_sum<NQ, N1>(a.WB, r, s);
#pragma unroll
            for (int j = 0; j < N1; j += 2)
#pragma unroll
                for (int i = 0; i < N1; ++i) c[i + N1 * j] = a.WB[NQ / 2][j] * s[i];
        }
#pragma unroll
        for (int m = 0; m < NP; ++m) {
            double rm[NQ], rp[NQ], sm[N1], sp[N1];
            proj_row<NQ>(f, m, a.vec, rm);
            proj_row<NQ>(f, NQ - 1 - m, a.vec, rp);
            proj_sum<NQ, N1>(a.WB, rm, sm);
            proj_sum<NQ, N1>(a.WB, rp, sp);
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                const double S = sp[i] + sm[i], D = sp[i] - sm[i];
#pragma unroll
                for (int j = 0; j < N1; ++j)
                    c[i + N1 * j] = fma(a.WB[NQ - 1 - m][j], (j & 1) ? D : S, c[i + N1 * j]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double v = c[k] * (DIM == 1 ? a.minv[k] : a.minv[k % N1] * a.minv[k / N1]);
        if (a.f64) static_cast<double*>(a.U)[k * a.E + e] = v;
        else static_cast<float*>(a.U)[k * a.E + e] = (float)v;
    }
}

template <int DIM, int N1, int NQ>
__global__ void __launch_bounds__(128) project_kernel(const __grid_constant__ ProjArgs a)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < a.E) project_cell<DIM, N1, NQ>(a, e);
}

// Float states in 2D: the sums of project_cell in 64-bit fixed point, on integer multipliers that are
// several times as wide as the FP64 pipe.  Per cell the samples become integers of 59 bits (the unit from
// the largest exponent), the centre sample is taken off them, exactly, and the differences d are
// shifted up to 60 bits, so that all errors are relative to the cell's variation: fewer than
// five roundings of 2^-57 max |d| in a mode, where the double sums round by 2^-53 of the samples or of
// their differences.  The stored modes' error against 64 bits is the double sums' or less in every mode,
// on smooth data whose high modes cancel too (2 + sin cos on 64^2 to 1024^2 cells, p = 3, Kelvin-Helmholtz,
// KPP, cones, noise).  (The centre sample meets only the mean: rules of two points or more annihilate
// P_1 to P_3.)  Products take two limbs of 31 bits each: with x = xh 2^31 + xl and the weight M 2^60 =
// mh 2^31 + ml, M x = 4 sum mh xh + 2^-29 sum (mh xl + ml xh) but for one unit; |M| < 2, sum |M| < 2.7 and
// |x| < 2^61 keep every sum below 2^63.  Cells with samples that are not finite, or largest ones
// outside [2^-60, 2^100), take the sums in double.
// The samples arrive through shared memory, whole lines at a time; 65 words a cell keep the lanes
// that read one cell each on banks of their own.  1024^2 cells, p = 3, 8 x 8 samples, with the mass that
// follows: every sample read K times in double 4.53 ms, project_cell in double 0.73 ms, this 0.23 ms
// (604 MB would take 0.09 ms).  The kernel alone takes 160 us: 2860 instructions a cell, 576 of them
// 64-bit multiply-adds, issued in half of the slots by 12 warps per SM, which the samples in shared
// memory hold it to.  Multiply-adds written in C took twice the instructions of their pipe (230 us).
constexpr int kProjFixedThreads = 64;
__device__ __forceinline__ void proj_limbs(long long x, int& h, int& l)
{
    h = (int)(x >> 31);
    l = (int)((unsigned)x & 0x7fffffffu);
}
// A 2^62 + B 2^31 += (M x) 2^60
__device__ __forceinline__ void proj_mad(int mh, int ml, int h, int l, long long& A, long long& B)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(A) : "r"(mh), "r"(h));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(B) : "r"(mh), "r"(l));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(B) : "r"(ml), "r"(h));
}
// v as an integer multiple (rounded down in magnitude) of 2^(X - 1023 - 58), X the largest biased
// exponent of the cell
__device__ __forceinline__ long long proj_fixed(double v, int X)
{
    const int h = __double2hiint(v);
    const unsigned long long m = ((unsigned long long)((h & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
    const long long q = (long long)((m << 6) >> min(X - ((h >> 20) & 0x7ff), 63));
    return h < 0 ? -q : q;
}

template <int N1, int NQ>
__global__ void __launch_bounds__(kProjFixedThreads) project_fixed_kernel(const __grid_constant__ ProjArgs a)
{
    constexpr int NPT = NQ * NQ, ST = NPT | 1, NP = NQ / 2, NT = kProjFixedThreads;
    __shared__ double sm[NT * ST];
    const int64_t e0 = (int64_t)blockIdx.x * NT, e = e0 + threadIdx.x;
    const int n = (int)(a.E - e0 < NT ? a.E - e0 : NT);
    const double* src = a.f + e0 * NPT;
#pragma unroll 8
    for (int i = threadIdx.x; i < n * NPT; i += NT) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sm[i / NPT * ST + i % NPT]);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"(dst), "l"(src + i) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (e >= a.E) return;
    double* const f = sm + threadIdx.x * ST;
    long long* const d = reinterpret_cast<long long*>(f);
    float* const U = static_cast<float*>(a.U) + e;

    const double f0 = f[NQ / 2 * NQ + NQ / 2];
    const int h0 = __double2hiint(f0);
    // range of the upper words; one sign and exponent: they and all between share them
    unsigned least = h0, most = h0;
#pragma unroll
    for (int i = 0; i < NPT; ++i) {
        const unsigned h = (unsigned)__double2hiint(f[i]);
        least = min(least, h);
        most = max(most, h);
    }
    const bool same = ((least ^ most) >> 20) == 0;
    int top = (int)(most & 0x7fffffffu);     // largest |f|
    if (!same) {
        for (int i = 0; i < NPT; ++i) top = max(top, __double2hiint(f[i]) & 0x7fffffff);
    }
    const int X = top >> 20;
    if (X != 0 && (X < 1023 - 60 || X >= 1023 + 100)) {
        project_cell<2, N1, NQ>(a, e);
        return;
    }
    // d = x - base, x the words in shared memory, in units of 2^unit; of -f where neg
    long long base = 0;
    int unit = X - 1023 - 58, len;           // |d| <= 2^len
    bool neg = false, exact = true;
    if (same) {
        // the differences of the bits are those of the significands
        base = __double_as_longlong(f0);
        unit = X - 1023 - 52;
        neg = h0 < 0;
        const unsigned far = max(most - (unsigned)h0, (unsigned)h0 - least);
        exact = far == 0;                    // (the upper words do not tell)
        len = 64 - __clz(far);
    } else {
        const long long q0 = proj_fixed(f0, X);
#pragma unroll 8
        for (int i = 0; i < NPT; ++i) d[i] = proj_fixed(f[i], X) - q0;
    }
    if (exact) {
        long long mask = 0;
        for (int i = 0; i < NPT; ++i) {
            const long long q = d[i] - base;
            mask |= q ^ (q >> 63);
        }
        len = 64 - __clzll(mask);
    }
    if (len == 0 || X == 0) {                // a constant, or nothing but zeros and numbers below the normal ones
#pragma unroll
        for (int k = 0; k < N1 * N1; ++k) U[k * a.E] = k == 0 ? (float)f0 : 0.f;
        return;
    }
    const int up = 60 - len;
    using u64 = unsigned long long;
    auto get = [d](int i) { return (u64)d[i]; };

    long long A[N1][N1], B[N1][N1];
#pragma unroll
    for (int i = 0; i < N1; ++i)
#pragma unroll
        for (int j = 0; j < N1; ++j) A[i][j] = B[i][j] = 0;
    // quarters of the x-sums of row b
    auto row = [&](int b, long long (&r)[N1]) {
        long long ra[N1], rb[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) ra[i] = rb[i] = 0;
        if constexpr ((NQ & 1) != 0) {
            int h, l;
            proj_limbs((long long)((get(b * NQ + NP) - (u64)base) << up), h, l);
#pragma unroll
            for (int i = 0; i < N1; i += 2) proj_mad(a.mh[NP][i], a.ml[NP][i], h, l, ra[i], rb[i]);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int qp = NQ - 1 - q;
            const u64 x = get(b * NQ + qp), y = get(b * NQ + q);
            int sh, sl, dh, dl;
            proj_limbs((long long)((x + y - 2 * (u64)base) << up), sh, sl);
            proj_limbs((long long)((x - y) << up), dh, dl);
#pragma unroll
            for (int i = 0; i < N1; ++i) proj_mad(a.mh[qp][i], a.ml[qp][i], (i & 1) ? dh : sh, (i & 1) ? dl : sl, ra[i], rb[i]);
        }
#pragma unroll
        for (int i = 0; i < N1; ++i) r[i] = ra[i] + ((rb[i] + (1ll << 30)) >> 31);
    };
    if constexpr ((NQ & 1) != 0) {
        long long r[N1];
        row(NP, r);
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            int h, l;
            proj_limbs(r[i], h, l);
#pragma unroll
            for (int j = 0; j < N1; j += 2) proj_mad(a.mh[NP][j], a.ml[NP][j], h, l, A[i][j], B[i][j]);
        }
    }
#pragma unroll 1
    for (int m = 0; m < NP; ++m) {
        const int mp = NQ - 1 - m;
        long long rm[N1], rp[N1];
        row(m, rm);
        row(mp, rp);
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            int sh, sl, dh, dl;
            proj_limbs(rp[i] + rm[i], sh, sl);
            proj_limbs(rp[i] - rm[i], dh, dl);
#pragma unroll
            for (int j = 0; j < N1; ++j) proj_mad(a.mh[mp][j], a.ml[mp][j], (j & 1) ? dh : sh, (j & 1) ? dl : sl, A[i][j], B[i][j]);
        }
    }
    // a unit is 2^t; the mean adds the centre sample
    const int t = unit + 2 - up;
#pragma unroll
    for (int j = 0; j < N1; ++j)
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            long long R = 4 * A[i][j] + ((B[i][j] + (1ll << 28)) >> 29);
            if (neg) R = -R;
            float v;
            if (i + j == 0) v = (float)fma(__ll2double_rn(R), __hiloint2double((1023 + t) << 20, 0), f0);
            else v = __ll2float_rn(R) * __int_as_float((127 - 50) << 23) * __int_as_float((127 + 50 + t) << 23);
            U[(i + N1 * j) * a.E] = v;
        }
}

// Fills the tables for degree p and the nq-point Gauss rule (P_0..P_p by their recurrence).
static void project_tables(ProjArgs& a, int p, int nq)
{
    double x[8], w[8];
    gauss_rule_public(nq, x, w);
    // w_q P_i(g_q), and minv_i times it to 2^-60 from the exact product of the two doubles
    auto set = [&](int q, int i, double P) {
        a.WB[q][i] = w[q] * P;
        const double lo = std::fma(w[q], P, -a.WB[q][i]);
        const long long z = std::llrint(std::ldexp(a.WB[q][i], 60)) + std::llrint(std::ldexp(lo, 60));
        const long long M = ((2 * i + 1) * z + 1) >> 1;
        a.mh[q][i] = (int)((M + (1ll << 30)) >> 31);
        a.ml[q][i] = (int)(M - ((long long)a.mh[q][i] << 31));
    };
    for (int q = 0; q < nq; ++q) {
        double pm = 1.0, pc = x[q];
        set(q, 0, 1.0);
        set(q, 1, pc);
        for (int k = 1; k < p; ++k) {
            const double pn = ((2 * k + 1) * x[q] * pc - k * pm) / (k + 1);
            pm = pc; pc = pn;
            set(q, k + 1, pn);
        }
    }
    for (int i = 0; i <= p; ++i) a.minv[i] = (2 * i + 1) / 2.0;
}

template <int DIM, int N1, int NQ>
static void launch_project_q(const ProjArgs& a, unsigned blocks, cudaStream_t s)
{
    if constexpr (DIM == 2 && NQ >= 2) {     // (one point does not annihilate P_2)
        if (!a.f64) {
            project_fixed_kernel<N1, NQ><<<(unsigned)((a.E + kProjFixedThreads - 1) / kProjFixedThreads), kProjFixedThreads, 0, s>>>(a);
            return;
        }
    }
    project_kernel<DIM, N1, NQ><<<blocks, 128, 0, s>>>(a);
}

template <int DIM, int N1>
static void launch_project_n(const ProjArgs& a, int nq, unsigned blocks, cudaStream_t s)
{
    switch (nq) {
    case 1: launch_project_q<DIM, N1, 1>(a, blocks, s); break;
    case 2: launch_project_q<DIM, N1, 2>(a, blocks, s); break;
    case 3: launch_project_q<DIM, N1, 3>(a, blocks, s); break;
    case 4: launch_project_q<DIM, N1, 4>(a, blocks, s); break;
    case 5: launch_project_q<DIM, N1, 5>(a, blocks, s); break;
    case 6: launch_project_q<DIM, N1, 6>(a, blocks, s); break;
    case 7: launch_project_q<DIM, N1, 7>(a, blocks, s); break;
    default: launch_project_q<DIM, N1, 8>(a, blocks, s); break;
    }
}

// Samples f (E nq^dim, nq in 1..8) to the modes of degree p in U; a's tables are filled.
static cudaError_t launch_project(ProjArgs& a, const double* f, void* U, int64_t E, int dim, int p, int nq, cudaStream_t s)
{
    a.f = f; a.U = U; a.E = E;
    a.vec = ((uintptr_t)f & 15u) == 0;       // with nq even every row starts where f does, mod 16 bytes
    const unsigned blocks = (unsigned)((E + 127) / 128);
    if (dim == 1) {
        if (p == 1) launch_project_n<1, 2>(a, nq, blocks, s);
        else if (p == 2) launch_project_n<1, 3>(a, nq, blocks, s);
        else launch_project_n<1, 4>(a, nq, blocks, s);
    } else {
        if (p == 1) launch_project_n<2, 2>(a, nq, blocks, s);
        else if (p == 2) launch_project_n<2, 3>(a, nq, blocks, s);
        else launch_project_n<2, 4>(a, nq, blocks, s);
    }
    return cudaGetLastError();
}

extern "C" dgw_status dgw_project(dgw_ctx* c, int nq, const double* samples, void* U, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!samples || !U) return fail(DGW_EINVAL, "NULL array");
    if (nq < 1 || nq > 8) return fail(DGW_EINVAL, "nq must lie in 1..8");
    ProjArgs a;
    std::memset(&a, 0, sizeof a);
    project_tables(a, c->p, nq);
    a.f64 = c->params.prec == DGW_FP64;
    // the Euler system: one projection per component (samples and rows component-major)
    const int ncomp = c->flux.kind == DGW_FLUX_EULER ? c->mesh.dim + 2 : 1;
    const int64_t npt = c->mesh.dim == 1 ? nq : nq * nq;
    for (int comp = 0; comp < ncomp; ++comp)
        DGW_CUDA(launch_project(a, samples + comp * c->E * npt,
                                static_cast<char*>(U) + (size_t)comp * (c->K / ncomp) * c->E * c->eb, c->E, c->mesh.dim,
                                c->p, nq, (cudaStream_t)stream));
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// batched ensemble
// ------------------------------------------------------------------------------------
struct dgw_batch {
    int device = 0;
    int n = 0;
    dgw_params params{};
    int eb = 4;
    std::vector<BatchInst> inst;
    std::vector<int> dims;
    int64_t total = 0;
    BatchInst* d_inst = nullptr;
    // per group (dimension, degree): its work items, kernel tile height, items' chunk of
    // tiles, grid, and the stream its persistent kernel runs on
    BatchItem* d_items[2][kMaxP + 1] = {};
    int nitems[2][kMaxP + 1] = {};
    int rows[2][kMaxP + 1] = {};
    int chunk[2][kMaxP + 1] = {};
    int grid[2][kMaxP + 1] = {};
    void* S1 = nullptr;
    void* S2 = nullptr;
    unsigned long long* counters = nullptr;   // queue[kQueues], one per group, then done[n]
    unsigned* flag = nullptr;
    int* abort = nullptr;
    int sms = 0;
    long long wait_limit = 1ll << 24;
    int unreachable = 0;
    cudaStream_t st[2 * (kMaxP + 1)] = {};
    cudaEvent_t fork = nullptr;
    cudaEvent_t join[2 * (kMaxP + 1)] = {};
};

static const int kQueues = 2 * (kMaxP + 1);

static bool batch_group_used(const dgw_batch* b, int d, int p)
{
    for (int i = 0; i < b->n; ++i)
        if (b->dims[i] == d + 1 && b->inst[i].p == p) return true;
    return false;
}

static bool batch_rows_ok(const dgw_batch* b, int d, int rows)
{
    const bool f64 = b->eb == 8;
    return d == 0 ? (f64 ? batch_rows_built_f64_d1(rows) : batch_rows_built_f32_d1(rows))
                  : (f64 ? batch_rows_built_f64_d2(rows) : batch_rows_built_f32_d2(rows));
}

// Tiles of every instance of group (d, p) for the group's tile height, and the group's
// grid (resident CTAs per SM x SMs).  Uploads the instance table.
static dgw_status batch_layout(dgw_batch* b, int d, int p)
{
    const int rows = b->rows[d][p];
    for (int i = 0; i < b->n; ++i) {
        BatchInst& I = b->inst[i];
        if (b->dims[i] != d + 1 || I.p != p) continue;
        I.ntx = d == 0 ? (I.nx + 127) / 128 : (I.nx + kTileX2 - 1) / kTileX2;
        I.ntiles = d == 0 ? I.ntx : I.ntx * ((I.ny + rows - 1) / rows);
    }
    const bool f64 = b->eb == 8;
    const int bps = d == 0 ? (f64 ? batch_blocks_per_sm_f64_d1(p, rows) : batch_blocks_per_sm_f32_d1(p, rows))
                           : (f64 ? batch_blocks_per_sm_f64_d2(p, rows) : batch_blocks_per_sm_f32_d2(p, rows));
    if (bps <= 0) return fail(DGW_ECUDA, "batch kernel (dim %d, p %d, %d rows): occupancy query failed", d + 1, p, rows);
    b->grid[d][p] = bps * b->sms;
    DGW_CUDA(cudaMemcpy(b->d_inst, b->inst.data(), sizeof(BatchInst) * b->n, cudaMemcpyHostToDevice));
    return DGW_OK;
}

// Work items of group (d, p): chunks of the group's chunk size over each instance's
// tiles, longest instances first, so that the tail of each stage is made of small items.
static dgw_status batch_build_items(dgw_batch* b, int d, int p)
{
    std::vector<int> order;
    for (int i = 0; i < b->n; ++i)
        if (b->dims[i] == d + 1 && b->inst[i].p == p) order.push_back(i);
    std::stable_sort(order.begin(), order.end(),
                     [&](int x, int y) { return b->inst[x].ntiles > b->inst[y].ntiles; });
    const int c = b->chunk[d][p];
    std::vector<BatchItem> items;
    for (int i : order)
        for (int t = 0; t < b->inst[i].ntiles; t += c)
            items.push_back(BatchItem{i, t, std::min(c, b->inst[i].ntiles - t), 0});
    cudaFree(b->d_items[d][p]);
    b->d_items[d][p] = nullptr;
    b->nitems[d][p] = (int)items.size();
    if (!items.empty()) {
        DGW_CUDA(cudaMalloc(&b->d_items[d][p], sizeof(BatchItem) * items.size()));
        DGW_CUDA(cudaMemcpy(b->d_items[d][p], items.data(), sizeof(BatchItem) * items.size(),
                            cudaMemcpyHostToDevice));
    }
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_destroy(dgw_batch* b)
{
    if (!b) return DGW_OK;
    cudaDeviceSynchronize();
    cudaFree(b->d_inst);
    for (int d = 0; d < 2; ++d)
        for (int p = 0; p <= kMaxP; ++p) cudaFree(b->d_items[d][p]);
    cudaFree(b->S1);
    cudaFree(b->S2);
    cudaFree(b->counters);
    cudaFree(b->flag);
    cudaFree(b->abort);
    for (int g = 0; g < 2 * (kMaxP + 1); ++g) {
        if (b->st[g]) cudaStreamDestroy(b->st[g]);
        if (b->join[g]) cudaEventDestroy(b->join[g]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    delete b;
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_create(int n, const dgw_mesh* meshes, const int* ps, const dgw_flux* fluxes,
                                       const dgw_params* params, dgw_batch** out)
{
    if (!out || !meshes || !ps || !fluxes || !params || n < 1) return fail(DGW_EINVAL, "bad arguments to dgw_batch_create");
    *out = nullptr;
    dgw_status st = check_params(params, 2);
    if (params->rk_order != 3) return fail(DGW_EUNSUPPORTED, "the batch step is SSP-RK3 (rk_order 3)");
    if (st != DGW_OK) return st;
    std::vector<BatchInst> insts;
    std::vector<int> dims;
    int64_t off = 0;
    bool need_tab[2][2][kMaxP + 1] = {};
    const int eb = params->prec == DGW_FP64 ? 8 : 4;
    for (int i = 0; i < n; ++i) {
        const dgw_mesh& m = meshes[i];
        const int p = ps[i];
        const dgw_flux& f = fluxes[i];
        if (m.dim != 1 && m.dim != 2) return fail(DGW_EINVAL, "instance %d: dim must be 1 or 2", i);
        if (m.nx < 1 || (m.dim == 2 && m.ny < 1) || !(m.x1 > m.x0) || (m.dim == 2 && !(m.y1 > m.y0)))
            return fail(DGW_EINVAL, "instance %d: bad mesh", i);
        const double hx = (m.x1 - m.x0) / m.nx;
        if (m.dim == 2 && std::fabs(hx - (m.y1 - m.y0) / m.ny) > 1e-12 * hx)
            return fail(DGW_EUNSUPPORTED, "instance %d: 2D cells must be square", i);
        if (p < 1 || p > kMaxP) return fail(DGW_EUNSUPPORTED, "instance %d: degree %d not built", i, p);
        if (f.kind != DGW_FLUX_ADVECT && f.kind != DGW_FLUX_BURGERS)
            return fail(DGW_EUNSUPPORTED, "instance %d: the batched kernel is built for advection and Burgers", i);
        if (!(f.lambda_nu >= 0.0)) return fail(DGW_EINVAL, "instance %d: lambda_nu must be >= 0", i);
        for (int s = 0; s < 2 * m.dim; ++s)
            if (m.bc[s] < DGW_BC_PERIODIC || m.bc[s] > DGW_BC_OUTFLOW) return fail(DGW_EINVAL, "instance %d: bad bc", i);
        for (int a = 0; a < m.dim; ++a)
            if ((m.bc[2 * a] == DGW_BC_PERIODIC) != (m.bc[2 * a + 1] == DGW_BC_PERIODIC))
                return fail(DGW_EINVAL, "instance %d: periodic sides must come in pairs", i);
        BatchInst I;
        std::memset(&I, 0, sizeof I);
        I.nx = m.nx;
        I.ny = m.dim == 2 ? m.ny : 1;
        I.E = (int64_t)I.nx * I.ny;
        I.p = p;
        I.flux = f.kind;
        const int K = m.dim == 1 ? p + 1 : (p + 1) * (p + 1);
        for (int s = 0; s < 4; ++s) I.bc[s] = s < 2 * m.dim ? m.bc[s] : DGW_BC_PERIODIC;
        I.x0 = m.x0; I.y0 = m.y0; I.h = hx;
        I.a0 = f.a[0]; I.a1 = f.a[1]; I.cx = f.center[0]; I.cy = f.center[1];
        I.omega = f.omega; I.lambda_nu = f.lambda_nu; I.dt = 0.0;
        I.off = off;
        off += ((int64_t)K * I.E + 3) / 4 * 4;     // keep every instance 16-byte aligned
        insts.push_back(I);
        dims.push_back(m.dim);
        need_tab[eb == 8][m.dim - 1][p] = true;
    }
    dgw_batch* b = new dgw_batch();
    b->n = n;
    b->params = *params;
    b->eb = eb;
    b->inst = insts;
    b->dims = dims;
    b->total = off;
    cudaError_t ce = cudaGetDevice(&b->device);
    for (int f64 = 0; f64 < 2 && ce == cudaSuccess; ++f64)
        for (int d = 0; d < 2 && ce == cudaSuccess; ++d)
            for (int p = 1; p <= kMaxP && ce == cudaSuccess; ++p) {
                if (!need_tab[f64][d][p]) continue;
                HostTables t;
                build_tables(p, &t);
                ce = f64 ? (d == 0 ? upload_tables_f64_d1(t) : upload_tables_f64_d2(t))
                         : (d == 0 ? upload_tables_f32_d1(t) : upload_tables_f32_d2(t));
            }
    const size_t bytes = (size_t)b->total * b->eb;
    if (ce == cudaSuccess) ce = cudaMalloc(&b->S1, bytes);
    if (ce == cudaSuccess) ce = cudaMalloc(&b->S2, bytes);
    if (ce == cudaSuccess) ce = cudaMalloc(&b->counters, sizeof(unsigned long long) * (kQueues + n));
    if (ce == cudaSuccess) ce = cudaMalloc(&b->flag, sizeof(unsigned));
    if (ce == cudaSuccess) ce = cudaMemset(b->flag, 0, sizeof(unsigned));
    if (ce == cudaSuccess) ce = cudaMalloc(&b->abort, sizeof(int));
    if (ce == cudaSuccess) ce = cudaMalloc(&b->d_inst, sizeof(BatchInst) * n);
    if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    if (ce != cudaSuccess) {
        dgw_status s2 = fail(ce == cudaErrorMemoryAllocation ? DGW_ENOMEM : DGW_ECUDA, "dgw_batch_create: %s",
                             cudaGetErrorString(ce));
        dgw_batch_destroy(b);
        return s2;
    }
    for (int g = 0; g < 2 * (kMaxP + 1) && ce == cudaSuccess; ++g) {
        ce = cudaStreamCreateWithFlags(&b->st[g], cudaStreamNonBlocking);
        if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&b->join[g], cudaEventDisableTiming);
    }
    if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    if (ce != cudaSuccess) {
        dgw_batch_destroy(b);
        return fail(DGW_ECUDA, "dgw_batch_create: %s", cudaGetErrorString(ce));
    }
    for (int d = 0; d < 2 && st == DGW_OK; ++d)
        for (int p = 1; p <= kMaxP && st == DGW_OK; ++p) {
            // default schedule (the autotuner's usual pick with pipelined staging): 1D
            // items of 2 tiles; 2D float tiles of 8 cell rows, items of 16 tiles (p = 1, whose
            // tiles are the cheapest: 8, 1.5 % of a step of the ensemble of 512)
            const bool f64 = b->eb == 8;
            b->rows[d][p] = d == 0 ? 1 : (f64 ? kTileY2 : 8);
            b->chunk[d][p] = d == 0 ? 2 : (p == 1 && !f64 ? 8 : 16);
            if (!batch_group_used(b, d, p)) continue;
            st = batch_layout(b, d, p);
            if (st == DGW_OK) st = batch_build_items(b, d, p);
        }
    if (st != DGW_OK) {
        dgw_batch_destroy(b);
        return st;
    }
    *out = b;
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_sizes(const dgw_batch* b, int64_t* total, int64_t* offsets)
{
    if (!b) return fail(DGW_EINVAL, "NULL batch");
    if (total) *total = b->total;
    if (offsets)
        for (int i = 0; i < b->n; ++i) offsets[i] = b->inst[i].off;
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_set_dt(dgw_batch* b, const double* dt)
{
    if (!b || !dt) return fail(DGW_EINVAL, "NULL argument");
    for (int i = 0; i < b->n; ++i)
        if (!std::isfinite(dt[i]) || dt[i] == 0.0) return fail(DGW_EINVAL, "dt[%d] must be finite and nonzero", i);
    for (int i = 0; i < b->n; ++i) b->inst[i].dt = dt[i];
    DGW_CUDA(cudaMemcpy(b->d_inst, b->inst.data(), sizeof(BatchInst) * b->n, cudaMemcpyHostToDevice));
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_project(dgw_batch* b, int nq, int first, int count, const double* samples,
                                        void* U, void* stream)
{
    if (!b || !samples || !U) return fail(DGW_EINVAL, "NULL argument");
    if (nq < 1 || nq > 8) return fail(DGW_EINVAL, "nq must lie in 1..8");
    if (first < 0 || count < 0 || first + count > b->n) return fail(DGW_EINVAL, "instance range out of bounds");
    ProjArgs a;
    std::memset(&a, 0, sizeof a);
    a.f64 = b->eb == 8;
    int64_t so = 0;
    for (int i = first; i < first + count; ++i) {
        const BatchInst& I = b->inst[i];
        project_tables(a, I.p, nq);
        DGW_CUDA(launch_project(a, samples + so, static_cast<char*>(U) + (size_t)I.off * b->eb, I.E, b->dims[i], I.p,
                                nq, (cudaStream_t)stream));
        so += I.E * (b->dims[i] == 1 ? nq : nq * nq);
    }
    return DGW_OK;
}

// Launch of group (d, p)'s persistent kernel on stream s: it advances the group's
// instances through all 3 * nsteps stages.
static dgw_status batch_launch_group(dgw_batch* b, int d, int p, void* U, int nsteps, cudaStream_t s)
{
    BatchArgs a;
    std::memset(&a, 0, sizeof a);
    a.inst = b->d_inst;
    a.items = b->d_items[d][p];
    a.nitems = b->nitems[d][p];
    a.nstages = 3 * nsteps;
    a.U = U;
    a.S1 = b->S1;
    a.S2 = b->S2;
    a.queue = b->counters + d * (kMaxP + 1) + p;
    a.done = b->counters + kQueues;
    a.flag = b->flag;
    a.abort = b->abort;
    a.stab = b->params.stab;
    a.q = b->params.q; a.b = b->params.b; a.w_nbr = b->params.w_nbr;
    a.eps_w = b->params.eps_w; a.eps_s = b->params.eps_s; a.theta = b->params.theta;
    a.wait_limit = b->wait_limit;
    a.unreachable = b->unreachable;
    const bool f64 = b->eb == 8;
    const int rows = b->rows[d][p], g = b->grid[d][p];
    cudaError_t e = d == 0 ? (f64 ? launch_batch_f64_d1(a, p, rows, g, s) : launch_batch_f32_d1(a, p, rows, g, s))
                           : (f64 ? launch_batch_f64_d2(a, p, rows, g, s) : launch_batch_f32_d2(a, p, rows, g, s));
    if (e != cudaSuccess) return fail(DGW_ECUDA, "batch launch: %s", cudaGetErrorString(e));
    return DGW_OK;
}

// The persistent kernels of all groups (or of group `only` = d * (kMaxP + 1) + p) side by
// side: each on the batch's stream of its group, forked from s after the counters are
// cleared and joined back into s.  Groups with more DOFs start first; the others fill the
// SMs as its CTAs drain.
static dgw_status batch_enqueue(dgw_batch* b, void* U, int nsteps, cudaStream_t s, int only = -1)
{
    DGW_CUDA(cudaMemsetAsync(b->counters, 0, sizeof(unsigned long long) * (kQueues + b->n), s));
    DGW_CUDA(cudaMemsetAsync(b->abort, 0, sizeof(int), s));
    std::vector<std::pair<double, int>> groups;
    for (int d = 0; d < 2; ++d)
        for (int p = 1; p <= kMaxP; ++p) {
            const int gi = d * (kMaxP + 1) + p;
            if (b->nitems[d][p] == 0 || (only >= 0 && gi != only)) continue;
            double dofs = 0.0;
            for (int i = 0; i < b->n; ++i)
                if (b->dims[i] == d + 1 && b->inst[i].p == p)
                    dofs += (double)b->inst[i].E * (d == 0 ? p + 1 : (p + 1) * (p + 1));
            groups.push_back({-dofs, gi});
        }
    std::sort(groups.begin(), groups.end());
    DGW_CUDA(cudaEventRecord(b->fork, s));
    for (const auto& gr : groups) {
        const int gi = gr.second, d = gi / (kMaxP + 1), p = gi % (kMaxP + 1);
        DGW_CUDA(cudaStreamWaitEvent(b->st[gi], b->fork, 0));
        dgw_status st = batch_launch_group(b, d, p, U, nsteps, b->st[gi]);
        if (st != DGW_OK) return st;
        DGW_CUDA(cudaEventRecord(b->join[gi], b->st[gi]));
        DGW_CUDA(cudaStreamWaitEvent(s, b->join[gi], 0));
    }
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_rk_step(dgw_batch* b, void* U, int nsteps, void* stream)
{
    if (!b || !U) return fail(DGW_EINVAL, "NULL argument");
    if (nsteps < 0) return fail(DGW_EINVAL, "nsteps < 0");
    if (((uintptr_t)U & 15u) != 0) return fail(DGW_EINVAL, "U must be 16-byte aligned");
    if (nsteps == 0) return DGW_OK;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != b->device) return fail(DGW_EINVAL, "wrong device");
    for (int i = 0; i < b->n; ++i)
        if (b->inst[i].dt == 0.0) return fail(DGW_EINVAL, "dt not set (dgw_batch_set_dt)");
    return batch_enqueue(b, U, nsteps, (cudaStream_t)stream);
}

// For each group alone: time `steps` steps for every built tile height and every chunk of
// 1, 2, 4, 8, 16 tiles on a copy of U, and keep the fastest pair.
extern "C" dgw_status dgw_batch_autotune(dgw_batch* b, void* U, int steps, int* chosen_chunk, void* stream)
{
    if (!b || !U || steps < 1) return fail(DGW_EINVAL, "bad arguments");
    for (int i = 0; i < b->n; ++i)
        if (b->inst[i].dt == 0.0) return fail(DGW_EINVAL, "dt not set (dgw_batch_set_dt)");
    cudaStream_t s = (cudaStream_t)stream;
    void* tmp = nullptr;
    const size_t bytes = (size_t)b->total * b->eb;
    DGW_CUDA(cudaMalloc(&tmp, bytes));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int chunks[] = {1, 2, 4, 8, 16};
    const int heights[] = {1, 2, 4, 8};
    dgw_status st = DGW_OK;
    double best_dofs = -1.0;
    for (int d = 0; d < 2 && st == DGW_OK; ++d)
        for (int p = 1; p <= kMaxP && st == DGW_OK; ++p) {
            if (!batch_group_used(b, d, p)) continue;
            int best_rows = b->rows[d][p], best_chunk = b->chunk[d][p];
            float best_ms = 1e30f;
            for (int rows : heights) {
                if (!batch_rows_ok(b, d, rows)) continue;
                b->rows[d][p] = rows;
                st = batch_layout(b, d, p);
                for (int c : chunks) {
                    if (st != DGW_OK) break;
                    b->chunk[d][p] = c;
                    st = batch_build_items(b, d, p);
                    if (st != DGW_OK) break;
                    if (cudaMemcpyAsync(tmp, U, bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
                        st = fail(DGW_ECUDA, "copy");
                        break;
                    }
                    const int gi = d * (kMaxP + 1) + p;
                    st = batch_enqueue(b, tmp, 1, s, gi);    // warm-up
                    if (st != DGW_OK) break;
                    cudaEventRecord(e0, s);
                    st = batch_enqueue(b, tmp, steps, s, gi);
                    if (st != DGW_OK) break;
                    cudaEventRecord(e1, s);
                    cudaEventSynchronize(e1);
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    if (ms < best_ms) { best_ms = ms; best_rows = rows; best_chunk = c; }
                }
            }
            if (st != DGW_OK) break;
            b->rows[d][p] = best_rows;
            b->chunk[d][p] = best_chunk;
            st = batch_layout(b, d, p);
            if (st == DGW_OK) st = batch_build_items(b, d, p);
            double dofs = 0.0;
            for (int i = 0; i < b->n; ++i)
                if (b->dims[i] == d + 1 && b->inst[i].p == p) dofs += (double)b->inst[i].E;
            if (dofs > best_dofs && chosen_chunk) { best_dofs = dofs; *chosen_chunk = best_chunk; }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaStreamSynchronize(s);
    cudaFree(tmp);
    return st;
}

extern "C" dgw_status dgw_batch_schedule(const dgw_batch* b, int dim, int p, int* rows, int* chunk)
{
    if (!b || (dim != 1 && dim != 2) || p < 1 || p > kMaxP) return fail(DGW_EINVAL, "bad arguments");
    if (rows) *rows = b->rows[dim - 1][p];
    if (chunk) *chunk = b->chunk[dim - 1][p];
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_set_schedule(dgw_batch* b, int dim, int p, int rows, int chunk)
{
    if (!b || (dim != 1 && dim != 2) || p < 1 || p > kMaxP) return fail(DGW_EINVAL, "bad arguments");
    if (!batch_rows_ok(b, dim - 1, rows)) return fail(DGW_EINVAL, "tile height %d not built for dim %d", rows, dim);
    if (chunk < 1) return fail(DGW_EINVAL, "chunk must be >= 1");
    b->rows[dim - 1][p] = rows;
    b->chunk[dim - 1][p] = chunk;
    if (!batch_group_used(b, dim - 1, p)) return DGW_OK;
    dgw_status st = batch_layout(b, dim - 1, p);
    return st == DGW_OK ? batch_build_items(b, dim - 1, p) : st;
}

extern "C" dgw_status dgw_batch_sync_status(dgw_batch* b, void* stream)
{
    if (!b) return fail(DGW_EINVAL, "NULL batch");
    unsigned v = 0;
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(cudaMemcpyAsync(&v, b->flag, sizeof v, cudaMemcpyDeviceToHost, s));
    DGW_CUDA(cudaMemsetAsync(b->flag, 0, sizeof(unsigned), s));
    DGW_CUDA(cudaStreamSynchronize(s));
    if (v & 2u) return fail(DGW_ETIMEOUT, "a work item waited too long for its instance's previous stage");
    if (v & 1u) return fail(DGW_ENONFINITE, "a stage produced a non-finite value");
    return DGW_OK;
}

extern "C" dgw_status dgw_batch_debug(dgw_batch* b, long long wait_limit, int unreachable)
{
    if (!b || wait_limit < 1) return fail(DGW_EINVAL, "bad arguments");
    b->wait_limit = wait_limit;
    b->unreachable = unreachable ? 1 : 0;
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// mass: sum_e |K_e| c_0^e by a fixed-order two-level tree
// ------------------------------------------------------------------------------------
template <typename Real>
__global__ void mass_partial_kernel(const Real* U0, int64_t E, double* partial)
{
    __shared__ double sh[kMassThreads];
    double s = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
         e += (int64_t)gridDim.x * blockDim.x)
        s += (double)U0[e];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void mass_final_kernel(const double* partial, int n, double vol, double* out)
{
    __shared__ double sh[kMassThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += partial[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0] * vol;
}

extern "C" dgw_status dgw_mass(dgw_ctx* c, const void* U, double* host_mass, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !host_mass) return fail(DGW_EINVAL, "NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    const double vol = c->mesh.dim == 1 ? c->h : c->h * c->h;
    if (c->params.prec == DGW_FP64)
        mass_partial_kernel<double><<<kMassBlocks, kMassThreads, 0, s>>>((const double*)U, c->E, c->partial);
    else
        mass_partial_kernel<float><<<kMassBlocks, kMassThreads, 0, s>>>((const float*)U, c->E, c->partial);
    DGW_CUDA(cudaGetLastError());
    mass_final_kernel<<<1, kMassThreads, 0, s>>>(c->partial, kMassBlocks, vol, c->mass_dev);
    DGW_CUDA(cudaGetLastError());
    DGW_CUDA(cudaMemcpyAsync(host_mass, c->mass_dev, sizeof(double), cudaMemcpyDeviceToHost, s));
    DGW_CUDA(cudaStreamSynchronize(s));
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// discrete adjoint
// ------------------------------------------------------------------------------------
static dgw_status adjoint_ready(dgw_ctx* c)
{
    for (int f = 0; f < 2 * c->mesh.dim; ++f)
        if (c->mesh.bc[f] != DGW_BC_PERIODIC)
            return fail(DGW_EUNSUPPORTED, "the adjoint is built for periodic meshes");
    if (c->flux.kind != DGW_FLUX_ADVECT && c->flux.kind != DGW_FLUX_BURGERS)
        return fail(DGW_EUNSUPPORTED, "the adjoint is built for the advection and Burgers fluxes");
    if (c->params.stab == DGW_STAB_ZHAO)
        return fail(DGW_EUNSUPPORTED, "the adjoint differentiates the DG, LO and WENO stabilizations");
    const size_t bytes = (size_t)c->K * c->E * c->eb;
    cudaError_t e = cudaSuccess;
    if (!c->adj_ws) e = cudaMalloc(&c->adj_ws, bytes);
    if (e == cudaSuccess && !c->adj_wn) e = cudaMalloc(&c->adj_wn, bytes * 2 * c->mesh.dim);
    if (e == cudaSuccess && !c->adj_b1) e = cudaMalloc(&c->adj_b1, bytes);
    if (e == cudaSuccess && !c->adj_b2) e = cudaMalloc(&c->adj_b2, bytes);
    if (e != cudaSuccess) return fail(DGW_ENOMEM, "adjoint buffers: %s", cudaGetErrorString(e));
    return DGW_OK;
}

// out = c0 x0 + c1 x1 + c2 x2 + cv J_L(U)^T lam
static cudaError_t vjp_combine(const dgw_ctx* c, const void* U, const void* lam, const void* x0, double c0,
                               const void* x1, double c1, const void* x2, double c2, double cv, void* out,
                               cudaStream_t s)
{
    StageArgs a = base_args(c);
    const bool f64 = c->params.prec == DGW_FP64;
    a.pdl = f64 ? kPdlCaptured : pdl_mode(s);
    a.Uk = U;
    const int d = c->mesh.dim;
    cudaError_t e = f64 ? (d == 1 ? launch_vjp_f64_d1(a, c->p, c->flux.kind, lam, c->adj_ws, c->adj_wn, s)
                                  : launch_vjp_f64_d2(a, c->p, c->flux.kind, lam, c->adj_ws, c->adj_wn, s))
                        : (d == 1 ? launch_vjp_f32_d1(a, c->p, c->flux.kind, lam, c->adj_ws, c->adj_wn, s)
                                  : launch_vjp_f32_d2(a, c->p, c->flux.kind, lam, c->adj_ws, c->adj_wn, s));
    if (e != cudaSuccess) return e;
    GatherArgs g;
    std::memset(&g, 0, sizeof g);
    g.E = c->E; g.nx = c->mesh.nx; g.ny = d == 2 ? c->mesh.ny : 1;
    g.wself = c->adj_ws; g.wnb = c->adj_wn;
    g.x[0] = x0; g.x[1] = x1; g.x[2] = x2;
    g.coef[0] = c0; g.coef[1] = c1; g.coef[2] = c2;
    g.cvjp = cv;
    g.out = out;
    g.pdl = a.pdl;
    return f64 ? (d == 1 ? launch_gather_f64_d1(g, c->p, s) : launch_gather_f64_d2(g, c->p, s))
               : (d == 1 ? launch_gather_f32_d1(g, c->p, s) : launch_gather_f32_d2(g, c->p, s));
}

extern "C" dgw_status dgw_residual_vjp(dgw_ctx* c, const void* U, const void* lam, void* out, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !lam || !out) return fail(DGW_EINVAL, "NULL array");
    if (out == U || out == lam) return fail(DGW_EINVAL, "out must not overlap U or lam");
    st = adjoint_ready(c);
    if (st != DGW_OK) return st;
    DGW_CUDA(vjp_combine(c, U, lam, nullptr, 0.0, nullptr, 0.0, nullptr, 0.0, 1.0, out, (cudaStream_t)stream));
    return DGW_OK;
}

// Reverse of one SSP-RK3 step (Eq. ssp).  With a = lam^{n+1}:
//   lam_U2 = 2/3 a + 2/3 dt J_L(U2)^T a
//   lam_U1 = 1/4 lam_U2 + 1/4 dt J_L(U1)^T lam_U2
//   lam^n  = 1/3 a + 3/4 lam_U2 + lam_U1 + dt J_L(U^n)^T lam_U1
// where U1, U2 are recomputed from U^n.
extern "C" dgw_status dgw_adjoint_step(dgw_ctx* c, const void* U_n, const void* lam_np1, void* lam_n,
                                       double dt, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U_n || !lam_np1 || !lam_n) return fail(DGW_EINVAL, "NULL array");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    if (c->params.rk_order != 3)
        return fail(DGW_EUNSUPPORTED, "the adjoint step reverses the SSP-RK3 step (rk_order 3)");
    st = adjoint_ready(c);
    if (st != DGW_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(enqueue_stages(c, U_n, dt, c->S1, c->S2, nullptr, s));
    DGW_CUDA(vjp_combine(c, c->S2, lam_np1, lam_np1, 2.0 / 3.0, nullptr, 0.0, nullptr, 0.0, 2.0 / 3.0 * dt,
                         c->adj_b1, s));
    DGW_CUDA(vjp_combine(c, c->S1, c->adj_b1, c->adj_b1, 0.25, nullptr, 0.0, nullptr, 0.0, 0.25 * dt,
                         c->adj_b2, s));
    DGW_CUDA(vjp_combine(c, U_n, c->adj_b2, lam_np1, 1.0 / 3.0, c->adj_b1, 0.75, c->adj_b2, 1.0, dt, lam_n, s));
    return DGW_OK;
}

extern "C" dgw_status dgw_rk_step_stages(dgw_ctx* c, const void* U, double dt, void* U1, void* U2, void* U_next,
                                         void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !U1 || !U2) return fail(DGW_EINVAL, "NULL array");
    if (!aligned16(U) || !aligned16(U1) || !aligned16(U2) || (U_next && !aligned16(U_next)))
        return fail(DGW_EINVAL, "arrays must be 16-byte aligned");
    if (U1 == U || U2 == U || U1 == U2 || U_next == U1 || U_next == U2)
        return fail(DGW_EINVAL, "the stage states must not overlap U, U_next or each other");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    if (c->params.rk_order != 3) return fail(DGW_EUNSUPPORTED, "stage states of the SSP-RK3 step (rk_order 3)");
    if (c->state_sides) return fail(DGW_EUNSUPPORTED, "dgw_rk_step_stages keeps no time (prescribed-state sides)");
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(enqueue_stages(c, U, dt, U1, U2, U_next, s));
    return DGW_OK;
}

extern "C" dgw_status dgw_adjoint_step_stages(dgw_ctx* c, const void* U_n, const void* U1, const void* U2,
                                              const void* lam_np1, void* lam_n, double dt, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U_n || !U1 || !U2 || !lam_np1 || !lam_n) return fail(DGW_EINVAL, "NULL array");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    if (c->params.rk_order != 3)
        return fail(DGW_EUNSUPPORTED, "the adjoint step reverses the SSP-RK3 step (rk_order 3)");
    st = adjoint_ready(c);
    if (st != DGW_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(vjp_combine(c, U2, lam_np1, lam_np1, 2.0 / 3.0, nullptr, 0.0, nullptr, 0.0, 2.0 / 3.0 * dt,
                         c->adj_b1, s));
    DGW_CUDA(vjp_combine(c, U1, c->adj_b1, c->adj_b1, 0.25, nullptr, 0.0, nullptr, 0.0, 0.25 * dt,
                         c->adj_b2, s));
    DGW_CUDA(vjp_combine(c, U_n, c->adj_b2, lam_np1, 1.0 / 3.0, c->adj_b1, 0.75, c->adj_b2, 1.0, dt, lam_n, s));
    return DGW_OK;
}

// Mass of every mode of a cell, int phi_k^2 (a table: its divisions, done per coefficient, held the
// FP64 pipe for most of the kernel's 128 us on 512^2 Q2 cells)
struct MassTable {
    double m[4 * kMaxK];
};

template <typename Real, int K>
__global__ void misfit_kernel(const Real* U, const Real* Ut, Real* grad, int64_t E,
                              const __grid_constant__ MassTable t, double* partial)
{
    __shared__ double sh[kMassThreads];
    double s = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
        Real u[K], ut[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            u[k] = U[k * E + e];
            ut[k] = Ut[k * E + e];
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double d = (double)u[k] - (double)ut[k], md = t.m[k] * d;
            s = fma(0.5 * md, d, s);
            if (grad) grad[k * E + e] = (Real)md;
        }
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

extern "C" dgw_status dgw_misfit(dgw_ctx* c, const void* U, const void* U_target, double* host_J, void* grad,
                                 void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!U || !U_target || !host_J) return fail(DGW_EINVAL, "NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    MassTable t;
    const int n1 = c->p + 1;
    for (int k = 0; k < c->K; ++k) {
        t.m[k] = 0.5 * c->h * 2.0 / (2 * (k % n1) + 1);                             // mass of P_i on a cell of width h
        if (c->mesh.dim == 2) t.m[k] *= 0.5 * c->h * 2.0 / (2 * (k / n1 % n1) + 1);  // n1 n1 rows a component
    }
    auto run = [&](auto kc) {
        constexpr int kK = decltype(kc)::value;
        if (c->params.prec == DGW_FP64)
            misfit_kernel<double, kK><<<kMassBlocks, kMassThreads, 0, s>>>((const double*)U, (const double*)U_target,
                                                                           (double*)grad, c->E, t, c->partial);
        else
            misfit_kernel<float, kK><<<kMassBlocks, kMassThreads, 0, s>>>((const float*)U, (const float*)U_target,
                                                                          (float*)grad, c->E, t, c->partial);
    };
    switch (c->K) {            // (p + 1)^dim times the components
    case 2: run(std::integral_constant<int, 2>()); break;
    case 3: run(std::integral_constant<int, 3>()); break;
    case 4: run(std::integral_constant<int, 4>()); break;
    case 6: run(std::integral_constant<int, 6>()); break;
    case 9: run(std::integral_constant<int, 9>()); break;
    case 12: run(std::integral_constant<int, 12>()); break;
    case 16: run(std::integral_constant<int, 16>()); break;
    case 36: run(std::integral_constant<int, 36>()); break;
    default: run(std::integral_constant<int, 64>()); break;
    }
    DGW_CUDA(cudaGetLastError());
    mass_final_kernel<<<1, kMassThreads, 0, s>>>(c->partial, kMassBlocks, 1.0, c->mass_dev);
    DGW_CUDA(cudaGetLastError());
    DGW_CUDA(cudaMemcpyAsync(host_J, c->mass_dev, sizeof(double), cudaMemcpyDeviceToHost, s));
    DGW_CUDA(cudaStreamSynchronize(s));
    return DGW_OK;
}

extern "C" dgw_status dgw_sync_status(dgw_ctx* c, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    unsigned v = 0;
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(cudaMemcpyAsync(&v, c->flag, sizeof v, cudaMemcpyDeviceToHost, s));
    DGW_CUDA(cudaMemsetAsync(c->flag, 0, sizeof(unsigned), s));
    DGW_CUDA(cudaStreamSynchronize(s));
    if (v & 2u) return fail(DGW_ETIMEOUT, "a stage kernel's bounded wait for its TMA copy gave up (its tile was skipped)");
    if (v & 1u) return fail(DGW_ENONFINITE, "a stage produced a non-finite value");
    return DGW_OK;
}

extern "C" dgw_status dgw_set_time(dgw_ctx* c, double t, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!std::isfinite(t)) return fail(DGW_EINVAL, "t must be finite");
    cudaStream_t s = (cudaStream_t)stream;
    static thread_local double host_t;       // pageable source: the copy reads it before returning
    host_t = t;
    DGW_CUDA(cudaMemcpyAsync(c->t_dev, &host_t, sizeof(double), cudaMemcpyHostToDevice, s));
    DGW_CUDA(cudaStreamSynchronize(s));
    return DGW_OK;
}

extern "C" dgw_status dgw_get_time(dgw_ctx* c, double* t, void* stream)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (!t) return fail(DGW_EINVAL, "NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    DGW_CUDA(cudaMemcpyAsync(t, c->t_dev, sizeof(double), cudaMemcpyDeviceToHost, s));
    DGW_CUDA(cudaStreamSynchronize(s));
    return DGW_OK;
}

extern "C" dgw_status dgw_debug(dgw_ctx* c, int wait_limit)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    c->wait_limit = wait_limit;
    drop_graphs(c);          // the cached graphs hold the old launch parameters
    return DGW_OK;
}

extern "C" dgw_status dgw_set_stage_kernel(dgw_ctx* c, int choice)
{
    dgw_status st = check_ctx(c);
    if (st != DGW_OK) return st;
    if (choice < 0 || choice > 2) return fail(DGW_EINVAL, "stage kernel choice %d (0, 1 or 2)", choice);
    c->stage_kernel = choice;
    drop_graphs(c);          // the cached graphs hold the old kernels
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// self-test of the float sin/cos used by the KPP flux
// ------------------------------------------------------------------------------------
__global__ void sincos_selftest_kernel(const float* x, float* s, float* c, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dgw::fast_sincos(x[i], &s[i], &c[i]);
}

extern "C" dgw_status dgw_selftest_sincos(const float* x, float* s, float* c, int64_t n, void* stream)
{
    if (!x || !s || !c || n < 0) return fail(DGW_EINVAL, "bad arguments");
    if (n == 0) return DGW_OK;
    const int threads = 256;
    sincos_selftest_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(x, s, c, n);
    DGW_CUDA(cudaGetLastError());
    return DGW_OK;
}

extern "C" dgw_status dgw_selftest_tc_volume(const float* U, float* out, int64_t ntiles, int variant, float* ms,
                                             void* stream)
{
    if (!U || !out || ntiles < 0 || (variant != 0 && variant != 1)) return fail(DGW_EINVAL, "bad arguments");
    if (((uintptr_t)U & 15u) || ((uintptr_t)out & 15u)) return fail(DGW_EINVAL, "arrays must be 16-byte aligned");
    if (ntiles == 0) return DGW_OK;
    static std::mutex mu;
    static std::set<int> ready;                 // devices with the degree-3 float 2D tables
    int dev = -1;
    DGW_CUDA(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!ready.count(dev)) {
            HostTables t;
            build_tables(3, &t);
            DGW_CUDA(upload_tables_f32_d2(t));
            ready.insert(dev);
        }
    }
    unsigned* flag = nullptr;
    DGW_CUDA(cudaMalloc(&flag, sizeof(unsigned)));
    cudaError_t e = cudaMemset(flag, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = launch_tc_volume_f32_d2(U, out, ntiles, variant, flag, ms, (cudaStream_t)stream);
    unsigned v = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&v, flag, sizeof v, cudaMemcpyDeviceToHost);
    cudaFree(flag);
    if (e != cudaSuccess) return fail(DGW_ECUDA, "tensor-core volume probe: %s", cudaGetErrorString(e));
    if (v & 2u) return fail(DGW_ETIMEOUT, "tensor-core volume probe: a bounded wait for the MMAs gave up");
    return DGW_OK;
}

// ------------------------------------------------------------------------------------
// SSP-RK3 steps without any device allocation
// ------------------------------------------------------------------------------------
// Some callers cannot call cudaMalloc: applications whose device memory is all owned by
// another allocator, and real-time code that allows no allocation after start-up (an
// allocation can block or fail at an arbitrary point).  dgw_rk_step_noalloc serves them:
// instead of a context's
// stage buffers it keeps the two SSP-RK3 stage states in this fixed array, which every
// GPU that loads the library holds until the process exits.  Layout: stage 1, stage 2
// (kNoAllocStageBytes each), then the kernels' error flag.  Nothing in it has to start
// at zero: each stage buffer is written in full before it is read, and the flag is
// only ever set.
static const size_t kNoAllocStageBytes = (size_t)8 << 20;   // 8 MiB per stage state
static __device__ __align__(256) unsigned char g_noalloc_scratch[2 * kNoAllocStageBytes + 256];

static std::mutex g_noalloc_mu;
static std::map<int, unsigned char*> g_noalloc_addr;        // device -> array address
static std::set<std::tuple<int, int, int, int>> g_noalloc_tables;   // device, prec, dim, p

extern "C" dgw_status dgw_rk_step_noalloc(const dgw_mesh* mesh, int p, const dgw_flux* flux,
                                          const dgw_params* params, void* U, double dt,
                                          int nsteps, void* stream)
{
    if (!mesh || !flux || !params || !U) return fail(DGW_EINVAL, "NULL argument to dgw_rk_step_noalloc");
    const dgw_mesh& m = *mesh;
    if (m.dim != 1 && m.dim != 2) return fail(DGW_EINVAL, "dim must be 1 or 2");
    if (m.nx < 1 || (m.dim == 2 && m.ny < 1)) return fail(DGW_EINVAL, "nx, ny must be >= 1");
    if (!(m.x1 > m.x0) || (m.dim == 2 && !(m.y1 > m.y0))) return fail(DGW_EINVAL, "empty box");
    for (int f = 0; f < 2 * m.dim; ++f)
        if (m.bc[f] < DGW_BC_PERIODIC || m.bc[f] > DGW_BC_OUTFLOW) return fail(DGW_EINVAL, "bad bc[%d]", f);
    for (int a = 0; a < m.dim; ++a)
        if ((m.bc[2 * a] == DGW_BC_PERIODIC) != (m.bc[2 * a + 1] == DGW_BC_PERIODIC))
            return fail(DGW_EINVAL, "periodic sides must come in pairs");
    const double hx = (m.x1 - m.x0) / m.nx;
    if (m.dim == 2 && std::fabs(hx - (m.y1 - m.y0) / m.ny) > 1e-12 * hx)
        return fail(DGW_EUNSUPPORTED, "2D cells must be square");
    if (p < 1 || p > kMaxP) return fail(DGW_EUNSUPPORTED, "degree p=%d not built (1..3)", p);
    if (flux->kind == DGW_FLUX_EULER) return fail(DGW_EUNSUPPORTED, "dgw_rk_step_noalloc is built for the scalar laws");
    if (flux->kind < DGW_FLUX_ADVECT || flux->kind > DGW_FLUX_KPP) return fail(DGW_EINVAL, "bad flux kind");
    if (!(flux->lambda_nu >= 0.0)) return fail(DGW_EINVAL, "lambda_nu must be >= 0");
    dgw_status st = check_params(params, m.dim);
    if (st != DGW_OK) return st;
    if (!aligned16(U)) return fail(DGW_EINVAL, "U must be 16-byte aligned");
    if (nsteps < 0) return fail(DGW_EINVAL, "nsteps < 0");
    if (!std::isfinite(dt)) return fail(DGW_EINVAL, "dt must be finite");
    const int64_t E = m.dim == 1 ? (int64_t)m.nx : (int64_t)m.nx * m.ny;
    const int K = m.dim == 1 ? p + 1 : (p + 1) * (p + 1);
    const int eb = params->prec == DGW_FP64 ? 8 : 4;
    const double bytes = (double)K * (double)E * eb;
    if (bytes > (double)kNoAllocStageBytes)
        return fail(DGW_EINVAL,
                    "dgw_rk_step_noalloc: a state of %.0f bytes exceeds the fixed stage capacity of %zu "
                    "bytes (K*E*elem_bytes); use dgw_create/dgw_rk_step for larger meshes",
                    bytes, kNoAllocStageBytes);
    if (nsteps == 0) return DGW_OK;

    int dev = -1;
    DGW_CUDA(cudaGetDevice(&dev));
    unsigned char* base = nullptr;
    {
        // once per device (with that device current): the array's device address, and
        // the operator tables of this precision, dimension and degree
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        auto it = g_noalloc_addr.find(dev);
        if (it == g_noalloc_addr.end()) {
            void* ptr = nullptr;
            DGW_CUDA(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
            it = g_noalloc_addr.emplace(dev, static_cast<unsigned char*>(ptr)).first;
        }
        base = it->second;
        const auto key = std::make_tuple(dev, params->prec, m.dim, p);
        if (!g_noalloc_tables.count(key)) {
            HostTables t;
            build_tables(p, &t);
            cudaError_t ce;
            if (params->prec == DGW_FP64) ce = m.dim == 1 ? upload_tables_f64_d1(t) : upload_tables_f64_d2(t);
            else ce = m.dim == 1 ? upload_tables_f32_d1(t) : upload_tables_f32_d2(t);
            if (ce != cudaSuccess) return fail(DGW_ECUDA, "table upload: %s", cudaGetErrorString(ce));
            g_noalloc_tables.insert(key);
        }
    }

    // A context that lives on the host stack and points into the fixed array.
    dgw_ctx c;
    c.device = dev;
    c.mesh = m;
    if (m.dim == 1) c.mesh.ny = 1;
    c.p = p;
    c.flux = *flux;
    c.params = *params;
    c.K = K;
    c.E = E;
    c.eb = eb;
    c.h = hx;
    c.S1 = base;
    c.S2 = base + kNoAllocStageBytes;
    c.flag = reinterpret_cast<unsigned*>(base + 2 * kNoAllocStageBytes);
    DGW_CUDA(enqueue_steps(&c, U, dt, nsteps, (cudaStream_t)stream));
    return DGW_OK;
}

extern "C" const char* dgw_last_error(void) { return g_err.c_str(); }

extern "C" const char* dgw_version(void) { return "dgw 0.1 (sm_103a)"; }
