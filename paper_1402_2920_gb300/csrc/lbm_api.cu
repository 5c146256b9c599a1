// Host side of the C ABI declared in include/lbm.h.
//
// A simulation owns its device buffers and four CUDA graphs: one time step
// and two time steps, each for either population buffer as the source.  A
// time step is the chain moments -> force -> u-solve -> derivatives ->
// collide; the u-solve is a WHILE conditional node whose body is one Jacobi
// sweep (q, j~new) followed by a one-thread control kernel that tests
// convergence on the device and sets the loop condition, so a step never
// returns to the host.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include <cudaTypedefs.h>

#include "lbm.h"
#include "lbm_batch.h"
#include "lbm_common.h"
#include "lbm_lattice.h"
#include "lbm_plan.h"

using namespace lbm;

namespace {

constexpr int MAX_AUX = 26;
// extrapolation factor of the u-solve start j~_n + theta (j~_n - j~_n-1) (usolve_warm_start = 2):
// of 0.5, 0.75 and 1 measured on the 256^3 spinodal, 0.75 took the fewest sweeps over steps 6-25
// (5.95 against 6.35 and 6.4) at one sweep per step later on
constexpr double kWarmTheta = 0.75;

struct Graphs {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
};

}  // namespace

struct lbm_sim {
    int device = 0;
    cudaStream_t stream = nullptr;
    int lattice = 0, d = 0, Q = 0;
    int64_t dims[3] = {0, 0, 0};
    lbm_eos eos{};
    lbm_params prm{};
    KernelTable kt{};
    const void* sweep = nullptr;  // the sweep kernel in use: kt.sweep, or kt.sweep_tma when selected
    DevSim dev{};
    int cur = 0;  // population buffer holding the current pre-collision populations
    int64_t steps = 0;
    std::vector<void*> allocs;
    double* red_part = nullptr;
    HostView* view = nullptr;  // the device block that DevSim::us and DevSim::status point into
    Graphs one[2], two[2];
    bool graphs = false;  // the step graphs are built on the first lbm_step
};

namespace {

#define LBM_CK(call)                                                  \
    do {                                                              \
        cudaError_t e_ = (call);                                      \
        if (e_ != cudaSuccess) {                                      \
            (void)cudaGetLastError();                                 \
            return e_ == cudaErrorMemoryAllocation ? LBM_E_OOM : LBM_E_CUDA; \
        }                                                             \
    } while (0)

int nblocks(long long N, int block) { return int((N + block - 1) / block); }

// grid of a tiled kernel: one CTA per TX x TY column tile and z-slab
dim3 tile_grid(const lbm_sim* s, TiledKernel k);
dim3 moments_grid(const lbm_sim* s);
int moments_block(const lbm_sim* s);
cudaError_t launch_moments(const lbm_sim* s, DevSim dv, int src, int pair);

void host_eos(const lbm_eos& e, double rho, double out[4])
{
    double p, dp, d2p;
    if (e.kind == LBM_EOS_VDW) {
        const double g = 1.0 - e.b * rho;
        p = rho * e.T / g - e.a * rho * rho;
        dp = e.T / (g * g) - 2.0 * e.a * rho;
        d2p = 2.0 * e.b * e.T / (g * g * g) - 2.0 * e.a;
    } else {
        const double D = e.rho2 - e.rho1, rho3 = 2.0 * e.rho2 - e.rho1;
        double psi = 0.0, dpsi = 0.0, integ = 0.0;
        if (rho > e.rho1 && rho < rho3) {
            const double ph = M_PI * (rho - e.rho1) / D;
            psi = e.A * std::sin(ph);
            dpsi = e.A * M_PI / D * std::cos(ph);
            integ = e.A * D / M_PI * (1.0 - std::cos(ph));
        }
        const double cs2 = e.cs2_rho1 * std::exp(integ);
        p = rho * cs2;
        dp = cs2 * (1.0 + rho * psi);
        d2p = cs2 * psi * (1.0 + rho * psi) + cs2 * (psi + rho * dpsi);
    }
    out[0] = p;
    out[1] = dp;
    out[2] = p - rho * dp;
    out[3] = rho * d2p;
}

template <int LAT>
double host_weight(int k, double s)
{
    using L = Lat<LAT>;
    return L::wc(k, 0) + s * (L::wc(k, 1) + s * (L::wc(k, 2) + s * L::wc(k, 3)));
}

template <int LAT>
double min_weight(double s)
{
    double m = 1e300;
    for (int k = 0; k < Lat<LAT>::NSHELL; ++k) m = std::fmin(m, host_weight<LAT>(k, s));
    return m;
}

// edges of the interval around s_in where every shell weight is positive
template <int LAT>
void weight_window(double& lo, double& hi)
{
    const double s_in = 0.6;  // inside the window of both lattices
    double a = 0.01, b = s_in;
    for (int it = 0; it < 200; ++it) {
        const double m = 0.5 * (a + b);
        (min_weight<LAT>(m) > 0.0 ? b : a) = m;
    }
    lo = b;
    a = s_in;
    b = 3.0;
    for (int it = 0; it < 200; ++it) {
        const double m = 0.5 * (a + b);
        (min_weight<LAT>(m) > 0.0 ? a : b) = m;
    }
    hi = a;
}

// The parameters and derived constants of the kernels in arithmetic T (see Phys).
template <typename T>
void fill_phys(Phys<T>& q, const DevSim& dv, const lbm_eos& e)
{
    const double g = dv.gamma, c0 = dv.cs0;
    q.rho0 = T(dv.rho0);
    q.cs0 = T(c0);
    q.gamma = T(g);
    q.kappa = T(dv.kappa);
    q.omega = T(dv.omega);
    q.a = T(e.a);
    q.b = T(e.b);
    q.Teos = T(e.T);
    q.bT = T(e.b * e.T);
    q.g0 = T(1.0 - e.b * dv.rho0);
    {
        const double g0 = 1.0 - e.b * dv.rho0;
        const double F0 = e.b * e.T / (g0 * g0) - e.a;
        q.F0 = T(F0);
        q.F0lo = T(F0 - double(T(F0)));
        q.b2T_g02 = T(e.b * e.b * e.T / (g0 * g0));
    }
    const double D = e.kind == LBM_EOS_PSI_SINE ? e.rho2 - e.rho1 : 1.0;
    q.rho1 = T(e.rho1);
    q.rho3 = T(2.0 * e.rho2 - e.rho1);
    q.cs2_1 = T(e.cs2_rho1);
    q.A = T(e.A);
    q.pi_D = T(M_PI / D);
    q.A_pi_D = T(e.A * M_PI / D);
    q.AD_pi = T(e.A * D / M_PI);
    q.ph0 = T(M_PI * (dv.rho0 - e.rho1) / D);
    q.cs2_lo = T(dv.cs2_lo);
    q.cs2_hi = T(dv.cs2_hi);
    for (int k = 0; k < 8; ++k) {
        q.w0[k] = T(dv.w0[k]);
        q.off[k] = T(dv.off[k]);
        q.offc[k] = T(dv.off[k] - double(T(dv.off[k])));
        q.isc[k] = dv.w0[k] > 0.0 ? T(1.0 / dv.w0[k]) : T(0);
    }
    q.k1 = T(-0.25 * (g + 1.0) * (g + 1.0) / (g - 1.0));
    q.k2 = T((1.0 / 6.0) * (g * g + 4.0 * g + 1.0) / (g - 1.0));
    q.k3 = T((1.0 / 3.0) * (g * g + 4.0 * g + 1.0) / (g + 1.0));
    q.cf_int = T(0.5 * (1.0 + g) / c0);
    q.cf_jt = T((g - 1.0) / c0);
    q.cf_h2 = T(0.5 / (c0 * c0));
    q.cf_h3 = T(1.0 / (6.0 * c0 * c0 * c0));
    q.cj = T((1.0 - g) * c0);
    for (int k = 0; k < 8; ++k) q.w0h2[k] = T(dv.w0[k] * 0.5 / (c0 * c0));
}

// warm-start j~ buffers: two for the start extrapolated from the last two steps
int warm_buffers(const DevSim& dv) { return dv.warm == 2 ? 2 : 1; }

bool is_local(int storage)
{
    return storage == LBM_STORE_F32_LOC || storage == LBM_STORE_F16_LOC || storage == LBM_STORE_BF16_LOC;
}

size_t bytes_per_site(int lattice, int storage, size_t* ssize_out = nullptr)
{
    const int Q = lattice == LBM_D3Q59 ? 59 : 21;
    const int naux = lattice == LBM_D3Q59 ? 26 : 13;
    size_t ssize = 4, tsize = 4;
    if (storage == LBM_STORE_F16_DEV || storage == LBM_STORE_BF16_DEV || storage == LBM_STORE_F16_LOC ||
        storage == LBM_STORE_BF16_LOC)
        ssize = 2;
    if (storage == LBM_STORE_F64) ssize = tsize = 8;
    if (ssize_out) *ssize_out = ssize;
    const size_t usize = 8;  // worst case: FP64 u-solve
    const size_t rest = storage == LBM_STORE_F64 ? 0 : 2 * 8 + 4;  // two float-pair rest planes, rho_lo
    // the senders' references of the local-reference storages, one set per population buffer
    const size_t wref = is_local(storage) ? 2 * (lattice == LBM_D3Q59 ? 8 : 6) * 4 : 0;
    // populations (two buffers), rest planes, rho - rho0, j0', f, aux; u iterates (2 x 2),
    // warm-start j~ (two buffers with the extrapolated start) and the two Chebyshev update vectors
    return 2 * Q * ssize + rest + wref + tsize * (1 + 3 + 3 + naux) + usize * (4 * 3 + 2 * 3 + 2 * 3);
}

int validate(int lattice, const int64_t dims[3], int storage)
{
    if (lattice != LBM_D2Q21 && lattice != LBM_D3Q59) return LBM_E_INVALID_ARG;
    if (!dims) return LBM_E_INVALID_ARG;
    if (storage < LBM_STORE_F32 || storage > LBM_STORE_BF16_LOC) return LBM_E_INVALID_ARG;
    if (dims[0] < 4 || dims[1] < 4) return LBM_E_INVALID_ARG;
    if (lattice == LBM_D2Q21 && dims[2] != 1) return LBM_E_INVALID_ARG;
    if (lattice == LBM_D3Q59 && dims[2] < 4) return LBM_E_INVALID_ARG;
    if (dims[0] > (1 << 20) || dims[1] > (1 << 20) || dims[2] > (1 << 20)) return LBM_E_INVALID_ARG;
    const double N = double(dims[0]) * double(dims[1]) * double(dims[2]);
    const int Q = lattice == LBM_D3Q59 ? 59 : 21;
    if (N * Q > 9.0e18 / 8.0) return LBM_E_INVALID_ARG;
    // site indices inside a plane stack are 32-bit in the streaming kernel; the tiled kernels' grids have
    // ceil(ny / 8) rows of CTAs (wide_tiles keeps to lattices whose four-row tiles fit)
    if (N >= 2147483648.0 || dims[1] > kGridRows * 8) return LBM_E_INVALID_ARG;
    return LBM_OK;
}

cudaError_t add_kernel(cudaGraph_t g, cudaGraphNode_t* out, const void* fn, dim3 grid, int block, void** args,
                       const cudaGraphNode_t* deps, size_t ndeps, size_t smem = 0)
{
    cudaKernelNodeParams kp{};
    kp.func = const_cast<void*>(fn);
    kp.gridDim = grid;
    kp.blockDim = dim3(block);
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = args;
    kp.extra = nullptr;
    return cudaGraphAddKernelNode(out, g, deps, ndeps, &kp);
}

// Append one time step (source buffer src) to graph g after dependency dep.
int add_step(lbm_sim* s, cudaGraph_t g, cudaGraphNode_t dep, int src, cudaGraphNode_t* last)
{
    DevSim& dv = s->dev;
    const int B = s->kt.block;
    const int G = nblocks(dv.N, B);
    int pair = 0, mode = SWEEP_IN_GRAPH;
    cudaGraphNode_t n1, n2[2], nc, n5, n6;
    const cudaGraphNode_t* d0 = dep ? &dep : nullptr;
    size_t nd0 = dep ? 1 : 0;
    {
        void* a[] = {&dv, &src, &pair};
        LBM_CK(add_kernel(g, &n1, s->kt.moments, moments_grid(s), moments_block(s), a, d0, nd0));
    }
    const TileShape* ts = s->kt.tile;
    {
        void* a[] = {&dv, &pair};
        LBM_CK(add_kernel(g, &n2[0], s->kt.force, tile_grid(s, TK_FORCE), ts[TK_FORCE].threads, a, &n1, 1, s->kt.smem_force));
    }
    {  // beside the force kernel: the solve's start needs the density range alone
        void* a[] = {&dv, &pair};
        LBM_CK(add_kernel(g, &n2[1], s->kt.us_begin, dim3(1), 32, a, &n1, 1));
    }
    cudaGraphConditionalHandle h;
    LBM_CK(cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault));
    // One sweep and its control step after `deps`.
    auto add_sweep = [&](cudaGraph_t to, const cudaGraphNode_t* deps, size_t ndeps, cudaGraphNode_t* out) -> int {
        cudaGraphNode_t b1;
        void* a1[] = {&dv, &pair, &mode};
        LBM_CK(add_kernel(to, &b1, s->sweep, tile_grid(s, TK_SWEEP), ts[TK_SWEEP].threads, a1, deps, ndeps, s->kt.smem_sweep));
        void* a2[] = {&dv, &pair, &h, &mode};
        LBM_CK(add_kernel(to, out, s->kt.us_ctl, dim3(1), 1, a2, &b1, 1));
        return LBM_OK;
    };
    const cudaGraphNode_t* deps = n2;
    size_t ndeps = 2;
    // The first sweeps as plain nodes, which return at once when the solve has stopped before them; the loop takes
    // the rest.  An iteration of the WHILE node costs 4 us more than a plain node, an idle sweep 1 to 3.
    // Measured, us per step with 0 / 1 / 2 / 3 / 4 plain sweeps: 64^2 59 / 56 / 50 / 47 / 48, 512^2 105 / 102 / 99 / 96 / 96,
    // 333 x 217 77 / 72 / 68 / 64 / 65, 32^3 62 / 59 / 55 / 56 / 58, 128^3 484 / 478 / 472 / 473 / 475.
    constexpr int kPlainSweeps = 3;
    cudaGraphNode_t ahead[kPlainSweeps];
    for (int k = 0; k < kPlainSweeps; ++k) {
        const int rc = add_sweep(g, deps, ndeps, &ahead[k]);
        if (rc) return rc;
        deps = &ahead[k];
        ndeps = 1;
    }
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    LBM_CK(cudaGraphAddNode(&nc, g, deps, nullptr, ndeps, &cp));
    {
        cudaGraphNode_t last_sweep;
        const int rc = add_sweep(cp.conditional.phGraph_out[0], nullptr, 0, &last_sweep);
        if (rc) return rc;
    }
    {
        void* a[] = {&dv};
        LBM_CK(add_kernel(g, &n5, s->kt.derivs, tile_grid(s, TK_DERIVS), ts[TK_DERIVS].threads, a, &nc, 1, s->kt.smem_derivs));
    }
    {
        void* a[] = {&dv, &src};
        LBM_CK(add_kernel(g, &n6, s->kt.collide, tile_grid(s, TK_COLLIDE), ts[TK_COLLIDE].threads, a, &n5, 1, s->kt.smem_collide));
    }
    *last = n6;
    return LBM_OK;
}

int build_graphs(lbm_sim* s)
{
    for (int src = 0; src < 2; ++src) {
        LBM_CK(cudaGraphCreate(&s->one[src].g, 0));
        cudaGraphNode_t last;
        int rc = add_step(s, s->one[src].g, nullptr, src, &last);
        if (rc) return rc;
        LBM_CK(cudaGraphInstantiate(&s->one[src].x, s->one[src].g, 0));
        LBM_CK(cudaGraphCreate(&s->two[src].g, 0));
        cudaGraphNode_t mid;
        rc = add_step(s, s->two[src].g, nullptr, src, &mid);
        if (rc) return rc;
        rc = add_step(s, s->two[src].g, mid, src ^ 1, &last);
        if (rc) return rc;
        LBM_CK(cudaGraphInstantiate(&s->two[src].x, s->two[src].g, 0));
    }
    return LBM_OK;
}

// Device buffers come from the stream-ordered allocator on the simulation's stream:
// creating and destroying simulations (a serving loop does it per request) then
// neither synchronises the device nor stalls the other simulations' streams.
int dev_alloc(lbm_sim* s, void** p, size_t bytes)
{
    cudaError_t e = cudaMallocAsync(p, bytes, s->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        *p = nullptr;
        return e == cudaErrorMemoryAllocation ? LBM_E_OOM : LBM_E_CUDA;
    }
    s->allocs.push_back(*p);
    return LBM_OK;
}

template <class... A>
cudaError_t launch(const lbm_sim* s, const void* fn, int grid, int block, A... args)
{
    void* a[] = {&args...};
    return cudaLaunchKernel(fn, dim3(grid), dim3(block), a, 0, s->stream);
}

template <class... A>
cudaError_t launch_tiled(const lbm_sim* s, TiledKernel k, A... args)
{
    const void* fn[kTiled] = {s->kt.force, s->sweep, s->kt.derivs, s->kt.collide};
    const size_t smem[kTiled] = {s->kt.smem_force, s->kt.smem_sweep, s->kt.smem_derivs, s->kt.smem_collide};
    void* a[] = {&args...};
    return cudaLaunchKernel(fn[k], tile_grid(s, k), dim3(s->kt.tile[k].threads), a, smem[k], s->stream);
}

// Everything issued so far is done, and the block is in *v.
int read_view(lbm_sim* s, HostView* v)
{
    LBM_CK(cudaMemcpyAsync(v, s->view, sizeof(HostView), cudaMemcpyDeviceToHost, s->stream));
    LBM_CK(cudaStreamSynchronize(s->stream));
    return LBM_OK;
}
int clear_status(lbm_sim* s, int bits)
{
    if (!bits) return LBM_OK;
    LBM_CK(cudaMemsetAsync(s->dev.status, 0, sizeof(int), s->stream));
    LBM_CK(cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

int status_code(int bits)
{
    if (bits & STB_TIMEOUT) return LBM_E_TIMEOUT;
    if (bits & (STB_WEIGHTS | STB_NONFINITE_RHO)) return LBM_E_WEIGHTS;
    if (bits & (STB_USOLVE_CAP | STB_USOLVE_NAN)) return LBM_E_USOLVE_DIVERGED;
    return LBM_OK;
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
using EncodeTiledFn = PFN_cuTensorMapEncodeTiled_v12000;
EncodeTiledFn tensor_map_encoder()
{
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// Tensor map of a field [ncomp][nz][ny][nx] (rank 3 when ncomp = 1) read in boxes of one plane of
// box_x x box_y sites and box_comps components, out-of-range elements read as zero.
bool encode_plane_map(CUtensorMap* m, void* base, int ncomp, size_t esize, const DevSim& dv, int box_x, int box_y,
                      int box_comps)
{
    const EncodeTiledFn enc = tensor_map_encoder();
    if (!enc || !base) return false;
    const cuuint32_t rank = ncomp > 1 ? 4 : 3;
    const cuuint64_t dims[4] = {cuuint64_t(dv.nx), cuuint64_t(dv.ny), cuuint64_t(dv.nz), cuuint64_t(ncomp)};
    const cuuint64_t strides[3] = {cuuint64_t(dv.nx) * esize, cuuint64_t(dv.nx) * cuuint64_t(dv.ny) * esize,
                                   cuuint64_t(dv.N) * esize};
    const cuuint32_t boxd[4] = {cuuint32_t(box_x), cuuint32_t(box_y), 1, cuuint32_t(box_comps)};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    const CUresult r = enc(m, esize == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, rank, base,
                           dims, strides, boxd, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// The sweep kernel: the tensor-copy (TMA) form, whose tensor maps need a 3D lattice with rows a
// multiple of 16 bytes, or per-thread plane copies (2D, other sizes, or LBM_SWEEP_COPY=cp_async in
// the environment).  The two are close: Chebyshev sweep with tensor / per-thread copies, us, 256^3 368 / 366, 192^3 173 / 170,
// 160^3 110 / 107, 128^3 61.6 / 59.5, 288 x 192 x 224 280 / 281.  The tensor form is the default: it wins on the
// largest of these, and leaves the threads no copies to issue.
void setup_sweep_maps(lbm_sim* s)
{
    DevSim& dv = s->dev;
    dv.tma = 0;
    dv.tmaps = nullptr;
    s->sweep = s->kt.sweep;
    const char* sel = std::getenv("LBM_SWEEP_COPY");
    if ((sel && std::strcmp(sel, "cp_async") == 0) || !s->kt.sweep_tma) return;
    if (s->d != 3 || !dv.aligned16 || dv.nx % 4 != 0) return;
    SweepMaps m;
    const int bx = s->kt.sweep_box[0], by = s->kt.sweep_box[1];
    bool ok = true;
    for (int pr = 0; pr < 2; ++pr)
        for (int b = 0; b < 2; ++b)
            ok = ok && encode_plane_map(&m.u[pr][b], dv.uit[pr][b], 3, s->kt.usize, dv, bx, by, dv.pm_scaled ? 3 : 1);
    ok = ok && (dv.pm_scaled ? encode_plane_map(&m.rho, dv.pm, 2, sizeof(float), dv, bx, s->kt.pm_rows, 2)
                      : encode_plane_map(&m.rho, dv.rho, 1, s->kt.tsize, dv, bx, by, 1));
    void* dm = nullptr;
    ok = ok && dev_alloc(s, &dm, sizeof(SweepMaps)) == LBM_OK;
    ok = ok && cudaMemcpyAsync(dm, &m, sizeof(SweepMaps), cudaMemcpyHostToDevice, s->stream) == cudaSuccess &&
         cudaStreamSynchronize(s->stream) == cudaSuccess;  // m lives on this stack
    if (!ok) (void)cudaGetLastError();
    dv.tmaps = ok ? static_cast<const SweepMaps*>(dm) : nullptr;
    dv.tma = ok ? 1 : 0;
    if (ok) s->sweep = s->kt.sweep_tma;
}

// The u iterates need no reset: each solve's force kernel writes the one that its first sweep reads.
int reset_usolve(lbm_sim* s)
{
    LBM_CK(launch(s, s->kt.reset, 1, 256, s->dev));
    const size_t jbytes = 3 * size_t(s->dev.N) * s->kt.usize;
    LBM_CK(cudaMemsetAsync(s->dev.jt_warm, 0, warm_buffers(s->dev) * jbytes, s->stream));
    return LBM_OK;
}

// moments kernel: flat grid, or for the local-reference storages the row grid (x-blocks of
// kMomentsRowBlock threads, y, z), which gives each thread its coordinates
constexpr int kMomentsRowBlock = 128;
dim3 moments_grid(const lbm_sim* s)
{
    if (!s->kt.local_ref) return dim3(nblocks(s->dev.N, s->kt.block));
    return dim3((s->dev.nx + kMomentsRowBlock - 1) / kMomentsRowBlock, s->dev.ny, s->d == 3 ? s->dev.nz : 1);
}
int moments_block(const lbm_sim* s) { return s->kt.local_ref ? kMomentsRowBlock : s->kt.block; }

cudaError_t launch_moments(const lbm_sim* s, DevSim dv, int src, int pair)
{
    void* a[] = {&dv, &src, &pair};
    return cudaLaunchKernel(s->kt.moments, moments_grid(s), dim3(moments_block(s)), a, 0, s->stream);
}

dim3 tile_grid(const lbm_sim* s, TiledKernel k)
{
    const TileShape& t = s->kt.tile[k];
    const int zb = s->dev.zb[k];
    return dim3((s->dev.nx + t.tx - 1) / t.tx, (s->dev.ny + t.ty - 1) / t.ty, s->d == 3 ? (s->dev.nz + zb - 1) / zb : 1);
}

// z-slab depth of each tiled kernel.  A CTA marches zb planes plus its halo, and the grid's
// tiles_xy * ceil(nz / zb) CTAs run in waves of (resident CTAs per SM) x SMs.  Deep slabs repeat
// less halo; shallow ones give a small lattice enough CTAs to fill the chip, and a last wave that
// is nearly empty costs as much as a full one.  The depth taken minimises the modelled time
//   (zb + halo) x (full waves x l[resident] + l[CTAs per SM of the last wave]),
// with l[r] the time (us) a CTA takes per plane when r share an SM and halo the cost of a CTA's
// other planes in the same unit, both fitted to cubes of 16^3 to 192^3 at depths 2 to 48 on GB300
// (the model is within 10 % of those measurements).  Measured, us per step of force + 3 sweeps +
// derivatives + collision against the one depth of 32 of before: 32^3 359 -> 70, 64^3 377 -> 118, 96^3 406 -> 264,
// 160^3 1129 -> 1002.  With FP64 fields or sweeps the CTAs of an SM share its FP64 units,
// so l grows with r (48^3 FP64: 4.9 -> 0.78 ms).  LBM_TILE_Z=<n> in the environment at lbm_create
// sets the depth of all (any depth gives the same results, bit for bit).
void choose_zb(lbm_sim* s)
{
    DevSim& dv = s->dev;
    for (int& zb : dv.zb) zb = 1;
    if (s->d != 3) return;
    const int nz = dv.nz;
    for (int& zb : dv.zb) zb = nz < 32 ? nz : 32;
    if (const char* env = std::getenv("LBM_TILE_Z")) {
        const int v = std::atoi(env);
        if (v >= 1) {
            for (int& zb : dv.zb) zb = v < nz ? v : nz;
            return;
        }
    }
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, s->device) != cudaSuccess || nsm < 1) {
        (void)cudaGetLastError();
        return;
    }
    constexpr int RMAX = 4;
    const bool f64 = s->kt.tsize == 8 || s->kt.usize == 8;
    struct Kern {
        const void* fn;
        size_t smem;
        double halo, l[RMAX];
        double l64;  // per plane and resident CTA with FP64 arithmetic
    } ks[kTiled] = {{s->kt.force, s->kt.smem_force, 2.0, {0.9, 1.2, 1.5, 1.9}, 6.0},
                    {s->sweep, s->kt.smem_sweep, 6.0, {1.3, 1.65, 2.2, 2.9}, 16.6},
                    {s->kt.derivs, s->kt.smem_derivs, 1.5, {1.8, 2.2, 2.9, 3.9}, 31.0},
                    {s->kt.collide, s->kt.smem_collide, 0.5, {3.3, 6.6, 9.9, 13.2}, 60.0}};
    auto set = [&](TiledKernel k, double halo, double l1, double l2, double l3, double l4) {
        ks[k].halo = halo;
        ks[k].l[0] = l1, ks[k].l[1] = l2, ks[k].l[2] = l3, ks[k].l[3] = l4;
    };
    if (s->kt.pm_rows) {  // b_sweep_pm, and the force kernel that writes its pressure pair
        set(TK_FORCE, 2.0, 1.0, 1.35, 1.7, 2.1);
        set(TK_SWEEP, 8.0, 0.95, 1.4, 1.7, 2.3);
    }
    if (s->kt.derivs == s->kt.pair_derivs) {  // the kernels on pairs of sites
        set(TK_DERIVS, 1.3, 1.5, 2.0, 2.55, 3.4);
        set(TK_COLLIDE, 0.3, 2.75, 5.0, 7.5, 10.0);
    }
    for (int q = 0; q < kTiled; ++q) {
        Kern& k = ks[q];
        const TileShape& t = s->kt.tile[q];
        const long long txy = (long long)((dv.nx + t.tx - 1) / t.tx) * ((dv.ny + t.ty - 1) / t.ty);
        int r = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k.fn, t.threads, k.smem) != cudaSuccess) {
            (void)cudaGetLastError();
            r = 1;
        }
        r = r < 1 ? 1 : r > RMAX ? RMAX : r;
        if (f64)
            for (int m = 0; m < RMAX; ++m) k.l[m] = k.l64 * (m + 1);
        double cbest = 1e300;
        for (int zb = 1; zb <= 48 && zb <= nz; ++zb) {
            if ((nz + zb - 1) / zb > 65535) continue;  // gridDim.z
            const long long ctas = txy * ((nz + zb - 1) / zb), slots = (long long)r * nsm;
            const long long full = ctas / slots, rem = ctas % slots;
            const double c = (zb + k.halo) * (double(full) * k.l[r - 1] + (rem ? k.l[(rem + nsm - 1) / nsm - 1] : 0.0));
            if (c < cbest * (1.0 - 1e-9)) {
                dv.zb[q] = zb;
                cbest = c;
            }
        }
    }
}

// S1-S8 on the current populations with the scratch j~ pair, and the fields to device memory.  The sweeps are
// launched kAhead at a time, the fields' kernel behind them: sweeps that come after the solve has stopped
// return at once, a fields' kernel before it has too, and one copy tells whether it has.  (One sweep and one copy in turn
// left the device idle for the host's round trip at each sweep.)
int run_fields(lbm_sim* s, double* rho, double* u, HostView* v)
{
    constexpr int kAhead = 4;
    DevSim& dv = s->dev;
    const int B = s->kt.block, G = nblocks(dv.N, B);
    const int pair = 1, mode = SWEEP_BY_HOST;
    const cudaGraphConditionalHandle h{};
    LBM_CK(launch_moments(s, dv, s->cur, pair));
    LBM_CK(launch_tiled(s, TK_FORCE, dv, pair));
    LBM_CK(launch(s, s->kt.us_begin, 1, 32, dv, pair));
    for (int it = 0; it < dv.maxit + 1; it += kAhead) {
        for (int k = 0; k < kAhead; ++k) {
            LBM_CK(launch_tiled(s, TK_SWEEP, dv, pair, mode));
            LBM_CK(launch(s, s->kt.us_ctl, 1, 1, dv, pair, h, mode));
        }
        LBM_CK(launch(s, s->kt.fields_out, G, B, dv, 1, rho, u));
        const int rc = read_view(s, v);
        if (rc) return rc;
        if (!v->us[1].running) break;  // the control step recorded a stop
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

const char* lbm_error_string(int code)
{
    switch (code) {
    case LBM_OK: return "ok";
    case LBM_E_INVALID_ARG: return "invalid argument";
    case LBM_E_WEIGHTS: return "c_s^2 left the positive-weight window or a density became non-finite";
    case LBM_E_BULKVISC: return "equation of state not admissible (bulk viscosity or weights)";
    case LBM_E_USOLVE_DIVERGED: return "u-solve did not converge within its sweep cap";
    case LBM_E_OOM: return "out of device memory";
    case LBM_E_CUDA: return "CUDA error or no usable device";
    case LBM_E_TIMEOUT: return "device wait timed out";
    case LBM_E_IO: return "checkpoint file error";
    default: return "unknown error";
    }
}

int lbm_velocities(int lattice, int* c_out)
{
    if (lattice == LBM_D2Q21) {
        using L = Lat<0>;
        if (c_out)
            for (int i = 0; i < L::Q; ++i) { c_out[3 * i] = L::cx(i); c_out[3 * i + 1] = L::cy(i); c_out[3 * i + 2] = 0; }
        return L::Q;
    }
    if (lattice == LBM_D3Q59) {
        using L = Lat<1>;
        if (c_out)
            for (int i = 0; i < L::Q; ++i) { c_out[3 * i] = L::cx(i); c_out[3 * i + 1] = L::cy(i); c_out[3 * i + 2] = L::cz(i); }
        return L::Q;
    }
    return LBM_E_INVALID_ARG;
}

size_t lbm_footprint_bytes(int lattice, const int64_t dims[3], int storage)
{
    if (validate(lattice, dims, storage) != LBM_OK) return 0;
    const size_t N = size_t(dims[0]) * size_t(dims[1]) * size_t(dims[2]);
    return N * bytes_per_site(lattice, storage) + 64 * 1024;
}

void lbm_destroy(lbm_sim* s)
{
    if (!s) return;
    cudaSetDevice(s->device);
    if (s->stream) cudaStreamSynchronize(s->stream);
    for (int k = 0; k < 2; ++k) {
        if (s->one[k].x) cudaGraphExecDestroy(s->one[k].x);
        if (s->one[k].g) cudaGraphDestroy(s->one[k].g);
        if (s->two[k].x) cudaGraphExecDestroy(s->two[k].x);
        if (s->two[k].g) cudaGraphDestroy(s->two[k].g);
    }
    for (void* p : s->allocs) cudaFreeAsync(p, s->stream);
    if (s->stream) cudaStreamSynchronize(s->stream);
    (void)cudaGetLastError();
    delete s;
}

int lbm_create(int lattice, const int64_t dims[3], const lbm_eos* eos, const lbm_params* params, void* cuda_stream,
               lbm_sim** out)
{
    if (!out || !eos || !params) return LBM_E_INVALID_ARG;
    *out = nullptr;
    int rc = validate(lattice, dims, params->storage);
    if (rc) return rc;
    if (!(params->gamma > -1.0 && params->gamma < 1.0)) return LBM_E_INVALID_ARG;
    if (!(params->kappa >= 0.0) || !(params->rho0 > 0.0)) return LBM_E_INVALID_ARG;
    if (eos->kind != LBM_EOS_VDW && eos->kind != LBM_EOS_PSI_SINE) return LBM_E_INVALID_ARG;
    if (eos->kind == LBM_EOS_PSI_SINE && !(eos->rho2 > eos->rho1 && eos->cs2_rho1 > 0.0)) return LBM_E_INVALID_ARG;
    if (params->usolve_precision != LBM_USOLVE_NATIVE && params->usolve_precision != LBM_USOLVE_F64)
        return LBM_E_INVALID_ARG;

    const int d = lattice == LBM_D3Q59 ? 3 : 2;
    double lo, hi;
    if (lattice == LBM_D3Q59) weight_window<1>(lo, hi); else weight_window<0>(lo, hi);

    // create-time admissibility of the EOS (App. B) over the density range of the run
    double e0[4];
    host_eos(*eos, params->rho0, e0);
    const double cs0 = e0[0] / params->rho0;
    if (!(cs0 > lo && cs0 < hi)) return LBM_E_WEIGHTS;
    if (params->rho_check_max > params->rho_check_min && params->rho_check_min > 0.0) {
        for (int k = 0; k <= 2000; ++k) {
            const double r = params->rho_check_min + (params->rho_check_max - params->rho_check_min) * k / 2000.0;
            double e[4];
            host_eos(*eos, r, e);
            const double cs2 = e[0] / r;
            if (!(cs2 > lo && cs2 < hi)) return LBM_E_WEIGHTS;
            if (!(r * e[1] / e[0] < 1.0 + 2.0 / d)) return LBM_E_BULKVISC;
        }
    }

    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        (void)cudaGetLastError();
        return LBM_E_CUDA;
    }
    lbm_sim* s = new (std::nothrow) lbm_sim();
    if (!s) return LBM_E_OOM;
    cudaGetDevice(&s->device);
    s->stream = static_cast<cudaStream_t>(cuda_stream);
    s->lattice = lattice;
    s->d = d;
    s->Q = lattice == LBM_D3Q59 ? 59 : 21;
    for (int k = 0; k < 3; ++k) s->dims[k] = dims[k];
    s->eos = *eos;
    s->prm = *params;

    const bool f64 = params->storage == LBM_STORE_F64;
    const bool us64 = f64 || params->usolve_precision == LBM_USOLVE_F64;
    const bool read_pops = params->gamma != 0.0;
    bool ok = lattice == LBM_D3Q59 ? get_kernels_d3q59(params->storage, us64, read_pops, &s->kt)
                                   : get_kernels_d2q21(params->storage, us64, read_pops, &s->kt);
    if (!ok) { delete s; return LBM_E_INVALID_ARG; }
    // the kernels on pairs of sites need pairs that stay aligned words: nx even
    if (s->kt.pair_derivs && pairs_of_sites(dims)) {
        KernelTable& kt = s->kt;
        kt.derivs = kt.pair_derivs;
        kt.kb_derivs = kt.kb_pair_derivs;
        kt.tile[TK_DERIVS] = kt.tile_pair_derivs;
        kt.smem_derivs = kt.smem_pair_derivs;
        const PairCollide& c = kt.pair_collide[wide_tiles(dims) ? 1 : 0];
        kt.collide = c.collide;
        kt.kb_collide = c.kb_collide;
        kt.tile[TK_COLLIDE] = c.tile;
        kt.smem_collide = c.smem;
    }

    DevSim& dv = s->dev;
    dv.lattice = lattice;
    dv.d = d;
    dv.Q = s->Q;
    dv.nx = int(dims[0]);
    dv.ny = int(dims[1]);
    dv.nz = int(dims[2]);
    dv.N = (long long)dims[0] * dims[1] * dims[2];
    dv.gamma = params->gamma;
    dv.kappa = params->kappa;
    dv.rho0 = params->rho0;
    dv.cs0 = cs0;
    const int nshell = lattice == LBM_D3Q59 ? 8 : 6;
    for (int k = 0; k < 8; ++k) {
        dv.w0[k] = k < nshell ? (lattice == LBM_D3Q59 ? host_weight<1>(k, cs0) : host_weight<0>(k, cs0)) : 0.0;
        dv.off[k] = dv.w0[k] * params->rho0;
    }
    dv.eos_kind = eos->kind;
    dv.a = eos->a; dv.b = eos->b; dv.T = eos->T;
    dv.rho1 = eos->rho1; dv.rho2 = eos->rho2; dv.A = eos->A; dv.cs2_1 = eos->cs2_rho1;
    dv.cs2_lo = lo;
    dv.cs2_hi = hi;
    if (params->usolve_tol > 0.0 || params->usolve_rtol > 0.0) {
        dv.tol = params->usolve_tol > 0.0 ? params->usolve_tol : 0.0;
        dv.rtol = params->usolve_rtol > 0.0 ? params->usolve_rtol : 0.0;
    } else if (us64) {
        dv.tol = 1e-14;
        dv.rtol = 0.0;
    } else {
        // below the rounding noise the stored populations put into j0 each step: tighter
        // stops only chase that noise
        dv.tol = s->kt.ssize == 2 ? 4e-8 : 5e-9;
        dv.rtol = 0.0;
    }
    if (!(params->usolve_omega >= 0.0 && params->usolve_omega < 2.0)) { lbm_destroy(s); return LBM_E_INVALID_ARG; }
    dv.omega = params->usolve_omega;  // 0: 2/(2 - g) per solve
    dv.maxit = params->usolve_max_iter > 0 ? params->usolve_max_iter : 500;
    if (params->usolve_warm_start < 0 || params->usolve_warm_start > 2) { lbm_destroy(s); return LBM_E_INVALID_ARG; }
    dv.warm = params->usolve_warm_start;
    dv.wtheta = kWarmTheta;
    {
        double smax = 0.0;  // max_k |(4/3) sin k - (1/6) sin 2k|, the Sec. IV.B symbol
        for (int k = 0; k <= 20000; ++k) {
            const double x = M_PI * k / 20000.0;
            smax = std::fmax(smax, std::fabs(4.0 / 3.0 * std::sin(x) - std::sin(2.0 * x) / 6.0));
        }
        dv.s2max = smax * smax;
        // the bound of each solve comes from its density range.  16-bit storages stay Chebyshev throughout:
        // their tolerance is far above the rounding of u, and 6 sweeps became 5 at best
        dv.cheb = params->usolve_chebyshev ? (s->kt.ssize == 2 ? 2 : 1) : 0;
    }
    fill_phys<float>(dv.pf, dv, *eos);
    fill_phys<double>(dv.pd, dv, *eos);
    for (int k = 0; k < nshell; ++k) {
        // velocities of shell k as multiples of {-1, 0, 1}^3 ones
        int m = 1;
        for (int i = 1; i < s->Q; ++i) {
            const int ks = lattice == LBM_D3Q59 ? Lat<1>::shell(i) : Lat<0>::shell(i);
            const int cx = lattice == LBM_D3Q59 ? Lat<1>::cx(i) : Lat<0>::cx(i);
            if (ks == k && std::abs(cx) > m) m = std::abs(cx);
        }
        dv.pc.wh2[k] = float(dv.w0[k] * m * m * 0.5 / (cs0 * cs0));
        dv.pc.wl[k] = float(dv.w0[k] * m);
        dv.pc.wh3[k] = float(dv.w0[k] * m * m * m / (6.0 * cs0 * cs0 * cs0));
    }

    const size_t N = size_t(dv.N);
    const size_t T = s->kt.tsize, U = s->kt.usize, SS = s->kt.ssize;
    rc = LBM_OK;
    rc = rc ? rc : dev_alloc(s, &dv.pop[0], size_t(s->Q) * N * SS);
    rc = rc ? rc : dev_alloc(s, &dv.pop[1], size_t(s->Q) * N * SS);
    if (s->kt.rsize) {  // separate rest plane of the reduced storages
        rc = rc ? rc : dev_alloc(s, &dv.pop0[0], N * s->kt.rsize);
        rc = rc ? rc : dev_alloc(s, &dv.pop0[1], N * s->kt.rsize);
    }
    for (int b = 0; b < 2 && !rc; ++b)
        for (int i = 0; i < s->Q; ++i) dv.popp[b][i] = static_cast<char*>(dv.pop[b]) + size_t(i) * N * SS;
    if (s->kt.exact) rc = rc ? rc : dev_alloc(s, &dv.rho_lo, N * sizeof(float));
    rc = rc ? rc : dev_alloc(s, &dv.rho, N * T);
    rc = rc ? rc : dev_alloc(s, &dv.j0p, 3 * N * T);
    rc = rc ? rc : dev_alloc(s, &dv.f, 3 * N * T);
    for (int pr = 0; pr < 2; ++pr)
        for (int b = 0; b < 2; ++b) rc = rc ? rc : dev_alloc(s, &dv.uit[pr][b], 3 * N * U);
    rc = rc ? rc : dev_alloc(s, &dv.jt_warm, size_t(warm_buffers(dv)) * 3 * N * U);
    if (s->kt.local_ref) {
        const int nshell = lattice == LBM_D3Q59 ? 8 : 6;
        for (int b = 0; b < 2; ++b) {
            void* w = nullptr;
            rc = rc ? rc : dev_alloc(s, &w, size_t(nshell) * N * sizeof(float));
            dv.wref[b] = static_cast<float*>(w);
        }
    }
    if (dv.cheb) {
        rc = rc ? rc : dev_alloc(s, &dv.dvec[0], 3 * N * U);
        rc = rc ? rc : dev_alloc(s, &dv.dvec[1], 3 * N * U);
    }
    rc = rc ? rc : dev_alloc(s, &dv.aux, size_t(MAX_AUX) * N * T);
    dv.pm = dv.aux;
    dv.pm_scaled = s->kt.pm_rows ? 1 : 0;
    if (!rc) {
        for (int c = 0; c < MAX_AUX; ++c) dv.auxp[c] = static_cast<char*>(dv.aux) + size_t(c) * N * T;
        for (int a = 0; a < 3; ++a) {
            dv.j0pp[a] = static_cast<char*>(dv.j0p) + size_t(a) * N * T;
            dv.fpp[a] = static_cast<char*>(dv.f) + size_t(a) * N * T;
            for (int b = 0; b < 2; ++b)
                dv.jwp[b][a] = static_cast<char*>(dv.jt_warm) + size_t((warm_buffers(dv) - 1) * b * 3 + a) * N * U;
        }
    }
    void* vp = nullptr;
    rc = rc ? rc : dev_alloc(s, &vp, sizeof(HostView));
    s->view = static_cast<HostView*>(vp);
    if (!rc) {
        dv.us = s->view->us;
        dv.status = &s->view->status;
    }
    void* rgp = nullptr;
    rc = rc ? rc : dev_alloc(s, &rgp, 4 * kRangeSlots * sizeof(unsigned));
    dv.range = static_cast<unsigned*>(rgp);
    void* rp = nullptr;
    rc = rc ? rc : dev_alloc(s, &rp, kRedGrid * 4 * sizeof(double));
    s->red_part = static_cast<double*>(rp);
    dv.red = s->red_part;
    if (rc) { lbm_destroy(s); return rc; }
    {  // vector (16-byte) copies of the tiled kernels need 16-byte aligned field arrays
        auto a16 = [](const void* q) { return q == nullptr || (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
        bool ok = a16(dv.rho) && a16(dv.j0p) && a16(dv.f) && a16(dv.aux) && a16(dv.jt_warm);
        for (int pr = 0; pr < 2; ++pr)
            for (int b = 0; b < 2; ++b) ok = ok && a16(dv.uit[pr][b]);
        dv.aligned16 = ok ? 1 : 0;
    }
    setup_sweep_maps(s);
    choose_zb(s);
    // well-defined contents before the first lbm_init
    for (int b = 0; b < 2; ++b) {
        const size_t wbytes = dv.wref[b] ? size_t(lattice == LBM_D3Q59 ? 8 : 6) * N * sizeof(float) : 0;
        if (cudaMemsetAsync(dv.pop[b], 0, size_t(s->Q) * N * SS, s->stream) != cudaSuccess ||
            (dv.pop0[b] && cudaMemsetAsync(dv.pop0[b], 0, N * s->kt.rsize, s->stream) != cudaSuccess) ||
            (wbytes && cudaMemsetAsync(dv.wref[b], 0, wbytes, s->stream) != cudaSuccess)) {
            lbm_destroy(s);
            return LBM_E_CUDA;
        }
    }
    for (int pr = 0; pr < 2; ++pr)
        for (int b = 0; b < 2; ++b)
            if (cudaMemsetAsync(dv.uit[pr][b], 0, 3 * N * U, s->stream) != cudaSuccess) rc = LBM_E_CUDA;
    if (!rc) rc = reset_usolve(s);
    if (!rc && cudaStreamSynchronize(s->stream) != cudaSuccess) rc = LBM_E_CUDA;
    if (rc) { lbm_destroy(s); return rc; }
    *out = s;
    return LBM_OK;
}

int lbm_init(lbm_sim* s, const double* rho, const double* u, int on_device)
{
    if (!s || !rho) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    const size_t N = size_t(s->dev.N);
    const double* drho = rho;
    const double* du = u;
    // staging buffer of host inputs, released on every return path (stream-ordered)
    struct Staging {
        double* p = nullptr;
        cudaStream_t st;
        ~Staging() { if (p) (void)cudaFreeAsync(p, st); }
    } stage{nullptr, s->stream};
    double*& tmp = stage.p;
    if (!on_device) {
        LBM_CK(cudaMallocAsync(&tmp, (1 + s->d) * N * sizeof(double), s->stream));
        LBM_CK(cudaMemcpyAsync(tmp, rho, N * sizeof(double), cudaMemcpyHostToDevice, s->stream));
        drho = tmp;
        if (u) {
            LBM_CK(cudaMemcpyAsync(tmp + N, u, s->d * N * sizeof(double), cudaMemcpyHostToDevice, s->stream));
            du = tmp + N;
        }
    }
    int rc = reset_usolve(s);
    if (rc) return rc;
    s->cur = 0;
    s->steps = 0;
    const int B = s->kt.block, G = nblocks(s->dev.N, B);
    if (s->kt.init_ref) LBM_CK(launch(s, s->kt.init_ref, G, B, s->dev, drho, 0));
    LBM_CK(launch(s, s->kt.init_eq, G, B, s->dev, drho, du, 0));
    if (tmp) {
        double* p = tmp;
        tmp = nullptr;
        LBM_CK(cudaFreeAsync(p, s->stream));
        LBM_CK(cudaStreamSynchronize(s->stream));  // the caller's host arrays are borrowed for the call only
    }
    return LBM_OK;
}

}  // extern "C"

namespace {

bool trace_mode()
{
    const char* v = std::getenv("LBM_TRACE");
    return v && v[0] == '1';
}

// One step with every kernel launched on its own and the u-solve loop driven
// from the host (the same kernels and order as the graph).
int step_direct(lbm_sim* s)
{
    DevSim& dv = s->dev;
    const int B = s->kt.block, G = nblocks(dv.N, B);
    const int pair = 0, mode = SWEEP_BY_HOST, src = s->cur;
    const cudaGraphConditionalHandle h{};
    LBM_CK(launch_moments(s, dv, src, pair));
    LBM_CK(launch_tiled(s, TK_FORCE, dv, pair));
    LBM_CK(launch(s, s->kt.us_begin, 1, 32, dv, pair));
    for (int it = 0; it < dv.maxit + 1; ++it) {
        LBM_CK(launch_tiled(s, TK_SWEEP, dv, pair, mode));
        LBM_CK(launch(s, s->kt.us_ctl, 1, 1, dv, pair, h, mode));
        UsolveState u;
        LBM_CK(cudaMemcpyAsync(&u, &dv.us[0], sizeof(u), cudaMemcpyDeviceToHost, s->stream));
        LBM_CK(cudaStreamSynchronize(s->stream));
        if (trace_mode())  // the residual history of every u-solve, for tuning the solver
            std::fprintf(stderr, "lbm usolve step %lld sweep %d resid %.3e mode %d next c1 %.4f c2 %.4f\n",
                         (long long)s->steps, u.iter, u.running ? u.resid_min : u.resid_last, u.mode, u.c1, u.c2);
        if (!u.running) break;
    }
    LBM_CK(launch_tiled(s, TK_DERIVS, dv));
    LBM_CK(launch_tiled(s, TK_COLLIDE, dv, src));
    s->cur ^= 1;
    return LBM_OK;
}

bool direct_mode()
{
    const char* v = std::getenv("LBM_LAUNCH");
    return v && std::strcmp(v, "direct") == 0;
}

}  // namespace

extern "C" {

int lbm_step(lbm_sim* s, int64_t nsteps)
{
    if (!s || nsteps < 0) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    if (direct_mode()) {
        for (int64_t k = 0; k < nsteps; ++k) {
            const int rc = step_direct(s);
            if (rc) return rc;
            s->steps += 1;
        }
        return LBM_OK;
    }
    if (!s->graphs && nsteps > 0) {  // built on first use: simulations stepped in batches never need them
        const int rc = build_graphs(s);
        if (rc) return rc;
        s->graphs = true;
    }
    int64_t n = nsteps;
    while (n >= 2) {
        LBM_CK(cudaGraphLaunch(s->two[s->cur].x, s->stream));
        n -= 2;
    }
    if (n == 1) {
        LBM_CK(cudaGraphLaunch(s->one[s->cur].x, s->stream));
        s->cur ^= 1;
    }
    s->steps += nsteps;
    return LBM_OK;
}

int lbm_sync(lbm_sim* s)
{
    if (!s) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    HostView v;
    int rc = read_view(s, &v);
    rc = rc ? rc : clear_status(s, v.status);
    return rc ? rc : status_code(v.status);
}

int lbm_fields(lbm_sim* s, double* rho, double* u, int on_device)
{
    if (!s) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    const size_t N = size_t(s->dev.N);
    double* drho = rho;
    double* du = u;
    double* tmp = nullptr;
    if (!on_device && (rho || u)) {
        LBM_CK(cudaMallocAsync(&tmp, (1 + s->d) * N * sizeof(double), s->stream));
        drho = rho ? tmp : nullptr;
        du = u ? tmp + N : nullptr;
    }
    HostView v;
    int rc = run_fields(s, drho, du, &v);
    if (tmp) {
        if (!rc && rho && cudaMemcpyAsync(rho, drho, N * sizeof(double), cudaMemcpyDeviceToHost, s->stream) != cudaSuccess)
            rc = LBM_E_CUDA;
        if (!rc && u && cudaMemcpyAsync(u, du, s->d * N * sizeof(double), cudaMemcpyDeviceToHost, s->stream) != cudaSuccess)
            rc = LBM_E_CUDA;
        if (cudaFreeAsync(tmp, s->stream) != cudaSuccess && !rc) rc = LBM_E_CUDA;
        if (!rc && cudaStreamSynchronize(s->stream) != cudaSuccess) rc = LBM_E_CUDA;
        if (rc) (void)cudaGetLastError();
    }
    rc = rc ? rc : clear_status(s, v.status);
    return rc ? rc : status_code(v.status);
}

int lbm_populations(lbm_sim* s, double* out, int on_device)
{
    if (!s || !out) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    const size_t bytes = size_t(s->Q) * size_t(s->dev.N) * sizeof(double);
    double* d = out;
    if (!on_device) LBM_CK(cudaMallocAsync(&d, bytes, s->stream));
    const int B = s->kt.block, G = nblocks(s->dev.N, B);
    LBM_CK(launch(s, s->kt.pops_out, G, B, s->dev, s->cur, d));
    if (!on_device) {
        LBM_CK(cudaMemcpyAsync(out, d, bytes, cudaMemcpyDeviceToHost, s->stream));
        LBM_CK(cudaFreeAsync(d, s->stream));
    }
    LBM_CK(cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

int lbm_set_populations(lbm_sim* s, const double* in, int on_device)
{
    if (!s || !in) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    const size_t bytes = size_t(s->Q) * size_t(s->dev.N) * sizeof(double);
    const double* d = in;
    double* tmp = nullptr;
    if (!on_device) {
        LBM_CK(cudaMallocAsync(&tmp, bytes, s->stream));
        LBM_CK(cudaMemcpyAsync(tmp, in, bytes, cudaMemcpyHostToDevice, s->stream));
        d = tmp;
    }
    int rc = reset_usolve(s);
    if (rc) return rc;
    s->cur = 0;
    const int B = s->kt.block, G = nblocks(s->dev.N, B);
    double* rho = nullptr;
    if (s->kt.init_ref) {
        // local-reference storages: every site's references from the density of the given
        // populations, then the populations relative to their senders'
        LBM_CK(cudaMallocAsync(&rho, size_t(s->dev.N) * sizeof(double), s->stream));
        LBM_CK(launch(s, s->kt.pops_rho, G, B, s->dev, d, rho));
        LBM_CK(launch(s, s->kt.init_ref, G, B, s->dev, (const double*)rho, 0));
    }
    LBM_CK(launch(s, s->kt.pops_in, G, B, s->dev, d, 0));
    if (rho) LBM_CK(cudaFreeAsync(rho, s->stream));
    if (tmp) LBM_CK(cudaFreeAsync(tmp, s->stream));
    LBM_CK(cudaStreamSynchronize(s->stream));
    return LBM_OK;
}

int lbm_stats_get(lbm_sim* s, lbm_stats* out)
{
    if (!s || !out) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    LBM_CK(launch(s, s->kt.red_partial, kRedGrid, kRedBlock, s->dev, s->cur, s->red_part));
    LBM_CK(launch(s, s->kt.red_final, 1, kRedBlock, s->dev, (const double*)s->red_part, kRedGrid, s->view->sums));
    HostView v;
    const int rc = read_view(s, &v);
    if (rc) return rc;
    const UsolveState& u = v.us[0];
    out->mass = v.sums[0];
    out->mom[0] = v.sums[1];
    out->mom[1] = v.sums[2];
    out->mom[2] = v.sums[3];
    out->steps = s->steps;
    out->usolve_iters_last = u.iters_last;
    out->usolve_iters_max = u.iters_max;
    out->usolve_resid = u.resid_last;
    out->status = v.status;
    out->usolve_sweeps_total = u.sweeps_total;
    out->usolve_tensor_copies = u.tma;
    return LBM_OK;
}

int lbm_profile(lbm_sim* s, int reps, double* ms_out, int n)
{
    if (!s || reps < 1 || !ms_out || n < 0) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    DevSim& dv = s->dev;
    const int B = s->kt.block, G = nblocks(dv.N, B);
    const int src = s->cur, pair = 1;
    // the collision kernel rewrites the warm-start j~: keep the run's copy aside
    const size_t jbytes = size_t(warm_buffers(dv)) * 3 * size_t(dv.N) * s->kt.usize;
    void* keep = nullptr;
    LBM_CK(cudaMallocAsync(&keep, jbytes, s->stream));
    LBM_CK(cudaMemcpyAsync(keep, dv.jt_warm, jbytes, cudaMemcpyDeviceToDevice, s->stream));
    cudaEvent_t e0, e1;
    LBM_CK(cudaEventCreate(&e0));
    LBM_CK(cudaEventCreate(&e1));
    // the scratch u-solve pair; the collision writes the spare population buffer
    LBM_CK(launch_moments(s, dv, src, pair));
    LBM_CK(launch_tiled(s, TK_FORCE, dv, pair));
    LBM_CK(launch(s, s->kt.us_begin, 1, 32, dv, pair));
    const int alone = SWEEP_ALONE;
    if (dv.cheb) {
        // the sweep as a Chebyshev solve runs it after its first, which reads and writes the update vector (us_begin
        // alone would leave c1 = 0: 60 instead of 72 bytes per site in FP32)
        UsolveState u{};
        LBM_CK(cudaMemcpyAsync(&u, &dv.us[pair], sizeof(u), cudaMemcpyDeviceToHost, s->stream));
        LBM_CK(cudaStreamSynchronize(s->stream));
        cheb_first(u);
        usolve_next(u, 2, 0.0, 0.0);
        LBM_CK(cudaMemcpyAsync(&dv.us[pair], &u, sizeof(u), cudaMemcpyHostToDevice, s->stream));
        LBM_CK(cudaStreamSynchronize(s->stream));  // u lives on this stack
        LBM_CK(cudaMemsetAsync(dv.dvec[pair], 0, 3 * size_t(dv.N) * s->kt.usize, s->stream));
    }
    int rc = LBM_OK;
    for (int k = 0; k < 5 && rc == LBM_OK; ++k) {
        for (int r = 0; r <= reps && rc == LBM_OK; ++r) {
            if (r == 1 && cudaEventRecord(e0, s->stream) != cudaSuccess) rc = LBM_E_CUDA;
            cudaError_t e = cudaSuccess;
            switch (k) {
            case 0: e = launch_moments(s, dv, src, pair); break;
            case 1: e = launch_tiled(s, TK_FORCE, dv, pair); break;
            case 2: e = launch_tiled(s, TK_SWEEP, dv, pair, alone); break;
            case 3: e = launch_tiled(s, TK_DERIVS, dv); break;
            case 4: e = launch_tiled(s, TK_COLLIDE, dv, src); break;
            }
            if (e != cudaSuccess) rc = LBM_E_CUDA;
        }
        if (rc == LBM_OK && cudaEventRecord(e1, s->stream) != cudaSuccess) rc = LBM_E_CUDA;
        if (rc == LBM_OK && cudaEventSynchronize(e1) != cudaSuccess) rc = LBM_E_CUDA;
        float ms = 0.f;
        if (rc == LBM_OK && cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) rc = LBM_E_CUDA;
        if (rc == LBM_OK && k < n) ms_out[k] = double(ms) / reps;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    (void)cudaGetLastError();
    if (rc == LBM_OK && trace_mode()) {
        UsolveState u{};
        if (cudaMemcpy(&u, &dv.us[pair], sizeof(u), cudaMemcpyDeviceToHost) != cudaSuccess) rc = LBM_E_CUDA;
        std::fprintf(stderr, "lbm profile sweep c1 %.4f c2 %.4f\n", u.c1, u.c2);
    }
    // the scratch solve's density ranges hold this state's (lbm_fields would widen its own with them): empty them; its
    // residual accumulators were left mid-loop: clear them; restore the warm start
    if (rc == LBM_OK && launch(s, s->kt.us_begin, 1, 32, dv, pair) != cudaSuccess) rc = LBM_E_CUDA;
    UsolveState u1{};
    if (rc == LBM_OK && cudaMemcpyAsync(&dv.us[1], &u1, sizeof(u1), cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
        rc = LBM_E_CUDA;
    if (cudaMemcpyAsync(dv.jt_warm, keep, jbytes, cudaMemcpyDeviceToDevice, s->stream) != cudaSuccess) rc = LBM_E_CUDA;
    if (cudaFreeAsync(keep, s->stream) != cudaSuccess) rc = LBM_E_CUDA;
    if (rc == LBM_OK && cudaStreamSynchronize(s->stream) != cudaSuccess) rc = LBM_E_CUDA;
    return rc;
}

namespace {
struct CkptHeader {
    char magic[8];
    int32_t lattice, storage, usize, Q;
    int32_t warm_buffers, pad;
    int64_t dims[3];
    int64_t steps;
    double gamma, kappa, rho0;
};
}  // namespace

int lbm_save(lbm_sim* s, const char* path)
{
    if (!s || !path) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    LBM_CK(cudaStreamSynchronize(s->stream));
    const size_t N = size_t(s->dev.N);
    const size_t pbytes = size_t(s->Q) * N * s->kt.ssize;
    const size_t zbytes = N * s->kt.rsize;
    const size_t jbytes = size_t(warm_buffers(s->dev)) * 3 * N * s->kt.usize;
    const size_t wbytes = s->dev.wref[0] ? size_t(s->d == 3 ? 8 : 6) * N * sizeof(float) : 0;
    std::vector<char> buf(pbytes + zbytes + jbytes + wbytes);
    UsolveState us[2];
    LBM_CK(cudaMemcpy(us, s->dev.us, sizeof(us), cudaMemcpyDeviceToHost));
    LBM_CK(cudaMemcpy(buf.data(), s->dev.pop[s->cur], pbytes, cudaMemcpyDeviceToHost));
    if (zbytes) LBM_CK(cudaMemcpy(buf.data() + pbytes, s->dev.pop0[s->cur], zbytes, cudaMemcpyDeviceToHost));
    LBM_CK(cudaMemcpy(buf.data() + pbytes + zbytes, s->dev.jt_warm, jbytes, cudaMemcpyDeviceToHost));
    if (wbytes)  // the senders' references the stored populations are relative to
        LBM_CK(cudaMemcpy(buf.data() + pbytes + zbytes + jbytes, s->dev.wref[s->cur], wbytes, cudaMemcpyDeviceToHost));
    CkptHeader h{};
    std::memcpy(h.magic, "LBM2PH03", 8);
    h.lattice = s->lattice;
    h.storage = s->prm.storage;
    h.usize = int32_t(s->kt.usize);
    h.Q = s->Q;
    h.warm_buffers = warm_buffers(s->dev);
    for (int k = 0; k < 3; ++k) h.dims[k] = s->dims[k];
    h.steps = s->steps;
    h.gamma = s->prm.gamma;
    h.kappa = s->prm.kappa;
    h.rho0 = s->prm.rho0;
    FILE* fp = std::fopen(path, "wb");
    if (!fp) return LBM_E_IO;
    bool ok = std::fwrite(&h, sizeof(h), 1, fp) == 1 && std::fwrite(&us[0], sizeof(UsolveState), 1, fp) == 1 &&
              std::fwrite(buf.data(), 1, buf.size(), fp) == buf.size();
    ok = (std::fclose(fp) == 0) && ok;
    return ok ? LBM_OK : LBM_E_IO;
}

int lbm_load(lbm_sim* s, const char* path)
{
    if (!s || !path) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(s->device));
    FILE* fp = std::fopen(path, "rb");
    if (!fp) return LBM_E_IO;
    CkptHeader h{};
    UsolveState u0{};
    bool ok = std::fread(&h, sizeof(h), 1, fp) == 1 && std::fread(&u0, sizeof(u0), 1, fp) == 1;
    ok = ok && std::memcmp(h.magic, "LBM2PH03", 8) == 0 && h.lattice == s->lattice && h.storage == s->prm.storage &&
         h.warm_buffers == warm_buffers(s->dev) &&
         h.usize == int32_t(s->kt.usize) && h.Q == s->Q && h.dims[0] == s->dims[0] && h.dims[1] == s->dims[1] &&
         h.dims[2] == s->dims[2];
    const size_t N = size_t(s->dev.N);
    const size_t pbytes = size_t(s->Q) * N * s->kt.ssize;
    const size_t zbytes = N * s->kt.rsize;
    const size_t jbytes = size_t(warm_buffers(s->dev)) * 3 * N * s->kt.usize;
    const size_t wbytes = s->dev.wref[0] ? size_t(s->d == 3 ? 8 : 6) * N * sizeof(float) : 0;
    std::vector<char> buf;
    if (ok) {
        buf.resize(pbytes + zbytes + jbytes + wbytes);
        ok = std::fread(buf.data(), 1, buf.size(), fp) == buf.size();
    }
    std::fclose(fp);
    if (!ok) return LBM_E_IO;
    LBM_CK(cudaStreamSynchronize(s->stream));
    int rc = reset_usolve(s);
    if (rc) return rc;
    LBM_CK(cudaStreamSynchronize(s->stream));  // the copies below do not go through the stream
    s->cur = 0;
    u0.cur = 0;
    u0.resid_bits = 0;
    u0.jmax_bits = 0;
    LBM_CK(cudaMemcpy(s->dev.pop[0], buf.data(), pbytes, cudaMemcpyHostToDevice));
    if (zbytes) LBM_CK(cudaMemcpy(s->dev.pop0[0], buf.data() + pbytes, zbytes, cudaMemcpyHostToDevice));
    LBM_CK(cudaMemcpy(s->dev.jt_warm, buf.data() + pbytes + zbytes, jbytes, cudaMemcpyHostToDevice));
    if (wbytes) LBM_CK(cudaMemcpy(s->dev.wref[0], buf.data() + pbytes + zbytes + jbytes, wbytes, cudaMemcpyHostToDevice));
    LBM_CK(cudaMemcpy(&s->dev.us[0], &u0, sizeof(u0), cudaMemcpyHostToDevice));
    s->steps = h.steps;
    return LBM_OK;
}

int lbm_step_batch(lbm_sim* const* sims, int n, const int64_t* nsteps)
{
    if ((!sims || !nsteps) && n > 0) return LBM_E_INVALID_ARG;
    for (int k = 0; k < n; ++k)
        if (!sims[k] || nsteps[k] < 0) return LBM_E_INVALID_ARG;
    for (int k = 0; k < n; ++k) {
        int rc = lbm_step(sims[k], nsteps[k]);
        if (rc) return rc;
    }
    return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched stepping (lbm_batch.h)
// ---------------------------------------------------------------------------
namespace lbm {

struct Batch {
    KernelTable kt{};
    int key = 0;
    int device = 0;
    cudaStream_t stream = nullptr;
    DevSim* d_sims = nullptr;    // [kBatchSlots] device table
    BatchWork* d_work = nullptr;
    DevSim* h_sims = nullptr;    // pinned mirrors of the table and the work list (copied from
    BatchWork* h_work = nullptr; // these asynchronously, so they change only between chunks)
    cudaEvent_t copied = nullptr; // the mirrors' last copy to the device has been done
    lbm_sim* slot[kBatchSlots] = {};
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
};

// The class of nx (odd, or the pairwise collision's tile width) tells batches apart for every combination, also where
// no kernel depends on it: a batch steps in lockstep, and up to three smaller ones on their own streams overlap.
// Measured, ms against one batch: 15 requests of 96^2, 113^2, 120^2 54.5 / 64.5, of 352^2, 480^2, 511^2 200 / 212;
// 12 of 40^3, 48^3, 51^3 with 16-bit populations 69.9 / 72.7, with FP32 n_i 132 / 134.
int batch_key(int lattice, const int64_t dims[3], const lbm_params& prm)
{
    const bool us64 = prm.storage == LBM_STORE_F64 || prm.usolve_precision == LBM_USOLVE_F64;
    const int combo = (((lattice * 16 + prm.storage) * 2 + (us64 ? 1 : 0)) * 2 + (prm.gamma != 0.0 ? 1 : 0)) * 3 +
                      (pairs_of_sites(dims) ? (wide_tiles(dims) ? 2 : 1) : 0);
    int64_t n = dims[0] * dims[1] * (lattice == LBM_D3Q59 ? dims[2] : 1);
    int size_class = 0;
    while (n >= 4) {
        n >>= 2;
        ++size_class;
    }
    return combo * 64 + size_class;
}

int batch_key_of(const lbm_sim* s) { return batch_key(s->lattice, s->dims, s->prm); }

namespace {

// persistent grid of a batched kernel: the blocks that fit on the device at once
int resident_grid(const void* fn, int threads, size_t smem)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem) != cudaSuccess || per < 1) {
        (void)cudaGetLastError();
        per = 1;
    }
    return sms * per;
}

int build_batch_graph(Batch* b)
{
    LBM_CK(cudaGraphCreate(&b->g, 0));
    const KernelTable& kt = b->kt;
    DevSim* sims = b->d_sims;
    BatchWork* w = b->d_work;
    int pair = 0;
    const int FB = kt.tile[TK_FORCE].threads, SB = kt.tile[TK_SWEEP].threads, DB = kt.tile[TK_DERIVS].threads,
              CB = kt.tile[TK_COLLIDE].threads;
    const int MB = kt.local_ref ? kMomentsRowBlock : kt.block;
    cudaGraphNode_t n0, n1, n2, n3, nc, n5, n6, n7;
    {
        void* a[] = {&sims, &w};
        LBM_CK(add_kernel(b->g, &n0, kt.kb_step_begin, dim3(1), 32, a, nullptr, 0));
    }
    {
        void* a[] = {&sims, &w, &pair};
        LBM_CK(add_kernel(b->g, &n1, kt.kb_moments, dim3(resident_grid(kt.kb_moments, MB, 0)), MB, a, &n0, 1));
    }
    {
        void* a[] = {&sims, &w, &pair};
        LBM_CK(add_kernel(b->g, &n2, kt.kb_force, dim3(resident_grid(kt.kb_force, FB, kt.smem_force)), FB, a, &n1, 1,
                          kt.smem_force));
    }
    {
        void* a[] = {&sims, &w, &pair};
        LBM_CK(add_kernel(b->g, &n3, kt.kb_us_begin, dim3(1), 32 * kBatchSlots, a, &n2, 1));
    }
    cudaGraphConditionalHandle h;
    LBM_CK(cudaGraphConditionalHandleCreate(&h, b->g, 1, cudaGraphCondAssignDefault));
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    LBM_CK(cudaGraphAddNode(&nc, b->g, &n3, nullptr, 1, &cp));
    {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        cudaGraphNode_t b1, b2;
        void* a1[] = {&sims, &w, &pair};
        LBM_CK(add_kernel(body, &b1, kt.kb_sweep, dim3(resident_grid(kt.kb_sweep, SB, kt.smem_sweep)), SB, a1, nullptr, 0,
                          kt.smem_sweep));
        void* a2[] = {&sims, &w, &pair, &h};
        LBM_CK(add_kernel(body, &b2, kt.kb_us_ctl, dim3(1), 32, a2, &b1, 1));
    }
    {
        void* a[] = {&sims, &w};
        LBM_CK(add_kernel(b->g, &n5, kt.kb_derivs, dim3(resident_grid(kt.kb_derivs, DB, kt.smem_derivs)), DB, a, &nc, 1,
                          kt.smem_derivs));
    }
    {
        void* a[] = {&sims, &w};
        LBM_CK(add_kernel(b->g, &n6, kt.kb_collide, dim3(resident_grid(kt.kb_collide, CB, kt.smem_collide)), CB, a, &n5,
                          1, kt.smem_collide));
    }
    {
        void* a[] = {&sims, &w};
        LBM_CK(add_kernel(b->g, &n7, kt.kb_step_end, dim3(1), 32, a, &n6, 1));
    }
    LBM_CK(cudaGraphInstantiate(&b->x, b->g, 0));
    return LBM_OK;
}

}  // namespace

int batch_create(const lbm_sim* proto, cudaStream_t stream, Batch** out)
{
    if (!proto || !out) return LBM_E_INVALID_ARG;
    *out = nullptr;
    Batch* b = new (std::nothrow) Batch();
    if (!b) return LBM_E_OOM;
    b->kt = proto->kt;
    b->key = batch_key_of(proto);
    b->device = proto->device;
    b->stream = stream;
    int rc = LBM_OK;
    if (cudaSetDevice(b->device) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&b->d_sims), sizeof(DevSim) * kBatchSlots) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&b->d_work), sizeof(BatchWork)) != cudaSuccess ||
        cudaMallocHost(reinterpret_cast<void**>(&b->h_sims), sizeof(DevSim) * kBatchSlots) != cudaSuccess ||
        cudaMallocHost(reinterpret_cast<void**>(&b->h_work), sizeof(BatchWork)) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->copied, cudaEventDisableTiming) != cudaSuccess) {
        (void)cudaGetLastError();
        rc = LBM_E_OOM;
    }
    if (!rc) {
        std::memset(static_cast<void*>(b->h_sims), 0, sizeof(DevSim) * kBatchSlots);
        std::memset(static_cast<void*>(b->h_work), 0, sizeof(BatchWork));
        rc = build_batch_graph(b);
    }
    if (rc) {
        batch_destroy(b);
        return rc;
    }
    *out = b;
    return LBM_OK;
}

int batch_attach(Batch* b, int slot, lbm_sim* s)
{
    if (!b || !s || slot < 0 || slot >= kBatchSlots || b->slot[slot] || batch_key_of(s) != b->key) return LBM_E_INVALID_ARG;
    b->slot[slot] = s;
    return LBM_OK;
}

void batch_detach(Batch* b, int slot)
{
    if (b && slot >= 0 && slot < kBatchSlots) b->slot[slot] = nullptr;
}

int batch_launch(Batch* b, const int64_t* steps)
{
    if (!b || !steps) return LBM_E_INVALID_ARG;
    LBM_CK(cudaSetDevice(b->device));
    LBM_CK(cudaEventSynchronize(b->copied));  // the mirrors may be rewritten
    BatchWork& w = *b->h_work;
    int nslot = 0;
    int64_t most = 0;
    for (int k = 0; k < kBatchSlots; ++k)
        if (b->slot[k]) nslot = k + 1;
    w.nslot = nslot;
    for (int q = 0; q < kTiled; ++q) w.tstart[q][0] = 0;
    w.mstart[0] = 0;
    for (int k = 0; k < kBatchSlots; ++k) {
        lbm_sim* s = b->slot[k];
        const int64_t n = s ? steps[k] : 0;
        if (n < 0) return LBM_E_INVALID_ARG;
        most = n > most ? n : most;
        w.live[k] = 0;
        w.todo[k] = int(n);
        w.src[k] = s ? s->cur : 0;
        if (s) b->h_sims[k] = s->dev;
        for (int q = 0; q < kTiled; ++q) {
            const dim3 g = s ? tile_grid(s, TiledKernel(q)) : dim3(1, 1, 0);
            w.tgx[q][k] = int(g.x);
            w.tgy[q][k] = int(g.y);
            w.tstart[q][k + 1] = w.tstart[q][k] + int(g.x * g.y * g.z);
        }
        const dim3 m = s ? moments_grid(s) : dim3(1, 1, 0);
        w.mgx[k] = int(m.x);
        w.mgy[k] = int(m.y);
        w.mstart[k + 1] = w.mstart[k] + int(m.x * m.y * m.z);
    }
    if (most == 0) return LBM_OK;
    LBM_CK(cudaMemcpyAsync(b->d_sims, b->h_sims, sizeof(DevSim) * size_t(nslot), cudaMemcpyHostToDevice, b->stream));
    LBM_CK(cudaMemcpyAsync(b->d_work, b->h_work, sizeof(BatchWork), cudaMemcpyHostToDevice, b->stream));
    LBM_CK(cudaEventRecord(b->copied, b->stream));
    for (int64_t i = 0; i < most; ++i) LBM_CK(cudaGraphLaunch(b->x, b->stream));
    return LBM_OK;
}

void batch_account(Batch* b, const int64_t* steps)
{
    if (!b || !steps) return;
    for (int k = 0; k < kBatchSlots; ++k) {
        lbm_sim* s = b->slot[k];
        if (!s || steps[k] <= 0) continue;
        s->cur ^= int(steps[k] & 1);
        s->steps += steps[k];
    }
}

void batch_destroy(Batch* b)
{
    if (!b) return;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->x) cudaGraphExecDestroy(b->x);
    if (b->g) cudaGraphDestroy(b->g);
    if (b->d_sims) cudaFree(b->d_sims);
    if (b->d_work) cudaFree(b->d_work);
    if (b->h_sims) cudaFreeHost(b->h_sims);
    if (b->h_work) cudaFreeHost(b->h_work);
    if (b->copied) cudaEventDestroy(b->copied);
    (void)cudaGetLastError();
    delete b;
}

}  // namespace lbm
