// Host side of the C ABI declared in include/nlbm.h: parameter validation,
// workspace layout, kernel dispatch and checkpoints.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstdint>
#include <cstring>
#include <algorithm>
#include <iterator>
#include <new>
#include <vector>

#include <cuda.h>

#include "../../include/nlbm.h"
#include "nlbm_internal.cuh"
#include "adjoint.cuh"

using namespace nlbm;

namespace {

thread_local char g_err[512] = "";

constexpr size_t kMaxPlane = (size_t)1 << 28;   // keeps 9 * plane in 32-bit offsets

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace layout.  FP32 storage: two copies of f [N-1][9] and g [8]
// planes, phi and P single (phi is updated in place, P written on request).
// 16-bit storage: two copies of the f deviations [N-1][8], the FP32 rest
// populations f0 [N-1], the g deviations [8], phi and P.  f[k] and g[k] are
// adjacent, so an idle f/g pair can stage N + 3 planes for host downloads.
struct Layout {
    size_t f[2], g[2], f0[2], phi[2], u[2], mphi, P[2], partials, mass, total;
    size_t fbytes, gbytes;
};

Layout make_layout(int ns, size_t plane, bool half)
{
    Layout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align256(off + bytes);
        return o;
    };
    const size_t es = half ? 2 : 4;
    L.fbytes = es * ns * (half ? 8 : 9) * plane;
    L.gbytes = es * 8 * plane;
    for (int k = 0; k < 2; ++k) {
        L.f[k] = take(L.fbytes);
        L.g[k] = take(L.gbytes);
    }
    for (int k = 0; k < 2; ++k) L.f0[k] = half ? take(sizeof(float) * ns * plane) : 0;
    L.phi[0] = take(sizeof(float) * ns * plane);
    L.phi[1] = half ? take(sizeof(float) * ns * plane) : L.phi[0];
    L.u[0] = take(sizeof(float) * 2 * plane);
    L.u[1] = take(sizeof(float) * 2 * plane);
    L.mphi = take(sizeof(float) * 2 * plane);
    L.P[0] = take(sizeof(float) * plane);
    L.P[1] = half ? take(sizeof(float) * plane) : L.P[0];
    L.partials = take(sizeof(double) * kMassBlocks * (ns + 2));
    L.mass = take(sizeof(double) * (ns + 2) + sizeof(int));
    L.total = off;
    return L;
}

bool is_half(int storage) { return storage == NLBM_STORE_BF16 || storage == NLBM_STORE_F16; }

void set_err(char *buf, const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, 512, fmt, ap);
    va_end(ap);
}

bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

// Whether a kernel may read the caller's [src, src + bytes) where it lies: a
// float array within one allocation of the current device's own memory.
// Everything else that a copy takes (memory of another device, managed or
// host memory, an odd address) or refuses (a range beyond its allocation) is
// left to the copy.
bool device_readable(const void *src, size_t bytes)
{
    using Get = CUresult (*)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const Get get = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<Get>(f) : nullptr;
    }();
    if (!get || ((uintptr_t)src & (sizeof(float) - 1))) return false;
    unsigned type = 0, managed = 0;   // left 0 for an address the driver does not know
    int ordinal = -1, device = -1;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                  CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *out[] = {&type, &managed, &ordinal, &start, &size};
    if (get(5, what, out, (CUdeviceptr)src) != CUDA_SUCCESS || type != CU_MEMORYTYPE_DEVICE || managed) return false;
    if (cudaGetDevice(&device) != cudaSuccess || ordinal != device) return false;
    const CUdeviceptr at = (CUdeviceptr)src;
    return at >= start && at - start <= size && bytes <= size - (at - start);
}

bool overlap(const void *a, size_t na, const void *b, size_t nb)
{
    return (uintptr_t)a < (uintptr_t)b + nb && (uintptr_t)b < (uintptr_t)a + na;
}

// Validates the problem statement; fills the derived kernel parameters.
nlbm_status validate(const nlbm_params *p, StepParams *kp, char *err)
{
    if (!p) { set_err(err, "params is NULL"); return NLBM_EINVAL; }
    const int N = p->n_phases;
    if (N < 2 || N > kMaxPhases) { set_err(err, "n_phases=%d outside 2..%d", N, kMaxPhases); return NLBM_EINVAL; }
    if (p->nx < 1 || p->ny < 1) { set_err(err, "lattice %dx%d is empty", p->nx, p->ny); return NLBM_EINVAL; }
    if ((p->bc_x != NLBM_BC_PERIODIC && p->bc_x != NLBM_BC_WALL) ||
        (p->bc_y != NLBM_BC_PERIODIC && p->bc_y != NLBM_BC_WALL)) {
        set_err(err, "unknown boundary type"); return NLBM_EINVAL;
    }
    if ((p->bc_x == NLBM_BC_WALL && p->nx < 4) || (p->bc_y == NLBM_BC_WALL && p->ny < 4)) {
        set_err(err, "a wall axis needs at least 4 nodes"); return NLBM_EINVAL;
    }
    if ((size_t)p->nx * (size_t)p->ny > kMaxPlane) {
        set_err(err, "lattice of %zu nodes exceeds %zu", (size_t)p->nx * p->ny, kMaxPlane);
        return NLBM_EINVAL;
    }
    if (p->model != NLBM_MODEL_A && p->model != NLBM_MODEL_B) { set_err(err, "unknown model"); return NLBM_EINVAL; }
    if (p->model == NLBM_MODEL_A && !finite_pos(p->model_a_n)) { set_err(err, "Model A exponent n must be > 0"); return NLBM_EINVAL; }
    if (!finite_pos(p->eps)) { set_err(err, "eps must be > 0"); return NLBM_EINVAL; }
    if (!finite_pos(p->mobility)) { set_err(err, "mobility must be > 0"); return NLBM_EINVAL; }
    if (!p->rho || !p->mu || !p->sigma) { set_err(err, "rho, mu and sigma must be given"); return NLBM_EINVAL; }
    for (int a = 0; a < N; ++a) {
        if (!finite_pos(p->rho[a])) { set_err(err, "rho[%d] must be > 0", a); return NLBM_EINVAL; }
        if (!finite_pos(p->mu[a])) { set_err(err, "mu[%d] must be > 0", a); return NLBM_EINVAL; }
        for (int b = 0; b < N; ++b) {
            const double s = p->sigma[a * N + b];
            if (a == b && s != 0.0) { set_err(err, "sigma[%d][%d] must be 0", a, a); return NLBM_EINVAL; }
            if (a != b && !finite_pos(s)) { set_err(err, "sigma[%d][%d] must be > 0", a, b); return NLBM_EINVAL; }
            if (s != p->sigma[b * N + a]) { set_err(err, "sigma is not symmetric at (%d,%d)", a, b); return NLBM_EINVAL; }
        }
    }
    if (p->reserved != 0) { set_err(err, "reserved must be 0"); return NLBM_EINVAL; }
    if (!std::isfinite(p->unit_delta) || p->unit_delta < 0.0) { set_err(err, "unit_delta must be >= 0"); return NLBM_EINVAL; }
    if (!std::isfinite(p->gx) || !std::isfinite(p->gy)) { set_err(err, "gravity not finite"); return NLBM_EINVAL; }
    bool wet = false;
    if (p->wall_cos) {
        for (int a = 0; a < 2 * (N - 1); ++a) {
            const double c = p->wall_cos[a];
            if (!(std::fabs(c) <= 1.0)) { set_err(err, "wall_cos[%d] must lie in [-1, 1]", a); return NLBM_EINVAL; }
            if (c != 0.0) wet = true;
        }
        if (wet && p->bc_y != NLBM_BC_WALL) { set_err(err, "wall_cos needs walls on y"); return NLBM_EINVAL; }
    }
    if (p->storage != NLBM_STORE_F32 && !is_half(p->storage)) { set_err(err, "unknown storage"); return NLBM_EINVAL; }
    if (is_half(p->storage) && (p->nx & 1)) {
        set_err(err, "16-bit storage needs an even nx (got %d)", p->nx); return NLBM_EINVAL;
    }
    if (kp) {
        memset(kp, 0, sizeof *kp);
        kp->nx = p->nx;
        kp->ny = p->ny;
        kp->wall_x = p->bc_x == NLBM_BC_WALL;
        kp->wall_y = p->bc_y == NLBM_BC_WALL;
        kp->model = p->model;
        kp->plane = (unsigned)((size_t)p->nx * p->ny);
        const double rhoN = p->rho[N - 1], muN = p->mu[N - 1];
        kp->rhoN = (float)rhoN;
        kp->muN = (float)muN;
        for (int a = 0; a < N - 1; ++a) {
            kp->drho[a] = (float)(p->rho[a] - rhoN);
            kp->dmu[a] = (float)(p->mu[a] - muN);
        }
        for (int a = 0; a < N; ++a)
            for (int b = 0; b < N; ++b) {
                const double s = p->sigma[a * N + b];
                kp->beta2[a][b] = (float)(6.0 * s / p->eps);       // 2 beta_pq, Eq. (15)
                kp->kap[a][b] = (float)(0.75 * p->eps * s);        // -k_pq, Eq. (15)
            }
        kp->four_over_eps = (float)(4.0 / p->eps);
        kp->unit_delta2 = (float)(p->unit_delta * p->unit_delta);
        kp->six_over_eps = (float)(6.0 / p->eps);
        kp->three_eps_over_4 = (float)(0.75 * p->eps);
        kp->mob = (float)p->mobility;
        kp->s1 = (float)(1.0 / (0.5 + 3.0 * p->mobility));        // Eq. (20), c_s^2 = 1/3
        kp->model_n = (float)p->model_a_n;
        kp->gx = (float)p->gx;
        kp->gy = (float)p->gy;
        // Sec. 4.2: cos theta_pq from the N-1 angles against phase N by
        // Young's relation, cos theta_qp = -cos theta_pq; stored times 4/eps
        kp->wet = wet ? 1 : 0;
        for (int w = 0; wet && w < 2; ++w) {
            const double *cn = p->wall_cos + w * (N - 1);
            for (int a = 0; a < N; ++a)
                for (int b = 0; b < N; ++b) {
                    double c = 0.0;
                    if (a != b) {
                        if (b == N - 1) c = cn[a];
                        else if (a == N - 1) c = -cn[b];
                        else c = (p->sigma[a * N + N - 1] * cn[a] - p->sigma[b * N + N - 1] * cn[b]) / p->sigma[a * N + b];
                    }
                    kp->wetc[w][a][b] = (float)(4.0 / p->eps * c);
                }
        }
        const double n = p->model_a_n;
        kp->model_n_int = (n == std::floor(n) && n >= 1.0 && n <= 8.0) ? (int)n : 0;
    }
    return NLBM_OK;
}

}  // namespace

struct nlbm_sim {
    StepParams kp;
    int N, ns, model, storage;
    size_t plane;
    cudaStream_t stream;
    char *ws;
    Layout L;
    int cur;
    int64_t steps;
    int64_t launches;
    int tx, ty;
    char err[512];
    bool half() const { return is_half(storage); }
    float *f(int k) const { return (float *)(ws + L.f[k]); }
    float *g(int k) const { return (float *)(ws + L.g[k]); }
    float *f0(int k) const { return half() ? (float *)(ws + L.f0[k]) : nullptr; }
    float *u(int k) const { return (float *)(ws + L.u[k]); }
    float *phi(int k) const { return (float *)(ws + L.phi[k]); }
    float *mphi() const { return (float *)(ws + L.mphi); }
    float *P(int k) const { return (float *)(ws + L.P[k]); }
};

namespace {

nlbm_status cuda_fail(nlbm_sim *s, cudaError_t e, const char *what)
{
    set_err(s->err, "%s: %s", what, cudaGetErrorString(e));
    return NLBM_ECUDA;
}

void default_tile(nlbm_sim *s)
{
    // 124-column strips; narrower lattices use 60-column strips, and so does
    // FP32 storage at N = 7 (2048^2: 8,562 against 8,090 MLUPS)
    s->tx = s->kp.nx > 96 && !(s->ns == 6 && s->storage == NLBM_STORE_F32) ? 128 : 64;
    s->ty = 0;
}

// Number of state bytes in a checkpoint, excluding the trailing counter.
size_t state_payload(const nlbm_sim *s)
{
    const size_t pb = sizeof(float) * s->plane;
    return s->L.fbytes + s->L.gbytes + (s->half() ? pb * s->ns : 0) + pb * (2 + s->ns + 2 + 1);
}

// Kernel parameters with the buffers of state a (input) -> b (output).
StepParams step_params(const nlbm_sim *s, int a, int b)
{
    StepParams kp = s->kp;
    kp.fin = s->f(a);
    kp.fout = s->f(b);
    kp.f0in = s->f0(a);
    kp.f0out = s->f0(b);
    kp.gin = s->g(a);
    kp.gout = s->g(b);
    kp.uin = s->u(a);
    kp.uout = s->u(b);
    kp.phi_prev = s->phi(a);
    kp.phi = s->phi(b);
    kp.mphi = s->mphi();
    kp.mphi_in = kp.mphi;
    kp.pin = s->P(a);
    kp.pout = s->P(b);
    return kp;
}

// Where the initial state's kernel reads the caller's phase fields from:
// dev_phi itself, or, where it may not be read in place or lies in memory
// ([own, own + own_bytes)) that the kernel writes, the state's phi planes,
// copied there first.
cudaError_t initial_fields(const float *dev_phi, float *phi, size_t bytes, const void *own, size_t own_bytes,
                           cudaStream_t stream, const float **src)
{
    *src = dev_phi;
    if (dev_phi == phi || (!overlap(dev_phi, bytes, own, own_bytes) && device_readable(dev_phi, bytes)))
        return cudaSuccess;
    *src = phi;
    return cudaMemcpyAsync(phi, dev_phi, bytes, cudaMemcpyDeviceToDevice, stream);
}

// Initial state into the buffers of state c from the phase fields src.
cudaError_t launch_initial_state(nlbm_sim *s, int c, const float *src)
{
    // init writes the populations of state c; kp.uin / kp.pin name the
    // other velocity / pressure buffers, zeroed as well
    StepParams kp = step_params(s, c ^ 1, c);
    kp.phi = s->phi(c);
    return launch_init(s->ns, kp, src, s->stream);
}

cudaError_t launch_step(const nlbm_sim *s, const StepParams &kp)
{
    const bool a = s->model == NLBM_MODEL_A;
    switch (s->storage) {
    case NLBM_STORE_BF16: return a ? launch_step_a_bf16(s->ns, kp, s->tx, s->ty, s->stream)
                                   : launch_step_b_bf16(s->ns, kp, s->tx, s->ty, s->stream);
    case NLBM_STORE_F16: return a ? launch_step_a_f16(s->ns, kp, s->tx, s->ty, s->stream)
                                  : launch_step_b_f16(s->ns, kp, s->tx, s->ty, s->stream);
    default: return a ? launch_step_a_f32(s->ns, kp, s->tx, s->ty, s->stream)
                      : launch_step_b_f32(s->ns, kp, s->tx, s->ty, s->stream);
    }
}

// A simulation in the workspace ws laid out as L (ws nullptr: without state).
nlbm_status make_sim(const nlbm_params *p, const StepParams &kp, char *ws, const Layout &L, void *cuda_stream,
                     nlbm_sim **out)
{
    nlbm_sim *s = new (std::nothrow) nlbm_sim();
    if (!s) { set_err(g_err, "host allocation failed"); return NLBM_ENOMEM; }
    s->kp = kp;
    s->N = p->n_phases;
    s->ns = p->n_phases - 1;
    s->model = p->model;
    s->storage = p->storage;
    s->plane = (size_t)p->nx * p->ny;
    s->stream = (cudaStream_t)cuda_stream;
    s->ws = ws;
    s->L = L;
    s->cur = 0;
    s->steps = 0;
    s->launches = 0;
    s->err[0] = 0;
    default_tile(s);
    *out = s;
    return NLBM_OK;
}

}  // namespace

extern "C" {

nlbm_status nlbm_workspace_bytes(const nlbm_params *p, size_t *bytes)
{
    if (!bytes) { set_err(g_err, "bytes is NULL"); return NLBM_EINVAL; }
    nlbm_status st = validate(p, nullptr, g_err);
    if (st != NLBM_OK) return st;
    *bytes = make_layout(p->n_phases - 1, (size_t)p->nx * p->ny, is_half(p->storage)).total;
    return NLBM_OK;
}

nlbm_status nlbm_create(const nlbm_params *p, void *dev_workspace, size_t workspace_bytes,
                        void *cuda_stream, nlbm_sim **out)
{
    if (!out) { set_err(g_err, "out is NULL"); return NLBM_EINVAL; }
    *out = nullptr;
    StepParams kp;
    nlbm_status st = validate(p, &kp, g_err);
    if (st != NLBM_OK) return st;
    const Layout L = make_layout(p->n_phases - 1, (size_t)p->nx * p->ny, is_half(p->storage));
    if (!dev_workspace) { set_err(g_err, "workspace is NULL"); return NLBM_EINVAL; }
    if (((uintptr_t)dev_workspace & 255) != 0) { set_err(g_err, "workspace must be 256-byte aligned"); return NLBM_EINVAL; }
    if (workspace_bytes < L.total) {
        set_err(g_err, "workspace of %zu bytes is smaller than the %zu needed", workspace_bytes, L.total);
        return NLBM_ENOMEM;
    }
    return make_sim(p, kp, (char *)dev_workspace, L, cuda_stream, out);
}

nlbm_status nlbm_set_phi(nlbm_sim *s, const float *dev_phi)
{
    if (!s || !dev_phi) return NLBM_EINVAL;
    const float *src;
    cudaError_t e = initial_fields(dev_phi, s->phi(s->cur), sizeof(float) * s->ns * s->plane, s->ws, s->L.total,
                                   s->stream, &src);
    if (e != cudaSuccess) return cuda_fail(s, e, "copy of the initial phase fields");
    e = launch_initial_state(s, s->cur, src);
    if (e != cudaSuccess) return cuda_fail(s, e, "init kernel");
    s->launches++;
    s->steps = 0;
    return NLBM_OK;
}

nlbm_status nlbm_set_phi_host(nlbm_sim *s, const float *host_phi)
{
    if (!s || !host_phi) return NLBM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(s->phi(s->cur), host_phi, sizeof(float) * s->ns * s->plane,
                                    cudaMemcpyHostToDevice, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "upload of the initial phase fields");
    // the device copy in the phi planes is its own source for the init kernel
    e = launch_initial_state(s, s->cur, s->phi(s->cur));
    if (e != cudaSuccess) return cuda_fail(s, e, "init kernel");
    s->launches++;
    s->steps = 0;
    return NLBM_OK;
}

nlbm_status nlbm_set_velocity(nlbm_sim *s, const float *dev_u)
{
    if (!s || !dev_u) return NLBM_EINVAL;
    if (s->half()) {
        set_err(s->err, "a state in motion is set for FP32 population storage only");
        return NLBM_ENOTSUP;
    }
    if (s->kp.wet) {
        set_err(s->err, "a state in motion is not set with wetting walls");
        return NLBM_ENOTSUP;
    }
    if (s->steps != 0) {
        set_err(s->err, "set the velocity after nlbm_set_phi and before the first step");
        return NLBM_EINVAL;
    }
    const int c = s->cur;
    // the populations of state c; u(c) becomes the first step's previous
    // velocity, and the other velocity buffer holds P' until the first step
    // overwrites it
    const StepParams kp = step_params(s, c ^ 1, c);
    cudaError_t e = launch_velocity_state(s->ns, s->model, kp, dev_u, s->u(c), s->u(c ^ 1), s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "velocity initial state");
    s->launches += 2;
    return NLBM_OK;
}

nlbm_status nlbm_step(nlbm_sim *s, int64_t nsteps)
{
    if (!s || nsteps < 0) return NLBM_EINVAL;
    for (int64_t k = 0; k < nsteps; ++k) {
        const int a = s->cur, b = s->cur ^ 1;
        StepParams kp = step_params(s, a, b);
        // FP32 storage writes P on the last step of a call only; 16-bit
        // storage needs it every step (the pullers add 3 w_i P back)
        if (!s->half() && k != nsteps - 1) kp.pout = nullptr;
        cudaError_t e = launch_step(s, kp);
        if (e != cudaSuccess) return cuda_fail(s, e, "step kernel");
        s->launches++;
        s->cur = b;
        s->steps++;
    }
    return NLBM_OK;
}

nlbm_status nlbm_get_moments(nlbm_sim *s, float *dev_phi, float *dev_u, float *dev_p)
{
    if (!s) return NLBM_EINVAL;
    if (!dev_phi && !dev_u && !dev_p) return NLBM_OK;
    cudaError_t e = launch_export(s->ns, s->phi(s->cur), s->u(s->cur), s->P(s->cur), (unsigned)s->plane,
                                  dev_phi, dev_u, dev_p, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "export kernel");
    s->launches++;
    return NLBM_OK;
}

nlbm_status nlbm_get_moments_host(nlbm_sim *s, float *host_phi, float *host_u, float *host_p)
{
    if (!s) return NLBM_EINVAL;
    if (!host_phi && !host_u && !host_p) return NLBM_OK;
    // Stage through the idle population buffers (rewritten by the next
    // step): N + 3 planes fit in one f copy and the g copy after it.
    const size_t pl = s->plane, pb = sizeof(float) * pl;
    float *stage = s->f(s->cur ^ 1);
    float *sphi = stage, *su = stage + (size_t)s->N * pl, *sp = su + 2 * pl;
    cudaError_t e = launch_export(s->ns, s->phi(s->cur), s->u(s->cur), s->P(s->cur), (unsigned)pl,
                                  host_phi ? sphi : nullptr, host_u ? su : nullptr,
                                  host_p ? sp : nullptr, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "export kernel");
    s->launches++;
    if (host_phi && (e = cudaMemcpyAsync(host_phi, sphi, pb * s->N, cudaMemcpyDeviceToHost, s->stream)) != cudaSuccess)
        return cuda_fail(s, e, "download of phi");
    if (host_u && (e = cudaMemcpyAsync(host_u, su, 2 * pb, cudaMemcpyDeviceToHost, s->stream)) != cudaSuccess)
        return cuda_fail(s, e, "download of u");
    if (host_p && (e = cudaMemcpyAsync(host_p, sp, pb, cudaMemcpyDeviceToHost, s->stream)) != cudaSuccess)
        return cuda_fail(s, e, "download of P");
    e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "synchronize");
    return NLBM_OK;
}

nlbm_status nlbm_phase_mass(nlbm_sim *s, double *host_mass)
{
    if (!s || !host_mass) return NLBM_EINVAL;
    double *partials = (double *)(s->ws + s->L.partials);
    double *mass = (double *)(s->ws + s->L.mass);
    int *flag = (int *)(mass + s->N);
    cudaError_t e = launch_phase_mass(s->ns, s->phi(s->cur), (unsigned)s->plane, partials, mass, flag, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "phase-mass kernels");
    s->launches += 2;
    double buf[kMaxPhases + 1];
    e = cudaMemcpyAsync(buf, mass, sizeof(double) * s->N + sizeof(int), cudaMemcpyDeviceToHost, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "download of the phase masses");
    e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "synchronize");
    memcpy(host_mass, buf, sizeof(double) * s->N);
    int fl = 0;
    memcpy(&fl, (const char *)buf + sizeof(double) * s->N, sizeof(int));
    if (fl) {
        set_err(s->err, "a phase field is non-finite or outside [-0.5, 1.5]");
        return NLBM_EDIVERGED;
    }
    return NLBM_OK;
}

nlbm_status nlbm_state_bytes(const nlbm_sim *s, size_t *bytes)
{
    if (!s || !bytes) return NLBM_EINVAL;
    *bytes = state_payload(s) + 16;
    return NLBM_OK;
}

nlbm_status nlbm_save(nlbm_sim *s, void *dev_dst)
{
    if (!s || !dev_dst || ((uintptr_t)dev_dst & 15)) return NLBM_EINVAL;
    char *d = (char *)dev_dst;
    const size_t pb = sizeof(float) * s->plane;
    const int c = s->cur;
    struct Part { const void *src; size_t n; } parts[] = {
        {s->f(c), s->L.fbytes}, {s->g(c), s->L.gbytes}, {s->f0(c), s->half() ? pb * s->ns : 0},
        {s->u(c), pb * 2}, {s->phi(c), pb * s->ns}, {s->mphi(), pb * 2}, {s->P(c), pb}};
    for (const Part &pt : parts) {
        if (!pt.n) continue;
        cudaError_t e = cudaMemcpyAsync(d, pt.src, pt.n, cudaMemcpyDeviceToDevice, s->stream);
        if (e != cudaSuccess) return cuda_fail(s, e, "checkpoint copy");
        d += pt.n;
    }
    int64_t counter[2] = {s->steps, 0x6e6c626d};   // step count and a tag
    cudaError_t e = cudaMemcpyAsync(d, counter, sizeof counter, cudaMemcpyHostToDevice, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "checkpoint counter");
    e = cudaStreamSynchronize(s->stream);   // counter is a host stack value
    if (e != cudaSuccess) return cuda_fail(s, e, "synchronize");
    return NLBM_OK;
}

nlbm_status nlbm_restore(nlbm_sim *s, const void *dev_src)
{
    if (!s || !dev_src || ((uintptr_t)dev_src & 15)) return NLBM_EINVAL;
    const char *d = (const char *)dev_src;
    const size_t pb = sizeof(float) * s->plane;
    s->cur = 0;
    struct Part { void *dst; size_t n; } parts[] = {
        {s->f(0), s->L.fbytes}, {s->g(0), s->L.gbytes}, {s->f0(0), s->half() ? pb * s->ns : 0},
        {s->u(0), pb * 2}, {s->phi(0), pb * s->ns}, {s->mphi(), pb * 2}, {s->P(0), pb}};
    for (const Part &pt : parts) {
        if (!pt.n) continue;
        cudaError_t e = cudaMemcpyAsync(pt.dst, d, pt.n, cudaMemcpyDeviceToDevice, s->stream);
        if (e != cudaSuccess) return cuda_fail(s, e, "restore copy");
        d += pt.n;
    }
    int64_t counter[2] = {0, 0};
    cudaError_t e = cudaMemcpyAsync(counter, d, sizeof counter, cudaMemcpyDeviceToHost, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "restore counter");
    e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "synchronize");
    if (counter[1] != 0x6e6c626d) {
        set_err(s->err, "checkpoint tag mismatch");
        return NLBM_EINVAL;
    }
    s->steps = counter[0];
    return NLBM_OK;
}

nlbm_status nlbm_synchronize(nlbm_sim *s)
{
    if (!s) return NLBM_EINVAL;
    cudaError_t e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "synchronize");
    return NLBM_OK;
}

int64_t nlbm_steps_done(const nlbm_sim *s) { return s ? s->steps : -1; }

int64_t nlbm_kernel_launches(const nlbm_sim *s) { return s ? s->launches : -1; }

nlbm_status nlbm_set_tile(nlbm_sim *s, int32_t tx, int32_t ty)
{
    if (!s) return NLBM_EINVAL;
    if ((tx != 64 && tx != 128 && tx != 256) || ty < 0) {
        set_err(s->err, "tile %dx%d outside tx in {64, 128, 256}, ty >= 0", tx, ty);
        return NLBM_EINVAL;
    }
    s->tx = tx;
    s->ty = ty;
    return NLBM_OK;
}

nlbm_status nlbm_get_tile(const nlbm_sim *s, int32_t *tx, int32_t *ty)
{
    if (!s || !tx || !ty) return NLBM_EINVAL;
    *tx = s->tx;
    *ty = s->ty;
    return NLBM_OK;
}

nlbm_status nlbm_autotune(nlbm_sim *s, void *dev_scratch, size_t scratch_bytes, int32_t steps_per_trial,
                          int32_t *best_tx, int32_t *best_ty, float *best_ms_per_step)
{
    if (!s || !dev_scratch || steps_per_trial < 1) return NLBM_EINVAL;
    const size_t need = state_payload(s) + 16;
    if (scratch_bytes < need) {
        set_err(s->err, "scratch of %zu bytes is smaller than the %zu of state", scratch_bytes, need);
        return NLBM_ENOMEM;
    }
    nlbm_status st = nlbm_save(s, dev_scratch);
    if (st != NLBM_OK) return st;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e;
    if ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return cuda_fail(s, e, "timing events");
    }
    // Trials: for every width that the lattice can fill (strips of tx - 4
    // columns) the explicit rows and the library's own choice, ty = 0, which
    // only a one-wave march makes depend on tx; where it is another form, the
    // one-wave march is tried by its rows.  16-bit storage has one shape.
    static const int kTx[] = {64, 128, 256};
    static const int kTy[] = {8, 12, 16, 20, 24, 32, 48};
    struct Trial { int tx, ty; } trials[3 * 9];
    int count = 0;
    bool seen[3] = {false, false, false};
    if (s->half()) {
        s->ty = 0;
        trials[count++] = Trial{s->tx, 0};
    }
    for (int tx : kTx) {
        if (s->half() || (tx > 64 && (tx / 2 - 4) >= s->kp.nx)) continue;
        StepForm form;
        int rows = 0;
        const StepParams kp = step_params(s, s->cur, s->cur ^ 1);
        e = (s->model == NLBM_MODEL_A ? step_form_a_f32 : step_form_b_f32)(s->ns, kp, tx, &form, &rows);
        if (e != cudaSuccess) { st = cuda_fail(s, e, "trial shapes"); break; }
        if (form == StepForm::OneWave || !seen[(int)form]) trials[count++] = Trial{tx, 0};
        seen[(int)form] = true;
        for (int ty : kTy) trials[count++] = Trial{tx, ty};
        if (form != StepForm::OneWave && rows > kTy[0] && std::find(std::begin(kTy), std::end(kTy), rows) == std::end(kTy))
            trials[count++] = Trial{tx, rows};
    }
    float best = 1e30f;
    int btx = s->tx, bty = s->ty;
    for (int i = 0; i < count && st == NLBM_OK; ++i) {
        s->tx = trials[i].tx;
        s->ty = trials[i].ty;
        for (int k = 0; k <= steps_per_trial && st == NLBM_OK; ++k) {
            if (k == 1 && (e = cudaEventRecord(e0, s->stream)) != cudaSuccess) st = cuda_fail(s, e, "event");
            StepParams kp = step_params(s, s->cur, s->cur ^ 1);
            if (!s->half()) kp.pout = nullptr;
            if (st == NLBM_OK && (e = launch_step(s, kp)) != cudaSuccess) st = cuda_fail(s, e, "trial step");
            s->launches++;
            s->cur ^= 1;
        }
        float ms = 0.f;
        if (st == NLBM_OK &&
            ((e = cudaEventRecord(e1, s->stream)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess ||
             (e = cudaEventElapsedTime(&ms, e0, e1)) != cudaSuccess))
            st = cuda_fail(s, e, "trial timing");
        if (st != NLBM_OK) break;
        ms /= steps_per_trial;
        if (ms < best) {
            best = ms;
            btx = s->tx;
            bty = s->ty;
        }
        st = nlbm_restore(s, dev_scratch);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    s->tx = btx;
    s->ty = bty;
    if (st != NLBM_OK) return st;
    if (best_tx) *best_tx = btx;
    if (best_ty) *best_ty = bty;
    if (best_ms_per_step) *best_ms_per_step = best;
    return NLBM_OK;
}

void nlbm_destroy(nlbm_sim *s) { delete s; }

}  // extern "C"

// ------------------------------------------------------------------ ensembles

struct nlbm_batch {
    int count, ns;
    std::vector<nlbm_sim *> sims;
    std::vector<size_t> sim_off;         // workspace offset of each simulation
    size_t state_begin, state_end;       // span of all simulations' state
    cudaStream_t stream;
    char *ws;
    StepParams *d_params;                // [4][count]: parity 0/1 x (no P / P)
    BatchTile *d_tiles;
    size_t max_tiles;
    int ntiles;
    int *d_counters;                     // [2]
    int cur;                             // state parity shared by every simulation
    int tx, ty;
    int px, rows;                        // the tiles they give, see choose_tiles()
    cudaGraphExec_t graph;               // two steps (parity 0 then 1), no P output
    bool graph_ok;
    int64_t steps, launches;
    char err[512];
};

namespace {

constexpr int kBatchMaxSims = 4096;

struct BatchLayout {
    size_t params, tiles, counters, sims_begin, total;
    size_t max_tiles;
    std::vector<size_t> sim_off;
};

// Largest number of tiles any allowed tile shape gives (tx = 64, ty = 1, or
// patches of 16 x 8 on a lattice of few rows).
size_t worst_tiles(const nlbm_params *p, int count)
{
    size_t t = 0;
    for (int k = 0; k < count; ++k)
        t += std::max((size_t)((p[k].nx + 59) / 60) * (size_t)p[k].ny,
                      (size_t)((p[k].nx + 15) / 16) * (size_t)((p[k].ny + 7) / 8));
    return t;
}

nlbm_status batch_layout(const nlbm_params *p, int count, BatchLayout *B, char *err)
{
    if (!p || count < 1 || count > kBatchMaxSims) {
        set_err(err, "count=%d outside 1..%d (or params NULL)", count, kBatchMaxSims);
        return NLBM_EINVAL;
    }
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align256(off + bytes);
        return o;
    };
    B->max_tiles = worst_tiles(p, count);
    B->params = take(sizeof(StepParams) * 4 * (size_t)count);
    B->tiles = take(sizeof(BatchTile) * B->max_tiles);
    B->counters = take(2 * sizeof(int));
    B->sims_begin = off;
    B->sim_off.resize(count);
    for (int k = 0; k < count; ++k) {
        nlbm_status st = validate(&p[k], nullptr, err);
        if (st != NLBM_OK) {
            char tmp[512];
            snprintf(tmp, sizeof tmp, "simulation %d: %s", k, err);
            memcpy(err, tmp, sizeof tmp);
            return st;
        }
        if (p[k].n_phases != p[0].n_phases) {
            set_err(err, "simulation %d has N=%d, simulation 0 N=%d: an ensemble shares N", k,
                    p[k].n_phases, p[0].n_phases);
            return NLBM_EINVAL;
        }
        if (p[k].storage != NLBM_STORE_F32) {
            set_err(err, "simulation %d: ensembles store FP32 populations", k);
            return NLBM_ENOTSUP;
        }
        B->sim_off[k] = take(make_layout(p[k].n_phases - 1, (size_t)p[k].nx * p[k].ny, false).total);
    }
    B->total = off;
    return NLBM_OK;
}

nlbm_status batch_fail(nlbm_batch *b, cudaError_t e, const char *what)
{
    set_err(b->err, "%s: %s", what, cudaGetErrorString(e));
    return NLBM_ECUDA;
}

// Tiles for the current tx and ty: px > 0 patches of px columns and 8 rows,
// px = 0 strips of tx - 4 columns marched down `rows` rows.
//
// ty = 8 with more than 64 threads: patches of those threads; other ty > 0: a
// march.  ty = 0: the library's choice, wide patches unless a march of 32
// rows costs less.  Patches win on small members, whose marches repeat their
// 6 pre-roll rows often and end in narrow strips (us a step, march 128 x 32 /
// best march / narrow / wide patches: 64 lenses of 512 x 256 to 128 x 64, N =
// 3, 228 / 215 / 233 / 195; 8 of them 78 / 44 / 38 / 33; 32 members N = 5 304 /
// 292 / 260 / 250; 16 members N = 8 413 / 331 / 253 / 242).  On large ones a
// march spends `gain` of a patch's time on a node of its tiles (strips padded
// to tx - 4 columns, 6 rows more a tile), and part of its last wave idles
// (N = 5, march / wide patches: 2 of 2048^2 713 / 790, 3 of 1536^2 625 / 673, 2
// of 1280^2 293 / 321, but 1 of 1536^2 274 / 232; N = 3: 4 of 2048^2 785 / 832,
// 1 of 2048^2 221 / 216).  Without row windows it gains less, and at N = 8
// nothing.  Over 160 ensembles of 0.4 to 17 million nodes at N = 2..8 the worse
// form is taken by at most 2.5 %, 5 % for 3 of 1536^2 at N = 2.
cudaError_t choose_tiles(nlbm_batch *b)
{
    b->px = b->ty == 8 && b->tx > 64 ? b->tx / 8 : 0;
    b->rows = b->ty;
    if (b->ty > 0) return cudaSuccess;
    static const double kGain[2][kMaxPhases - 1] = {{.91, 1., 1., .91, .91, .91, 1.}, {.88, .90, .89, .83, .90, .92, 1.}};
    const int W = b->tx - 4;
    double nodes = 0., march = 0., gain = 0.;
    long long tiles = 0;
    for (const nlbm_sim *s : b->sims) {
        const int strips = (s->kp.nx + W - 1) / W, chunks = (s->kp.ny + 31) / 32;
        const double g = kGain[row_windows(step_params(s, 0, 1))][b->ns - 1];
        nodes += (double)s->plane;
        march += g * strips * W * (s->kp.ny + 6. * chunks) * (32. / 38.);
        gain = std::max(gain, g);
        tiles += (long long)strips * chunks;
    }
    b->px = 32;
    b->rows = 8;
    if (march >= nodes) return cudaSuccess;
    int resident = 0, sms = 0;
    const cudaError_t e = batch_march_blocks(b->ns, b->tx, &resident, &sms);
    if (e != cudaSuccess) return e;
    const double idle = (double)((resident - tiles % resident) % resident);
    march += gain * std::min(0.68 * sms, sms / 6. + 0.5 * idle) * W * 32.;
    if (march < nodes) {
        b->px = 0;
        b->rows = 32;
    }
    return cudaSuccess;
}

// Tile table for the current tile shape: every strip and row chunk of every
// simulation, the largest simulations first (so the last tiles are small).
nlbm_status build_tiles(nlbm_batch *b)
{
    cudaError_t e = choose_tiles(b);
    if (e != cudaSuccess) return batch_fail(b, e, "choice of the tiles");
    const int W = b->px ? b->px : b->tx - 4;
    std::vector<int> order(b->count);
    for (int k = 0; k < b->count; ++k) order[k] = k;
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        return b->sims[a]->plane > b->sims[c]->plane;
    });
    std::vector<BatchTile> t;
    for (int k : order) {
        const nlbm_sim *s = b->sims[k];
        const int nx = s->kp.nx, ny = s->kp.ny;
        int ty = b->rows;
        if (ty > ny) ty = ny;
        for (int y0 = 0; y0 < ny; y0 += ty)
            for (int x0 = 0; x0 < nx; x0 += W) t.push_back(BatchTile{k, x0, y0, ty});
    }
    if (t.size() > b->max_tiles) {
        set_err(b->err, "tile table of %zu entries exceeds the %zu reserved", t.size(), b->max_tiles);
        return NLBM_EINVAL;
    }
    e = cudaMemcpyAsync(b->d_tiles, t.data(), sizeof(BatchTile) * t.size(), cudaMemcpyHostToDevice,
                                    b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);   // t is a host temporary
    if (e != cudaSuccess) return batch_fail(b, e, "upload of the tile table");
    b->ntiles = (int)t.size();
    b->graph_ok = false;
    return NLBM_OK;
}

nlbm_status upload_params(nlbm_batch *b)
{
    std::vector<StepParams> h(4 * (size_t)b->count);
    for (int par = 0; par < 2; ++par)
        for (int k = 0; k < b->count; ++k) {
            StepParams kp = step_params(b->sims[k], par, par ^ 1);
            kp.row_window = row_windows(kp);
            kp.pout = nullptr;
            h[(size_t)(2 * par) * b->count + k] = kp;
            kp.pout = b->sims[k]->P(0);
            h[(size_t)(2 * par + 1) * b->count + k] = kp;
        }
    cudaError_t e = cudaMemcpyAsync(b->d_params, h.data(), sizeof(StepParams) * h.size(), cudaMemcpyHostToDevice,
                                    b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return batch_fail(b, e, "upload of the parameter blocks");
    return NLBM_OK;
}

// One step of every simulation from state parity b->cur; with_p selects the
// parameter blocks that also write P.
cudaError_t batch_launch(nlbm_batch *b, int parity, bool with_p)
{
    const StepParams *tab = b->d_params + (size_t)(2 * parity + (with_p ? 1 : 0)) * b->count;
    if (b->px) return launch_batch_patches(b->ns, b->px, tab, b->d_tiles, b->ntiles, b->d_counters, parity, b->stream);
    return launch_batch_step(b->ns, b->tx, tab, b->d_tiles, b->ntiles, b->d_counters, parity, b->stream);
}

void sync_sims(nlbm_batch *b)
{
    for (nlbm_sim *s : b->sims) {
        s->cur = b->cur;
        s->steps = b->steps;
    }
}

nlbm_status capture_graph(nlbm_batch *b)
{
    if (b->graph_ok) return NLBM_OK;
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return batch_fail(b, e, "stream capture");
    cudaError_t e0 = batch_launch(b, 0, false);
    cudaError_t e1 = batch_launch(b, 1, false);
    e = cudaStreamEndCapture(b->stream, &g);
    if (e0 != cudaSuccess) e = e0;
    if (e == cudaSuccess && e1 != cudaSuccess) e = e1;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) return batch_fail(b, e, "graph of two ensemble steps");
    b->graph_ok = true;
    return NLBM_OK;
}

}  // namespace

extern "C" {

nlbm_status nlbm_batch_workspace_bytes(const nlbm_params *sims, int32_t count, size_t *bytes)
{
    if (!bytes) { set_err(g_err, "bytes is NULL"); return NLBM_EINVAL; }
    BatchLayout B;
    nlbm_status st = batch_layout(sims, count, &B, g_err);
    if (st != NLBM_OK) return st;
    *bytes = B.total;
    return NLBM_OK;
}

nlbm_status nlbm_batch_create(const nlbm_params *sims, int32_t count, void *dev_workspace, size_t workspace_bytes,
                              void *cuda_stream, nlbm_batch **out)
{
    if (!out) { set_err(g_err, "out is NULL"); return NLBM_EINVAL; }
    *out = nullptr;
    BatchLayout B;
    nlbm_status st = batch_layout(sims, count, &B, g_err);
    if (st != NLBM_OK) return st;
    if (!dev_workspace || ((uintptr_t)dev_workspace & 255)) {
        set_err(g_err, "workspace must be non-NULL and 256-byte aligned");
        return NLBM_EINVAL;
    }
    if (workspace_bytes < B.total) {
        set_err(g_err, "workspace of %zu bytes is smaller than the %zu needed", workspace_bytes, B.total);
        return NLBM_ENOMEM;
    }
    nlbm_batch *b = new (std::nothrow) nlbm_batch();
    if (!b) { set_err(g_err, "host allocation failed"); return NLBM_ENOMEM; }
    b->count = count;
    b->ns = sims[0].n_phases - 1;
    b->stream = (cudaStream_t)cuda_stream;
    b->ws = (char *)dev_workspace;
    b->d_params = (StepParams *)(b->ws + B.params);
    b->d_tiles = (BatchTile *)(b->ws + B.tiles);
    b->max_tiles = B.max_tiles;
    b->d_counters = (int *)(b->ws + B.counters);
    b->sim_off = B.sim_off;
    b->state_begin = B.sims_begin;
    b->state_end = B.total;
    b->cur = 0;
    b->tx = 128;
    b->ty = 0;
    b->graph = nullptr;
    b->graph_ok = false;
    b->steps = 0;
    b->launches = 0;
    b->err[0] = 0;
    for (int k = 0; k < count; ++k) {
        nlbm_sim *s = nullptr;
        const size_t need = make_layout(b->ns, (size_t)sims[k].nx * sims[k].ny, false).total;
        st = nlbm_create(&sims[k], b->ws + B.sim_off[k], need, cuda_stream, &s);
        if (st != NLBM_OK) {
            for (nlbm_sim *q : b->sims) delete q;
            delete b;
            return st;
        }
        b->sims.push_back(s);
    }
    cudaError_t e = cudaMemsetAsync(b->d_counters, 0, 2 * sizeof(int), b->stream);
    if (e != cudaSuccess) {
        set_err(g_err, "counter reset: %s", cudaGetErrorString(e));
        for (nlbm_sim *q : b->sims) delete q;
        delete b;
        return NLBM_ECUDA;
    }
    if ((st = upload_params(b)) != NLBM_OK || (st = build_tiles(b)) != NLBM_OK) {
        memcpy(g_err, b->err, sizeof b->err);
        for (nlbm_sim *q : b->sims) delete q;
        delete b;
        return st;
    }
    *out = b;
    return NLBM_OK;
}

nlbm_status nlbm_batch_set_phi(nlbm_batch *b, int32_t sim, const float *dev_phi)
{
    if (!b || sim < 0 || sim >= b->count || !dev_phi) return NLBM_EINVAL;
    nlbm_sim *s = b->sims[sim];
    s->cur = b->cur;
    nlbm_status st = nlbm_set_phi(s, dev_phi);
    b->launches++;
    if (st != NLBM_OK) memcpy(b->err, s->err, sizeof b->err);
    return st;
}

nlbm_status nlbm_batch_step(nlbm_batch *b, int64_t nsteps)
{
    if (!b || nsteps < 0) return NLBM_EINVAL;
    if (nsteps == 0) return NLBM_OK;
    int64_t k = 0;
    const bool use_graph = b->stream != nullptr && nsteps >= 3;
    cudaError_t e;
    if (use_graph) {
        if (b->cur == 1) {   // align to the graph's parity order
            if ((e = batch_launch(b, 1, false)) != cudaSuccess) return batch_fail(b, e, "ensemble step");
            b->launches++;
            b->cur = 0;
            ++k;
        }
        nlbm_status st = capture_graph(b);
        if (st != NLBM_OK) return st;
        for (; k + 2 < nsteps; k += 2) {
            if ((e = cudaGraphLaunch(b->graph, b->stream)) != cudaSuccess) return batch_fail(b, e, "graph launch");
            b->launches += 2;
        }
    }
    for (; k < nsteps; ++k) {
        if ((e = batch_launch(b, b->cur, k == nsteps - 1)) != cudaSuccess) return batch_fail(b, e, "ensemble step");
        b->launches++;
        b->cur ^= 1;
    }
    b->steps += nsteps;
    sync_sims(b);
    return NLBM_OK;
}

nlbm_status nlbm_batch_get_moments(nlbm_batch *b, int32_t sim, float *dev_phi, float *dev_u, float *dev_p)
{
    if (!b || sim < 0 || sim >= b->count) return NLBM_EINVAL;
    nlbm_sim *s = b->sims[sim];
    nlbm_status st = nlbm_get_moments(s, dev_phi, dev_u, dev_p);
    if (dev_phi || dev_u || dev_p) b->launches++;
    if (st != NLBM_OK) memcpy(b->err, s->err, sizeof b->err);
    return st;
}

nlbm_status nlbm_batch_phase_mass(nlbm_batch *b, int32_t sim, double *host_mass)
{
    if (!b || sim < 0 || sim >= b->count || !host_mass) return NLBM_EINVAL;
    nlbm_sim *s = b->sims[sim];
    nlbm_status st = nlbm_phase_mass(s, host_mass);
    b->launches += 2;
    if (st != NLBM_OK) memcpy(b->err, s->err, sizeof b->err);
    return st;
}

nlbm_status nlbm_batch_set_tile(nlbm_batch *b, int32_t tx, int32_t ty)
{
    if (!b) return NLBM_EINVAL;
    if ((tx != 64 && tx != 128 && tx != 256) || ty < 0) {
        set_err(b->err, "tile %dx%d outside tx in {64, 128, 256}, ty >= 0", tx, ty);
        return NLBM_EINVAL;
    }
    b->tx = tx;
    b->ty = ty;
    return build_tiles(b);
}

nlbm_status nlbm_batch_get_tile(const nlbm_batch *b, int32_t *tx, int32_t *ty, int32_t *ntiles)
{
    if (!b || !tx || !ty) return NLBM_EINVAL;
    *tx = b->tx;
    *ty = b->ty;
    if (ntiles) *ntiles = b->ntiles;
    return NLBM_OK;
}

nlbm_status nlbm_batch_state_bytes(const nlbm_batch *b, size_t *bytes)
{
    if (!b || !bytes) return NLBM_EINVAL;
    *bytes = b->state_end - b->state_begin;
    return NLBM_OK;
}

nlbm_status nlbm_batch_autotune(nlbm_batch *b, void *dev_scratch, size_t scratch_bytes, int32_t steps_per_trial,
                                int32_t *best_tx, int32_t *best_ty, float *best_ms_per_step)
{
    if (!b || !dev_scratch || steps_per_trial < 1) return NLBM_EINVAL;
    const size_t span = b->state_end - b->state_begin;
    if (scratch_bytes < span) {
        set_err(b->err, "scratch of %zu bytes is smaller than the %zu of state", scratch_bytes, span);
        return NLBM_ENOMEM;
    }
    char *state = b->ws + b->state_begin;
    const int cur0 = b->cur;
    cudaError_t e = cudaMemcpyAsync(dev_scratch, state, span, cudaMemcpyDeviceToDevice, b->stream);
    if (e != cudaSuccess) return batch_fail(b, e, "state copy");
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return batch_fail(b, e, "timing events");
    }
    static const int kTx[] = {64, 128, 256};
    static const int kTy[] = {8, 16, 32, 64, 128};
    float best = 1e30f;
    int btx = b->tx, bty = b->ty;
    nlbm_status st = NLBM_OK;
    for (int tx : kTx) {
        for (int ty : kTy) {
            b->tx = tx;
            b->ty = ty;
            if ((st = build_tiles(b)) != NLBM_OK) break;
            // one untimed step, then the timed ones, from the saved state
            for (int k = 0; k <= steps_per_trial && st == NLBM_OK; ++k) {
                if (k == 1 && (e = cudaEventRecord(e0, b->stream)) != cudaSuccess) st = batch_fail(b, e, "event");
                if (st == NLBM_OK && (e = batch_launch(b, b->cur, false)) != cudaSuccess)
                    st = batch_fail(b, e, "trial step");
                b->launches++;
                b->cur ^= 1;
            }
            if (st != NLBM_OK) break;
            float ms = 0.f;
            if ((e = cudaEventRecord(e1, b->stream)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess ||
                (e = cudaEventElapsedTime(&ms, e0, e1)) != cudaSuccess) {
                st = batch_fail(b, e, "trial timing");
                break;
            }
            ms /= steps_per_trial;
            if (ms < best) {
                best = ms;
                btx = tx;
                bty = ty;
            }
            // back to the saved state; the tile counters restart from zero
            // since the parity sequence is broken here
            b->cur = cur0;
            if ((e = cudaMemcpyAsync(state, dev_scratch, span, cudaMemcpyDeviceToDevice, b->stream)) != cudaSuccess ||
                (e = cudaMemsetAsync(b->d_counters, 0, 2 * sizeof(int), b->stream)) != cudaSuccess) {
                st = batch_fail(b, e, "state restore");
                break;
            }
        }
        if (st != NLBM_OK) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->cur = cur0;
    if (st == NLBM_OK) {   // state restored after the last trial
        b->tx = btx;
        b->ty = bty;
        st = build_tiles(b);
    }
    if (st == NLBM_OK && (e = cudaStreamSynchronize(b->stream)) != cudaSuccess) st = batch_fail(b, e, "synchronize");
    if (st != NLBM_OK) return st;
    if (best_tx) *best_tx = btx;
    if (best_ty) *best_ty = bty;
    if (best_ms_per_step) *best_ms_per_step = best;
    return NLBM_OK;
}

nlbm_status nlbm_batch_synchronize(nlbm_batch *b)
{
    if (!b) return NLBM_EINVAL;
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return batch_fail(b, e, "synchronize");
    return NLBM_OK;
}

int64_t nlbm_batch_steps_done(const nlbm_batch *b) { return b ? b->steps : -1; }

int64_t nlbm_batch_kernel_launches(const nlbm_batch *b) { return b ? b->launches : -1; }

void nlbm_batch_destroy(nlbm_batch *b)
{
    if (!b) return;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    for (nlbm_sim *s : b->sims) delete s;
    delete b;
}

const char *nlbm_batch_last_error(const nlbm_batch *b) { return b ? b->err : g_err; }

}  // extern "C"

// ------------------------------------------------------------------- adjoint

struct nlbm_adjoint {
    nlbm_sim *sim;             // parameters, tile and launch count of the steps (no state of its own)
    int ns, N, nsteps, every, nckpt;
    size_t plane, state_floats;
    cudaStream_t stream;
    char *ws;
    size_t ws_bytes, sums_bytes;
    float *ckpt;               // [nckpt][state]
    float *seg;                // [every + 1][state]
    float *tapes;              // [every][tape] the rebuilt segment's tapes
    AdjTape T;                 // the tape of nlbm_adjoint_reverse_step
    float *seed[2];            // two sets of step-output adjoints
    AdjFields A;               // intermediates (the seed pointers are set per step)
    double *partials, *acc;    // [kAdjRedBlocks][NP+1], [NP+1]
    float *seed_buf;           // [N][plane] copy of the caller's dL/dphi(T)
    float *grad_buf;           // [N-1][plane] dL/dphi_0
    int taped;                 // segment whose states and tapes seg / tapes hold, -1: none
    int unswept;               // forwards since the last sweep, counted to kUnswept
    // the whole reverse sweep as a graph: [0] from the last segment's tapes
    // that forward kept, captured on first use; [1] rebuilding them, captured
    // on second use (a handle often needs that sweep once or never)
    cudaGraphExec_t graph[2];
    int sweeps[2];
    bool forward_done;
    char err[512];
};

namespace {

constexpr int kUnswept = 3;   // see nlbm_adjoint_forward()

// State of a simulation between steps: f [9 NS], g [8], u [2], phi [NS],
// m_phi [2] planes (FP32 storage).
size_t adj_state_floats(int ns, size_t plane) { return plane * ((size_t)ns * 9 + 8 + 2 + ns + 2); }

// Planes of a step's tape in a sweep, of one seed set and of the
// intermediates, and values of the parameter gradient (the tensions, M).
struct AdjCounts {
    int tape, seedset, inter, params;
};

AdjCounts adj_counts(int ns)
{
    return AdjCounts{8 * ns + 12, 10 * ns + 12, 9 * ns + 12, (ns + 1) * ns / 2 + 1};
}

struct AdjLayout {
    size_t ckpt, seg, tapes, fields, sums, partials, acc, total;
    size_t sums_bytes;   // FP64 sums of the parameter gradient, one a block of the reverse passes
};

nlbm_status adj_layout(const nlbm_params *p, int nsteps, int every, AdjLayout *L, char *err)
{
    nlbm_status st = validate(p, nullptr, err);
    if (st != NLBM_OK) return st;
    bool wet = false;
    for (int a = 0; p->wall_cos && a < 2 * (p->n_phases - 1); ++a) wet = wet || p->wall_cos[a] != 0.0;
    if (p->storage != NLBM_STORE_F32 || wet) {
        set_err(err, "the adjoint covers FP32 storage and walls without wetting (contact angles of 90 degrees)");
        return NLBM_ENOTSUP;
    }
    if (nsteps < 1 || every < 1) { set_err(err, "nsteps and checkpoint interval must be >= 1"); return NLBM_EINVAL; }
    const int ns = p->n_phases - 1;
    const size_t plane = (size_t)p->nx * p->ny;
    const int nckpt = (nsteps + every - 1) / every;
    const AdjCounts c = adj_counts(ns);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align256(off + bytes);
        return o;
    };
    L->ckpt = take(sizeof(float) * adj_state_floats(ns, plane) * nckpt);
    // a segment's states and one spare (the output of its last step), and
    // the tape of each of its steps
    const size_t seglen = (size_t)(every < nsteps ? every : nsteps);
    L->seg = take(sizeof(float) * adj_state_floats(ns, plane) * (seglen + 1));
    L->tapes = take(sizeof(float) * plane * (size_t)c.tape * seglen);
    // (a single reverse step's tape has one plane more, w)
    L->fields = take(sizeof(float) * plane * (size_t)(c.tape + 1 + 2 * c.seedset + c.inter + 2 * ns + 1));
    L->sums_bytes = sizeof(double) * c.params * (size_t)adj_sum_blocks(p->nx, p->ny);
    L->sums = take(L->sums_bytes);
    L->partials = take(sizeof(double) * kAdjRedBlocks * c.params);
    L->acc = take(sizeof(double) * c.params);
    L->total = off;
    return NLBM_OK;
}

nlbm_status adj_fail(nlbm_adjoint *a, cudaError_t e, const char *what)
{
    set_err(a->err, "%s: %s", what, cudaGetErrorString(e));
    return NLBM_ECUDA;
}

// Step parameters whose inputs are a packed state record.
StepParams adj_params_from_state(const nlbm_adjoint *a, const float *state)
{
    StepParams kp = a->sim->kp;
    const size_t pl = a->plane;
    kp.fin = state;
    kp.gin = state + pl * 9 * a->ns;
    kp.uin = kp.gin + pl * 8;
    kp.phi_prev = kp.uin + pl * 2;
    kp.mphi = const_cast<float *>(kp.phi_prev + pl * a->ns);
    kp.mphi_in = kp.mphi;
    return kp;
}

// One forward step from one packed state record to another; tape: also the
// step's intermediate fields.
cudaError_t adj_step(nlbm_adjoint *a, const float *in, float *out, float *tape)
{
    const size_t pl = a->plane;
    const int ns = a->ns;
    StepParams kp = adj_params_from_state(a, in);
    kp.fout = out;
    kp.gout = out + pl * 9 * ns;
    kp.uout = kp.gout + pl * 8;
    kp.phi = kp.uout + pl * 2;
    kp.mphi = kp.phi + pl * ns;   // read from the input state, written to the output
    kp.pout = nullptr;
    kp.tape = tape;
    if (!tape) return launch_step(a->sim, kp);
    return (kp.model == NLBM_MODEL_A ? launch_step_tape_a_f32 : launch_step_tape_b_f32)(ns, kp, a->stream);
}

// Input state of step s (0-based) of segment k: the checkpoint, then the
// states that the segment's own steps wrote.
float *adj_segment_state(const nlbm_adjoint *a, int k, int s)
{
    return s == 0 ? a->ckpt + a->state_floats * k : a->seg + a->state_floats * s;
}

int adj_segment_length(const nlbm_adjoint *a, int k)
{
    return (k + 1) * a->every <= a->nsteps ? a->every : a->nsteps - k * a->every;
}

// `steps` steps from checkpoint k without tapes, through the first two slots
// of the segment's states or, the last one, into `end` if given; returns
// where that one was written.
cudaError_t adj_run_segment(nlbm_adjoint *a, int k, int steps, float *end, const float **last)
{
    const float *in = a->ckpt + a->state_floats * k;
    for (int t = 0; t < steps; ++t) {
        float *out = end && t + 1 == steps ? end : a->seg + a->state_floats * (t & 1);
        const cudaError_t e = adj_step(a, in, out, nullptr);
        if (e != cudaSuccess) return e;
        in = out;
    }
    *last = in;
    return cudaSuccess;
}

// The states and tapes of segment k from its checkpoint: one taping step
// launch per step (the last step's output state goes to the spare slot).
cudaError_t adj_tape_segment(nlbm_adjoint *a, int k)
{
    const size_t tape = a->plane * (size_t)adj_counts(a->ns).tape;
    const int len = adj_segment_length(a, k);
    for (int s = 0; s < len; ++s) {
        const cudaError_t e =
            adj_step(a, adj_segment_state(a, k, s), a->seg + a->state_floats * (s + 1), a->tapes + tape * s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Adjoint-field pointers for a step whose output adjoints are seed set so
// and input adjoints seed set si.
AdjFields adj_fields(const nlbm_adjoint *a, float *so, float *si)
{
    const size_t pl = a->plane;
    const int ns = a->ns;
    AdjFields A = a->A;
    A.lf_out = so;
    A.lg_out = so + pl * 9 * ns;
    A.lphi_out = A.lg_out + pl * 8;
    A.lu_out = A.lphi_out + pl * ns;
    A.lm_out = A.lu_out + pl * 2;
    A.lf_in = si;
    A.lg_in = si + pl * 9 * ns;
    A.lphi_in = A.lg_in + pl * 8;
    A.lu_in = A.lphi_in + pl * ns;
    A.lm_in = A.lu_in + pl * 2;
    return A;
}

// Tape k of the segment (the field order of launch_step_tape_{a,b}_f32).
AdjTape adj_tape(const nlbm_adjoint *a, int k)
{
    const size_t pl = a->plane;
    const int ns = a->ns;
    float *b = a->tapes + pl * (size_t)adj_counts(ns).tape * k;
    AdjTape T;
    T.phi = b;
    T.j = b + pl * ns;
    T.g = b + pl * 3 * ns;
    T.grad = b + pl * (3 * ns + 8);
    T.lap = b + pl * (5 * ns + 8);
    T.R = b + pl * (6 * ns + 8);
    T.mphi = b + pl * (8 * ns + 8);
    T.w = nullptr;
    T.F = b + pl * (8 * ns + 10);
    return T;
}

// Kernel launches of one reverse sweep (counted, not queried).
int64_t adj_sweep_launches(const nlbm_adjoint *a, bool rebuild_last)
{
    // fold + per step: 2 reverse kernels and, unless forward has kept the
    // last segment's tapes, one taping step kernel while its segment is
    // rebuilt; the phi0 sum and the two-kernel reduction
    const int64_t kept = rebuild_last ? 0 : adj_segment_length(a, a->nckpt - 1);
    return 1 + 3 * (int64_t)a->nsteps - kept + 1 + 2;
}

// The reverse sweep, asynchronous and capturable: seeds from seed_buf,
// dL/dphi_0 into grad_buf, dL/dsigma and dL/dM into acc.
cudaError_t adj_backward_body(nlbm_adjoint *a, bool rebuild_last)
{
    const size_t pl = a->plane, pb = sizeof(float) * pl;
    const int ns = a->ns, np = (ns + 1) * ns / 2, blocks = adj_sum_blocks(a->sim->kp.nx, a->sim->kp.ny);
    cudaError_t e;
    // No step follows the last: what its first pass gathers (the adjoints of
    // j and of the pulled g in the seed set, of phi in lphi_tot) is 0, and so
    // are the seeds of u and m_phi.
    if ((e = cudaMemsetAsync(a->seed[0], 0, pb * (2 * ns + 8), a->stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a->seed[0] + pl * (10 * ns + 8), 0, pb * 4, a->stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a->A.lphi_tot, 0, pb * ns, a->stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a->A.gacc, 0, a->sums_bytes, a->stream)) != cudaSuccess) return e;
    if ((e = launch_fold_seed(ns, a->seed_buf, (unsigned)pl, a->seed[0] + pl * (9 * ns + 8), a->stream)) != cudaSuccess)
        return e;
    int cur = 0;
    for (int k = a->nckpt - 1; k >= 0; --k) {
        if ((k < a->nckpt - 1 || rebuild_last) && (e = adj_tape_segment(a, k)) != cudaSuccess) return e;
        for (int s = adj_segment_length(a, k) - 1; s >= 0; --s) {
            const StepParams kp = adj_params_from_state(a, adj_segment_state(a, k, s));
            AdjFields A = adj_fields(a, a->seed[cur], a->seed[cur ^ 1]);
            // the sweep's seed sets hold j and pulled g adjoints (2 ns + 8
            // planes) where a single step's hold those of the populations
            A.lj_next = a->seed[cur];
            A.lg_next = a->seed[cur] + 2 * ns * pl;
            A.lj = a->seed[cur ^ 1];
            A.lg_pull = a->seed[cur ^ 1] + 2 * ns * pl;
            if ((e = launch_reverse_step(ns, kp, adj_tape(a, s), A, true, a->stream)) != cudaSuccess) return e;
            cur ^= 1;
        }
    }
    // phi0 entered step 1 as its pulled phase populations (f_i = w_i phi0,
    // so the adjoint is that of phi) and as its phi_prev
    const float *lphi_in = a->seed[cur] + pl * (9 * ns + 8);
    if ((e = launch_add_planes(a->A.lphi_tot, lphi_in, (unsigned)(pl * ns), a->grad_buf, a->stream)) != cudaSuccess)
        return e;
    return launch_grad_reduce(a->A.gacc, np + 1, (unsigned)blocks, a->partials, a->acc, a->stream);
}

}  // namespace

extern "C" {

nlbm_status nlbm_adjoint_workspace_bytes(const nlbm_params *p, int32_t nsteps, int32_t checkpoint_every,
                                         size_t *bytes)
{
    if (!bytes) { set_err(g_err, "bytes is NULL"); return NLBM_EINVAL; }
    AdjLayout L;
    nlbm_status st = adj_layout(p, nsteps, checkpoint_every, &L, g_err);
    if (st != NLBM_OK) return st;
    *bytes = L.total;
    return NLBM_OK;
}

nlbm_status nlbm_adjoint_create(const nlbm_params *p, int32_t nsteps, int32_t checkpoint_every, void *dev_workspace,
                                size_t workspace_bytes, void *cuda_stream, nlbm_adjoint **out)
{
    if (!out) { set_err(g_err, "out is NULL"); return NLBM_EINVAL; }
    *out = nullptr;
    AdjLayout L;
    nlbm_status st = adj_layout(p, nsteps, checkpoint_every, &L, g_err);
    if (st != NLBM_OK) return st;
    if (!dev_workspace || ((uintptr_t)dev_workspace & 255)) {
        set_err(g_err, "workspace must be non-NULL and 256-byte aligned");
        return NLBM_EINVAL;
    }
    if (workspace_bytes < L.total) {
        set_err(g_err, "workspace of %zu bytes is smaller than the %zu needed", workspace_bytes, L.total);
        return NLBM_ENOMEM;
    }
    nlbm_adjoint *a = new (std::nothrow) nlbm_adjoint();
    if (!a) { set_err(g_err, "host allocation failed"); return NLBM_ENOMEM; }
    char *ws = (char *)dev_workspace;
    StepParams kp;
    st = validate(p, &kp, g_err);
    if (st == NLBM_OK) st = make_sim(p, kp, nullptr, Layout{}, cuda_stream, &a->sim);
    if (st != NLBM_OK) {
        delete a;
        return st;
    }
    a->ns = p->n_phases - 1;
    a->N = p->n_phases;
    a->nsteps = nsteps;
    a->every = checkpoint_every;
    a->nckpt = (nsteps + checkpoint_every - 1) / checkpoint_every;
    a->plane = (size_t)p->nx * p->ny;
    a->state_floats = adj_state_floats(a->ns, a->plane);
    a->stream = (cudaStream_t)cuda_stream;
    a->ws = ws;
    a->ws_bytes = L.total;
    a->ckpt = (float *)(ws + L.ckpt);
    a->seg = (float *)(ws + L.seg);
    a->tapes = (float *)(ws + L.tapes);
    const AdjCounts c = adj_counts(a->ns);
    const size_t pl = a->plane;
    float *f = (float *)(ws + L.fields);
    auto take = [&](int planes) {
        float *q = f;
        f += (size_t)planes * pl;
        return q;
    };
    const int ns = a->ns;
    a->T.phi = take(ns);
    a->T.j = take(2 * ns);
    a->T.g = take(8);
    a->T.grad = take(2 * ns);
    a->T.lap = take(ns);
    a->T.R = take(2 * ns);
    a->T.mphi = take(2);
    a->T.w = take(1);
    a->T.F = take(2);
    a->seed[0] = take(c.seedset);
    a->seed[1] = take(c.seedset);
    a->A.lF = take(2);
    a->A.lphi_pw = take(ns);
    a->A.lj = take(2 * ns);
    a->A.lgrad = take(2 * ns);
    a->A.llap = take(ns);
    a->A.lR = take(2 * ns);
    a->A.lmphi = take(2);
    a->A.lg_pull = take(8);
    a->A.lphi_tot = take(ns);
    a->seed_buf = take(ns + 1);
    a->grad_buf = take(ns);
    a->A.gacc = (double *)(ws + L.sums);
    a->sums_bytes = L.sums_bytes;
    a->partials = (double *)(ws + L.partials);
    a->acc = (double *)(ws + L.acc);
    a->taped = -1;
    a->unswept = 0;
    a->forward_done = false;
    a->err[0] = 0;
    *out = a;
    return NLBM_OK;
}

nlbm_status nlbm_adjoint_forward(nlbm_adjoint *a, const float *dev_phi0, float *dev_phi_final)
{
    if (!a || !dev_phi0) return NLBM_EINVAL;
    nlbm_sim *s = a->sim;
    // The initial state is written as the first checkpoint; from there on a
    // step reads one packed record and writes the next, every segment's last
    // step straight into the next checkpoint.  The last segment runs the
    // taping kernel, as its states and tapes are the first that a sweep needs,
    // until kUnswept forwards in a row were not followed by one.  Taping every
    // step costs a forward 25 to 40 % (1024^2, us a step: N = 2 42 -> 60, N = 3
    // 55 -> 76, N = 5 96 -> 121) and saves the sweep as much as the taped
    // forward takes, so that a few of them unread (a line search) still pay.
    const size_t pl = a->plane;
    const int ns = a->ns, last = a->nckpt - 1;
    StepParams kp = adj_params_from_state(a, a->ckpt);
    kp.fout = a->ckpt;
    kp.gout = a->ckpt + pl * 9 * ns;
    kp.uout = kp.gout + pl * 8;
    kp.uin = kp.uout;             // one velocity buffer in a record
    kp.phi = kp.uout + pl * 2;
    kp.pout = a->A.lF;            // the initial pressure is no part of it: into a plane of the sweep's
    const float *src;
    cudaError_t e = initial_fields(dev_phi0, kp.phi, sizeof(float) * pl * ns, a->ws, a->ws_bytes, a->stream, &src);
    if (e != cudaSuccess) return adj_fail(a, e, "copy of the initial phase fields");
    e = launch_init(ns, kp, src, a->stream);
    if (e != cudaSuccess) return adj_fail(a, e, "initial state");
    s->launches++;
    a->forward_done = false;
    a->taped = -1;
    const bool tape = a->unswept < kUnswept;
    a->unswept += tape;
    const float *end;
    for (int k = 0; k < last; ++k)
        if ((e = adj_run_segment(a, k, a->every, a->ckpt + a->state_floats * (k + 1), &end)) != cudaSuccess)
            return adj_fail(a, e, "forward step");
    const int len = adj_segment_length(a, last);
    e = tape ? adj_tape_segment(a, last) : adj_run_segment(a, last, len, nullptr, &end);
    if (e != cudaSuccess) return adj_fail(a, e, "forward step");
    if (tape) {
        end = a->seg + a->state_floats * len;
        a->taped = last;
    }
    s->launches += a->nsteps;
    if (dev_phi_final) {
        e = launch_export(ns, end + pl * (9 * ns + 10), nullptr, nullptr, (unsigned)pl, dev_phi_final, nullptr, nullptr,
                          a->stream);
        if (e != cudaSuccess) return adj_fail(a, e, "export kernel");
        s->launches++;
    }
    a->forward_done = true;
    return NLBM_OK;
}

nlbm_status nlbm_adjoint_backward(nlbm_adjoint *a, const float *dev_seed, float *dev_grad_phi0,
                                  double *host_grad_sigma, double *host_grad_mobility)
{
    if (!a || !dev_seed) return NLBM_EINVAL;
    if (!a->forward_done) { set_err(a->err, "backward before forward"); return NLBM_EINVAL; }
    const size_t pl = a->plane, pb = sizeof(float) * pl;
    const int ns = a->ns, N = a->N, np = N * (N - 1) / 2;
    const AdjCounts c = adj_counts(ns);
    cudaError_t e = cudaMemcpyAsync(a->seed_buf, dev_seed, pb * N, cudaMemcpyDeviceToDevice, a->stream);
    if (e != cudaSuccess) return adj_fail(a, e, "seed copy");
    // After a forward that taped, and after one that did not or for another
    // sweep of the same forward, the sweep is one sequence of launches each
    // on every call of this handle: captured into a CUDA graph (on a
    // capturable stream) and replayed (256^2 N = 3, another sweep of 20 steps,
    // launched / replayed: 26.2 / 24.8 us a step).
    const bool rebuild_last = a->taped != a->nckpt - 1;
    const int kind = rebuild_last ? 1 : 0;
    if (!a->graph[kind] && a->sweeps[kind] == kind && a->stream != nullptr) {
        cudaGraph_t g = nullptr;
        if (cudaStreamBeginCapture(a->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            cudaError_t eb = adj_backward_body(a, rebuild_last);
            cudaError_t ec = cudaStreamEndCapture(a->stream, &g);
            if (eb == cudaSuccess && ec == cudaSuccess && cudaGraphInstantiate(&a->graph[kind], g, 0) != cudaSuccess)
                a->graph[kind] = nullptr;
            if (g) cudaGraphDestroy(g);
        }
        cudaGetLastError();   // a failed capture leaves the direct path
    }
    a->sweeps[kind] += a->sweeps[kind] <= kind;   // counted as far as it matters
    a->unswept = 0;
    a->taped = -1;
    if (a->graph[kind]) {
        e = cudaGraphLaunch(a->graph[kind], a->stream);
        if (e != cudaSuccess) return adj_fail(a, e, "graph launch");
    } else if ((e = adj_backward_body(a, rebuild_last)) != cudaSuccess) {
        return adj_fail(a, e, "reverse sweep");
    }
    a->taped = 0;   // the segment that the sweep ends with
    a->sim->launches += adj_sweep_launches(a, rebuild_last);
    if (dev_grad_phi0 &&
        (e = cudaMemcpyAsync(dev_grad_phi0, a->grad_buf, pb * ns, cudaMemcpyDeviceToDevice, a->stream)) != cudaSuccess)
        return adj_fail(a, e, "phi0 gradient");
    double acc[kMaxPhases * kMaxPhases + 1];
    if ((e = cudaMemcpyAsync(acc, a->acc, sizeof(double) * (np + 1), cudaMemcpyDeviceToHost, a->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(a->stream)) != cudaSuccess)
        return adj_fail(a, e, "gradient download");
    (void)c;
    if (host_grad_sigma) {
        for (int i = 0; i < N * N; ++i) host_grad_sigma[i] = 0.0;
        int q = 0;
        for (int i = 0; i < N; ++i)
            for (int j = i + 1; j < N; ++j, ++q) host_grad_sigma[i * N + j] = host_grad_sigma[j * N + i] = acc[q];
    }
    if (host_grad_mobility) *host_grad_mobility = acc[np];
    return NLBM_OK;
}

nlbm_status nlbm_adjoint_reverse_step(nlbm_adjoint *a, const float *dev_state, const float *dev_seed_out,
                                      float *dev_seed_in, double *host_grad_sigma, double *host_grad_mobility)
{
    if (!a || !dev_state || !dev_seed_out || !dev_seed_in) return NLBM_EINVAL;
    const size_t pl = a->plane, pb = sizeof(float) * pl;
    const int ns = a->ns, N = a->N, np = N * (N - 1) / 2;
    const AdjCounts c = adj_counts(ns);
    cudaError_t e;
    if ((e = cudaMemcpyAsync(a->seed[0], dev_seed_out, pb * c.seedset, cudaMemcpyDeviceToDevice, a->stream)) != cudaSuccess ||
        (e = cudaMemsetAsync(a->A.gacc, 0, a->sums_bytes, a->stream)) != cudaSuccess)
        return adj_fail(a, e, "seed");
    const StepParams kp = adj_params_from_state(a, dev_state);
    if ((e = launch_reverse_step(ns, kp, a->T, adj_fields(a, a->seed[0], a->seed[1]), false, a->stream)) != cudaSuccess ||
        (e = launch_grad_reduce(a->A.gacc, np + 1, (unsigned)adj_sum_blocks(kp.nx, kp.ny), a->partials, a->acc, a->stream)) != cudaSuccess)
        return adj_fail(a, e, "reverse step");
    a->sim->launches += 8;
    double acc[kMaxPhases * kMaxPhases + 1];
    if ((e = cudaMemcpyAsync(dev_seed_in, a->seed[1], pb * c.seedset, cudaMemcpyDeviceToDevice, a->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync(acc, a->acc, sizeof(double) * (np + 1), cudaMemcpyDeviceToHost, a->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(a->stream)) != cudaSuccess)
        return adj_fail(a, e, "reverse step results");
    if (host_grad_sigma) {
        for (int i = 0; i < N * N; ++i) host_grad_sigma[i] = 0.0;
        int q = 0;
        for (int i = 0; i < N; ++i)
            for (int j = i + 1; j < N; ++j, ++q) host_grad_sigma[i * N + j] = host_grad_sigma[j * N + i] = acc[q];
    }
    if (host_grad_mobility) *host_grad_mobility = acc[np];
    return NLBM_OK;
}

int32_t nlbm_adjoint_uses_graph(const nlbm_adjoint *a) { return a && (a->graph[0] || a->graph[1]) ? 1 : 0; }

int64_t nlbm_adjoint_kernel_launches(const nlbm_adjoint *a) { return a ? a->sim->launches : -1; }

void nlbm_adjoint_destroy(nlbm_adjoint *a)
{
    if (!a) return;
    for (cudaGraphExec_t g : a->graph)
        if (g) cudaGraphExecDestroy(g);
    nlbm_destroy(a->sim);
    delete a;
}

const char *nlbm_adjoint_last_error(const nlbm_adjoint *a) { return a ? a->err : g_err; }

}  // extern "C"

extern "C" {

const char *nlbm_last_error(const nlbm_sim *s) { return s ? s->err : g_err; }

const char *nlbm_status_string(nlbm_status st)
{
    switch (st) {
    case NLBM_OK: return "ok";
    case NLBM_EINVAL: return "invalid argument";
    case NLBM_ENOMEM: return "insufficient memory";
    case NLBM_ECUDA: return "CUDA error";
    case NLBM_ENOTSUP: return "not supported";
    case NLBM_EDIVERGED: return "diverged";
    default: return "unknown status";
    }
}

}  // extern "C"
