// gl_capi.cu -- host implementation of the C ABI declared in include/gl_map.h:
// argument validation, device-memory ownership, the keyframe store, and the
// sequencing of the kernels of one optimisation step on the map's stream.
#include <cuda.h>   // types only: the driver's entry points are looked up at run time
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "gl_internal.h"

struct gl_ctx {
    gl::gl_ctx_impl impl;
};

namespace gl {

namespace {
thread_local std::string g_err;
}

void set_error(const std::string& msg) { g_err = msg; }

namespace {
std::atomic<int64_t> g_launches{0};
const char* kPhaseNames[PH_COUNT] = {"preprocess", "depth_sort", "scan_duplicate", "tile_sort",
                                     "tile_ranges", "raster_forward", "loss", "raster_backward",
                                     "params_adam", "expand"};
}

void count_launches(int64_t n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

namespace {
constexpr int kMaxDev = 64;
std::mutex g_dev_mu;
int g_sms[kMaxDev] = {};
struct SmemLimit { const void* fn; int dev; int bytes; };
std::vector<SmemLimit> g_smem;
}

int sm_count()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return 152;
    }
    std::lock_guard<std::mutex> lk(g_dev_mu);
    if (!g_sms[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 152;
        }
        g_sms[dev] = n;
    }
    return g_sms[dev];
}

gl_status ensure_smem_limit(const void* fn, int bytes)
{
    int dev = 0;
    GL_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_dev_mu);
    for (const SmemLimit& e : g_smem)
        if (e.fn == fn && e.dev == dev && e.bytes >= bytes) return GL_OK;
    GL_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    g_smem.push_back({fn, dev, bytes});
    return GL_OK;
}

cudaEvent_t Prof::begin(cudaStream_t s)
{
    cudaEvent_t e;
    if (npool > 0) e = pool[--npool];
    else if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    cudaEventRecord(e, s);
    return e;
}

void Prof::end(int phase, cudaEvent_t a, cudaStream_t s)
{
    cudaEvent_t b;
    if (npool > 0) b = pool[--npool];
    else if (cudaEventCreate(&b) != cudaSuccess) return;
    cudaEventRecord(b, s);
    if (npend == cap) {
        int nc = cap ? 2 * cap : 256;
        Pending* np = static_cast<Pending*>(realloc(pend, sizeof(Pending) * nc));
        if (!np) return;
        pend = np;
        cap = nc;
    }
    pend[npend++] = Pending{phase, a, b};
}

void Prof::harvest()
{
    for (int i = 0; i < npend; i++) {
        float t = 0.f;
        cudaEventSynchronize(pend[i].b);
        if (cudaEventElapsedTime(&t, pend[i].a, pend[i].b) == cudaSuccess) {
            ms[pend[i].phase] += t;
            calls[pend[i].phase] += 1;
        }
        for (cudaEvent_t e : {pend[i].a, pend[i].b}) {
            if (npool == poolcap) {
                int nc = poolcap ? 2 * poolcap : 512;
                cudaEvent_t* np = static_cast<cudaEvent_t*>(realloc(pool, sizeof(cudaEvent_t) * nc));
                if (!np) { cudaEventDestroy(e); continue; }
                pool = np;
                poolcap = nc;
            }
            pool[npool++] = e;
        }
    }
    npend = 0;
}

void Prof::reset()
{
    harvest();
    for (int i = 0; i < PH_COUNT; i++) { ms[i] = 0; calls[i] = 0; }
}

void Prof::prefill(int count)
{
    // Creating events inside a timed region stalls the host while the GPU
    // idles; create them up front.
    while (npool < count) {
        if (npool == poolcap) {
            int nc = poolcap ? 2 * poolcap : 512;
            cudaEvent_t* np = static_cast<cudaEvent_t*>(realloc(pool, sizeof(cudaEvent_t) * nc));
            if (!np) return;
            pool = np;
            poolcap = nc;
        }
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return;
        pool[npool++] = e;
    }
}

void Prof::release()
{
    harvest();
    for (int i = 0; i < npool; i++) cudaEventDestroy(pool[i]);
    free(pool);
    free(pend);
    pool = nullptr;
    pend = nullptr;
    npool = poolcap = npend = cap = 0;
}

namespace {
thread_local int t_freeze = 0;
// gl_selftest_alloc_limit: allocations above it fail on this thread (0: none)
thread_local int64_t t_alloc_limit = 0, t_alloc_refused = 0;
}
AllocFreeze::AllocFreeze() { t_freeze++; }
AllocFreeze::~AllocFreeze() { t_freeze--; }
bool alloc_frozen() { return t_freeze > 0; }

gl_status DevBuf::reserve(size_t need)
{
    if (need <= bytes && p) return GL_OK;
    if (t_freeze) {
        set_error("buffer growth while capturing a step graph");
        return GL_ERR_CAPACITY;
    }
    if (p) {
        cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    if (need == 0) need = 16;
    cudaError_t e = cudaErrorMemoryAllocation;
    if (t_alloc_limit && need > (size_t)t_alloc_limit) t_alloc_refused++;
    else e = cudaMalloc(&p, need);
    if (e != cudaSuccess) {
        p = nullptr;
        set_error(std::string("cudaMalloc(") + std::to_string(need) + "): " + cudaGetErrorString(e));
        return GL_ERR_OOM;
    }
    bytes = need;
    return GL_OK;
}

void DevBuf::release()
{
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
}

gl_status View::init()
{
    if (!count.p) {
        GL_TRY(count.reserve(128));
        GL_CUDA_TRY(cudaMemset(count.p, 0, 128));
    }
    if (!h_count) {
        GL_CUDA_TRY(cudaMallocHost(&h_count, 128));
        std::memset(h_count, 0, 128);
    }
    if (!hpin) GL_CUDA_TRY(cudaMallocHost(&hpin, kDescBlock * kDescRing));
    for (int i = 0; i < kDescRing; i++)
        if (!pin_ev[i]) GL_CUDA_TRY(cudaEventCreateWithFlags(&pin_ev[i], cudaEventDisableTiming));
    GL_TRY(desc.reserve(kDescBlock));
    return GL_OK;
}

// Copy hdesc[0..V) to the device through the next pinned slot; a slot is
// reused only after its previous copy has executed.
gl_status View::upload_descs(cudaStream_t s)
{
    const int slot = pin_slot;
    pin_slot = (pin_slot + 1) % kDescRing;
    if (pin_used[slot]) GL_CUDA_TRY(cudaEventSynchronize(pin_ev[slot]));
    char* h = hpin + (size_t)slot * kDescBlock;
    std::memcpy(h, &hscal, sizeof(StepScalars));
    std::memcpy(h + sizeof(StepScalars), hdesc, sizeof(ViewDesc) * (size_t)V);
    const size_t bytes = sizeof(StepScalars) + sizeof(ViewDesc) * (size_t)V;
    GL_CUDA_TRY(cudaMemcpyAsync(desc.p, h, bytes, cudaMemcpyHostToDevice, s));
    GL_CUDA_TRY(cudaEventRecord(pin_ev[slot], s));
    pin_used[slot] = true;
    return GL_OK;
}

void View::release()
{
    DevBuf* all[] = {&rec, &radius, &brec, &touched, &dkey, &gidx, &dkey2, &gidx2,
                     &dup_off, &bsum, &count, &itile, &ival, &itile2, &ival2, &iowner, &srec0, &srec1, &srec2, &srec3, &sgid, &g2d, &gpart, &gmask, &work, &items, &heads, &segstate,
                     &hist, &sctl, &ranges, &tile_order, &Tfin, &ncon, &rgb, &depth, &opac};
    for (DevBuf* b : all) b->release();
    desc.release();
    if (h_count) cudaFreeHost(h_count);
    h_count = nullptr;
    if (hpin) cudaFreeHost(hpin);
    hpin = nullptr;
    for (int i = 0; i < kDescRing; i++) {
        if (pin_ev[i]) cudaEventDestroy(pin_ev[i]);
        pin_ev[i] = nullptr;
        pin_used[i] = false;
    }
}

namespace {

bool finite_all(const float* x, int n)
{
    for (int i = 0; i < n; i++)
        if (!std::isfinite(x[i])) return false;
    return true;
}

gl_status make_cam(const gl_pose* pose, const gl_intrinsics* K, Cam& cam)
{
    if (!pose || !K) { set_error("pose and intrinsics are required"); return GL_ERR_INVALID; }
    if (!finite_all(pose->R_cw, 9) || !finite_all(pose->t_cw, 3)) {
        set_error("pose contains NaN or Inf");
        return GL_ERR_INVALID;
    }
    if (!(K->fx > 0.f) || !(K->fy > 0.f) || !std::isfinite(K->fx) || !std::isfinite(K->fy) ||
        !std::isfinite(K->cx) || !std::isfinite(K->cy)) {
        set_error("intrinsics: focal lengths must be positive and finite");
        return GL_ERR_INVALID;
    }
    if (K->width <= 0 || K->height <= 0 || K->width > 16384 || K->height > 16384) {
        set_error("image size must be in 1..16384");
        return GL_ERR_INVALID;
    }
    std::memcpy(cam.R, pose->R_cw, sizeof(cam.R));
    std::memcpy(cam.t, pose->t_cw, sizeof(cam.t));
    cam.fx = K->fx; cam.fy = K->fy; cam.cx = K->cx; cam.cy = K->cy;
    cam.W = K->width; cam.H = K->height;
    return GL_OK;
}

// Twists xi = (rho, phi) in R^6, translation part first.  se3_exp maps a
// twist to a rigid motion (R, t); the left Jacobian J_l(xi) relates a change
// of the twist to a left perturbation of the motion it gives:
// exp((xi + d)^) = exp((J_l(xi) d)^) exp(xi^) to first order.  Closed forms
// of SO(3)/SE(3) (Barfoot, "State Estimation for Robotics", 2017, Sec. 7.1),
// with Taylor series of the coefficients below 0.1 rad, in double.
void so3_hat(const double w[3], double W[9])
{
    W[0] = 0.0;   W[1] = -w[2]; W[2] = w[1];
    W[3] = w[2];  W[4] = 0.0;   W[5] = -w[0];
    W[6] = -w[1]; W[7] = w[0];  W[8] = 0.0;
}

void mat3_mul(const double A[9], const double B[9], double C[9])
{
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++)
            C[i * 3 + j] = A[i * 3] * B[j] + A[i * 3 + 1] * B[3 + j] + A[i * 3 + 2] * B[6 + j];
}

// Coefficients of the rotation angle th: sin(th)/th, (1 - cos th)/th^2,
// (th - sin th)/th^3, (th^2 + 2 cos th - 2)/(2 th^4), (2 th - 3 sin th + th cos th)/(2 th^5).
void so3_coefs(double th, double c[5])
{
    const double t2 = th * th;
    if (th < 0.1) {
        c[0] = 1.0 - t2 / 6.0 + t2 * t2 / 120.0;
        c[1] = 0.5 - t2 / 24.0 + t2 * t2 / 720.0;
        c[2] = 1.0 / 6.0 - t2 / 120.0 + t2 * t2 / 5040.0;
        c[3] = 1.0 / 24.0 - t2 / 720.0 + t2 * t2 / 40320.0;
        c[4] = 1.0 / 120.0 - t2 / 2520.0 + t2 * t2 / 120960.0;
        return;
    }
    const double s = std::sin(th), co = std::cos(th);
    c[0] = s / th;
    c[1] = (1.0 - co) / t2;
    c[2] = (th - s) / (t2 * th);
    c[3] = (t2 + 2.0 * co - 2.0) / (2.0 * t2 * t2);
    c[4] = (2.0 * th - 3.0 * s + th * co) / (2.0 * t2 * t2 * th);
}

// SO(3) left Jacobian J(phi) = I + c1 phi^ + c2 phi^2.
void so3_left_jacobian(const double phi[3], const double c[5], double J[9])
{
    double P[9], P2[9];
    so3_hat(phi, P);
    mat3_mul(P, P, P2);
    for (int i = 0; i < 9; i++) J[i] = (i % 4 == 0 ? 1.0 : 0.0) + c[1] * P[i] + c[2] * P2[i];
}

void se3_exp(const double xi[6], double R[9], double t[3])
{
    const double* phi = xi + 3;
    const double th = std::sqrt(phi[0] * phi[0] + phi[1] * phi[1] + phi[2] * phi[2]);
    double c[5], P[9], P2[9], J[9];
    so3_coefs(th, c);
    so3_hat(phi, P);
    mat3_mul(P, P, P2);
    for (int i = 0; i < 9; i++) R[i] = (i % 4 == 0 ? 1.0 : 0.0) + c[0] * P[i] + c[1] * P2[i];
    so3_left_jacobian(phi, c, J);
    for (int i = 0; i < 3; i++) t[i] = J[i * 3] * xi[0] + J[i * 3 + 1] * xi[1] + J[i * 3 + 2] * xi[2];
}

// J_l(xi) (6 x 6, row-major) = [[J, Q], [0, J]], Q(rho, phi) from Barfoot's
// series summed in closed form.
void se3_left_jacobian(const double xi[6], double Jl[36])
{
    const double* rho = xi;
    const double* phi = xi + 3;
    const double th = std::sqrt(phi[0] * phi[0] + phi[1] * phi[1] + phi[2] * phi[2]);
    double c[5], J[9], P[9], Rh[9];
    so3_coefs(th, c);
    so3_left_jacobian(phi, c, J);
    so3_hat(phi, P);
    so3_hat(rho, Rh);
    double PR[9], RP[9], PRP[9], PP[9], PPR[9], RPP[9], PRPP[9], PPRP[9];
    mat3_mul(P, Rh, PR);
    mat3_mul(Rh, P, RP);
    mat3_mul(PR, P, PRP);
    mat3_mul(P, P, PP);
    mat3_mul(PP, Rh, PPR);
    mat3_mul(RP, P, RPP);
    mat3_mul(PRP, P, PRPP);
    mat3_mul(P, PRP, PPRP);
    double Q[9];
    for (int i = 0; i < 9; i++)
        Q[i] = 0.5 * Rh[i] + c[2] * (PR[i] + RP[i] + PRP[i]) + c[3] * (PPR[i] + RPP[i] - 3.0 * PRP[i]) +
               c[4] * (PRPP[i] + PPRP[i]);
    for (int i = 0; i < 36; i++) Jl[i] = 0.0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            Jl[i * 6 + j] = J[i * 3 + j];
            Jl[i * 6 + 3 + j] = Q[i * 3 + j];
            Jl[(3 + i) * 6 + 3 + j] = J[i * 3 + j];
        }
}

// Records a raster warp stages per batch, in 32-record sub-batches.
int batch_subs(int batch_depth, bool det)
{
    return det ? 1 : std::max(1, batch_depth / 32);
}

bool valid_batch_depth(int b) { return b == 32 || b == 64 || b == 128 || b == 256; }

// -1: the library's choice, 0: no splitting
bool valid_segment(int s) { return s == -1 || s == 0 || (s >= 64 && s <= 65536 && (s & (s - 1)) == 0); }

bool is_device_ptr(const void* p)
{
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Bytes from p to the end of the device allocation that holds it; 0 if none
// does (or the driver does not say).
size_t bytes_left(const void* p)
{
    using Range = CUresult(CUDAAPI*)(CUdeviceptr*, size_t*, CUdeviceptr);
    static const Range range = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Range>(f);
    }();
    CUdeviceptr base = 0;
    size_t size = 0;
    const CUdeviceptr at = (CUdeviceptr)(uintptr_t)p;
    if (!range || range(&base, &size, at) != CUDA_SUCCESS || at < base || at - base >= size) return 0;
    return size - (size_t)(at - base);
}

// `count` floats that a kernel on the current device can read and write: one
// allocation holds them (a copy looks at that itself, a kernel does not).
bool is_local_array(const void* p, size_t count)
{
    cudaPointerAttributes a;
    int dev = -1;
    if (!p || ((uintptr_t)p & 3) || cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev)) &&
           bytes_left(p) >= 4 * count;
}

// Refuses device memory that ends before `count` floats with nothing mapped
// behind it.  (What spans several allocations is left to the copy.)
gl_status check_extent(const void* p, size_t count)
{
    const size_t left = is_device_ptr(p) ? bytes_left(p) : 0;
    if (left && left < 4 * count && bytes_left(static_cast<const char*>(p) + left) == 0) {
        set_error("a device array ends before its last row");
        return GL_ERR_INVALID;
    }
    return GL_OK;
}

bool overlap(const float* a, size_t na, const float* b, size_t nb) { return a && b && a < b + nb && b < a + na; }

gl_status check_tile(int t)
{
    if (t != 8 && t != 16 && t != 32) { set_error("tile_size must be 8, 16 or 32"); return GL_ERR_INVALID; }
    return GL_OK;
}

gl_status check_gauss(const gl_gaussians* g, bool need_ptrs)
{
    if (!g) { set_error("null gaussians"); return GL_ERR_INVALID; }
    if (g->n < 0 || g->n > (int64_t)0x7fffffff) { set_error("gaussian count out of range"); return GL_ERR_INVALID; }
    if (g->sh_degree < 0 || g->sh_degree > 3) { set_error("sh_degree must be 0..3"); return GL_ERR_INVALID; }
    if (need_ptrs && g->n > 0 &&
        (!g->means || !g->log_scales || !g->quats || !g->logits || !g->sh)) {
        set_error("null parameter array");
        return GL_ERR_INVALID;
    }
    for (const float* a : {g->means, g->log_scales, g->quats, g->logits, g->sh})
        if (a && (reinterpret_cast<uintptr_t>(a) & 15u)) {
            set_error("parameter arrays must be 16-byte aligned");
            return GL_ERR_INVALID;
        }
    return GL_OK;
}

GParams params_of(const gl_gaussians* g)
{
    GParams p;
    p.means = g->means; p.log_scales = g->log_scales; p.quats = g->quats; p.logits = g->logits;
    p.sh = g->sh; p.n = g->n; p.deg = g->sh_degree; p.K = (g->sh_degree + 1) * (g->sh_degree + 1);
    return p;
}

GMut mut_of(const gl_gaussians* g)
{
    GMut m;
    m.means = g->means; m.log_scales = g->log_scales; m.quats = g->quats; m.logits = g->logits; m.sh = g->sh;
    return m;
}

}  // namespace
}  // namespace gl

using namespace gl;

// ===========================================================================
// Library
// ===========================================================================
extern "C" const char* gl_last_error(void) { return g_err.c_str(); }

extern "C" int32_t gl_version(void) { return 102; }

extern "C" gl_status gl_config_default(gl_config* c)
{
    if (!c) return GL_ERR_INVALID;
    std::memset(c, 0, sizeof(*c));
    c->sh_degree = 3;
    c->tile_size = 16;
    c->sparse_adam = 1;
    c->seed = 0x5eedULL;
    c->lambda_dssim = 0.2f;    // Sec. IV-A
    c->tau = 0.99f;            // Sec. IV-A
    c->opacity_fg = 0.1f;      // o_a
    c->opacity_sky = 0.7f;     // o_b
    c->sky_radius = 1.0e4f;    // R
    c->n_sky = 100000;         // N_s
    c->lr_pos = 1.6e-4f;       // 3DGS learning rates, not decayed
    c->lr_sh_dc = 2.5e-3f;
    c->lr_sh_rest = 2.5e-3f / 20.0f;
    c->lr_opacity = 0.05f;
    c->lr_scale = 5e-3f;
    c->lr_rot = 1e-3f;
    c->lr_exposure = 1e-3f;
    c->adam_b1 = 0.9f;
    c->adam_b2 = 0.999f;
    c->adam_eps = 1e-15f;
    c->capacity_hint = 1 << 20;
    return GL_OK;
}

// ===========================================================================
// Stateless differentiable API
// ===========================================================================
extern "C" gl_status gl_ctx_create(void* stream, gl_ctx** out)
{
    if (!out) { set_error("null out"); return GL_ERR_INVALID; }
    std::unique_ptr<gl_ctx> c(new gl_ctx());
    c->impl.stream = static_cast<cudaStream_t>(stream);
    GL_TRY(c->impl.view.init());
    *out = c.release();
    return GL_OK;
}

extern "C" gl_status gl_ctx_set_exec(gl_ctx* ctx, const gl_exec_config* e)
{
    if (!ctx || !e) { set_error("null argument"); return GL_ERR_INVALID; }
    if (!valid_batch_depth(e->batch_depth) || (e->batch_depth > 64 && e->pixels_per_lane != 1) ||
        (e->deterministic != 0 && e->deterministic != 1) ||
        (e->pixels_per_lane != 1 && e->pixels_per_lane != 2 && e->pixels_per_lane != 4) ||
        !valid_segment(e->segment) || (e->exact_cull != 0 && e->exact_cull != 1) ||
        (e->per_gaussian != 0 && e->per_gaussian != 1)) {
        set_error("invalid execution config");
        return GL_ERR_INVALID;
    }
    ctx->impl.exec = *e;
    return GL_OK;
}

extern "C" gl_status gl_ctx_destroy(gl_ctx* ctx)
{
    if (!ctx) return GL_OK;
    cudaStreamSynchronize(ctx->impl.stream);
    ctx->impl.view.release();
    ctx->impl.pose_part.release();
    ctx->impl.loss_part.release();
    delete ctx;
    return GL_OK;
}

extern "C" gl_status gl_rasterize_forward(gl_ctx* ctx, const gl_gaussians* g, const gl_pose* pose,
                                          const float* twist6, const gl_intrinsics* K, int32_t tile_size,
                                          float* out_rgb, float* out_depth, float* out_opacity)
{
    if (!ctx || !out_rgb) { set_error("null ctx or out_rgb"); return GL_ERR_INVALID; }
    GL_TRY(check_gauss(g, true));
    GL_TRY(check_tile(tile_size));
    Cam cam;
    GL_TRY(make_cam(pose, K, cam));
    gl_ctx_impl& c = ctx->impl;
    c.has_forward = 0;
    // the pose rendered: exp(xi^) T_cw (T_cw itself when twist6 is null)
    double xi[6] = {0, 0, 0, 0, 0, 0};
    if (twist6) {
        if (!finite_all(twist6, 6)) { set_error("twist contains NaN or Inf"); return GL_ERR_INVALID; }
        for (int i = 0; i < 6; i++) xi[i] = twist6[i];
    }
    double Rd[9], td[3], Jl[36];
    se3_exp(xi, Rd, td);
    se3_left_jacobian(xi, Jl);
    double R0[9], R1[9];
    for (int i = 0; i < 9; i++) R0[i] = pose->R_cw[i];
    mat3_mul(Rd, R0, R1);
    for (int i = 0; i < 3; i++) {
        cam.t[i] = (float)(Rd[i * 3] * pose->t_cw[0] + Rd[i * 3 + 1] * pose->t_cw[1] + Rd[i * 3 + 2] * pose->t_cw[2] +
                           td[i]);
        for (int j = 0; j < 3; j++) cam.R[i * 3 + j] = (float)R1[i * 3 + j];
    }
    if (!finite_all(cam.R, 9) || !finite_all(cam.t, 3)) { set_error("twisted pose is not finite"); return GL_ERR_INVALID; }
    for (int i = 0; i < 36; i++) c.pose_jac[i] = (float)Jl[i];
    c.view.det = c.exec.deterministic != 0;
    c.view.nb = batch_subs(c.exec.batch_depth, c.view.det);
    c.view.pd = std::min(c.exec.pixels_per_lane, tile_size / 4);
    c.view.persistent = c.exec.persistent != 0;
    c.view.set_segment(c.exec.segment);
    c.view.cull = c.exec.exact_cull != 0;
    c.view.pg = c.exec.per_gaussian != 0;
    GL_TRY(bin_view(c.view, params_of(g), cam, tile_size, c.stream));
    GL_TRY(raster_forward(c.view, out_rgb, out_depth, out_opacity, c.stream));
    c.has_forward = 1;
    c.deg = g->sh_degree;
    return GL_OK;
}

extern "C" gl_status gl_rasterize_backward(gl_ctx* ctx, const gl_gaussians* g, const float* dL_drgb,
                                           const float* dL_ddepth, const float* dL_dopacity,
                                           gl_gaussians* grad, float* grad_pose6)
{
    if (!ctx || !dL_drgb) { set_error("null ctx or dL_drgb"); return GL_ERR_INVALID; }
    gl_ctx_impl& c = ctx->impl;
    if (!c.has_forward) { set_error("backward without a forward on this ctx"); return GL_ERR_INVALID; }
    GL_TRY(check_gauss(g, true));
    GL_TRY(check_gauss(grad, true));
    if (g->n != c.view.n || grad->n != g->n || grad->sh_degree != g->sh_degree) {
        set_error("gaussians differ from the forward");
        return GL_ERR_INVALID;
    }
    GL_TRY(raster_backward(c.view, dL_drgb, dL_ddepth, dL_dopacity, c.stream));
    const int npart = pose_partials_needed(g->n);
    float* pp = nullptr;
    if (grad_pose6) {
        GL_TRY(c.pose_part.reserve(sizeof(float) * 6 * (size_t)npart));
        pp = c.pose_part.as<float>();
    }
    GL_TRY(params_backward(c.view, params_of(g), mut_of(grad), pp, npart, c.stream));
    if (grad_pose6) {
        if (g->n == 0) GL_CUDA_TRY(cudaMemsetAsync(grad_pose6, 0, 24, c.stream));
        else GL_TRY(pose_reduce(pp, npart, c.pose_jac, grad_pose6, c.stream));
    }
    return GL_OK;
}

extern "C" gl_status gl_photometric_loss(gl_ctx* ctx, const float* rgb, const float* target,
                                         const float* E34, int32_t width, int32_t height,
                                         float lambda_dssim, float* loss_out, float* dL_drgb,
                                         float* dL_dE)
{
    if (!ctx || !rgb || !target || !E34 || !dL_drgb) { set_error("null argument"); return GL_ERR_INVALID; }
    if (width <= 0 || height <= 0) { set_error("bad image size"); return GL_ERR_INVALID; }
    if (!(lambda_dssim >= 0.f && lambda_dssim <= 1.f)) { set_error("lambda must be in [0,1]"); return GL_ERR_INVALID; }
    gl_ctx_impl& c = ctx->impl;
    GL_TRY(c.loss_part.reserve(sizeof(float) * (size_t)loss_partials_needed(width, height)));
    return photometric_loss(rgb, target, E34, width, height, lambda_dssim, dL_drgb, c.loss_part.as<float>(),
                            loss_out, dL_dE, c.stream);
}

extern "C" gl_status gl_ctx_get_preprocess(gl_ctx* ctx, int32_t* radius, int32_t* rect, float* mean2d,
                                           float* conic, float* opacity, float* rgb, float* depth)
{
    if (!ctx || !ctx->impl.has_forward) { set_error("no forward on this ctx"); return GL_ERR_INVALID; }
    View& v = ctx->impl.view;
    cudaStream_t s = ctx->impl.stream;
    const size_t n = (size_t)v.n;
    if (n == 0) return GL_OK;
    if (radius) GL_CUDA_TRY(cudaMemcpyAsync(radius, v.radius.p, 4 * n, cudaMemcpyDeviceToDevice, s));
    return export_preprocess(v, rect, mean2d, conic, opacity, rgb, depth, s);
}

extern "C" gl_status gl_ctx_num_instances(gl_ctx* ctx, int64_t* I_out)
{
    if (!ctx || !I_out || !ctx->impl.has_forward) { set_error("no forward on this ctx"); return GL_ERR_INVALID; }
    *I_out = ctx->impl.view.I;
    return GL_OK;
}

extern "C" gl_status gl_ctx_get_instances(gl_ctx* ctx, uint64_t* keys, uint32_t* vals, uint32_t* ranges)
{
    if (!ctx || !ctx->impl.has_forward) { set_error("no forward on this ctx"); return GL_ERR_INVALID; }
    View& v = ctx->impl.view;
    GL_TRY(export_instances(v, keys, vals, ctx->impl.stream));
    if (ranges)
        GL_CUDA_TRY(cudaMemcpyAsync(ranges, v.ranges.p, 8 * (size_t)v.ntiles, cudaMemcpyDeviceToDevice,
                                    ctx->impl.stream));
    return GL_OK;
}

extern "C" gl_status gl_ctx_get_pixel_state(gl_ctx* ctx, float* T_final, uint32_t* n_contrib)
{
    if (!ctx || !ctx->impl.has_forward) { set_error("no forward on this ctx"); return GL_ERR_INVALID; }
    View& v = ctx->impl.view;
    const size_t P = (size_t)v.P;
    if (T_final) GL_CUDA_TRY(cudaMemcpyAsync(T_final, v.Tfin.p, 4 * P, cudaMemcpyDeviceToDevice, ctx->impl.stream));
    if (n_contrib) GL_CUDA_TRY(cudaMemcpyAsync(n_contrib, v.ncon.p, 4 * P, cudaMemcpyDeviceToDevice, ctx->impl.stream));
    return GL_OK;
}

// ===========================================================================
// Map API
// ===========================================================================
namespace {

struct Keyframe {
    gl_pose pose{};
    gl_intrinsics K{};
    DevBuf image;       // H*W*3 floats when registered
    bool has_image = false;
    DevBuf expo;        // 36 floats: E, m, v
    int64_t steps = 0;
};

enum { PM = 0, PS, PQ, PO, PH, NPARAM };

}  // namespace

struct gl_map {
    gl_config cfg{};
    cudaStream_t stream = nullptr;
    int deg = 3, K = 16;
    int64_t n = 0, cap = 0;
    DevBuf prm[NPARAM], mom1[NPARAM], mom2[NPARAM];
    DevBuf kind;                 // u8 per Gaussian: 0 LiDAR, 1 visual, 2 sky
    int64_t step = 0;
    gl_ctx_impl ctx;
    DevBuf stage_img, stage_pts, dLdC, loss_dev;
    DevBuf flags, scan;
    float* h_loss = nullptr;             // pinned: losses of a step's views
    float* h_expo = nullptr;             // pinned: an exposure on its way to the caller
    std::unordered_map<int64_t, std::unique_ptr<Keyframe>> kfs;
    Prof prof;
    // step execution and the captured step graph
    gl_exec_config exec{0, 0, 32, 1, 0, 0, -1, 1, 0};
    cudaStream_t gstream = nullptr;      // capture stream (the map's may be the legacy one)
    // caller host images of a step are copied on cstream while the step's
    // first kernels run; the loss waits for stage_ev (ready_ev: the map's
    // stream has finished with the staging buffer)
    cudaStream_t cstream = nullptr;
    cudaEvent_t stage_ev = nullptr, ready_ev = nullptr;
    struct StepGraph {
        std::vector<int64_t> key;        // the step shape it was captured for
        cudaGraphExec_t exec = nullptr;
        int64_t nodes = 0;               // kernels per replay
    };
    std::vector<StepGraph> graphs;       // most recently used last, at most kMaxGraphs
    static constexpr size_t kMaxGraphs = 8;
    int64_t graph_captures = 0, graph_replays = 0, graph_reruns = 0;
    // counts of the steps taken while the phase timers are on (device u64:
    // visible pairs, instances, contributor sum, pixels), and their views
    DevBuf timed_counts;
    int64_t timed_steps = 0, timed_views = 0;

    size_t row_floats(int which) const
    {
        switch (which) {
            case PM: return 3;
            case PS: return 3;
            case PQ: return 4;
            case PO: return 1;
            default: return (size_t)K * 3;
        }
    }
    GParams params() const
    {
        GParams p;
        p.means = prm[PM].as<float>(); p.log_scales = prm[PS].as<float>(); p.quats = prm[PQ].as<float>();
        p.logits = prm[PO].as<float>(); p.sh = prm[PH].as<float>(); p.n = n; p.deg = deg; p.K = K;
        return p;
    }
    static GMut mut(DevBuf* b)
    {
        GMut m;
        m.means = b[PM].as<float>(); m.log_scales = b[PS].as<float>(); m.quats = b[PQ].as<float>();
        m.logits = b[PO].as<float>(); m.sh = b[PH].as<float>();
        return m;
    }
};

namespace {

gl_status map_reserve(gl_map* m, int64_t need)
{
    if (need <= m->cap) return GL_OK;
    int64_t nc = std::max<int64_t>({need, 2 * m->cap, m->cfg.capacity_hint, 1024});
    for (int set = 0; set < 3; set++) {
        DevBuf* arr = set == 0 ? m->prm : (set == 1 ? m->mom1 : m->mom2);
        for (int w = 0; w < NPARAM; w++) {
            const size_t rb = 4 * m->row_floats(w);
            void* np = nullptr;
            cudaError_t e = cudaMalloc(&np, rb * (size_t)nc);
            if (e != cudaSuccess) { set_error("map growth: out of device memory"); return GL_ERR_OOM; }
            if (m->n > 0) GL_CUDA_TRY(cudaMemcpyAsync(np, arr[w].p, rb * (size_t)m->n, cudaMemcpyDeviceToDevice, m->stream));
            GL_CUDA_TRY(cudaMemsetAsync(static_cast<char*>(np) + rb * (size_t)m->n, 0, rb * (size_t)(nc - m->n), m->stream));
            GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
            arr[w].release();
            arr[w].p = np;
            arr[w].bytes = rb * (size_t)nc;
        }
    }
    {
        void* np = nullptr;
        GL_CUDA_TRY(cudaMalloc(&np, (size_t)nc));
        if (m->n > 0) GL_CUDA_TRY(cudaMemcpyAsync(np, m->kind.p, (size_t)m->n, cudaMemcpyDeviceToDevice, m->stream));
        GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
        m->kind.release();
        m->kind.p = np;
        m->kind.bytes = (size_t)nc;
    }
    m->cap = nc;
    return GL_OK;
}

gl_status zero_moments(gl_map* m, int64_t from, int64_t count)
{
    if (count <= 0) return GL_OK;
    ArrayMove mv[2 * NPARAM];
    for (int w = 0; w < NPARAM; w++) {
        const size_t row = m->row_floats(w);
        mv[2 * w] = {m->mom1[w].as<float>() + row * from, nullptr, row * count};
        mv[2 * w + 1] = {m->mom2[w].as<float>() + row * from, nullptr, row * count};
    }
    return move_arrays(mv, 2 * NPARAM, m->stream);
}

gl_status from_device(float* dst, const float* src, size_t count, cudaStream_t s)
{
    GL_TRY(check_extent(dst, count));
    GL_CUDA_TRY(cudaMemcpyAsync(dst, src, 4 * count, is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    return GL_OK;
}

// The live rows of five map arrays into the caller's arrays (null: skipped).
// Arrays that share memory are copied one after the other, the later one
// winning; the others move in one launch.
gl_status copy_rows_out(gl_map* m, DevBuf* src, float* const dst[NPARAM])
{
    size_t cnt[NPARAM];
    for (int w = 0; w < NPARAM; w++) cnt[w] = m->row_floats(w) * (size_t)m->n;
    bool shared = false;
    for (int w = 1; w < NPARAM; w++)
        for (int u = 0; u < w; u++) shared = shared || overlap(dst[u], cnt[u], dst[w], cnt[w]);
    ArrayMove mv[NPARAM];
    int k = 0;
    for (int w = 0; w < NPARAM; w++) {
        if (!dst[w] || m->n == 0) continue;
        if (!shared && is_local_array(dst[w], cnt[w])) mv[k++] = {dst[w], src[w].as<float>(), cnt[w]};
        else GL_TRY(from_device(dst[w], src[w].as<float>(), cnt[w], m->stream));
    }
    return move_arrays(mv, k, m->stream);
}

Keyframe* get_kf(gl_map* m, int64_t id, bool create, gl_status* st)
{
    auto it = m->kfs.find(id);
    if (it != m->kfs.end()) return it->second.get();
    if (!create) { *st = GL_ERR_NOT_FOUND; set_error("unknown keyframe id"); return nullptr; }
    std::unique_ptr<Keyframe> kf(new Keyframe());
    if ((*st = kf->expo.reserve(36 * 4)) != GL_OK) return nullptr;
    float init[36] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0};
    if (cudaMemcpyAsync(kf->expo.p, init, sizeof(init), cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        *st = GL_ERR_CUDA;
        set_error("keyframe exposure init failed");
        return nullptr;
    }
    Keyframe* raw = kf.get();
    m->kfs[id] = std::move(kf);
    *st = GL_OK;
    return raw;
}

// Render into the given device images, or the view's own where null.
gl_status render_internal(gl_map* m, const Cam& cam, int Ts, float* rgb = nullptr, float* depth = nullptr,
                          float* opac = nullptr)
{
    View& v = m->ctx.view;
    const size_t P = (size_t)cam.W * cam.H;
    if (!rgb) GL_TRY(v.rgb.reserve(12 * P));
    if (!depth) GL_TRY(v.depth.reserve(4 * P));
    if (!opac) GL_TRY(v.opac.reserve(4 * P));
    map_exec_knobs(m, v, Ts);
    GL_TRY(bin_view(v, m->params(), cam, Ts, m->stream));
    return raster_forward(v, rgb ? rgb : v.rgb.as<float>(), depth ? depth : v.depth.as<float>(),
                          opac ? opac : v.opac.as<float>(), m->stream);
}

}  // namespace

gl_status check_runtime_config(const gl_config* cfg)
{
    GL_TRY(check_tile(cfg->tile_size));
    const float lrs[] = {cfg->lr_pos, cfg->lr_sh_dc, cfg->lr_sh_rest, cfg->lr_opacity, cfg->lr_scale, cfg->lr_rot,
                         cfg->lr_exposure};
    for (float x : lrs)
        if (!(x >= 0.f) || !std::isfinite(x)) { set_error("learning rates must be finite and >= 0"); return GL_ERR_INVALID; }
    if (!(cfg->adam_b1 >= 0.f && cfg->adam_b1 < 1.f) || !(cfg->adam_b2 >= 0.f && cfg->adam_b2 < 1.f) ||
        !(cfg->adam_eps >= 0.f) || !(cfg->lambda_dssim >= 0.f && cfg->lambda_dssim <= 1.f) ||
        !(cfg->tau > 0.f && cfg->tau <= 1.f) || !(cfg->opacity_fg > 0.f && cfg->opacity_fg < 1.f) ||
        !std::isfinite(cfg->lr_window_exp) || cfg->lr_window_exp < -2.f || cfg->lr_window_exp > 2.f) {
        set_error("invalid config value");
        return GL_ERR_INVALID;
    }
    return GL_OK;
}

extern "C" gl_status gl_map_create(const gl_config* cfg, void* stream, gl_map** out)
{
    if (!cfg || !out) { set_error("null argument"); return GL_ERR_INVALID; }
    if (cfg->sh_degree < 0 || cfg->sh_degree > 3) { set_error("sh_degree must be 0..3"); return GL_ERR_INVALID; }
    GL_TRY(check_runtime_config(cfg));
    if (cfg->n_sky < 0 || !(cfg->sky_radius > 0.f) || !(cfg->opacity_sky > 0.f && cfg->opacity_sky < 1.f) ||
        !(cfg->opacity_fg > 0.f && cfg->opacity_fg < 1.f) || !(cfg->adam_b1 >= 0.f && cfg->adam_b1 < 1.f) ||
        !(cfg->adam_b2 >= 0.f && cfg->adam_b2 < 1.f)) {
        set_error("invalid config value");
        return GL_ERR_INVALID;
    }
    std::unique_ptr<gl_map> m(new gl_map());
    m->cfg = *cfg;
    m->stream = static_cast<cudaStream_t>(stream);
    m->deg = cfg->sh_degree;
    m->K = (m->deg + 1) * (m->deg + 1);
    m->ctx.stream = m->stream;
    m->ctx.view.prof = &m->prof;
    GL_TRY(m->ctx.view.init());
    GL_CUDA_TRY(cudaMallocHost(&m->h_loss, sizeof(float) * kMaxViews));
    GL_CUDA_TRY(cudaMallocHost(&m->h_expo, sizeof(float) * 12));
    GL_TRY(m->loss_dev.reserve(16));
    GL_TRY(map_reserve(m.get(), std::max<int64_t>(cfg->n_sky, 1)));
    if (cfg->n_sky > 0) {
        GMut p = gl_map::mut(m->prm);
        GL_TRY(sky_create(p.means, p.log_scales, p.quats, p.logits, p.sh, m->K, cfg->n_sky, cfg->sky_radius,
                          cfg->seed, cfg->opacity_sky, m->stream));
        GL_CUDA_TRY(cudaMemsetAsync(m->kind.p, 2, (size_t)cfg->n_sky, m->stream));
        m->n = cfg->n_sky;
    }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    *out = m.release();
    return GL_OK;
}

extern "C" gl_status gl_map_destroy(gl_map* m)
{
    if (!m) return GL_OK;
    cudaStreamSynchronize(m->stream);
    for (int w = 0; w < NPARAM; w++) { m->prm[w].release(); m->mom1[w].release(); m->mom2[w].release(); }
    m->kind.release();
    m->ctx.view.release();
    m->ctx.pose_part.release();
    m->ctx.loss_part.release();
    m->stage_img.release(); m->stage_pts.release(); m->dLdC.release(); m->loss_dev.release();
    m->flags.release(); m->scan.release(); m->timed_counts.release();
    for (auto& kv : m->kfs) { kv.second->image.release(); kv.second->expo.release(); }
    if (m->h_loss) cudaFreeHost(m->h_loss);
    if (m->h_expo) cudaFreeHost(m->h_expo);
    for (auto& g : m->graphs) cudaGraphExecDestroy(g.exec);
    if (m->gstream) cudaStreamDestroy(m->gstream);
    if (m->cstream) {
        cudaStreamSynchronize(m->cstream);
        cudaStreamDestroy(m->cstream);
    }
    if (m->stage_ev) cudaEventDestroy(m->stage_ev);
    if (m->ready_ev) cudaEventDestroy(m->ready_ev);
    m->prof.release();
    delete m;
    return GL_OK;
}

extern "C" gl_status gl_map_size(gl_map* m, int64_t* n_out)
{
    if (!m || !n_out) { set_error("null argument"); return GL_ERR_INVALID; }
    *n_out = m->n;
    return GL_OK;
}

extern "C" gl_status gl_map_add_points(gl_map* m, const float* xyz, const float* rgb, int64_t n, int32_t kind,
                                       const gl_pose* pose, const gl_intrinsics* K, int32_t use_mask,
                                       int64_t* n_added)
{
    if (!m || (n > 0 && (!xyz || !rgb))) { set_error("null argument"); return GL_ERR_INVALID; }
    if (n < 0) { set_error("negative point count"); return GL_ERR_INVALID; }
    Cam cam;
    GL_TRY(make_cam(pose, K, cam));
    if (n_added) *n_added = 0;
    if (n == 0) return GL_OK;
    const float *dx, *dc;
    GL_TRY(m->stage_pts.reserve(24 * (size_t)n));
    {
        // stage both arrays into one buffer when they live on the host
        if (is_device_ptr(xyz)) dx = xyz;
        else {
            GL_CUDA_TRY(cudaMemcpyAsync(m->stage_pts.p, xyz, 12 * (size_t)n, cudaMemcpyHostToDevice, m->stream));
            dx = m->stage_pts.as<float>();
        }
        if (is_device_ptr(rgb)) dc = rgb;
        else {
            float* dst = m->stage_pts.as<float>() + 3 * (size_t)n;
            GL_CUDA_TRY(cudaMemcpyAsync(dst, rgb, 12 * (size_t)n, cudaMemcpyHostToDevice, m->stream));
            dc = dst;
        }
    }
    const float* opac = nullptr;
    if (use_mask) {
        GL_TRY(render_internal(m, cam, m->cfg.tile_size));
        opac = m->ctx.view.opac.as<float>();
    }
    int64_t added = 0;
    PhaseScope ps(&m->prof, PH_EXPAND, m->stream);
    GMut none{};
    GL_TRY(expand_points(dx, dc, n, cam, opac, m->cfg.tau, use_mask ? 1 : 0, m->cfg.opacity_fg, m->K, none, 0, 0,
                         m->flags, m->scan, &added, m->stream));
    if (added > 0) {
        GL_TRY(map_reserve(m, m->n + added));
        GL_TRY(expand_points(dx, dc, n, cam, opac, m->cfg.tau, use_mask ? 1 : 0, m->cfg.opacity_fg, m->K,
                             gl_map::mut(m->prm), m->n, m->cap, m->flags, m->scan, &added, m->stream));
        GL_TRY(zero_moments(m, m->n, added));
        GL_CUDA_TRY(cudaMemsetAsync(static_cast<char*>(m->kind.p) + m->n, kind ? 1 : 0, (size_t)added, m->stream));
        m->n += added;
    }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    if (n_added) *n_added = added;
    return GL_OK;
}

extern "C" gl_status gl_map_add_keyframe(gl_map* m, const gl_keyframe* kf)
{
    if (!m || !kf || !kf->image) { set_error("null argument"); return GL_ERR_INVALID; }
    Cam cam;
    GL_TRY(make_cam(&kf->pose, &kf->K, cam));
    gl_status st;
    Keyframe* k = get_kf(m, kf->id, true, &st);
    if (!k) return st;
    const size_t cnt = (size_t)kf->K.width * kf->K.height * 3;
    GL_TRY(k->image.reserve(4 * cnt));
    GL_CUDA_TRY(cudaMemcpyAsync(k->image.p, kf->image, 4 * cnt,
                                is_device_ptr(kf->image) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                m->stream));
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    k->has_image = true;
    k->pose = kf->pose;
    k->K = kf->K;
    return GL_OK;
}

extern "C" gl_status gl_render(gl_map* m, const gl_pose* pose, const gl_intrinsics* K, const float* E34,
                               float* out_rgb, float* out_depth, float* out_opacity)
{
    if (!m || !out_rgb) { set_error("null argument"); return GL_ERR_INVALID; }
    Cam cam;
    GL_TRY(make_cam(pose, K, cam));
    if (E34 && !finite_all(E34, 12)) { set_error("exposure contains NaN or Inf"); return GL_ERR_INVALID; }
    // images in the caller's device memory are rendered in place (the colour
    // only without an exposure); images that share memory are copied out one
    // after the other, the later one winning
    const size_t px = (size_t)cam.W * cam.H;
    const bool shared = overlap(out_rgb, 3 * px, out_depth, px) || overlap(out_rgb, 3 * px, out_opacity, px) ||
                        overlap(out_depth, px, out_opacity, px);
    float* depth = !shared && is_local_array(out_depth, px) ? out_depth : nullptr;
    float* opac = !shared && is_local_array(out_opacity, px) ? out_opacity : nullptr;
    float* rgb = !shared && !E34 && is_local_array(out_rgb, 3 * px) ? out_rgb : nullptr;
    GL_TRY(render_internal(m, cam, m->cfg.tile_size, rgb, depth, opac));
    View& v = m->ctx.view;
    const float ident[12] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0};
    if (!rgb && is_device_ptr(out_rgb)) {
        GL_TRY(check_extent(out_rgb, 3 * px));
        GL_TRY(apply_exposure(v.rgb.as<float>(), out_rgb, E34 ? E34 : ident, (int64_t)px, m->stream));
    } else if (!rgb) {
        const float* src = v.rgb.as<float>();
        if (E34) {
            GL_TRY(m->stage_img.reserve(12 * px));
            GL_TRY(apply_exposure(src, m->stage_img.as<float>(), E34, (int64_t)px, m->stream));
            src = m->stage_img.as<float>();
        }
        GL_CUDA_TRY(cudaMemcpyAsync(out_rgb, src, 12 * px, cudaMemcpyDeviceToHost, m->stream));
    }
    if (out_depth && !depth) GL_TRY(from_device(out_depth, v.depth.as<float>(), px, m->stream));
    if (out_opacity && !opac) GL_TRY(from_device(out_opacity, v.opac.as<float>(), px, m->stream));
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return sort_wait_status(v, m->stream);
}

namespace {

// Host side of one step: cameras, keyframes and targets (caller host images
// are staged into one device buffer at each view's pixel offset).
struct StepPlan {
    int V = 0;
    int64_t P = 0;
    Cam cams[kMaxViews];
    ViewExtra extra[kMaxViews];
    Keyframe* kfs[kMaxViews];
};

// The copy stream and its events (created once per map, before the first
// staging or capture, so that every captured step holds the loss's wait).
gl_status ensure_stage(gl_map* m)
{
    if (!m->cstream) GL_CUDA_TRY(cudaStreamCreateWithFlags(&m->cstream, cudaStreamNonBlocking));
    if (!m->stage_ev) GL_CUDA_TRY(cudaEventCreateWithFlags(&m->stage_ev, cudaEventDisableTiming));
    if (!m->ready_ev) GL_CUDA_TRY(cudaEventCreateWithFlags(&m->ready_ev, cudaEventDisableTiming));
    return GL_OK;
}

gl_status plan_step(gl_map* m, const gl_keyframe* views, int V, StepPlan& sp)
{
    if (!m || !views || V < 1) { set_error("need at least one view"); return GL_ERR_INVALID; }
    if (V > kMaxViews) { set_error("at most 64 views per step"); return GL_ERR_INVALID; }
    sp.V = V;
    for (int i = 0; i < V; i++) {
        GL_TRY(make_cam(&views[i].pose, &views[i].K, sp.cams[i]));
        for (int j = 0; j < i; j++)
            if (views[j].id == views[i].id) { set_error("a keyframe appears twice in one window"); return GL_ERR_INVALID; }
        gl_status st;
        sp.kfs[i] = get_kf(m, views[i].id, true, &st);
        if (!sp.kfs[i]) return st;
        if (!views[i].image) {
            if (!sp.kfs[i]->has_image) { set_error("keyframe has no stored image"); return GL_ERR_NOT_FOUND; }
            if (sp.kfs[i]->K.width != sp.cams[i].W || sp.kfs[i]->K.height != sp.cams[i].H) {
                set_error("stored image size differs");
                return GL_ERR_INVALID;
            }
        }
    }
    sp.P = 0;
    for (int i = 0; i < V; i++) sp.P += (int64_t)sp.cams[i].W * sp.cams[i].H;
    bool need_stage = false;
    for (int i = 0; i < V; i++)
        if (views[i].image && !is_device_ptr(views[i].image)) need_stage = true;
    if (need_stage) {
        GL_TRY(m->stage_img.reserve(12 * (size_t)sp.P));
        GL_TRY(ensure_stage(m));
        GL_CUDA_TRY(cudaEventRecord(m->ready_ev, m->stream));
        GL_CUDA_TRY(cudaStreamWaitEvent(m->cstream, m->ready_ev, 0));
    }
    int64_t off = 0;
    for (int i = 0; i < V; i++) {
        const size_t Pi = (size_t)sp.cams[i].W * sp.cams[i].H;
        const float* tgt = nullptr;
        if (!views[i].image) tgt = sp.kfs[i]->image.as<float>();
        else if (is_device_ptr(views[i].image)) tgt = views[i].image;
        else {
            float* dst = m->stage_img.as<float>() + 3 * off;
            GL_CUDA_TRY(cudaMemcpyAsync(dst, views[i].image, 12 * Pi, cudaMemcpyHostToDevice, m->cstream));
            tgt = dst;
        }
        off += (int64_t)Pi;
        float* e = sp.kfs[i]->expo.as<float>();
        sp.extra[i].target = tgt;
        sp.extra[i].E = e;
        sp.extra[i].Em = e + 12;
        sp.extra[i].weight = 1.0f / (float)V;
    }
    if (need_stage) GL_CUDA_TRY(cudaEventRecord(m->stage_ev, m->cstream));
    return GL_OK;
}

// Advance the Adam step counters (the map's and each view's exposure) and
// set the exposure bias corrections of the plan.
void begin_step(gl_map* m, StepPlan& sp)
{
    const gl_config& c = m->cfg;
    m->step++;
    for (int i = 0; i < sp.V; i++) {
        Keyframe* kf = sp.kfs[i];
        kf->steps++;
        sp.extra[i].e_bc1 = (float)(1.0 - std::pow((double)c.adam_b1, (double)kf->steps));
        sp.extra[i].e_bc2 = (float)(1.0 - std::pow((double)c.adam_b2, (double)kf->steps));
    }
}

StepScalars step_scalars(const gl_map* m)
{
    const gl_config& c = m->cfg;
    StepScalars sc;
    sc.ibc1 = (float)(1.0 / (1.0 - std::pow((double)c.adam_b1, (double)m->step)));
    sc.isbc2 = (float)(1.0 / std::sqrt(1.0 - std::pow((double)c.adam_b2, (double)m->step)));
    return sc;
}

int step_tile(const gl_map* m) { return m->exec.tile_size ? m->exec.tile_size : m->cfg.tile_size; }

void apply_exec(gl_map* m)
{
    View& v = m->ctx.view;
    v.det = m->exec.deterministic != 0;
    v.nb = batch_subs(m->exec.batch_depth, v.det);
    v.pd = m->exec.pixels_per_lane;
    v.persistent = m->exec.persistent != 0;
    v.set_segment(m->exec.segment);
    v.cull = m->exec.exact_cull != 0;
    v.pg = m->exec.per_gaussian != 0;
}

// Enqueue the whole step on `s`.  sync_free: the descriptors were uploaded by
// the caller, nothing is read back (the step being captured into a graph).
gl_status enqueue_step(gl_map* m, const StepPlan& sp, cudaStream_t s, bool sync_free)
{
    const gl_config& c = m->cfg;
    View& v = m->ctx.view;
    const int V = sp.V;
    GL_TRY(v.rgb.reserve(12 * (size_t)sp.P));
    GL_TRY(bin_views(v, m->params(), sp.cams, sp.extra, V, step_tile(m), s, sync_free, true));
    GL_TRY(raster_forward(v, v.rgb.as<float>(), nullptr, nullptr, s, false));
    GL_TRY(m->dLdC.reserve(12 * (size_t)sp.P));
    GL_TRY(m->ctx.loss_part.reserve(sizeof(float) * 14 * (size_t)v.nltiles));
    GL_TRY(m->loss_dev.reserve(sizeof(float) * kMaxViews));
    const uint64_t* ctl = v.count.as<uint64_t>();
    // the targets copied from host memory (if any) have landed; captured
    // steps hold this wait as an external event node, so a replay waits for
    // the copy of its own step
    if (m->stage_ev) GL_CUDA_TRY(cudaStreamWaitEvent(s, m->stage_ev, sync_free ? cudaEventWaitExternal : 0));
    {
        PhaseScope ps(&m->prof, PH_LOSS, s);
        GL_TRY(photometric_loss_views(v, v.rgb.as<float>(), c.lambda_dssim, m->dLdC.as<float>(),
                                      m->ctx.loss_part.as<float>(), m->loss_dev.as<float>(), c.adam_b1, c.adam_b2,
                                      c.adam_eps, c.lr_exposure, s, ctl));
    }
    GL_TRY(raster_backward(v, m->dLdC.as<float>(), nullptr, nullptr, s));
    AdamArgs a;
    a.m = gl_map::mut(m->mom1);
    a.v = gl_map::mut(m->mom2);
    a.lr_pos = c.lr_pos; a.lr_dc = c.lr_sh_dc; a.lr_rest = c.lr_sh_rest; a.lr_op = c.lr_opacity;
    a.lr_scale = c.lr_scale; a.lr_rot = c.lr_rot;
    a.b1 = c.adam_b1; a.b2 = c.adam_b2; a.eps = c.adam_eps;
    if (c.lr_window_exp != 0.0f && V > 1) {
        const float f = std::pow((float)V, c.lr_window_exp);
        a.lr_pos *= f; a.lr_dc *= f; a.lr_rest *= f; a.lr_op *= f; a.lr_scale *= f; a.lr_rot *= f;
    }
    const StepScalars sc = step_scalars(m);
    a.ibc1 = sc.ibc1;
    a.isbc2 = sc.isbc2;
    a.sparse = c.sparse_adam;
    a.abort = ctl;
    if (sync_free) a.bc = v.d_scal();
    GL_TRY(params_adam(v, m->params(), gl_map::mut(m->prm), a, s));
    return report_step(v, m->loss_dev.as<float>(), m->h_loss, s);
}

// The mean loss of the step just synchronised with (report_step).
void read_loss(const gl_map* m, int V, float* out_loss)
{
    if (!out_loss) return;
    double sum = 0.0;
    for (int i = 0; i < V; i++) sum += m->h_loss[i];
    *out_loss = (float)(sum / V);
}

// Everything a captured step bakes in: its shape, the execution knobs and
// the address and size of every buffer its kernels touch directly (targets
// and exposures are reached through the descriptors, uploaded per replay).
std::vector<int64_t> graph_key(const gl_map* m, const StepPlan& sp)
{
    std::vector<int64_t> k = {sp.V, step_tile(m), m->exec.batch_depth, m->exec.pixels_per_lane,
                              m->exec.persistent, m->exec.deterministic, m->exec.segment, m->exec.exact_cull,
                              m->exec.per_gaussian,
                              m->n, m->deg,
                              m->cfg.sparse_adam};
    for (int i = 0; i < sp.V; i++) {
        k.push_back(sp.cams[i].W);
        k.push_back(sp.cams[i].H);
    }
    const View& v = m->ctx.view;
    const DevBuf* bufs[] = {&v.rec, &v.radius, &v.brec, &v.touched, &v.dkey,
                            &v.gidx, &v.dkey2, &v.gidx2, &v.dup_off, &v.g2d, &v.bsum, &v.count, &v.itile,
                            &v.ival, &v.itile2, &v.ival2, &v.iowner, &v.srec0, &v.srec1, &v.srec2, &v.srec3,
                            &v.sgid, &v.hist, &v.sctl, &v.ranges, &v.tile_order, &v.Tfin, &v.ncon, &v.rgb, &v.work, &v.gpart, &v.gmask,
                            &v.items, &v.heads, &v.segstate,
                            &v.desc, &m->dLdC, &m->ctx.loss_part, &m->loss_dev};
    for (const DevBuf* b : bufs) {
        k.push_back((int64_t)(uintptr_t)b->p);
        k.push_back((int64_t)b->bytes);
    }
    for (int w = 0; w < NPARAM; w++) {
        k.push_back((int64_t)(uintptr_t)m->prm[w].p);
        k.push_back((int64_t)(uintptr_t)m->mom1[w].p);
        k.push_back((int64_t)(uintptr_t)m->mom2[w].p);
    }
    return k;
}

void drop_graph(gl_map* m)
{
    for (auto& g : m->graphs) cudaGraphExecDestroy(g.exec);
    m->graphs.clear();
}

// The cached graph of this key (moved to most recently used), or null.
gl_map::StepGraph* find_graph(gl_map* m, const std::vector<int64_t>& key)
{
    for (size_t i = 0; i < m->graphs.size(); i++)
        if (m->graphs[i].key == key) {
            gl_map::StepGraph g = std::move(m->graphs[i]);
            m->graphs.erase(m->graphs.begin() + i);
            m->graphs.push_back(std::move(g));
            return &m->graphs.back();
        }
    return nullptr;
}

// Capture the step shape of `sp` (sized by the eager step just taken).  A
// failure leaves no graph and is not an error: steps stay eager.
void capture_step(gl_map* m, const StepPlan& sp)
{
    if (ensure_stage(m) != GL_OK) return;
    if (!m->gstream && cudaStreamCreateWithFlags(&m->gstream, cudaStreamNonBlocking) != cudaSuccess) {
        m->gstream = nullptr;
        return;
    }
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return;
    const int64_t l0 = g_launches.load();
    cudaGraph_t g = nullptr;
    gl_status st;
    {
        AllocFreeze freeze;
        if (cudaStreamBeginCapture(m->gstream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return;
        st = enqueue_step(m, sp, m->gstream, true);
        const cudaError_t e = cudaStreamEndCapture(m->gstream, &g);
        if (e != cudaSuccess) st = GL_ERR_CUDA;
    }
    const int64_t nodes = g_launches.load() - l0;
    count_launches(-nodes);   // nothing ran yet
    cudaGetLastError();
    if (st != GL_OK || !g) {
        if (g) cudaGraphDestroy(g);
        return;
    }
    cudaGraphExec_t ex = nullptr;
    const cudaError_t e = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    std::vector<int64_t> key = graph_key(m, sp);
    for (size_t i = 0; i < m->graphs.size(); i++)
        if (m->graphs[i].key == key) {   // replaces a stale entry of the same shape
            cudaGraphExecDestroy(m->graphs[i].exec);
            m->graphs.erase(m->graphs.begin() + i);
            break;
        }
    if (m->graphs.size() >= gl_map::kMaxGraphs) {
        cudaGraphExecDestroy(m->graphs.front().exec);
        m->graphs.erase(m->graphs.begin());
    }
    gl_map::StepGraph entry;
    entry.key = std::move(key);
    entry.exec = ex;
    entry.nodes = nodes;
    m->graphs.push_back(std::move(entry));
    m->graph_captures++;
}

gl_status run_step(gl_map* m, StepPlan& sp, float* out_loss)
{
    apply_exec(m);
    begin_step(m, sp);
    View& v = m->ctx.view;
    const bool graphs = m->exec.use_graphs && !m->prof.on;
    gl_map::StepGraph* g = graphs ? find_graph(m, graph_key(m, sp)) : nullptr;
    if (g) {
        v.set_views(sp.cams, sp.extra, sp.V, step_tile(m));
        v.hscal = step_scalars(m);
        GL_TRY(v.upload_descs(m->stream));
        GL_CUDA_TRY(cudaGraphLaunch(g->exec, m->stream));
        count_launches(g->nodes);
        m->graph_replays++;
        GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
        GL_TRY(sort_wait_status(v, m->stream));
        if (v.h_count[1] == 0) {
            read_loss(m, sp.V, out_loss);
            return GL_OK;
        }
        // the instances outgrew the buffers: the replay updated nothing; run
        // the same step (same counters) eagerly, which grows them
        m->graph_reruns++;
    }
    GL_TRY(enqueue_step(m, sp, m->stream, false));
    if (m->prof.on && m->timed_counts.p) {
        GL_TRY(accumulate_view_counts(v, m->timed_counts.as<uint64_t>(), m->stream));
        m->timed_steps++;
        m->timed_views += sp.V;
    }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    read_loss(m, sp.V, out_loss);
    GL_TRY(sort_wait_status(v, m->stream));
    if (graphs) capture_step(m, sp);
    return GL_OK;
}

}  // namespace

extern "C" gl_status gl_optimize_step(gl_map* m, const gl_keyframe* views, int32_t n_views, float* out_loss)
{
    StepPlan sp;
    GL_TRY(plan_step(m, views, n_views, sp));
    return run_step(m, sp, out_loss);
}

extern "C" gl_status gl_map_get_params(gl_map* m, gl_gaussians* out, int64_t* n_out)
{
    if (!m || !out) { set_error("null argument"); return GL_ERR_INVALID; }
    if (out->sh_degree != m->deg) { set_error("sh_degree differs from the map"); return GL_ERR_INVALID; }
    if (n_out) *n_out = m->n;
    if (out->n < m->n) { set_error("output arrays too small"); return GL_ERR_INVALID; }
    float* dst[NPARAM] = {out->means, out->log_scales, out->quats, out->logits, out->sh};
    GL_TRY(copy_rows_out(m, m->prm, dst));
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GL_OK;
}

extern "C" gl_status gl_map_get_moments(gl_map* m, int32_t which, gl_gaussians* out)
{
    if (!m || !out || (which != 1 && which != 2)) { set_error("bad argument"); return GL_ERR_INVALID; }
    if (out->sh_degree != m->deg || out->n < m->n) { set_error("output shape differs"); return GL_ERR_INVALID; }
    DevBuf* src = which == 1 ? m->mom1 : m->mom2;
    float* dst[NPARAM] = {out->means, out->log_scales, out->quats, out->logits, out->sh};
    GL_TRY(copy_rows_out(m, src, dst));
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GL_OK;
}

extern "C" gl_status gl_map_set_params(gl_map* m, const gl_gaussians* in)
{
    if (!m || !in) { set_error("null argument"); return GL_ERR_INVALID; }
    GL_TRY(check_gauss(in, true));
    if (in->sh_degree != m->deg) { set_error("sh_degree differs from the map"); return GL_ERR_INVALID; }
    GL_TRY(map_reserve(m, in->n));
    const float* src[NPARAM] = {in->means, in->log_scales, in->quats, in->logits, in->sh};
    ArrayMove mv[3 * NPARAM];
    int k = 0;
    for (int w = 0; w < NPARAM; w++) {
        const size_t cnt = m->row_floats(w) * (size_t)in->n;
        if (is_local_array(src[w], cnt)) {
            mv[k++] = {m->prm[w].as<float>(), src[w], cnt};
        } else {
            GL_TRY(check_extent(src[w], cnt));
            GL_CUDA_TRY(cudaMemcpyAsync(m->prm[w].p, src[w], 4 * cnt,
                                        is_device_ptr(src[w]) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                        m->stream));
        }
        mv[k++] = {m->mom1[w].as<float>(), nullptr, cnt};
        mv[k++] = {m->mom2[w].as<float>(), nullptr, cnt};
    }
    GL_TRY(move_arrays(mv, k, m->stream));
    GL_CUDA_TRY(cudaMemsetAsync(m->kind.p, 0, (size_t)in->n, m->stream));
    m->n = in->n;
    m->step = 0;
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GL_OK;
}

extern "C" gl_status gl_map_get_exposure(gl_map* m, int64_t id, float* E34_out)
{
    if (!m || !E34_out) { set_error("null argument"); return GL_ERR_INVALID; }
    gl_status st;
    Keyframe* kf = get_kf(m, id, false, &st);
    if (!kf) return st;
    // through pinned memory: a copy to pageable memory is staged by the driver
    // (what the host cannot write is left to the driver)
    const bool host = !is_device_ptr(E34_out);
    GL_CUDA_TRY(cudaMemcpyAsync(host ? m->h_expo : E34_out, kf->expo.p, 48, cudaMemcpyDeviceToHost, m->stream));
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    if (host) std::memcpy(E34_out, m->h_expo, 48);
    return GL_OK;
}

extern "C" gl_status gl_map_set_timing(gl_map* m, int32_t enable)
{
    if (!m) { set_error("null map"); return GL_ERR_INVALID; }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    m->prof.reset();
    m->prof.on = enable != 0;
    if (m->prof.on) m->prof.prefill(8192);
    m->timed_steps = m->timed_views = 0;
    GL_TRY(m->timed_counts.reserve(4 * sizeof(uint64_t)));
    GL_CUDA_TRY(cudaMemset(m->timed_counts.p, 0, 4 * sizeof(uint64_t)));
    return GL_OK;
}

extern "C" gl_status gl_map_get_stats(gl_map* m, gl_stats* out)
{
    if (!m || !out) { set_error("null argument"); return GL_ERR_INVALID; }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    m->prof.harvest();
    std::memset(out, 0, sizeof(*out));
    out->n_gaussians = m->n;
    out->steps = m->step;
    const View& v = m->ctx.view;
    out->n_instances = v.I;
    if (v.I < 0) {   // a graph step: the count lives on the device
        uint64_t c = 0;
        GL_CUDA_TRY(cudaMemcpy(&c, v.count.p, sizeof(c), cudaMemcpyDeviceToHost));
        out->n_instances = (int64_t)c;
    }
    out->graph_captures = m->graph_captures;
    out->graph_replays = m->graph_replays;
    out->graph_reruns = m->graph_reruns;
    out->pixels = (int64_t)v.W * v.H;
    GL_TRY(view_counts(v, &out->n_visible, &out->sum_contrib, m->stream));
    out->timed_steps = m->timed_steps;
    out->timed_views = m->timed_views;
    if (m->timed_counts.p && m->timed_steps) {
        uint64_t h[4];
        GL_CUDA_TRY(cudaMemcpy(h, m->timed_counts.p, sizeof(h), cudaMemcpyDeviceToHost));
        out->timed_visible = (int64_t)h[0];
        out->timed_instances = (int64_t)h[1];
        out->timed_contrib = (int64_t)h[2];
        out->timed_pixels = (int64_t)h[3];
    }
    for (int i = 0; i < PH_COUNT && i < GL_NUM_PHASES; i++) {
        out->phase_ms[i] = m->prof.ms[i];
        out->phase_calls[i] = m->prof.calls[i];
    }
    return GL_OK;
}

extern "C" const char* gl_phase_name(int32_t i)
{
    if (i < 0 || i >= PH_COUNT) return "";
    return kPhaseNames[i];
}

extern "C" int64_t gl_kernel_launch_count(void) { return g_launches.load(); }

extern "C" gl_status gl_selftest_bounded_wait(int32_t* expired)
{
    if (!expired) { set_error("null expired"); return GL_ERR_INVALID; }
    *expired = 0;
    return sort_wait_selftest(expired);
}

extern "C" gl_status gl_selftest_alloc_limit(int64_t bytes, int64_t* refused)
{
    if (bytes < 0) { set_error("bytes must not be negative"); return GL_ERR_INVALID; }
    t_alloc_limit = bytes;
    if (refused) *refused = t_alloc_refused;
    t_alloc_refused = 0;
    return GL_OK;
}

// ---------------------------------------------------------------------------
// Step execution and the autotuner
// ---------------------------------------------------------------------------
namespace {

gl_status check_exec_config(const gl_map* m, const gl_exec_config& e)
{
    const int ts = e.tile_size ? e.tile_size : m->cfg.tile_size;
    if (e.tile_size != 0 && e.tile_size != 8 && e.tile_size != 16 && e.tile_size != 32) {
        set_error("tile_size must be 0, 8, 16 or 32");
        return GL_ERR_INVALID;
    }
    if (!valid_batch_depth(e.batch_depth)) { set_error("batch_depth must be 32, 64, 128 or 256"); return GL_ERR_INVALID; }
    if (e.batch_depth > 64 && e.pixels_per_lane != 1) {
        set_error("batch depths of 128 and 256 take one pixel per lane");
        return GL_ERR_INVALID;
    }
    if (e.deterministic != 0 && e.deterministic != 1) { set_error("deterministic must be 0 or 1"); return GL_ERR_INVALID; }
    if (e.exact_cull != 0 && e.exact_cull != 1) { set_error("exact_cull must be 0 or 1"); return GL_ERR_INVALID; }
    if (e.per_gaussian != 0 && e.per_gaussian != 1) { set_error("per_gaussian must be 0 or 1"); return GL_ERR_INVALID; }
    if (!valid_segment(e.segment)) {
        set_error("segment must be -1, 0 or a power of two in 64..65536");
        return GL_ERR_INVALID;
    }
    if ((e.pixels_per_lane != 1 && e.pixels_per_lane != 2 && e.pixels_per_lane != 4) || 4 * e.pixels_per_lane > ts) {
        set_error("pixels_per_lane must be 1, 2 or 4 with 4 x pixels_per_lane <= tile size");
        return GL_ERR_INVALID;
    }
    return GL_OK;
}

// Device copy of everything a step changes: the Gaussians, both Adam
// moments, the views' exposures (E, m, v) and the step counters.
struct Snapshot {
    DevBuf rows[3][NPARAM];
    DevBuf expo;
    int64_t step = 0, n = 0;
    std::vector<int64_t> kf_steps;
};

gl_status snap_take(gl_map* m, const std::vector<Keyframe*>& kfs, Snapshot& S)
{
    S.step = m->step;
    S.n = m->n;
    S.kf_steps.resize(kfs.size());
    GL_TRY(S.expo.reserve(36 * 4 * std::max<size_t>(kfs.size(), 1)));
    for (size_t i = 0; i < kfs.size(); i++) {
        S.kf_steps[i] = kfs[i]->steps;
        GL_CUDA_TRY(cudaMemcpyAsync(S.expo.as<float>() + 36 * i, kfs[i]->expo.p, 36 * 4, cudaMemcpyDeviceToDevice,
                                    m->stream));
    }
    for (int set = 0; set < 3; set++) {
        DevBuf* arr = set == 0 ? m->prm : (set == 1 ? m->mom1 : m->mom2);
        for (int w = 0; w < NPARAM; w++) {
            const size_t bytes = 4 * m->row_floats(w) * (size_t)m->n;
            GL_TRY(S.rows[set][w].reserve(bytes));
            GL_CUDA_TRY(cudaMemcpyAsync(S.rows[set][w].p, arr[w].p, bytes, cudaMemcpyDeviceToDevice, m->stream));
        }
    }
    return GL_OK;
}

gl_status snap_restore(gl_map* m, const std::vector<Keyframe*>& kfs, const Snapshot& S)
{
    m->step = S.step;
    for (size_t i = 0; i < kfs.size(); i++) {
        kfs[i]->steps = S.kf_steps[i];
        GL_CUDA_TRY(cudaMemcpyAsync(kfs[i]->expo.p, S.expo.as<float>() + 36 * i, 36 * 4, cudaMemcpyDeviceToDevice,
                                    m->stream));
    }
    for (int set = 0; set < 3; set++) {
        DevBuf* arr = set == 0 ? m->prm : (set == 1 ? m->mom1 : m->mom2);
        for (int w = 0; w < NPARAM; w++) {
            const size_t bytes = 4 * m->row_floats(w) * (size_t)S.n;
            GL_CUDA_TRY(cudaMemcpyAsync(arr[w].p, S.rows[set][w].p, bytes, cudaMemcpyDeviceToDevice, m->stream));
        }
    }
    return GL_OK;
}

void snap_release(Snapshot& S)
{
    for (auto& set : S.rows)
        for (DevBuf& b : set) b.release();
    S.expo.release();
}

}  // namespace

extern "C" gl_status gl_map_set_exec(gl_map* m, const gl_exec_config* e)
{
    if (!m || !e) { set_error("null argument"); return GL_ERR_INVALID; }
    GL_TRY(check_exec_config(m, *e));
    m->exec = *e;
    return GL_OK;
}

extern "C" gl_status gl_map_get_exec(gl_map* m, gl_exec_config* e)
{
    if (!m || !e) { set_error("null argument"); return GL_ERR_INVALID; }
    *e = m->exec;
    return GL_OK;
}

extern "C" gl_status gl_map_autotune(gl_map* m, const gl_keyframe* views, int32_t n_views, int32_t window,
                                     int32_t reps, int32_t keep_tile_size, gl_exec_config* best, float* best_ms)
{
    if (!m || !best || !views) { set_error("null argument"); return GL_ERR_INVALID; }
    if (reps < 1) { set_error("reps must be >= 1"); return GL_ERR_INVALID; }
    if (window < 1 || n_views < window || n_views % window != 0 || n_views / window > 64) {
        set_error("n_views must be 1..64 windows of `window` views");
        return GL_ERR_INVALID;
    }
    const int nw = n_views / window;
    std::vector<StepPlan> plans(nw);
    for (int w = 0; w < nw; w++) GL_TRY(plan_step(m, views + (size_t)w * window, window, plans[w]));
    const gl_exec_config saved = m->exec;
    const bool timing = m->prof.on;
    m->prof.on = false;
    std::vector<Keyframe*> kfs;   // every keyframe the windows touch, once
    for (const StepPlan& sp : plans)
        for (int i = 0; i < sp.V; i++)
            if (std::find(kfs.begin(), kfs.end(), sp.kfs[i]) == kfs.end()) kfs.push_back(sp.kfs[i]);
    Snapshot S;
    gl_status st = snap_take(m, kfs, S);
    auto restore = [&]() { return snap_restore(m, kfs, S); };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (st == GL_OK && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)) {
        set_error("event creation failed");
        st = GL_ERR_CUDA;
    }
    // time one candidate: per window one eager step (sizes buffers, captures
    // the graph) and one replay, then reps timed rounds of every window
    auto trial = [&](const gl_exec_config& cand, float* ms_out) -> gl_status {
        m->exec = cand;
        gl_status r = GL_OK;
        for (int w = 0; w < nw && r == GL_OK; w++)
            for (int k = 0; k < 2 && r == GL_OK; k++) r = run_step(m, plans[w], nullptr);
        if (r != GL_OK) return r;
        cudaEventRecord(e0, m->stream);
        for (int k = 0; k < reps && r == GL_OK; k++)
            for (int w = 0; w < nw && r == GL_OK; w++) r = run_step(m, plans[w], nullptr);
        cudaEventRecord(e1, m->stream);
        if (r != GL_OK) return r;
        if (cudaEventSynchronize(e1) != cudaSuccess) return GL_ERR_CUDA;
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        *ms_out = ms / (float)(reps * nw);
        return restore();
    };
    // coordinate descent from the defaults: each knob in turn takes the
    // value that is fastest with the others fixed
    float best_t = -1.0f;
    gl_exec_config best_e{1, 1, 32, 1, keep_tile_size ? 0 : m->cfg.tile_size, saved.deterministic, 1024,
                          saved.exact_cull, 0};
    if (st == GL_OK) st = trial(best_e, &best_t);
    const int tile_vals[3] = {8, 16, 32}, seg_vals[4] = {0, 256, 512, 1024}, pers_vals[2] = {0, 1},
              bd_vals[4] = {32, 64, 128, 256}, ppl_vals[3] = {1, 2, 4}, pg_vals[2] = {0, 1};
    struct Dim { int32_t gl_exec_config::*field; const int* vals; int n; };
    const Dim dims[6] = {{&gl_exec_config::tile_size, tile_vals, keep_tile_size ? 0 : 3},
                         {&gl_exec_config::segment, seg_vals, 4},
                         {&gl_exec_config::persistent, pers_vals, 2},
                         {&gl_exec_config::batch_depth, bd_vals, saved.deterministic ? 1 : 4},
                         {&gl_exec_config::pixels_per_lane, ppl_vals, 3},
                         {&gl_exec_config::per_gaussian, pg_vals, 2}};
    for (const Dim& d : dims) {
        for (int i = 0; i < d.n && st == GL_OK; i++) {
            gl_exec_config cand = best_e;
            cand.*(d.field) = d.vals[i];
            if (cand.*(d.field) == best_e.*(d.field)) continue;
            const int ts = cand.tile_size ? cand.tile_size : m->cfg.tile_size;
            if (4 * cand.pixels_per_lane > ts) continue;
            if (cand.batch_depth > 64 && cand.pixels_per_lane != 1) continue;
            float ms = 0.0f;
            st = trial(cand, &ms);
            if (st == GL_OK && ms < best_t) {
                best_t = ms;
                best_e = cand;
            }
        }
    }
    if (st == GL_OK) st = restore();
    cudaStreamSynchronize(m->stream);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    snap_release(S);
    drop_graph(m);
    m->prof.on = timing;
    if (st != GL_OK) {
        m->exec = saved;
        return st;
    }
    m->exec = best_e;
    *best = best_e;
    if (best_ms) *best_ms = best_t;
    return GL_OK;
}

// ---------------------------------------------------------------------------
// Checkpoint: the whole optimisation state in one host byte buffer
// ---------------------------------------------------------------------------
namespace {

constexpr char kCkMagic[8] = {'G', 'L', 'M', 'A', 'P', 'C', 'K', '1'};
constexpr uint32_t kCkVersion = 1;

struct CkHeader {
    char magic[8];
    uint32_t version;
    int32_t deg;
    int64_t n, step, n_kf;
    int32_t with_images, reserved;
};

struct CkKeyframe {
    int64_t id;
    gl_pose pose;
    gl_intrinsics K;
    int64_t steps;
    float expo[36];
    int32_t has_image, reserved;
};

size_t pad8(size_t x) { return (x + 7) & ~size_t(7); }

int64_t ck_bytes(const gl_map* m, bool with_images)
{
    size_t b = sizeof(CkHeader);
    for (int w = 0; w < NPARAM; w++) b += 3 * 4 * m->row_floats(w) * (size_t)m->n;
    b += pad8((size_t)m->n);
    for (const auto& kv : m->kfs) {
        b += sizeof(CkKeyframe);
        if (with_images && kv.second->has_image) b += 12 * (size_t)kv.second->K.width * kv.second->K.height;
    }
    return (int64_t)b;
}

std::vector<int64_t> sorted_ids(const gl_map* m)
{
    std::vector<int64_t> ids;
    for (const auto& kv : m->kfs) ids.push_back(kv.first);
    std::sort(ids.begin(), ids.end());
    return ids;
}

}  // namespace

extern "C" gl_status gl_map_checkpoint_size(gl_map* m, int32_t with_images, int64_t* bytes)
{
    if (!m || !bytes) { set_error("null argument"); return GL_ERR_INVALID; }
    *bytes = ck_bytes(m, with_images != 0);
    return GL_OK;
}

extern "C" gl_status gl_map_save(gl_map* m, int32_t with_images, void* host_buf, int64_t bytes)
{
    if (!m || !host_buf) { set_error("null argument"); return GL_ERR_INVALID; }
    const bool wi = with_images != 0;
    if (bytes < ck_bytes(m, wi)) { set_error("checkpoint buffer too small"); return GL_ERR_INVALID; }
    char* out = static_cast<char*>(host_buf);
    CkHeader h{};
    std::memcpy(h.magic, kCkMagic, 8);
    h.version = kCkVersion;
    h.deg = m->deg;
    h.n = m->n;
    h.step = m->step;
    h.n_kf = (int64_t)m->kfs.size();
    h.with_images = wi ? 1 : 0;
    std::memcpy(out, &h, sizeof(h));
    size_t off = sizeof(h);
    for (int set = 0; set < 3; set++) {
        DevBuf* arr = set == 0 ? m->prm : (set == 1 ? m->mom1 : m->mom2);
        for (int w = 0; w < NPARAM; w++) {
            const size_t b = 4 * m->row_floats(w) * (size_t)m->n;
            if (b) GL_CUDA_TRY(cudaMemcpyAsync(out + off, arr[w].p, b, cudaMemcpyDeviceToHost, m->stream));
            off += b;
        }
    }
    if (m->n) GL_CUDA_TRY(cudaMemcpyAsync(out + off, m->kind.p, (size_t)m->n, cudaMemcpyDeviceToHost, m->stream));
    std::memset(out + off + m->n, 0, pad8((size_t)m->n) - (size_t)m->n);
    off += pad8((size_t)m->n);
    for (int64_t id : sorted_ids(m)) {
        const Keyframe& k = *m->kfs[id];
        CkKeyframe c{};
        c.id = id;
        c.pose = k.pose;
        c.K = k.K;
        c.steps = k.steps;
        c.has_image = (wi && k.has_image) ? 1 : 0;
        GL_CUDA_TRY(cudaMemcpyAsync(c.expo, k.expo.p, sizeof(c.expo), cudaMemcpyDeviceToHost, m->stream));
        GL_CUDA_TRY(cudaStreamSynchronize(m->stream));   // c lives on this stack frame
        std::memcpy(out + off, &c, sizeof(c));
        off += sizeof(c);
        if (c.has_image) {
            const size_t b = 12 * (size_t)k.K.width * k.K.height;
            GL_CUDA_TRY(cudaMemcpyAsync(out + off, k.image.p, b, cudaMemcpyDeviceToHost, m->stream));
            off += b;
        }
    }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GL_OK;
}

extern "C" gl_status gl_map_load(gl_map* m, const void* host_buf, int64_t bytes)
{
    if (!m || !host_buf) { set_error("null argument"); return GL_ERR_INVALID; }
    const char* in = static_cast<const char*>(host_buf);
    if (bytes < (int64_t)sizeof(CkHeader)) { set_error("checkpoint too short"); return GL_ERR_INVALID; }
    CkHeader h;
    std::memcpy(&h, in, sizeof(h));
    if (std::memcmp(h.magic, kCkMagic, 8) != 0 || h.version != kCkVersion) {
        set_error("not a map checkpoint of this version");
        return GL_ERR_INVALID;
    }
    if (h.deg != m->deg) { set_error("checkpoint SH degree differs from the map's"); return GL_ERR_INVALID; }
    if (h.n < 0 || h.n_kf < 0 || h.step < 0) { set_error("corrupt checkpoint header"); return GL_ERR_INVALID; }
    // validate the whole layout before touching the map
    size_t need = sizeof(CkHeader);
    for (int w = 0; w < NPARAM; w++) need += 3 * 4 * m->row_floats(w) * (size_t)h.n;
    need += pad8((size_t)h.n);
    {
        size_t off = need;
        for (int64_t i = 0; i < h.n_kf; i++) {
            if ((int64_t)(off + sizeof(CkKeyframe)) > bytes) { set_error("checkpoint truncated"); return GL_ERR_INVALID; }
            CkKeyframe c;
            std::memcpy(&c, in + off, sizeof(c));
            off += sizeof(c);
            Cam tmp;
            GL_TRY(make_cam(&c.pose, &c.K, tmp));
            if (c.has_image) off += 12 * (size_t)c.K.width * c.K.height;
        }
        if ((int64_t)off > bytes) { set_error("checkpoint truncated"); return GL_ERR_INVALID; }
    }
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    GL_TRY(map_reserve(m, std::max<int64_t>(h.n, 1)));
    size_t off = sizeof(CkHeader);
    for (int set = 0; set < 3; set++) {
        DevBuf* arr = set == 0 ? m->prm : (set == 1 ? m->mom1 : m->mom2);
        for (int w = 0; w < NPARAM; w++) {
            const size_t b = 4 * m->row_floats(w) * (size_t)h.n;
            if (b) GL_CUDA_TRY(cudaMemcpyAsync(arr[w].p, in + off, b, cudaMemcpyHostToDevice, m->stream));
            off += b;
        }
    }
    if (h.n) GL_CUDA_TRY(cudaMemcpyAsync(m->kind.p, in + off, (size_t)h.n, cudaMemcpyHostToDevice, m->stream));
    off += pad8((size_t)h.n);
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    for (auto& kv : m->kfs) { kv.second->image.release(); kv.second->expo.release(); }
    m->kfs.clear();
    for (int64_t i = 0; i < h.n_kf; i++) {
        CkKeyframe c;
        std::memcpy(&c, in + off, sizeof(c));
        off += sizeof(c);
        gl_status st;
        Keyframe* k = get_kf(m, c.id, true, &st);
        if (!k) return st;
        k->pose = c.pose;
        k->K = c.K;
        k->steps = c.steps;
        GL_CUDA_TRY(cudaMemcpyAsync(k->expo.p, in + off - sizeof(c) + offsetof(CkKeyframe, expo), sizeof(c.expo),
                                    cudaMemcpyHostToDevice, m->stream));
        if (c.has_image) {
            const size_t b = 12 * (size_t)c.K.width * c.K.height;
            GL_TRY(k->image.reserve(b));
            GL_CUDA_TRY(cudaMemcpyAsync(k->image.p, in + off, b, cudaMemcpyHostToDevice, m->stream));
            k->has_image = true;
            off += b;
        }
    }
    m->n = h.n;
    m->step = h.step;
    drop_graph(m);
    GL_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GL_OK;
}

extern "C" gl_status gl_map_set_config(gl_map* m, const gl_config* cfg)
{
    if (!m || !cfg) { set_error("null argument"); return GL_ERR_INVALID; }
    if (cfg->sh_degree != m->deg) { set_error("sh_degree cannot change"); return GL_ERR_INVALID; }
    GL_TRY(check_runtime_config(cfg));
    gl_config c = *cfg;
    c.seed = m->cfg.seed;
    c.n_sky = m->cfg.n_sky;
    c.sky_radius = m->cfg.sky_radius;
    c.opacity_sky = m->cfg.opacity_sky;
    c.capacity_hint = m->cfg.capacity_hint;
    m->cfg = c;
    drop_graph(m);   // learning rates and flags are baked into captured steps
    return GL_OK;
}

extern "C" gl_status gl_map_get_config(gl_map* m, gl_config* cfg)
{
    if (!m || !cfg) { set_error("null argument"); return GL_ERR_INVALID; }
    *cfg = m->cfg;
    return GL_OK;
}

// ---------------------------------------------------------------------------
// Hooks for the serving loop (gl_server.cu)
// ---------------------------------------------------------------------------
namespace gl {

gl_status camera_from(const gl_pose* pose, const gl_intrinsics* K, Cam& cam) { return make_cam(pose, K, cam); }
cudaStream_t map_stream(const gl_map* m) { return m->stream; }

void map_exec_knobs(const gl_map* m, View& v, int Ts)
{
    v.nb = batch_subs(m->exec.batch_depth, m->exec.deterministic != 0);
    v.pd = std::min(m->exec.pixels_per_lane, Ts / 4);
    v.persistent = m->exec.persistent != 0;
    v.set_segment(m->exec.segment);
    v.cull = m->exec.exact_cull != 0;
    v.pg = m->exec.per_gaussian != 0;
}
int map_sh_degree(const gl_map* m) { return m->deg; }
int map_tile_size(const gl_map* m) { return m->cfg.tile_size; }
int64_t map_size_now(const gl_map* m) { return m->n; }
void map_keep_free(gl_map* m, size_t bytes) { m->ctx.view.keep_free = bytes; }

int64_t map_capacity(const gl_map* m) { return m->cap; }

gl_status map_snapshot(gl_map* m, DevBuf* dst, int64_t* n_out, cudaEvent_t done)
{
    ArrayMove mv[NPARAM];
    for (int w = 0; w < NPARAM; w++) {
        const size_t cnt = m->row_floats(w) * (size_t)m->n;
        GL_TRY(dst[w].reserve(4 * m->row_floats(w) * (size_t)std::max<int64_t>(m->n, 1)));
        mv[w] = {dst[w].as<float>(), m->prm[w].as<float>(), cnt};
    }
    GL_TRY(move_arrays(mv, NPARAM, m->stream));
    GL_CUDA_TRY(cudaEventRecord(done, m->stream));
    *n_out = m->n;
    return GL_OK;
}

GParams snapshot_params(const gl_map* m, const DevBuf* src, int64_t n)
{
    GParams p;
    p.means = src[PM].as<float>(); p.log_scales = src[PS].as<float>(); p.quats = src[PQ].as<float>();
    p.logits = src[PO].as<float>(); p.sh = src[PH].as<float>();
    p.n = n; p.deg = m->deg; p.K = m->K;
    return p;
}

void map_keyframes(const gl_map* m, std::vector<gl_keyframe>& out)
{
    out.clear();
    std::vector<int64_t> ids;
    for (const auto& kv : m->kfs)
        if (kv.second->has_image) ids.push_back(kv.first);
    std::sort(ids.begin(), ids.end());
    for (int64_t id : ids) {
        const Keyframe& k = *m->kfs.at(id);
        gl_keyframe kf{};
        kf.id = id;
        kf.pose = k.pose;
        kf.K = k.K;
        kf.image = nullptr;
        out.push_back(kf);
    }
}

}  // namespace gl
