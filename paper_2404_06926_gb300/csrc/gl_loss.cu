// gl_loss.cu -- exposure-compensated photometric loss (Eq. 9) and its adjoint.
//
// L = (1 - lambda) mean |E[C] - C_bar| + lambda (1 - mean SSIM(E[C], C_bar)),
// E[C] = A C + b with the 3x4 exposure [A | b] of the view (Sec. III-C 3).
// SSIM uses an 11x11 Gaussian window (sigma 1.5), zero padding, C1 = 0.01^2,
// C2 = 0.03^2 -- the D-SSIM of 3DGS the paper cites.
//
// One CTA per 32x32 output tile and channel, the three channels of a tile in
// one cluster (k_loss_split), or for large launches one CTA per tile that
// takes the channels in turn (k_loss; the rule is at launch_loss).  A CTA loads the channel's exposed colour x and target y over
// the tile plus a 10-pixel halo as (x, y) pairs, blurs the five moment maps
// separably over a 5-pixel halo, forms the SSIM map and its partials w.r.t. (mu_x, E[x^2], E[xy]) and
// blurs those back (the adjoint of a zero-padded symmetric correlation is the
// same correlation).  dL/dC = A^T dL/dE[C] needs all three channels: k_loss adds
// them up in registers; in a cluster each CTA leaves its dL/dE[C] in shared memory and, after a cluster barrier, CTA j
// reads the other two and writes component j.
//
// Bound: FP32 issue.  Four of the maps are kept as pairs, (mu_x, mu_y) and
// (E[x^2], E[y^2]), so a tap is one 8-byte load and one two-lane FMA per pair,
// and the tap weights are literals.  In every pass a thread slides the 11 taps
// along a run of 3-8 outputs held in registers; the run lengths give the 256
// threads 728 = 2.8 x 256, 252, 168 and 256 equal items, and the row strides
// (43 and 33) keep the passes whose lanes go down rows off shared bank
// conflicts.  The maps of later passes reuse the space of those consumed:
// 63.8 KB, three CTAs (24 warps) per SM.  A CTA per channel also cuts the
// length of the longest chain to a third where a small image leaves SMs idle.
// One CTA for all three channels -> this: 115.7 -> 104.9 us (1280x1024), 40.6 ->
// 32.9 (647x481), 24.2 -> 13.8 (256x192: 48 tiles).
// Per-CTA partial sums of |.|, SSIM and dL/dE are reduced afterwards in a
// fixed order (k_loss_final).
#include "gl_internal.h"

#include <cooperative_groups.h>

#include <algorithm>

namespace gl {

namespace {

constexpr int LT = 32;
constexpr int HW = 5;                 // window half width
constexpr int RA = LT + 4 * HW;       // 52
constexpr int RB = LT + 2 * HW;       // 42
constexpr int kThreads = 256;
constexpr int kNP = 14;               // partials per CTA: 12 dL/dE, sum|d|, sum SSIM
constexpr int HR = 3;                 // outputs per thread, horizontal moment pass (RB = 14 x 3)
constexpr int VR = 7;                 // outputs per thread, vertical moment pass (RB = 6 x 7)
constexpr int AHR = 8;                // outputs per thread, horizontal adjoint pass (LT = 4 x 8)
constexpr int AVR = 4;                // outputs per thread, vertical adjoint pass (LT = 8 x 4)
constexpr int GS = RB + 1;            // row stride of the partial maps
constexpr int HS = LT + 1;            // row stride of their horizontal blur
static_assert(RB % HR == 0 && RB % VR == 0 && LT % AHR == 0 && LT % AVR == 0, "run lengths must tile the maps");
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

// The window exp(-k^2 / (2 1.5^2)) / sum, |k| <= 5, every operation rounded to
// single precision.  SSIM divides small differences of blurred squares, where
// the image is flat by little more than C2: there the rounding of the taps and
// of the moments shows in the gradient (exact taps move dL/dC by 2.6e-5; x^2 +
// y^2 blurred as one map costs the loss digits, because 2 xy no longer rounds
// as it does; means by fused instead of rounded products move dL/dC by 1.6e-5).
// So every sum here takes its terms in one fixed form and order.
constexpr float kT0 = 0x1.0d957p-10f;
constexpr float kT1 = 0x1.f1fe06p-8f;
constexpr float kT2 = 0x1.26eb18p-5f;
constexpr float kT3 = 0x1.bff102p-4f;
constexpr float kT4 = 0x1.b43c4p-3f;
constexpr float kT5 = 0x1.106562p-2f;
__host__ __device__ constexpr float tap(int k)
{
    return k == 0 || k == 10 ? kT0 : k == 1 || k == 9 ? kT1 : k == 2 || k == 8 ? kT2 : k == 3 || k == 7 ? kT3
         : k == 4 || k == 6 ? kT4 : kT5;
}

// two FMAs on a register pair, both lanes rounded to nearest
__device__ __forceinline__ float2 fma2(float a, float2 b, float2 c)
{
    return __ffma2_rn(make_float2(a, a), b, c);
}

// (x, y) over the tile and halo (later the three SSIM partial maps: a pair
// map and a single one), then the two pair maps and the single one of the
// moments (later the horizontally blurred partials)
constexpr size_t kXYBytes = 12 * RB * GS;   // >= 8 RA RA
constexpr size_t kSmemBytes = kXYBytes + 20 * RA * RB;
static_assert(8 * RA * RA <= kXYBytes && 12 * RB * HS <= 16 * RA * RB && kXYBytes % 8 == 0, "aliased maps must fit");
static_assert(4 * LT * LT <= 8 * RA * RA, "the channel's gradient map reuses the partial maps");

// One view passed by value (the stateless and allocation-free entry points).
struct LossOne {
    const float* rgb;
    const float* target;
    const float* E;
    float* dL;
    int W, H;
};

// Grid: a cluster of three CTAs (the channels; SPLIT) or one CTA per 32x32
// loss tile over all views.  With `views` null the single view `one` is used; otherwise view,
// images, exposure and weight come from the descriptors and images are the
// concatenated ones.
template <bool SPLIT>
__device__ __forceinline__ void
loss_tile(LossOne one, const ViewDesc* __restrict__ views, int V, const float* __restrict__ rgb_all,
       float* __restrict__ dL_all, float lambda, float* __restrict__ part)
{
    namespace cg = cooperative_groups;
    const float* rgb = one.rgb;
    const float* target = one.target;
    const float* E = one.E;
    float* dL_drgb = one.dL;
    int W = one.W, H = one.H;
    float weight = 1.0f;
    int lt = SPLIT ? blockIdx.x / 3 : blockIdx.x;
    const int tile = lt;
    if (views) {
        const int v = view_of_ltile(views, V, lt);
        const ViewDesc& d = views[v];
        lt -= d.ltile_base;
        rgb = rgb_all + 3 * d.pix_base;
        dL_drgb = dL_all + 3 * d.pix_base;
        target = d.target;
        E = d.E;
        W = d.cam.W;
        H = d.cam.H;
        weight = d.weight;
    }
    extern __shared__ __align__(16) unsigned char smraw[];
    float2* xy = reinterpret_cast<float2*>(smraw);                 // RA x RA
    float2* gab = xy;                                              // RB x GS (reuses xy after the horizontal pass)
    float* gcm = reinterpret_cast<float*>(gab + RB * GS);          // RB x GS
    float* gout = reinterpret_cast<float*>(smraw);                 // LT x LT (reuses the partial maps)
    float2* hm = reinterpret_cast<float2*>(smraw + kXYBytes);      // 2 maps, RA rows x RB cols
    float* hp = reinterpret_cast<float*>(hm + 2 * RA * RB);        // E[xy]
    float2* hab = hm;                                              // RB rows x HS (reuses hm)
    float* hc = reinterpret_cast<float*>(hab + RB * HS);           // RB rows x HS
    __shared__ float red[kNP][kThreads / 32];
    __shared__ float chsum[2];       // SPLIT: the channel's sums of |.| and SSIM
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int LTX = (W + LT - 1) / LT;
    const int ox = (lt % LTX) * LT, oy = (lt / LTX) * LT;
    const float invN = 1.0f / (3.0f * (float)W * (float)H);
    const float gS = -lambda * invN * weight;
    const float gL1 = (1.0f - lambda) * invN * weight;

    float l1acc = 0.0f, sacc = 0.0f;
    static_assert(LT * (LT / AVR) == kThreads, "one adjoint run per thread");
    const int c = tid % LT, r0 = (tid / LT) * AVR;
    float dC[AVR][3];   // !SPLIT: dL/dC of the thread's pixels
    const int first = SPLIT ? blockIdx.x % 3 : 0;   // SPLIT: the rank in the cluster
#pragma unroll 1
    for (int ch = first; ch < (SPLIT ? first + 1 : 3); ch++) {
    const float e0 = E ? E[4 * ch] : (ch == 0 ? 1.0f : 0.0f), e1 = E ? E[4 * ch + 1] : (ch == 1 ? 1.0f : 0.0f);
    const float e2 = E ? E[4 * ch + 2] : (ch == 2 ? 1.0f : 0.0f), e3 = E ? E[4 * ch + 3] : 0.0f;
    // a warp per row, two columns per lane; a tile whose halo lies inside the
    // image takes the loads without bounds
    const bool inner = ox >= 2 * HW && oy >= 2 * HW && ox + LT + 2 * HW <= W && oy + LT + 2 * HW <= H;
    if (inner) {
        const size_t p0 = 3 * ((size_t)(oy - 2 * HW + wid) * W + (ox - 2 * HW + lane));
        const float* cp = rgb + p0;
        const float* tp = target + p0 + ch;
        const size_t step = 3 * (size_t)(kThreads / 32) * W;
#pragma unroll 4
        for (int r = wid; r < RA; r += kThreads / 32, cp += step, tp += step) {
            xy[r * RA + lane] = make_float2(e0 * cp[0] + e1 * cp[1] + e2 * cp[2] + e3, tp[0]);
            if (lane < RA - 32)
                xy[r * RA + 32 + lane] = make_float2(e0 * cp[96] + e1 * cp[97] + e2 * cp[98] + e3, tp[96]);
        }
    } else {
        for (int r = wid; r < RA; r += kThreads / 32) {
            const int gy = oy - 2 * HW + r;
            const bool rowin = gy >= 0 && gy < H;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int c = lane + 32 * k, gx = ox - 2 * HW + c;
                float2 v = make_float2(0.0f, 0.0f);
                if (rowin && c < RA && gx >= 0 && gx < W) {
                    const size_t p = 3 * ((size_t)gy * W + gx);
                    v.x = e0 * rgb[p] + e1 * rgb[p + 1] + e2 * rgb[p + 2] + e3;
                    v.y = target[p + ch];
                }
                if (c < RA) xy[r * RA + c] = v;
            }
        }
    }
    __syncthreads();
    // horizontal pass of the moments: runs of HR outputs of one row
    for (int e = tid; e < RA * (RB / HR); e += kThreads) {
        const int r = e / (RB / HR), c0 = (e % (RB / HR)) * HR;
        float2 m[HR], q[HR];
        float p[HR];
#pragma unroll
        for (int o = 0; o < HR; o++) {
            m[o] = q[o] = make_float2(0.0f, 0.0f);
            p[o] = 0.0f;
        }
#pragma unroll
        for (int k = 0; k < HR + 10; k++) {
            const float2 v = xy[r * RA + c0 + k];
#pragma unroll
            for (int o = 0; o < HR; o++)
                if (k >= o && k - o < 11) {
                    const float w = tap(k - o);
                    const float2 t = __fmul2_rn(make_float2(w, w), v);
                    m[o] = __fadd2_rn(m[o], t);
                    q[o] = __ffma2_rn(t, v, q[o]);
                    p[o] = fmaf(t.x, v.y, p[o]);
                }
        }
#pragma unroll
        for (int o = 0; o < HR; o++) {
            const int i = r * RB + c0 + o;
            hm[i] = m[o];
            hm[RA * RB + i] = q[o];
            hp[i] = p[o];
        }
    }
    __syncthreads();
    // vertical pass, SSIM and its partials: runs of VR rows of one column
    if (tid < RB * (RB / VR)) {
        const int c = tid % RB, r0 = (tid / RB) * VR;
        float2 m[VR], q[VR];
        float p[VR];
#pragma unroll
        for (int o = 0; o < VR; o++) {
            m[o] = q[o] = make_float2(0.0f, 0.0f);
            p[o] = 0.0f;
        }
#pragma unroll
        for (int k = 0; k < VR + 10; k++) {
            const int i = (r0 + k) * RB + c;
            const float2 v = hm[i], s = hm[RA * RB + i];
            const float z = hp[i];
#pragma unroll
            for (int o = 0; o < VR; o++)
                if (k >= o && k - o < 11) {
                    m[o] = fma2(tap(k - o), v, m[o]);
                    q[o] = fma2(tap(k - o), s, q[o]);
                    p[o] = fmaf(tap(k - o), z, p[o]);
                }
        }
        const int gx = ox - HW + c;
        const bool colin = gx >= 0 && gx < W, core = c >= HW && c < HW + LT;
#pragma unroll
        for (int o = 0; o < VR; o++) {
            const int r = r0 + o;
            const int gy = oy - HW + r;
            float ga = 0.0f, gb = 0.0f, gc = 0.0f;
            if (colin && gy >= 0 && gy < H) {
                const float mx = m[o].x, my = m[o].y, exx = q[o].x, eyy = q[o].y, exy = p[o];
                const float sxx = exx - mx * mx, syy = eyy - my * my, sxy = exy - mx * my;
                const float N1 = 2.f * mx * my + kC1, N2 = 2.f * sxy + kC2;
                const float D1 = mx * mx + my * my + kC1, D2 = sxx + syy + kC2;
                // one approximate reciprocal (a few ulp) serves S and both
                // partials: 1/D1 = D2 iD, 1/D2 = D1 iD
                const float iD = __fdividef(1.0f, D1 * D2);
                const float S = N1 * N2 * iD;
                if (core && r >= HW && r < HW + LT) sacc += S;
                const float dN1 = N2 * iD, dN2 = N1 * iD, dD1 = -S * (D2 * iD), dD2 = -S * (D1 * iD);
                const float dmx = dN1 * 2.f * my - dN2 * 2.f * my + dD1 * 2.f * mx - dD2 * 2.f * mx;
                ga = gS * dmx;
                gb = gS * dD2;
                gc = gS * 2.f * dN2;
            }
            gab[r * GS + c] = make_float2(ga, gb);
            gcm[r * GS + c] = gc;
        }
    }
    __syncthreads();
    // adjoint, horizontal: a thread per (row, run of AHR outputs), lanes down the rows
    if (tid < RB * (LT / AHR)) {
        const int r = tid % RB, c0 = (tid / RB) * AHR;
        float2 a[AHR];
        float b[AHR];
#pragma unroll
        for (int o = 0; o < AHR; o++) { a[o] = make_float2(0.0f, 0.0f); b[o] = 0.0f; }
#pragma unroll
        for (int k = 0; k < AHR + 10; k++) {
            const float2 v = gab[r * GS + c0 + k];
            const float s = gcm[r * GS + c0 + k];
#pragma unroll
            for (int o = 0; o < AHR; o++)
                if (k >= o && k - o < 11) {
                    a[o] = fma2(tap(k - o), v, a[o]);
                    b[o] = fmaf(tap(k - o), s, b[o]);
                }
        }
#pragma unroll
        for (int o = 0; o < AHR; o++) {
            hab[r * HS + c0 + o] = a[o];
            hc[r * HS + c0 + o] = b[o];
        }
    }
    __syncthreads();
    // adjoint, vertical, and dL/dE[C] of the tile's pixels: runs of AVR rows
    // of a column (x, y read again: their shared copy is overwritten)
    float pe[4] = {0.0f, 0.0f, 0.0f, 0.0f};   // exposure gradient: sum g C_j (j < 3), sum g
    float g[AVR];
    {
        float2 a[AVR];
        float b[AVR];
#pragma unroll
        for (int o = 0; o < AVR; o++) { a[o] = make_float2(0.0f, 0.0f); b[o] = 0.0f; }
#pragma unroll
        for (int k = 0; k < AVR + 10; k++) {
            const float2 v = hab[(r0 + k) * HS + c];
            const float s = hc[(r0 + k) * HS + c];
#pragma unroll
            for (int o = 0; o < AVR; o++)
                if (k >= o && k - o < 11) {
                    a[o] = fma2(tap(k - o), v, a[o]);
                    b[o] = fmaf(tap(k - o), s, b[o]);
                }
        }
#pragma unroll
        for (int o = 0; o < AVR; o++) {
            const int gx = ox + c, gy = oy + r0 + o;
            g[o] = 0.0f;
            if (gx < W && gy < H) {
                const size_t p = 3 * ((size_t)gy * W + gx);
                const float c0 = rgb[p], c1 = rgb[p + 1], c2 = rgb[p + 2];
                const float x = e0 * c0 + e1 * c1 + e2 * c2 + e3, y = target[p + ch];
                const float d = x - y;
                l1acc += fabsf(d);
                g[o] = a[o].x + 2.f * x * a[o].y + y * b[o] + gL1 * (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f));
                pe[0] += g[o] * c0; pe[1] += g[o] * c1; pe[2] += g[o] * c2; pe[3] += g[o];
            }
            if (SPLIT) {
                gout[(r0 + o) * LT + c] = g[o];
            } else {
                dC[o][0] = ch == 0 ? e0 * g[o] : fmaf(e0, g[o], dC[o][0]);
                dC[o][1] = ch == 0 ? e1 * g[o] : fmaf(e1, g[o], dC[o][1]);
                dC[o][2] = ch == 0 ? e2 * g[o] : fmaf(e2, g[o], dC[o][2]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        float v = pe[i];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
        if (lane == 0) red[4 * ch + i][wid] = v;
    }
    }
    {
        const float vals[2] = {l1acc, sacc};
#pragma unroll
        for (int i = 0; i < 2; i++) {
            float v = vals[i];
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
            if (lane == 0) red[12 + i][wid] = v;
        }
    }
    __syncthreads();
    float* prow = part + (size_t)tile * kNP;
    if constexpr (SPLIT) {
        const int ch = first;
        cg::cluster_group cluster = cg::this_cluster();
        if (tid < 6) {
            const int k = tid < 4 ? 4 * ch + tid : 8 + tid;
            float v = 0.0f;
            for (int ww = 0; ww < kThreads / 32; ww++) v += red[k][ww];
            if (tid < 4) prow[k] = v;
            else chsum[tid - 4] = v;
        }
        // a CTA's shared memory may be touched from another one only once all
        // are known to run: sums and gradients are left at home and read after
        // this barrier
        cluster.sync();
        // component ch of dL/dC = sum over channels k of A[k][ch] dL/dE[C]_k
        const float f0 = E ? E[ch] : (ch == 0 ? 1.0f : 0.0f), f1 = E ? E[4 + ch] : (ch == 1 ? 1.0f : 0.0f);
        const float f2 = E ? E[8 + ch] : (ch == 2 ? 1.0f : 0.0f);
        const float* g0 = cluster.map_shared_rank(gout, 0);
        const float* g1 = cluster.map_shared_rank(gout, 1);
        const float* g2 = cluster.map_shared_rank(gout, 2);
        float s1 = 0.0f, s2 = 0.0f;   // on their way while the gradients are added
        if (ch == 0 && tid < 2) {
            s1 = cluster.map_shared_rank(chsum, 1)[tid];
            s2 = cluster.map_shared_rank(chsum, 2)[tid];
        }
#pragma unroll
        for (int o = 0; o < AVR; o++) {
            const int gx = ox + c, gy = oy + r0 + o, i = (r0 + o) * LT + c;
            const float v = fmaf(f2, g2[i], fmaf(f1, g1[i], f0 * g0[i]));
            if (gx < W && gy < H) dL_drgb[3 * ((size_t)gy * W + gx) + ch] = v;
        }
        if (ch == 0 && tid < 2) prow[12 + tid] = chsum[tid] + s1 + s2;
        cluster.sync();   // the shared memory read by the other CTAs stays until they are done
    } else {
        if (tid < kNP) {
            float v = 0.0f;
            for (int ww = 0; ww < kThreads / 32; ww++) v += red[tid][ww];
            prow[tid] = v;
        }
#pragma unroll
        for (int o = 0; o < AVR; o++) {
            const int gx = ox + c, gy = oy + r0 + o;
            if (gx < W && gy < H) {
                const size_t p = 3 * ((size_t)gy * W + gx);
                dL_drgb[p] = dC[o][0];
                dL_drgb[p + 1] = dC[o][1];
                dL_drgb[p + 2] = dC[o][2];
            }
        }
    }
}

__global__ void __cluster_dims__(3, 1, 1) __launch_bounds__(kThreads, 3)
k_loss_split(LossOne one, const ViewDesc* __restrict__ views, int V, const float* __restrict__ rgb_all,
             float* __restrict__ dL_all, float lambda, float* __restrict__ part)
{
    loss_tile<true>(one, views, V, rgb_all, dL_all, lambda, part);
}

__global__ void __launch_bounds__(kThreads, 3)
k_loss(LossOne one, const ViewDesc* __restrict__ views, int V, const float* __restrict__ rgb_all,
       float* __restrict__ dL_all, float lambda, float* __restrict__ part)
{
    loss_tile<false>(one, views, V, rgb_all, dL_all, lambda, part);
}

// Sums the per-tile partials in a fixed order (in three floats, FloatSum; again
// in double where that overflows).  Single view (views null): block 0 over
// [0, nblk) -> loss_out, dE_out.  Views: block v over the view's loss tiles ->
// loss_v[v] (unweighted) and, if the view has Em, one Adam step of its exposure
// on the (already weighted) gradient.
// Bound by latency: one CTA reads nblk x 14 floats in order (thread t takes
// elements t, t + 1022, ...: 1022 = 73 x 14, so always the same partial),
// eight loads in flight, then a warp per partial adds the 73 sums.
// A warp per partial in double -> this: 13.3 -> 5.2 us (1280x1024).
constexpr int kRedBatch = 8;
constexpr int kRedRows = 73;
constexpr int kRedThreads = 1024;
static_assert(kRedRows * kNP <= kRedThreads && kRedRows <= 96, "a warp takes at most three sums a lane");
__global__ void __launch_bounds__(kRedThreads)
k_loss_final(const float* __restrict__ part, int nblk, int W, int H, float lambda,
             float* __restrict__ loss_out, float* __restrict__ dE_out,
             const ViewDesc* __restrict__ views, float* __restrict__ loss_v, float b1,
             float b2, float eps, float lr, const uint64_t* __restrict__ abort)
{
    __shared__ FloatSum sums[kRedRows * kNP];
    __shared__ FloatSum tot[kNP];
    __shared__ double s_invN;
    int begin = 0;
    float* Ev = nullptr;
    float* Em = nullptr;
    float bc1 = 1.f, bc2 = 1.f;
    if (views) {
        const ViewDesc& d = views[blockIdx.x];
        begin = d.ltile_base;
        W = d.cam.W;
        H = d.cam.H;
        nblk = ((W + LT - 1) / LT) * ((H + LT - 1) / LT);
        Ev = d.E;
        Em = d.Em;
        bc1 = d.e_bc1;
        bc2 = d.e_bc2;
    }
    const int tid = threadIdx.x;
    constexpr int STRIDE = kRedRows * kNP;
    if (tid < STRIDE) {
        const float* src = part + (size_t)begin * kNP + tid;
        int left = (nblk * kNP - tid + STRIDE - 1) / STRIDE;   // elements of this thread
        FloatSum S{};
        for (; left > 0; left -= kRedBatch, src += STRIDE * kRedBatch) {
            float x[kRedBatch];
#pragma unroll
            for (int b = 0; b < kRedBatch; b++) x[b] = b < left ? src[STRIDE * b] : 0.0f;
#pragma unroll
            for (int b = 0; b < kRedBatch; b++)
                if (b < left) S.add(x[b]);
        }
        sums[tid] = S;
    } else if (tid == kRedThreads - 1) {
        s_invN = 1.0 / (3.0 * (double)W * (double)H);   // while the others load
    }
    __syncthreads();
    const int k = tid >> 5, lane = tid & 31;
    if (k < kNP) {
        FloatSum S{};
        FloatSum q[3];
#pragma unroll
        for (int j = 0; j < 3; j++) q[j] = lane + 32 * j < kRedRows ? sums[(lane + 32 * j) * kNP + k] : FloatSum{};
#pragma unroll
        for (int j = 0; j < 3; j++) S.add(q[j]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) S.add(S.xor_lane(off));
        if (lane == 0) tot[k] = S;
    }
    __syncthreads();
    // (few warps take the sums to double: its lanes are few)
    if (tid == 32) {
        const float* src = part + (size_t)begin * kNP;
        const double l1 = sum_value(tot[12], src + 12, nblk, kNP), ss = sum_value(tot[13], src + 13, nblk, kNP);
        const double L = (1.0 - lambda) * l1 * s_invN + lambda * (1.0 - ss * s_invN);
        if (views) { if (loss_v) loss_v[blockIdx.x] = (float)L; }
        else if (loss_out) *loss_out = (float)L;
    }
    if (tid < 12) {
        const int i = tid;
        const float g = (float)sum_value(tot[i], part + (size_t)begin * kNP + i, nblk, kNP);
        if (!views && dE_out) dE_out[i] = g;
        if (Ev && Em && !(abort && abort[1])) {
            const float m = b1 * Em[i] + (1.0f - b1) * g;
            const float v = b2 * Em[12 + i] + (1.0f - b2) * g * g;
            Em[i] = m;
            Em[12 + i] = v;
            Ev[i] -= lr * (m / bc1) / (sqrtf(v / bc2) + eps);
        }
    }
}

__global__ void k_apply_exposure(const float* __restrict__ src, float* __restrict__ dst, int64_t P,
                                 float e0, float e1, float e2, float e3, float e4, float e5, float e6,
                                 float e7, float e8, float e9, float e10, float e11)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < P;
         p += (int64_t)gridDim.x * blockDim.x) {
        const float c0 = src[3 * p], c1 = src[3 * p + 1], c2 = src[3 * p + 2];
        dst[3 * p] = e0 * c0 + e1 * c1 + e2 * c2 + e3;
        dst[3 * p + 1] = e4 * c0 + e5 * c1 + e6 * c2 + e7;
        dst[3 * p + 2] = e8 * c0 + e9 * c1 + e10 * c2 + e11;
    }
}

}  // namespace

int loss_partials_needed(int W, int H)
{
    return ((W + LT - 1) / LT) * ((H + LT - 1) / LT) * kNP;
}

namespace {
// Tiles per two SMs from which a CTA takes all three channels of a tile: one
// and a half waves of three CTAs per SM.  Then no cluster waits for its slowest
// channel and the channels share the rows in L1; below, a third of the chain per
// CTA counts more.  A cluster and one CTA per tile, by tiles: 13 and 25 us (48),
// 33.2 and 37.3 (336), 44.3 and 38.1 (456, one full wave), 48.9 and 51.2 (525), 56.1
// and 58.2 (620), 61.7 and 59.4 (690), 67.9 and 67.6 (768), 78.3 and 69.0 (896), 108 and
// 98 (1,280), 167 and 146 (2,040), 850 and 656 (9.5k, 12 views): from 684 tiles the
// one CTA is never slower.
constexpr int kWholeTilesPer2Sms = 9;

gl_status launch_loss(const LossOne& one, const ViewDesc* views, int V, const float* rgb, float* dL, float lambda,
                      float* part, int tiles, cudaStream_t s)
{
    GL_TRY(ensure_smem_limit(reinterpret_cast<const void*>(&k_loss_split), (int)kSmemBytes));
    GL_TRY(ensure_smem_limit(reinterpret_cast<const void*>(&k_loss), (int)kSmemBytes));
    if (2 * (int64_t)tiles < kWholeTilesPer2Sms * (int64_t)sm_count()) {
        k_loss_split<<<3 * tiles, kThreads, kSmemBytes, s>>>(one, views, V, rgb, dL, lambda, part);
    } else {
        k_loss<<<tiles, kThreads, kSmemBytes, s>>>(one, views, V, rgb, dL, lambda, part);
    }
    return GL_OK;
}
}  // namespace

gl_status photometric_loss(const float* rgb, const float* target, const float* E, int W, int H,
                           float lambda, float* dL_drgb, float* part, float* loss_out, float* dE_out,
                           cudaStream_t s)
{
    const int nblk = ((W + LT - 1) / LT) * ((H + LT - 1) / LT);
    LossOne one{rgb, target, E, dL_drgb, W, H};
    GL_TRY(launch_loss(one, nullptr, 0, nullptr, nullptr, lambda, part, nblk, s));
    k_loss_final<<<1, kRedThreads, 0, s>>>(part, nblk, W, H, lambda, loss_out, dE_out, nullptr, nullptr, 0.f, 0.f,
                                        0.f, 0.f, nullptr);
    count_launches(2);
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

gl_status photometric_loss_views(const View& v, const float* rgb, float lambda, float* dL_drgb, float* part,
                                 float* loss_v, float b1, float b2, float eps, float lr, cudaStream_t s,
                                 const uint64_t* abort)
{
    LossOne one{};
    GL_TRY(launch_loss(one, v.d_desc(), v.V, rgb, dL_drgb, lambda, part, v.nltiles, s));
    k_loss_final<<<v.V, kRedThreads, 0, s>>>(part, 0, 0, 0, lambda, nullptr, nullptr, v.d_desc(), loss_v, b1, b2, eps,
                                          lr, abort);
    count_launches(2);
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

gl_status apply_exposure(const float* src, float* dst, const float E[12], int64_t P, cudaStream_t s)
{
    int blocks = (int)std::min<int64_t>(8 * (int64_t)sm_count(), (P + 255) / 256);
    if (blocks < 1) blocks = 1;
    k_apply_exposure<<<blocks, 256, 0, s>>>(src, dst, P, E[0], E[1], E[2], E[3], E[4], E[5], E[6], E[7],
                                            E[8], E[9], E[10], E[11]);
    count_launches(1);
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

}  // namespace gl
