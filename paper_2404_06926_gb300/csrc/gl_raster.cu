// gl_raster.cu -- front-to-back compositing (Eq. 4-7) and its adjoint.
//
// Work unit: one warp per (work item, block of 8 x 4D pixels).  A work item
// is a screen tile (TS x TS) or, for a tile whose list holds at least 2 seg
// records, one segment of seg consecutive records of that list.  Every
// pixel block of a tile is rendered by its own warp, and a long list is
// split along depth, so neither a heavy tile nor a deep one (the road's
// vanishing point gathers tens of thousands of far Gaussians in a few
// tiles) is the critical path of one warp.  Items are numbered heaviest
// first.  Lane l owns the D pixels (x0 + l % 8, y0 + l / 8 + 4 j), j < D:
// the records a warp stages and the warp reduction of the backward are
// shared by D pixels per lane.
//
// Records are permuted into sorted-instance order after binning, so a
// tile's Gaussians are contiguous: a batch is 32 NB records (NB per lane, the
// next batch prefetched into registers); the warp ballots which records'
// alpha boxes touch its pixel block, compacts the hits in shared memory in
// depth order and evaluates only those.  A Gaussian outside the block's box
// fails the alpha test at every pixel of the block, so skipping it changes
// no result.
//
// Forward of a whole tile: per pixel, blend until the transmittance would
// fall below 1e-4; keep the final transmittance and the position (in the
// tile's list) of the last blended Gaussian, so the backward recomputes T by
// division.
//
// Forward of a split tile: a CTA per pixel block walks the list in rounds,
// each warp blending the next run of kSub records from T = 1 (a pixel whose
// own run falls below 1e-4 stops there: it cannot matter what follows).  The
// stop rule fires inside a run exactly when the transmittance entering it
// times the run's own product falls below 1e-4 (the running value inside is
// the entering one times the run's running product, and that product only
// decreases), so the runs' products in order give the entering values and
// the run each pixel stops in; that run is replayed from its entering value
// to find the truncated sums, and the walk ends when every pixel has stopped:
// nothing behind the stop is blended.  Runs of a segment are folded into its
// sums, from which the backward's starting state of each segment follows
// back to front: the transmittance after the segment and the normalised
// colour blended behind it (R = C_next + T_next * R_next over the later
// segments).  The transmittance is the product of the per-run products, so
// it can differ from a single running product by float rounding.
// Against a segment pass over the whole list and three launches for prefix,
// replay and finish: 106 -> 79 us (250k Gaussians, 640x512), 236 -> 184 us (1M,
// 1280x1024), 3,853 -> 3,338 us (12 views of 2M), 225 -> 185 us (render,
// 1920x1080).
//
// Backward: every item walked back to front from its starting state (the
// final transmittance and R = 0 for a whole tile).  Per hit a lane leaves two
// numbers per pixel in shared memory, the blend weight and dL/d(exponent);
// every 16 / D hits the warp turns over: lanes own hits instead of pixels and
// form each hit's ten sums (colour 3, dL/dpower moments 6, depth 1) from
// those rows, then add them to the Gaussian's accumulator with two vector
// atomics (or, deterministic, store them per instance and pixel block).
//
// Scheduling: either one unit per warp of a grid that covers the bound on
// units, or a persistent grid (sized to the resident warps) whose warps take
// the next unit from a counter; the number of units is read on the device.
#include "gl_internal.h"

#include <map>
#include <mutex>

namespace gl {

namespace {

constexpr int kWarpsPerBlock = 8;
// Prefetch slots (32 records each) of a batch of 32 NB records: the whole
// next batch up to 64 records, one sub-batch ahead beyond.
template <int NB>
constexpr int pf_slots() { return NB <= 2 ? NB : 1; }
constexpr int kMinBlocksPg = 3;   // resident CTAs per SM, per-Gaussian backward
constexpr int kNG = 10;           // screen-space gradient sums per Gaussian (rows of kGradStride floats)
constexpr int kSegFields = 8;   // per (segment item, pixel): see below
constexpr int kSub = 128;       // records of a run (a warp's share of a round on a split tile)
constexpr int kBackBatch = 4;   // segments whose sums one load round trip brings (back walk)

// Warps per CTA of the forward; they walk a split tile's pixel block together.
// Eight shorten the deepest lists' walks, which is what a single frame waits
// for; four leave less idle at the rounds' barriers and overshoot the stop by
// less, which counts once there is far more work than the chip holds
// (8 and 4 warps: 79 and 112 us on 250k Gaussians at 640x512, 10k pixel
// blocks; 91 and 132 at 1280x1024, 41k; 1M Gaussians, one view: 241 and 303 us at
// 65k blocks, 247 and 267 at 88k, 249 and 251 at 93k, 252 and 244 at 102k, 255 and 238
// at 115k, 359 and 338 at 259k; 300k Gaussians: 115 and 113 at 88k, 125 and 120 at
// 102k; 3,968 and 3,338 us on 12 views of 2M, 303k; the line lies at 95k).  (The
// staging and exchange of every variant fit in 48 KB of static shared memory.)
template <int NB, int D>
constexpr int wpb_fwd(bool wide) { return D == 4 || NB == 8 ? 2 : (NB == 1 && D == 1 && wide ? 8 : 4); }
// pixel blocks per resident warp from which CTAs of four warps are taken
constexpr int kWideUnits = 26;
// registers: 80 a thread (24 warps per SM) at the default shape, which spill 92 to
// 128 bytes
template <int NB, int D>
constexpr int warps_fwd() { return D == 4 ? 12 : (NB == 1 && D == 1 ? 24 : 16); }

// segstate fields of a segment item: 0 transmittance after the segment, 1-3 R
// (colour behind it, normalised), 4 R depth, 5 R opacity; until the back walk
// 1-5 hold the segment's own sums from T = 1 and 6 its transmittance product.
// Written for the segments up to the one a pixel stops in.
__device__ __forceinline__ size_t seg_at(int w, int k, int p, int TS)
{
    return ((size_t)w * kSegFields + k) * (size_t)(TS * TS) + p;
}

// Inputs shared by the kernels (passed by value).
struct RasterArgs {
    int TS, V, nblk, seg;
    const uint2* items;          // (tile, segment), heaviest first
    const uint32_t* heads;       // first item of each split tile
    const uint64_t* ctl;         // ctl[6] work items, ctl[7] items of split tiles, ctl[11] split tiles
    const uint32_t* ranges;      // [first, last + 1) of each tile's list
    const float4 *s0, *s1, *s2, *s3;
    const uint32_t* sgid;        // owning (view, Gaussian) pair of each sorted instance
    const ViewDesc* views;
    float* segstate;
    int* work;                   // persistent grid: unit counters; nullptr: one unit per warp
};

struct RasterOut {
    float *rgb, *depth, *opac, *Tfin;
    uint32_t* ncon;
};

struct RasterGrad {
    const float* Tfin;
    const uint32_t* ncon;
    const float *dL_drgb, *dL_ddepth, *dL_dopac;
    float* g2d;                  // atomic accumulation per (view, Gaussian)
    // deterministic mode: per (instance, pixel block) sums, indexed by the
    // instance's emission index (sinst of its sorted position)
    float* part;
    const uint32_t* sinst;
    uint32_t* pmask;             // per instance: the pixel blocks whose sums are in `part`
};

struct Unit {
    int w, wb;             // work item, pixel block within the tile
    int j, nseg;           // segment of the item and segments of its tile
    int lx0, ly0;          // pixel block origin within the tile
    int x0, y0;            // absolute pixel origin of the pixel block in its view
    int W, H;              // the view's image size
    long long pix_base;    // the view's first pixel in the concatenated images
    uint32_t trs, tre;     // the tile's whole list
    uint32_t rs, re;       // the item's part of it
};

// Pixel block wb of item w.
template <int D>
__device__ __forceinline__ void unit_at(int w, int wb, const RasterArgs& A, Unit& U)
{
    // pixel blocks per tile, blocks per tile row and the segment length are
    // powers of two: shifts and masks instead of integer divisions
    const int TS = A.TS, bsh = __ffs(TS >> 3) - 1;
    U.w = w;
    U.wb = wb;
    const uint2 it = A.items[U.w];
    const int tile = (int)it.x;
    U.j = (int)it.y;
    const int v = view_of_tile(A.views, A.V, tile);
    const ViewDesc& d = A.views[v];
    const int lt = tile - d.tile_base;
    U.lx0 = (U.wb & ((1 << bsh) - 1)) * 8;
    U.ly0 = (U.wb >> bsh) * 4 * D;
    U.x0 = (lt % d.TX) * TS + U.lx0;
    U.y0 = (lt / d.TX) * TS + U.ly0;
    U.W = d.cam.W;
    U.H = d.cam.H;
    U.pix_base = d.pix_base;
    U.trs = A.ranges[2 * tile];
    U.tre = A.ranges[2 * tile + 1];
    const uint32_t L = U.tre - U.trs;
    U.nseg = (A.seg > 0 && L >= 2u * (uint32_t)A.seg) ? (int)((L + A.seg - 1) >> (__ffs(A.seg) - 1)) : 1;
    if (U.nseg > 1) {
        U.rs = U.trs + (uint32_t)U.j * (uint32_t)A.seg;
        U.re = min(U.tre, U.rs + (uint32_t)A.seg);
    } else {
        U.rs = U.trs;
        U.re = U.tre;
    }
}

template <int D>
__device__ __forceinline__ void unit_of(int u, const RasterArgs& A, Unit& U)
{
    unit_at<D>(u >> (__ffs(A.nblk) - 1), u & (A.nblk - 1), A, U);
}

__device__ __forceinline__ bool box_hit(const float4 box, float bx0, float bx1, float by0, float by1)
{
    return !(box.y < bx0 || box.x > bx1 || box.w < by0 || box.z > by1);
}

// Next unit from the counter (the same value in every lane).
__device__ __forceinline__ int next_unit(int* work, int lane)
{
    int u = 0;
    if (lane == 0) u = atomicAdd(work, 1);
    return __shfl_sync(kFull, u, 0);
}

// One warp's staged hits of the forward, from index 1: records r0, r1 and r2
// with the list position + 1 in r2.w (bits).  Entry 0 is a record that reaches
// no pixel, the partner of an odd count's first hit.
template <int NB>
struct FwdHits {
    float4 r0[32 * NB + 1], r1[32 * NB + 1], r2[32 * NB + 1];
    __device__ __forceinline__ void init(int lane)
    {
        if (lane == 0) {
            r0[0] = r2[0] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            r1[0] = make_float4(0.0f, -3.0e38f, 0.0f, 0.0f);
        }
        __syncwarp();
    }
};

// Front-to-back blend of the records [a, b) of a tile list for the warp's
// pixel block.  Per pixel: T (running transmittance), colour, depth and
// opacity sums (XD; without it they stay 0) and the last blended position
// (relative to trs).  A pixel stops, without blending, at the first record
// whose T * (1 - alpha) (SCALED: times its Tin) falls below 1e-4; its alpha
// threshold `thr` then becomes infinite, as it is from the start for pixels
// that take no part.
template <int NB, int D, bool XD, bool SCALED>
__device__ __forceinline__ void blend_range(const RasterArgs& A, uint32_t a, uint32_t b, uint32_t trs, float px,
                                            const float (&py)[D], float bx0, float bx1, float by0, float by1,
                                            const float (&Tin)[D], float (&thr)[D], float (&T)[D], float (&C0)[D],
                                            float (&C1)[D], float (&C2)[D], float (&Dd)[D], float (&Oo)[D],
                                            uint32_t (&last)[D], FwdHits<NB>& F, int lane)
{
    const unsigned lt = (1u << lane) - 1u;
    constexpr int PF = pf_slots<NB>();
    float4 n0[PF], n1[PF], n2[PF], n3[PF];
#pragma unroll
    for (int q = 0; q < PF; q++) {
        const uint32_t i = a + q * 32 + lane;
        if (i < b) { n0[q] = A.s0[i]; n1[q] = A.s1[i]; n2[q] = A.s2[i]; n3[q] = A.s3[i]; }
    }
    for (uint32_t base = a; base < b; base += 32 * NB) {
        bool lane_done = true;
#pragma unroll
        for (int j = 0; j < D; j++) lane_done = lane_done && thr[j] > 0.0f;
        if (__all_sync(kFull, lane_done)) break;
        int nh = 0;
#pragma unroll
        for (int q = 0; q < NB; q++) {
            const int sl = PF == NB ? q : 0;
            const float4 c0 = n0[sl], c1 = n1[sl], c3 = n3[sl];
            float4 c2 = n2[sl];
            const uint32_t i = base + q * 32 + lane;
            const uint32_t ni = i + 32 * PF;
            if (ni < b) { n0[sl] = A.s0[ni]; n1[sl] = A.s1[ni]; n2[sl] = A.s2[ni]; n3[sl] = A.s3[ni]; }
            const bool hit = i < b && box_hit(c3, bx0, bx1, by0, by1);
            const unsigned mask = __ballot_sync(kFull, hit);
            if (hit) {
                const int k = 1 + nh + __popc(mask & lt);
                c2.w = __uint_as_float(i - trs + 1u);
                F.r0[k] = c0; F.r1[k] = c1; F.r2[k] = c2;
            }
            nh += __popc(mask);
        }
        __syncwarp();
        // Two hits at a time: their alphas are independent, only T forms a
        // chain.  Branch-free: a pixel that is done or that a hit misses takes
        // alpha = 0, which leaves T and its sums exactly unchanged (and T at
        // or above the stop); one that stops here blends with weight 0 and
        // keeps its T.
        for (int k = 1 - (nh & 1); k <= nh; k += 2) {
            float4 g0[2], g1[2], c[2];
#pragma unroll
            for (int i = 0; i < 2; i++) { g0[i] = F.r0[k + i]; g1[i] = F.r1[k + i]; c[i] = F.r2[k + i]; }
            float al[2][D];
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < D; j++) {
                    float alpha;
                    al[i][j] = pair_alpha(g0[i], g1[i], px, py[j], thr[j], alpha) ? alpha : 0.0f;
                }
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < D; j++) {
                    const float al_ = i && thr[j] > 0.0f ? 0.0f : al[i][j];   // the first may have stopped the pixel
                    const float tT = __fmul_rn(T[j], __fsub_rn(1.0f, al_));
                    const bool halt = (SCALED ? __fmul_rn(Tin[j], tT) : tT) < kTransMin;
                    const float wgt = halt ? 0.0f : al_ * T[j];
                    T[j] = halt ? T[j] : tT;
                    thr[j] = halt ? kNoAlpha : thr[j];
                    last[j] = wgt > 0.0f ? __float_as_uint(c[i].w) : last[j];
                    C0[j] += c[i].x * wgt; C1[j] += c[i].y * wgt; C2[j] += c[i].z * wgt;
                    if (XD) {
                        Dd[j] += g1[i].z * wgt;
                        Oo[j] += wgt;
                    }
                }
        }
        __syncwarp();
    }
}

// Per-lane pixel geometry of a unit: lane l owns pixels (l % 8, l / 8 + 4 j),
// or (HALF) one pixel of its half-warp's 4 x 4 block: the lower half-warp has
// the left block, the upper one the right.
template <int D, bool HALF = false>
struct LanePix {
    int x, y;
    float px, py[D];   // relative to the tile's origin, as the records' means
    bool inside[D];
    int p[D];          // pixel index within the tile
    float bx0, bx1, by0, by1;
    __device__ __forceinline__ LanePix(const Unit& U, int TS, int lane)
    {
        static_assert(!HALF || D == 1, "a half-warp block has a pixel per lane");
        const int lx = HALF ? (lane >> 4) * 4 + (lane & 3) : lane & 7, ly = HALF ? (lane >> 2) & 3 : lane >> 3;
        x = U.x0 + lx;
        y = U.y0 + ly;
        px = (float)(U.lx0 + lx);
#pragma unroll
        for (int j = 0; j < D; j++) {
            py[j] = (float)(U.ly0 + ly + 4 * j);
            inside[j] = x < U.W && y + 4 * j < U.H;
            p[j] = (U.ly0 + ly + 4 * j) * TS + U.lx0 + lx;
        }
        bx0 = (float)U.x0;
        bx1 = (float)(U.x0 + 7);
        by0 = (float)U.y0;
        by1 = (float)(U.y0 + 4 * D - 1);
    }
    __device__ __forceinline__ size_t pix(const Unit& U, int j) const
    {
        return (size_t)U.pix_base + (size_t)(y + 4 * j) * U.W + x;
    }
};

// A whole tile's pixel block, by one warp.
template <int NB, int D, bool XD>
__device__ __forceinline__ void fwd_item(const Unit& U, const RasterArgs& A, const RasterOut& O, FwdHits<NB>& F,
                                         int lane)
{
    const LanePix<D> L(U, A.TS, lane);
    float T[D], C0[D], C1[D], C2[D], Dd[D], Oo[D], thr[D];
    uint32_t last[D];
#pragma unroll
    for (int j = 0; j < D; j++) {
        T[j] = 1.0f; C0[j] = C1[j] = C2[j] = Dd[j] = Oo[j] = 0.0f;
        last[j] = 0;
        thr[j] = L.inside[j] ? kLog2AlphaMin : kNoAlpha;
    }
    blend_range<NB, D, XD, false>(A, U.trs, U.tre, U.trs, L.px, L.py, L.bx0, L.bx1, L.by0, L.by1, T, thr, T, C0, C1,
                                  C2, Dd, Oo, last, F, lane);
#pragma unroll
    for (int j = 0; j < D; j++) {
        if (!L.inside[j]) continue;
        const size_t p = L.pix(U, j);
        O.rgb[3 * p] = C0[j]; O.rgb[3 * p + 1] = C1[j]; O.rgb[3 * p + 2] = C2[j];
        if (O.depth) O.depth[p] = Dd[j];
        if (O.opac) O.opac[p] = Oo[j];
        O.Tfin[p] = T[j];
        O.ncon[p] = last[j];
    }
}

// Shared memory of a CTA's forward.  ex: the runs of a round, per warp and
// pixel, in three buffers (one being written, one being replayed, one being
// folded); tot: warp 0's running sums per pixel.
template <int NB, int D, int WPB>
struct FwdShared {
    enum { ET, EC0, EC1, EC2, ELAST, ETR, ED, EO, NEX };   // ETR: product up to the stop
    enum { C0, C1, C2, LAST, S0, S1, S2, ST, DD, OO, SD, SO, NTOT };
    FwdHits<NB> hits[WPB];
    float ex[3][WPB][NEX][32 * D];
    float tot[NTOT][32 * D];
    int unit;
};

// Warp 0 adds the `runs` runs of a round, in order and up to the run `stop` a
// pixel stops in (-1: it stopped earlier), to the pixel's and the segment's
// sums; t is the transmittance entering the round.  A finished segment's sums
// go to its state.  At the stop, Tst and jstop get the final transmittance and
// the segment.
template <int NB, int D, bool XD, int WPB>
__device__ __forceinline__ void fold_round(const Unit& U, const RasterArgs& A, FwdShared<NB, D, WPB>& M, int buf, int s0,
                                           int runs, int nrun, int seg_runs, int p, int q, float t, int stop,
                                           float& Tst, int& jstop)
{
    using FS = FwdShared<NB, D, WPB>;
    float C0 = M.tot[FS::C0][p], C1 = M.tot[FS::C1][p], C2 = M.tot[FS::C2][p];
    float S0 = M.tot[FS::S0][p], S1 = M.tot[FS::S1][p], S2 = M.tot[FS::S2][p], ST = M.tot[FS::ST][p];
    float Dd = 0.f, Oo = 0.f, SD = 0.f, SO = 0.f;
    if (XD) {
        Dd = M.tot[FS::DD][p]; Oo = M.tot[FS::OO][p];
        SD = M.tot[FS::SD][p]; SO = M.tot[FS::SO][p];
    }
    uint32_t lp = __float_as_uint(M.tot[FS::LAST][p]);
    for (int v = 0; v < runs && v <= stop; v++) {
        const float (*e)[32 * D] = M.ex[buf][v];
        const bool at_stop = v == stop;
        const float f0 = e[FS::EC0][p], f1 = e[FS::EC1][p], f2 = e[FS::EC2][p];
        C0 += t * f0; C1 += t * f1; C2 += t * f2;
        S0 += ST * f0; S1 += ST * f1; S2 += ST * f2;
        if (XD) {
            const float fd = e[FS::ED][p], fo = e[FS::EO][p];
            Dd += t * fd; Oo += t * fo;
            SD += ST * fd; SO += ST * fo;
        }
        const uint32_t ls = __float_as_uint(e[FS::ELAST][p]);
        if (ls) lp = ls;
        const float tr = at_stop ? e[FS::ETR][p] : e[FS::ET][p];
        t = __fmul_rn(t, tr);
        ST = __fmul_rn(ST, tr);
        const int run = s0 + v;
        if (at_stop || (run & (seg_runs - 1)) == seg_runs - 1 || run == nrun - 1) {
            const int sg = run / seg_runs, wi = U.w + sg;
            float* S = A.segstate;
            S[seg_at(wi, 0, q, A.TS)] = t;
            S[seg_at(wi, 1, q, A.TS)] = S0;
            S[seg_at(wi, 2, q, A.TS)] = S1;
            S[seg_at(wi, 3, q, A.TS)] = S2;
            if (XD) {
                S[seg_at(wi, 4, q, A.TS)] = SD;
                S[seg_at(wi, 5, q, A.TS)] = SO;
            }
            S[seg_at(wi, 6, q, A.TS)] = ST;
            S0 = S1 = S2 = SD = SO = 0.0f;
            ST = 1.0f;
            if (at_stop) {
                Tst = t;
                jstop = sg;
            }
        }
    }
    M.tot[FS::C0][p] = C0; M.tot[FS::C1][p] = C1; M.tot[FS::C2][p] = C2;
    M.tot[FS::S0][p] = S0; M.tot[FS::S1][p] = S1; M.tot[FS::S2][p] = S2; M.tot[FS::ST][p] = ST;
    if (XD) {
        M.tot[FS::DD][p] = Dd; M.tot[FS::OO][p] = Oo;
        M.tot[FS::SD][p] = SD; M.tot[FS::SO][p] = SO;
    }
    M.tot[FS::LAST][p] = __uint_as_float(lp);
}

// A split tile's pixel block, by the whole CTA (every warp calls it).  One
// barrier per round: after it every warp finds the stops on its own, replays
// its run if one is in it, and goes on to the next round, while warp 0 folds
// the round before.
template <int NB, int D, bool XD, int WPB>
__device__ __forceinline__ void fwd_split(const Unit& U, const RasterArgs& A, const RasterOut& O,
                                          FwdShared<NB, D, WPB>& M, int lane, int w)
{
    using FS = FwdShared<NB, D, WPB>;
    const LanePix<D> L(U, A.TS, lane);
    const uint32_t sub = (uint32_t)min(A.seg, kSub);
    const int seg_runs = A.seg / (int)sub;   // a power of two
    const int nrun = (int)((U.tre - U.trs + sub - 1) / sub);
    float Trun[D];             // transmittance entering the round (of open pixels; the same in every warp)
    bool open[D];              // not stopped yet
    float Tprev[D], Tst[D];    // warp 0: entering the round to fold; at the stop
    int sprev[D], jstop[D];    // warp 0: stops of the round to fold; segment of the stop
#pragma unroll
    for (int j = 0; j < D; j++) {
        Trun[j] = Tprev[j] = 1.0f;
        Tst[j] = -1.0f;
        open[j] = L.inside[j];
        sprev[j] = -1;
        jstop[j] = U.nseg - 1;
        if (w == 0)
            for (int k = 0; k < FS::NTOT; k++) M.tot[k][j * 32 + lane] = k == FS::ST ? 1.0f : 0.0f;
    }
    int buf = 0, bprev = 0, s0 = 0, sp0 = 0;
    while (true) {
        const int s = s0 + w, runs = min(WPB, nrun - s0);
        const uint32_t a = U.trs + (uint32_t)s * sub, b = min(U.tre, a + sub);
        float T[D], c0[D], c1[D], c2[D], dd[D], oo[D], thr[D];
        uint32_t last[D];
#pragma unroll
        for (int j = 0; j < D; j++) {
            T[j] = 1.0f; c0[j] = c1[j] = c2[j] = dd[j] = oo[j] = 0.0f;
            last[j] = 0;
            thr[j] = open[j] ? kLog2AlphaMin : kNoAlpha;
        }
        if (s < nrun) {
            blend_range<NB, D, XD, false>(A, a, b, U.trs, L.px, L.py, L.bx0, L.bx1, L.by0, L.by1, T, thr, T, c0, c1,
                                          c2, dd, oo, last, M.hits[w], lane);
#pragma unroll
            for (int j = 0; j < D; j++) {
                const int p = j * 32 + lane;
                // a pixel that fell below 1e-4 within the run stops in it
                // whatever enters it
                M.ex[buf][w][FS::ET][p] = thr[j] > 0.0f ? 0.0f : T[j];
                M.ex[buf][w][FS::EC0][p] = c0[j];
                M.ex[buf][w][FS::EC1][p] = c1[j];
                M.ex[buf][w][FS::EC2][p] = c2[j];
                M.ex[buf][w][FS::ELAST][p] = __uint_as_float(last[j]);
                if (XD) {
                    M.ex[buf][w][FS::ED][p] = dd[j];
                    M.ex[buf][w][FS::EO][p] = oo[j];
                }
            }
        }
        __syncthreads();
        if (w == 0 && s0 > 0) {
#pragma unroll
            for (int j = 0; j < D; j++)
                fold_round<NB, D, XD, WPB>(U, A, M, bprev, sp0, WPB, nrun, seg_runs, j * 32 + lane, L.p[j], Tprev[j],
                                      sprev[j], Tst[j], jstop[j]);
        }
        // entering transmittance of every run, in order; the run each pixel
        // stops in
        float Tin[D];
        int stop[D];
        bool mine = false, any_open = false;
#pragma unroll
        for (int j = 0; j < D; j++) {
            float Tb = Trun[j];
            Tprev[j] = Tb;
            Tin[j] = 1.0f;
            stop[j] = open[j] ? WPB : -1;
            for (int v = 0; v < runs; v++) {
                const float t = __fmul_rn(Tb, M.ex[buf][v][FS::ET][j * 32 + lane]);
                if (stop[j] == WPB) {
                    if (v == w) Tin[j] = Tb;
                    if (t < kTransMin) stop[j] = v; else Tb = t;
                }
            }
            mine = mine || stop[j] == w;
            sprev[j] = stop[j];
            Trun[j] = Tb;
            open[j] = open[j] && stop[j] == WPB;
            any_open = any_open || open[j];
        }
        if (__any_sync(kFull, mine)) {
            // replay this warp's run from its entering transmittance for the
            // pixels that stop in it
#pragma unroll
            for (int j = 0; j < D; j++) {
                T[j] = 1.0f; c0[j] = c1[j] = c2[j] = dd[j] = oo[j] = 0.0f;
                last[j] = 0;
                thr[j] = stop[j] == w ? kLog2AlphaMin : kNoAlpha;
            }
            blend_range<NB, D, XD, true>(A, a, b, U.trs, L.px, L.py, L.bx0, L.bx1, L.by0, L.by1, Tin, thr, T, c0, c1,
                                         c2, dd, oo, last, M.hits[w], lane);
#pragma unroll
            for (int j = 0; j < D; j++) {
                const int p = j * 32 + lane;
                if (stop[j] != w) continue;
                M.ex[buf][w][FS::ETR][p] = T[j];
                M.ex[buf][w][FS::EC0][p] = c0[j];
                M.ex[buf][w][FS::EC1][p] = c1[j];
                M.ex[buf][w][FS::EC2][p] = c2[j];
                M.ex[buf][w][FS::ELAST][p] = __uint_as_float(last[j]);
                if (XD) {
                    M.ex[buf][w][FS::ED][p] = dd[j];
                    M.ex[buf][w][FS::EO][p] = oo[j];
                }
            }
        }
        bprev = buf;
        sp0 = s0;
        buf = buf == 2 ? 0 : buf + 1;
        s0 += WPB;
        // (the same in every warp)
        if (s0 >= nrun || !__any_sync(kFull, any_open)) break;
    }
    __syncthreads();
    if (w != 0) return;
    int smax = 0;
#pragma unroll
    for (int j = 0; j < D; j++) {
        const int p = j * 32 + lane;
        fold_round<NB, D, XD, WPB>(U, A, M, bprev, sp0, min(WPB, nrun - sp0), nrun, seg_runs, p, L.p[j], Tprev[j], sprev[j],
                              Tst[j], jstop[j]);
        if (!L.inside[j]) continue;
        const size_t o = L.pix(U, j);
        O.rgb[3 * o] = M.tot[FS::C0][p];
        O.rgb[3 * o + 1] = M.tot[FS::C1][p];
        O.rgb[3 * o + 2] = M.tot[FS::C2][p];
        if (XD && O.depth) O.depth[o] = M.tot[FS::DD][p];
        if (XD && O.opac) O.opac[o] = M.tot[FS::OO][p];
        O.Tfin[o] = Tst[j] >= 0.0f ? Tst[j] : Trun[j];
        O.ncon[o] = __float_as_uint(M.tot[FS::LAST][p]);
        smax = max(smax, jstop[j]);
    }
    // the backward's starting states, back to front from the stop segment
    // (each lane reads back only what it wrote)
    for (int off = 16; off > 0; off >>= 1) smax = max(smax, __shfl_xor_sync(kFull, smax, off));
    constexpr int NF = XD ? 6 : 4;   // sums (3 or 5) and the product
#pragma unroll
    for (int j = 0; j < D; j++) {
        if (!L.inside[j]) continue;
        const int q = L.p[j];
        float* S = A.segstate;
        float R[NF - 1];
#pragma unroll
        for (int k = 0; k < NF - 1; k++) R[k] = 0.0f;
        for (int b0 = smax; b0 >= 0; b0 -= kBackBatch) {
            float f[kBackBatch][NF];
#pragma unroll
            for (int b = 0; b < kBackBatch; b++) {
                const int sg = b0 - b;
                if (sg >= 0 && sg <= jstop[j]) {
#pragma unroll
                    for (int k = 0; k < NF - 1; k++) f[b][k] = S[seg_at(U.w + sg, 1 + k, q, A.TS)];
                    f[b][NF - 1] = S[seg_at(U.w + sg, 6, q, A.TS)];
                }
            }
#pragma unroll
            for (int b = 0; b < kBackBatch; b++) {
                const int sg = b0 - b;
                if (sg >= 0 && sg <= jstop[j]) {
#pragma unroll
                    for (int k = 0; k < NF - 1; k++) {
                        S[seg_at(U.w + sg, 1 + k, q, A.TS)] = R[k];
                        R[k] = f[b][k] + f[b][NF - 1] * R[k];
                    }
                }
            }
        }
    }
}

// Split tiles first (a CTA per pixel block; counters work[1] of a persistent
// grid, the first CTAs otherwise), then the other tiles (a warp per pixel
// block).
template <int NB, int D, bool XD, int WPB>
__global__ void __launch_bounds__(32 * WPB, warps_fwd<NB, D>() / WPB) k_raster_fwd(RasterArgs A, RasterOut O)
{
    __shared__ FwdShared<NB, D, WPB> M;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nsh = __ffs(A.nblk) - 1;
    const int nsplit = (int)A.ctl[11] * A.nblk;
    const int split_items = (int)A.ctl[7];
    const int nwhole = ((int)A.ctl[6] - split_items) * A.nblk;
    Unit U;
    M.hits[w].init(lane);
    if (A.work) {
        while (nsplit > 0) {
            __syncthreads();
            if (threadIdx.x == 0) M.unit = atomicAdd(A.work + 1, 1);
            __syncthreads();
            const int u = M.unit;
            if (u >= nsplit) break;
            unit_at<D>((int)A.heads[u >> nsh], u & (A.nblk - 1), A, U);
            fwd_split<NB, D, XD, WPB>(U, A, O, M, lane, w);
        }
        for (int u = next_unit(A.work, lane); u < nwhole; u = next_unit(A.work, lane)) {
            unit_at<D>(split_items + (u >> nsh), u & (A.nblk - 1), A, U);
            fwd_item<NB, D, XD>(U, A, O, M.hits[w], lane);
        }
    } else if ((int)blockIdx.x < nsplit) {
        unit_at<D>((int)A.heads[blockIdx.x >> nsh], blockIdx.x & (A.nblk - 1), A, U);
        fwd_split<NB, D, XD, WPB>(U, A, O, M, lane, w);
    } else {
        const int u = ((int)blockIdx.x - nsplit) * WPB + w;
        if (u < nwhole) {
            unit_at<D>(split_items + (u >> nsh), u & (A.nblk - 1), A, U);
            fwd_item<NB, D, XD>(U, A, O, M.hits[w], lane);
        }
    }
}

// Sum 16 per-lane values over the warp.  On return lane l holds the total of
// value (l >> 1): each butterfly level halves the slots a lane keeps.
__device__ __forceinline__ float warp_transpose_reduce16(float (&v)[16])
{
    const unsigned lane = threadIdx.x & 31u;
    {
        const bool up = lane & 16u;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            float send = up ? v[k] : v[k + 8];
            float keep = up ? v[k + 8] : v[k];
            v[k] = keep + __shfl_xor_sync(kFull, send, 16);
        }
    }
    {
        const bool up = lane & 8u;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            float send = up ? v[k] : v[k + 4];
            float keep = up ? v[k + 4] : v[k];
            v[k] = keep + __shfl_xor_sync(kFull, send, 8);
        }
    }
    {
        const bool up = lane & 4u;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            float send = up ? v[k] : v[k + 2];
            float keep = up ? v[k + 2] : v[k];
            v[k] = keep + __shfl_xor_sync(kFull, send, 4);
        }
    }
    {
        const bool up = lane & 2u;
        float send = up ? v[0] : v[1];
        float keep = up ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(kFull, send, 2);
    }
    return v[0] + __shfl_xor_sync(kFull, v[0], 1);
}

// Warps per CTA of the per-pixel backward: its staging takes 6.5 KB a warp at
// the default shape, and CTAs of 4 warps (2 with 256-record batches) keep
// every variant's within 48 KB of static shared memory.
template <int NB>
constexpr int wpb_bwd() { return NB <= 4 ? 4 : 2; }
// registers: 96 a thread (20 warps per SM) at the default shape (32 bytes spilled
// without depth gradients)
template <int NB, int D>
constexpr int minb_bwd() { return (D > 1 ? 12 : (NB <= 2 ? 20 : 16)) / wpb_bwd<NB>(); }

constexpr uint32_t kNoOwner = 0xffffffffu;

// The per-pixel backward.  Bound by instruction issue (the deepest tiles'
// latency in small frames).  Folding every hit's nine sums across the warp
// took 37 of its ~100 instructions and the moments behind them ten more; the
// turn-over replaces both by one 8-byte store per hit and about ten
// instructions.  Two hits are evaluated together because a warp's chain, not
// its throughput, ends the kernel on a single frame; the registers that takes
// are worth more than warps: 64 / 80 / 96 / 128 a thread (32 / 24 / 20 / 16
// warps per SM) gave 107 / 85 / 79 / 79 us on the 250k-Gaussian street at
// 640x512 and 264 / 237 / 233 / 258 us on the 1M one at 1280x1024 (before: 126
// and 306 us, and 1,218 -> 650 us with unsplit lists and depth gradients).
// Staging of one warp: `sv` holds a row per
// pending hit: (blend weight, dL/d(exponent)) of each of the block's 32 D
// pixels.  The turn-over reads a row in parts of 16 pixels (two pixel rows),
// one part per lane: the row stride S and the part stride PS (in float2) put
// the 16 lanes of each half-warp phase of the 8-byte loads on different banks
// (2 S mod 32 and 2 PS mod 32 are (2, -), (4, 2) and (8, 2) words for D = 1,
// 2, 4).
template <int NB, int D>
struct BwdWarp {
    static constexpr int H = 16 / D;                  // pending hits per turn-over
    static constexpr int PARTS = 2 * D;               // lanes per hit, 16 pixels each
    static constexpr int PS = D == 1 ? 16 : 17;
    static constexpr int S = D == 1 ? 33 : (D == 2 ? 82 : 148);
    static_assert(H * PARTS == 32 && S >= PARTS * PS, "one lane per (hit, part)");
    // hit records from index 1, r1.w owner, r2.w list position (bits); entry 0
    // is a record that reaches no pixel, the partner of an odd last hit
    float4 r0[32 * NB + 1], r1[32 * NB + 1], r2[32 * NB + 1];
    float4 pix[32 * D];                               // per pixel: dL/dC, dL/dD
    float4 info[H];                                   // pending hits: tile-relative mean, owner (bits; kNoOwner: none)
    float2 sv[H * S];
};

// The n pending hits' sums: lane (h, part) adds up hit h over the part's two
// pixel rows, the parts are folded across the warp, and the lower half-warp
// emits slots 0-3 and 8-9, the upper one slots 4-7.  The moments take dx, dy
// per pixel (no expansion about the block), so they round as per-pixel sums.
template <bool EXTRA, int NB, int D, bool DET>
__device__ __forceinline__ void bwd_turn_over(const RasterArgs& A, const RasterGrad& G, const BwdWarp<NB, D>& W,
                                              int n, float bx, float by, int wb, int lane)
{
    using BW = BwdWarp<NB, D>;
    constexpr int H = BW::H;
    const int h = lane % H, part = lane / H;
    const float4 in = W.info[h];
    const float2* row = W.sv + h * BW::S + part * BW::PS;
    const float4* pc = W.pix + part * 16;
    const float dya = in.y - (by + (float)(2 * part)), dyb = in.y - (by + (float)(2 * part + 1));
    // even and odd columns apart: chains of four terms (the column moments) or
    // eight fused ones, then pairs of sums.  Against 64 bits the gradients are as
    // far off as with a fold of the pixels' terms (rms of five gradients, 5k
    // Gaussians at 256x192: 3.2 3.8 2.6 4.2 3.1e-6, folded 3.3 3.9 2.7 4.1 3.1e-6);
    // chains of four throughout gain nothing and cost 3 to 11% of the half-warp
    // kernel.
    float c0[2] = {0.f, 0.f}, c1[2] = {0.f, 0.f}, c2[2] = {0.f, 0.f}, cD[2] = {0.f, 0.f}, mxx[2] = {0.f, 0.f};
    float m0a[2] = {0.f, 0.f}, m0b[2] = {0.f, 0.f}, mxa[2] = {0.f, 0.f}, mxb[2] = {0.f, 0.f};
#pragma unroll
    for (int x = 0; x < 8; x++) {
        const int e = x & 1;
        const float2 va = row[x], vb = row[8 + x];
        const float4 ga = pc[x], gb = pc[8 + x];
        const float dx = in.x - (bx + (float)x), dx2 = dx * dx;
        c0[e] = fmaf(va.x, ga.x, c0[e]); c1[e] = fmaf(va.x, ga.y, c1[e]); c2[e] = fmaf(va.x, ga.z, c2[e]);
        c0[e] = fmaf(vb.x, gb.x, c0[e]); c1[e] = fmaf(vb.x, gb.y, c1[e]); c2[e] = fmaf(vb.x, gb.z, c2[e]);
        if (EXTRA) cD[e] = fmaf(vb.x, gb.w, fmaf(va.x, ga.w, cD[e]));
        m0a[e] += va.y; m0b[e] += vb.y;
        mxa[e] = fmaf(va.y, dx, mxa[e]); mxb[e] = fmaf(vb.y, dx, mxb[e]);
        mxx[e] = fmaf(vb.y, dx2, fmaf(va.y, dx2, mxx[e]));
    }
    const float ma = m0a[0] + m0a[1], mb = m0b[0] + m0b[1], xa = mxa[0] + mxa[1], xb = mxb[0] + mxb[1];
    // slots 0-3 (lo), 4-7 (hi), 8-9
    float lo[4] = {c0[0] + c0[1], c1[0] + c1[1], c2[0] + c2[1], ma + mb};
    float hi[4] = {xa + xb, fmaf(dya, ma, dyb * mb), mxx[0] + mxx[1], fmaf(dya, xa, dyb * xb)};
    float s8 = fmaf(dya * dya, ma, dyb * dyb * mb), s9 = cD[0] + cD[1];
#pragma unroll
    for (int off = H; off < 16; off <<= 1) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            lo[k] += __shfl_xor_sync(kFull, lo[k], off);
            hi[k] += __shfl_xor_sync(kFull, hi[k], off);
        }
        s8 += __shfl_xor_sync(kFull, s8, off);
        if (EXTRA) s9 += __shfl_xor_sync(kFull, s9, off);
    }
    const bool up = lane & 16;
    float4 r;
    float* rp = &r.x;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float send = up ? lo[k] : hi[k], keep = up ? hi[k] : lo[k];
        rp[k] = keep + __shfl_xor_sync(kFull, send, 16);
    }
    s8 += __shfl_xor_sync(kFull, s8, 16);
    if (EXTRA) s9 += __shfl_xor_sync(kFull, s9, 16);
    const uint32_t id = __float_as_uint(in.z);
    if (h < n && (lane & 15) < H && id != kNoOwner) {
        float* dst = DET ? G.part + ((size_t)id * A.nblk + wb) * kGradStride : G.g2d + (size_t)id * kGradStride;
        if (DET) {
            *reinterpret_cast<float4*>(dst + (up ? 4 : 0)) = r;
            if (!up) {
                *reinterpret_cast<float2*>(dst + 8) = make_float2(s8, EXTRA ? s9 : 0.0f);
                atomicOr(G.pmask + id, 1u << wb);
            }
        } else {
            atomicAdd(reinterpret_cast<float4*>(dst + (up ? 4 : 0)), r);
            if (!up) {
                if (EXTRA) atomicAdd(reinterpret_cast<float2*>(dst + 8), make_float2(s8, s9));
                else atomicAdd(dst + 8, s8);
            }
        }
    }
}

template <bool EXTRA, int NB, int D, bool DET>
__device__ __forceinline__ void bwd_item(int u, const RasterArgs& A, const RasterGrad& G, BwdWarp<NB, D>& W, int lane)
{
    using BW = BwdWarp<NB, D>;
    Unit U;
    unit_of<D>(u, A, U);
    const LanePix<D> L(U, A.TS, lane);
    const unsigned lt = (1u << lane) - 1u;
    // per pixel: transmittance, what is blended behind (colour; EXTRA: depth,
    // opacity), the gradients of the pixel's outputs
    float T[D], R[D][5], g0[D], g1[D], g2[D], gD[D], gO[D];
    uint32_t last[D];
    uint32_t wmax = 0;
#pragma unroll
    for (int j = 0; j < D; j++) {
        T[j] = 1.0f;
        g0[j] = g1[j] = g2[j] = gD[j] = gO[j] = 0.0f;
#pragma unroll
        for (int k = 0; k < 5; k++) R[j][k] = 0.0f;
        last[j] = 0;
        if (L.inside[j]) {
            const size_t p = L.pix(U, j);
            last[j] = G.ncon[p];
            g0[j] = G.dL_drgb[3 * p]; g1[j] = G.dL_drgb[3 * p + 1]; g2[j] = G.dL_drgb[3 * p + 2];
            if (EXTRA) {
                gD[j] = G.dL_ddepth ? G.dL_ddepth[p] : 0.0f;
                gO[j] = G.dL_dopac ? G.dL_dopac[p] : 0.0f;
            }
            if (U.nseg == 1) {
                T[j] = G.Tfin[p];
            } else if (last[j] > U.rs - U.trs) {   // (no state behind the stop segment)
                const float* S = A.segstate;
                const int i = L.p[j];
                T[j] = S[seg_at(U.w, 0, i, A.TS)];
#pragma unroll
                for (int k = 0; k < (EXTRA ? 5 : 3); k++) R[j][k] = S[seg_at(U.w, 1 + k, i, A.TS)];
            }
        }
        W.pix[j * 32 + lane] = make_float4(g0[j], g1[j], g2[j], gD[j]);
        wmax = max(wmax, last[j]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wmax = max(wmax, __shfl_xor_sync(kFull, wmax, off));
    // positions at or beyond the last contributor reach no pixel of the block
    const uint32_t end = min(U.re, U.trs + wmax);
    if (end <= U.rs) return;
    const float bx = (float)U.lx0, by = (float)U.ly0;
    int slot = 0;   // pending hits
    if (lane == 0) {
        W.r0[0] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        W.r1[0] = make_float4(0.0f, -3.0e38f, 0.0f, __uint_as_float(kNoOwner));
        W.r2[0] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    // batches from the back: [bstart, bstart + 32 NB) with bstart = end - 32 NB k, clipped at rs
    constexpr int BS = 32 * NB;
    constexpr int PF = pf_slots<NB>();
    int64_t bstart = (int64_t)end - BS;
    float4 n0[PF], n1[PF], n2[PF], n3[PF];
    uint32_t ng[PF];
#pragma unroll
    for (int b = 0; b < PF; b++) {
        const int64_t i = bstart + b * 32 + lane;
        ng[b] = 0;
        if (i >= (int64_t)U.rs) {
            n0[b] = A.s0[i]; n1[b] = A.s1[i]; n2[b] = A.s2[i]; n3[b] = A.s3[i];
            ng[b] = DET ? G.sinst[i] : A.sgid[i];
        }
    }
    for (; bstart + BS > (int64_t)U.rs; bstart -= BS) {
        int nh = 0;
#pragma unroll
        for (int b = 0; b < NB; b++) {
            const int sl = PF == NB ? b : 0;
            const float4 c0 = n0[sl], c3 = n3[sl];
            float4 c1 = n1[sl], c2 = n2[sl];
            c1.w = __uint_as_float(ng[sl]);
            const int64_t i = bstart + b * 32 + lane;
            // next: the same sub-batch of the batch before (whole-batch
            // prefetch), else the next sub-batch of this one, or the first
            // of the batch before
            const int64_t ni = PF == NB ? i - BS : (b < NB - 1 ? i + 32 : i + 32 - 2 * BS);
            if (ni >= (int64_t)U.rs) {
                n0[sl] = A.s0[ni]; n1[sl] = A.s1[ni]; n2[sl] = A.s2[ni]; n3[sl] = A.s3[ni];
                ng[sl] = DET ? G.sinst[ni] : A.sgid[ni];
            }
            const bool hit = i >= (int64_t)U.rs && box_hit(c3, L.bx0, L.bx1, L.by0, L.by1);
            const unsigned mask = __ballot_sync(kFull, hit);
            if (hit) {
                const int k = 1 + nh + __popc(mask & lt);
                c2.w = __uint_as_float((uint32_t)(i - U.trs));
                W.r0[k] = c0; W.r1[k] = c1; W.r2[k] = c2;
            }
            nh += __popc(mask);
        }
        __syncwarp();
        // Two hits at a time: their alphas are independent, only T and what is
        // behind form a chain.  Branch-free, without selects where arithmetic
        // does: a pixel a hit does not reach takes alpha = 0, which leaves T
        // (T / 1) and the state behind exactly unchanged and zeroes its sums.
        // (Hits that reach no pixel at all are too few to be worth a vote.)
        for (int k = nh; k >= 1; k -= 2) {
            float4 a[2], b[2], c[2];
#pragma unroll
            for (int i = 0; i < 2; i++) { a[i] = W.r0[k - i]; b[i] = W.r1[k - i]; c[i] = W.r2[k - i]; }
            float al[2][D];
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const uint32_t pos = __float_as_uint(c[i].w);
#pragma unroll
                for (int j = 0; j < D; j++) {
                    float dx, dy, alpha;
                    bool capped;
                    const bool live = pair_eval_nb(a[i], b[i], L.px, L.py[j], dx, dy, alpha, capped) && pos < last[j];
                    al[i][j] = live ? alpha : 0.0f;
                }
            }
#pragma unroll
            for (int i = 0; i < 2; i++) {
                float2* sv = W.sv + (slot + i) * BW::S;
#pragma unroll
                for (int j = 0; j < D; j++) {
                    const float al_ = al[i][j];
                    T[j] = __fdividef(T[j], 1.0f - al_);
                    const float wgt = al_ * T[j];
                    // dL/dalpha = T g . (c - R); what is blended behind moves
                    // toward this Gaussian by alpha.  (Keeping only g . R of
                    // the colour behind saves four instructions and loses
                    // digits of the pose gradient: c is close to R.)
                    const float d0 = c[i].x - R[j][0], d1 = c[i].y - R[j][1], d2 = c[i].z - R[j][2];
                    float dot = g0[j] * d0 + g1[j] * d1 + g2[j] * d2;
                    R[j][0] = fmaf(al_, d0, R[j][0]);
                    R[j][1] = fmaf(al_, d1, R[j][1]);
                    R[j][2] = fmaf(al_, d2, R[j][2]);
                    if (EXTRA) {
                        const float dD = b[i].z - R[j][3], dO = 1.0f - R[j][4];
                        dot += gD[j] * dD + gO[j] * dO;
                        R[j][3] = fmaf(al_, dD, R[j][3]);
                        R[j][4] = fmaf(al_, dO, R[j][4]);
                    }
                    // dL/d(exponent) = alpha dL/dalpha, none at the cap
                    const float gp = al_ < kAlphaMax ? wgt * dot : 0.0f;
                    const int p = j * 32 + lane;
                    sv[p + (p >> 4) * (BW::PS - 16)] = make_float2(wgt, gp);
                }
                if (lane == 0) W.info[slot + i] = make_float4(a[i].x, a[i].y, b[i].w, 0.0f);
            }
            slot += 2;
            if (slot == BW::H) {
                __syncwarp();
                bwd_turn_over<EXTRA, NB, D, DET>(A, G, W, BW::H, bx, by, U.wb, lane);
                slot = 0;
                __syncwarp();
            }
        }
        __syncwarp();
    }
    if (slot > 0) bwd_turn_over<EXTRA, NB, D, DET>(A, G, W, slot, bx, by, U.wb, lane);
    __syncwarp();
}

// Half-warp blocks (one pixel per lane).  A Gaussian of the usual few pixels
// reaches a quarter to a third of an 8 x 4 block, so a warp whose lanes all
// evaluate the same hit idles most of them.  Here each half-warp has its own
// 4 x 4 block and its own list of hits, and the two lists are walked side by
// side: a step evaluates two different Gaussians.  Hits wait in a ring per
// half-warp until sixteen are there, so that the halves' shares of a batch
// even out.
// Against the whole-warp backward: 79 -> 72 us (250k Gaussians, 640x512), 235 ->
// 220 us (1M, 1280x1024), 92 -> 81 us (300k, 957x717), 3,959 -> 3,772 us (12
// views of 2M).  The forward has no sums to add up and loses what its two
// lists cost (185 -> 193 us, 1M; 3,347 -> 3,566 us): it keeps whole warps.
constexpr int kRing = 48;    // three groups of 16: up to 16 waiting, a batch of 32 staged on top
struct HalfRing {
    float4 r0[kRing], r1[kRing], r2[kRing];
    __device__ __forceinline__ void put(int k, const float4 a, const float4 b, const float4 c)
    {
        r0[k] = a; r1[k] = b; r2[k] = c;
    }
};

// The waiting hits of the two half-warps (the same values in every lane):
// entries tail .. tail + n of the ring, tail a multiple of 16.
struct HalfQueue {
    int head[2], tail[2], n[2];
    __device__ __forceinline__ HalfQueue() { head[0] = head[1] = tail[0] = tail[1] = n[0] = n[1] = 0; }
    // stage a batch's hits of half h (lane mask m), REV: in reverse lane order
    template <bool REV>
    __device__ __forceinline__ void stage(HalfRing& R, int h, unsigned m, unsigned lt, bool hit, const float4 a,
                                          const float4 b, const float4 c)
    {
        const int cnt = __popc(m);
        if (hit) {
            const int r = __popc(m & lt);
            int k = head[h] + (REV ? cnt - 1 - r : r);
            if (k >= kRing) k -= kRing;
            R.put(k, a, b, c);
        }
        head[h] += cnt;
        if (head[h] >= kRing) head[h] -= kRing;
        n[h] += cnt;
    }
    // the group of half h (up to 16 hits) has been walked
    __device__ __forceinline__ void pop(int h)
    {
        tail[h] = tail[h] == kRing - 16 ? 0 : tail[h] + 16;
        if (n[h] < 16) {   // all of them: the next hits start a group
            n[h] = 0;
            head[h] = tail[h];
        } else {
            n[h] -= 16;
            if (n[h] == 0) head[h] = tail[h];
        }
    }
};

// The per-pixel backward over half-warp blocks (one pixel per lane, not
// deterministic; the sums of a hit's two halves would need a row each).  A
// group of up to sixteen hits per half-warp is walked, then the warp turns
// over: lane (half, hit) adds up its hit over the half's sixteen pixels, so no
// sum crosses lanes.  Bound by
// instruction issue (67% of the cycles issue on the 1M view).
struct BwdHalf {
    static constexpr int S = 17;      // row stride (float2): the rows of a half on different banks
    HalfRing ring[2];                 // hits; r1.w owner, r2.w list position (bits)
    float4 pix[32];                   // per lane's pixel: dL/dC, dL/dD
    float2 sv[32 * S];                // per (half, hit): (blend weight, dL/d(exponent)) of its pixels
};

template <bool EXTRA>
__device__ __forceinline__ void half_turn_over(const RasterGrad& G, const BwdHalf& W, int at, bool on, float bx,
                                               float by, int lane)
{
    const int half = lane >> 4;
    const HalfRing& R = W.ring[half];
    const float4 a = R.r0[at + (lane & 15)];
    const float2* row = W.sv + lane * BwdHalf::S;
    const float4* pc = W.pix + half * 16;
    // chains of four to eight terms, then pairs of sums (see bwd_turn_over)
    float c0[2] = {0.f, 0.f}, c1[2] = {0.f, 0.f}, c2[2] = {0.f, 0.f}, cD[2] = {0.f, 0.f}, mxx[2] = {0.f, 0.f};
    float m0[4] = {0.f, 0.f, 0.f, 0.f}, mx[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int x = 0; x < 4; x++) {
        const float dx = a.x - (bx + (float)x), dx2 = dx * dx;
#pragma unroll
        for (int y = 0; y < 4; y++) {
            const int e = y & 1;
            const float2 v = row[y * 4 + x];
            const float4 g = pc[y * 4 + x];
            c0[e] = fmaf(v.x, g.x, c0[e]); c1[e] = fmaf(v.x, g.y, c1[e]); c2[e] = fmaf(v.x, g.z, c2[e]);
            if (EXTRA) cD[e] = fmaf(v.x, g.w, cD[e]);
            m0[y] += v.y;
            mx[y] = fmaf(v.y, dx, mx[y]);
            mxx[e] = fmaf(v.y, dx2, mxx[e]);
        }
    }
    float gy = 0.f, gxy = 0.f, gyy = 0.f;
#pragma unroll
    for (int y = 0; y < 4; y++) {
        const float dy = a.y - (by + (float)y), t = dy * m0[y];
        gy += t;
        gxy = fmaf(dy, mx[y], gxy);
        gyy = fmaf(dy, t, gyy);
    }
    if (on) {
        const uint32_t id = __float_as_uint(R.r1[at + (lane & 15)].w);
        float* dst = G.g2d + (size_t)id * kGradStride;
        atomicAdd(reinterpret_cast<float4*>(dst), make_float4(c0[0] + c0[1], c1[0] + c1[1], c2[0] + c2[1],
                                                                (m0[0] + m0[1]) + (m0[2] + m0[3])));
        atomicAdd(reinterpret_cast<float4*>(dst + 4), make_float4((mx[0] + mx[1]) + (mx[2] + mx[3]), gy, mxx[0] + mxx[1], gxy));
        if (EXTRA) atomicAdd(reinterpret_cast<float2*>(dst + 8), make_float2(gyy, cD[0] + cD[1]));
        else atomicAdd(dst + 8, gyy);
    }
}

template <bool EXTRA>
__device__ __forceinline__ void bwd_half_item(int u, const RasterArgs& A, const RasterGrad& G, BwdHalf& W, int lane)
{
    Unit U;
    unit_of<1>(u, A, U);
    const LanePix<1, true> L(U, A.TS, lane);
    const unsigned lt = (1u << lane) - 1u;
    const int half = lane >> 4, l16 = lane & 15;
    HalfRing& R = W.ring[half];
    float T = 1.0f, R0 = 0.f, R1 = 0.f, R2 = 0.f, RD = 0.f, RO = 0.f;   // as bwd_item
    float g0 = 0.f, g1 = 0.f, g2 = 0.f, gD = 0.f, gO = 0.f;
    uint32_t last = 0;
    if (L.inside[0]) {
        const size_t p = L.pix(U, 0);
        last = G.ncon[p];
        g0 = G.dL_drgb[3 * p]; g1 = G.dL_drgb[3 * p + 1]; g2 = G.dL_drgb[3 * p + 2];
        if (EXTRA) {
            gD = G.dL_ddepth ? G.dL_ddepth[p] : 0.0f;
            gO = G.dL_dopac ? G.dL_dopac[p] : 0.0f;
        }
        if (U.nseg == 1) {
            T = G.Tfin[p];
        } else if (last > U.rs - U.trs) {   // (no state behind the stop segment)
            const float* S = A.segstate;
            const int i = L.p[0];
            T = S[seg_at(U.w, 0, i, A.TS)];
            R0 = S[seg_at(U.w, 1, i, A.TS)];
            R1 = S[seg_at(U.w, 2, i, A.TS)];
            R2 = S[seg_at(U.w, 3, i, A.TS)];
            if (EXTRA) {
                RD = S[seg_at(U.w, 4, i, A.TS)];
                RO = S[seg_at(U.w, 5, i, A.TS)];
            }
        }
    }
    W.pix[lane] = make_float4(g0, g1, g2, gD);
    // positions at or beyond a half's last contributor reach none of its pixels
    uint32_t hmax = last;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) hmax = max(hmax, __shfl_xor_sync(kFull, hmax, off));
    const uint32_t last0 = __shfl_sync(kFull, hmax, 0), last1 = __shfl_sync(kFull, hmax, 16);
    const uint32_t end = min(U.re, U.trs + max(last0, last1));
    if (end <= U.rs) return;
    const float bx = (float)(U.lx0 + 4 * half), by = (float)U.ly0;
    HalfQueue Q;
    // batches of 32 from the back, the last one clipped at rs: i = hi - 32 + lane
    uint32_t hi = end;
    float4 n0, n1, n2, n3;
    uint32_t ng = 0;
    if (hi - U.rs + lane >= 32u) {
        const uint32_t i = hi - 32u + lane;
        n0 = A.s0[i]; n1 = A.s1[i]; n2 = A.s2[i]; n3 = A.s3[i];
        ng = A.sgid[i];
    }
    while (true) {
        const uint32_t left = hi - U.rs;   // records of this and the batches before it
        const bool valid = left + lane >= 32u, more = left > 32u;
        const uint32_t pos = hi - 32u + lane - U.trs;
        const float4 c0 = n0, c3 = n3;
        float4 c1 = n1, c2 = n2;
        c1.w = __uint_as_float(ng);
        c2.w = __uint_as_float(pos);
        if (more && left - 32u + lane >= 32u) {
            const uint32_t i = hi - 64u + lane;
            n0 = A.s0[i]; n1 = A.s1[i]; n2 = A.s2[i]; n3 = A.s3[i];
            ng = A.sgid[i];
        }
        const bool rows = valid && !(c3.w < L.by0 || c3.z > L.by1);
        const bool h0 = rows && pos < last0 && !(c3.y < L.bx0 || c3.x > L.bx0 + 3.0f);
        const bool h1 = rows && pos < last1 && !(c3.y < L.bx0 + 4.0f || c3.x > L.bx0 + 7.0f);
        const unsigned m0 = __ballot_sync(kFull, h0), m1 = __ballot_sync(kFull, h1);
        Q.stage<true>(W.ring[0], 0, m0, lt, h0, c0, c1, c2);
        Q.stage<true>(W.ring[1], 1, m1, lt, h1, c0, c1, c2);
        const int keep = more ? 16 : 0;   // the last batch leaves none waiting
        while (max(Q.n[0], Q.n[1]) > keep) {
            const int k0 = min(Q.n[0], 16), k1 = min(Q.n[1], 16), steps = max(k0, k1);
            const int mine = half ? k1 : k0, at = half ? Q.tail[1] : Q.tail[0];
            if (l16 >= mine && l16 < ((steps + 1) & ~1)) {
                R.r0[at + l16] = R.r2[at + l16] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                R.r1[at + l16] = make_float4(0.0f, -3.0e38f, 0.0f, 0.0f);
            }
            __syncwarp();
            float2* sv = W.sv + half * 16 * BwdHalf::S + l16;
            for (int k = 0; k < steps; k += 2, sv += 2 * BwdHalf::S) {
                float4 a[2], b[2], c[2];
                float al[2];
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    a[e] = R.r0[at + k + e];
                    b[e] = R.r1[at + k + e];
                    c[e] = R.r2[at + k + e];
                }
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    float dx, dy, alpha;
                    bool capped;
                    const bool live = pair_eval_nb(a[e], b[e], L.px, L.py[0], dx, dy, alpha, capped) &&
                                      __float_as_uint(c[e].w) < last;
                    al[e] = live ? alpha : 0.0f;
                }
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    // as bwd_item
                    T = __fdividef(T, 1.0f - al[e]);
                    const float wgt = al[e] * T;
                    const float d0 = c[e].x - R0, d1 = c[e].y - R1, d2 = c[e].z - R2;
                    float dot = g0 * d0 + g1 * d1 + g2 * d2;
                    R0 = fmaf(al[e], d0, R0);
                    R1 = fmaf(al[e], d1, R1);
                    R2 = fmaf(al[e], d2, R2);
                    if (EXTRA) {
                        const float dD = b[e].z - RD, dO = 1.0f - RO;
                        dot += gD * dD + gO * dO;
                        RD = fmaf(al[e], dD, RD);
                        RO = fmaf(al[e], dO, RO);
                    }
                    sv[e * BwdHalf::S] = make_float2(wgt, al[e] < kAlphaMax ? wgt * dot : 0.0f);
                }
            }
            __syncwarp();
            half_turn_over<EXTRA>(G, W, at, l16 < mine, bx, by, lane);
            __syncwarp();
            Q.pop(0);
            Q.pop(1);
        }
        if (!more) break;
        hi -= 32u;
    }
}

constexpr int kWpbHalf = 4;       // 37.0 KB of shared memory a CTA
static_assert(sizeof(BwdHalf) * kWpbHalf == 37888, "five CTAs in an SM's 227 KB");
// Instances per visible (view, Gaussian) pair up to which blocks are half-warps
// (street maps have 1.3 to 1.5).  A half-warp block adds a row of its own, so a
// large Gaussian's sums take twice as many additions: against 64 bits the
// gradients are as far off with either block up to 28 instances a Gaussian, 2 to
// 4% further with half-warps at 240, and on 20k Gaussians of 4 to 84 pixels (64
// instances) the quaternions' 4.6e-6 instead of 3.9e-6, the scales' 4.5e-6 instead
// of 4.1e-6.  Whole-warp blocks' times there, 1280x960: 440 -> 485 us (63 instances), 442
// -> 482 (219), 574 -> 495 (1,150).  The counts are on the device, so the choice is made
// there; the whole-warp item is a call, which leaves the half-warp loop's registers
// as they are (inlined, the loop took 3% longer).
constexpr uint64_t kHalfInstances = 32;
constexpr int kMinBlocksHalf = 5; // 96 registers (at most 8 bytes spilled), 20 warps per SM

template <bool EXTRA>
__device__ __noinline__ void bwd_item_call(int u, const RasterArgs& A, const RasterGrad& G, BwdWarp<1, 1>& W, int lane)
{
    bwd_item<EXTRA, 1, 1, false>(u, A, G, W, lane);
}

template <bool EXTRA>
__global__ void __launch_bounds__(32 * kWpbHalf, kMinBlocksHalf)
k_raster_bwd_half(const __grid_constant__ RasterArgs A, const __grid_constant__ RasterGrad G)
{
    __shared__ union {
        BwdHalf half;
        BwdWarp<1, 1> whole;
    } sw[kWpbHalf];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nunits = (int)A.ctl[6] * A.nblk;
    int u = A.work ? next_unit(A.work, lane) : blockIdx.x * kWpbHalf + w;
    if (A.ctl[0] <= kHalfInstances * A.ctl[9]) {
        while (u < nunits) {
            bwd_half_item<EXTRA>(u, A, G, sw[w].half, lane);
            __syncwarp();
            if (!A.work) break;
            u = next_unit(A.work, lane);
        }
    } else {
        while (u < nunits) {
            bwd_item_call<EXTRA>(u, A, G, sw[w].whole, lane);
            if (!A.work) break;
            u = next_unit(A.work, lane);
        }
    }
}

template <bool EXTRA, int NB, int D, bool DET>
__global__ void __launch_bounds__(32 * wpb_bwd<NB>(), minb_bwd<NB, D>()) k_raster_bwd(RasterArgs A, RasterGrad G)
{
    constexpr int WPB = wpb_bwd<NB>();
    __shared__ BwdWarp<NB, D> sw[WPB];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nunits = (int)A.ctl[6] * A.nblk;
    int u = A.work ? next_unit(A.work, lane) : blockIdx.x * WPB + w;
    while (u < nunits) {
        bwd_item<EXTRA, NB, D, DET>(u, A, G, sw[w], lane);
        if (!A.work) break;
        u = next_unit(A.work, lane);
    }
}

// ---------------------------------------------------------------------------
// Per-Gaussian backward (Sec. III-D 1: threads assigned to the Gaussians
// rather than to the pixels).  A warp takes a (work item, 8x4 pixel block)
// unit like the kernel above and walks, back to front, the Gaussians whose
// alpha box touches the block (the hits); lane l owns hits l, l + 32, l + 64,
// ... and sums each one's gradient over the block's 32 pixels in its own
// registers.  The pixels' backward state -- the transmittance and the colour
// (depth, opacity) blended behind -- travels round the warp: at step s, lane
// l serves pixel p = (s - l) mod 32 for its hit s - p and then hands the
// pixel's state to lane l + 1, which holds the next hit.  Every pixel thus
// meets the hits in back-to-front order, one step apart, and H hits take
// H + 31 steps.  At step s lane s mod 32 is done with hit s - 32: it leaves
// its sums in a shared-memory slot and takes up hit s; every 32 steps the
// warp adds the 32 finished hits to their Gaussians' accumulators (or, in
// deterministic mode, stores them per instance and pixel block).  So a hit
// costs no warp reduction, and a Gaussian's sums stay in one lane.
// Hits are compacted from the sorted records in batches of 32, as above,
// into a per-warp ring of kPgQ entries, at least 32 ahead of the steps.  A
// list short enough to fit in the first fill (under 64 hits) is walked per
// pixel instead: there the 31 steps of filling and draining the ring would
// cost more than the per-hit reductions they save.
// ---------------------------------------------------------------------------
constexpr int kPgQ = 64;   // hit ring per warp: live hits are < 32 ahead + one batch of 32

struct PgWarp {
    float4 q0[kPgQ], q1[kPgQ], q2[kPgQ];   // hit records (sorted-order r0, r1, r2)
    uint32_t qpos[kPgQ], qg[kPgQ];          // list position (relative to the tile) and owner
    float4 pix[32];                         // per pixel: dL/dC and the last contributor (bits)
    float2 pxy[32];                         // per pixel: tile-relative coordinates
    float2 pde[32];                         // per pixel: dL/dD, dL/dO (EXTRA)
    float4 st0[32], st1[32];                // finished hits' sums, one slot per lane:
    float2 st2[32];                         //   0-3, 4-7, 8-9
    uint32_t stg[32];                       // their owners (0xffffffff: empty)
};
static_assert(sizeof(PgWarp) * 8 <= 48 * 1024, "static shared memory of the per-Gaussian backward");

template <bool EXTRA, bool DET>
__device__ __forceinline__ void pg_flush(const RasterArgs& A, const RasterGrad& G, int wb, uint32_t g,
                                         const float (&acc)[kNG])
{
    constexpr int NQ = EXTRA || DET ? kNG : kNG - 1;   // deterministic rows are stored whole
    if (DET) atomicOr(G.pmask + g, 1u << wb);
#pragma unroll
    for (int q = 0; q < NQ; q++) {
        if (DET) G.part[((size_t)g * A.nblk + wb) * kGradStride + q] = acc[q];
        else atomicAdd(G.g2d + (size_t)g * kGradStride + q, acc[q]);
    }
}

template <bool EXTRA, bool DET>
__device__ __forceinline__ void bwd_item_pg(int u, const RasterArgs& A, const RasterGrad& G, PgWarp& W, int lane)
{
    Unit U;
    unit_of<1>(u, A, U);
    const unsigned lt = (1u << lane) - 1u;
    // lane l starts with the state of pixel (32 - l) mod 32 of the block
    const int p0 = (32 - lane) & 31;
    const int lx = U.lx0 + (p0 & 7), ly = U.ly0 + (p0 >> 3);
    const int x = U.x0 + (p0 & 7), y = U.y0 + (p0 >> 3);
    float T = 1.0f, R0 = 0.0f, R1 = 0.0f, R2 = 0.0f, RD = 0.0f, RO = 0.0f;
    uint32_t last = 0;
    float4 pc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float2 pe = make_float2(0.0f, 0.0f);
    if (x < U.W && y < U.H) {
        const size_t p = (size_t)U.pix_base + (size_t)y * U.W + x;
        last = G.ncon[p];
        if (U.nseg == 1) {
            T = G.Tfin[p];
        } else if (last > U.rs - U.trs) {
            const float* S = A.segstate;
            const int q = ly * A.TS + lx;
            T = S[seg_at(U.w, 0, q, A.TS)];
            R0 = S[seg_at(U.w, 1, q, A.TS)];
            R1 = S[seg_at(U.w, 2, q, A.TS)];
            R2 = S[seg_at(U.w, 3, q, A.TS)];
            if (EXTRA) {
                RD = S[seg_at(U.w, 4, q, A.TS)];
                RO = S[seg_at(U.w, 5, q, A.TS)];
            }
        }
        pc = make_float4(G.dL_drgb[3 * p], G.dL_drgb[3 * p + 1], G.dL_drgb[3 * p + 2], __uint_as_float(last));
        if (EXTRA) pe = make_float2(G.dL_ddepth ? G.dL_ddepth[p] : 0.0f, G.dL_dopac ? G.dL_dopac[p] : 0.0f);
    }
    W.pix[p0] = pc;
    W.pxy[p0] = make_float2((float)lx, (float)ly);
    if (EXTRA) W.pde[p0] = pe;
    W.stg[lane] = 0xffffffffu;
    uint32_t wmax = last;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wmax = max(wmax, __shfl_xor_sync(kFull, wmax, off));
    const uint32_t end = min(U.re, U.trs + wmax);
    __syncwarp();
    if (end <= U.rs) return;

    // batches from the back: [bstart, bstart + 32) clipped at rs, next one prefetched
    int64_t bstart = (int64_t)end - 32;
    float4 n0, n1, n2, n3;
    uint32_t ng = 0;
    {
        const int64_t i = bstart + lane;
        if (i >= (int64_t)U.rs) {
            n0 = A.s0[i]; n1 = A.s1[i]; n2 = A.s2[i]; n3 = A.s3[i];
            ng = DET ? G.sinst[i] : A.sgid[i];
        }
    }
    bool exhausted = false;
    int qhead = 0;   // hits compacted so far (hit 0 is the deepest)

    // the lane's current hit
    bool cur = false;
    float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0, c2 = c0;
    uint32_t cpos = 0, cg = 0;
    float acc[kNG];
#pragma unroll
    for (int q = 0; q < kNG; q++) acc[q] = 0.0f;

    for (int S = 0;; S += 32) {
        if (S > 0) {
            // the hits finished in the last 32 steps, one per lane
            const uint32_t g = W.stg[lane];
            if (g != 0xffffffffu) {
                float a[kNG];
                const float4 v0 = W.st0[lane], v1 = W.st1[lane];
                const float2 v2 = W.st2[lane];
                a[0] = v0.x; a[1] = v0.y; a[2] = v0.z; a[3] = v0.w;
                a[4] = v1.x; a[5] = v1.y; a[6] = v1.z; a[7] = v1.w;
                a[8] = v2.x; a[9] = v2.y;
                pg_flush<EXTRA, DET>(A, G, U.wb, g, a);
                W.stg[lane] = 0xffffffffu;
            }
        }
        // refill: compacted hits must cover the steps S .. S + 31
        while (!exhausted && qhead < S + 32) {
            const float4 b0 = n0, b1 = n1, b2 = n2, b3 = n3;
            const uint32_t bg = ng;
            const int64_t i = bstart + lane;
            const int64_t ni = i - 32;
            if (ni >= (int64_t)U.rs) {
                n0 = A.s0[ni]; n1 = A.s1[ni]; n2 = A.s2[ni]; n3 = A.s3[ni];
                ng = DET ? G.sinst[ni] : A.sgid[ni];
            }
            const bool hit = i >= (int64_t)U.rs && box_hit(b3, (float)U.x0, (float)(U.x0 + 7), (float)U.y0,
                                                            (float)(U.y0 + 3));
            const unsigned mask = __ballot_sync(kFull, hit);
            const int nh = __popc(mask);
            if (hit) {
                // deepest first: the batch's hits in reverse list order
                const int k = (qhead + nh - 1 - __popc(mask & lt)) & (kPgQ - 1);
                W.q0[k] = b0; W.q1[k] = b1; W.q2[k] = b2;
                W.qpos[k] = (uint32_t)(i - U.trs);
                W.qg[k] = bg;
            }
            qhead += nh;
            bstart -= 32;
            if (bstart + 32 <= (int64_t)U.rs) exhausted = true;
        }
        __syncwarp();
        if (S == 0 && exhausted) {
            // a short list (all of it fitted in the first fill): the ring
            // would spend 31 steps filling and draining for fewer than 64
            // hits, so walk it per pixel instead, each lane with the pixel
            // it holds, and fold each hit's sums across the warp
            const float px = (float)lx, py = (float)ly;
            for (int k = 0; k < qhead; k++) {
                const float4 a = W.q0[k], b = W.q1[k], c = W.q2[k];
                const uint32_t pos = W.qpos[k];
                float v[16];
#pragma unroll
                for (int q = 0; q < 16; q++) v[q] = 0.0f;
                float dx, dy, alpha;
                bool capped;
                const bool on = pos < last && pair_eval(a, b, px, py, dx, dy, alpha, capped);
                if (on) {
                    const float om = 1.0f - alpha;
                    T = __fdividef(T, om);
                    const float wgt = alpha * T;
                    float ga = pc.x * (c.x - R0) + pc.y * (c.y - R1) + pc.z * (c.z - R2);
                    if (EXTRA) ga += pe.x * (b.z - RD) + pe.y * (1.0f - RO);
                    ga *= T;
                    R0 = alpha * c.x + om * R0;
                    R1 = alpha * c.y + om * R1;
                    R2 = alpha * c.z + om * R2;
                    if (EXTRA) {
                        RD = alpha * b.z + om * RD;
                        RO = alpha + om * RO;
                    }
                    const float gp = capped ? 0.0f : ga * alpha;
                    v[0] = wgt * pc.x; v[1] = wgt * pc.y; v[2] = wgt * pc.z;
                    v[3] = gp;
                    v[4] = gp * dx; v[5] = gp * dy;
                    v[6] = gp * dx * dx; v[7] = gp * dx * dy; v[8] = gp * dy * dy;
                    if (EXTRA) v[9] = wgt * pe.x;
                }
                if (__any_sync(kFull, on)) {
                    const float r = warp_transpose_reduce16(v);
                    const int q = lane >> 1;
                    if ((lane & 1) == 0 && q < (EXTRA || DET ? kNG : kNG - 1)) {
                        const uint32_t g = W.qg[k];
                        if (DET && lane == 0) atomicOr(G.pmask + g, 1u << U.wb);
                        if (DET) G.part[((size_t)g * A.nblk + U.wb) * kGradStride + q] = r;
                        else atomicAdd(G.g2d + (size_t)g * kGradStride + q, r);
                    }
                }
            }
            __syncwarp();
            return;
        }
        if (exhausted && S > qhead + 30) break;
        // 32 steps of the wavefront
#pragma unroll 2
        for (int j = 0; j < 32; j++) {
            const int s = S + j;
            if (lane == j) {
                // done with hit s - 32: park its sums; take up hit s
                if (cur) {
                    W.st0[lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
                    W.st1[lane] = make_float4(acc[4], acc[5], acc[6], acc[7]);
                    W.st2[lane] = make_float2(acc[8], acc[9]);
                    W.stg[lane] = cg;
                }
                cur = s < qhead;
                if (cur) {
                    const int k = s & (kPgQ - 1);
                    c0 = W.q0[k]; c1 = W.q1[k]; c2 = W.q2[k];
                    cpos = W.qpos[k];
                    cg = W.qg[k];
                }
#pragma unroll
                for (int q = 0; q < kNG; q++) acc[q] = 0.0f;
            }
            const int p = (s - lane) & 31;
            const float4 c = W.pix[p];
            const float2 xy = W.pxy[p];
            float dx, dy, alpha;
            bool capped;
            if (cur && cpos < __float_as_uint(c.w) && pair_eval(c0, c1, xy.x, xy.y, dx, dy, alpha, capped)) {
                const float om = 1.0f - alpha;
                T = __fdividef(T, om);
                const float wgt = alpha * T;
                float ga = c.x * (c2.x - R0) + c.y * (c2.y - R1) + c.z * (c2.z - R2);
                float2 e = make_float2(0.0f, 0.0f);
                if (EXTRA) {
                    e = W.pde[p];
                    ga += e.x * (c1.z - RD) + e.y * (1.0f - RO);
                }
                ga *= T;
                R0 = alpha * c2.x + om * R0;
                R1 = alpha * c2.y + om * R1;
                R2 = alpha * c2.z + om * R2;
                if (EXTRA) {
                    RD = alpha * c1.z + om * RD;
                    RO = alpha + om * RO;
                }
                const float gp = capped ? 0.0f : ga * alpha;
                acc[0] += wgt * c.x; acc[1] += wgt * c.y; acc[2] += wgt * c.z;
                acc[3] += gp;
                acc[4] += gp * dx; acc[5] += gp * dy;
                acc[6] += gp * dx * dx; acc[7] += gp * dx * dy; acc[8] += gp * dy * dy;
                if (EXTRA) acc[9] += wgt * e.x;
            }
            // the pixel's state moves on to the lane of the next hit
            const int src = (lane + 31) & 31;
            T = __shfl_sync(kFull, T, src);
            R0 = __shfl_sync(kFull, R0, src);
            R1 = __shfl_sync(kFull, R1, src);
            R2 = __shfl_sync(kFull, R2, src);
            if (EXTRA) {
                RD = __shfl_sync(kFull, RD, src);
                RO = __shfl_sync(kFull, RO, src);
            }
        }
    }
    // the hits still held by the lanes
    if (cur) pg_flush<EXTRA, DET>(A, G, U.wb, cg, acc);
    __syncwarp();
}

template <bool EXTRA, bool DET>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, kMinBlocksPg)
k_raster_bwd_pg(RasterArgs A, RasterGrad G)
{
    __shared__ PgWarp sw[kWarpsPerBlock];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nunits = (int)A.ctl[6] * A.nblk;
    int u = A.work ? next_unit(A.work, lane) : blockIdx.x * kWarpsPerBlock + w;
    while (u < nunits) {
        bwd_item_pg<EXTRA, DET>(u, A, G, sw[w], lane);
        if (!A.work) break;
        u = next_unit(A.work, lane);
    }
}

// Deterministic gradient sums: each (view, Gaussian) pair's instances
// (emission indices dup_off .. dup_off + touched), of each the pixel blocks
// its mask names.  Four lanes share a row (three of them hold its float4s)
// and a pair's instances are dealt to row streams: two of them for a pair of
// up to kHeavyPair instances (four pairs per warp), eight -- the warp -- for
// the others, one pair after the other.  The streams' sums are then added in
// a fixed order.  Only written rows are read, so neither the rows nor the
// blocks without a hit need clearing.  Bound by the latency of the pairs with
// hundreds of instances: 32 masks come in one load, the four pairs of a warp
// lie a quarter of all pairs apart (near Gaussians are neighbours in the
// map).  A thread per pair over every row, 173 us and a memset of the rows
// (115 MB, 18 us) -> 66 us (250k Gaussians, street, 640x512).
constexpr uint32_t kHeavyPair = 8;

// acc += the rows of one instance that its mask m names (this lane's float4).
__device__ __forceinline__ void part_rows(const float* __restrict__ part, uint64_t e, uint32_t m, int nblk, int f,
                                          float4& acc)
{
    const float4* row = reinterpret_cast<const float4*>(part + (size_t)e * nblk * kGradStride) + f;
    for (int b0 = 0; b0 < nblk; b0 += 8) {
        const uint32_t mb = f < 3 ? m >> b0 : 0u;
        float4 v[8];
#pragma unroll
        for (int b = 0; b < 8; b++)
            if ((mb >> b) & 1u) v[b] = row[(b0 + b) * (kGradStride / 4)];
#pragma unroll
        for (int b = 0; b < 8; b++)
            if ((mb >> b) & 1u) { acc.x += v[b].x; acc.y += v[b].y; acc.z += v[b].z; acc.w += v[b].w; }
    }
}

__device__ __forceinline__ void fold_streams(float4& a, int off)
{
    a.x += __shfl_xor_sync(kFull, a.x, off);
    a.y += __shfl_xor_sync(kFull, a.y, off);
    a.z += __shfl_xor_sync(kFull, a.z, off);
    a.w += __shfl_xor_sync(kFull, a.w, off);
}

__global__ void __launch_bounds__(256)
k_part_reduce(const float* __restrict__ part, const uint32_t* __restrict__ pmask,
              const uint32_t* __restrict__ touched, const uint32_t* __restrict__ dup_off, int nblk, int64_t pairs,
              const uint64_t* __restrict__ ctl, uint64_t cap, float* __restrict__ g2d)
{
    const bool overflow = ctl[1] != 0;   // the step's instances did not fit: nothing was written
    const int lane = threadIdx.x & 31, f = lane & 3;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5), quarter = (pairs + 3) / 4;
    for (int64_t t0 = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t0 < quarter; t0 += warps) {
        const int64_t t = t0 + (lane >> 3) * quarter;
        uint32_t cnt = t < pairs ? touched[t] : 0u;
        const uint64_t first = cnt ? dup_off[t] : 0u;
        if (overflow || first + cnt > cap) cnt = 0;
        const bool heavy = cnt > kHeavyPair;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t light = heavy ? 0u : cnt;
        // lane k of a pair's eight holds the mask of its instance k
        const uint32_t lm = (uint32_t)(lane & 7) < light ? pmask[first + (lane & 7)] : 0u;
        const int s = (lane >> 2) & 1;
#pragma unroll
        for (int i = 0; i < (int)kHeavyPair; i += 2) {
            const uint32_t m = __shfl_sync(kFull, lm, (lane & ~7) + i + s);
            if (m) part_rows(part, first + i + s, m, nblk, f, acc);
        }
        fold_streams(acc, 4);
        for (unsigned left = __ballot_sync(kFull, heavy && (lane & 7) == 0); left; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const uint64_t hf = __shfl_sync(kFull, first, src);
            const uint32_t hc = __shfl_sync(kFull, cnt, src);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            uint32_t hm = (uint32_t)lane < hc ? pmask[hf + lane] : 0u;
            for (uint32_t e0 = 0; e0 < hc; e0 += 32) {
                const uint32_t cur = hm;
                hm = e0 + 32 + lane < hc ? pmask[hf + e0 + 32 + lane] : 0u;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int k = i * 8 + (lane >> 2);
                    const uint32_t m = __shfl_sync(kFull, cur, k);
                    if (m) part_rows(part, hf + e0 + k, m, nblk, f, a);
                }
            }
            fold_streams(a, 4);
            fold_streams(a, 8);
            fold_streams(a, 16);
            if ((lane >> 3) == (src >> 3)) acc = a;
        }
        if (t < pairs && (lane & 7) < 3) reinterpret_cast<float4*>(g2d + (size_t)t * kGradStride)[f] = acc;
    }
}

// Records in sorted-instance order (and, where instance ids were sorted, the
// owning Gaussian of each), the
// mean made relative to the origin of the instance's tile: (u_hi - x0) is
// exact near the tile (Sterbenz), and adding u_lo leaves an offset accurate
// to float precision of a number of pixels, not of the image coordinate.
// The same pass marks each tile's list [first, last + 1) in `ranges` where
// the sorted tile id changes (tiles without instances keep the zeros the
// caller wrote).
__global__ void k_permute(const uint64_t* __restrict__ n_dev, uint32_t* __restrict__ ranges,
                          const uint32_t* __restrict__ sinst,
                          const uint32_t* __restrict__ stile, const ViewDesc* __restrict__ views, int V, int TS,
                          const uint32_t* __restrict__ owner, const float4* __restrict__ rec,
                          float4* __restrict__ s0, float4* __restrict__ s1,
                          float4* __restrict__ s2, float4* __restrict__ s3, uint32_t* __restrict__ sg)
{
    const uint64_t I = *n_dev;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < I; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t g = sinst ? owner[sinst[i]] : owner[i];
        const int tile = (int)stile[i];
        if (i == 0 || stile[i - 1] != (uint32_t)tile) ranges[2 * tile] = (uint32_t)i;
        if (i == I - 1 || stile[i + 1] != (uint32_t)tile) ranges[2 * tile + 1] = (uint32_t)(i + 1);
        const ViewDesc& d = views[view_of_tile(views, V, tile)];
        const int lt = tile - d.tile_base;
        const float x0 = (float)((lt % d.TX) * TS), y0 = (float)((lt / d.TX) * TS);
        float4 a, b, c, box;
        ld_sector(rec + 4 * (size_t)g, a, b);
        ld_sector(rec + 4 * (size_t)g + 2, c, box);
        a.x = __fadd_rn(__fsub_rn(a.x, x0), c.w);
        a.y = __fadd_rn(__fsub_rn(a.y, y0), b.w);
        s0[i] = a; s1[i] = b; s2[i] = c; s3[i] = box;
        if (sinst) sg[i] = g;
    }
}

// Resident CTAs of a kernel on the current device (SMs x CTAs per SM),
// looked up once per (kernel, device).
int resident_ctas(const void* kernel, int threads)
{
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find({kernel, dev});
    if (it != cache.end()) return it->second;
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
    const int r = std::max(1, sm_count() * std::max(1, per));
    cache[{kernel, dev}] = r;
    return r;
}

// Grid of `wpb`-warp CTAs for up to units_bound warp units: one unit per
// warp, or (persistent) the resident CTAs, whose warps take units from a
// counter.
template <typename K>
int grid_for(K kernel, int64_t units_bound, bool persistent, int wpb = kWarpsPerBlock)
{
    const int64_t need = std::max<int64_t>(1, (units_bound + wpb - 1) / wpb);
    if (!persistent) return (int)std::min<int64_t>(need, 0x7fffffff);
    const int res = resident_ctas(reinterpret_cast<const void*>(kernel), 32 * wpb);
    return (int)std::max<int64_t>(1, std::min<int64_t>(need, res));
}

int blocks_per_tile(const View& v) { return v.Ts * v.Ts / (32 * v.pd); }

// Split-tile items are bounded by 1.5 x capacity / seg: a tile of L >= 2 seg
// records has at most L / seg + 1 <= 1.5 L / seg segments.
int64_t split_items_bound(const View& v)
{
    return v.seg > 0 ? (int64_t)(v.itile.bytes / 4) * 3 / (2 * v.seg) + 1 : 0;
}

RasterArgs make_args(View& v, int* work)
{
    RasterArgs A;
    A.TS = v.Ts;
    A.V = v.V;
    A.nblk = blocks_per_tile(v);
    A.seg = v.seg;
    A.items = v.items.as<uint2>();
    A.heads = v.heads.as<uint32_t>();
    A.ctl = v.count.as<uint64_t>();
    A.ranges = v.ranges.as<uint32_t>();
    A.s0 = v.srec0.as<float4>();
    A.s1 = v.srec1.as<float4>();
    A.s2 = v.srec2.as<float4>();
    A.s3 = v.srec3.as<float4>();
    A.sgid = v.sorted_owner ? v.sorted_owner : v.sgid.as<uint32_t>();
    A.views = v.d_desc();
    A.segstate = v.segstate.as<float>();
    A.work = work;
    return A;
}

gl_status check_exec(const View& v)
{
    if (v.Ts != 8 && v.Ts != 16 && v.Ts != 32) { set_error("tile_size must be 8, 16 or 32"); return GL_ERR_INVALID; }
    if (v.nb != 1 && v.nb != 2 && v.nb != 4 && v.nb != 8) {
        set_error("batch depth must be 32, 64, 128 or 256");
        return GL_ERR_INVALID;
    }
    if (v.nb > 2 && v.pd != 1) {
        set_error("batch depths of 128 and 256 take one pixel per lane");
        return GL_ERR_INVALID;
    }
    if ((v.pd != 1 && v.pd != 2 && v.pd != 4) || 4 * v.pd > v.Ts) {
        set_error("pixels per lane must be 1, 2 or 4, with 4 x pixels per lane <= tile size");
        return GL_ERR_INVALID;
    }
    if (v.seg != 0 && (v.seg < 64 || v.seg > 65536 || (v.seg & (v.seg - 1)) != 0)) {
        set_error("segment length must be 0 or a power of two in 64..65536");
        return GL_ERR_INVALID;
    }
    return GL_OK;
}

// split_units and units bound the split and the whole tiles' pixel blocks.
template <int NB, int D, bool XD, int WPB>
void fwd_launch_wpb(const RasterArgs& A, const RasterOut& O, int64_t units, int64_t split_units, bool persistent,
                    cudaStream_t s)
{
    const int grid = grid_for(k_raster_fwd<NB, D, XD, WPB>, units + split_units * WPB, persistent, WPB);
    k_raster_fwd<NB, D, XD, WPB><<<grid, 32 * WPB, 0, s>>>(A, O);
}

template <int NB, int D, bool XD>
void fwd_launch(const RasterArgs& A, const RasterOut& O, int64_t units, int64_t split_units, bool persistent,
                cudaStream_t s)
{
    constexpr int wide = wpb_fwd<NB, D>(true), narrow = wpb_fwd<NB, D>(false);
    if (wide != narrow && units < (int64_t)kWideUnits * warps_fwd<NB, D>() * sm_count())
        fwd_launch_wpb<NB, D, XD, wide>(A, O, units, split_units, persistent, s);
    else
        fwd_launch_wpb<NB, D, XD, narrow>(A, O, units, split_units, persistent, s);
}

template <bool EXTRA, int NB, int D, bool DET>
void bwd_launch(const RasterArgs& A, const RasterGrad& G, int64_t units, bool persistent, cudaStream_t s)
{
    const int grid = grid_for(k_raster_bwd<EXTRA, NB, D, DET>, units, persistent, wpb_bwd<NB>());
    k_raster_bwd<EXTRA, NB, D, DET><<<grid, 32 * wpb_bwd<NB>(), 0, s>>>(A, G);
}

template <bool EXTRA, bool DET>
void bwd_pg_launch(const RasterArgs& A, const RasterGrad& G, int64_t units, bool persistent, cudaStream_t s)
{
    const int grid = grid_for(k_raster_bwd_pg<EXTRA, DET>, units, persistent);
    k_raster_bwd_pg<EXTRA, DET><<<grid, 32 * kWarpsPerBlock, 0, s>>>(A, G);
}

template <bool EXTRA>
void bwd_dispatch(int nb, int pd, bool det, bool pg, const RasterArgs& A, const RasterGrad& G, int64_t units,
                  int64_t blocks, bool persistent, cudaStream_t s)
{
    if (pg) {    // per-Gaussian: batch depth 32, one pixel per lane
        if (det) bwd_pg_launch<EXTRA, true>(A, G, units, persistent, s);
        else bwd_pg_launch<EXTRA, false>(A, G, units, persistent, s);
    } else if (det) {   // batch depth 32 only
        if (pd == 1) bwd_launch<EXTRA, 1, 1, true>(A, G, units, persistent, s);
        else if (pd == 2) bwd_launch<EXTRA, 1, 2, true>(A, G, units, persistent, s);
        else bwd_launch<EXTRA, 1, 4, true>(A, G, units, persistent, s);
    } else if (pd == 1 && nb == 1 && blocks >= (int64_t)kMinBlocksHalf * kWpbHalf * sm_count()) {
        // more pixel blocks than resident warps.  Below, a warp has one block
        // and its chain is the time, which the two lists lengthen: 17.8 -> 22.4
        // us on 5k Gaussians at 256x192 (1.5k blocks; the line lies at 3.0k).
        // Its batches are of 32 records (hits wait in a ring): deeper ones
        // were asked for and take the kernels that have them.
        // Whole- and half-warp blocks by footprint, 1280x960, standard
        // deviation in pixels: 1 (600k Gaussians) 245 and 188 us, 4 (100k) 224
        // and 193, 10 (30k) 297 and 268.  (Maps of much larger Gaussians take
        // whole-warp blocks within the kernel, see kHalfInstances.)
        const int grid = grid_for(k_raster_bwd_half<EXTRA>, units, persistent, kWpbHalf);
        k_raster_bwd_half<EXTRA><<<grid, 32 * kWpbHalf, 0, s>>>(A, G);
    } else if (nb == 4) {   // deeper batches: one pixel per lane
        bwd_launch<EXTRA, 4, 1, false>(A, G, units, persistent, s);
    } else if (nb == 8) {
        bwd_launch<EXTRA, 8, 1, false>(A, G, units, persistent, s);
    } else if (nb == 1) {
        if (pd == 1) bwd_launch<EXTRA, 1, 1, false>(A, G, units, persistent, s);
        else if (pd == 2) bwd_launch<EXTRA, 1, 2, false>(A, G, units, persistent, s);
        else bwd_launch<EXTRA, 1, 4, false>(A, G, units, persistent, s);
    } else {
        if (pd == 1) bwd_launch<EXTRA, 2, 1, false>(A, G, units, persistent, s);
        else if (pd == 2) bwd_launch<EXTRA, 2, 2, false>(A, G, units, persistent, s);
        else bwd_launch<EXTRA, 2, 4, false>(A, G, units, persistent, s);
    }
}

}  // namespace

gl_status permute_records(View& v, int64_t nmax, cudaStream_t s)
{
    if (nmax <= 0) return GL_OK;
    const size_t I = (size_t)nmax;
    GL_TRY(v.srec0.reserve(16 * I));
    GL_TRY(v.srec1.reserve(16 * I));
    GL_TRY(v.srec2.reserve(16 * I));
    GL_TRY(v.srec3.reserve(16 * I));
    if (v.sorted_inst) GL_TRY(v.sgid.reserve(4 * I));
    const int blocks = (int)std::min<size_t>(8 * (size_t)sm_count(), (I + 255) / 256);
    k_permute<<<blocks, 256, 0, s>>>(v.count.as<uint64_t>(), v.ranges.as<uint32_t>(), v.sorted_inst, v.sorted_tile, v.d_desc(), v.V, v.Ts,
                                     v.sorted_owner ? v.sorted_owner : v.iowner.as<uint32_t>(),
                                     v.rec.as<float4>(), v.srec0.as<float4>(), v.srec1.as<float4>(),
                                     v.srec2.as<float4>(), v.srec3.as<float4>(), v.sgid.as<uint32_t>());
    count_launches(1);
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

template <bool XD>
void fwd_dispatch(const View& v, const RasterArgs& A, const RasterOut& O, int64_t units, int64_t split_units,
                  cudaStream_t s)
{
    if (v.nb == 4) {
        fwd_launch<4, 1, XD>(A, O, units, split_units, v.persistent, s);
    } else if (v.nb == 8) {
        fwd_launch<8, 1, XD>(A, O, units, split_units, v.persistent, s);
    } else if (v.nb == 1) {
        if (v.pd == 1) fwd_launch<1, 1, XD>(A, O, units, split_units, v.persistent, s);
        else if (v.pd == 2) fwd_launch<1, 2, XD>(A, O, units, split_units, v.persistent, s);
        else fwd_launch<1, 4, XD>(A, O, units, split_units, v.persistent, s);
    } else {
        if (v.pd == 1) fwd_launch<2, 1, XD>(A, O, units, split_units, v.persistent, s);
        else if (v.pd == 2) fwd_launch<2, 2, XD>(A, O, units, split_units, v.persistent, s);
        else fwd_launch<2, 4, XD>(A, O, units, split_units, v.persistent, s);
    }
}

size_t segstate_bytes(const View& v)
{
    return sizeof(float) * kSegFields * (size_t)(v.Ts * v.Ts) * (size_t)split_items_bound(v);
}

gl_status reserve_segstate(View& v) { return v.segstate.reserve(segstate_bytes(v)); }

gl_status raster_forward(View& v, float* rgb, float* depth, float* opac, cudaStream_t s, bool extras)
{
    if (!extras && (depth || opac)) {
        set_error("raster_forward: depth and opacity outputs need the extra sums");
        return GL_ERR_INVALID;
    }
    const size_t P = (size_t)v.P;
    GL_TRY(v.Tfin.reserve(4 * P));
    GL_TRY(v.ncon.reserve(4 * P));
    if (v.ntiles == 0) return GL_OK;
    GL_TRY(check_exec(v));
    if (v.seg > 0) GL_TRY(reserve_segstate(v));
    PhaseScope ps(v.prof, PH_RASTER_FWD, s);
    int* work = v.persistent ? v.work.as<int>() : nullptr;   // cleared with the items
    const RasterArgs A = make_args(v, work);
    RasterOut O{rgb, depth, opac, v.Tfin.as<float>(), v.ncon.as<uint32_t>()};
    const int nblk = blocks_per_tile(v);
    // a split tile's list holds at least 2 seg records
    const int64_t tiles = v.seg > 0 ? std::min<int64_t>(v.ntiles, (int64_t)(v.itile.bytes / 4) / (2 * v.seg)) : 0;
    const int64_t units = (int64_t)v.ntiles * nblk, split_units = tiles * nblk;
    if (extras) fwd_dispatch<true>(v, A, O, units, split_units, s);
    else fwd_dispatch<false>(v, A, O, units, split_units, s);
    count_launches(1);
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

gl_status raster_backward(View& v, const float* dL_drgb, const float* dL_ddepth,
                          const float* dL_dopac, cudaStream_t s)
{
    const size_t pairs = (size_t)v.n * v.V;
    GL_TRY(v.g2d.reserve(sizeof(float) * kGradStride * std::max<size_t>(pairs, 1)));
    GL_TRY(check_exec(v));
    PhaseScope ps(v.prof, PH_RASTER_BWD, s);
    const bool det = v.det && v.ntiles > 0 && v.I != 0;
    // the per-Gaussian backward works on 8x4 pixel blocks whatever the
    // forward's pixels per lane
    const int nblk = v.pg ? v.Ts * v.Ts / 32 : blocks_per_tile(v);
    if (!det && !v.g2d_clean) GL_CUDA_TRY(cudaMemsetAsync(v.g2d.p, 0, sizeof(float) * kGradStride * pairs, s));
    v.g2d_clean = false;   // a second backward of the same binning starts over
    if (v.ntiles == 0 || v.I == 0) return GL_OK;
    int* work = nullptr;
    if (v.persistent) {
        work = v.work.as<int>() + 2;
        if (!v.work_clean) GL_CUDA_TRY(cudaMemsetAsync(work, 0, sizeof(int), s));
    }
    v.work_clean = false;
    RasterArgs A = make_args(v, work);
    A.nblk = nblk;
    RasterGrad G{v.Tfin.as<float>(), v.ncon.as<uint32_t>(), dL_drgb, dL_ddepth, dL_dopac, v.g2d.as<float>(),
                 nullptr, v.sorted_inst, nullptr};
    const size_t cap = v.itile.bytes / 4;
    if (det) {
        // every instance's block sums, and a mask of the blocks that have any;
        // the instance count is bounded by the capacity when it is known on
        // the device only
        const size_t inst = v.I > 0 ? (size_t)v.I : cap;
        GL_TRY(v.gpart.reserve(sizeof(float) * kGradStride * (size_t)nblk * std::max<size_t>(cap, 1)));
        GL_TRY(v.gmask.reserve(sizeof(uint32_t) * std::max<size_t>(cap, 1)));
        GL_CUDA_TRY(cudaMemsetAsync(v.gmask.p, 0, sizeof(uint32_t) * inst, s));
        G.part = v.gpart.as<float>();
        G.pmask = v.gmask.as<uint32_t>();
    }
    // pixel blocks, and the bound on units (a split tile's blocks count once per segment)
    const int64_t blocks = (int64_t)v.ntiles * nblk, units = work_items_bound(v) * nblk;
    if (dL_ddepth != nullptr || dL_dopac != nullptr)
        bwd_dispatch<true>(v.nb, v.pd, det, v.pg, A, G, units, blocks, v.persistent, s);
    else
        bwd_dispatch<false>(v.nb, v.pd, det, v.pg, A, G, units, blocks, v.persistent, s);
    count_launches(1);
    if (det) {
        const int blocks = (int)std::min<size_t>(8 * (size_t)sm_count(), (pairs + 31) / 32);
        k_part_reduce<<<std::max(blocks, 1), 256, 0, s>>>(v.gpart.as<float>(), v.gmask.as<uint32_t>(),
                                                          v.touched.as<uint32_t>(),
                                                          v.dup_off.as<uint32_t>(), nblk, (int64_t)pairs,
                                                          v.count.as<uint64_t>(), (uint64_t)cap, v.g2d.as<float>());
        count_launches(1);
    }
    GL_CUDA_TRY(cudaGetLastError());
    return GL_OK;
}

}  // namespace gl
