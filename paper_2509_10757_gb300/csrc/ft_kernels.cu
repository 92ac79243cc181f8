// ft_kernels.cu -- the fused, persistent tracking kernel for sm_103a.
//
// Work items (pulled in queue order by every CTA of one launch):
//   K_INDEX    per frame: the row sort of the pinhole stereo step (left and
//              right keypoints bucketed by image row, a counting sort), and
//              per camera the 64x48 keypoint grid of the search step (paper
//              section IV-E; grid reading 64x48), also a counting sort.
//   K_STEREO   pinhole: one horizontal strip of image rows.  The CTA stages
//              the row-sorted right keypoints that can reach the strip in
//              shared memory, then (1) a few lanes per left keypoint search
//              the staged candidates of its band (kernel 1 of section IV-C);
//              (2) rounds of matches: the 11x11 left patches and 11x21 right
//              strips of the next two rounds on their way into shared memory
//              while one thread per (match, patch row) adds its row to the SADs
//              of centre-subtracted patches and a warp finishes the round
//              before (best shift, parabola, disparity and depth: kernel 2 of
//              section IV-C).  The frame's last strip runs the median rejection.
//              (Fisheye frames' brute force is a kernel of its own:
//              ft_fisheye.cu.)
//   K_SEARCH   one tile of map points, one thread each: frustum test, FP32
//              projection, predicted level, scan of the grid window's packed
//              places on chip; a warp pools its points' candidates for the
//              exact tests and the Hamming distances; top-2 and ratio test;
//              accepted claims go to an atomicMin per keypoint.
//              A frame whose search is split around its stereo step scans its
//              candidates before waiting for the stereo step and applies the
//              stereo consistency after it, in the same item.
//   K_RESOLVE  one tile: final map-point -> keypoint and keypoint -> map
//              point tables from the per-keypoint winners.
// Floating point runs through __fmul_rn / __fadd_rn / __fsub_rn / __fdiv_rn /
// __fsqrt_rn so that no multiply-add is contracted and every operation is
// IEEE-rounded in the order the method defines it.
#include <cuda_runtime.h>

#include <cstdint>

#include "ft_internal.h"
#include "ft_rn.h"

namespace ft {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kNoKey = 0xffffffffu;
constexpr int kW = FT_SAD_W;
constexpr int kL = FT_SAD_L;
constexpr int kStripW = 2 * (kW + kL) + 1;                      // 21
constexpr int kShifts = 2 * kL + 1;                             // 11
constexpr int kBatch = 4;                                       // loads issued ahead per thread
constexpr int kScatter = 3;                                     // keypoints per thread per scatter batch
constexpr int kGridBatch = 8;                                   // the same in the grid build
constexpr float kPlaceX = 16383.0f, kPlaceY = 4095.0f;          // largest packed places (14 and 12 bits)

// resident CTAs per SM the register budget is sized for
#ifndef FT_MIN_CTAS_PER_SM
#define FT_MIN_CTAS_PER_SM 3
#endif

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fsqrt(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ int f2i(float x) { return __float2int_rz(x); }   // C (int) cast

__device__ __forceinline__ int ham8(uint4 a0, uint4 a1, uint4 b0, uint4 b1)
{
    return __popc(a0.x ^ b0.x) + __popc(a0.y ^ b0.y) + __popc(a0.z ^ b0.z) +
           __popc(a0.w ^ b0.w) + __popc(a1.x ^ b1.x) + __popc(a1.y ^ b1.y) +
           __popc(a1.z ^ b1.z) + __popc(a1.w ^ b1.w);
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// atan2 for y >= 0, x >= 0, from the mathematics: atan2(y, x) = atan(y/x)
// when y <= x, else pi/2 - atan(x/y); atan(t) = pi/4 + atan((t-1)/(t+1)) for
// t > tan(pi/8); below that the Taylor series of atan with terms up to a^17
// (coefficients (-1)^k / (2k+1) divided out in FP32), evaluated by Horner in
// a^2.
__device__ float atan_series(float a)
{
    const float a2 = fmul(a, a);
    float p = (1.0f / 17.0f);
    p = fadd(-(1.0f / 15.0f), fmul(a2, p));
    p = fadd((1.0f / 13.0f), fmul(a2, p));
    p = fadd(-(1.0f / 11.0f), fmul(a2, p));
    p = fadd((1.0f / 9.0f), fmul(a2, p));
    p = fadd(-(1.0f / 7.0f), fmul(a2, p));
    p = fadd((1.0f / 5.0f), fmul(a2, p));
    p = fadd(-(1.0f / 3.0f), fmul(a2, p));
    p = fadd(1.0f, fmul(a2, p));
    return fmul(a, p);
}

__device__ float atan_unit(float t)
{
    if (t > 0.41421356237309504880f)
        return fadd(0.78539816339744830962f, atan_series(fdiv(fsub(t, 1.0f), fadd(t, 1.0f))));
    return atan_series(t);
}

__device__ float atan2_pos(float y, float x)
{
    if (y == 0.0f) return 0.0f;
    if (y <= x) return atan_unit(fdiv(y, x));
    return fsub(1.57079632679489661923f, atan_unit(fdiv(x, y)));
}

// Exclusive scan of n ints (in place allowed), block-wide; returns the total.
__device__ int block_scan(const int *in, int *out, int n, int *warp_sums)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int per = (n + kThreads - 1) / kThreads;
    const int b = tid * per;
    int local = 0;
    for (int i = 0; i < per; ++i)
        if (b + i < n) local += in[b + i];
    int v = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) warp_sums[w] = v;
    __syncthreads();
    if (w == 0) {
        int s = lane < kWarps ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, s, o);
            if (lane >= o) s += t;
        }
        if (lane < kWarps) warp_sums[lane] = s;
    }
    __syncthreads();
    int run = v - local + (w > 0 ? warp_sums[w - 1] : 0);
    for (int i = 0; i < per; ++i) {
        if (b + i < n) {
            const int x = in[b + i];
            out[b + i] = run;
            run += x;
        }
    }
    const int total = warp_sums[kWarps - 1];
    __syncthreads();
    return total;
}

// ---------------------------------------------------------------- shared memory
// one match waiting for its SAD refinement
struct RefineJob {
    int i, j, d, l, ul, vl, ur0;
    float xi;
};

constexpr int kGroup = 4;                       // lanes per left keypoint in the Hamming phase
constexpr int kGroups = kThreads / kGroup;      // left keypoints in flight per CTA
constexpr int kSadChunk = 23;                   // matches refined per round: 253 of their patch rows, one a thread
constexpr int kSadBufs = 3;                     // rounds of patches on chip: one in use, two on their way
constexpr int kChunksL = 2;                     // 16-byte chunks holding a left patch row (11 bytes)
constexpr int kChunksR = 3;                     // chunks holding a right strip row (21 bytes)

// patches of one refinement round as the raw 16-byte chunks of their rows
// (copied asynchronously; a row's bytes start at offset (column & 15))
struct PatchBuf {
    uint4 l[kSadChunk][2 * kW + 1][kChunksL];
    uint4 r[kSadChunk][2 * kW + 1][kChunksR];
};
// left keypoints of a pass (Hamming phase)
struct LeftBuf {
    float4 lkp[kThreads];              // x, y, index, octave
    uint4 ldesc[2 * kThreads];
};

// what the Hamming phase reads: the staged right window and the pass's left
// keypoints
struct StageBuf {
    float4 rkp[kStageCap];             // staged right keypoints sorted by (octave, row)
    uint4 sdesc[2 * kStageCap];        // their descriptors in row order
    LeftBuf left;
    int bptr[kOctBuckets * kWinRows + 1];   // start of each (octave, window row) bucket
};

struct SmemStereo {
    union {                            // the window and the left keypoints are dead once
        StageBuf st;                   // the Hamming phase is over; the patches reuse them
        PatchBuf patch[kSadBufs];      // (a strip with a second pass stages its window again)
    } u;
    RefineJob ref[kThreads];
    int sad[2][kShifts][kSadChunk];    // this round's and the last one's
    int warp_sums[kWarps];
    int nref;
};

constexpr int kSortParts = kRowSortItems / 2;   // work items per side of a frame's row sort

struct SmemRows {
    int cnt[kSortParts][kMaxRows + 1];  // per-part row counts, then this part's write cursors
    int tot[kMaxRows + 1];              // row totals, then row starts
    int warp_sums[kWarps];
};

struct SmemGrid {
    int cnt[kCells];
    int warp_sums[kWarps];
};

constexpr int kMedianSmem = 8192;               // left keypoints whose SADs the median keeps on chip

struct SmemMedian {
    int hist[256], hist2[256];          // high bytes; low bytes within the median's high byte
    int count, bin, before;
    int vals[kMedianSmem];
};

constexpr int kCell16Bytes = (2 * (kCells + 1) + 15) / 16 * 16;   // 16-bit cell starts, whole chunks
constexpr int kStep = 4;                        // candidates a lane tests per step
constexpr int kList = 8;                        // candidates a lane collects before its warp compares them
constexpr int kSearchBuf = 56 * 1024;           // bytes for the staged grid and the split search's records
constexpr int kGridStage = (kSearchBuf - kCell16Bytes) / 6 / 8 * 8;   // keypoints of a camera's grid on chip at a time

// Where a keypoint lies, for the search's first test: x and y over the grid's
// span (one cell more at each side, so that every placed keypoint is inside)
// in 14 and 12 bits, and the octave in 4.
struct PlaceScale {
    float x0, y0, sx, sy;
};

// what a search item keeps on chip: the camera's pose, each warp's
// candidates, then (buf) the staged part of the grid (cell starts, packed
// places, indices) and, in a split search, its points' records
struct SmemSearch {
    float pose[12];
    PlaceScale ps;
    float iw, ih;                   // grid cells per pixel
    int motion;                     // of a last-frame search (f2)
    int e0, wide;                   // first staged keypoint of the grid; its indices are left in device memory
    unsigned list[kWarps][kList][32];   // candidates by lane, then the warp's pool of them
    unsigned pool[kWarps][kList * 32];
    uint4 buf[kSearchBuf / 16];
};

union Smem {
    SmemStereo s;
    SmemRows r;
    SmemGrid g;
    SmemMedian m;
    SmemSearch q;
};
// three CTAs per SM: dynamic + static shared memory + the 1 KB the SM
// reserves per CTA must stay within the SM's 228 KB
static_assert(3 * (sizeof(Smem) + sizeof(BatchHeader) + sizeof(FrameDev) + 256 + 1024) <= 228 * 1024,
              "shared memory above three CTAs per SM");

// ---------------------------------------------------------------- waits and signals
// time this CTA spent in waits during the current item, and phase marks (tracing)
__shared__ unsigned long long s_wait_ns;
__shared__ unsigned long long s_mark[4];

__device__ __forceinline__ void mark(const BatchHeader &B, int k)
{
    if (B.trace != nullptr && threadIdx.x == 0) s_mark[k] = global_ns();
}

// 16-byte asynchronous copy global -> shared (both 16-byte aligned)
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)),
                 "l"(gmem_src)
                 : "memory");
}

// Block-wide wait until *ctr >= target, bounded by the header's timeout.  On
// timeout (or when another CTA already reported one) it records the timeout in
// the status word and returns false.
// A second counter (ctr2 non-null) is polled in the same round trip.
__device__ bool wait_geq(const BatchHeader &B, const unsigned *ctr, unsigned target, int *s_flag,
                         const unsigned *ctr2 = nullptr, unsigned target2 = 0)
{
    if (threadIdx.x == 0) {
        int ok = 1;
        auto ready = [&]() {
            const unsigned a = ld_acquire(ctr);
            const unsigned b = ctr2 ? ld_acquire(ctr2) : target2;
            return a >= target && b >= target2;
        };
        if (!ready()) {
            const unsigned long long t0 = global_ns();
            unsigned spins = 0;
            while (!ready()) {
                if ((++spins & 31u) == 0) {
                    if (global_ns() - t0 > B.timeout_ns || (ld_acquire(B.status) & kStatusTimeout)) {
                        ok = 0;
                        break;
                    }
                }
                __nanosleep(256);
            }
            if (!ok) atomicOr(B.status, kStatusTimeout);
            s_wait_ns += global_ns() - t0;
        }
        *s_flag = ok;
    }
    __syncthreads();
    const bool ok = *s_flag != 0;
    __syncthreads();
    return ok;
}

// Publish this CTA's writes and add one to *ctr; returns true in every thread
// of the CTA that brought the counter to `total`.
__device__ bool signal_count(unsigned *ctr, unsigned total, int *s_flag)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned prev = atomicAdd(ctr, 1u);
        const int last = (prev + 1u == total);
        if (last) __threadfence();
        *s_flag = last;
    }
    __syncthreads();
    const bool last = *s_flag != 0;
    __syncthreads();
    return last;
}

// ---------------------------------------------------------------- K_INDEX
__device__ __forceinline__ int grid_cell(const CamDev &C, float iw, float ih, float x, float y)
{
    const int cx = f2i(roundf(fmul(fsub(x, C.minx), iw)));
    const int cy = f2i(roundf(fmul(fsub(y, C.miny), ih)));
    if (cx < 0 || cx >= FT_GRID_COLS || cy < 0 || cy >= FT_GRID_ROWS) return -1;
    return cy * FT_GRID_COLS + cx;
}

__device__ __forceinline__ PlaceScale place_scale(const CamDev &C)
{
    PlaceScale s;
    const float w = fsub(C.maxx, C.minx), h = fsub(C.maxy, C.miny);
    s.x0 = fsub(C.minx, fdiv(w, (float)FT_GRID_COLS));
    s.y0 = fsub(C.miny, fdiv(h, (float)FT_GRID_ROWS));
    s.sx = fdiv(kPlaceX * (float)FT_GRID_COLS / (float)(FT_GRID_COLS + 2), w);
    s.sy = fdiv(kPlaceY * (float)FT_GRID_ROWS / (float)(FT_GRID_ROWS + 2), h);
    // a span too small to scale: every place is 0 and passes the first test
    if (!(s.sx < 1e30f)) s.sx = 0.0f;
    if (!(s.sy < 1e30f)) s.sy = 0.0f;
    return s;
}

__device__ __forceinline__ unsigned place_of(float t, float top) { return (unsigned)f2i(fminf(fmaxf(t, 0.0f), top)); }

__device__ __forceinline__ unsigned pack_place(const PlaceScale &s, float x, float y, unsigned oct)
{
    return place_of(fmul(fsub(x, s.x0), s.sx), kPlaceX) | place_of(fmul(fsub(y, s.y0), s.sy), kPlaceY) << 16 |
           oct << 28;
}

// The keypoints that can be matched (in the grid, not taken, an octave below
// 16) in cell order: 6 bytes each, so that a search item's staging of a whole
// camera is short; coordinates, descriptors and right coordinates are read
// from the frame's own arrays, for the few candidates that pass the first
// test.  One block per camera; 8 keypoints' loads in flight per thread
// (1200 keypoints: 6 us; with 48-byte records copied in cell order 10 us;
// 8000 keypoints: 16 against 44 us).
__device__ void grid_item(const BatchHeader &B, const FrameDev &F, int cam, SmemGrid &G,
                          int *s_flag)
{
    const CamDev &C = F.cam[cam];
    const int tid = threadIdx.x;
    const float iw = fdiv((float)FT_GRID_COLS, fsub(C.maxx, C.minx));
    const float ih = fdiv((float)FT_GRID_ROWS, fsub(C.maxy, C.miny));
    const PlaceScale ps = place_scale(C);
    for (int c = tid; c < kCells; c += kThreads) G.cnt[c] = 0;
    __syncthreads();
    auto pass = [&](bool place) {
        for (int base = 0; base < C.nk; base += kGridBatch * kThreads) {
            float x[kGridBatch], y[kGridBatch];
            unsigned oct[kGridBatch], tk[kGridBatch];
#pragma unroll
            for (int u = 0; u < kGridBatch; ++u) {
                const int k = min(base + u * kThreads + tid, C.nk - 1);
                x[u] = __ldg(C.kx + k);
                y[u] = __ldg(C.ky + k);
                oct[u] = (unsigned)(int)__ldg(C.koct + k);
                tk[u] = C.taken ? (unsigned)__ldg(C.taken + k) : 0u;
            }
#pragma unroll
            for (int u = 0; u < kGridBatch; ++u) {
                const int k = base + u * kThreads + tid;
                if (k >= C.nk) continue;
                if (!place) C.owner[k] = ~0ull;
                const int c = grid_cell(C, iw, ih, x[u], y[u]);
                if (c < 0 || tk[u] || oct[u] > 15u) continue;
                const int pos = atomicAdd(&G.cnt[c], 1);
                if (!place) continue;
                C.gq[pos] = pack_place(ps, x[u], y[u], oct[u]);
                if (C.gk32) C.gk32[pos] = k;
                else C.gk16[pos] = (uint16_t)k;
            }
        }
    };
    pass(false);
    __syncthreads();
    mark(B, 0);
    const int total = block_scan(G.cnt, G.cnt, kCells, G.warp_sums);
    for (int c = tid; c < kCells; c += kThreads) C.cell_ptr[c] = G.cnt[c];
    if (tid == 0) C.cell_ptr[kCells] = total;
    __syncthreads();
    mark(B, 1);
    pass(true);
    mark(B, 2);
    signal_count(&F.ctr[C_GRID_DONE], (unsigned)F.n_grid_items, s_flag);
    mark(B, 3);
}

// ---------------------------------------------------------------- K_INDEX: row sort
__device__ __forceinline__ int floor_row(float y) { return f2i(floorf(y)); }

// Row that owns a keypoint in the row sort (rows outside the image go to the
// edge rows).
__device__ __forceinline__ int own_row(float y, int H)
{
    if (y < 0.0f) return 0;
    return min(f2i(y), H - 1);
}

// Right keypoints are bucketed by floor(y) clamped to the image, left
// keypoints by the row they search, (int)y clamped to the image.  Each side's
// sort is split over kSortParts work items that run side by side: every part
// counts all keypoints per row and per part, and scatters only its own
// contiguous share, starting each row after the parts before it.
__device__ __forceinline__ int sort_row(bool right, float y, int H)
{
    return right ? clampi(floor_row(y), 0, H - 1) : own_row(y, H);
}

__device__ void rowsort_item(const BatchHeader &B, const FrameDev &F, SmemRows &S, bool right, int part,
                             int *s_flag)
{
    const int tid = threadIdx.x, H = F.H;
    const int n = right ? F.nr : F.nl;
    const float *ys = right ? F.ry : F.ly;
    const int share = (n + kSortParts - 1) / kSortParts;
    for (int r = tid; r <= H; r += kThreads)
        for (int p = 0; p < kSortParts; ++p) S.cnt[p][r] = 0;
    __syncthreads();
    for (int base = 0; base < n; base += kBatch * kThreads) {
        float y[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = base + u * kThreads + tid;
            y[u] = i < n ? __ldg(ys + i) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = base + u * kThreads + tid;
            if (i < n) atomicAdd(&S.cnt[i / share][sort_row(right, y[u], H)], 1);
        }
    }
    __syncthreads();
    mark(B, 0);
    for (int r = tid; r < H; r += kThreads) {
        int t = 0;
        for (int p = 0; p < kSortParts; ++p) t += S.cnt[p][r];
        S.tot[r] = t;
    }
    __syncthreads();
    const int total = block_scan(S.tot, S.tot, H, S.warp_sums);
    // this part's write cursor per row: the row's start plus the earlier parts' counts
    for (int r = tid; r < H; r += kThreads) {
        int c = S.tot[r];
        for (int p = 0; p < part; ++p) c += S.cnt[p][r];
        S.cnt[part][r] = c;
    }
    if (part == 0) {
        int *row_ptr = right ? F.row_ptr_r : F.row_ptr_l;
        for (int r = tid; r < H; r += kThreads) row_ptr[r] = S.tot[r];
        if (tid == 0) row_ptr[H] = total;
    }
    __syncthreads();
    mark(B, 1);
    // the part's share: records (right: x, band rows, row, index | octave;
    // left: x, y, index, octave) and descriptors in row order, so that the
    // stereo strips read them contiguously (all loads of a batch are issued
    // before its shared-memory atomics)
    const int i0 = part * share, i1 = min(n, i0 + share);
    const float *xs = right ? F.rx : F.lx;
    const int8_t *os = right ? F.roct : F.loct;
    const uint4 *ds = right ? F.rdesc : F.ldesc;
    float4 *rec_out = right ? F.rs_kp : F.ls_kp;
    uint4 *desc_out = right ? F.rs_desc : F.ls_desc;
    for (int base = i0; base < i1; base += kScatter * kThreads) {
        float x[kScatter], y[kScatter];
        int oct[kScatter];
        uint4 d0[kScatter], d1[kScatter];
#pragma unroll
        for (int u = 0; u < kScatter; ++u) {
            const int i = min(base + u * kThreads + tid, i1 - 1);
            x[u] = __ldg(xs + i);
            y[u] = __ldg(ys + i);
            oct[u] = __ldg(os + i);
            d0[u] = __ldg(ds + 2 * i);
            d1[u] = __ldg(ds + 2 * i + 1);
        }
#pragma unroll
        for (int u = 0; u < kScatter; ++u) {
            const int i = base + u * kThreads + tid;
            if (i >= i1) continue;
            const int row = sort_row(right, y[u], H);
            const int pos = atomicAdd(&S.cnt[part][row], 1);
            if (right) {
                // the rows this keypoint lists: floor(y - r) .. ceil(y + r), r = 2 scale[oct],
                // clamped to the image (computed once here, tested per candidate later;
                // an empty band stays empty: lo in [0, H], hi in [-1, H - 1])
                const float r = B.p.band_r[clampi(oct[u], 0, B.p.nlevels - 1)];
                const int lo = min(max(f2i(floorf(fsub(y[u], r))), 0), H);
                const int hi = max(min(f2i(ceilf(fadd(y[u], r))), H - 1), -1);
                rec_out[pos] = make_float4(x[u], __int_as_float(lo | (hi << 16)), __int_as_float(row),
                                           __int_as_float(i | ((oct[u] & 0xff) << 20)));
            } else {
                rec_out[pos] = make_float4(x[u], y[u], __int_as_float(i), __int_as_float(oct[u]));
            }
            desc_out[2 * pos] = d0[u];
            desc_out[2 * pos + 1] = d1[u];
        }
    }
    mark(B, 2);
    signal_count(&F.ctr[C_ROWS_DONE], (unsigned)F.rowsort, s_flag);
    mark(B, 3);
}

// ---------------------------------------------------------------- K_STEREO, pinhole
// A row-sorted right keypoint record: x, band rows lo | hi << 16, bucket row,
// index | octave << 20.
__device__ __forceinline__ bool band_has(float packed, int row)
{
    const int b = __float_as_int(packed);
    return (b & 0xffff) <= row && row <= (b >> 16);
}
__device__ __forceinline__ int rec_index(float w) { return __float_as_int(w) & 0xfffff; }
__device__ __forceinline__ int rec_octave(float w) { return (int)(int8_t)((__float_as_int(w) >> 20) & 0xff); }

__device__ __forceinline__ void write_stereo(const FrameDev &F, int i, int best, int dist, int shift,
                                             int sadb, float ur, float dep)
{
    F.best_r[i] = best;
    F.dist[i] = dist;
    F.sad_shift[i] = shift;
    F.sad_best[i] = sadb;
    F.u_right[i] = ur;
    F.depth[i] = dep;
}

// Phase 1: the kGroup lanes of a group scan the band candidates of one left
// keypoint (consecutive candidates per lane, conflict-free shared loads) and
// reduce to the smallest (distance, right index); lane 0 of the group queues
// the match for refinement or writes the final "no match" outputs.
__device__ void hamming_phase(const DevParams &P, const FrameDev &F, SmemStereo &S, int npass,
                              bool staged, int w_a, int nrows)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane & (kGroup - 1), gw = lane / kGroup;
    const float disp_hi = fdiv(F.bf, F.b);
    for (int tb = warp * (32 / kGroup); tb < npass; tb += kGroups) {
        const int t = tb + gw;
        const bool have = t < npass;
        unsigned key = kNoKey;
        float xb = 0.0f;
        float xi = 0.0f, yi = 0.0f;
        int oi = 0, i = 0;
        if (have) {
            const float4 L = S.u.st.left.lkp[t];
            xi = L.x;
            yi = L.y;
            i = __float_as_int(L.z);
            oi = __float_as_int(L.w);
            const int row = f2i(yi);
            const float u_lo = fsub(xi, disp_hi);
            const float u_hi = fsub(xi, 0.0f);
            if (!(yi < 0.0f) && row < F.H && !(u_hi < 0.0f)) {
                const uint4 a0 = S.u.st.left.ldesc[2 * t], a1 = S.u.st.left.ldesc[2 * t + 1];
                if (staged) {
                    // candidate octaves oi-1 .. oi+1, each over the rows its band
                    // can reach: up to three ranges of records, taken as one
                    // list, two of a lane's candidates at a time (an octave
                    // after the other: one frame 28.1 us, now 27.6; 32 frames
                    // of 1920x1080 502 and 498)
                    const int olo = max(oi - 1, 0), ohi = min(oi + 1, kOctBuckets - 1);
                    int from[3], end[3], n = 0;             // record = place in the list + from
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const int o = min(olo + q, kOctBuckets - 1), h = P.halo_c[o];
                        const int ra = max(row - h, w_a) - w_a;
                        const int rb = min(row + h, w_a + nrows - 1) - w_a;
                        const int e0 = S.u.st.bptr[o * nrows + ra], e1 = S.u.st.bptr[o * nrows + rb + 1];
                        from[q] = e0 - n;
                        n += olo + q <= ohi ? e1 - e0 : 0;
                        end[q] = n;
                    }
                    auto record = [&](int j) { return j + (j < end[0] ? from[0] : j < end[1] ? from[1] : from[2]); };
                    for (int j = sub; j < n; j += 2 * kGroup) {
                        // past the list's end the first candidate comes again
                        const float4 g[2] = {S.u.st.rkp[record(j)], S.u.st.rkp[record(j + kGroup < n ? j + kGroup : j)]};
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int oj = rec_octave(g[u].w);
                            if (oj < oi - 1 || oj > oi + 1) continue;
                            if (!band_has(g[u].y, row)) continue;
                            if (g[u].x < u_lo || g[u].x > u_hi) continue;
                            const int at = __float_as_int(g[u].z);
                            const unsigned k = ((unsigned)ham8(a0, a1, S.u.st.sdesc[2 * at], S.u.st.sdesc[2 * at + 1]) << 20) |
                                               (unsigned)rec_index(g[u].w);
                            if (k < key) {
                                key = k;
                                xb = g[u].x;
                            }
                        }
                    }
                } else {
                    const int h = (oi >= 0 && oi < P.nlevels) ? P.halo_oct[oi] : P.halo;
                    const int e0 = __ldcg(F.row_ptr_r + max(row - h, 0));
                    const int e1 = __ldcg(F.row_ptr_r + min(row + h, F.H - 1) + 1);
                    for (int e = e0 + sub; e < e1; e += kGroup) {
                        const float4 g = __ldcg(F.rs_kp + e);
                        const int oj = rec_octave(g.w);
                        if (oj < oi - 1 || oj > oi + 1) continue;
                        if (!band_has(g.y, row)) continue;
                        if (g.x < u_lo || g.x > u_hi) continue;
                        const unsigned k = ((unsigned)ham8(a0, a1, __ldcg(F.rs_desc + 2 * e),
                                                           __ldcg(F.rs_desc + 2 * e + 1)) << 20) |
                                           (unsigned)rec_index(g.w);
                        if (k < key) {
                            key = k;
                            xb = g.x;
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int o = kGroup / 2; o > 0; o >>= 1) {
            const unsigned k2 = __shfl_xor_sync(kFull, key, o);
            const float x2 = __shfl_xor_sync(kFull, xb, o);
            if (k2 < key) {
                key = k2;
                xb = x2;
            }
        }
        // every lane of the group holds the reduced key
        if (have) {
            int best = -1, dist = -1;
            if (key != kNoKey) {
                dist = (int)(key >> 20);
                if (dist < P.th_stereo) best = (int)(key & 0xfffffu);
            }
            bool queued = false;
            if (best >= 0) {
                const int l = clampi(oi, 0, P.nlevels - 1);
                const int ul = f2i(roundf(fmul(xi, P.isc[l])));
                const int vl = f2i(roundf(fmul(yi, P.isc[l])));
                const int ur0 = f2i(roundf(fmul(xb, P.isc[l])));
                // windows inside both level images.  ul, vl and ur0 saturate at
                // INT_MAX / INT_MIN for coordinates of 2^31 and more (or +-inf), so
                // they are compared with the bounds and never offset: ul + kW would
                // wrap negative and let a window 2 GB past the level through.
                const bool inside = vl >= kW && vl <= F.lh[l] - 1 - kW && vl <= F.rh[l] - 1 - kW &&
                                    ul >= kW && ul <= F.lw[l] - 1 - kW &&
                                    ur0 >= kL + kW && ur0 <= F.rw[l] - 1 - kL - kW;
                if (inside) {
                    // the lanes ask L2 for the patch rows now, so that the
                    // refinement's copies find them there
                    for (int rr = sub; rr < 2 * kW + 1; rr += kGroup) {
                        const uint8_t *pl = F.pyrL[l] + (size_t)(vl - kW + rr) * F.lp[l] + (ul - kW);
                        const uint8_t *pr = F.pyrR[l] + (size_t)(vl - kW + rr) * F.rp[l] + (ur0 - kL - kW);
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(pl));
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(pr));
                        if (((reinterpret_cast<uintptr_t>(pr) & 127u) + kStripW - 1) >= 128u)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(pr + kStripW - 1));
                        if (((reinterpret_cast<uintptr_t>(pl) & 127u) + 2 * kW) >= 128u)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(pl + 2 * kW));
                    }
                    if (sub == 0) {
                        const int slot = atomicAdd(&S.nref, 1);
                        S.ref[slot] = RefineJob{i, best, dist, l, ul, vl, ur0, xi};
                    }
                    queued = true;
                }
            }
            if (!queued && sub == 0) write_stereo(F, i, best, dist, FT_NO_SHIFT, -1, -1.0f, -1.0f);
        }
    }
}

// Asks for the patches of refine round r (jobs r * kSadChunk ...) by
// asynchronous copies of the 16-byte chunks holding every patch row, and
// closes the group; a match has five chunk slots (two of a left row, three of
// a right row) and two threads per slot walk the 11 rows.  Level pointers and
// pitches are 16-byte aligned (checked on the host): a row's chunks start at
// its column rounded down to a multiple of 16 and end within the row's pitch.
__device__ __forceinline__ void refine_copy(const FrameDev &F, SmemStereo &S, int r, int nref)
{
    constexpr int kSlots = kChunksL + kChunksR, kRows = 2 * kW + 1, kHalf = (kRows + 1) / 2;
    const int nc = min(kSadChunk, nref - r * kSadChunk);
    const int q = threadIdx.x, mm = q / (2 * kSlots), w = (q - mm * 2 * kSlots) >> 1, row0 = (q & 1) * kHalf;
    PatchBuf &B = S.u.patch[r % kSadBufs];
    if (mm < nc) {
        const bool right = w >= kChunksL;
        const int k = right ? w - kChunksL : w;
        const RefineJob &J = S.ref[r * kSadChunk + mm];
        const int col = right ? J.ur0 - kL - kW : J.ul - kW;
        const int len = right ? kStripW : 2 * kW + 1;
        if (k <= (((col & 15) + len - 1) >> 4)) {           // else the chunk holds none of the row's bytes
            const int pitch = right ? F.rp[J.l] : F.lp[J.l];
            const uint8_t *src =
                (right ? F.pyrR[J.l] : F.pyrL[J.l]) + (size_t)(J.vl - kW + row0) * pitch + (col & ~15) + 16 * k;
            const unsigned dst = (unsigned)__cvta_generic_to_shared(right ? &B.r[mm][row0][k] : &B.l[mm][row0][k]);
            const unsigned dstep = 16u * (right ? kChunksR : kChunksL);
#pragma unroll
            for (int row = 0; row < kHalf; ++row)
                if (row0 + row < kRows)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + row * dstep),
                                 "l"(src + (size_t)row * pitch)
                                 : "memory");
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Adds this thread's patch row of round r to the 11 SADs of its match.  The
// pixels go in pairs: |p - q| = 2 max(p, q) - p - q, so a pair costs one
// instruction (an add of the centres' difference and the larger of the lanes;
// the larger is never below the right pixel, so sums of lanes do not borrow)
// and the two other sums come from dot products, the right one sliding from
// shift to shift.  (A difference and an absolute sum per pixel before: 64
// frames 98.0 us, now 96.2; 32 frames of 1920x1080 507 and 501.)
__device__ __forceinline__ void refine_row(SmemStereo &S, int r, int nref)
{
    constexpr int kRows = 2 * kW + 1;
    static_assert(kSadChunk * kRows <= kThreads, "one patch row a thread");
    const int nc = min(kSadChunk, nref - r * kSadChunk);
    const PatchBuf &B = S.u.patch[r % kSadBufs];
    const int dy = threadIdx.x / kSadChunk, mm = threadIdx.x - dy * kSadChunk;
    if (dy < kRows && mm < nc) {
        const RefineJob &J = S.ref[r * kSadChunk + mm];
        const int ol = (J.ul - kW) & 15, orr = (J.ur0 - kL - kW) & 15;
        // the rows as 32-bit words; byte b of a row is byte (o + b) of its chunks
        const unsigned *ql = reinterpret_cast<const unsigned *>(B.l[mm][dy]) + (ol >> 2);
        const unsigned *qr = reinterpret_cast<const unsigned *>(B.r[mm][dy]) + (orr >> 2);
        const unsigned *qc = reinterpret_cast<const unsigned *>(B.r[mm][kW]) + (orr >> 2);
        const unsigned *qlc = reinterpret_cast<const unsigned *>(B.l[mm][kW]) + (ol >> 2);
        const int sl = 8 * (ol & 3), sr = 8 * (orr & 3);
        // realigned words: byte b of the row is byte b & 3 of word b >> 2
        unsigned wl[3], wr[6], wc[4];
#pragma unroll
        for (int k = 0; k < 3; ++k) wl[k] = __funnelshift_r(ql[k], ql[k + 1], sl);
#pragma unroll
        for (int k = 0; k < 6; ++k) wr[k] = __funnelshift_r(qr[k], qr[k + 1], sr);
#pragma unroll
        for (int k = 1; k < 4; ++k) wc[k] = __funnelshift_r(qc[k], qc[k + 1], sr);
        // pairs of left pixels, and of right pixels that start at an even or
        // an odd byte, in 16-bit lanes; the left row's sixth pair is its last
        // pixel and a value below all others
        unsigned a[6], e[11], o[10];
#pragma unroll
        for (int i = 0; i < 6; ++i) a[i] = __byte_perm(wl[i >> 1], 0u, i & 1 ? 0x4342 : 0x4140);
        a[5] = (a[5] & 0xffffu) | 0x8ad00000u;              // -30000 in the upper lane
#pragma unroll
        for (int i = 0; i < 11; ++i) e[i] = __byte_perm(wr[i >> 1], 0u, i & 1 ? 0x4342 : 0x4140);
#pragma unroll
        for (int i = 0; i < 10; ++i)
            o[i] = i & 1 ? __byte_perm(__funnelshift_r(wr[i >> 1], wr[(i >> 1) + 1], 24), 0u, 0x4140)
                         : __byte_perm(wr[i >> 1], 0u, 0x4241);
        const int cl = (int)((__funnelshift_r(qlc[1], qlc[2], sl) >> 8) & 0xff);
        // minus the sums of the left row (centred) and of the shift's right
        // pixels, which slide by one
        int minus = 11 * cl;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int w = k < 2 ? (int)0xffffffff : 0x00ffffff;              // -1 per byte
            asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(minus) : "r"(wl[k]), "r"(w));
            asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(minus) : "r"(wr[k]), "r"(w));
        }
#pragma unroll
        for (int k = 0; k < kShifts; ++k) {
            const int c = (int)__byte_perm(wc[(k + kW) >> 2], 0u, 0x4440 + ((k + kW) & 3));
            const unsigned c2 = __byte_perm((unsigned)(c - cl), 0u, 0x1010);
            const unsigned *b = k & 1 ? o + (k >> 1) : e + (k >> 1);
            unsigned m[6];
#pragma unroll
            for (int i = 0; i < 5; ++i) m[i] = __viaddmax_s16x2(a[i], c2, b[i]);
            m[5] = __viaddmax_s16x2(a[5], c2, b[5] & 0xffffu);
            const unsigned sum = (m[0] + m[1] + m[2]) + (m[3] + m[4] + m[5]);
            atomicAdd(&S.sad[r & 1][k][mm], (int)__dp2a_lo(sum, 0x0202u, (unsigned)(minus - 11 * c)));
            if (k + 1 < kShifts) {
                const unsigned t = __byte_perm(wr[k >> 2], wr[(k + 11) >> 2], 0x0000 + (k & 3) + ((4 + ((k + 11) & 3)) << 4));
                asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(minus) : "r"(t), "r"(0xff01));     // + the first, - the next
            }
        }
    }
}

// Match m of round r: the first strict minimum over the shifts, the parabola,
// disparity and depth; its SADs are left zero for round r + 2.
__device__ __forceinline__ void refine_finish(const DevParams &P, const FrameDev &F, SmemStereo &S, int r, int nref, int m)
{
    if (m < min(kSadChunk, nref - r * kSadChunk)) {
        const RefineJob &J = S.ref[r * kSadChunk + m];
        int sad[kShifts];
#pragma unroll
        for (int k = 0; k < kShifts; ++k) {
            sad[k] = S.sad[r & 1][k][m];
            S.sad[r & 1][k][m] = 0;
        }
        // (the neighbours of the minimum are carried along: no dynamic index)
        int kb = 0, lo = 0, best = sad[0], hi = sad[1];
#pragma unroll
        for (int k = 1; k < kShifts; ++k)
            if (sad[k] < best) {
                kb = k;
                lo = sad[k - 1];
                best = sad[k];
                hi = k + 1 < kShifts ? sad[k + 1 < kShifts ? k + 1 : k] : 0;
            }
        const int shift = kb - kL;
        int sadb = -1;
        float ur = -1.0f, dep = -1.0f;
        if (kb != 0 && kb != 2 * kL) {
            const float d1 = (float)lo, d2 = (float)best, d3 = (float)hi;
            const float delta = fdiv(fsub(d1, d3), fmul(2.0f, fsub(fadd(d1, d3), fmul(2.0f, d2))));
            if (!(delta < -1.0f || delta > 1.0f)) {
                float ur_sub = fmul(P.sc[J.l], fadd(fadd((float)J.ur0, (float)shift), delta));
                float disparity = fsub(J.xi, ur_sub);
                const float disp_hi = fdiv(F.bf, F.b);
                if (disparity >= 0.0f && disparity < disp_hi) {
                    if (disparity <= 0.0f) {
                        disparity = 0.01f;
                        ur_sub = fsub(J.xi, 0.01f);
                    }
                    dep = fdiv(F.bf, disparity);
                    ur = ur_sub;
                    sadb = best;
                }
            }
        }
        write_stereo(F, J.i, J.j, J.d, shift, sadb, ur, dep);
    }
}

// Refinement of the pass's nref matches: rounds of kSadChunk, the copies of
// the next two rounds on their way while a round is summed and the last
// warp finishes the round before it; one block-wide synchronization a round.
// What bounds a round is the latency of its scattered rows: rounds of 64
// matches that waited for their own copies took 15.2 us a strip of 112
// matches (64 frames, 3 blocks an SM), these 12.5 us, 12 with paired pixels.
__device__ void refine_matches(const DevParams &P, const FrameDev &F, SmemStereo &S, int nref)
{
    const int tid = threadIdx.x, last = tid - (kThreads - 32);
    static_assert(kSadChunk <= 32 && kSadBufs == 3, "a warp finishes a round; two rounds of copies in flight");
    for (int q = tid; q < 2 * kShifts * kSadChunk; q += kThreads) (&S.sad[0][0][0])[q] = 0;
    refine_copy(F, S, 0, nref);
    refine_copy(F, S, 1, nref);
    const int rounds = (nref + kSadChunk - 1) / kSadChunk;
    for (int r = 0; r < rounds; ++r) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        refine_copy(F, S, r + 2, nref);             // into the buffer of round r - 1
        if (r > 0 && last >= 0) refine_finish(P, F, S, r - 1, nref, last);
        refine_row(S, r, nref);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (rounds > 0 && last >= 0) refine_finish(P, F, S, rounds - 1, nref, last);
}

// warp 0: bin of the k-th smallest value (0-based) of a 256-bin histogram
__device__ void select_bin(const int *hist, int k, int *bin, int *before)
{
    const int lane = threadIdx.x & 31;
    int s = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) s += hist[lane * 8 + j];
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    const int excl = incl - s;
    const unsigned m = __ballot_sync(kFull, excl <= k && k < incl);
    if (lane == __ffs(m) - 1) {
        int c = excl;
        for (int j = 0; j < 8; ++j) {
            const int h = hist[lane * 8 + j];
            if (k < c + h) {
                *bin = lane * 8 + j;
                *before = c;
                break;
            }
            c += h;
        }
    }
}

// a5: median of the frame's accepted SAD minima (radix select on 2 x 8 bits),
// then drop matches with SAD >= factor * median.  Frames of up to
// kMedianSmem left keypoints load the values once into shared memory;
// larger frames read them three times.
__device__ __forceinline__ int median_value(const FrameDev &F, const SmemMedian &M, bool on_chip, int i)
{
    return on_chip ? M.vals[i] : __ldcg(F.sad_best + i);
}

constexpr int kMedianBatch = 8;   // values a thread loads at once in the median's first pass

__device__ void median_reject(const BatchHeader &B, const FrameDev &F, SmemMedian &M)
{
    const DevParams &P = B.p;
    const int tid = threadIdx.x;
    const bool on_chip = F.nl <= kMedianSmem;
    for (int b = tid; b < 256; b += kThreads) M.hist[b] = M.hist2[b] = 0;
    if (tid == 0) M.count = 0;
    __syncthreads();
    // one pass over the values (kept on chip when they fit): the count and
    // the histogram of the high bytes; a thread loads kMedianBatch values
    // before it stores or counts any
    int local = 0;
    for (int i0 = tid; i0 < F.nl; i0 += kThreads * kMedianBatch) {
        int xv[kMedianBatch];
#pragma unroll
        for (int u = 0; u < kMedianBatch; ++u) {
            const int i = i0 + u * kThreads;
            xv[u] = i < F.nl ? __ldcg(F.sad_best + i) : -1;
        }
#pragma unroll
        for (int u = 0; u < kMedianBatch; ++u) {
            const int i = i0 + u * kThreads;
            if (i >= F.nl) continue;
            if (on_chip) M.vals[i] = xv[u];
            if (xv[u] >= 0) {
                atomicAdd(&M.hist[(xv[u] >> 8) & 255], 1);
                ++local;
            }
        }
    }
    local = __reduce_add_sync(kFull, local);
    if ((tid & 31) == 0 && local) atomicAdd(&M.count, local);
    __syncthreads();
    const int n = M.count;
    if (n == 0) return;
    const int k = n / 2;
    if (tid < 32) select_bin(M.hist, k, &M.bin, &M.before);
    __syncthreads();
    const int hi = M.bin;
    const int k2 = k - M.before;
    for (int i = tid; i < F.nl; i += kThreads) {
        const int x = median_value(F, M, on_chip, i);
        if (x >= 0 && ((x >> 8) & 255) == hi) atomicAdd(&M.hist2[x & 255], 1);
    }
    __syncthreads();
    if (tid < 32) select_bin(M.hist2, k2, &M.bin, &M.before);
    __syncthreads();
    const int median = (hi << 8) | M.bin;
    const float th = fmul(P.median_factor, (float)median);
    for (int i = tid; i < F.nl; i += kThreads) {
        const int x = median_value(F, M, on_chip, i);
        if (x < 0) continue;
        if ((float)x >= th) {
            F.u_right[i] = -1.0f;
            F.depth[i] = -1.0f;
        }
    }
}

// Stage the row-sorted right keypoints of window rows [w_a, w_a + nrows)
// in shared memory, re-bucketed by (octave, row) so that a left keypoint
// visits only its octaves; their descriptors keep row order (a staged record
// carries its row-order position) and arrive by asynchronous copies that the
// caller waits for.
__device__ __forceinline__ void stage_window(const FrameDev &F, SmemStereo &S, int w_a, int nrows, int e_base,
                                             int n_st)
{
    const int tid = threadIdx.x;
    for (int e = tid; e < 2 * n_st; e += kThreads) cp_async16(&S.u.st.sdesc[e], F.rs_desc + 2 * e_base + e);
    constexpr int Q = kStageCap / kThreads;
    const int nb = kOctBuckets * nrows;
    for (int b = tid; b <= nb; b += kThreads) S.u.st.bptr[b] = 0;
    __syncthreads();
    float4 g[Q];
    int bucket[Q], rank[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int e = q * kThreads + tid;
        if (e < n_st) {
            g[q] = __ldcg(F.rs_kp + e_base + e);
            bucket[q] = clampi(rec_octave(g[q].w), 0, kOctBuckets - 1) * nrows + (__float_as_int(g[q].z) - w_a);
            rank[q] = atomicAdd(&S.u.st.bptr[bucket[q]], 1);
        }
    }
    __syncthreads();
    block_scan(S.u.st.bptr, S.u.st.bptr, nb + 1, S.warp_sums);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int e = q * kThreads + tid;
        if (e < n_st) {
            g[q].z = __int_as_float(e);          // row-order position: its descriptor
            S.u.st.rkp[S.u.st.bptr[bucket[q]] + rank[q]] = g[q];
        }
    }
}

__device__ void stereo_pinhole_item(const BatchHeader &B, const FrameDev &F, int strip, Smem &U,
                                    int *s_flag)
{
    SmemStereo &S = U.s;
    const DevParams &P = B.p;
    const int tid = threadIdx.x;
    if (wait_geq(B, &F.ctr[C_ROWS_DONE], (unsigned)F.rowsort, s_flag)) {
        const int H = F.H;
        const int r_lo = strip * F.strip_rows;
        const int r_hi = min(H, r_lo + F.strip_rows);
        // the window of right keypoint rows [w_a, w_b] the strip's bands can reach
        const int w_a = max(r_lo - P.halo, 0);
        const int w_b = min(r_hi - 1 + P.halo, H - 1);
        const int nrows = w_b - w_a + 1;
        const int e_base = __ldcg(F.row_ptr_r + w_a);
        const int e_end = __ldcg(F.row_ptr_r + w_b + 1);
        const int l_lo = __ldcg(F.row_ptr_l + r_lo), l_hi = __ldcg(F.row_ptr_l + r_hi);
        const int n_st = e_end - e_base;
        const bool staged = n_st <= kStageCap && nrows <= kWinRows && P.nlevels <= kOctBuckets;
        if (tid == 0) S.nref = 0;
        for (int pass = l_lo; pass < l_hi; pass += kThreads) {
            // the pass's left keypoints arrive by asynchronous copies while the
            // window is staged (again for a later pass: the previous pass's
            // patches overwrote it)
            const int npass = min(kThreads, l_hi - pass);
            if (tid < npass) {
                cp_async16(&S.u.st.left.lkp[tid], F.ls_kp + pass + tid);
                cp_async16(&S.u.st.left.ldesc[2 * tid], F.ls_desc + 2 * (pass + tid));
                cp_async16(&S.u.st.left.ldesc[2 * tid + 1], F.ls_desc + 2 * (pass + tid) + 1);
            }
            if (staged) stage_window(F, S, w_a, nrows, e_base, n_st);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            mark(B, 0);
            hamming_phase(P, F, S, npass, staged, w_a, nrows);
            __syncthreads();
            mark(B, 1);
            wait_for_previous();                // the levels the refinement reads
            const int nref = S.nref;
            refine_matches(P, F, S, nref);
            __syncthreads();
            if (tid == 0) S.nref = 0;
            mark(B, 2);
        }
    }
    if (signal_count(&F.ctr[C_STEREO_DONE], (unsigned)F.n_stereo_items, s_flag)) {
        median_reject(B, F, U.m);
        __threadfence();
        __syncthreads();
        mark(B, 3);
        if (tid == 0 && !(B.debug_flags & kDebugWithholdStereoReady))
            atomicExch(&F.ctr[C_STEREO_READY], 1u);
    }
}

// ---------------------------------------------------------------- K_SEARCH
__device__ void resolve_range(const CamDev &C, int nm, int i0, int i1);

__device__ __forceinline__ void transform(const float *pose, float4 p, float &x, float &y, float &z)
{
    x = fadd(fadd(fadd(fmul(pose[0], p.x), fmul(pose[1], p.y)), fmul(pose[2], p.z)), pose[9]);
    y = fadd(fadd(fadd(fmul(pose[3], p.x), fmul(pose[4], p.y)), fmul(pose[5], p.z)), pose[10]);
    z = fadd(fadd(fadd(fmul(pose[6], p.x), fmul(pose[7], p.y)), fmul(pose[8], p.z)), pose[11]);
}

// distance window, viewing cosine, predicted level
__device__ __forceinline__ bool distance_scale(const DevParams &P, const float *O, float4 pos,
                                               float4 nrm, float &vc, int &level)
{
    const float px = fsub(pos.x, O[0]), py = fsub(pos.y, O[1]), pz = fsub(pos.z, O[2]);
    const float dist = fsqrt(fadd(fadd(fmul(px, px), fmul(py, py)), fmul(pz, pz)));
    const float d_far = fmul(P.dist_hi, nrm.w);
    const float d_near = fmul(P.dist_lo, pos.w);
    if (dist < d_near || dist > d_far) return false;
    vc = fdiv(fadd(fadd(fmul(px, nrm.x), fmul(py, nrm.y)), fmul(pz, nrm.z)), dist);
    if (vc < P.view_cos_min) return false;
    const float ratio = fdiv(nrm.w, dist);
    level = P.nlevels - 1;
    for (int l = 0; l < P.nlevels; ++l) {
        if (P.sc[l] >= ratio) {
            level = l;
            break;
        }
    }
    return true;
}

// a8 without the distance and viewing tests: camera z > 0 and the
// projection inside the image bounds
__device__ bool project_uv(const CamDev &C, const float *pose, float4 pos, float &u, float &v, float &ur)
{
    float x, y, z;
    transform(pose, pos, x, y, z);
    if (!(z > 0.0f)) return false;
    if (C.model == FT_CAMERA_PINHOLE) {
        const float invz = fdiv(1.0f, z);
        u = fadd(fmul(fmul(C.fx, x), invz), C.cx);
        v = fadd(fmul(fmul(C.fy, y), invz), C.cy);
        if (u < C.minx || u > C.maxx) return false;
        if (v < C.miny || v > C.maxy) return false;
        ur = fsub(u, fmul(C.bf, invz));
    } else {
        const float rho = fsqrt(fadd(fmul(x, x), fmul(y, y)));
        if (rho == 0.0f) {
            u = C.cx;
            v = C.cy;
        } else {
            const float theta = atan2_pos(rho, z);
            const float t2 = fmul(theta, theta);
            float poly = C.k[3];
            poly = fadd(C.k[2], fmul(t2, poly));
            poly = fadd(C.k[1], fmul(t2, poly));
            poly = fadd(C.k[0], fmul(t2, poly));
            poly = fadd(1.0f, fmul(t2, poly));
            const float thetad = fmul(theta, poly);
            u = fadd(fdiv(fmul(fmul(C.fx, thetad), x), rho), C.cx);
            v = fadd(fdiv(fmul(fmul(C.fy, thetad), y), rho), C.cy);
        }
        if (u < C.minx || u > C.maxx) return false;
        if (v < C.miny || v > C.maxy) return false;
        ur = -1.0f;
    }
    return true;
}

__device__ bool project(const DevParams &P, const CamDev &C, const float *pose, float4 pos,
                        float4 nrm, float &u, float &v, float &ur, float &vc, int &level)
{
    return project_uv(C, pose, pos, u, v, ur) && distance_scale(P, C.O, pos, nrm, vc, level);
}

// The search of one map point, as its lane holds it: the projection, the
// radius and the window of grid cells (active: the point is in view and its
// window meets the grid), the same window in packed places (widened by a
// place, so that it keeps every keypoint the exact test keeps) and the
// octaves searched (bit o).
struct PointWindow {
    bool active;
    int level, x0, x1, y0, y1;
    unsigned lo, hi, octs;
    float u, v, ur, vc, r;
};

// motion: for a last-frame search, +1 / -1 / 0 for a camera that moved
// forward / backward / neither along its viewing axis (f2).
__device__ __forceinline__ PointWindow point_window(const DevParams &P, const FrameDev &F, const CamDev &C,
                                                    const SmemSearch &Q, int m)
{
    const float *pose = Q.pose;
    const PlaceScale &ps = Q.ps;
    const float iw = Q.iw, ih = Q.ih;
    const int motion = Q.motion;
    PointWindow W;
    W.active = false;
    W.level = -1;
    W.u = W.v = W.ur = W.vc = W.r = 0.0f;
    W.x0 = W.x1 = W.y0 = W.y1 = 0;
    W.lo = W.hi = W.octs = 0u;
    const bool last = F.search_mode != 0;
    const int loct = last ? (int)__ldg(F.last_oct + m) : 0;
    const bool skipped = F.skip != nullptr && __ldg(F.skip + m) != 0;
    const float4 pos = __ldg(F.pos + m);
    const float4 nrm = last ? pos : __ldg(F.nrm + m);
    if (skipped || (last && (loct < 0 || loct >= P.nlevels))) return W;
    float u, v, ur, vc = 0.0f;
    int level = loct;
    const bool in_view = last ? project_uv(C, pose, pos, u, v, ur)
                              : project(P, C, pose, pos, nrm, u, v, ur, vc, level);
    if (!in_view) return W;
    W.level = level;
    W.u = u;
    W.v = v;
    W.ur = ur;
    W.vc = vc;
    float r;
    int min_oct = level - 1, max_oct = level;
    if (last) {
        // f2: radius of the last octave, octave window by the motion
        r = fmul(P.th_last, P.sc[level]);
        min_oct = motion > 0 ? level : (motion < 0 ? 0 : level - 1);
        max_oct = motion > 0 ? P.nlevels - 1 : (motion < 0 ? level : level + 1);
    } else {
        r = (vc > P.view_cos_narrow) ? P.radius_narrow : P.radius_wide;
        r = fmul(r, P.search_th);
        r = fmul(r, P.sc[level]);
    }
    W.r = r;
    const float du = fsub(u, C.minx), dv = fsub(v, C.miny);
    W.x0 = max(f2i(floorf(fmul(fsub(du, r), iw))), 0);
    W.x1 = min(f2i(ceilf(fmul(fadd(du, r), iw))), FT_GRID_COLS - 1);
    W.y0 = max(f2i(floorf(fmul(fsub(dv, r), ih))), 0);
    W.y1 = min(f2i(ceilf(fmul(fadd(dv, r), ih))), FT_GRID_ROWS - 1);
    W.active = !(W.x0 >= FT_GRID_COLS || W.x1 < 0 || W.y0 >= FT_GRID_ROWS || W.y1 < 0);
    const float pu = fsub(u, ps.x0), pv = fsub(v, ps.y0);
    W.lo = place_of(fsub(fmul(fsub(pu, r), ps.sx), 1.0f), kPlaceX) |
           place_of(fsub(fmul(fsub(pv, r), ps.sy), 1.0f), kPlaceY) << 16;
    W.hi = place_of(fadd(fmul(fadd(pu, r), ps.sx), 1.0f), kPlaceX) |
           place_of(fadd(fmul(fadd(pv, r), ps.sy), 1.0f), kPlaceY) << 16;
    W.octs = (0xffffu >> (15 - clampi(max_oct, 0, 15))) & ~((1u << clampi(min_oct, 0, 15)) - 1u);
    return W;
}

// The staged part of the grid: keypoints [e0, e0 + kGridStage) in cell order,
// which is all of them for a camera of up to kGridStage keypoints (8528);
// cell starts are relative to e0 and clamped to the part.
__device__ __forceinline__ int grid_start(const SmemSearch &Q, int c)
{
    return (int)reinterpret_cast<const uint16_t *>(Q.buf)[c];
}
__device__ __forceinline__ const unsigned *grid_places(const SmemSearch &Q)
{
    return reinterpret_cast<const unsigned *>(Q.buf) + kCell16Bytes / 4;
}
__device__ __forceinline__ int grid_index(const CamDev &C, const SmemSearch &Q, int n, int e)
{
    if (Q.wide) return __ldcg(C.gk32 + Q.e0 + e);
    return (int)reinterpret_cast<const uint16_t *>(grid_places(Q) + n)[e];
}

// entries of a staged part, rounded up to whole 16-byte chunks of indices
__device__ __forceinline__ int grid_part(const CamDev &C) { return min((C.nk + 7) & ~7, kGridStage); }

// Copies part `part` of a camera's grid on chip (the caller synchronizes).
// Every chunk read lies inside the arrays, whose sizes are whole chunks.
__device__ void stage_grid(const CamDev &C, SmemSearch &Q, int part)
{
    const int tid = threadIdx.x;
    const int e0 = part * kGridStage, n = grid_part(C);
    const int have = min(n, ((C.nk + 7) & ~7) - e0);         // entries of this part
    unsigned char *buf = reinterpret_cast<unsigned char *>(Q.buf);
    auto copy = [&](unsigned char *dst, const void *src, int bytes) {
        for (int c = 16 * tid; c < bytes; c += 16 * kThreads)
            cp_async16(dst + c, reinterpret_cast<const unsigned char *>(src) + c);
    };
    copy(buf + kCell16Bytes, C.gq + e0, 4 * have);
    if (C.gk16) copy(buf + kCell16Bytes + 4 * n, C.gk16 + e0, 2 * have);
    uint16_t *start = reinterpret_cast<uint16_t *>(buf);
    for (int c = 4 * tid; c < kCells; c += 4 * kThreads) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(C.cell_ptr + c));
        const unsigned a = (unsigned)clampi(v.x - e0, 0, n) | (unsigned)clampi(v.y - e0, 0, n) << 16;
        const unsigned b = (unsigned)clampi(v.z - e0, 0, n) | (unsigned)clampi(v.w - e0, 0, n) << 16;
        *reinterpret_cast<uint2 *>(start + c) = make_uint2(a, b);
    }
    if (tid == 0) {
        start[kCells] = (uint16_t)clampi(__ldcg(C.cell_ptr + kCells) - e0, 0, n);
        Q.e0 = e0;
        Q.wide = C.gk16 == nullptr;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// A warp's 32 map points (point mw + lane in lane `lane`) against the
// keypoints of their windows.  Each lane walks the cell rows of its own point
// and applies the first test (packed place and octave: one shared-memory
// word a candidate, four in flight; 19 in 20 fail), listing what passes.  The
// warp's listed candidates are then shared out over its lanes, whichever
// point they belong to, and get the exact tests and the Hamming distance
// from the frame's own arrays, all their loads in flight at once; then each
// lane takes its own point's keys (distance << 20 | keypoint) and keeps the
// four smallest and their number.  What bounds it is latency: a point has one
// or two candidates behind the first test, so comparing them lane by lane as
// they are found leaves most lanes idle and pays a round trip for each
// (1280x720, 4000 keypoints, 20000 points: 13 us a point and thread that
// way; 7 us with the candidates voted into the pool one step at a time).
// check_ur: the stereo consistency is among the tests (the first half of a
// search split around the stereo step leaves it out).
__device__ __forceinline__ void gather(const FrameDev &F, const CamDev &C, SmemSearch &Q, const PointWindow &W, int mw,
                                       bool check_ur, unsigned (&sk)[4], unsigned &count)
{
    const int lane = threadIdx.x & 31;
    unsigned *const list = &Q.list[threadIdx.x >> 5][0][lane], *const pool = Q.pool[threadIdx.x >> 5];
    const unsigned *const places = grid_places(Q);
    const int part = grid_part(C);
    bool active = W.active;
    int cy = W.y0, e = 0, e1 = 0;
    if (active) {
        e = grid_start(Q, cy * FT_GRID_COLS + W.x0);
        e1 = grid_start(Q, cy * FT_GRID_COLS + W.x1 + 1);
    }
    do {
        int n = 0;
        while (active && n <= kList - kStep) {
            if (e >= e1) {
                if (cy < W.y1) {
                    ++cy;
                    e = grid_start(Q, cy * FT_GRID_COLS + W.x0);
                    e1 = grid_start(Q, cy * FT_GRID_COLS + W.x1 + 1);
                } else {
                    active = false;
                }
            }
            unsigned w[kStep];
#pragma unroll
            for (int s = 0; s < kStep; ++s) w[s] = e + s < e1 ? places[e + s] : 0u;
#pragma unroll
            for (int s = 0; s < kStep; ++s) {
                const unsigned place = w[s] & 0x0fff3fffu;
                const bool pass = e + s < e1 & __vminu2(__vmaxu2(place, W.lo), W.hi) == place &
                                  ((W.octs >> (w[s] >> 28)) & 1u);
                list[32 * n] = (unsigned)(e + s) | ((unsigned)lane << 20);   // kept if it passes
                n += pass;
            }
            e += kStep;
        }
        __syncwarp();
        int end = n;                    // of this lane's candidates in the pool
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(kFull, end, d);
            if (lane >= d) end += t;
        }
        const int total = __shfl_sync(kFull, end, 31);
        for (int i = 0; i < n; ++i) pool[end - n + i] = list[32 * i];
        __syncwarp();
        for (int p = lane; p - lane < total; p += 32) {
            const bool have = p < total;
            const unsigned ent = have ? pool[p] : 0u;
            const int o = (int)(ent >> 20);
            const float uo = __shfl_sync(kFull, W.u, o), vo = __shfl_sync(kFull, W.v, o);
            const float ro = __shfl_sync(kFull, W.r, o), uro = __shfl_sync(kFull, W.ur, o);
            if (!have) continue;
            const int k = grid_index(C, Q, part, (int)(ent & 0xfffffu));
            const float x = __ldg(C.kx + k), y = __ldg(C.ky + k);
            const float w1 = check_ur ? __ldcg(F.u_right_in + k) : -1.0f;
            const uint4 b0 = __ldg(C.kdesc + 2 * k), b1 = __ldg(C.kdesc + 2 * k + 1);
            const uint4 q0 = __ldg(F.mdesc + 2 * (size_t)(mw + o)), q1 = __ldg(F.mdesc + 2 * (size_t)(mw + o) + 1);
            bool ok = fabsf(fsub(x, uo)) < ro && fabsf(fsub(y, vo)) < ro;
            if (w1 > 0.0f && fabsf(fsub(uro, w1)) > ro) ok = false;
            pool[p] = ok ? ((unsigned)ham8(q0, q1, b0, b1) << 20) | (unsigned)k : kNoKey;
        }
        __syncwarp();
        for (int p = end - n; p < end; ++p) {
            unsigned key = pool[p];
            count += key != kNoKey;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned lo = min(sk[q], key);
                key = max(sk[q], key);
                sk[q] = lo;
            }
        }
    } while (__any_sync(kFull, active));
}

// The top-2 rules (threshold, ratio test) on a point's two smallest keys, the
// claim of the keypoint, and the point's outputs.
__device__ __forceinline__ void claim_point(const DevParams &P, const FrameDev &F, const CamDev &C, int m,
                                            unsigned best, unsigned second)
{
    int d1 = -1, d2 = -1, kp = -1;
    if (best != kNoKey) {
        d1 = (int)(best >> 20);
        d2 = second != kNoKey ? (int)(second >> 20) : 256;
        if (d1 <= P.th_search) {
            const int k1 = (int)(best & 0xfffffu);
            bool ratio = F.search_mode == 0;
            if (ratio && !P.ratio_any_octave) {
                // the ratio test applies if both share an octave
                const int o1 = __ldg(C.koct + k1);
                const int o2 = second != kNoKey ? (int)__ldg(C.koct + (second & 0xfffffu)) : -1;
                ratio = o1 == o2;
            }
            if (!(ratio && (float)d1 > fmul(P.nn_ratio, (float)d2))) {
                atomicMin(C.owner + k1, ((unsigned long long)d1 << 32) | (unsigned)m);
                kp = k1;
            }
        }
    }
    C.mp_d1[m] = d1;
    C.mp_d2[m] = d2;
    C.mp_kp[m] = kp;
}

// How a search item passes over its points: the whole search; the first half
// of a search split around the stereo step (each point's four smallest keys,
// their number and the projection's right coordinate and radius go to its
// record); or the whole search of the points that the second half left.
enum SearchPass { kWhole, kFirstHalf, kLeftOver };

// Map points [m0, m1), 32 a warp at a time; scan: their records (2 a point).
__device__ __forceinline__ void search_points(const DevParams &P, const FrameDev &F, const CamDev &C, SmemSearch &Q,
                                              uint4 *scan, int m0, int m1, SearchPass pass)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool check_ur = pass != kFirstHalf && C.model == FT_CAMERA_PINHOLE && F.u_right_in != nullptr;
    // a grid of several parts is staged part by part for every 256 points (all
    // warps take part in each)
    const int parts = (C.nk + kGridStage - 1) / kGridStage;
    for (int mb = m0; mb < m1; mb += kThreads) {
        const int mw = mb + 32 * warp, m = mw + lane;
        if (parts <= 1 && mw >= m1) break;
        const bool mine = m < m1 && (pass != kLeftOver || scan[2 * (m - m0) + 1].w != 0u);
        PointWindow W;
        W.active = false;
        if (mine) {
            W = point_window(P, F, C, Q, m);
            C.level[m] = (int8_t)W.level;
            if (C.proj) C.proj[m] = make_float4(W.u, W.v, W.ur, W.vc);
        }
        unsigned sk[4] = {kNoKey, kNoKey, kNoKey, kNoKey}, count = 0;
        for (int part = 0; part < parts; ++part) {
            if (parts > 1) {
                __syncthreads();
                stage_grid(C, Q, part);
                __syncthreads();
            }
            __syncwarp();
            gather(F, C, Q, W, mw, check_ur, sk, count);
        }
        if (!mine) continue;
        if (pass == kFirstHalf) {
            scan[2 * (m - m0)] = make_uint4(sk[0], sk[1], sk[2], sk[3]);
            scan[2 * (m - m0) + 1] = make_uint4(__float_as_uint(W.ur), __float_as_uint(W.r), count, 0u);
        } else {
            claim_point(P, F, C, m, sk[0], sk[1]);
        }
    }
}

// The second half of a split search, after the stereo step: the stereo
// consistency applied to each point's four smallest candidates, then the
// top-2 rules and the claim, exactly as the unsplit search takes them.  The
// consistency test drops candidates and keys are unique, so the two smallest
// consistent keys among the four smallest candidates are the two smallest
// consistent candidates, unless fewer than two of the four are consistent
// while more than four passed: only those points are left to be searched
// again, with the consistency among the tests (true: there are some).
__device__ __forceinline__ bool finish_points(const DevParams &P, const FrameDev &F, const CamDev &C, uint4 *scan,
                                              int m0, int m1)
{
    const bool check_ur = C.model == FT_CAMERA_PINHOLE && F.u_right_in != nullptr;
    bool left = false;
    for (int m = m0 + (int)threadIdx.x; m < m1; m += kThreads) {
        const uint4 ks = scan[2 * (m - m0)], aux = scan[2 * (m - m0) + 1];
        const unsigned sk[4] = {ks.x, ks.y, ks.z, ks.w};
        const float ur = __uint_as_float(aux.x), r = __uint_as_float(aux.y);
        unsigned best = kNoKey, second = kNoKey;
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            w[q] = check_ur && sk[q] != kNoKey ? __ldcg(F.u_right_in + (sk[q] & 0xfffffu)) : -1.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (sk[q] == kNoKey || (w[q] > 0.0f && fabsf(fsub(ur, w[q])) > r)) continue;
            if (best == kNoKey) best = sk[q];
            else if (second == kNoKey) second = sk[q];
        }
        if (aux.z > 4u && second == kNoKey) {
            scan[2 * (m - m0) + 1].w = 1u;
            left = true;
        } else {
            claim_point(P, F, C, m, best, second);
        }
    }
    return left;
}

// The camera pose of a search item in shared memory (the right fisheye
// camera's composed from the rig), the grid scales and the last-frame motion.
__device__ void search_setup(const FrameDev &F, int cam, SmemSearch &Q)
{
    const CamDev &C = F.cam[cam];
    const int tid = threadIdx.x;
    if (tid < 12) {
        const CamDev &L = F.cam[0];
        float v;
        if (cam == 0 || F.camera == FT_CAMERA_PINHOLE) {
            v = tid < 9 ? L.R[tid] : L.t[tid - 9];
        } else if (tid < 9) {      // right camera: R_rw = R_rl * R_lw
            const int i = tid / 3, j = tid % 3;
            v = fadd(fadd(fmul(F.R_rl[3 * i], L.R[j]), fmul(F.R_rl[3 * i + 1], L.R[3 + j])),
                     fmul(F.R_rl[3 * i + 2], L.R[6 + j]));
        } else {                   // t_rw = R_rl * t_lw + t_rl
            const int i = tid - 9;
            v = fadd(fadd(fadd(fmul(F.R_rl[3 * i], L.t[0]), fmul(F.R_rl[3 * i + 1], L.t[1])),
                          fmul(F.R_rl[3 * i + 2], L.t[2])),
                     F.t_rl[i]);
        }
        Q.pose[tid] = v;
    }
    if (tid == 32) {
        Q.iw = fdiv((float)FT_GRID_COLS, fsub(C.maxx, C.minx));
        Q.ih = fdiv((float)FT_GRID_ROWS, fsub(C.maxy, C.miny));
        Q.ps = place_scale(C);
        Q.motion = 0;
        if (F.search_mode != 0) {
            // the current (left) camera centre in the last frame's camera
            // coordinates; its z against the baseline (f2)
            const float *O = F.cam[0].O;
            const float cz = fadd(fadd(fadd(fmul(F.last_R[6], O[0]), fmul(F.last_R[7], O[1])),
                                       fmul(F.last_R[8], O[2])),
                                  F.last_t[2]);
            Q.motion = cz > F.base ? 1 : (-cz > F.base ? -1 : 0);
        }
    }
}

// Defined outputs of map points [m0, m1) after a wait ran out (reported in
// the status word).
__device__ void search_abandon(const CamDev &C, int m0, int m1)
{
    for (int m = m0 + (int)threadIdx.x; m < m1; m += kThreads) {
        C.level[m] = -1;
        if (C.proj) C.proj[m] = make_float4(0.f, 0.f, 0.f, 0.f);
        C.mp_d1[m] = -1;
        C.mp_d2[m] = -1;
        C.mp_kp[m] = -1;
    }
}

// A tile of map points.  A frame whose search is split around its stereo
// step (split_search) runs the first half of every point without waiting
// for the stereo step, then waits for it and finishes the points: the first
// half overlaps the wait.
__device__ void search_item(const BatchHeader &B, const FrameDev &F, int tile, Smem &U, int *s_flag)
{
    const int cam = tile < F.n_search_items[0] ? 0 : 1;
    const int t = cam ? tile - F.n_search_items[0] : tile;
    const bool split = F.split_search != 0;
    const int m0 = t * F.search_tile;
    const int m1 = min(F.nm, m0 + F.search_tile);
    // the tile's map point records do not depend on the stereo step: ask L2
    // for them before waiting for it
    for (int m = m0 + (int)threadIdx.x; m < m1; m += kThreads) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(F.pos + m));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(F.mdesc + 2 * m));
        if (F.search_mode == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(F.nrm + m));
    }
    bool ok = true;
    if (F.wait_stereo && !split) ok = wait_geq(B, &F.ctr[C_STEREO_READY], 1u, s_flag);
    if (ok) ok = wait_geq(B, &F.ctr[C_GRID_DONE], (unsigned)F.n_grid_items, s_flag);
    const CamDev &C = F.cam[cam];
    if (ok) {
        SmemSearch &Q = U.q;
        search_setup(F, cam, Q);
        if (C.nk <= kGridStage) stage_grid(C, Q, 0);
        __syncthreads();
        mark(B, 0);
        // a split search runs its first halves (the right coordinates are not
        // read: they may not be final yet), then waits for the stereo step,
        // then runs the second halves; each thread finishes the points it
        // scanned, whose records stay on chip when they fit behind the grid
        const int used = kCell16Bytes + 6 * grid_part(C);
        uint4 *scan = used + 32 * (m1 - m0) <= kSearchBuf ? reinterpret_cast<uint4 *>(reinterpret_cast<char *>(Q.buf) + used)
                                                          : C.scan + 2 * (size_t)m0;
        SearchPass pass = split ? kFirstHalf : kWhole;
        for (;;) {
            search_points(B.p, F, C, Q, scan, m0, m1, pass);
            mark(B, 1);
            if (pass != kFirstHalf) break;
            if (!wait_geq(B, &F.ctr[C_STEREO_READY], 1u, s_flag)) {
                search_abandon(C, m0, m1);
                break;
            }
            const bool left = finish_points(B.p, F, C, scan, m0, m1);
            mark(B, 2);
            if (!__syncthreads_or(left)) break;
            pass = kLeftOver;
        }
    } else {
        search_abandon(C, m0, m1);
    }
    if (signal_count(&F.ctr[C_SEARCH_DONE0 + cam], (unsigned)F.n_search_items[cam], s_flag) &&
        F.fold_resolve) {
        // the last search item of this camera also writes the final tables
        // (small frames: no separate resolve items wait for the search)
        resolve_range(F.cam[cam], F.nm, 0, max(F.nm, F.cam[cam].nk));
    }
}

// ---------------------------------------------------------------- K_RESOLVE
// Final tables for entries [i0, i1): a map point keeps its keypoint only if
// it owns it; a keypoint gets its owner (or -1).  A thread takes kResolveBatch
// entries at a time and issues all their loads before any store, so a
// range's dependent reads (map point -> keypoint -> owner) cost two L2 round
// trips per batch rather than per entry.
constexpr int kResolveBatch = 8;

__device__ void resolve_range(const CamDev &C, int nm, int i0, int i1)
{
    const int me = min(i1, nm), ke = min(i1, C.nk);
    for (int m0 = i0 + (int)threadIdx.x; m0 < me; m0 += kThreads * kResolveBatch) {
        int kk[kResolveBatch];
#pragma unroll
        for (int u = 0; u < kResolveBatch; ++u) {
            const int m = m0 + u * kThreads;
            kk[u] = m < me ? __ldcg(C.mp_kp + m) : -1;
        }
        unsigned own[kResolveBatch];
#pragma unroll
        for (int u = 0; u < kResolveBatch; ++u)
            own[u] = kk[u] >= 0 && kk[u] < C.nk ? (unsigned)(__ldcg(C.owner + kk[u]) & 0xffffffffull) : 0u;
#pragma unroll
        for (int u = 0; u < kResolveBatch; ++u) {
            const int m = m0 + u * kThreads;
            if (m >= me || kk[u] < 0) continue;
            if (kk[u] >= C.nk || own[u] != (unsigned)m) C.mp_kp[m] = -1;   // never written / not the owner
        }
    }
    for (int k0 = i0 + (int)threadIdx.x; k0 < ke; k0 += kThreads * kResolveBatch) {
        unsigned long long own[kResolveBatch];
#pragma unroll
        for (int u = 0; u < kResolveBatch; ++u) {
            const int k = k0 + u * kThreads;
            own[u] = k < ke ? __ldcg(C.owner + k) : ~0ull;
        }
#pragma unroll
        for (int u = 0; u < kResolveBatch; ++u) {
            const int k = k0 + u * kThreads;
            if (k < ke) C.kp_mp[k] = own[u] == ~0ull ? -1 : (int)(own[u] & 0xffffffffull);
        }
    }
}

__device__ void resolve_item(const BatchHeader &B, const FrameDev &F, int tile, int *s_flag)
{
    const int cam = tile < F.n_resolve_items[0] ? 0 : 1;
    const int t = cam ? tile - F.n_resolve_items[0] : tile;
    // the grid build initialises the owners (a frame without map points has no
    // search item to order the two)
    const CamDev &C = F.cam[cam];
    const int i0 = t * F.resolve_tile, i1 = i0 + F.resolve_tile;
    if (!wait_geq(B, &F.ctr[C_GRID_DONE], (unsigned)F.n_grid_items, s_flag) ||
        !wait_geq(B, &F.ctr[C_SEARCH_DONE0 + cam], (unsigned)F.n_search_items[cam], s_flag)) {
        // the wait ran out (reported in the status word): leave defined outputs
        for (int m = i0 + threadIdx.x; m < min(i1, F.nm); m += kThreads) C.mp_kp[m] = -1;
        for (int k = i0 + threadIdx.x; k < min(i1, C.nk); k += kThreads) C.kp_mp[k] = -1;
        return;
    }
    resolve_range(C, F.nm, i0, i1);
}

// ---------------------------------------------------------------- the kernel
__device__ __forceinline__ void copy_words(void *dst, const void *src, size_t bytes)
{
    const unsigned *a = reinterpret_cast<const unsigned *>(src);
    unsigned *b = reinterpret_cast<unsigned *>(dst);
    for (size_t i = threadIdx.x; i < bytes / 4; i += kThreads) b[i] = __ldg(a + i);
}

// Words of a kernel parameter (not global memory).
__device__ __forceinline__ void copy_param(void *dst, const void *src, size_t bytes)
{
    const unsigned *a = reinterpret_cast<const unsigned *>(src);
    unsigned *b = reinterpret_cast<unsigned *>(dst);
    for (size_t i = threadIdx.x; i < bytes / 4; i += blockDim.x) b[i] = a[i];
}

// The persistent loop over the batch table at hdr, or (kOne) over the single
// frame of a call whose header hdr and descriptor one are kernel parameters.
template <bool kOne>
__device__ __forceinline__ void fused_run(const BatchHeader *hdr, const FrameDev *one)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    __shared__ int s_flag;
    // the launch header and the current frame's descriptor live in shared
    // memory: their many indexed fields (level sizes, pitches, scales) are
    // then shared-memory loads instead of dependent global loads
    __shared__ __align__(16) BatchHeader sB;
    __shared__ __align__(16) FrameDev sF;
    let_next_start();
    if (kOne) {
        copy_param(&sB, hdr, sizeof(BatchHeader));
        copy_param(&sF, one, sizeof(FrameDev));
    } else {
        copy_words(&sB, hdr, sizeof(BatchHeader));
    }
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(sB.queue, 1u);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= sB.total_items) break;
        // zero (items are not negative), which the compiler does not know: the
        // roles' addresses then depend on the item, and their arithmetic is not
        // hoisted out of this loop, all roles' at once, and spilled
        const unsigned zero = (unsigned)item >> 31;
        const BatchHeader &B = *reinterpret_cast<const BatchHeader *>(reinterpret_cast<const char *>(&sB) + 16 * zero);
        Smem &U = *reinterpret_cast<Smem *>(smem_raw + 16 * zero);
        int kind = 0;
        while (kind < K_KINDS - 1 && item >= B.kind_begin[kind + 1]) ++kind;
        const int local = item - B.kind_begin[kind];
        int lo = 0, first = 0;                   // the item's frame, and its first item of the kind
        if (!kOne) {
            const int *pre = B.prefix + kind * (B.nframes + 1);
            int hi = B.nframes - 1;              // last frame f with pre[f] <= local
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (pre[mid] <= local) lo = mid;
                else hi = mid - 1;
            }
            first = pre[lo];
            copy_words(&sF, B.frames + lo, sizeof(FrameDev));
            __syncthreads();
        }
        const FrameDev &F = *reinterpret_cast<const FrameDev *>(reinterpret_cast<const char *>(&sF) + 16 * zero);
        const int tile = local - first;
        unsigned long long t_start = 0;
        if (B.trace != nullptr && threadIdx.x == 0) {
            t_start = global_ns();
            s_wait_ns = 0;
            s_mark[0] = s_mark[1] = s_mark[2] = s_mark[3] = 0;
        }
        switch (kind) {
        case K_INDEX:
            if (tile < F.rowsort) {
                rowsort_item(B, F, U.r, tile >= kSortParts, tile % kSortParts, &s_flag);
            } else {
                grid_item(B, F, tile - F.rowsort, U.g, &s_flag);
            }
            break;
        case K_STEREO:
            stereo_pinhole_item(B, F, tile, U, &s_flag);
            break;
        case K_SEARCH: search_item(B, F, tile, U, &s_flag); break;
        default: resolve_item(B, F, tile, &s_flag); break;
        }
        if (B.trace != nullptr && threadIdx.x == 0) {
            const unsigned slot = atomicAdd(B.queue + 1, 1u);
            if (slot < (unsigned)B.trace_cap) {
                unsigned sm;
                asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
                ft_trace_record r;
                r.item = item;
                r.kind = kind;
                r.frame = lo;
                r.sm = (int)sm;
                r.t_start = t_start;
                r.t_end = global_ns();
                r.wait_ns = s_wait_ns;
                for (int q = 0; q < 4; ++q) r.mark[q] = s_mark[q];
                B.trace[slot] = r;
            }
        }
    }
    wait_for_previous();
    if (kOne && threadIdx.x == 0) {
        // the last block of the launch leaves the queue and the counters zero
        __threadfence();
        if (atomicAdd(sB.queue + 2, 1u) == gridDim.x - 1) {
            sB.queue[0] = sB.queue[2] = 0u;
            for (int c = 0; c < kCounters; ++c) sF.ctr[c] = 0u;
        }
    }
}

__global__ void __launch_bounds__(kThreads, FT_MIN_CTAS_PER_SM) ft_fused_kernel(const BatchHeader *__restrict__ hdr)
{
    fused_run<false>(hdr, nullptr);
}

__global__ void __launch_bounds__(kThreads, FT_MIN_CTAS_PER_SM) ft_fused_one_kernel(const __grid_constant__ FrameCall call)
{
    fused_run<true>(&call.h, &call.f);
}

}  // namespace

// ---------------------------------------------------------------- f4: pose optimization
// The refinement of the camera pose with all the map points the search found
// in the frame (paper section II-D; FastTrack switches it off, section
// IV-F), as the algorithm family's motion-only optimization (a reading):
// observations are the matched keypoints (x, y) and, where stereo gave one,
// u_right; weight 1/scale[oct]^2; po_rounds rounds of po_iters Gauss-Newton
// steps over the inliers with Huber weights, the update exp(d) multiplied on
// the left of the pose; every observation reclassified by its chi2 after
// each round.  FP32.  A kernel of its own, after the fused kernel on the
// same stream (the matches are final by then).
//
// What bounds it is the serial chain of a frame's Gauss-Newton steps (up to
// 40), so one frame gets a cluster of kPoseCtas blocks with one warp per
// scheduler instead of one block with four: 512 threads on one SM spent half
// of a 3.2 us step issuing the observations' 27 sums.  Every block keeps its
// threads' observations on chip; each warp reduce-scatters its 27 sums (lane q
// ends with sum q) and writes them to all blocks' shared
// memory, one cluster barrier makes them visible, and then every warp adds
// the 16 warps' sums in the same order and solves the 6x6 system itself, so
// nothing is broadcast back.  The additions are those of one 512-thread block
// in the same order, and a pose that repeats ends a round early (it fixes the
// round's remaining steps), so the results are the same bit for bit.  A step
// now spends 2200 cycles on three observations per thread, 250 on the
// reduction, 600 on the barrier and 1300 on the solve.  One frame of 1100
// matches: 135 us a call before, 80 to 95 us now by the steps its data needs
// (the call's table no longer travels ahead of it); 16 frames' share 116 -> 85 us.
namespace {

constexpr int kPoseLanes = 512;                       // threads of a frame, over all its blocks
constexpr int kPoseCtas = 4;                          // blocks of a frame (one cluster)
constexpr int kPoseThreads = kPoseLanes / kPoseCtas;
constexpr int kPoseWarps = kPoseLanes / 32;           // of a frame
constexpr int kPoseStage = 8192;                      // observations of a frame kept on chip
constexpr int kPoseSlots = kPoseStage / kPoseCtas;    // of a block
constexpr int kPoseSmem = 2 * kPoseSlots * (int)sizeof(float4);
constexpr int kPoseRead = 8;                          // matches a lane loads at once

struct PoseShared {
    float part[2][kPoseWarps][32];                    // every warp's sums, two steps' (written by all blocks)
    int count[2][kPoseWarps];
    alignas(16) float tot[kPoseThreads / 32][32];     // a warp's copy of the frame's sums
};

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of this block's shared-memory location p in block `rank` of the cluster
__device__ __forceinline__ unsigned remote_addr(const void *p, unsigned rank)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void remote_store(unsigned addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void remote_store(unsigned addr, int v)
{
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void remote_store(unsigned addr, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Observation (a, b) at pose Rt: residual, chi2 and Jacobian rows (rotation
// then translation of the left perturbation).  front: the point lies in
// front of the camera; if not, everything is finite and of no meaning.
struct PoseObs {
    float e[3], J[3][6], chi2;
    bool stereo, front;
};

__device__ __forceinline__ void pose_obs(const CamDev &C, const float (&Rt)[12], float4 a, float4 b, PoseObs &o)
{
    float x = Rt[0] * a.x + Rt[1] * a.y + Rt[2] * a.z + Rt[9];
    float y = Rt[3] * a.x + Rt[4] * a.y + Rt[5] * a.z + Rt[10];
    float z = Rt[6] * a.x + Rt[7] * a.y + Rt[8] * a.z + Rt[11];
    o.front = z > 0.0f;
    if (!o.front) {
        x = y = 0.0f;
        z = 1.0f;
    }
    const float iz = rn_range(z) ? rn_rcp(z) : 1.0f / z, iz2 = iz * iz;
    const float u = C.fx * x * iz + C.cx, v = C.fy * y * iz + C.cy;
    o.stereo = b.z >= 0.0f;
    o.e[0] = b.x - u;
    o.e[1] = b.y - v;
    o.e[2] = o.stereo ? b.z - (u - C.bf * iz) : 0.0f;
    o.chi2 = a.w * (o.e[0] * o.e[0] + o.e[1] * o.e[1] + o.e[2] * o.e[2]);
    // d projection / d Pc, times d Pc / d (w, v) = [ -[Pc]x | I ]
    const float D[3][3] = {{C.fx * iz, 0.0f, -C.fx * x * iz2},
                           {0.0f, C.fy * iz, -C.fy * y * iz2},
                           {C.fx * iz, 0.0f, -C.fx * x * iz2 + C.bf * iz2}};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        o.J[r][0] = -D[r][1] * z + D[r][2] * y;
        o.J[r][1] = D[r][0] * z - D[r][2] * x;
        o.J[r][2] = -D[r][0] * y + D[r][1] * x;
        o.J[r][3] = D[r][0];
        o.J[r][4] = D[r][1];
        o.J[r][5] = D[r][2];
    }
}

// Adds hw J^T J (upper triangle, 21) and hw J^T e (6) of one Jacobian row
// whose column kZero is zero for every observation (the y translation of the
// u rows, the x translation of the v row).
template <int kZero>
__device__ __forceinline__ void pose_row(float (&acc)[32], const float (&J)[6], float hw, float e)
{
    int q = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float wi = hw * J[i];
#pragma unroll
        for (int j = i; j < 6; ++j, ++q)
            if (i != kZero && j != kZero) acc[q] += wi * J[j];
        if (i != kZero) acc[21 + i] += wi * e;
    }
}

// Solve H d = g (H as its upper triangle, row by row, in tot[0..20], g in
// tot[21..26]) by Cholesky with one reciprocal per column, then (R, t) <-
// exp(d) (R, t); false if H is not positive definite.
__device__ __forceinline__ bool pose_step(const float *tot, float (&Rt)[12])
{
    float H[6][6], L[6][6], inv[6], y[6], d[6];
    float t[28];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const float4 v = reinterpret_cast<const float4 *>(tot)[k];
        t[4 * k] = v.x;
        t[4 * k + 1] = v.y;
        t[4 * k + 2] = v.z;
        t[4 * k + 3] = v.w;
    }
    int q = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = i; j < 6; ++j) H[i][j] = H[j][i] = t[q++];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        float s = H[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) s -= L[j][k] * L[j][k];
        if (!(s > 0.0f)) return false;
        if (rn_range(s)) {
            rn_sqrt_rcp(s, L[j][j], inv[j]);
        } else {
            L[j][j] = sqrtf(s);
            inv[j] = 1.0f / L[j][j];
        }
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            float t = H[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= L[i][k] * L[j][k];
            L[i][j] = t * inv[j];
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float s = t[21 + i];
#pragma unroll
        for (int k = 0; k < i; ++k) s -= L[i][k] * y[k];
        y[i] = s * inv[i];
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        float s = y[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) s -= L[k][i] * d[k];
        d[i] = s * inv[i];
    }
    // exp of the twist d = (w, v): R_d = I + a [w]x + b [w]x^2,
    // V = I + b [w]x + c [w]x^2 (series of a, b, c below theta = 0.01)
    const float th2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    float a, b, c;
    if (th2 < 1.0e-10f) {
        // the series below, whose th2 terms are less than half an ulp here
        a = 1.0f;
        b = 0.5f;
        c = 1.0f / 6.0f;
    } else {
        const float th = sqrtf(th2);
        if (th < 0.01f) {
            a = 1.0f - th2 / 6.0f;
            b = 0.5f - th2 / 24.0f;
            c = 1.0f / 6.0f - th2 / 120.0f;
        } else {
            const float sn = sinf(th), cs = cosf(th);
            a = sn / th;
            b = (1.0f - cs) / th2;
            c = (th - sn) / (th2 * th);
        }
    }
    const float W[9] = {0.0f, -d[2], d[1], d[2], 0.0f, -d[0], -d[1], d[0], 0.0f};
    float W2[9], Rd[9], V[9], Rn[12];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            W2[3 * i + j] = W[3 * i] * W[j] + W[3 * i + 1] * W[3 + j] + W[3 * i + 2] * W[6 + j];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float id = (i % 4 == 0) ? 1.0f : 0.0f;
        Rd[i] = id + a * W[i] + b * W2[i];
        V[i] = id + b * W[i] + c * W2[i];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Rn[3 * i + j] = Rd[3 * i] * Rt[j] + Rd[3 * i + 1] * Rt[3 + j] + Rd[3 * i + 2] * Rt[6 + j];
        Rn[9 + i] = Rd[3 * i] * Rt[9] + Rd[3 * i + 1] * Rt[10] + Rd[3 * i + 2] * Rt[11] +
                    V[3 * i] * d[3] + V[3 * i + 1] * d[4] + V[3 * i + 2] * d[5];
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) Rt[i] = Rn[i];
    return true;
}

__device__ __forceinline__ bool same_pose(const float (&a)[12], const float (&b)[12])
{
    bool same = true;
#pragma unroll
    for (int i = 0; i < 12; ++i) same = same && __float_as_int(a[i]) == __float_as_int(b[i]);
    return same;
}

// Sum over the frame of one int per thread (all threads get it); `slot` as
// the partial sums' (calls alternate).
__device__ int pose_sum(int v, PoseShared &S, unsigned rank, int slot)
{
    const int lane = threadIdx.x & 31, vw = (int)(rank * (kPoseThreads / 32) + (threadIdx.x >> 5));
    v = __reduce_add_sync(kFull, v);
    if (lane < kPoseCtas) remote_store(remote_addr(&S.count[slot][vw], (unsigned)lane), v);
    cluster_barrier();
    int sum = 0;
#pragma unroll
    for (int i = 0; i < kPoseWarps; ++i) sum += S.count[slot][i];
    return sum;
}

// kOne: the header and the frame are kernel parameters.
template <bool kOne>
__device__ __forceinline__ void pose_run(const BatchHeader *hdr, const FrameDev *one)
{
    extern __shared__ __align__(16) float4 pose_stage[];      // [2][kPoseSlots]: the observations' two parts
    __shared__ PoseShared S;
    __shared__ __align__(16) DevParams sP;
    __shared__ __align__(16) FrameDev sF;
    const int f = (int)blockIdx.x / kPoseCtas;
    if (!kOne && (f >= hdr->nframes || !hdr->frames[f].do_pose)) return;       // the whole cluster
    const unsigned rank = cluster_rank();
    const int tid = threadIdx.x, lane = tid & 31;
    const int vt = (int)rank * kPoseThreads + tid;            // thread of the frame
    const int vw = vt >> 5;                                   // warp of the frame
    if (kOne) {
        copy_param(&sF, one, sizeof(FrameDev));
        copy_param(&sP, &hdr->p, sizeof(DevParams));
    } else {
        const unsigned *a = reinterpret_cast<const unsigned *>(hdr->frames + f);
        unsigned *b = reinterpret_cast<unsigned *>(&sF);
        for (int i = tid; i < (int)(sizeof(FrameDev) / 4); i += kPoseThreads) b[i] = __ldg(a + i);
        const unsigned *pa = reinterpret_cast<const unsigned *>(&hdr->p);
        unsigned *pb = reinterpret_cast<unsigned *>(&sP);
        for (int i = tid; i < (int)(sizeof(DevParams) / 4); i += kPoseThreads) pb[i] = __ldg(pa + i);
    }
    __syncthreads();
    const FrameDev &F = sF;
    const DevParams &P = sP;
    const CamDev &C = F.cam[0];
    const int M = F.nm;
    float Rt[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) Rt[i] = i < 9 ? C.R[i] : C.t[i - 9];
    // observations in map-point order: each of the frame's warps takes a
    // contiguous chunk of map points, counts its matches, and writes them
    // after the chunks before it.  Observation e belongs to thread e % 512 of
    // the frame.
    const int per = ((M + kPoseWarps - 1) / kPoseWarps + 31) & ~31;
    const int m0 = min(M, vw * per), m1 = min(M, m0 + per);
    int cnt = 0;
    for (int m = m0 + lane; m < m1; m += 32 * kPoseRead) {
        int k[kPoseRead];
#pragma unroll
        for (int u = 0; u < kPoseRead; ++u) k[u] = m + 32 * u < m1 ? __ldg(F.po_mp_kp + m + 32 * u) : -1;
#pragma unroll
        for (int u = 0; u < kPoseRead; ++u) cnt += (k[u] >= 0 && k[u] < C.nk) ? 1 : 0;
    }
    cluster_barrier();                  // every block has started: its shared memory may be written
    const int total = pose_sum(cnt, S, rank, 0);
    int at = 0;                         // matches of the warps before this one
    for (int w = 0; w < vw; ++w) at += S.count[0][w];
    const bool staged = total <= kPoseStage;
    for (int mb = m0; mb < m1; mb += 32 * kPoseRead) {
        int k[kPoseRead];
        float4 a[kPoseRead], b[kPoseRead];
#pragma unroll
        for (int u = 0; u < kPoseRead; ++u) {
            const int m = mb + 32 * u + lane;
            k[u] = m < m1 ? __ldg(F.po_mp_kp + m) : -1;
            if (k[u] >= C.nk) k[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < kPoseRead; ++u) {
            if (k[u] < 0) continue;
            const int oct = __ldg(C.koct + k[u]);
            a[u] = __ldg(F.pos + mb + 32 * u + lane);
            a[u].w = (oct >= 0 && oct < P.nlevels) ? P.sc[oct] : 1.0f;
            b[u] = make_float4(__ldg(C.kx + k[u]), __ldg(C.ky + k[u]), F.u_right_in ? __ldg(F.u_right_in + k[u]) : -1.0f, 0.0f);
        }
#pragma unroll
        for (int u = 0; u < kPoseRead; ++u) {
            const int m = mb + 32 * u + lane;
            const unsigned all = __ballot_sync(kFull, k[u] >= 0);
            if (m < m1) F.po_inlier[m] = k[u] >= 0 ? 1 : -1;
            if (k[u] >= 0) {
                const int e = at + __popc(all & ((1u << lane) - 1u));
                const float sc = a[u].w;
                a[u].w = 1.0f / (sc * sc);
                if (!(b[u].z >= 0.0f)) b[u].z = -1.0f;
                b[u].w = __int_as_float(m | (int)0x80000000);
                if (staged) {
                    const int slot = e / kPoseLanes * kPoseThreads + e % kPoseThreads;
                    const unsigned owner = (unsigned)(e % kPoseLanes / kPoseThreads);
                    remote_store(remote_addr(pose_stage + slot, owner), a[u]);
                    remote_store(remote_addr(pose_stage + kPoseSlots + slot, owner), b[u]);
                } else {
                    F.po_list[2 * e] = a[u];
                    F.po_list[2 * e + 1] = b[u];
                }
            }
            at += __popc(all);
        }
    }
    cluster_barrier();
    // observation j of this thread
    auto obs_a = [&](int j) { return staged ? pose_stage[j * kPoseThreads + tid] : __ldcg(F.po_list + 2 * (j * kPoseLanes + vt)); };
    auto obs_b = [&](int j) -> float4 * {
        return staged ? pose_stage + kPoseSlots + j * kPoseThreads + tid : F.po_list + 2 * (j * kPoseLanes + vt) + 1;
    };
    const int mine = total > vt ? (total - vt + kPoseLanes - 1) / kPoseLanes : 0;
    const float th_mono = P.po_chi2_mono, th_stereo = P.po_chi2_stereo;
    int n_inliers = total, slot = 0;
    bool ok = true;
    for (int round = 0; round < P.po_rounds; ++round) {
        if (n_inliers < 3) break;
        float before[12];               // the pose two steps back
#pragma unroll
        for (int i = 0; i < 12; ++i) before[i] = Rt[i];
        for (int it = 0; it < P.po_iters; ++it) {
            float acc[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) acc[q] = 0.0f;
            for (int j = 0; j < mine; ++j) {
                const float4 a = obs_a(j), b = *obs_b(j);
                PoseObs o;
                pose_obs(C, Rt, a, b, o);
                const float th = o.stereo ? th_stereo : th_mono;
                const float h = (!P.po_huber || o.chi2 <= th) ? 1.0f : sqrtf(th / o.chi2);
                const float hw = o.front && __float_as_int(b.w) < 0 ? h * a.w : 0.0f;
                if (hw == 0.0f) continue;               // behind the camera, or an outlier
                pose_row<4>(acc, o.J[0], hw, o.e[0]);
                pose_row<3>(acc, o.J[1], hw, o.e[1]);
                if (o.stereo) pose_row<4>(acc, o.J[2], hw, o.e[2]);
            }
            // reduce-scatter: after the five butterfly stages lane q holds
            // the warp's sum of entry q
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) {
                const bool upper = (lane & s) != 0;
#pragma unroll
                for (int i = 0; i < s; ++i) {
                    const float send = upper ? acc[i] : acc[i + s];
                    const float keep = upper ? acc[i + s] : acc[i];
                    acc[i] = keep + __shfl_xor_sync(kFull, send, s);
                }
            }
            slot ^= 1;
#pragma unroll
            for (unsigned c = 0; c < (unsigned)kPoseCtas; ++c) remote_store(remote_addr(&S.part[slot][vw][lane], c), acc[0]);
            // (two steps' slots: a block that is a step ahead writes the other
            // one, and none gets further before all have read this one)
            cluster_barrier();
            float v = 0.0f;
#pragma unroll
            for (int w = 0; w < kPoseWarps; ++w) v += S.part[slot][w][lane];
            float *tot = S.tot[tid >> 5];
            __syncwarp();
            tot[lane] = v;
            __syncwarp();
            float now[12];
#pragma unroll
            for (int i = 0; i < 12; ++i) now[i] = Rt[i];
            ok = pose_step(tot, Rt);
            if (!ok) break;
            // a step depends on the pose alone: a pose that came back, from the
            // step before or two before, fixes all the round's later ones
            if (same_pose(Rt, now)) break;
            if (same_pose(Rt, before)) {
                if ((P.po_iters - 1 - it) & 1) {
#pragma unroll
                    for (int i = 0; i < 12; ++i) Rt[i] = now[i];
                }
                break;
            }
#pragma unroll
            for (int i = 0; i < 12; ++i) before[i] = now[i];
        }
        // classify every observation at the new pose
        int n_in = 0;
        for (int j = 0; j < mine; ++j) {
            float4 *pb = obs_b(j);
            const float4 b = *pb;
            PoseObs o;
            pose_obs(C, Rt, obs_a(j), b, o);
            const bool in = o.front && !(o.chi2 > (o.stereo ? th_stereo : th_mono));
            const int m = __float_as_int(b.w) & 0x7fffffff;
            pb->w = __int_as_float(in ? (m | (int)0x80000000) : m);
            n_in += in ? 1 : 0;
        }
        n_inliers = pose_sum(n_in, S, rank, 1 - (round & 1));
        if (!ok) break;
    }
    for (int j = 0; j < mine; ++j) {
        const int w = __float_as_int(obs_b(j)->w);
        F.po_inlier[w & 0x7fffffff] = w < 0 ? 1 : 0;
    }
    if (vt == 0) {
#pragma unroll
        for (int i = 0; i < 12; ++i) F.po_Rt[i] = Rt[i];
        *F.po_n = n_inliers;
    }
}

__global__ void __cluster_dims__(kPoseCtas, 1, 1) __launch_bounds__(kPoseThreads)
    ft_pose_kernel(const BatchHeader *__restrict__ hdr)
{
    pose_run<false>(hdr, nullptr);
}

__global__ void __cluster_dims__(kPoseCtas, 1, 1) __launch_bounds__(kPoseThreads)
    ft_pose_one_kernel(const __grid_constant__ FrameCall call)
{
    pose_run<true>(&call.h, &call.f);
}

}  // namespace

// A batch table's 16-byte words from mapped pinned host memory: small blocks
// without shared memory, which find room beside a running fused kernel.
__global__ void __launch_bounds__(128) ft_table_kernel(uint4 *__restrict__ dst, const uint4 *src, unsigned n)
{
    const unsigned i = blockIdx.x * 128u + threadIdx.x;
    if (i < n) dst[i] = __ldcv(src + i);
}

cudaError_t launch_table_copy(void *dst, const void *pinned, size_t bytes, cudaStream_t stream)
{
    const unsigned n = (unsigned)((bytes + 15) / 16);
    if (n == 0) return cudaSuccess;
    ft_table_kernel<<<(n + 127) / 128, 128, 0, stream>>>(static_cast<uint4 *>(dst), static_cast<const uint4 *>(pinned), n);
    return cudaGetLastError();
}

int fused_smem_bytes() { return (int)sizeof(Smem); }

const void *fused_kernel_ptr() { return (const void *)ft_fused_kernel; }

cudaError_t fused_occupancy(int *ctas_per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(ft_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(Smem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ft_fused_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ft_pose_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPoseSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ft_pose_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPoseSmem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, ft_fused_kernel, kThreads,
                                                         sizeof(Smem));
}

cudaError_t launch_fused(const BatchHeader *dev_hdr, int grid, cudaStream_t stream, bool overlap)
{
    OverlapLaunch l(dim3((unsigned)grid), kThreads, sizeof(Smem), stream, overlap);
    return l.run(ft_fused_kernel, dev_hdr);
}

cudaError_t launch_fused(const FrameCall &call, int grid, cudaStream_t stream, bool overlap)
{
    OverlapLaunch l(dim3((unsigned)grid), kThreads, sizeof(Smem), stream, overlap);
    return l.run(ft_fused_one_kernel, call);
}

cudaError_t launch_pose(const FrameCall &call, cudaStream_t stream)
{
    ft_pose_one_kernel<<<kPoseCtas, kPoseThreads, kPoseSmem, stream>>>(call);
    return cudaGetLastError();
}

cudaError_t launch_pose(const BatchHeader *dev_hdr, int nframes, cudaStream_t stream)
{
    if (nframes <= 0) return cudaSuccess;
    ft_pose_kernel<<<nframes * kPoseCtas, kPoseThreads, kPoseSmem, stream>>>(dev_hdr);
    return cudaGetLastError();
}

}  // namespace ft
