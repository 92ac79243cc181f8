// ft_pyramid.cu -- levels 1.. of an image pyramid resampled from level 0 on
// the device (next row f3, the pyramid part).  The paper builds the pyramid
// on the GPU as part of its ORB extraction so that it never crosses the bus
// (section IV-B) and prints no resampling; the library's reading: level l is
// round(W / sc[l]) x round(H / sc[l]); pixel (x, y) samples level 0 at
// xs = (x + 0.5) * (W / w) - 0.5 (ys likewise), clamped to the image,
// bilinear in FP32 in the order top = I00 (1 - fx) + I01 fx, bottom
// likewise, value = top (1 - fy) + bottom fy, rounded half to even.  Every
// level comes straight from level 0.
//
// One block per tile of level 0: kPyrTileRows source rows (plus the next
// row) by kPyrTileCols source columns (plus the next 16).  The block
//   1. reads the tile and stores in shared memory one 32-bit word per source
//      pixel: its own byte, the next column's, and the same two of the next
//      row, the four values of the formula, so that an output pixel is one
//      shared load (a float per pixel took two per source row, and the
//      shared-memory pipe and the issue slots were both two thirds busy);
//   2. finds, for every level, the output rows whose upper source row y0
//      and the output columns whose left source column c0 lie in the tile
//      (searches over the same FP32 operations as the formula, one lane of
//      the last warp per level while the tile loads are in flight; y0 and
//      c0 never decrease along a level), and tabulates those rows'
//      source-row offsets and vertical weights;
//   3. gives each thread kPyrCols output columns (x, x + 32, ...) of one
//      level at a time (all levels' columns in one list, so few threads
//      idle) and walks those columns' rows in the tile, two columns to a
//      packed operation.  The lanes of a warp take 32 neighbouring columns,
//      so the byte stores of a row coalesce.
// Past the image's last column and row the words hold other bytes (or zero):
// the formula clamps the source coordinate there, its weight is zero, and zero
// times any byte is the same zero.
// Every tile is independent: no block waits for another.
// What bounds it is instruction issue and the shared-memory pipe together: 128
// images of 752x480, 97 M output pixels, take 103 us (131 with a float per
// pixel and scalar products; 25 against 31 warp instructions a pixel, 10 against
// 25 M shared-memory wavefronts of loads).  Two, four and six columns a thread:
// 300 / 297 / 306 us for the call of 64 frames with pose; 384 and 512 threads
// 309 and 323.
//
// A byte b placed in the mantissa of 2^23 is the float 2^23 + b, and
// fma(2^23 + b, w, -2^23 w) rounds the exact b w once: the product b w as one
// FP32 multiplication gives it, without the conversion.  The vertical
// products are fused multiply-adds of -0.0 (a x b - 0 rounds as a x b) that
// the compiler does not know to be zero: a packed multiply that feeds a packed
// add it contracts even when both carry a rounding mode.  Sums are single
// packed FP32 additions.  The value v lies in [0, 255] up to rounding (a
// convex combination of bytes), so adding 1.5 * 2^23 rounds it to the
// nearest integer, ties to even, and the low mantissa byte is the result.
// Levels therefore equal the per-pixel formula bit for bit.
#include "ft_internal.h"

#ifndef FT_PYR_COLS
#define FT_PYR_COLS 4
#endif

namespace ft {
namespace {

constexpr int kPyrCols = FT_PYR_COLS;        // output columns per thread (32 apart), an even count
constexpr int kPyrFillRows = 4;              // tile rows a thread fills at a time

__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ int f2i(float x) { return __float2int_rz(x); }   // C (int) cast

typedef unsigned long long f32x2;        // lane 0 in the low 32 bits

__device__ __forceinline__ f32x2 f2_pack(unsigned lo, unsigned hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 a, unsigned &lo, unsigned &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(a));
}
__device__ __forceinline__ f32x2 f2_dup(float a) { return f2_pack(__float_as_uint(a), __float_as_uint(a)); }
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

constexpr unsigned kExp23 = 0x4B000000u;     // bits of 2^23
constexpr float kTwo23 = 8388608.0f;         // 2^23
constexpr float kRound23 = 12582912.0f;      // 1.5 * 2^23

// Upper source row (or left source column) of output coordinate y of a level
// with scale s = (source size) / (level size): the formula's operations.
__device__ __forceinline__ float pyr_src(int y, float s, int n)
{
    const float ys = fsub(fmul(fadd((float)y, 0.5f), s), 0.5f);
    return fminf(fmaxf(ys, 0.0f), (float)(n - 1));
}
__device__ __forceinline__ int pyr_floor(int y, float s, int n) { return f2i(floorf(pyr_src(y, s, n))); }

// First output coordinate in [0, m] whose floor source coordinate is >= t
// (m if none); the floor never decreases with the coordinate.  Starts from
// the real-valued solution of (y + 0.5) s - 0.5 = t and steps to the exact
// answer (one or two steps: the estimate is off by less than one).
__device__ int pyr_first_at_least(int t, float s, int n, int m)
{
    int y = (int)ceilf(fsub(fdiv(fadd((float)t, 0.5f), s), 0.5f));
    y = min(max(y, 0), m);
    while (y > 0 && pyr_floor(y - 1, s, n) >= t) --y;
    while (y < m && pyr_floor(y, s, n) < t) ++y;
    return y;
}

// Per level of the tile: output rows [ylo, ylo + nrows), output columns
// [xlo, xlo + ncols) (the columns from the level's width to its width
// rounded up to 4 get zeros), and the level's first unit.  A unit is one
// thread's kPyrCols columns x, x + 32, ... of a group of 32 kPyrCols
// columns, so a warp (32 units) covers one group of one level.
struct PyrLevelInfo {
    int ylo, nrows, xlo, ncols, wreal, unit0, dp;
    float sx;
    uint8_t *dst;
};

// A tile's output row of a level in the row table: its upper source row r0
// (offset in words of the staged tile; the lower one is the next staged
// row), weights fy and 1 - fy, and the row's byte offset in the level.
struct alignas(16) PyrRow {
    unsigned r0;
    float fy, gy;
    unsigned doff;
};

// side: 0 the left image, 1 the right one; nl: levels.
__device__ __forceinline__ void pyramid_run(const FrameDev &F, const int side, const int nl)
{
    extern __shared__ uint4 pyr_smem[];
    unsigned *tile = reinterpret_cast<unsigned *>(pyr_smem);                 // [kPyrTileRows][kPyrTileCols]
    PyrRow *tab = reinterpret_cast<PyrRow *>(tile + kPyrTileRows * kPyrTileCols);       // [levels][kPyrRowsPerLevel]
    __shared__ PyrLevelInfo info[FT_MAX_LEVELS + 1];

    if (!(F.build_pyr & (1 << side))) return;
    const uint8_t *src = side ? F.pyrR[0] : F.pyrL[0];
    const int *lw = side ? F.rw : F.lw, *lh = side ? F.rh : F.lh, *lp = side ? F.rp : F.lp;
    const int W = lw[0], H = lh[0], sp = lp[0];
    const int ntx = (W + kPyrTileCols - 1) / kPyrTileCols;
    if ((int)blockIdx.x >= pyr_tiles(W, H)) return;
    const int Y0 = ((int)blockIdx.x / ntx) * kPyrTileRows, X0 = ((int)blockIdx.x % ntx) * kPyrTileCols;
    const int tid = (int)threadIdx.x;

    // 1. the tile's words: four columns (one 4-byte word) of kPyrFillRows rows
    // per thread at a time, each row's bytes joined with the next row's (W
    // rounded up to 16 is within the pitch)
    const int nr = min(kPyrTileRows, H - Y0);
    const int left = ((W + 15) & ~15) - X0;          // bytes of a row from the tile on
    const int nw = min(kPyrTileCols, left) >> 2;
    const unsigned inv = (1u << 20) / (unsigned)nw + 1u;      // k / nw = k inv >> 20 for k nw < 2^20
    for (int k = tid; k < nw * (kPyrTileRows / kPyrFillRows); k += kPyrThreads) {
        const int g = (int)(((unsigned)k * inv) >> 20), c = k - g * nw;
        const int r0 = g * kPyrFillRows;
        if (r0 >= nr) break;
        const uint8_t *p = src + X0 + 4 * c;
        const bool more = 4 * c + 4 < left;
        unsigned a[kPyrFillRows + 1], t[kPyrFillRows + 1];
#pragma unroll
        for (int i = 0; i <= kPyrFillRows; ++i) {
            const uint8_t *q = p + (size_t)min(Y0 + r0 + i, H - 1) * sp;
            a[i] = __ldg(reinterpret_cast<const unsigned *>(q));
            t[i] = more ? __ldg(reinterpret_cast<const unsigned *>(q) + 1) : 0u;
        }
#pragma unroll
        for (int i = 0; i <= kPyrFillRows; ++i) t[i] = __byte_perm(a[i], t[i], 0x0043);     // columns 3, 4
#pragma unroll
        for (int i = 0; i < kPyrFillRows; ++i)
            *reinterpret_cast<uint4 *>(tile + (r0 + i) * kPyrTileCols + 4 * c) =
                make_uint4(__byte_perm(a[i], a[i + 1], 0x5410), __byte_perm(a[i], a[i + 1], 0x6521),
                           __byte_perm(a[i], a[i + 1], 0x7632), __byte_perm(t[i], t[i + 1], 0x5410));
    }
    // 2. the rows and columns of every level whose source lies in the tile:
    // lane l - 1 of the last warp takes level l (nlevels <= 16 <= 32), while
    // the other warps' tile loads are in flight
    if (tid >= kPyrThreads - 32) {
        const int lane = tid - (kPyrThreads - 32), l = 1 + lane;
        int units = 0;
        if (l < nl) {
            const int w = lw[l], h = lh[l];
            const float sx = fdiv((float)W, (float)w), sy = fdiv((float)H, (float)h);
            const int ylo = pyr_first_at_least(Y0, sy, H, h);
            const int yhi = pyr_first_at_least(Y0 + kPyrTileRows, sy, H, h);
            const int xlo = pyr_first_at_least(X0, sx, W, w);
            int xhi = pyr_first_at_least(X0 + kPyrTileCols, sx, W, w);
            if (xhi == w) xhi = (w + 3) & ~3;         // zeros up to w rounded to 4
            PyrLevelInfo &I = info[l];
            I.ylo = ylo;
            // scale_factor >= 1 makes H / h >= 1, so at most two consecutive
            // output rows share an upper source row: a tile holds at most
            // 2 x kPyrTileRows rows of a level (the bound keeps the table safe)
            I.nrows = min(yhi - ylo, kPyrRowsPerLevel);
            I.xlo = xlo;
            I.ncols = xhi - xlo;
            I.wreal = w;
            I.dp = lp[l];
            I.sx = sx;
            I.dst = const_cast<uint8_t *>(side ? F.pyrR[l] : F.pyrL[l]);
            units = 32 * ((I.ncols + 32 * kPyrCols - 1) / (32 * kPyrCols));
        }
        int end = units;                              // inclusive prefix sum over the levels
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, end, d);
            if (lane >= d) end += o;
        }
        if (l < nl) info[l].unit0 = end - units;
        if (l == nl - 1 || (nl <= 1 && lane == 0)) info[nl].unit0 = nl <= 1 ? 0 : end;   // end of the unit list
    }
    __syncthreads();
    for (int k = tid; k < (nl - 1) * kPyrRowsPerLevel; k += kPyrThreads) {
        const int l = 1 + k / kPyrRowsPerLevel, i = k - (l - 1) * kPyrRowsPerLevel;
        if (i >= info[l].nrows) continue;
        const int y = info[l].ylo + i;
        const float ys = pyr_src(y, fdiv((float)H, (float)lh[l]), H);
        const int y0 = f2i(floorf(ys));
        PyrRow e;
        e.r0 = (unsigned)((y0 - Y0) * kPyrTileCols);
        e.fy = fsub(ys, (float)y0);
        e.gy = fsub(1.0f, e.fy);
        e.doff = (unsigned)(y * info[l].dp);
        tab[k] = e;
    }
    __syncthreads();
    // 3. one unit (kPyrCols output columns 32 apart) of one level per thread
    // at a time, down the level's rows in this tile
    const int units = info[nl].unit0;
    const f32x2 minus0 = f2_dup(__uint_as_float(0x80000000u | ((unsigned)nl >> 8)));     // nl <= 16: -0.0
    int l = 1;
    for (int u = tid; u < units; u += kPyrThreads) {
        while (u >= info[l + 1].unit0) ++l;          // units are in level order; u only grows
        const int k = u - info[l].unit0;
        const int x0 = info[l].xlo + 32 * kPyrCols * (k >> 5) + (k & 31);
        const int xend = info[l].xlo + info[l].ncols, w = info[l].wreal;
        const int n = info[l].nrows;
        uint8_t *out = info[l].dst;
        const PyrRow *T = tab + (l - 1) * kPyrRowsPerLevel;
        // columns from the width to the width rounded up to 4 get zeros
#pragma unroll
        for (int j = 0; j < kPyrCols; ++j) {
            const int x = x0 + 32 * j;
            if (x >= w && x < xend)
                for (int i = 0; i < n; ++i) out[T[i].doff + x] = 0;
        }
        // sampled columns: below the width and owned by this tile (the last
        // group of a level may run past both); an unsampled column repeats
        // the first one's arithmetic and stores nothing
        const int xs_end = min(w, xend);
        if (x0 >= xs_end) continue;
        const float sx = info[l].sx;
        bool st[kPyrCols];
        const unsigned *P[kPyrCols];
        float fx[kPyrCols], gx[kPyrCols];
#pragma unroll
        for (int j = 0; j < kPyrCols; ++j) {
            st[j] = x0 + 32 * j < xs_end;
            const float xs = pyr_src(st[j] ? x0 + 32 * j : x0, sx, W);
            const int c0 = f2i(floorf(xs));
            fx[j] = fsub(xs, (float)c0);
            gx[j] = fsub(1.0f, fx[j]);
            P[j] = tile + (c0 - X0);
        }
        // the weights of a pair of columns, and -2^23 times them
        f32x2 fx2[kPyrCols / 2], gx2[kPyrCols / 2], nf2[kPyrCols / 2], ng2[kPyrCols / 2];
#pragma unroll
        for (int q = 0; q < kPyrCols / 2; ++q) {
            const float f0 = fx[2 * q], f1 = fx[2 * q + 1], g0 = gx[2 * q], g1 = gx[2 * q + 1];
            fx2[q] = f2_pack(__float_as_uint(f0), __float_as_uint(f1));
            gx2[q] = f2_pack(__float_as_uint(g0), __float_as_uint(g1));
            nf2[q] = f2_pack(__float_as_uint(fmul(f0, -kTwo23)), __float_as_uint(fmul(f1, -kTwo23)));
            ng2[q] = f2_pack(__float_as_uint(fmul(g0, -kTwo23)), __float_as_uint(fmul(g1, -kTwo23)));
        }
        uint8_t *o0 = out + x0;
        for (int i = 0; i < n; ++i) {
            const PyrRow e = T[i];
            const f32x2 fy2 = f2_dup(e.fy), gy2 = f2_dup(e.gy);
            uint8_t *o = o0 + e.doff;
            unsigned w4[kPyrCols];
#pragma unroll
            for (int j = 0; j < kPyrCols; ++j) w4[j] = P[j][e.r0];
#pragma unroll
            for (int q = 0; q < kPyrCols / 2; ++q) {
                const unsigned wa = w4[2 * q], wb = w4[2 * q + 1];
                const f32x2 t0 = f2_pack(__byte_perm(wa, kExp23, 0x7440), __byte_perm(wb, kExp23, 0x7440));
                const f32x2 t1 = f2_pack(__byte_perm(wa, kExp23, 0x7441), __byte_perm(wb, kExp23, 0x7441));
                const f32x2 b0 = f2_pack(__byte_perm(wa, kExp23, 0x7442), __byte_perm(wb, kExp23, 0x7442));
                const f32x2 b1 = f2_pack(__byte_perm(wa, kExp23, 0x7443), __byte_perm(wb, kExp23, 0x7443));
                const f32x2 top = f2_add(f2_fma(t0, gx2[q], ng2[q]), f2_fma(t1, fx2[q], nf2[q]));
                const f32x2 bot = f2_add(f2_fma(b0, gx2[q], ng2[q]), f2_fma(b1, fx2[q], nf2[q]));
                const f32x2 v = f2_add(f2_fma(top, gy2, minus0), f2_fma(bot, fy2, minus0));
                unsigned va, vb;
                f2_unpack(f2_add(v, f2_dup(kRound23)), va, vb);
                if (st[2 * q]) o[64 * q] = (uint8_t)va;
                if (st[2 * q + 1]) o[64 * q + 32] = (uint8_t)vb;
            }
        }
    }
}

__global__ void __launch_bounds__(kPyrThreads, 4) ft_pyramid_kernel(const BatchHeader *__restrict__ hdr)
{
    let_next_start();
    const int f = (int)(blockIdx.y >> 1);
    if (f >= hdr->nframes) return;
    pyramid_run(hdr->frames[f], (int)(blockIdx.y & 1), hdr->p.nlevels);
}

// one frame, its header and descriptor as kernel parameters (a 320x240 image's
// levels 13.6 us a call with a table, 8.6 us; 752x480 14.0 and 10.2)
__global__ void __launch_bounds__(kPyrThreads, 4) ft_pyramid_one_kernel(const __grid_constant__ FrameCall call)
{
    let_next_start();
    pyramid_run(call.f, (int)blockIdx.y, call.h.p.nlevels);
}

// Dynamic shared memory of the pyramid kernel for nlevels levels.
size_t pyr_smem_bytes(int nlevels)
{
    return sizeof(unsigned) * kPyrTileRows * kPyrTileCols +
           sizeof(PyrRow) * (size_t)(nlevels > 1 ? nlevels - 1 : 1) * kPyrRowsPerLevel;
}

}  // namespace

cudaError_t pyramid_setup()
{
    const int smem = (int)pyr_smem_bytes(FT_MAX_LEVELS);
    const cudaError_t e = cudaFuncSetAttribute(ft_pyramid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(ft_pyramid_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t launch_pyramids(const FrameCall &call, int tiles_per_image, cudaStream_t stream)
{
    const dim3 grid((unsigned)(tiles_per_image > 0 ? tiles_per_image : 1), 2);
    ft_pyramid_one_kernel<<<grid, kPyrThreads, pyr_smem_bytes(call.h.p.nlevels), stream>>>(call);
    return cudaGetLastError();
}

cudaError_t launch_pyramids(const BatchHeader *dev_hdr, int nframes, int nlevels, int tiles_per_image,
                            cudaStream_t stream)
{
    if (nframes <= 0) return cudaSuccess;
    const dim3 grid((unsigned)(tiles_per_image > 0 ? tiles_per_image : 1), (unsigned)(nframes * 2));
    ft_pyramid_kernel<<<grid, kPyrThreads, pyr_smem_bytes(nlevels), stream>>>(dev_hdr);
    return cudaGetLastError();
}

}  // namespace ft
