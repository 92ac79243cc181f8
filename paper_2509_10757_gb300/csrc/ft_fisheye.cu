// ft_fisheye.cu -- fisheye stereo matching (paper sections II-B and IV-C: brute
// force over the overlap, best and second best, ratio test) and the
// triangulation of its matches (f1), for sm_103a.
//
// The brute force compares every left overlap descriptor with every right one:
// a contraction.  With a descriptor's 256 bits as +-1 in FP8 (E4M3), the dot
// product of two is 256 - 2 * (Hamming distance), and FP32 accumulators hold
// it exactly, so the fifth-generation tensor cores give the distances
// themselves; eight 32-bit popcounts per pair, at 16 a clock and SM, were the
// bound before (34.6 M pairs of 32 frames: 58 us at the popcount peak, 91 us
// an item of 128 keypoints while three shared an SM).
//
// One block of 256 threads per 128 left keypoints of the overlap (compacted in
// index order), or a cluster of two or four that share the right keypoints
// step by step where the blocks would not fill the chip (one frame of 1500
// keypoints has eight).  It expands their descriptors into shared memory once (128
// rows x 256 bytes, K-major, 128-byte swizzle), then takes the right overlap
// keypoints 128 at a time: all threads expand the next 128 into one of two
// buffers while the tensor core multiplies the other (eight tcgen05.mma of
// K = 32, one thread issues), accumulators in one of two 128-column halves of
// the block's tensor memory; the epilogue reads a row per lane (two warps
// share a row's columns) and keeps the two smallest 16-bit keys (distance << 7
// | column) of even and odd columns with packed minima and maxima, then folds
// them into the row's 32-bit keys (distance << 20 | right index).  What bounds
// it now is the latency of the chain of steps at two blocks an SM (32 frames, 36
// us: issue slots 37 % busy, the tensor pipe 16 %, stalls on loads, waits and the
// step's barrier in equal parts); the epilogue spends three instructions a pair.
#include <cuda_runtime.h>

#include <cstdint>

#include "ft_internal.h"

namespace ft {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kNoKey = 0xffffffffu;
constexpr int kFishRows = 128;          // left keypoints of a block (rows of the product)
constexpr int kFishCols = 128;          // right keypoints of a step (columns)
constexpr int kFishThreads = 256;
constexpr int kFishWarps = kFishThreads / 32;
constexpr int kFishWindow = 2048;       // keypoints scanned for the overlap at a time
constexpr int kFishRowBytes = 256;      // an expanded descriptor
constexpr int kFishTile = kFishRows * kFishRowBytes;
constexpr int kFishSplit = 4;           // blocks that share a row's columns, at most (a cluster)
constexpr unsigned kTmemCols = 2 * kFishCols;
constexpr unsigned long long kDrainNs = 2000000000ull;       // bound of the wait for products after a wait ran out
static_assert(kFishRows == kFishCols, "both operands share the tile layout");
static_assert(kFishThreads == 2 * kFishRows, "two threads expand a row, two warps read a row");

struct SmemFish {
    uint8_t a[kFishTile];                   // left rows
    uint8_t b[2][kFishTile];                // right rows of this step and the next
    uint16_t list[kFishWindow];             // right overlap keypoints of the window, relative to its start
    int row[kFishRows];                     // left keypoint of each row
    unsigned best[2 * kFishSplit][kFishRows], second[2 * kFishSplit][kFishRows];  // by block of the cluster and half
    int count[kFishWarps];
    float rig[28];                          // kb of both cameras, R_rl, t_rl
    unsigned long long mbar[2];
    unsigned tmem;
};
constexpr int kFishSmem = (int)sizeof(SmemFish) + 1024;      // + alignment of the tiles
static_assert(2 * (kFishSmem + 1024) <= 228 * 1024, "shared memory above two blocks per SM");

__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fsqrt(float a) { return __fsqrt_rn(a); }

// ---------------------------------------------------------------- f1: fisheye triangulation
// sin and cos by their Taylor series (to t^13 and t^14; |t| <= 2 keeps the
// remainder under 2e-8), Horner in t^2, every operation explicitly rounded
__device__ __forceinline__ float sin_series(float t)
{
    const float t2 = fmul(t, t);
    float s = 1.60590444e-10f;               //  1/13!
    s = fadd(-2.50521079e-08f, fmul(t2, s)); // -1/11!
    s = fadd(2.75573188e-06f, fmul(t2, s));  //  1/9!
    s = fadd(-1.98412701e-04f, fmul(t2, s)); // -1/7!
    s = fadd(8.33333377e-03f, fmul(t2, s));  //  1/5!
    s = fadd(-1.66666672e-01f, fmul(t2, s)); // -1/3!
    s = fadd(1.0f, fmul(t2, s));
    return fmul(t, s);
}

__device__ __forceinline__ float cos_series(float t)
{
    const float t2 = fmul(t, t);
    float c = -1.14707454e-11f;              // -1/14!
    c = fadd(2.08767559e-09f, fmul(t2, c));  //  1/12!
    c = fadd(-2.75573200e-07f, fmul(t2, c)); // -1/10!
    c = fadd(2.48015876e-05f, fmul(t2, c));  //  1/8!
    c = fadd(-1.38888892e-03f, fmul(t2, c)); // -1/6!
    c = fadd(4.16666679e-02f, fmul(t2, c));  //  1/4!
    c = fadd(-0.5f, fmul(t2, c));            // -1/2!
    return fadd(1.0f, fmul(t2, c));
}

// Ray of a Kannala-Brandt pixel (kb = fx, fy, cx, cy, k1..k4): theta solves
// theta * (1 + k1 t + k2 t^2 + k3 t^3 + k4 t^4) = |m| (t = theta^2) by
// `iters` Newton steps from theta = |m|; false if the residual stays above
// 2e-6 rad, the model no longer rises there, or theta leaves [0, 2].
__device__ bool unproject_kb8(const float *kb, int iters, float u, float v, float *ray)
{
    const float mx = fdiv(fsub(u, kb[2]), kb[0]);
    const float my = fdiv(fsub(v, kb[3]), kb[1]);
    const float thd = fsqrt(fadd(fmul(mx, mx), fmul(my, my)));
    if (thd == 0.0f) {
        ray[0] = 0.0f;
        ray[1] = 0.0f;
        ray[2] = 1.0f;
        return true;
    }
    float th = thd, f = 0.0f, dp = 1.0f;
    for (int it = 0; it <= iters; ++it) {
        const float t2 = fmul(th, th);
        float poly = kb[7];
        poly = fadd(kb[6], fmul(t2, poly));
        poly = fadd(kb[5], fmul(t2, poly));
        poly = fadd(kb[4], fmul(t2, poly));
        poly = fadd(1.0f, fmul(t2, poly));
        f = fsub(fmul(th, poly), thd);
        dp = fmul(9.0f, kb[7]);
        dp = fadd(fmul(7.0f, kb[6]), fmul(t2, dp));
        dp = fadd(fmul(5.0f, kb[5]), fmul(t2, dp));
        dp = fadd(fmul(3.0f, kb[4]), fmul(t2, dp));
        dp = fadd(1.0f, fmul(t2, dp));
        if (it == iters) break;             // the last pass only measures the residual
        // a step that changes nothing leaves nothing to the later ones: the
        // residual is that of this pass (about 4 steps instead of 10)
        const float next = fsub(th, fdiv(f, dp));
        if (next == th) break;
        th = next;
    }
    if (!(fabsf(f) <= 2e-6f && dp > 0.0f && th >= 0.0f && th <= 2.0f)) return false;
    const float sn = fdiv(sin_series(th), thd);
    ray[0] = fmul(mx, sn);
    ray[1] = fmul(my, sn);
    ray[2] = cos_series(th);
    return true;
}

__device__ __forceinline__ float dot3f(const float *a, const float *b)
{
    return fadd(fadd(fmul(a[0], b[0]), fmul(a[1], b[1])), fmul(a[2], b[2]));
}

__device__ __forceinline__ void cross3f(const float *a, const float *b, float *c)
{
    c[0] = fsub(fmul(a[1], b[2]), fmul(a[2], b[1]));
    c[1] = fsub(fmul(a[2], b[0]), fmul(a[0], b[2]));
    c[2] = fsub(fmul(a[0], b[1]), fmul(a[1], b[0]));
}

// Midpoint of the common perpendicular of the left ray l (from the left
// centre) and the right ray r (right camera coordinates; X_r = R_rl X_l +
// t_rl), in left-camera coordinates: with C = -R^T t, d = R^T r and
// n = l x d, s = ((C x d).n)/(n.n), t = ((C x l).n)/(n.n).  Kept if the rays
// are not parallel, both parameters are positive and the depth exceeds
// min_depth.
__device__ bool triangulate(const float *l, const float *r, const float *R, const float *t, float min_depth,
                            float *X)
{
    float C[3], d[3], n[3], cd[3], cl[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        C[i] = -fadd(fadd(fmul(R[i], t[0]), fmul(R[3 + i], t[1])), fmul(R[6 + i], t[2]));
        d[i] = fadd(fadd(fmul(R[i], r[0]), fmul(R[3 + i], r[1])), fmul(R[6 + i], r[2]));
    }
    cross3f(l, d, n);
    const float nn = dot3f(n, n);
    if (!(nn > fmul(1e-10f, fmul(dot3f(l, l), dot3f(d, d))))) return false;
    cross3f(C, d, cd);
    cross3f(C, l, cl);
    const float s = fdiv(dot3f(cd, n), nn);
    const float tt = fdiv(dot3f(cl, n), nn);
    if (!(s > 0.0f && tt > 0.0f)) return false;
#pragma unroll
    for (int i = 0; i < 3; ++i) X[i] = fmul(0.5f, fadd(fmul(s, l[i]), fadd(C[i], fmul(tt, d[i]))));
    return X[2] > min_depth;
}

// f1 for left keypoint i with accepted right keypoint j (j < 0: none); rig:
// the left and right cameras' kb, R_rl, t_rl (on chip)
__device__ void triangulate_match(const DevParams &P, const FrameDev &F, const float *rig, int i, int j)
{
    float X[3] = {0.0f, 0.0f, 0.0f}, rl[3], rr[3];
    bool ok = false;
    if (j >= 0) {
        const float ul = __ldg(F.lx + i), vl = __ldg(F.ly + i), ur = __ldg(F.rx + j), vr = __ldg(F.ry + j);
        const bool left = unproject_kb8(rig, P.kb_iters, ul, vl, rl);
        const bool right = unproject_kb8(rig + 8, P.kb_iters, ur, vr, rr);
        if (left && right) ok = triangulate(rl, rr, rig + 16, rig + 25, P.min_depth, X);
    }
    F.fdepth[i] = ok ? X[2] : -1.0f;
    if (F.fxyz) F.fxyz[i] = ok ? make_float4(X[0], X[1], X[2], 1.0f) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---------------------------------------------------------------- tensor core
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Matrix descriptor of a K-major tile with 128-byte swizzle: 8-row groups of
// 1024 bytes (stride offset), descriptor version 1, swizzle mode 2.
__device__ __forceinline__ unsigned long long tile_desc(unsigned addr)
{
    return (unsigned long long)((addr & 0x3ffffu) >> 4) | (1ull << 16) | ((unsigned long long)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

// kind::f8f6f4: FP32 accumulators, E4M3 operands, both K-major, M = 128, N = 128
constexpr unsigned kInstrDesc = (1u << 4) | ((unsigned)(kFishCols >> 3) << 17) | ((unsigned)(kFishRows >> 4) << 24);

__device__ __forceinline__ void mma_f8(unsigned d, unsigned long long a, unsigned long long b, bool accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                 "l"(a), "l"(b), "r"(kInstrDesc), "r"((unsigned)accumulate)
                 : "memory");
}

// One step's product: 128 rows x 128 columns x 256, then an arrival on mbar.
__device__ __forceinline__ void mma_step(unsigned d, unsigned a, unsigned b, unsigned mbar)
{
#pragma unroll
    for (int k = 0; k < kFishRowBytes / 32; ++k) {
        // 128 bytes of K per sub-tile of 16 KB, 32 bytes per instruction
        const unsigned off = (unsigned)(k / 4) * (kFishTile / 2) + (unsigned)(k % 4) * 32u;
        mma_f8(d, tile_desc(a + off), tile_desc(b + off), k > 0);
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

// Bounded wait for the phase `parity` of mbar to end.
__device__ bool mbar_wait(unsigned mbar, unsigned parity, unsigned long long timeout_ns)
{
    unsigned long long t0 = 0;
    for (unsigned spins = 0;; ++spins) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(mbar), "r"(parity)
                     : "memory");
        if (done) return true;
        if ((spins & 31u) == 31u) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            else if (t - t0 > timeout_ns) return false;
        }
    }
}

// 32 accumulator columns of this warp's 32 lanes, from column `col`
__device__ __forceinline__ void tmem_load(unsigned (&v)[32], unsigned addr)
{
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Half a descriptor (16 bytes: 128 bits) as 128 bytes of +-1 into row r of a
// tile's half h.  Which bit lands on which byte is the same for every row, so
// it does not matter.  Threads of a warp take consecutive rows: the swizzle
// spreads their 16-byte stores over all banks.
__device__ __forceinline__ void expand(uint8_t *tile, int r, int h, uint4 d)
{
    const unsigned w[4] = {d.x, d.y, d.z, d.w};
    uint8_t *row = tile + h * (kFishTile / 2) + (r >> 3) * 1024 + (r & 7) * 128;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        unsigned o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = ((w[q] << (7 - i)) & 0x80808080u) | 0x38383838u;
        *reinterpret_cast<uint4 *>(row + 16 * ((2 * q) ^ (r & 7))) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4 *>(row + 16 * ((2 * q + 1) ^ (r & 7))) = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// Keypoints of [j0, j0 + n), n <= kFishWindow, with lo <= x <= hi, in index
// order: put(rank, j - j0) for each; returns how many.  The caller
// synchronizes before it reads what was put.
template <class Put>
__device__ __forceinline__ int compact(const float *xs, int j0, int n, float lo, float hi, int *count, Put put)
{
    constexpr int kPer = kFishWindow / kFishWarps, kIter = kPer / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned in[kIter];
    int mine = 0;
    float x[kIter];
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
        const int e = warp * kPer + 32 * i + lane;
        x[i] = e < n ? __ldg(xs + j0 + e) : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
        const int e = warp * kPer + 32 * i + lane;
        in[i] = __ballot_sync(kFull, e < n && x[i] >= lo && x[i] <= hi);
        mine += __popc(in[i]);
    }
    __syncthreads();                                // the previous use of count
    if (lane == 0) count[warp] = mine;
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kFishWarps; ++w) {
        base += w < warp ? count[w] : 0;
        total += count[w];
    }
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
        if ((in[i] >> lane) & 1u) put(base + __popc(in[i] & ((1u << lane) - 1u)), warp * kPer + 32 * i + lane);
        base += __popc(in[i]);
    }
    return total;
}

// Stores v at this shared-memory location of the cluster's first block.
__device__ __forceinline__ void store_first(unsigned *p, unsigned v)
{
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %0, 0;\n\t"
                 "st.shared::cluster.u32 [a], %1;\n\t}" ::"r"(smem_addr(p)),
                 "r"(v)
                 : "memory");
}

__device__ __forceinline__ void top2_push(unsigned key, unsigned &best, unsigned &second)
{
    second = min(second, max(best, key));
    best = min(best, key);
}

// The two smallest keys of 32 accumulator columns in each 16-bit lane (even
// and odd columns): (256 - v) / 2 << 7 | column is 16384 - 64 v + column,
// formed in the low mantissa bits of 2^23 + it (exact; the column is a
// constant, so a key is one instruction).  n: columns that count, from col0 = 0.
template <bool kAll>
__device__ __forceinline__ void scan_columns(const unsigned (&v)[32], const int col0, int n, unsigned &best,
                                             unsigned &second)
{
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const unsigned k0 =
            __float_as_uint(__fmaf_rn(__uint_as_float(v[i]), -64.0f, 8388608.0f + 16384.0f + (float)(col0 + i)));
        const unsigned k1 =
            __float_as_uint(__fmaf_rn(__uint_as_float(v[i + 1]), -64.0f, 8388608.0f + 16384.0f + (float)(col0 + i + 1)));
        unsigned k = __byte_perm(k0, k1, 0x5410);
        if (!kAll) {
            if (col0 + i >= n) k |= 0xffffu;
            if (col0 + i + 1 >= n) k |= 0xffff0000u;
        }
        second = __vminu2(second, __vmaxu2(best, k));
        best = __vminu2(best, k);
    }
}

// tile: of 128 left keypoints.
__device__ __forceinline__ void fisheye_run(const BatchHeader *hdr, const FrameDev &F, const int tile)
{
    extern __shared__ unsigned char fish_raw[];
    SmemFish &S = *reinterpret_cast<SmemFish *>(fish_raw + ((1024u - (smem_addr(fish_raw) & 1023u)) & 1023u));
    if (F.camera != FT_CAMERA_FISHEYE || !F.do_stereo || tile * kFishRows >= F.nl) return;
    const DevParams &P = hdr->p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nl = F.nl, nr = F.nr;
    const float *const rx = F.rx;
    const uint4 *const rdesc = F.rdesc;
    const float lap_r0 = F.lap_r0, lap_r1 = F.lap_r1;
    const unsigned long long timeout_ns = hdr->timeout_ns;

    if (tid < 28) S.rig[tid] = tid < 8 ? F.kbl[tid] : tid < 16 ? F.kbr[tid - 8] : tid < 25 ? F.R_rl[tid - 16] : F.t_rl[tid - 25];
    const int split = (int)blockIdx.z, splits = (int)gridDim.z;     // of the cluster

    // this block's share of the left keypoints outside the overlap: no match
    const int i_out = tile * kFishRows + tid;
    if (split == 0 && tid < kFishRows && i_out < nl) {
        const float x = __ldg(F.lx + i_out);
        if (!(x >= F.lap_l0 && x <= F.lap_l1)) {
            F.r_idx[i_out] = -1;
            F.fd1[i_out] = -1;
            F.fd2[i_out] = -1;
            if (F.fdepth) triangulate_match(P, F, nullptr, i_out, -1);
        }
    }
    // the rows: left keypoints of the overlap with ranks [128 tile, 128 tile + 128)
    int seen = 0;
    for (int i0 = 0; i0 < nl && seen < (tile + 1) * kFishRows; i0 += kFishWindow) {
        const int n = min(kFishWindow, nl - i0);
        seen += compact(F.lx, i0, n, F.lap_l0, F.lap_l1, S.count, [&](int rank, int e) {
            const int r = seen + rank - tile * kFishRows;
            if (r >= 0 && r < kFishRows) S.row[r] = i0 + e;
        });
    }
    const int rows = min(seen - tile * kFishRows, kFishRows);
    if (rows <= 0) return;                          // the whole cluster
    // says that this block has started; the first block's shared memory may be
    // written by the others once all have said so (waited for below, long over
    // by then: the matching lies between)
    if (splits > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");

    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&S.tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&S.mbar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&S.mbar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();                                // rows, tensor memory address, barriers
    const int er = tid & (kFishRows - 1), eh = tid / kFishRows;     // row and half this thread expands
    if (er < rows) expand(S.a, er, eh, __ldg(F.ldesc + 2 * S.row[er] + eh));
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = S.tmem;

    unsigned best = kNoKey, second = kNoKey;        // of row 32 (warp & 3) + lane, half the columns
    const int half = warp >> 2;
    const unsigned lanes = (unsigned)(32 * (warp & 3)) << 16;
    unsigned phase = 0, flying = 0;                 // bit k: parity of mbar[k]; a product that arrives on it is on its way
    bool ok = true;
    for (int j0 = 0; j0 < nr && ok; j0 += kFishWindow) {
        const int cnt = compact(rx, j0, min(kFishWindow, nr - j0), lap_r0, lap_r1, S.count,
                                [&](int rank, int e) { S.list[rank] = (uint16_t)e; });
        __syncthreads();
        const int steps = (cnt + kFishCols - 1) / kFishCols;
        // this block's steps: split, split + splits, ...; its i-th uses buffers i & 1
        const int mine = steps > split ? (steps - split + splits - 1) / splits : 0;
        uint4 next = make_uint4(0, 0, 0, 0);        // what this thread expands next
        auto fetch = [&](int i) {
            const int c = (split + i * splits) * kFishCols + er;
            if (i < mine && c < cnt) next = __ldg(rdesc + 2 * (j0 + S.list[c]) + eh);
        };
        auto stage = [&](int i) {
            if ((split + i * splits) * kFishCols + er < cnt) expand(S.b[i & 1], er, eh, next);
            // the tensor core reads shared memory through the async proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            ok = __syncthreads_and(ok);
            if (!ok) return;
            flying |= 1u << (i & 1);
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                mma_step(tmem + (unsigned)(i & 1) * kFishCols, smem_addr(S.a), smem_addr(S.b[i & 1]),
                         smem_addr(&S.mbar[i & 1]));
            }
            fetch(i + 1);
        };
        fetch(0);
        if (mine > 0) stage(0);
        for (int i = 0; i < mine; ++i) {
            // the buffer of step i + 1 was read by step i - 1, whose product
            // every thread has waited for; its accumulators were read before
            // stage()'s block-wide synchronization
            if (i + 1 < mine) stage(i + 1);
            if (!ok) break;                         // a wait ran out: known to the whole block
            const int s = split + i * splits;
            ok = __all_sync(kFull, mbar_wait(smem_addr(&S.mbar[i & 1]), (phase >> (i & 1)) & 1u, timeout_ns));
            if (!ok) continue;                      // the others learn of it at the next block-wide synchronization
            phase ^= 1u << (i & 1);
            flying &= ~(1u << (i & 1));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int n = cnt - s * kFishCols - 64 * half;       // of this warp's 64 columns
            unsigned b2 = 0xffffffffu, s2 = 0xffffffffu;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (32 * q >= n) continue;                  // the same in the whole warp
                unsigned v[32];
                tmem_load(v, tmem + lanes + (unsigned)((i & 1) * kFishCols + 64 * half + 32 * q));
                if (32 * q + 32 <= n) scan_columns<true>(v, 32 * q, n, b2, s2);
                else scan_columns<false>(v, 32 * q, n, b2, s2);
            }
            // the step's two smallest; right indices ascend, so one whose
            // distance is not below the row's second cannot enter any more
            const unsigned bl = b2 & 0xffffu, bh = b2 >> 16, sl = s2 & 0xffffu, sh = s2 >> 16;
            const unsigned k1 = min(bl, bh), k2 = min(max(bl, bh), min(sl, sh));
            if (k1 != 0xffffu && k1 >> 7 < second >> 20) {
                const uint16_t *at = S.list + s * kFishCols + 64 * half;
                top2_push((k1 >> 7) << 20 | (unsigned)(j0 + at[k1 & 127u]), best, second);
                if (k2 != 0xffffu && k2 >> 7 < second >> 20)
                    top2_push((k2 >> 7) << 20 | (unsigned)(j0 + at[k2 & 127u]), best, second);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        ok = __syncthreads_and(ok);                 // the list is read before the next window's
    }
    if (!ok) {
        if (tid == 0) atomicOr(hdr->status, kStatusTimeout);
        best = second = kNoKey;
        // products still on their way write tensor memory and read the tiles:
        // they end before either is given back
        for (int k = 0; k < 2; ++k)
            if (flying >> k & 1u) (void)mbar_wait(smem_addr(&S.mbar[k]), (phase >> k) & 1u, kDrainNs);
        __syncthreads();
    }
    // the parts of a row's columns (two halves of every block's steps) meet in
    // the cluster's first block, which then writes the match
    const int r = 32 * (warp & 3) + lane;
    if (splits == 1) {
        S.best[half][r] = best;
        S.second[half][r] = second;
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.wait;" ::: "memory");             // every block has started
        store_first(&S.best[2 * split + half][r], best);
        store_first(&S.second[2 * split + half][r], second);
        __syncthreads();
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    if (split == 0 && half == 0 && r < rows) {
        for (int p = 1; p < 2 * splits; ++p) {
            const unsigned ob = S.best[p][r], os = S.second[p][r];
            second = min(min(second, os), max(best, ob));
            best = min(best, ob);
        }
        const int i = S.row[r];
        int match = -1, d1 = -1, d2 = -1;
        if (best != kNoKey) {
            d1 = (int)(best >> 20);
            d2 = second != kNoKey ? (int)(second >> 20) : 256;
            if ((float)d1 < fmul(P.fisheye_ratio, (float)d2)) match = (int)(best & 0xfffffu);
        }
        F.r_idx[i] = match;
        F.fd1[i] = d1;
        F.fd2[i] = d2;
        if (F.fdepth) triangulate_match(P, F, S.rig, i, match);
    }
}

// A frame's blocks follow one another along x, which alone holds a batch of 65536
// frames (frames along x and blocks along y: 32 frames 74.0 us, this way 72.1).
__global__ void __launch_bounds__(kFishThreads, 2) ft_fisheye_kernel(const BatchHeader *__restrict__ hdr, unsigned blocks)
{
    let_next_start();
    wait_for_previous();
    const unsigned f = blockIdx.x / blocks;
    if ((int)f >= hdr->nframes) return;
    fisheye_run(hdr, hdr->frames[f], (int)(blockIdx.x - f * blocks));
}

// one frame, its header and descriptor as kernel parameters
__global__ void __launch_bounds__(kFishThreads, 2) ft_fisheye_one_kernel(const __grid_constant__ FrameCall call)
{
    let_next_start();
    fisheye_run(&call.h, call.f, (int)blockIdx.x);
}

// Columns are shared out while that still leaves the chip's 152 SMs a block
// each (about 60 % of a frame's blocks have rows: the overlap).
int fisheye_splits(int nframes, int blocks)
{
    int splits = 1;
    while (splits < kFishSplit && 2 * splits * blocks * nframes <= 256) splits *= 2;
    return splits;
}

}  // namespace

cudaError_t fisheye_setup()
{
    cudaError_t e = cudaFuncSetAttribute(ft_fisheye_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFishSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ft_fisheye_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFishSmem);
    return e;
}

int fisheye_blocks(int nl) { return (nl + kFishRows - 1) / kFishRows; }

cudaError_t launch_fisheye(const BatchHeader *dev_hdr, int nframes, int blocks, cudaStream_t stream, bool overlap)
{
    if (nframes <= 0 || blocks <= 0) return cudaSuccess;
    const unsigned splits = (unsigned)fisheye_splits(nframes, blocks);
    // (at most 65536 frames of 8192 blocks: below 2^31)
    OverlapLaunch l(dim3((unsigned)blocks * (unsigned)nframes, 1, splits), kFishThreads, kFishSmem, stream, overlap);
    l.cluster(1, 1, splits);
    return l.run(ft_fisheye_kernel, dev_hdr, (unsigned)blocks);
}

cudaError_t launch_fisheye(const FrameCall &call, int blocks, cudaStream_t stream)
{
    if (blocks <= 0) return cudaSuccess;
    const unsigned splits = (unsigned)fisheye_splits(1, blocks);
    OverlapLaunch l(dim3((unsigned)blocks, 1, splits), kFishThreads, kFishSmem, stream, false);
    l.cluster(1, 1, splits);
    return l.run(ft_fisheye_one_kernel, call);
}

}  // namespace ft
