// ft_orb.cu -- keypoint detection and description on the pyramid levels
// (next row f3).  The paper's ORB extraction builds the image pyramid, finds
// keypoints on every level, describes each one and filters them (section
// II-A); FastTrack reuses an existing GPU extractor (section IV-B) and
// prints none of its steps.  This file implements the reading stated in the
// public header: FAST-9 corners with the maximum-threshold score, 3x3
// non-maximum suppression (ties: the earlier raster position), the best
// max_kp[l] corners per level by (score descending, y, x) in fixed slots,
// intensity-centroid orientation over the radius-15 disk, and 256 steered
// tests on the level smoothed by the 5x5 binomial filter.
//
// Three launches per call, each over every image of the call:
//   detect    one block of 256 threads per 62x30 tile of a level (64x32 with
//             its suppression ring): the tile and a 4-pixel halo in shared
//             memory as two planes of packed pixel pairs, a compass test of
//             every pair (two pixels per step in 16-bit lanes), the arcs and
//             the FAST score of the pairs that pass, for their polarity, a
//             16-bit suppression key per corner that orders score and raster
//             position at once, suppression of the listed corners by their
//             eight neighbours' largest key, the kept ones appended as
//             keys (255 - score) << 24 | y << 12 | x (one atomic per warp),
//             and the smoothed level written from the same tile (separable,
//             two pixels per word);
//   select    one block per (image, level): the max_kp best of the level's
//             corners in two reads of them (the deciding score, then the
//             gather), sorted in shared memory by counting or a bitonic
//             network;
//   describe  one warp per output slot: the keypoint's two neighbourhoods
//             (level and smoothed level) copied to shared memory in one
//             round trip of 16-byte asynchronous copies, the moments over
//             the disk (integer warp sums), the orientation, and lane b
//             computes descriptor byte b (tests 8b .. 8b+7).
// Integer work is exact; the orientation and the rotated test positions use
// IEEE-rounded FP32 in the order the reading gives (the moment magnitude,
// a double square root rounded to float in the reading, is the same value
// from an FP32 square root settled by integer comparisons: ft_sqrt.h), so
// results equal the oracle's bit for bit.
#include <cuda_runtime.h>

#include <cstdint>

#include "ft_internal.h"
#include "ft_sqrt.h"

namespace ft {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kDetThreads = 256;
constexpr int kDetWarps = kDetThreads / 32;
constexpr int kHaloRows = kOrbTileH + 2 * kOrbHalo;     // 38 rows of 70 columns
constexpr int kHaloCols = kOrbTileW + 2 * kOrbHalo;
constexpr int kHalfW = 36;                              // words per row of a pixel-pair plane (35 used)
constexpr int kRingRows = kOrbTileH + 2;                // tile + suppression ring: 32 rows of 32 pixel pairs
constexpr int kRingPairs = (kOrbTileW + 2) / 2;
constexpr int kListCap = kRingRows * kRingPairs;
constexpr int kDescribeWarps = 8;
static_assert(kRingPairs == 32 && kRingRows == 4 * kDetWarps, "a warp takes whole ring rows, one pixel pair a lane");
static_assert(kHaloCols <= 72, "18 words of a level row hold a halo row");

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Offsets of the 16 pixels of the radius-3 circle, clockwise from (0, -3):
// x offsets 0 1 2 3 3 3 2 1 0 -1 -2 -3 -3 -3 -2 -1, stored + 3 as 4-bit
// nibbles of one constant; the y offset of pixel i is the x offset of pixel
// i + 12.
__device__ __forceinline__ int circle_dx(int i)
{
    constexpr unsigned long long kPacked = 0x2100012345666543ull;
    return (int)((kPacked >> (4 * i)) & 15ull) - 3;
}
__device__ __forceinline__ int circle_dy(int i) { return circle_dx((i + 12) & 15); }

// lane-wise minimum / maximum of two pixel pairs (16-bit lanes)
__device__ __forceinline__ unsigned vmin2(unsigned a, unsigned b) { return __vminu2(a, b); }
__device__ __forceinline__ unsigned vmax2(unsigned a, unsigned b) { return __vmaxu2(a, b); }

// The best arc of a pixel pair's 16 circle values v (one pixel per 16-bit
// lane): for kBright the largest, over the 16 arcs of 9 contiguous circle
// pixels, of the arc's smallest value; otherwise the smallest of the arcs'
// largest values.  Two arcs that start next to each other share eight pixels:
// for even k, the better of the arcs from k and from k + 1 is the extreme of
// pixels k + 1 .. k + 8 and of the better of pixels k and k + 9.  36
// operations a polarity (40 with the extremes of all 16 arcs formed).
template <bool kBright>
__device__ __forceinline__ unsigned best_arc(const unsigned (&v)[16])
{
    auto in2 = [](unsigned a, unsigned b) { return kBright ? vmin2(a, b) : vmax2(a, b); };
    auto out2 = [](unsigned a, unsigned b) { return kBright ? vmax2(a, b) : vmin2(a, b); };
    auto in3 = [](unsigned a, unsigned b, unsigned c) { return kBright ? __vimin3_u16x2(a, b, c) : __vimax3_u16x2(a, b, c); };
    auto out3 = [](unsigned a, unsigned b, unsigned c) { return kBright ? __vimax3_u16x2(a, b, c) : __vimin3_u16x2(a, b, c); };
    unsigned p[8], q[8], w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) p[j] = in2(v[2 * j + 1], v[(2 * j + 2) & 15]);
#pragma unroll
    for (int j = 0; j < 8; ++j) q[j] = in2(p[j], p[(j + 1) & 7]);          // pixels 2j + 1 .. 2j + 4
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = in3(q[j], q[(j + 2) & 7], out2(v[2 * j], v[(2 * j + 9) & 15]));
    const unsigned r0 = out3(w[0], w[1], w[2]), r1 = out3(w[3], w[4], w[5]);
    return out2(out3(w[6], w[7], r0), r1);
}

// The 16 circle values of the pixel pair (ring row ry, ring columns 2h and
// 2h + 1), whose centre is po[ry + 3][h + 1].
__device__ __forceinline__ void load_circle(const unsigned (*pe)[kHalfW], const unsigned (*po)[kHalfW], int ry, int h,
                                            unsigned (&v)[16])
{
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int dx = circle_dx(i), dy = circle_dy(i);     // halo column of the pair: 2h + 3 + dx
        v[i] = (dx & 1) ? pe[ry + 3 + dy][h + ((3 + dx) >> 1)] : po[ry + 3 + dy][h + 1 + (dx >> 1)];
    }
}

// One block per tile of 62 x 30 pixels of a level, so that the tile with its
// one-pixel suppression ring is 64 x 32 pixels: a warp takes whole rows, a
// lane two adjacent pixels, every shared-memory row read is conflict-free and
// nothing divides (32 x 32 tiles, 17 pairs a ring row, ran 6.0 warp
// instructions per tile pixel row of 32 and 80 % of the shared-memory
// wavefronts; this form 2.7).  The tile and its 4-pixel halo are held as two
// planes of pixel pairs: pe[r][k] packs the pixels of halo columns 2k and
// 2k + 1 of halo row r in its low and high 16-bit lanes, po[r][k] those of
// columns 2k + 1 and 2k + 2.  Any two horizontally adjacent pixels are then
// one word.
//
// Every corner of the tile and its ring gets a suppression key, (FAST score +
// 1) << 8 | (255 - g) with g = 3 * ring row + ring column (0: not a corner).
// Between 8-neighbours, 3 * dy + dx orders the earlier raster position first,
// so "the neighbour's score is larger, or equal and the neighbour comes
// first" is "the neighbour's key is larger" and a corner survives suppression
// when its key exceeds its 8 neighbours'.
//
// Nine contiguous circle pixels hold two neighbouring ones of the four
// compass pixels, so a bright corner has one of the upper and lower and one of
// the left and right compass pixels above I + t, and a dark one below I - t.
// That test (five loads, a dozen packed operations for a pixel pair and both
// polarities) goes first; pairs with a pixel that passes are listed by
// polarity, and only they get the 16 loads and the arcs, in full warps and
// for their polarity alone; corners are listed again for the suppression.
// What bounds the kernel is instruction issue, and a pixel of footage is
// rarely a corner: 128 images of 752x480 footage-like content (2.4 % corners;
// 14 % of the pixels pass the test), 143 M pixels, took 1176 us with every
// pair's arcs in both polarities, 975 us with the test on 32 x 32 tiles,
// 743 us on these.  A warp then takes its rows of a phase together, their loads
// in flight at once and one reservation for all its listed pairs: 648 us (79 %
// of the shared-memory wavefronts, 77 % of the issue slots).  62 x 62 tiles of
// 512 threads load fewer halo rows but cover more outside the small levels:
// extraction 853 us against 808.
__global__ void __launch_bounds__(kDetThreads, 6) orb_detect_kernel(const OrbHeader *__restrict__ hdr)
{
    __shared__ __align__(16) unsigned pe[kHaloRows][kHalfW];
    __shared__ __align__(16) unsigned po[kHaloRows][kHalfW];
    __shared__ unsigned key[kRingRows][kRingPairs];         // two 16-bit keys per word
    __shared__ unsigned hs[kOrbTileH + 4][kRingPairs];      // horizontal binomial sums of rows -2 .. H + 1, two per word
    __shared__ uint16_t listed[2][kListCap];                // pairs that passed the compass test: bright, dark
    __shared__ uint16_t corner[2 * kListCap];               // corners of the tile: ring row << 6 | ring column
    __shared__ unsigned n_listed[2];                        // bright | dark << 16, corners
    let_next_start();
    const OrbHeader &H = *hdr;
    const OrbImage &I = H.images[blockIdx.y];
    const int tile = blockIdx.x;
    if (tile >= I.tiles) return;
    int l = 0;
#pragma unroll
    for (int k = 0; k < FT_MAX_LEVELS; k += 4) {             // levels past the last start past every tile
        const int4 f = __ldg(reinterpret_cast<const int4 *>(I.tile0 + k));
        l += (f.x <= tile) + (f.y <= tile) + (f.z <= tile) + (f.w <= tile);
    }
    --l;                                                     // level 0 starts at tile 0
    const OrbLevel &L = I.lv[l];
    const int t = tile - L.tile0;
    // t / tiles_x by its reciprocal in 32.32 fixed point, rounded up: exact
    // for t, tiles_x < 2^16 (a level has at most 67 x 137 tiles)
    const int tx = L.tiles_x, ty = tx > 1 ? (int)__umulhi((unsigned)t, L.tiles_x_inv) : t;
    const int x0 = (t - ty * tx) * kOrbTileW, y0 = ty * kOrbTileH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int W = L.w, Hl = L.h, pitch = L.pitch;
    const uint8_t *const img = L.img;
    if (tile == 0 && tid == 0) I.n_level[H.nlevels] = 0;     // the select blocks add to it
    if (tid < 2) n_listed[tid] = 0;
    // the tile and its halo, coordinates clamped to the level (the smoothing
    // replicates the border; FAST only runs where its circle is inside), as
    // whole words: level rows are 16-byte aligned (checked on the host), and a
    // lane's word and the next lane's give four pixels and the one after
    // them.  x0 is even: the halo starts at byte 0 or 2 of a word.
    {
        const int xa = x0 >= kOrbHalo ? (x0 - kOrbHalo) & ~3 : -kOrbHalo;
        const unsigned shift = 8u * (unsigned)((x0 - kOrbHalo) & 3);
        const int p = xa + 4 * lane;                         // first pixel of this lane's word
        const bool wide = x0 < kOrbHalo || x0 + kOrbTileW + kOrbHalo > W;    // some columns lie outside
        const int pc = min(max(p, 0), (W - 1) & ~3);         // the word that is read
        const unsigned have = (unsigned)(W - pc);            // pixels of the level from there
        constexpr int kRows = (kHaloRows + kDetWarps - 1) / kDetWarps;      // of a warp, all in flight at once
        unsigned word[kRows];
#pragma unroll
        for (int s = 0; s < kRows; ++s) {
            const int r = min(warp + s * kDetWarps, kHaloRows - 1);
            const uint8_t *row = img + (size_t)clampi(y0 - kOrbHalo + r, 0, Hl - 1) * pitch;
            word[s] = lane < 18 ? __ldg(reinterpret_cast<const unsigned *>(row + pc)) : 0u;
        }
#pragma unroll
        for (int s = 0; s < kRows; ++s) {
            const int r = warp + s * kDetWarps;
            if (r >= kHaloRows) break;                       // the whole warp
            unsigned w = word[s];
            if (wide) {
                // bytes past the level's last pixel repeat it; words before
                // the first or past the last pixel repeat that one
                if (have < 4u) {
                    const unsigned last = (w >> (8u * (have - 1u))) & 0xffu, keep = (1u << (8u * have)) - 1u;
                    w = (w & keep) | (last * 0x01010101u & ~keep);
                }
                if (p < 0) w = (w & 0xffu) * 0x01010101u;
                if (p > pc) w = (w >> 24) * 0x01010101u;
            }
            const unsigned a = __funnelshift_r(w, __shfl_down_sync(kFull, w, 1), shift);
            const unsigned b = __shfl_down_sync(kFull, a, 1);
            if (lane < 18) {
                *reinterpret_cast<uint2 *>(&pe[r][2 * lane]) = make_uint2(__byte_perm(a, 0u, 0x4140), __byte_perm(a, 0u, 0x4342));
                *reinterpret_cast<uint2 *>(&po[r][2 * lane]) =
                    make_uint2(__byte_perm(a, 0u, 0x4241), __byte_perm(__funnelshift_r(a, b, 24), 0u, 0x4140));
            }
        }
    }
    __syncthreads();
    // the compass test of the tile and its ring, a row per warp at a time; the
    // pair's centre is po[ry + 3][lane + 1].  Pixels closer than E to a border
    // (or outside the level) are not corners; a pair with neither pixel inside
    // is not listed.
    const int E = H.edge, th = H.fast_th;
    const unsigned th2 = (unsigned)(256 + th) * 0x00010001u;
    const int px = x0 - 1 + 2 * lane;
    const bool in0 = px >= E && px < W - E, in1 = px + 1 >= E && px + 1 < W - E;
    constexpr int kRows = kRingRows / kDetWarps;            // of a warp
    unsigned mb[kRows], md[kRows], n2 = 0u;
#pragma unroll
    for (int s = 0; s < kRows; ++s) {
        const int ry = warp + s * kDetWarps, py = y0 - 1 + ry;
        key[ry][lane] = 0u;
        const unsigned c = po[ry + 3][lane + 1], up = po[ry][lane + 1], dn = po[ry + 6][lane + 1];
        const unsigned lf = pe[ry + 3][lane], rt = pe[ry + 3][lane + 3];
        // the best a corner could score, + 256 in each lane (the lanes stay
        // in [1, 511]); above t + 256 in one of them?
        const unsigned br = vmin2(vmax2(up, dn), vmax2(lf, rt)) + 0x01000100u - c;
        const unsigned dk = c + 0x01000100u - vmax2(vmin2(up, dn), vmin2(lf, rt));
        const bool in = (in0 || in1) && py >= E && py < Hl - E;
        mb[s] = __ballot_sync(kFull, in && vmax2(br, th2) != th2);
        md[s] = __ballot_sync(kFull, in && vmax2(dk, th2) != th2);
        n2 += (unsigned)__popc(mb[s]) | (unsigned)__popc(md[s]) << 16;
    }
    if (n2 != 0u) {
        // both lists' counters in one word (each stays below 2^16), one
        // reservation for all the warp's rows
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&n_listed[0], n2);
        at = __shfl_sync(kFull, at, 0);
        const unsigned below = (1u << lane) - 1u;
        uint16_t *lb = listed[0] + (at & 0xffffu), *ld = listed[1] + (at >> 16);
#pragma unroll
        for (int s = 0; s < kRows; ++s) {
            const uint16_t q = (uint16_t)((warp + s * kDetWarps) * kRingPairs + lane);
            if (mb[s] >> lane & 1u) lb[__popc(mb[s] & below)] = q;
            if (md[s] >> lane & 1u) ld[__popc(md[s] & below)] = q;
            lb += __popc(mb[s]);
            ld += __popc(md[s]);
        }
    }
    // horizontal binomial sums (1 4 6 4 1) of halo rows 2 .. 35, output
    // columns 2k and 2k + 1 (taps at halo columns 2k + 2 .. 2k + 7)
#pragma unroll
    for (int s = 0; s < (kOrbTileH + 4 + kDetWarps - 1) / kDetWarps; ++s) {
        const int r = warp + s * kDetWarps;
        if (r < kOrbTileH + 4 && lane < kOrbTileW / 2) {
            const unsigned *e = pe[r + 2], *o = po[r + 2];
            hs[r][lane] = e[lane + 1] + 4u * o[lane + 1] + 6u * e[lane + 2] + 4u * o[lane + 2] + e[lane + 3];
        }
    }
    __syncthreads();
    // the listed pairs' arcs; a pixel is a corner of one polarity at most (9 of
    // 16 circle pixels each), so no key is written and no corner listed twice
    const int nb = (int)(n_listed[0] & 0xffffu), nk = nb + (int)(n_listed[0] >> 16);
    for (int e0 = 32 * warp; e0 < nk; e0 += kDetThreads) {
        const int e = e0 + lane;
        bool k0 = false, k1 = false;
        int ry = 0, h = 0;
        if (e < nk) {
            const bool bright = e < nb;
            const int q = bright ? listed[0][e] : listed[1][e - nb];
            ry = q / kRingPairs;
            h = q % kRingPairs;
            unsigned v[16];
            load_circle(pe, po, ry, h, v);
            const unsigned c = po[ry + 3][h + 1];
            // the best arc's smallest difference, + 256 in each lane
            const unsigned d = bright ? best_arc<true>(v) + 0x01000100u - c : c + 0x01000100u - best_arc<false>(v);
            const int b0 = (int)(d & 0xffffu) - 256, b1 = (int)(d >> 16) - 256;
            const int qx = x0 - 1 + 2 * h;                  // the row is inside: the pair was listed
            k0 = b0 > th && qx >= E && qx < W - E;
            k1 = b1 > th && qx + 1 >= E && qx + 1 < W - E;
            const unsigned g = 3u * (unsigned)ry + 2u * (unsigned)h;
            uint16_t *k = reinterpret_cast<uint16_t *>(&key[ry][h]);
            if (k0) k[0] = (uint16_t)(((unsigned)b0 << 8) | (255u - g));
            if (k1) k[1] = (uint16_t)(((unsigned)b1 << 8) | (254u - g));
        }
        __syncwarp();
        // the tile's own corners (not its ring's)
        const bool own = ry >= 1 && ry <= kOrbTileH;
        k0 = k0 && own && h > 0;
        k1 = k1 && own && h < kRingPairs - 1;
        const unsigned m0 = __ballot_sync(kFull, k0), m1 = __ballot_sync(kFull, k1);
        if ((m0 | m1) == 0u) continue;
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&n_listed[1], (unsigned)(__popc(m0) + __popc(m1)));
        at = __shfl_sync(kFull, at, 0);
        const unsigned below = (1u << lane) - 1u;
        if (k0) corner[at + __popc(m0 & below)] = (uint16_t)(ry << 6 | 2 * h);
        if (k1) corner[at + __popc(m0) + __popc(m1 & below)] = (uint16_t)(ry << 6 | (2 * h + 1));
    }
    // vertical sums: a warp's four rows (two of the last warp's) from eight
    // rows of horizontal sums
    if (lane < kOrbTileW / 2) {
        const int iy0 = 4 * warp, sx = x0 + 2 * lane;
        const int spitch = L.spitch;
        uint8_t *o = L.smooth + (size_t)(y0 + iy0) * spitch + sx;
        unsigned v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = iy0 + r < kOrbTileH + 4 ? hs[iy0 + r][lane] : 0u;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (iy0 + r >= kOrbTileH || y0 + iy0 + r >= Hl || sx >= W) continue;
            const unsigned acc = v[r] + 4u * v[r + 1] + 6u * v[r + 2] + 4u * v[r + 3] + v[r + 4] + 0x00800080u;
            const unsigned sv = __byte_perm(acc, 0u, 0x4431);       // the two lanes' bits 8-15
            if (sx + 1 < W) *reinterpret_cast<uint16_t *>(o + r * spitch) = (uint16_t)sv;
            else o[r * spitch] = (uint8_t)sv;
        }
    }
    __syncthreads();
    // suppression of the listed corners; one atomic per warp and step reserves
    // the survivors' places
    const int nc = (int)n_listed[1];
    const uint16_t *keys = reinterpret_cast<const uint16_t *>(&key[0][0]);
    for (int e0 = 32 * warp; e0 < nc; e0 += kDetThreads) {
        const int e = e0 + lane;
        bool keep = false;
        unsigned kv = 0u;
        if (e < nc) {
            const int at = corner[e];                       // = index into keys: 64 per ring row
            const unsigned kp = keys[at];
            unsigned m = max(max((unsigned)keys[at - 65], (unsigned)keys[at - 64]), (unsigned)keys[at - 63]);
            m = max(max(m, (unsigned)keys[at - 1]), (unsigned)keys[at + 1]);
            m = max(max(m, (unsigned)keys[at + 63]), max((unsigned)keys[at + 64], (unsigned)keys[at + 65]));
            keep = kp > m;
            kv = ((256u - (kp >> 8)) << 24) | ((unsigned)(y0 - 1 + (at >> 6)) << 12) | (unsigned)(x0 - 1 + (at & 63));
        }
        const unsigned mk = __ballot_sync(kFull, keep);
        if (mk == 0u) continue;
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&I.cnt[l], (unsigned)__popc(mk));
        base = __shfl_sync(kFull, base, 0) + (unsigned)__popc(mk & ((1u << lane) - 1u));
        if (keep && (int)base < L.cand_cap) L.cand[base] = kv;
    }
}

// The bin of a byte histogram in which the running count reaches `rank`
// (warp 0: lane t sums bins 8t .. 8t + 7, a warp scan finds the lane), and the
// rank within the bin.  Block-wide; hist is not read after it returns.
__device__ __forceinline__ void find_bin(const int *hist, int rank, int *s_out, int &bin, int &rank_in)
{
    const int tid = threadIdx.x;
    if (tid < 32) {
        int s8 = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) s8 += hist[8 * tid + q];
        int incl = s8;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (tid >= o) incl += v;
        }
        const unsigned hit = __ballot_sync(kFull, incl >= rank);
        if (tid == __ffs(hit) - 1) {
            int cum = incl - s8;
            for (int q = 0; q < 8; ++q) {
                const int k = 8 * tid + q;
                if (cum + hist[k] >= rank) {
                    s_out[0] = k;
                    s_out[1] = rank - cum;
                    break;
                }
                cum += hist[k];
            }
        }
    }
    __syncthreads();
    bin = s_out[0];
    rank_in = s_out[1];
    __syncthreads();
}

// f(key) for every key of list[0, n), four loads in flight per thread
template <class F>
__device__ __forceinline__ void for_keys(const unsigned *list, int n, F f)
{
    for (int i0 = threadIdx.x; i0 < n; i0 += 4 * kOrbSelectThreads) {
        unsigned k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) k[u] = i0 + u * kOrbSelectThreads < n ? list[i0 + u * kOrbSelectThreads] : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + u * kOrbSelectThreads < n) f(k[u]);
    }
}

// The K-th smallest of the keys of list[0, n) whose bytes above byte `from`
// equal prefix's (keys are distinct), by an exact radix select on bytes
// from .. 0; rank: K among those keys.
__device__ unsigned kth_key(const unsigned *list, int n, unsigned prefix, int from, int rank, int *hist, int *s_out)
{
    unsigned mask = from == 3 ? 0u : 0xffffffffu << (8 * (from + 1));
    for (int b = from; b >= 0; --b) {
        if (threadIdx.x < 256) hist[threadIdx.x] = 0;
        __syncthreads();
        for_keys(list, n, [&](unsigned k) {
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> (8 * b)) & 255u], 1);
        });
        __syncthreads();
        int bin;
        find_bin(hist, rank, s_out, bin, rank);
        prefix |= (unsigned)bin << (8 * b);
        mask |= 255u << (8 * b);
    }
    return prefix;
}

// One block per (level, image).  The corners of a level are read twice: for a
// histogram of their top byte (the score), and to gather those that score
// above the deciding value and, apart, those that score exactly it, among
// which the remaining three bytes decide on chip.  A few hundred survivors are
// ranked by counting, all threads sharing the comparisons; more are sorted by
// a bitonic network.  What bounds it is the chain of block-wide steps: four
// histogram passes over device memory, a gather and a 45-step network took 24
// us for two images' levels, this form 14 us.
__global__ void __launch_bounds__(kOrbSelectThreads) orb_select_kernel(const OrbHeader *__restrict__ hdr)
{
    __shared__ __align__(16) unsigned keys[kOrbMaxSlots];
    __shared__ __align__(16) unsigned tied[kOrbMaxSlots];   // corners of the deciding score, then the ranks
    __shared__ int hist[256];
    __shared__ int s_out[2];
    __shared__ int s_n[2];
    const OrbHeader &H = *hdr;
    const int l = blockIdx.x;
    let_next_start();
    wait_for_previous();                // the detection's corners
    if (l >= H.nlevels) return;
    const OrbImage &I = H.images[blockIdx.y];
    const OrbLevel &L = I.lv[l];
    const int tid = threadIdx.x;
    const int c = min((int)I.cnt[l], L.cand_cap);
    const int K = L.max_kp;
    const unsigned *const cand = L.cand;
    if (tid < 256) hist[tid] = 0;
    if (tid < 2) s_n[tid] = 0;
    __syncthreads();
    auto keep = [&](unsigned k) {
        const int at = atomicAdd(&s_n[0], 1);
        if (at < kOrbMaxSlots) keys[at] = k;
    };
    if (K <= 0) {
        // no slots
    } else if (c <= K) {
        for_keys(cand, c, keep);
    } else {
        for_keys(cand, c, [&](unsigned k) { atomicAdd(&hist[k >> 24], 1); });
        __syncthreads();
        int bin, rank;
        find_bin(hist, K, s_out, bin, rank);
        const unsigned top = (unsigned)bin << 24;
        for_keys(cand, c, [&](unsigned k) {
            if (k < top) {
                keep(k);
            } else if (k >> 24 == (unsigned)bin) {
                const int at = atomicAdd(&s_n[1], 1);
                if (at < kOrbMaxSlots) tied[at] = k;
            }
        });
        __syncthreads();
        const int nt = s_n[1];
        if (nt == rank && nt <= kOrbMaxSlots) {
            for_keys(tied, nt, keep);
        } else {
            // more of them than fit on chip: select among them in device memory
            const bool on_chip = nt <= kOrbMaxSlots;
            const unsigned *list = on_chip ? tied : cand;
            const int n = on_chip ? nt : c;
            const unsigned kth = kth_key(list, n, top, 2, rank, hist, s_out);
            for_keys(list, n, [&](unsigned k) {
                if (k >= top && k <= kth) keep(k);
            });
        }
    }
    __syncthreads();
    const int n = min(s_n[0], K);
    unsigned *const sel = I.sel + L.slot0;
    if (n <= kOrbSelectThreads / 2) {
        // `parts` threads count, for each key, the smaller ones in a part of
        // the list each
        int p2 = 32;
        while (p2 < n) p2 <<= 1;
        const int parts = kOrbSelectThreads / p2, i = tid & (p2 - 1), part = tid / p2;
        if (tid < n) tied[tid] = 0u;
        if (tid < 4 && n + tid < kOrbMaxSlots) keys[n + tid] = 0xffffffffu;     // whole words of four
        __syncthreads();
        if (i < n) {
            const unsigned k = keys[i];
            unsigned smaller = 0;
            for (int j = 4 * part; j < n; j += 4 * parts) {
                const uint4 q = *reinterpret_cast<const uint4 *>(keys + j);
                smaller += (q.x < k) + (q.y < k) + (q.z < k) + (q.w < k);
            }
            atomicAdd(&tied[i], smaller);
        }
        __syncthreads();
        if (tid < n) sel[tied[tid]] = keys[tid];
    } else {
        int P = 1;
        while (P < n) P <<= 1;
        for (int i = n + tid; i < P; i += kOrbSelectThreads) keys[i] = 0xffffffffu;
        __syncthreads();
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = tid; i < P; i += kOrbSelectThreads) {
                    const int ixj = i ^ j;
                    if (ixj > i) {
                        const unsigned a = keys[i], b = keys[ixj];
                        if ((a > b) == ((i & k) == 0)) {
                            keys[i] = b;
                            keys[ixj] = a;
                        }
                    }
                }
                __syncthreads();
            }
        for (int i = tid; i < n; i += kOrbSelectThreads) sel[i] = keys[i];
    }
    if (tid == 0) {
        I.n_level[l] = n;
        atomicAdd(&I.n_level[H.nlevels], n);
    }
}

// Staged neighbourhoods of one keypoint (one warp): rows y - 15 .. y + 15 of
// the level for the moments and rows y - 18 .. y + 18 of the smoothed level
// for the tests (rotated pattern points within [-13, 13]^2 land within
// round(13 sqrt 2) = 18 pixels), each row copied from the 16-byte boundary at
// or before its first column.
constexpr int kMomR = 15, kTestR = 18;
constexpr int kMomRows = 2 * kMomR + 1, kTestRows = 2 * kTestR + 1;
constexpr int kMomChunks = 3, kTestChunks = 4;      // 16-byte chunks per staged row (31 + 15, 37 + 15 bytes)
constexpr int kMomStride = 16 * kMomChunks, kTestStride = 16 * kTestChunks;

// Byte masks of the disk's rows: entry v + 15, byte u + 15 is set if
// u^2 + v^2 <= 225 (entry 31 and byte 31 are empty).
struct DiskMask {
    unsigned w[32][8];
    constexpr DiskMask() : w()
    {
        for (int v = -kMomR; v <= kMomR; ++v)
            for (int u = -kMomR; u <= kMomR; ++u)
                if (u * u + v * v <= kMomR * kMomR) w[v + kMomR][(u + kMomR) / 4] |= 0xffu << (8 * ((u + kMomR) & 3));
    }
};
__device__ const DiskMask kDiskMaskTable __attribute__((aligned(16))) = DiskMask();
#define kDiskMask kDiskMaskTable.w

// Nearest integer, halves away from zero, for |x| < 2^22: the largest float
// below one half is added with x's sign and the sum truncated (the sum of a
// half and it rounds up to the next integer, of anything less it does not).
__device__ __forceinline__ int round_away(float x)
{
    return __float2int_rz(__fadd_rn(x, copysignf(__uint_as_float(0x3effffffu), x)));
}

__device__ __forceinline__ void copy16_async(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

__global__ void __launch_bounds__(32 * kDescribeWarps, 7) orb_describe_kernel(const OrbHeader *__restrict__ hdr)
{
    __shared__ __align__(16) uint8_t mom[kDescribeWarps][kMomRows * kMomStride];
    __shared__ __align__(16) uint8_t tst[kDescribeWarps][kTestRows * kTestStride];
    const OrbHeader &H = *hdr;
    const OrbImage &I = H.images[blockIdx.y];
    const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
    const int slot = blockIdx.x * kDescribeWarps + wv;
    wait_for_previous();                // the selection's keypoints
    if (slot >= I.nslots) return;
    int l = 0;
    for (int k = 0; k < H.nlevels; ++k)
        if (slot >= I.lv[k].slot0 && slot < I.lv[k].slot0 + I.lv[k].max_kp) l = k;
    const OrbLevel &L = I.lv[l];
    const int i = slot - L.slot0;
    if (i >= I.n_level[l]) {
        // a slot without a keypoint
        if (lane == 0) {
            I.x[slot] = -1.0e9f;
            I.y[slot] = -1.0e9f;
            I.oct[slot] = 0;
            I.score[slot] = -1;
            I.cs[2 * slot] = 1.0f;
            I.cs[2 * slot + 1] = 0.0f;
        }
        I.desc[(size_t)slot * 32 + lane] = 0;
        return;
    }
    const unsigned key = I.sel[slot];
    const int x = (int)(key & 4095u), y = (int)((key >> 12) & 4095u);
    // both neighbourhoods in one round trip, 8 rows of 4 chunks at a time;
    // keypoints lie at least 19 pixels inside the level, and a chunk that
    // holds a column of a row lies inside the row's 16-byte padded pitch
    const int a1 = (x - kMomR) & ~15, n1 = ((x + kMomR) >> 4) - (a1 >> 4) + 1;
    const int a0 = (x - kTestR) & ~15, n0 = ((x + kTestR) >> 4) - (a0 >> 4) + 1;
    const int ch = lane & 3, r0 = lane >> 2;
    {
        const uint8_t *src = L.img + (size_t)(y - kMomR + r0) * L.pitch + a1 + 16 * ch;
        uint8_t *dst = &mom[wv][r0 * kMomStride + 16 * ch];
        const size_t step = (size_t)8 * L.pitch;
#pragma unroll
        for (int r = 0; r < kMomRows; r += 8) {
            if (ch < n1 && r0 + r < kMomRows) copy16_async(dst + r * kMomStride, src);
            src += step;
        }
        src = L.smooth + (size_t)(y - kTestR + r0) * L.spitch + a0 + 16 * ch;
        dst = &tst[wv][r0 * kTestStride + 16 * ch];
        const size_t step2 = (size_t)8 * L.spitch;
#pragma unroll
        for (int r = 0; r < kTestRows; r += 8) {
            if (ch < n0 && r0 + r < kTestRows) copy16_async(dst + r * kTestStride, src);
            src += step2;
        }
    }
    // the disk's bytes of this lane's row (row v of the disk: |u| <= the
    // largest with u^2 + v^2 <= 225)
    const uint4 k0 = __ldg(reinterpret_cast<const uint4 *>(kDiskMask[lane])), k1 = __ldg(reinterpret_cast<const uint4 *>(kDiskMask[lane]) + 1);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncwarp();
    // intensity centroid over the disk u^2 + v^2 <= 225 (exact integer sums):
    // lane v + 15 takes row v, four pixels a dot product (lane 31 has an
    // empty mask); the row's bytes are realigned to its first column
    int m10 = 0, m01 = 0;
    {
        const uint4 *row = reinterpret_cast<const uint4 *>(&mom[wv][min(lane, kMomRows - 1) * kMomStride]);
        const uint4 q0 = row[0], q1 = row[1], q2 = row[2];
        const unsigned raw[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
        const unsigned msk[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
        const int off = x - kMomR - a1;                     // 0 .. 15, the same in the warp
        const unsigned sh = 8u * (unsigned)(off & 3);
        unsigned sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            // words i + off / 4 and the next one (a select by the two bits of off / 4)
            const unsigned lo = off & 8 ? (off & 4 ? raw[i + 3] : raw[i + 2]) : (off & 4 ? raw[i + 1] : raw[i]);
            const unsigned hi = off & 8 ? (off & 4 ? (i + 4 < 12 ? raw[i + 4 < 12 ? i + 4 : 11] : 0u) : raw[i + 3])
                                        : (off & 4 ? raw[i + 2] : raw[i + 1]);
            const unsigned p = __funnelshift_r(lo, hi, sh) & msk[i];
            // columns u = 4 i - 15 .. 4 i - 12
            const int u = 4 * i - kMomR;
            const unsigned uw = ((unsigned)u & 0xffu) | ((unsigned)(u + 1) & 0xffu) << 8 | ((unsigned)(u + 2) & 0xffu) << 16 |
                                ((unsigned)(u + 3) & 0xffu) << 24;
            asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(m10) : "r"(p), "r"(uw));
            sum = __dp4a(p, 0x01010101u, sum);
        }
        m01 = (lane - kMomR) * (int)sum;
    }
    m10 = __reduce_add_sync(kFull, m10);
    m01 = __reduce_add_sync(kFull, m01);
    float c = 1.0f, s = 0.0f;
    if (m10 != 0 || m01 != 0) {
        // |m| = sqrt(m10^2 + m01^2) as the double square root rounded to
        // float, which for these integers is the correctly rounded FP32
        // square root (ft_sqrt.h)
        const float nm = float_sqrt_rn((uint64_t)((long long)m10 * m10 + (long long)m01 * m01));
        c = __fdiv_rn((float)m10, nm);
        s = __fdiv_rn((float)m01, nm);
    }
    // byte `lane` of the descriptor: tests 8 lane .. 8 lane + 7 (their 32
    // pattern coordinates in two 16-byte loads)
    const uint8_t *tp = &tst[wv][kTestR * kTestStride + (x - a0)];
    const uint4 *pw = reinterpret_cast<const uint4 *>(H.pattern) + 2 * lane;
    const uint4 pa = __ldg(pw), pb = __ldg(pw + 1);
    const unsigned pws[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
    unsigned byte = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        int val[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            // test point q: bytes 2q (x) and 2q + 1 (y) of the test's word, signed
            const int xi = (int)(pws[k] << (24 - 16 * q)) >> 24, yi = (int)(pws[k] << (16 - 16 * q)) >> 24;
            const float px = (float)xi, py = (float)yi;
            const int u = round_away(__fsub_rn(__fmul_rn(c, px), __fmul_rn(s, py)));
            const int v = round_away(__fadd_rn(__fmul_rn(s, px), __fmul_rn(c, py)));
            val[q] = tp[v * kTestStride + u];
        }
        byte |= (val[0] < val[1] ? 1u : 0u) << k;
    }
    I.desc[(size_t)slot * 32 + lane] = (uint8_t)byte;
    if (lane == 0) {
        I.x[slot] = __fmul_rn((float)x, H.sc[l]);
        I.y[slot] = __fmul_rn((float)y, H.sc[l]);
        I.oct[slot] = (int8_t)l;
        I.score[slot] = 255 - (int)(key >> 24);
        I.cs[2 * slot] = c;
        I.cs[2 * slot + 1] = s;
    }
}

}  // namespace

cudaError_t launch_orb(const OrbHeader *dev_hdr, int nimages, int nlevels, int max_tiles, int max_slots,
                       cudaStream_t stream)
{
    if (nimages <= 0) return cudaSuccess;
    orb_detect_kernel<<<dim3((unsigned)max(max_tiles, 1), (unsigned)nimages), kDetThreads, 0, stream>>>(
        dev_hdr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    OverlapLaunch select(dim3((unsigned)nlevels, (unsigned)nimages), kOrbSelectThreads, 0, stream, true);
    e = select.run(orb_select_kernel, dev_hdr);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)((max(max_slots, 1) + kDescribeWarps - 1) / kDescribeWarps);
    OverlapLaunch describe(dim3(blocks, (unsigned)nimages), 32 * kDescribeWarps, 0, stream, true);
    return describe.run(orb_describe_kernel, dev_hdr);
}

}  // namespace ft
