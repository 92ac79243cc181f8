// ft_internal.h -- structures shared by the library's host and device code.
//
// One persistent kernel runs the index, pinhole stereo, search and resolve
// work of every entry point; pyramids, fisheye matching and pose optimization
// are kernels before and after it, and extraction has three of its own.  The
// host writes a "batch table" (header, per-frame descriptors, per-kind work
// prefixes, zeroed counters) into pinned memory and copies it to the slot's
// device table; a call of one frame passes its header and descriptor as kernel
// parameters instead.  The fused kernel's CTAs pull work items from a queue (an
// atomic head counter) in a fixed order: row sorts and grid builds, stereo
// items, search items, resolve items.  An item waits only on items that sit
// before it in the queue, so the queue drains without deadlock whatever the
// number of resident CTAs.
#pragma once

#include <cstddef>
#include <cstdint>

#include "fasttrack.h"

#include <cuda_runtime.h>

namespace ft {

constexpr int kThreads = 256;                       // threads per CTA
constexpr int kWarps = kThreads / 32;
constexpr int kCells = FT_GRID_COLS * FT_GRID_ROWS; // 3072 grid cells
constexpr int kStageCap = 512;                      // right keypoints staged per stereo item
constexpr int kMaxRows = 4096;                      // image rows the row sort handles
constexpr int kWinRows = 192;                       // rows of a stereo item's staged window
constexpr int kOctBuckets = 8;                      // octaves a staged window separates
constexpr int kFoldResolveMax = 8192;               // frames up to this size resolve in their last search item
constexpr int kCounters = 8;                        // per-frame counters (u32)
constexpr int kRowSortItems = 4;                    // row-sort work items per pinhole frame (2 per side)
constexpr int kPyrThreads = 256;                    // threads per pyramid block
constexpr int kPyrTileRows = 16;                    // source rows a pyramid block owns
constexpr int kPyrTileCols = 752;                   // source columns a pyramid block owns (a multiple of 16)
constexpr int kPyrRowsPerLevel = 2 * kPyrTileRows;  // output rows of one level in a tile, at most

// Tiles of a pyramid's level 0 (one pyramid block each).
__host__ __device__ inline int pyr_tiles(int W, int H)
{
    return ((H + kPyrTileRows - 1) / kPyrTileRows) * ((W + kPyrTileCols - 1) / kPyrTileCols);
}
// Byte offsets within one pyramid image are 32-bit in the pyramid kernel.
constexpr long long kPyrMaxLevelBytes = 1ll << 31;

// work item kinds, in queue order
enum Kind { K_INDEX = 0, K_STEREO = 1, K_SEARCH = 2, K_RESOLVE = 3, K_KINDS = 4 };

// per-frame counter slots
enum Ctr { C_GRID_DONE = 0, C_STEREO_DONE = 1, C_STEREO_READY = 2, C_SEARCH_DONE0 = 3,
           C_SEARCH_DONE1 = 4, C_ROWS_DONE = 5 };

// device status bits (ORed into the context's status word)
constexpr unsigned kStatusTimeout = 1u;

// debug flags of the batch header
constexpr unsigned kDebugWithholdStereoReady = 1u;   // never publish stereo-ready

struct DevParams {
    int nlevels, th_stereo, th_search, ratio_any_octave;
    float sc[FT_MAX_LEVELS], isc[FT_MAX_LEVELS], band_r[FT_MAX_LEVELS];
    float median_factor, fisheye_ratio, nn_ratio, search_th;
    float view_cos_min, view_cos_narrow, radius_narrow, radius_wide, dist_lo, dist_hi;
    float th_last;
    int kb_iters;
    float min_depth;
    int po_rounds, po_iters, po_huber;
    float po_chi2_mono, po_chi2_stereo;
    int halo;            // rows a right keypoint's band can reach beyond floor(y), any octave
    int halo_oct[FT_MAX_LEVELS];   // same for the octave window of a left keypoint of octave o
    int halo_c[FT_MAX_LEVELS];     // same for a right keypoint of octave o
};

// One camera of the search step (pinhole: the left camera only).
struct CamDev {
    int model;           // ft_camera_model
    int nk;
    float fx, fy, cx, cy, bf;
    float k[4];
    float minx, maxx, miny, maxy;
    float iw, ih;        // grid cells per pixel (computed on the device)
    float R[9], t[3], O[3];
    const float *kx, *ky;
    const int8_t *koct;
    const uint4 *kdesc;
    const uint8_t *taken;
    int8_t *level;
    float4 *proj;
    int *mp_kp, *mp_d1, *mp_d2, *kp_mp;
    // the keypoint grid (scratch), in cell order; keypoints already taken
    // are left out
    int *cell_ptr;                 // [kCells + 1] cell starts, 16-byte aligned
    unsigned *gq;                  // [nk] packed place and octave of each placed keypoint (see pack_place)
    uint16_t *gk16;                // [nk] its index (nk < 65536, else NULL); this and gq in whole 16-byte chunks
    int *gk32;                     // [nk] its index (nk >= 65536, else NULL)
    unsigned long long *owner;     // [nk] (distance << 32) | map index
    uint4 *scan;                   // [2 * nm] split search: per map point its four smallest candidate keys,
                                   // then (right coordinate, radius, how many passed, 0)
};

struct FrameDev {
    int camera, do_stereo, do_search, wait_stereo;
    int nl, nr, nm, ncam;
    // stereo inputs
    const float *lx, *ly, *rx, *ry;
    const int8_t *loct, *roct;
    const uint4 *ldesc, *rdesc;
    const uint8_t *pyrL[FT_MAX_LEVELS], *pyrR[FT_MAX_LEVELS];
    int lw[FT_MAX_LEVELS], lh[FT_MAX_LEVELS], lp[FT_MAX_LEVELS];
    int rw[FT_MAX_LEVELS], rh[FT_MAX_LEVELS], rp[FT_MAX_LEVELS];
    int H;
    float b, bf;
    float lap_l0, lap_l1, lap_r0, lap_r1;
    // row sort of the pinhole stereo step (scratch): keypoints bucketed by row
    int *row_ptr_l, *row_ptr_r;    // [H + 1]
    float4 *ls_kp;                 // [nl] left x, y, index, octave in row order
    uint4 *ls_desc;                // [2 * nl]
    float4 *rs_kp;                 // [nr] right x, band rows lo | hi << 16, row, index | octave << 20
    uint4 *rs_desc;                // [2 * nr]
    // stereo outputs (pinhole)
    int *best_r, *dist, *sad_shift, *sad_best;
    float *u_right, *depth;
    // stereo outputs (fisheye)
    int *r_idx, *fd1, *fd2;
    float *fdepth;                 // triangulated depth per left keypoint (NULL: no triangulation)
    float4 *fxyz;                  // triangulated point (may be NULL)
    float kbl[8], kbr[8];          // fx, fy, cx, cy, k1..k4 of the left and right fisheye cameras
    // search
    const float *u_right_in;       // stereo consistency input (NULL: none)
    int build_pyr;                 // levels 1.. built from level 0 before the launch: bit 0 left, bit 1 right
    int search_mode;               // 0: local map; 1: the last frame's points
    const int8_t *last_oct;        // last mode: octave of each point's last observation
    float last_R[9], last_t[3];    // last mode: the last frame's pose
    float base;                    // stereo baseline (the motion test of the last mode)
    float R_rl[9], t_rl[3];        // fisheye rig (right camera pose is composed on the device)
    CamDev cam[2];
    const float4 *pos, *nrm;
    const uint4 *mdesc;
    const uint8_t *skip;
    // work decomposition
    int strip_rows, n_stereo_items;
    int search_tile, resolve_tile;
    int rowsort;                   // row-sort index items (kRowSortItems: the first half the left
                                   // keypoints, the second half the right ones), 0 without stereo
    int fold_resolve;              // 1: the last search item of a camera writes the final tables
    int split_search;              // 1: search items scan their candidates before waiting for the stereo
                                   // step and apply the stereo consistency after it
    int n_grid_items, n_index_items, n_search_items[2], n_resolve_items[2];
    unsigned *ctr;                 // [kCounters]
    // pose optimization (next row f4): the pose kernel, launched after the
    // fused kernel, takes one cluster per frame with do_pose (pinhole frames)
    int do_pose;
    const int *po_mp_kp;           // [nm] matches: map point -> keypoint (cam[0])
    float *po_Rt;                  // [12] out: R row-major, t
    int8_t *po_inlier;             // [nm] out: 1 inlier, 0 outlier, -1 unmatched
    int *po_n;                     // [1] out: inliers
    float4 *po_list;               // [2 * nm] scratch: observations in map-point order
};

struct BatchHeader {
    DevParams p;
    int nframes, total_items;
    int kind_begin[K_KINDS + 1];
    unsigned debug_flags;
    const int *prefix;             // [K_KINDS][nframes + 1]
    const FrameDev *frames;
    unsigned *queue;               // [0]: next item, [1]: trace records written
    unsigned *status;              // context status word (persistent, not in the table)
    unsigned long long timeout_ns; // bound of every device-side wait
    ft_trace_record *trace;        // NULL: tracing off
    int trace_cap;
    int pad_;
};

// A call of one frame: its header and descriptor travel as kernel parameters
// (no table copy ahead of the kernel, and no descriptor loads in it).  Its
// queue and counters are a few words of the arena that are zero between
// launches: the fused kernel's last block zeroes them again.
struct FrameCall {
    BatchHeader h;                 // prefix and frames are not used; queue[2] counts finished blocks
    FrameDev f;
};
static_assert(sizeof(FrameCall) <= 4096, "a frame's call exceeds the kernel parameters");

// ---------------------------------------------------------------- f3: keypoint extraction
constexpr int kOrbTileW = 62;           // detection tile: with its suppression ring 64 x 32 pixels
constexpr int kOrbTileH = 30;
constexpr int kOrbHalo = 4;             // FAST circle (3) + suppression neighbours (1)
constexpr int kOrbMaxDim = 4096;        // level sizes the 12-bit key coordinates allow
constexpr int kOrbMaxSlots = 4096;      // slots per level (sorted in shared memory)
constexpr int kOrbSelectThreads = 1024;

// One pyramid level of an image being described.
struct OrbLevel {
    const uint8_t *img;                 // level image
    int w, h, pitch;
    uint8_t *smooth;                    // [h][spitch] binomial-smoothed level (scratch)
    int spitch;                         // its row pitch: w rounded up to 16 bytes
    unsigned *cand;                     // [cand_cap] suppressed corners as keys (scratch)
    int cand_cap;
    int tiles_x, tile0;                 // tiles per row, first tile of the level in the image
    unsigned tiles_x_inv;               // ceil(2^32 / tiles_x) (tiles_x 1: 0, handled by the kernel)
    int slot0, max_kp;                  // first output slot of the level and its slots
};

struct OrbImage {
    alignas(16) int tile0[FT_MAX_LEVELS];   // first tile of each level (levels that do not exist: past all tiles)
    OrbLevel lv[FT_MAX_LEVELS];
    int tiles, nslots;
    float *x, *y;                       // outputs, [nslots] each
    int8_t *oct;
    int *score;
    float *cs;                          // [nslots][2]
    uint8_t *desc;                      // [nslots][32]
    int *n_level;                       // [nlevels + 1]
    unsigned *sel;                      // [nslots] selected keys in slot order (scratch)
    unsigned *cnt;                      // [nlevels] candidate counters (zeroed by the table copy)
};

struct OrbHeader {
    int nimages, nlevels, fast_th, edge, max_tiles, max_slots;
    float sc[FT_MAX_LEVELS];
    alignas(16) int8_t pattern[256 * 4];      // test i: x1, y1, x2, y2 at 4 i (16-byte aligned: vector loads)
    const OrbImage *images;
};

}  // namespace ft

// Kernels of one call overlap their launches (programmatic dependent launch):
// a kernel lets the call's next one start when all its blocks run, and waits
// for the ones before it only where it needs their results, at the latest
// before it ends, so that a kernel's end is the end of all before it.  A wait
// in a kernel launched the ordinary way returns at once.  The pose kernel is
// launched the ordinary way: started early, its clusters crowd on the SMs that
// the fused kernel leaves first (16 frames with pose: 136 us, early 146 us).
// Measured against ordinary launches: 32 fisheye frames 92.5 -> 76.8 us (the
// matching, 128 threads a block, and the search share the chip), 64 frames from
// images with pose 335 -> 327 us (index and Hamming phases beside the pyramids).
namespace ft {
#ifdef __CUDACC__
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif
// launch attributes: the kernel may start before the stream's previous one ends
struct OverlapLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    OverlapLaunch(dim3 grid, int threads, size_t smem, cudaStream_t stream, bool overlap)
    {
        cfg.gridDim = grid;
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = overlap ? 1 : 0;
    }
    void cluster(unsigned x, unsigned y, unsigned z)
    {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = x;
        attr[cfg.numAttrs].val.clusterDim.y = y;
        attr[cfg.numAttrs].val.clusterDim.z = z;
        ++cfg.numAttrs;
    }
    template <class... P, class... A>
    cudaError_t run(void (*kernel)(P...), const A &...args)
    {
        return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess ? cudaSuccess : cudaGetLastError();
    }
};
}  // namespace ft

// Copies a batch table from pinned host memory (bytes rounded up to whole 16).
namespace ft {
cudaError_t launch_table_copy(void *dst, const void *pinned, size_t bytes, cudaStream_t stream);
}  // namespace ft

// Launch helpers implemented in ft_kernels.cu (host-callable).  overlap: the
// call's previous kernel lets this one start before it ends.
namespace ft {
cudaError_t launch_fused(const BatchHeader *dev_hdr, int grid, cudaStream_t stream, bool overlap = false);
cudaError_t launch_fused(const FrameCall &call, int grid, cudaStream_t stream, bool overlap);
cudaError_t launch_pose(const FrameCall &call, cudaStream_t stream);
cudaError_t launch_fisheye(const FrameCall &call, int blocks, cudaStream_t stream);
cudaError_t launch_pyramids(const FrameCall &call, int tiles_per_image, cudaStream_t stream);
// pose optimization of the frames with do_pose (one cluster per frame of the
// first nframes; after the fused kernel on the same stream)
cudaError_t launch_pose(const BatchHeader *dev_hdr, int nframes, cudaStream_t stream);
// levels 1.. of the pyramids of the frames that build them (before the fused
// launch); blocks_per_image blocks stride over each image's virtual blocks
cudaError_t launch_pyramids(const BatchHeader *dev_hdr, int nframes, int nlevels, int tiles_per_image,
                            cudaStream_t stream);
// brute-force matching and triangulation of the fisheye frames among the first
// nframes (any order with the fused kernel: neither reads the other's
// outputs); blocks: of the frame with the most left keypoints
cudaError_t launch_fisheye(const BatchHeader *dev_hdr, int nframes, int blocks, cudaStream_t stream, bool overlap);
int fisheye_blocks(int nl);    // blocks of a frame of nl left keypoints
cudaError_t fisheye_setup();   // the fisheye kernel's shared-memory attribute (once per context)
cudaError_t pyramid_setup();   // the pyramid kernel's shared-memory attribute (once per context)
int fused_smem_bytes();
// device set-up of the fused and pose kernels (shared-memory attributes),
// then the fused kernel's resident CTAs per SM
cudaError_t fused_occupancy(int *ctas_per_sm);
const void *fused_kernel_ptr();
// keypoint extraction of the images of an OrbHeader (ft_orb.cu): detection,
// selection and description, three launches on the stream
cudaError_t launch_orb(const OrbHeader *dev_hdr, int nimages, int nlevels, int max_tiles, int max_slots,
                       cudaStream_t stream);
// set the text ft_last_error() returns on this thread (ft_api.cu)
void set_last_error(const char *msg);
// host checks and derived tables shared by the entry points (ft_api.cu)
ft_status check_params(const ft_params &p);   // FT_EINVAL + ft_last_error() text on a bad field
DevParams make_dev_params(const ft_params &p);
int strip_rows_for(long long rows);
int stereo_strip_rows(int want, int H, int nr, int halo);
}  // namespace ft
