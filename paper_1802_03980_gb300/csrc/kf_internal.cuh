// Internal device-side structures of the tracking library (not part of the ABI).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kf_track.h"

namespace kf {

constexpr int kSums = 29;           // 21 upper(A^T A) + 6 A^T b + n + sum b^2
// Work-item partial sums, one row of 32 floats (29 used) per warp of the
// block that ran the item, in two slots: slot A (offset 0) holds the
// association pass's sums of the pixels surely inside the band, slot B
// (offset kSlotB) the reduction pass's sums (the window pixels, or the whole
// band). Per-warp rows keep the passes free of block barriers; the combine
// adds them in a fixed order.
constexpr int kBlockWarps = 8;      // warps per block of the ICP kernels
constexpr int kSlotB = kBlockWarps * 32;
constexpr int kPartialStride = 2 * kSlotB;  // floats per work-item partial
constexpr int kBlock = kBlockWarps * 32;  // threads per block of the ICP kernels
constexpr int kChunk = 4096;        // frame pixels per work item at level 0
// Coarser levels use smaller items so that their (4x, 16x fewer) pixels still
// spread over enough blocks: 4096, 2048, 1024, 1024.
__host__ __device__ constexpr int level_chunk(int level) {
  return (kChunk >> level) > 1024 ? (kChunk >> level) : 1024;
}
constexpr int kMaxBins = 4096;
// Default band-edge windows of the association pass (KParams::win_*): the
// next iteration at a level expects its edge within [g - 5, g + 3] of this
// one's, a finer level's first iteration within [g - 8, g + 2] of the
// coarser level's last edge.
#ifndef KF_WIN_SAME_BELOW
#define KF_WIN_SAME_BELOW 5
#endif
#ifndef KF_WIN_SAME_ABOVE
#define KF_WIN_SAME_ABOVE 3
#endif
#ifndef KF_WIN_NEXT_BELOW
#define KF_WIN_NEXT_BELOW 8
#endif
#ifndef KF_WIN_NEXT_ABOVE
#define KF_WIN_NEXT_ABOVE 2
#endif
constexpr int kMaxWindow = 8;
constexpr int kDescListMax = 64;    // pairs per front-end launch

// Maps of one pyramid level: a pixel's vertex and normal as two records, A =
// (v.x, v.y, v.z, n.x) and B = (n.y, n.z), in float32 (16 and 8 bytes) or
// float16 (8 and 4). One wide load or store a record instead of one a
// component: a gather of a model pixel is two instructions and addresses
// instead of six, the front end's output three stores instead of seven, a
// normal-shooting candidate one load instead of three.
struct LevelMaps {
  int fw, fh;                 // frame level size
  int mw, mh;                 // model level size
  float ffx, ffy, fcx, fcy;   // frame level intrinsics (vertex map)
  float fifx, fify;           // 1 / ffx and 1 / ffy, rounded once
  float mfx, mfy, mcx, mcy;   // model level intrinsics (projection)
  float* fdepth;              // filtered depth, fw * fh
  void* fA;                   // frame records, camera frame; vertex and normal NaN where
  void* fB;                   // either is invalid
  void* mA;                   // model records, world frame; NaN at holes
  void* mB;
};

struct PairState {
  double T[12];               // current estimate, 3x4 row-major camera->world
  float xf[24];               // float32 Rw[9] tw[3] (camera->world) Rr[9] tr[3]
                              // (camera->model camera) used by the decisions
  double lambda_c;
  int cur_level;              // level being iterated, -1 when finished
  int stopped;                // 1 after an error stop
  int status;
  int iters[KF_MAX_LEVELS];
  int median_bin[KF_MAX_LEVELS];
  int total_iters;
  int hist_len;
  int kmed_hist[kMaxWindow];
  int N, kmed, klo, khi;      // current iteration (written by the histogram stage)
  int w0, w1;                 // band-edge window of the current iteration: the
                              // association pass sums bins < w0 and records bins
                              // in [w0, w1); w0 = -1: no window (histogram only)
  int hit;                    // 1: the band edge fell in the window, the
                              // reduction pass adds the recorded pixels only
  int valid_pairs, inliers;   // last completed iteration
  double sb2;                 // sum b^2 over its inliers
  double dbg_sums[kSums];     // filled by the reduction stage in inspection mode
  double prior_R[9];          // IMU prior rotation (valid when has_prior)
  int has_prior;
  int pad2_;
  int trace_len;
  int pad_;
  kf_iter_record trace[KF_TRACE_MAX];
};

struct PairDesc {
  LevelMaps lv[KF_MAX_LEVELS];
  int levels;
  int iw, ih;                 // level-0 frame size
  const float* depth_raw;     // level-0 raw depth (tracker buffer)
  double Tm[12];              // model pose 3x4 camera->world
  PairState* st;
  unsigned* hist;             // [bins]
  float* partials;            // [items][kPartialStride]
  unsigned* counters;         // [2]: histogram stage, reduction stage
  float4* recs;               // [2 * rec_cap] records of the window pixels:
                              // row a[0..5], b and bin (int bits), written by the
                              // association pass, read by the reduction pass;
                              // warp w of item li packs its records from place
                              // li * chunk + w * chunk / kBlockWarps (in a team
                              // launch a block's are its own, see TeamPair)
  unsigned* wcount;           // [items * kBlockWarps] records per item and warp
  // team launch (null when the tracker's frames are too large for it): rotating
  // histograms, the leader's message and the half items' sums (packets
  // of a value and its tag), all zero between launches but for the packets
  unsigned* team_hist;        // [kTeamHists * team_hist_words(bins)]
  unsigned long long* team_msg;   // [32]
  unsigned long long* team_rows;  // [2 * items * 32]
  int* dbg_index;             // [iw*ih] inspection outputs (may be null)
  int* dbg_bin;
  int partial_cap;            // work-item partials the buffer holds
  int px_cap;                 // frame pixels dbg_* hold
  int rec_cap;                // record places
  int pad_;
};

// Active work list of one launch, built on the device (int buffer):
//   [0] items in the list  [1] pairs in the list  [2] level  [3] unused
//   [4 .. 4+cap)            pair index (into the descriptor list) per entry
//   [4+cap .. 4+2cap+1)     item prefix: entry s owns items [prefix[s], prefix[s+1])
// Item j of a pair at level l covers frame pixels [j c, min(w h, (j+1) c)),
// c = level_chunk(l).
__host__ __device__ constexpr int list_ints(int cap) { return 4 + 2 * cap + 1; }

// Queue of the scheduled ICP launch: header words (each on its own 128-byte
// line), then a ring of 64-bit task slots. Zeroed before each launch.
constexpr int kQHead = 0;    // next ticket to claim
constexpr int kQTail = 32;   // next ticket to reserve
constexpr int kQDone = 64;   // pairs finished
constexpr int kQErr = 96;    // 1: a bounded wait ran out
constexpr int kQSeed = 128;  // next pair to seed
constexpr int kQHeaderWords = 256;
constexpr int kMaxItemsPerLevel = 131071;  // 17-bit item field of a task
constexpr int kMaxSchedPairs = 65535;      // 16-bit pair field

// Team launch (kf_team.cu): words of one histogram (the bins to a multiple of
// four, then the count of unmatched pixels), half items a worker block can
// take, pairs of a launch.
__host__ __device__ constexpr int team_hist_none(int bins) { return (bins + 3) / 4 * 4; }
__host__ __device__ constexpr int team_hist_words(int bins) { return team_hist_none(bins) + 4; }
constexpr unsigned kTeamHists = 16;   // rotating histograms, a power of two
constexpr unsigned kTeamAcquire = 8;  // iterations between two acquires, a power of two
static_assert(kTeamHists >= kTeamAcquire + 1 + 2, "a clear comes before the messages of two iterations on");
// Half items of a worker at most: beyond, the queue's blocks, which share all
// items of all pairs, come near the team's whole slots. Measured on GB300, set
// frame and align of a batch, team against queue, us: one slot a worker 162 / 302
// (one pair 640x480), two 183 / 338 (700x525), 178 / 321 (800x600) and 179 / 314
// (two 640x480), four 272 / 430 (1280x960), seven 417 / 580 (1920x1080) and 356 /
// 434 (six 640x480), eight 391 / 456 (seven).
constexpr int kTeamSlots = 8;
constexpr int kTeamPlaces = level_chunk(0) / kBlockWarps;  // record places of an item warp, at any level
constexpr int kTeamMaxItems = 1024;  // items of the largest frame
// pairs whose inputs go with the launch; 16 pairs 320x240: 308 us team, 424 queue,
// 160x120: 256 and 424
constexpr int kTeamMaxPairs = 16;

struct DescList {
  const PairDesc* d[kDescListMax];
  const float* depth[kDescListMax];  // level-0 raw depth of each pair (device)
  int n;
};

// Parameters shared by every kernel, passed by value.
struct KParams {
  int levels;
  int caps[KF_MAX_LEVELS];
  int bins;
  float d_max32;
  float scale32;              // (float)(bins / d_max)
  int tiny_bins;              // d_max or a bin's width at or below 2^-49
  double kappa;
  int kappa_one;              // kappa == 1
  float cos_min32;
  int use_angle;
  int conv_window;
  int lambda_mode;
  int n_min;
  unsigned flags;
  int precision;
  // band-edge windows of the association pass: the next iteration at the
  // same level expects its band edge in [g - below, g + above] around this
  // iteration's edge g; the first iteration of a finer level around the
  // coarser level's last edge
  int split_ok;               // a window can hit (the band always starts at bin 0)
  int win_same_below, win_same_above, win_next_below, win_next_above;
  // front end
  int bil_radius;
  float bil_inv2sr2;          // 1 / (2 sigma_r^2)
  float bil_sw[81];           // -(dx^2 + dy^2) / (2 sigma_s^2), (2r+1)^2 entries
  float bil_sw2[81];          // the same times log2(e) (exponent for exp2)
  float bil_nsw[33];          // (dx^2 + dy^2) log2(e) / (2 sigma_s^2) by dx^2 + dy^2
  float bil_c2;               // log2(e) / (2 sigma_r^2)
  float bil_k;                // sqrt(bil_c2): the range term is (k zn - k z)^2
  float thr3sr32;             // (float)(3 sigma_r)
  // normals and association variants
  int normal_mode;            // KF_NORMALS_CROSS | KF_NORMALS_INTEGRAL
  float ii_a, ii_b;           // window half-size a + b z at level 0
  float ii_delta;             // relative depth change of an edge
  int ii_rmax;                // cap on the half-size
  int shoot_w;                // normal-shooting window half-size (0: projective)
};

// d_max or a bin's width at or below 2^-49 (KParams::tiny_bins)
inline bool tiny_bins(float d_max32, float scale32) { return !(d_max32 > 0x1p-49f && scale32 < 0x1p49f); }

struct PairInput {
  double prior_R[9];
  double init[16];
  double lambda;
  int has_prior;
  int pad_;
};

struct PairOutput;

// One pair of a team launch: its blocks are [first, first + 1 + workers), the
// first its leader; a worker takes up to `slots` half items, worker w's records
// of the s-th at places (w slots + s) 4 kTeamPlaces on. tag: distinguishes this launch's packets from all earlier
// ones (plus an iteration's number, below kTeamTags).
struct TeamPair {
  const PairDesc* d;
  PairOutput* out;
  unsigned tag;
  int first, workers, slots;
};
constexpr unsigned kTeamTags = 4096;  // > the iterations of an alignment + 1

struct TeamArgs {
  TeamPair pair[kTeamMaxPairs];
  PairInput in[kTeamMaxPairs];
  int n;
  unsigned long long limit_ns;
};

struct PairOutput {
  double pose[16];
  kf_result res;
};

// ---- checked builds (-DKF_CHECKED): guarded accesses record the first
// violation (code and two values) in a device fault word and are skipped;
// the host reports it as KF_ERR_INTERNAL. Unchecked builds compile the guard
// away and the access runs unconditionally.
#ifdef KF_CHECKED
#define KF_GUARD(cond, code, a, b) \
  if (!(cond)) {                   \
    kf_fault((code), (a), (b));    \
  } else
#else
#define KF_GUARD(cond, code, a, b)
#endif
#ifdef KF_CHECKED
void checked_fault_team(long long out[3]);
#endif
// host side of checked builds: copies and clears the fault word (0 = none)
void checked_fault(long long out[3]);

// ---- storage-type helpers -------------------------------------------------
template <class T> struct Store;
template <> struct Store<float> {
  using A = float4;
  using B = float2;
  static __device__ __forceinline__ float4 value_a(float4 w) { return w; }
  static __device__ __forceinline__ float2 value_b(float2 w) { return w; }
  static __device__ __forceinline__ float4 load_a(const void* p, int i) { return __ldg(static_cast<const float4*>(p) + i); }
  static __device__ __forceinline__ float2 load_b(const void* p, int i) { return __ldg(static_cast<const float2*>(p) + i); }
  static __device__ __forceinline__ void store_a(void* p, int i, float4 v) { static_cast<float4*>(p)[i] = v; }
  static __device__ __forceinline__ void store_b(void* p, int i, float2 v) { static_cast<float2*>(p)[i] = v; }
};
template <> struct Store<__half> {
  using A = uint2;
  using B = unsigned;
  static __device__ __forceinline__ float2 pair(unsigned w) {
    return __half22float2(*reinterpret_cast<const __half2*>(&w));
  }
  static __device__ __forceinline__ unsigned pack(float x, float y) {
    const __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<const unsigned*>(&h);
  }
  static __device__ __forceinline__ float4 value_a(uint2 w) {
    const float2 a = pair(w.x), b = pair(w.y);
    return make_float4(a.x, a.y, b.x, b.y);
  }
  static __device__ __forceinline__ float2 value_b(unsigned w) { return pair(w); }
  static __device__ __forceinline__ float4 load_a(const void* p, int i) {
    return value_a(__ldg(static_cast<const uint2*>(p) + i));
  }
  static __device__ __forceinline__ float2 load_b(const void* p, int i) {
    return value_b(__ldg(static_cast<const unsigned*>(p) + i));
  }
  static __device__ __forceinline__ void store_a(void* p, int i, float4 v) {
    static_cast<uint2*>(p)[i] = make_uint2(pack(v.x, v.y), pack(v.z, v.w));
  }
  static __device__ __forceinline__ void store_b(void* p, int i, float2 v) {
    static_cast<unsigned*>(p)[i] = pack(v.x, v.y);
  }
};

}  // namespace kf

// ---- launchers implemented in the .cu files ---------------------------------
namespace kf {
// Frames of a batch pulled from page-locked host memory into device buffers
// by one kernel (16-byte loads, several in flight per thread), instead of
// one copy per frame issued by the host.
constexpr int kPullMax = 32;                 // page-locked host frames per launch, and the
constexpr long long kPullPixels = 1200000;   // pixels from which on a launch takes no more
struct FrameCopyList {
  const float* src[kPullMax];
  float* dst[kPullMax];
  int count[kPullMax];  // floats
  int n;
  int layers;           // of the front end's grid (launch_frontend)
};
cudaError_t launch_copy_frames(const FrameCopyList& list, cudaStream_t s);
// next: page-locked host frames of a later launch, copied by a few of this one's
// blocks meanwhile
cudaError_t launch_frontend(const DescList& list, const FrameCopyList& next, int max_w, int max_h, int levels,
                            const KParams& P, cudaStream_t s);
// integral-image normals of every level of the listed frames (after the
// front end): replaces the frame normals and drops vertices without one
cudaError_t launch_integral_normals(const DescList& list, int max_w, int max_h, int levels,
                                    const KParams& P, cudaStream_t s);
// the model's records of every level, and the pair's device descriptor := desc
cudaError_t launch_model_prep(const PairDesc& desc, PairDesc* d_desc, const float* V, const float* N, int w,
                              int h, int precision, cudaStream_t s);
// the shared memory that the variant's kernels may take (before any query or
// launch of them in a context): the attribute belongs to the kernel, not to a
// tracker, so it is always that of the most bins
cudaError_t icp_attributes(const KParams& P);
cudaError_t team_attributes(const KParams& P);
// grid sizes (one wave) of the per-stage and the scheduled ICP kernels
void icp_grids(const KParams& P, int* g_assoc, int* g_reduce, int* g_sched);
cudaError_t launch_icp_init(const PairDesc* const* descs, const PairInput* in, int n, int* list,
                            const KParams& P, cudaStream_t s);
// mode 0: an iteration; 1: inspection (per-pixel outputs, no window);
// 2: inspection of the sums (the band and window set by launch_debug_setup)
cudaError_t launch_assoc_hist(const PairDesc* const* descs, const int* list, int cap, int grid,
                              int level, int mode, const KParams& P, cudaStream_t s);
// in_list: the pairs to reduce; out_list: where the launch's last block writes
// the next launch's active list (level next_level; -1: none)
cudaError_t launch_reduce_solve(const PairDesc* const* descs, int n, const int* in_list,
                                int* out_list, int cap, unsigned* launch_counter, int grid,
                                int level, int next_level, int mode, const KParams& P,
                                cudaStream_t s);
// the whole ICP of a batch in one persistent launch; queue: kQHeaderWords
// header words then (qmask + 1) slots, zeroed; a block whose wait for its
// next task exceeds wait_limit_ns sets queue[kQErr] and returns
constexpr unsigned long long kSchedWaitLimitNs = 2000000000ull;  // 2 s
cudaError_t launch_icp_sched(const PairDesc* const* descs, const PairInput* in, PairOutput* out,
                             int n, unsigned* queue, unsigned qmask, int grid,
                             unsigned long long wait_limit_ns, const KParams& P, cudaStream_t s);
// the whole ICP of a few pairs, each by a team of resident blocks
// (cooperative); team_blocks: blocks that can be resident at once
int team_blocks(const KParams& P);
cudaError_t launch_icp_team(const TeamArgs& args, int grid, const KParams& P, cudaStream_t s);
cudaError_t launch_icp_finish(const PairDesc* const* descs, PairOutput* out, int n,
                              const KParams& P, cudaStream_t s);
// inspection set-up of one pair: pose, level, band [klo, khi] and window
// [w0, w1) (w0 = -1: none) with its hit flag
cudaError_t launch_debug_setup(const PairDesc* const* d_self, const double* d_pose, int level,
                               int klo, int khi, int w0, int w1, int hit, int* list,
                               const KParams& P, cudaStream_t s);
}  // namespace kf
