// ICP hot path: projective association + distance histogram (Sec. 3.2),
// median from the CDF and the inlier band (Sec. 3.3), filtered point-to-plane
// normal-equation reduction (Eq. 3), the regularised FP64 solve (Eq. 4, 5),
// the pose update and the median-driven convergence control (Sec. 3.4).
//
// Work is split into items of consecutive frame pixels of one pair at one
// level. An iteration of a pair is two stages over its items. The association
// pass reads each frame vertex and gathers its model vertex and normal once:
// it counts the distance histogram and, knowing where the band edge fell the
// iteration before, sums the rows of the pixels surely inside the band and
// records the rows of the pixels near the edge. The reduction pass then only
// adds the recorded rows that the new band keeps, or, when the edge moved out
// of that window, associates again with the band known. Each stage's per-pair
// epilogue (median and band after the histogram; solve and update after the
// reduction) runs in the pair's last block to finish, found with a per-pair
// arrival counter: no block waits for the others of its stage (the queue's blocks
// wait for their next task only, each for a bounded time).
#include "kf_icp.cuh"

// Tuning of the ICP kernels: minimum resident blocks per SM (register cap).
#ifndef KF_ASSOC_MINB
#define KF_ASSOC_MINB 2
#endif
#ifndef KF_REDUCE_MINB
#define KF_REDUCE_MINB 2
#endif
#ifndef KF_SCHED_MINB
#define KF_SCHED_MINB 2
#endif
// Scheduled kernel: the pair's median epilogue also runs the reduction pass
// of a hit while the pairs still running number at least the launch's
// blocks / KF_FUSE_GRID_DIV (0: never; a large value: always). Measured at
// 640x480 on 304 blocks: 256 pairs 3.40 ms never, 3.31 ms from 76 pairs on. Below,
// spread over blocks for latency (with register gathers, before the ring: 64 pairs
// 1.45 ms never, 1.49 ms from 32 on).
#ifndef KF_FUSE_GRID_DIV
#define KF_FUSE_GRID_DIV 4
#endif
namespace kf {

#ifdef KF_CHECKED
void checked_fault(long long out[3]) {
  out[0] = out[1] = out[2] = 0;
  take_fault(out);
  checked_fault_team(out);
}
#else
void checked_fault(long long out[3]) { out[0] = out[1] = out[2] = 0; }
#endif

namespace {

// Median bin k_med = min{k : 2 C(k) >= N} from the pair's histogram and the
// band of bins around it (Sec. 3.3). Block-wide; the caller is the pair's last
// block of the histogram stage. Returns (in thread 0) 1 when the pair stops
// here (fewer than n_min valid pairs), else 0.
__device__ __noinline__ int median_and_band(const PairDesc* d, PairState* st, const KParams& P) {
  __shared__ unsigned s_wsum[kBlockWarps];
  __shared__ int s_kmed;
  const int B = P.bins;
  const int per = (B + kBlock - 1) / kBlock;
  const int b0 = threadIdx.x * per;
  const int b1 = min(b0 + per, B);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned local = 0;
  for (int b = b0; b < b1; ++b) local += __ldcg(d->hist + b);
  if (threadIdx.x == 0) s_kmed = 0;
  // inclusive scan of the threads' counts: within each warp by shuffles,
  // then over the warps' totals (exact integer sums)
  unsigned incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    unsigned w = lane < kBlockWarps ? s_wsum[lane] : 0u;
#pragma unroll
    for (int o = 1; o < kBlockWarps; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kBlockWarps) s_wsum[lane] = w;
  }
  __syncthreads();
  if (warp > 0) incl += s_wsum[warp - 1];
  const unsigned N = s_wsum[kBlockWarps - 1];
  const unsigned before = incl - local;
  if (N > 0 && 2ull * incl >= N && 2ull * before < N) {
    unsigned c = before;
    for (int b = b0; b < b1; ++b) {
      c += __ldcg(d->hist + b);
      if (2ull * c >= N) {
        s_kmed = b;
        break;
      }
    }
  }
  __syncthreads();
  int stop = 0;
  if (threadIdx.x == 0) {
    const int kmed = s_kmed;
    st->N = (int)N;
    st->kmed = kmed;
    if ((int)N < P.n_min) {
      st->status = KF_ERR_TOO_FEW_INLIERS;
      st->stopped = 1;
      stop = 1;
    }
    int klo, khi;
    band_of(P, kmed, klo, khi);
    st->klo = klo;
    st->khi = khi;
    st->hit = band_hits(klo, khi, __ldcg(&st->w0), __ldcg(&st->w1)) ? 1 : 0;
  }
  return stop;
}

// solve_update for the launches whose pair state lies in memory that other
// blocks wrote.
__device__ __noinline__ int solve_update_warp(const PairDesc* d, PairState* st, const double* S,
                                               int level, const KParams& P, int passes,
                                               const PairPre& pre) {
  double Tc[3], Tmc[3], Tmt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) Tc[k] = __ldcg(&st->T[4 * k + (threadIdx.x & 3)]);
  load_tm(d->Tm, Tmc, Tmt);
  const NextStep next = next_step(pre, level, P);
  const double lam2c = lane_of(2.0 * pre.lambda_c, 0);
  return solve_update(d, st, S, level, P, passes, pre, next, solve_lane(), lam2c, Tc, Tmc, Tmt,
                      [](const Solved&, int, int, int) {});
}

// ---------------------------------------------------------------------------
// Active work list (see kf_internal.cuh for the layout).
// ---------------------------------------------------------------------------
// Block-wide exclusive scan of one int per thread (kBlock threads); returns the
// exclusive prefix and writes the block total to *total.
__device__ int block_exclusive_scan(int v, int* total) {
  __shared__ int s_buf[kBlock];
  s_buf[threadIdx.x] = v;
  __syncthreads();
  for (int off = 1; off < kBlock; off <<= 1) {
    const int t = threadIdx.x >= off ? s_buf[threadIdx.x - off] : 0;
    __syncthreads();
    s_buf[threadIdx.x] += t;
    __syncthreads();
  }
  const int incl = s_buf[threadIdx.x];
  *total = s_buf[kBlock - 1];
  __syncthreads();
  return incl - v;
}

// Build the list of pairs still iterating at `level` and their items. One
// block of kBlock threads; every pair's state must be final when it runs.
__device__ void build_active_list(const PairDesc* const* descs, int n, int level, int* list, int cap) {
  int* pairs = list + 4;
  int* prefix = list + 4 + cap;
  int npairs = 0, nitems = 0;
  for (int base = 0; base < n; base += kBlock) {
    const int p = base + threadIdx.x;
    int cnt = 0;
    if (p < n && level >= 0) {
      // other blocks of this launch wrote these fields: read them from L2
      const PairState* st = descs[p]->st;
      if (__ldcg(&st->cur_level) == level && !__ldcg(&st->stopped))
        cnt = items_of(descs[p], level);
    }
    int tot_flags, tot_items;
    const int slot = block_exclusive_scan(cnt > 0 ? 1 : 0, &tot_flags);
    const int off = block_exclusive_scan(cnt, &tot_items);
    if (cnt > 0) {
      KF_GUARD(npairs + slot < cap, 8, npairs + slot, cap) {
        pairs[npairs + slot] = p;
        prefix[npairs + slot] = nitems + off;
      }
    }
    npairs += tot_flags;
    nitems += tot_items;
  }
  if (threadIdx.x == 0) {
    KF_GUARD(npairs <= cap, 9, npairs, cap)
    prefix[npairs] = nitems;
    list[0] = nitems;
    list[1] = npairs;
    list[2] = level;
  }
  __syncthreads();
}

// Entry s with prefix[s] <= f < prefix[s+1] (binary search).
__device__ __forceinline__ int find_slot(const int* prefix, int npairs, int f) {
  int lo = 0, hi = npairs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldcg(prefix + mid) <= f) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Writes the warp's row of item li's partial, in slot A or slot B.
__device__ __forceinline__ void write_row(const PairDesc* d, int li, bool slot_b, const float* sum) {
  const float v = warp_sums(sum);
  const int lane = threadIdx.x & 31;
  if (lane < kSums)
    d->partials[(size_t)li * kPartialStride + (slot_b ? kSlotB : 0) + (threadIdx.x >> 5) * 32 + lane] = v;
}

// An association pass over the items [first, first + run) of one pair, in
// order, batch after batch; kPassSplit / kPassBand write each item's partial
// (slot A / slot B). Block-wide: ends with a barrier, so the block's shared
// histogram is complete on return.
template <class T, int kA, int kPass, int kMode>
__device__ void assoc_items(const PairDesc* d, const LevelMaps& L, int first, int run, int chunk,
                            const float* sxf, const KParams& P, unsigned* sh_hist, int lo, int hi) {
  constexpr bool kGate = (kA & kAGate) != 0;
  const int fn = L.fw * L.fh;
  float sum[kSumRegs];
  constexpr int kN = kBatchU<kA>, kPixels = kN * kBlock;  // of a lane, of the block
  Verts<kN> va;
  Batch<kGate, kN> sa;
  const int warp = threadIdx.x >> 5;
  for (int li = first; li < first + run; ++li) {
    const int ib = li * chunk, ie = min(fn, ib + chunk);
    // the warp's record region of the item: as many places as the warp has
    // pixels in it (chunk / kBlockWarps: kU of each batch's 32-pixel groups)
    const int rbase = ib + warp * (chunk / kBlockWarps);
    int wc = 0;
    zero_sums(sum);
    // batches of the item; the last one may be partial (kPixels need not
    // divide the item)
    for (int b0 = ib; b0 < ie; b0 += kPixels) {
      const int e = min(ie, b0 + kPixels);
      load_verts<T>(L, b0, e, threadIdx.x, va);
      associate_batch<T, kA, kPass>(L, b0, threadIdx.x, va, sxf, P, sa);
      {  // L2 hints for this warp's next batch (of this item or the next)
        int nb0 = b0 + kPixels, ne = e + kPixels;
        if (nb0 >= ie) {
          nb0 = ie;
          ne = li + 1 < first + run ? min(fn, ie + kPixels) : ie;
        }
        ne = min(ne, fn);
        // the match offset of the warp's first matched pixel (0: none)
        const unsigned ok = __ballot_sync(0xffffffffu, sa.j[0] >= 0);
        const int src = ok ? __ffs(ok) - 1 : 0;
        const int off = __shfl_sync(0xffffffffu, sa.j[0] - (b0 + threadIdx.x), src);
        prefetch_next<T>(L, nb0, ne, ok ? off : 0);
      }
      finish_batch<kA, kPass, kMode>(d, b0, e, threadIdx.x, sa, sxf, P, sh_hist, lo, hi, sum, rbase, wc);
    }
    if constexpr (kPass == kPassSplit) {
      if ((threadIdx.x & 31) == 0) {
        KF_GUARD(li < d->partial_cap, 7, li, d->partial_cap)
        d->wcount[li * kBlockWarps + warp] = wc;
      }
    }
    if constexpr (kPass != kPassHist) {
      KF_GUARD(li < d->partial_cap, 1, li, d->partial_cap)
      write_row(d, li, kPass == kPassBand, sum);
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// The scheduled kernel's association pass (projective, no gate): as
// assoc_items, with the frame and model records passing through a ring in
// shared memory. A thread copies its pixels' records into its own places
// (cp.async), kAhead + 1 batches ahead for the frame and kAhead for the model,
// so a gather is in flight while the batches before it are summed and holds no
// registers meanwhile. What bounds the pass is the latency of a batch's
// dependent loads (frame record, then the model pixel it projects to) against
// the 16 to 24 warps an SM holds; with register gathers a warp spent 1850
// cycles a pixel of its own at 43 % issue. Only a thread's own copies are waited for
// (cp.async.wait_group): no barrier. The same pixels in the same order as
// assoc_items: the same sums.
// Measured on GB300, the whole alignment of a batch, register gathers -> ring:
// 256 pairs 640x480 3.92 -> 3.55 ms (3.31 since), 64 mixed pairs float16 2.27 -> 2.03 ms, 32
// pairs 0.85 -> 0.81 ms. Two pixels a batch: one pixel 4.2 ms (256 pairs), four
// 3.74 (its registers); model records two or three batches ahead 3.53, 3.57; 24
// warps on an SM 5.3 (spills).
// ---------------------------------------------------------------------------
#ifndef KF_RING_U
#define KF_RING_U 2
#endif
constexpr int kRingU = KF_RING_U;  // pixels of a thread per batch
static_assert(level_chunk(KF_MAX_LEVELS - 1) % (kRingU * kBlock) == 0, "a batch lies in one item");
// bytes of the block's histogram, rounded up for what follows it
__host__ __device__ __forceinline__ size_t hist_bytes(int bins) {
  return ((size_t)bins * sizeof(unsigned) + 15) / 16 * 16;
}
#ifndef KF_RING_AHEAD
#define KF_RING_AHEAD 1
#endif
constexpr int kAhead = KF_RING_AHEAD;  // batches whose model records are under way
template <class T>
struct Ring {
  typename Store<T>::A frame[kAhead + 2][kRingU][kBlock];
  typename Store<T>::A model[kAhead + 1][kRingU][kBlock];
  typename Store<T>::B normal[kAhead + 1][kRingU][kBlock];
};

template <class W>
__device__ __forceinline__ void copy_async(W* dst, const W* src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(W) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s), "l"(src), "n"(sizeof(W)) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

template <class T, int kPass>
__device__ void assoc_ring(const PairDesc* d, const LevelMaps& L, int first, int run, int chunk,
                           const float* sxf, const KParams& P, unsigned* sh_hist, Ring<T>* ring, int lo,
                           int hi) {
  using A = typename Store<T>::A;
  using B = typename Store<T>::B;
  constexpr int kN = kRingU, kPixels = kN * kBlock;
  const int t = threadIdx.x, warp = t >> 5;
  const int begin = first * chunk, end = min(L.fw * L.fh, begin + run * chunk);
  const A* fA = static_cast<const A*>(L.fA);
  const A* mA = static_cast<const A*>(L.mA);
  const B* mB = static_cast<const B*>(L.mB);
  auto fetch_frame = [&](int b0, int stage) {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const int i = b0 + t + u * kBlock;
      if (i < end) copy_async(&ring->frame[stage][u][t], fA + i);
    }
    copy_commit();
  };
  // model pixels of the batches under way, oldest first
  int j[kAhead + 1][kN];
  // projects a batch whose frame records have come and sends for its model records
  auto fetch_model = [&](int b0, int fstage, int mstage, int (&jj)[kN]) {
    float xr[12];
    load_xf<12>(sxf + 12, xr);
    bool far = false;
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const float4 v = Store<T>::value_a(ring->frame[fstage][u][t]);
      jj[u] = project(L, v.x, v.y, v.z, xr, far);
    }
    if (far) {
#pragma unroll
      for (int u = 0; u < kN; ++u) {
        const float4 v = Store<T>::value_a(ring->frame[fstage][u][t]);
        jj[u] = project_far(v.x, v.y, v.z, L.mw, L.mh, L.mfx, L.mfy, L.mcx, L.mcy, sxf);
      }
    }
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      if (b0 + t + u * kBlock >= end) jj[u] = -1;
      if (jj[u] >= 0) {
        copy_async(&ring->model[mstage][u][t], mA + jj[u]);
        if constexpr (kPass != kPassHist) copy_async(&ring->normal[mstage][u][t], mB + jj[u]);
      }
    }
    copy_commit();
  };
  // the loop's order of groups from the start on: the frame of batch k + 1, then
  // the model of batch k
  fetch_frame(begin, 0);
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    fetch_frame(begin + (k + 1) * kPixels, k + 1);
    if (k == 0) copy_wait<1>();
    else copy_wait<2>();
    fetch_model(begin + k * kPixels, k, k, j[k]);
  }
  float sum[kSumRegs];
  zero_sums(sum);
  int wc = 0, fs = 0, ms = 0;  // the ring places of the batch being summed
  // the item of the batch, where it ends and the warp's record region in it,
  // stepped: dividing by the item's size twice a batch cost 7 % (256 pairs
  // 640x480 3.55 ms, now 3.31)
  int li = first, ie = begin + chunk, rbase = begin + warp * (chunk / kBlockWarps);
  for (int b0 = begin; b0 < end; b0 += kPixels) {
    // the batch kAhead later: its frame records have come (one model group
    // stands behind them); the frame records after them take the free place
    copy_wait<1>();
    const int fl = fs + kAhead < kAhead + 2 ? fs + kAhead : fs - 2;
    const int ff = fl + 1 < kAhead + 2 ? fl + 1 : 0;
    fetch_frame(b0 + (kAhead + 1) * kPixels, ff);
    fetch_model(b0 + kAhead * kPixels, fl, ms > 0 ? ms - 1 : kAhead, j[kAhead]);
    copy_wait<2 * kAhead>();  // this batch's model records
    Batch<false, kN> cur;
    {
      float xw[12];
      load_xf<12>(sxf, xw);
#pragma unroll
      for (int u = 0; u < kN; ++u) {
        const float4 v = Store<T>::value_a(ring->frame[fs][u][t]);
        world_point(v.x, v.y, v.z, xw, cur.p[u]);
        cur.j[u] = j[0][u];
        const float4 q = Store<T>::value_a(ring->model[ms][u][t]);
        cur.q[u][0] = q.x;
        cur.q[u][1] = q.y;
        cur.q[u][2] = q.z;
        cur.nq[u][0] = q.w;
        if constexpr (kPass != kPassHist) {
          const float2 n = Store<T>::value_b(ring->normal[ms][u][t]);
          cur.nq[u][1] = n.x;
          cur.nq[u][2] = n.y;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
#pragma unroll
      for (int u = 0; u < kN; ++u) j[k][u] = j[k + 1][u];
    fs = fs + 1 < kAhead + 2 ? fs + 1 : 0;
    ms = ms < kAhead ? ms + 1 : 0;
    finish_batch<0, kPass, 0>(d, b0, end, t, cur, sxf, P, sh_hist, lo, hi, sum, rbase, wc);
    const int after = b0 + kPixels;
    if (after >= end || after == ie) {  // the item's last batch
      if constexpr (kPass == kPassSplit) {
        if ((t & 31) == 0) {
          KF_GUARD(li < d->partial_cap, 7, li, d->partial_cap)
          d->wcount[li * kBlockWarps + warp] = wc;
        }
        wc = 0;
      }
      if constexpr (kPass != kPassHist) {
        KF_GUARD(li < d->partial_cap, 1, li, d->partial_cap)
        write_row(d, li, kPass == kPassBand, sum);
        zero_sums(sum);
      }
      ++li;
      ie += chunk;
      rbase += chunk;
    }
  }
  copy_wait<0>();
  __syncthreads();
}

__device__ __forceinline__ int record_count(const PairDesc* d, int li) {
  return li < d->partial_cap ? (int)__ldcg(d->wcount + li * kBlockWarps + (threadIdx.x >> 5)) : 0;
}

__device__ __forceinline__ void fixup_item(const PairDesc* d, int li, int chunk, int klo, int khi,
                                           float* sum) {
  FixLoad f;
  f.total = record_count(d, li);
  fix_issue(d, li, chunk, threadIdx.x >> 5, f);
  fix_consume(d, li, chunk, threadIdx.x >> 5, klo, khi, f, sum);
}

// The reduction pass of a hit over every item of a pair by one block (the
// block that ran the pair's median): warp w takes region w of items 0, 1,
// ..., count - 1, with the next item's loads in flight while it adds the
// current one. Each item's slot B rows are the ones the reduction tasks
// would write (the same warp-to-region map, the same order): which way runs
// changes no bit. Block-wide: ends with a barrier.
__device__ __noinline__ void fixup_all(const PairDesc* d, int count, int chunk, int klo, int khi) {
  const int warp = threadIdx.x >> 5;
  FixLoad cur, nxt = {};
  if (count > 0) {
    cur.total = record_count(d, 0);
    fix_issue(d, 0, chunk, warp, cur);
  }
  for (int li = 0; li < count; ++li) {
    if (li + 1 < count) {
      nxt.total = record_count(d, li + 1);
      fix_issue(d, li + 1, chunk, warp, nxt);
    }
    float sum[kSumRegs];
    zero_sums(sum);
    fix_consume(d, li, chunk, warp, klo, khi, cur, sum);
    KF_GUARD(li < d->partial_cap, 1, li, d->partial_cap)
    write_row(d, li, true, sum);
    cur = nxt;
  }
  __threadfence_block();
  __syncthreads();
}

// The reduction pass over items [first, first + run) of one pair, last item
// first (the association pass left the latest items' data in L2): the
// recorded window pixels on a hit, else a re-association with the band known.
// Each item writes slot B of its partial.
template <class T, int kA>
__device__ void reduce_items(const PairDesc* d, const LevelMaps& L, int first, int run, int chunk,
                             const float* sxf, const KParams& P, int hit, int klo, int khi) {
  for (int li = first + run - 1; li >= first; --li) {
    if (hit) {
      float sum[kSumRegs];
      zero_sums(sum);
      fixup_item(d, li, chunk, klo, khi, sum);
      KF_GUARD(li < d->partial_cap, 1, li, d->partial_cap)
      write_row(d, li, true, sum);
    } else {
      assoc_items<T, kA, kPassBand, 0>(d, L, li, 1, chunk, sxf, P, nullptr, klo, khi);
    }
  }
}

// The pair's reduction epilogue (block-wide, run by the block that finished
// its last item): per sum, the items' partials in a fixed order (slot A +
// slot B on a hit, slot B alone otherwise; 8 strided sub-sums, then the 8), the histogram cleared for the next iteration, then the solve and
// update (mode 2: the sums are stored instead). Returns (in thread 0) the
// solve's next level (-1: finished or stopped).
__device__ __noinline__ int combine_and_solve(const PairDesc* d, PairState* st, int count,
                                               int level, const KParams& P, int mode,
                                               SubSums& s_part, double* s_sums) {
  __shared__ int s_hit;
  PairPre pre;
  if (threadIdx.x == 0) {
    if (mode == 0) pre = load_pre(st, level);
    s_hit = __ldcg(&st->hit);
  }
  KF_GUARD(count <= d->partial_cap, 2, count, d->partial_cap) {}
#ifdef KF_CHECKED
  if (count > d->partial_cap) count = d->partial_cap;  // the violation is recorded; stay inside
#endif
  __syncthreads();
  const int hit = s_hit;
  // warp `sub` takes items sub, sub + 8, ...; lane k < 29 sums, per item, the
  // 16 rows of sum k (slot A's 8 warps, zero on a miss, and slot B's) in
  // float32 by pairwise halving, then adds the items in increasing order
  // (ItemSum), four items' loads in flight
  const int k = threadIdx.x & 31, sub = threadIdx.x >> 5;
  auto item_value = [&](int l) {
    const float* a = d->partials + (size_t)l * kPartialStride + k;
    float v[2 * kBlockWarps];
#pragma unroll
    for (int w = 0; w < kBlockWarps; ++w) {
      v[w] = hit ? __ldcg(a + w * 32) : 0.f;
      v[kBlockWarps + w] = __ldcg(a + kSlotB + w * 32);
    }
#pragma unroll
    for (int h = kBlockWarps; h >= 1; h >>= 1)
#pragma unroll
      for (int i = 0; i < h; ++i) v[i] = __fadd_rn(v[i], v[i + h]);
    return v[0];
  };
  static_assert(kItemFold % 4 == 0, "folds where the other launches have them");
  FoldedSum t;
  if (k < kSums) {
    int l = sub;
    for (; l + 24 < count; l += 32) {
      const float e0 = item_value(l), e1 = item_value(l + 8), e2 = item_value(l + 16),
                  e3 = item_value(l + 24);
      t.room(4);
      t.s.add(e0);
      t.s.add(e1);
      t.s.add(e2);
      t.s.add(e3);
    }
    for (; l < count; l += 8) {
      t.room(1);
      t.s.add(item_value(l));
    }
    s_part.put(sub, k, t, count);
  }
  for (int b = threadIdx.x; b < P.bins; b += kBlock) d->hist[b] = 0u;
  __syncthreads();
  if (threadIdx.x < kSums) s_sums[threadIdx.x] = s_part.total(threadIdx.x, count);
  __syncthreads();
  int next = -1;
  if (threadIdx.x < 32) {
    if (mode != 0) {
      if (threadIdx.x == 0)
        for (int k = 0; k < kSums; ++k) st->dbg_sums[k] = s_sums[k];
    } else {
      next = solve_update_warp(d, st, s_sums, level, P, hit ? 1 : 2, pre);
    }
    if (threadIdx.x == 0) d->counters[1] = 0u;
  }
  __syncthreads();
  return next;
}

// ---------------------------------------------------------------------------
// Per-stage launches (KF_LAUNCH_PER_ITERATION and the inspection hooks): the
// same items, passes and epilogues as the scheduled kernel, one launch per
// stage and iteration over the active list; each block takes a contiguous
// run of items.
// ---------------------------------------------------------------------------
// Stage 1: association pass (histogram, and the split sums when the pair has
// a window); the pair's last item to finish computes the median, band and hit
// (not in mode 2, whose band is given).
template <class T, int kA>
__global__ void __launch_bounds__(kBlock, KF_ASSOC_MINB) k_assoc_hist(const PairDesc* const* descs,
                                                                      const int* list, int cap,
                                                                      int level, int mode, KParams P) {
  extern __shared__ unsigned sh_hist[];
  __shared__ __align__(16) float sxf[24];  // 16-byte vector loads (load_xf)
  __shared__ int s_active, s_last, s_w0, s_w1;
  const int n_items = __ldcg(list);
  const int M = (n_items + gridDim.x - 1) / gridDim.x;
  int f = blockIdx.x * M;
  const int f1 = min(n_items, f + M);
  if (f >= f1) return;
  const int* pairs = list + 4;
  const int* prefix = list + 4 + cap;
  int slot = find_slot(prefix, __ldcg(list + 1), f);
  const int chunk = level_chunk(level);
  while (f < f1) {
    const int pstart = __ldcg(prefix + slot);
    const int run_end = min(f1, __ldcg(prefix + slot + 1));
    const PairDesc* d = descs[__ldcg(pairs + slot)];
    PairState* st = d->st;
    __syncthreads();  // shared memory of the previous run is free again
    if (threadIdx.x == 0) {
      s_active = (st->cur_level == level) && !st->stopped;
      s_w0 = mode == 1 ? -1 : st->w0;
      s_w1 = st->w1;
    }
    if (threadIdx.x < 24) sxf[threadIdx.x] = st->xf[threadIdx.x];
    for (int b = threadIdx.x; b < P.bins; b += kBlock) sh_hist[b] = 0u;
    __syncthreads();
    if (s_active) {
      const LevelMaps L = d->lv[level];
      const int fn = L.fw * L.fh;
      const int count = (fn + chunk - 1) / chunk;
      const int first = f - pstart, run = run_end - f;
      if (s_w0 >= 0)
        assoc_items<T, kA, kPassSplit, 0>(d, L, first, run, chunk, sxf, P, sh_hist, s_w0, s_w1);
      else if (mode == 1)
        assoc_items<T, kA, kPassHist, 1>(d, L, first, run, chunk, sxf, P, sh_hist, 0, 0);
      else
        assoc_items<T, kA, kPassHist, 0>(d, L, first, run, chunk, sxf, P, sh_hist, 0, 0);
      for (int b = threadIdx.x; b < P.bins; b += kBlock) {
        const unsigned c = sh_hist[b];
        if (c) atomicAdd(d->hist + b, c);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        const unsigned nrun = (unsigned)run;
        s_last = (atomicAdd(d->counters + 0, nrun) + nrun == (unsigned)count);
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        if (mode != 2) median_and_band(d, st, P);
        if (threadIdx.x == 0) d->counters[0] = 0u;
      }
    }
    f = run_end;
    ++slot;
  }
}

// Stage 2: reduction pass; the pair's last item to finish combines, solves
// and updates (mode 2: stores the sums instead). The launch's last block
// builds the active list of the next launch (level next_level; -1: none).
template <class T, int kA>
__global__ void __launch_bounds__(kBlock, KF_REDUCE_MINB) k_reduce_solve(const PairDesc* const* descs, int n,
                                                            const int* list, int* out_list, int cap,
                                                            unsigned* launch_counter, int level,
                                                            int next_level, int mode, KParams P) {
  __shared__ __align__(16) float sxf[24];  // 16-byte vector loads (load_xf)
  __shared__ int s_active, s_klo, s_khi, s_hit, s_last;
  __shared__ double s_sums[kSums];
  __shared__ SubSums s_part;
  const int n_items = __ldcg(list);
  const int M = (n_items + gridDim.x - 1) / gridDim.x;
  int f = blockIdx.x * M;
  const int f1 = min(n_items, f + M);
  const int* pairs = list + 4;
  const int* prefix = list + 4 + cap;
  const int chunk = level_chunk(level);
  const int npairs = f < f1 ? __ldcg(list + 1) : 0;
  int slot = f < f1 ? find_slot(prefix, npairs, f) : 0;
  while (f < f1) {
    const int pstart = __ldcg(prefix + slot);
    const int run_end = min(f1, __ldcg(prefix + slot + 1));
    const PairDesc* d = descs[__ldcg(pairs + slot)];
    PairState* st = d->st;
    __syncthreads();
    if (threadIdx.x == 0) {
      s_active = (st->cur_level == level) && !st->stopped;
      s_klo = st->klo;
      s_khi = st->khi;
      s_hit = st->hit;
    }
    if (threadIdx.x < 24) sxf[threadIdx.x] = st->xf[threadIdx.x];
    __syncthreads();
    if (s_active) {
      const LevelMaps L = d->lv[level];
      const int fn = L.fw * L.fh;
      const int count = (fn + chunk - 1) / chunk;
      reduce_items<T, kA>(d, L, f - pstart, run_end - f, chunk, sxf, P, s_hit, s_klo, s_khi);
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        const unsigned nrun = (unsigned)(run_end - f);
        s_last = (atomicAdd(d->counters + 1, nrun) + nrun == (unsigned)count);
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        combine_and_solve(d, st, count, level, P, mode, s_part, s_sums);
      }
    }
    f = run_end;
    ++slot;
  }
  // the launch's last block to finish builds the next launch's active list
  __shared__ int s_glast;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_glast = (atomicAdd(launch_counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (s_glast) {
    __threadfence();
    if (next_level >= 0) build_active_list(descs, n, next_level, out_list, cap);
    if (threadIdx.x == 0) *launch_counter = 0u;
  }
}

// ---------------------------------------------------------------------------
// Seed (one block for all pairs, then the first active list), finish, and
// inspection set-up.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock) k_icp_init(const PairDesc* const* descs,
                                                     const PairInput* in, int n, int* list,
                                                     KParams P) {
  for (int p = 0; p < n; ++p) {
    const PairDesc* d = descs[p];
    for (int b = threadIdx.x; b < P.bins; b += kBlock) d->hist[b] = 0u;
  }
  for (int p = threadIdx.x; p < n; p += kBlock) {
    double sT[12];
    init_state(descs[p], in[p], P, sT);
    compute_xf(sT, descs[p]->Tm, descs[p]->st->xf);
  }
  __threadfence();
  __syncthreads();
  build_active_list(descs, n, P.levels - 1, list, n);
}

__global__ void k_icp_finish(const PairDesc* const* descs, PairOutput* out) {
  write_output(descs[blockIdx.x], out + blockIdx.x);
}

__global__ void __launch_bounds__(kBlock) k_debug_setup(const PairDesc* const* self,
                                                        const double* pose, int level, int klo,
                                                        int khi, int w0, int w1, int hit,
                                                        int* list, KParams P) {
  const PairDesc* d = self[0];
  PairState* st = d->st;
  for (int b = threadIdx.x; b < P.bins; b += blockDim.x) d->hist[b] = 0u;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 12; ++i) st->T[i] = pose[i];
    st->cur_level = level;
    st->stopped = 0;
    st->status = KF_OK;
    st->has_prior = 0;
    st->klo = klo;
    st->khi = khi;
    st->w0 = w0;
    st->w1 = w1;
    st->hit = hit;
    st->N = 0;
    d->counters[0] = 0u;
    d->counters[1] = 0u;
    compute_xf(st->T, d->Tm, st->xf);
  }
  __threadfence();
  __syncthreads();
  build_active_list(self, 1, level, list, 1);
}

// ---------------------------------------------------------------------------
// Scheduled ICP: every level and iteration of every pair of a batch in one
// persistent launch. Work is the same two kinds of task as in the per-stage
// launches (association pass of a run of items; reduction pass of a run of
// items), but pairs advance independently: the block that finishes a pair's
// last item of a stage runs that stage's epilogue and queues the pair's next
// stage at once, so one pair's median, solve and update overlap the other
// pairs' items instead of ending a launch.
//
// Device queue: a ring of 64-bit slots, each a ticket's tag and its task (a
// run of consecutive items of one stage of one pair). A producer reserves
// tickets at the tail and writes their slots; a block claims the next ticket
// at the head (one ahead of the task it is running) and waits for its slot to
// carry that ticket's tag. Every wait is bounded in time: a wait that runs
// out sets the queue's error word, which the host reports, and the block
// returns. The ring holds every task that can be outstanding at once (each
// pair has at most one stage queued) plus one exit word per block; it is
// zeroed before each launch.
// ---------------------------------------------------------------------------
constexpr unsigned long long kTaskExit = 0xffffffffffull;  // 40-bit payload, all ones
constexpr unsigned long long kTaskAbort = 1ull << 62;      // never stored in a slot
#ifndef KF_MAX_RUN
#define KF_MAX_RUN 16
#endif
// runs per block and round of stages the run length aims at (shorter runs
// shorten each pair's stages, longer ones cost fewer task claims)
#ifndef KF_RUNS_PER_BLOCK
#define KF_RUNS_PER_BLOCK 2
#endif
constexpr int kMaxRun = KF_MAX_RUN;  // <= 16 (the task word's 4-bit run field)
static_assert(kMaxRun >= 1 && kMaxRun <= 16, "run length field");

// slot: tag (24 bits) << 40 | task (40 bits):
//   pair (16) | level (2) | stage (1: reduction) | run length - 1 (4) | first item (17)
__device__ __forceinline__ unsigned long long task_word(int p, int level, int stage, int run,
                                                        int item) {
  return ((unsigned long long)p << 24) | ((unsigned long long)level << 22) |
         ((unsigned long long)stage << 21) | ((unsigned long long)(run - 1) << 17) |
         (unsigned long long)item;
}

__device__ __forceinline__ void slot_store(unsigned long long* a, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long slot_load_acquire(const unsigned long long* a) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
  return v;
}

__device__ __forceinline__ unsigned word_load_relaxed(const unsigned* a) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

// 1 .. 2^24 - 1, never the 0 of a zeroed slot; a slot's earlier tickets
// (ticket - m * slots, slots a power of two) never repeat its tag
__device__ __forceinline__ unsigned slot_tag(unsigned ticket) { return ticket % 0xffffffu + 1u; }

// Block-wide: make this block's writes visible, then queue `count` tasks;
// task i is word(i).
template <class F>
__device__ void push_tasks(unsigned* qh, unsigned long long* qs, unsigned qmask, int count, F word) {
  __shared__ unsigned s_base;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_base = atomicAdd(qh + kQTail, (unsigned)count);
  __syncthreads();
  const unsigned base = s_base;
  for (int i = threadIdx.x; i < count; i += kBlock) {
    const unsigned t = base + (unsigned)i;
    slot_store(qs + (t & qmask), ((unsigned long long)slot_tag(t) << 40) | word(i));
  }
  __syncthreads();
}

// Queue one stage of a pair: `count` items in runs of g consecutive items,
// g chosen from the items of all pairs still running so that a round of
// stages gives every block about KF_RUNS_PER_BLOCK runs (a lone pair gets
// single items).
// The association stage queues its runs first to last, the reduction last to
// first (the items associated last are the ones most likely still in L2).
// Scheduling only: items, partials and their order do not depend on g.
__device__ void push_stage(unsigned* qh, unsigned long long* qs, unsigned qmask, int n, int p,
                           int level, int stage, int count) {
  __shared__ int s_g;
  if (threadIdx.x == 0) {
    const int active = n - (int)word_load_relaxed(qh + kQDone);
    const long long want = (long long)active * count / ((long long)KF_RUNS_PER_BLOCK * gridDim.x);
    s_g = (int)(want < 1 ? 1 : (want > kMaxRun ? kMaxRun : want));
  }
  __syncthreads();
  const int g = s_g;
  const int ntask = (count + g - 1) / g;
  push_tasks(qh, qs, qmask, ntask, [=](int i) {
    const int j = stage ? ntask - 1 - i : i;
    const int first = j * g;
    return task_word(p, level, stage, min(g, count - first), first);
  });
}

// Thread 0: the task of `ticket` once its slot is written; kTaskAbort when
// the wait ran out (or another block's did).
__device__ unsigned long long wait_task(unsigned* qh, const unsigned long long* qs, unsigned qmask,
                                        unsigned ticket, unsigned long long limit_ns) {
  const unsigned long long* slot = qs + (ticket & qmask);
  const unsigned tag = slot_tag(ticket);
  unsigned long long t0 = 0;
  unsigned ns = 0;
  for (int spin = 0;; ++spin) {
    const unsigned long long v = slot_load_acquire(slot);
    if ((unsigned)(v >> 40) == tag) return v & 0xffffffffffull;
    if (spin == 0) {
      t0 = globaltimer_ns();
    } else {
      if (word_load_relaxed(qh + kQErr) != 0u) return kTaskAbort;
      if (globaltimer_ns() - t0 > limit_ns) {
        atomicExch(qh + kQErr, 1u);
        return kTaskAbort;
      }
    }
    if (ns) __nanosleep(ns);
    ns = ns < 256 ? ns + 32 : 256;
  }
}

// Block-wide: initial state of one pair (as the per-stage path's seed).
__device__ void seed_pair(const PairDesc* d, const PairInput& pi, const KParams& P, double* sT) {
  for (int b = threadIdx.x; b < P.bins; b += kBlock) d->hist[b] = 0u;
  if (threadIdx.x == 0) init_state(d, pi, P, sT);
  __syncthreads();
  if (threadIdx.x < 24) d->st->xf[threadIdx.x] = xf_entry(sT, d->Tm, threadIdx.x);
}

// Block-wide: the pair's outputs; the block that finishes the batch's last
// pair queues one exit word per block.
__device__ void finish_pair(const PairDesc* d, PairOutput* o, int n, unsigned* qh,
                            unsigned long long* qs, unsigned qmask) {
  __shared__ int s_lastpair;
  if (threadIdx.x == 0) write_output(d, o);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_lastpair = atomicAdd(qh + kQDone, 1u) == (unsigned)(n - 1);
  __syncthreads();
  if (s_lastpair) push_tasks(qh, qs, qmask, gridDim.x, [](int) { return kTaskExit; });
}

template <class T, int kA>
__global__ void __launch_bounds__(kBlock, KF_SCHED_MINB) k_icp_sched(const PairDesc* const* descs,
                                                                     const PairInput* in,
                                                                     PairOutput* out, int n,
                                                                     unsigned* qh,
                                                                     unsigned long long* qs,
                                                                     unsigned qmask,
                                                                     unsigned long long limit_ns,
                                                                     KParams P) {
  extern __shared__ __align__(16) unsigned char sh_raw[];
  unsigned* sh_hist = reinterpret_cast<unsigned*>(sh_raw);
  [[maybe_unused]] Ring<T>* ring = reinterpret_cast<Ring<T>*>(sh_raw + hist_bytes(P.bins));
  __shared__ __align__(16) float sxf[24];  // 16-byte vector loads (load_xf)
  __shared__ unsigned long long s_word;
  __shared__ int s_last, s_flag, s_a, s_b, s_hit;
  __shared__ double s_sums[kSums];
  __shared__ SubSums s_part;
  __shared__ double s_seed[12];
  // seed: every block that starts takes unseeded pairs until none is left
  for (;;) {
    if (threadIdx.x == 0) s_word = atomicAdd(qh + kQSeed, 1u);
    __syncthreads();
    const unsigned p = (unsigned)s_word;
    __syncthreads();
    if (p >= (unsigned)n) break;
    const PairDesc* d = descs[p];
    seed_pair(d, in[p], P, s_seed);
    const int level = P.levels - 1;
    push_stage(qh, qs, qmask, n, (int)p, level, 0, items_of(d, level));
  }
  unsigned ticket = 0;
  if (threadIdx.x == 0) ticket = atomicAdd(qh + kQHead, 1u);
  for (;;) {
    if (threadIdx.x == 0) {
      const unsigned long long w = wait_task(qh, qs, qmask, ticket, limit_ns);
      if (w < kTaskExit) ticket = atomicAdd(qh + kQHead, 1u);  // claim the next one ahead
      s_word = w;
    }
    __syncthreads();
    const unsigned long long w = s_word;
    if (w >= kTaskExit) break;
    const int p = (int)(w >> 24), level = (int)((w >> 22) & 3u);
    const int run = (int)((w >> 17) & 15u) + 1, first = (int)(w & 0x1ffffu);
    const PairDesc* d = descs[p];
    PairState* st = d->st;
    const LevelMaps L = d->lv[level];
    const int fn = L.fw * L.fh;
    const int chunk = level_chunk(level);
    const int count = (fn + chunk - 1) / chunk;
    if (threadIdx.x < 24) sxf[threadIdx.x] = __ldcg(&st->xf[threadIdx.x]);
    if (!((w >> 21) & 1u)) {
      // association pass of items [first, first + run)
      if (threadIdx.x == 0) {
        s_a = __ldcg(&st->w0);
        s_b = __ldcg(&st->w1);
      }
      for (int b = threadIdx.x; b < P.bins; b += kBlock) sh_hist[b] = 0u;
      __syncthreads();
      if constexpr (kA == 0) {
        if (s_a >= 0)
          assoc_ring<T, kPassSplit>(d, L, first, run, chunk, sxf, P, sh_hist, ring, s_a, s_b);
        else
          assoc_ring<T, kPassHist>(d, L, first, run, chunk, sxf, P, sh_hist, ring, 0, 0);
      } else if (s_a >= 0) {
        assoc_items<T, kA, kPassSplit, 0>(d, L, first, run, chunk, sxf, P, sh_hist, s_a, s_b);
      } else {
        assoc_items<T, kA, kPassHist, 0>(d, L, first, run, chunk, sxf, P, sh_hist, 0, 0);
      }
      for (int b = threadIdx.x; b < P.bins; b += kBlock) {
        const unsigned c = sh_hist[b];
        if (c) atomicAdd(d->hist + b, c);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0)
        s_last = atomicAdd(d->counters + 0, (unsigned)run) + (unsigned)run == (unsigned)count;
      __syncthreads();
      if (s_last) {
        __threadfence();
        const int stop = median_and_band(d, st, P);
        if (threadIdx.x == 0) {
          d->counters[0] = 0u;
          s_flag = stop;
          // while many pairs run, a hit's reduction pass is done here, by this
          // block (its item tasks would each wait on a round trip for a few
          // records); with few pairs left, spread over blocks for latency
          const int active = n - (int)word_load_relaxed(qh + kQDone);
          s_hit = !stop && st->hit && (long long)active * KF_FUSE_GRID_DIV >= (long long)gridDim.x;
          s_a = st->klo;
          s_b = st->khi;
        }
        __syncthreads();
        if (s_flag) {
          finish_pair(d, out + p, n, qh, qs, qmask);
        } else if (s_hit) {
          fixup_all(d, count, chunk, s_a, s_b);
          __threadfence();
          const int next = combine_and_solve(d, st, count, level, P, 0, s_part, s_sums);
          if (threadIdx.x == 0) s_flag = next;
          __syncthreads();
          const int nl = s_flag;
          if (nl >= 0) push_stage(qh, qs, qmask, n, p, nl, 0, items_of(d, nl));
          else finish_pair(d, out + p, n, qh, qs, qmask);
        } else {
          push_stage(qh, qs, qmask, n, p, level, 1, count);
        }
      }
    } else {
      // reduction pass of items first + run - 1 down to first, slot B each
      if (threadIdx.x == 0) {
        s_a = __ldcg(&st->klo);
        s_b = __ldcg(&st->khi);
        s_hit = __ldcg(&st->hit);
      }
      __syncthreads();
      if (s_hit) {
        reduce_items<T, kA>(d, L, first, run, chunk, sxf, P, 1, s_a, s_b);
      } else {
        // re-association with the band known (items in increasing order; the
        // partials do not depend on it)
        if constexpr (kA == 0)
          assoc_ring<T, kPassBand>(d, L, first, run, chunk, sxf, P, nullptr, ring, s_a, s_b);
        else
          assoc_items<T, kA, kPassBand, 0>(d, L, first, run, chunk, sxf, P, nullptr, s_a, s_b);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0)
        s_last = atomicAdd(d->counters + 1, (unsigned)run) + (unsigned)run == (unsigned)count;
      __syncthreads();
      if (s_last) {
        __threadfence();
        const int next = combine_and_solve(d, st, count, level, P, 0, s_part, s_sums);
        if (threadIdx.x == 0) s_flag = next;
        __syncthreads();
        const int nl = s_flag;
        if (nl >= 0) push_stage(qh, qs, qmask, n, p, nl, 0, items_of(d, nl));
        else finish_pair(d, out + p, n, qh, qs, qmask);
      }
    }
    __syncthreads();
  }
}

// the block's histogram, and the ring of the variants that have one
template <class T, int kA>
size_t sched_smem(int bins) { return hist_bytes(bins) + (kA == 0 ? sizeof(Ring<T>) : 0); }

template <class K>
int wave(K kernel, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kBlock, smem);
  return sms * (per > 0 ? per : 1);
}

}  // namespace

cudaError_t icp_attributes(const KParams& P) {
  const int sm = kMaxBins * (int)sizeof(unsigned);
  cudaError_t e = cudaSuccess;
#define KF_X(T, A)                                                                                     \
  e = cudaFuncSetAttribute(k_assoc_hist<T, A>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);       \
  if (e == cudaSuccess)                                                                                \
    e = cudaFuncSetAttribute(k_icp_sched<T, A>, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                             (int)sched_smem<T, A>(kMaxBins))
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return e == cudaSuccess ? team_attributes(P) : e;
}

void icp_grids(const KParams& P, int* g_assoc, int* g_reduce, int* g_sched) {
  const size_t sm = (size_t)P.bins * sizeof(unsigned);
#define KF_X(T, A)                                 \
  *g_assoc = wave(k_assoc_hist<T, A>, sm);         \
  *g_reduce = wave(k_reduce_solve<T, A>, 0);       \
  *g_sched = wave(k_icp_sched<T, A>, sched_smem<T, A>(P.bins))
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  // one partition of the items for both passes
  *g_assoc = *g_reduce = (*g_assoc < *g_reduce ? *g_assoc : *g_reduce);
}

cudaError_t launch_icp_sched(const PairDesc* const* descs, const PairInput* in, PairOutput* out,
                             int n, unsigned* queue, unsigned qmask, int grid,
                             unsigned long long wait_limit_ns, const KParams& P, cudaStream_t s) {
  unsigned long long* slots = reinterpret_cast<unsigned long long*>(queue + kQHeaderWords);
#define KF_X(T, A) \
  k_icp_sched<T, A><<<grid, kBlock, sched_smem<T, A>(P.bins), s>>>(descs, in, out, n, queue, slots, qmask, wait_limit_ns, P)
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return cudaGetLastError();
}

cudaError_t launch_icp_init(const PairDesc* const* descs, const PairInput* in, int n, int* list,
                            const KParams& P, cudaStream_t s) {
  k_icp_init<<<1, kBlock, 0, s>>>(descs, in, n, list, P);
  return cudaGetLastError();
}

cudaError_t launch_assoc_hist(const PairDesc* const* descs, const int* list, int cap, int grid,
                              int level, int mode, const KParams& P, cudaStream_t s) {
  const size_t sm = (size_t)P.bins * sizeof(unsigned);
#define KF_X(T, A) k_assoc_hist<T, A><<<grid, kBlock, sm, s>>>(descs, list, cap, level, mode, P)
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return cudaGetLastError();
}

cudaError_t launch_reduce_solve(const PairDesc* const* descs, int n, const int* in_list,
                                int* out_list, int cap, unsigned* launch_counter, int grid,
                                int level, int next_level, int mode, const KParams& P,
                                cudaStream_t s) {
#define KF_X(T, A)                                                                        \
  k_reduce_solve<T, A><<<grid, kBlock, 0, s>>>(descs, n, in_list, out_list, cap, launch_counter, \
                                               level, next_level, mode, P)
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return cudaGetLastError();
}

cudaError_t launch_icp_finish(const PairDesc* const* descs, PairOutput* out, int n,
                              const KParams& /*P*/, cudaStream_t s) {
  k_icp_finish<<<n, 1, 0, s>>>(descs, out);
  return cudaGetLastError();
}

cudaError_t launch_debug_setup(const PairDesc* const* d_self, const double* d_pose, int level,
                               int klo, int khi, int w0, int w1, int hit, int* list,
                               const KParams& P, cudaStream_t s) {
  k_debug_setup<<<1, kBlock, 0, s>>>(d_self, d_pose, level, klo, khi, w0, w1, hit, list, P);
  return cudaGetLastError();
}

}  // namespace kf

// ===========================================================================
// Allocation-free reduction entry point. The paper has no counterpart: this
// serves callers that may not allocate device memory themselves (a host
// application whose allocator is owned by another runtime, a plug-in running
// inside someone else's CUDA context, a caller that must not add
// cudaMalloc / cudaFree synchronisation points while other work is in
// flight). Its scratch lives in the file-scope array below instead.
// ===========================================================================
#include <atomic>
#include <cstring>
#include <mutex>

namespace kf {
namespace {

constexpr int kNoAllocMaxItems = 1024;  // 1024 items x 4096 px = 4,194,304 frame pixels
constexpr size_t kNoAllocHeader = 512;  // the arrivals' word
constexpr int kNoAllocStride = 32;     // floats per block partial (29 used)
constexpr size_t kNoAllocBytes = kNoAllocHeader + sizeof(float) * kNoAllocStride * kNoAllocMaxItems;
constexpr int kNoAllocMaxDevices = 64;

// Scratch of kf_reduce_noalloc: 131,584 bytes held on every device that loads
// the library, until the process exits. Every call shares it.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

struct NoAllocArgs {
  const float* fv;            // frame vertices, interleaved xyz, camera frame
  const float* mv;            // model vertices, interleaved xyz, world frame
  const float* mn;            // model normals, interleaved xyz, world frame
  int fw, fh, mw, mh;
  float mfx, mfy, mcx, mcy;
  double T[12];               // current pose 3x4
  double Tm[12];              // model pose 3x4
  KParams P;                  // d_max32, scale32, bins, tiny_bins used
  int klo, khi;
  unsigned long long first;   // the arrivals' word before this call's first arrival
  double* out;                // 29 sums (device)
};

// One block per item of 4096 frame pixels; the last block to arrive adds the
// items (ItemSum). The arrivals' word holds the number of the call in its upper
// half, so a call starts from zero whatever an earlier one left there: each block
// raises the word to the call's first value (a store that nobody waits for)
// before it counts itself. A captured call has the same number in every replay; a
// node of its own zeroes the word there. A thread takes its pixels kNoAllocFly
// at a time, every load of a batch before its first use, then adds the rows in
// pixel order: what bounds it is the two round trips of a batch (vertices, then
// model pixels), which a pixel-by-pixel loop pays 16 times over. kShort: a model up to 2^22
// pixels wide and high and no tiny bins (see project, bin_of).
// Measured on GB300, 640x480: 28.4 us with a set-up launch, pixel by pixel and
// a float64 chain over the items; 12.5 us now (calls in a row, the host's
// part included).
constexpr int kNoAllocFly = 8;
template <bool kShort>
__global__ void __launch_bounds__(kBlock) k_noalloc_reduce(unsigned char* scratch,
                                                           const __grid_constant__ NoAllocArgs a, int nitems) {
  __shared__ __align__(16) float sxf[24];  // 16-byte vector loads (load_xf)
  __shared__ float s_red[kBlock / 32][kSums];
  __shared__ SubSums s_part;
  __shared__ int s_last;
  unsigned long long* arrivals = reinterpret_cast<unsigned long long*>(scratch);
  if (threadIdx.x == 0) atomicMax(arrivals, a.first);
  float* partials = reinterpret_cast<float*>(scratch + kNoAllocHeader);
  const int npx = a.fw * a.fh;
  const int begin = blockIdx.x * kChunk;
  const int end = min(npx, begin + kChunk);
  LevelMaps L = {};
  L.fw = a.fw;
  L.fh = a.fh;
  L.mw = a.mw;
  L.mh = a.mh;
  L.mfx = a.mfx;
  L.mfy = a.mfy;
  L.mcx = a.mcx;
  L.mcy = a.mcy;
  if (threadIdx.x < 24) sxf[threadIdx.x] = xf_entry(a.T, a.Tm, threadIdx.x);
  float sum[kSums];
#pragma unroll
  for (int k = 0; k < kSums; ++k) sum[k] = 0.f;
  __syncthreads();
  for (int i0 = begin + threadIdx.x; i0 < end; i0 += kNoAllocFly * kBlock) {
    float v[kNoAllocFly][3], p[kNoAllocFly][3], q[kNoAllocFly][3], n[kNoAllocFly][3];
    int j[kNoAllocFly];
#pragma unroll
    for (int u = 0; u < kNoAllocFly; ++u) {
      const int i = i0 + u * kBlock;
      const bool in = i < end;
#pragma unroll
      for (int c = 0; c < 3; ++c) v[u][c] = in ? __ldg(a.fv + 3 * i + c) : __int_as_float(0x7fc00000);
    }
    bool far = false;
#pragma unroll
    for (int u = 0; u < kNoAllocFly; ++u) {
      if constexpr (kShort) {
        world_point(v[u][0], v[u][1], v[u][2], sxf, p[u]);
        j[u] = project(L, v[u][0], v[u][1], v[u][2], sxf + 12, far);
      } else {
        world_point(v[u][0], v[u][1], v[u][2], sxf, p[u]);
        j[u] = project_any(L, v[u][0], v[u][1], v[u][2], sxf);
      }
    }
    if (far) {
#pragma unroll
      for (int u = 0; u < kNoAllocFly; ++u)
        j[u] = project_far(v[u][0], v[u][1], v[u][2], L.mw, L.mh, L.mfx, L.mfy, L.mcx, L.mcy, sxf);
    }
#pragma unroll
    for (int u = 0; u < kNoAllocFly; ++u) {
      const int jj = max(j[u], 0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        q[u][c] = __ldg(a.mv + 3 * jj + c);
        n[u][c] = __ldg(a.mn + 3 * jj + c);
      }
    }
#pragma unroll
    for (int u = 0; u < kNoAllocFly; ++u) {
      const float n0 = n[u][0], n1 = n[u][1], n2 = n[u][2];
      const int k = kShort ? bin_of(p[u], q[u], a.P) : bin_any(p[u], q[u], a.P);
      // a model hole: any vertex or normal component non-finite, or a zero
      // normal (the tracker's model preparation drops the same pixels)
      const bool whole = isfinite(q[u][0]) && isfinite(q[u][1]) && isfinite(q[u][2]) && isfinite(n0) &&
                         isfinite(n1) && isfinite(n2) && (n0 != 0.f || n1 != 0.f || n2 != 0.f);
      if (j[u] < 0 || !whole || k < a.klo || k > a.khi) continue;
      const float av[6] = {p[u][1] * n2 - p[u][2] * n1, p[u][2] * n0 - p[u][0] * n2, p[u][0] * n1 - p[u][1] * n0,
                           n0, n1, n2};
      const float b = n0 * (q[u][0] - p[u][0]) + n1 * (q[u][1] - p[u][1]) + n2 * (q[u][2] - p[u][2]);
      int s = 0;
#pragma unroll
      for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int c = r; c < 6; ++c) {
          sum[s] = fmaf(av[r], av[c], sum[s]);
          ++s;
        }
#pragma unroll
      for (int r = 0; r < 6; ++r) sum[21 + r] = fmaf(av[r], b, sum[21 + r]);
      sum[27] += 1.f;
      sum[28] = fmaf(b, b, sum[28]);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kSums; ++k) {
    float v = sum[k];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) s_red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kSums) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kBlock / 32; ++w) v += s_red[w][threadIdx.x];
    partials[blockIdx.x * kNoAllocStride + threadIdx.x] = v;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(arrivals, 1ull) == a.first + (unsigned)(nitems - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (lane < kSums) {
    FoldedSum t;
    for (int l0 = warp; l0 < nitems; l0 += kItemFold * (kBlock / 32)) {
      const int l1 = min(nitems, l0 + kItemFold * (kBlock / 32));
      t.room(kItemFold);
#pragma unroll 8
      for (int l = l0; l < l1; l += kBlock / 32) t.s.add(__ldcg(partials + l * kNoAllocStride + lane));
    }
    s_part.put(warp, lane, t, nitems);
  }
  __syncthreads();
  if (threadIdx.x < kSums) a.out[threadIdx.x] = s_part.total(threadIdx.x, nitems);
  if (threadIdx.x == 0) *arrivals = 0ull;
}

std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_ptr[kNoAllocMaxDevices] = {nullptr};

}  // namespace
}  // namespace kf

extern "C" kf_status kf_reduce_noalloc(const float* frame_vertex, int width, int height,
                                       const float* model_vertex, const float* model_normal,
                                       const kf_intrinsics* model_K, const double pose[16],
                                       const double model_pose[16], double d_max, int hist_bins,
                                       int klo, int khi, double* sums, void* cuda_stream) {
  using namespace kf;
  if (!frame_vertex || !model_vertex || !model_normal || !model_K || !pose || !model_pose || !sums)
    return KF_ERR_INVALID_ARG;
  if (width < 1 || height < 1 || model_K->width < 1 || model_K->height < 1) return KF_ERR_INVALID_ARG;
  if (!(d_max > 0) || hist_bins < 1 || hist_bins > kMaxBins || klo < 0 || khi < klo)
    return KF_ERR_INVALID_ARG;
  if (!(model_K->fx > 0) || !(model_K->fy > 0)) return KF_ERR_INVALID_ARG;
  // model indices are 32-bit: 3 w h interleaved floats must stay below 2^31
  if (3LL * model_K->width * model_K->height > 2147483647LL) return KF_ERR_INVALID_ARG;
  const long long npx = (long long)width * height;
  if (npx > (long long)kNoAllocMaxItems * kChunk) return KF_ERR_SCRATCH_LIMIT;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return KF_ERR_CUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return KF_ERR_INTERNAL;
  unsigned char* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      // the host-side name of the array is not a device address: ask the
      // runtime for this device's copy (once per device, this device current)
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return KF_ERR_CUDA;
      g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
    }
    scratch = g_noalloc_ptr[dev];
  }
  NoAllocArgs a;
  memset(&a, 0, sizeof(a));
  a.fv = frame_vertex;
  a.mv = model_vertex;
  a.mn = model_normal;
  a.fw = width;
  a.fh = height;
  a.mw = model_K->width;
  a.mh = model_K->height;
  a.mfx = (float)model_K->fx;
  a.mfy = (float)model_K->fy;
  a.mcx = (float)model_K->cx;
  a.mcy = (float)model_K->cy;
  for (int i = 0; i < 12; ++i) {
    a.T[i] = pose[i];
    a.Tm[i] = model_pose[i];
  }
  a.P.bins = hist_bins;
  a.P.d_max32 = (float)d_max;
  a.P.scale32 = (float)((double)hist_bins / d_max);
  a.klo = klo;
  a.khi = khi;
  a.out = sums;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int nitems = (int)((npx + kChunk - 1) / kChunk);
  static std::atomic<unsigned> next_call{1};
  a.first = (unsigned long long)next_call.fetch_add(1) << 32;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &capture);
  if (e == cudaSuccess && capture == cudaStreamCaptureStatusActive) e = cudaMemsetAsync(scratch, 0, sizeof(a.first), s);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return KF_ERR_CUDA;
  }
  a.P.tiny_bins = tiny_bins(a.P.d_max32, a.P.scale32);
  const bool brief = !a.P.tiny_bins && a.mw <= (1 << 22) && a.mh <= (1 << 22);
  auto kernel = brief ? k_noalloc_reduce<true> : k_noalloc_reduce<false>;
  kernel<<<nitems, kBlock, 0, s>>>(scratch, a, nitems);
  return cudaGetLastError() == cudaSuccess ? KF_OK : KF_ERR_CUDA;
}
