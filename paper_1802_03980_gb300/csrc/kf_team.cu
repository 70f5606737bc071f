// Team launch of the ICP loop: a few pairs, one kernel, every block of a pair
// resident and bound to the same frame pixels for the whole alignment.
//
// What bounds a small batch is the chain of each iteration, not the pixels:
// the queue of kf_icp.cu hands every stage of every iteration out anew (claim,
// descriptor, transforms, fence, arrival, epilogue, publication: about 29 us
// an iteration for one 640x480 pair, whatever its size). Here a pair has a
// leader block and up to kTeamSlots half items per worker block, and an
// iteration crosses between blocks three times, each time as the data itself:
//
//  1. workers add their histograms to the pair's (one atomic per filled bin)
//     and read it until its total, unmatched pixels included, is the level's
//     pixel count; each then finds the median and the band for itself;
//  2. workers send the float32 sums of each half item as packets of a value
//     and the iteration's tag (a 64-bit store each), the leader reads until
//     every tag has come, adds the items and solves;
//  3. the leader sends transforms, level and window the same way.
//
// No arrival counter stands before any of them: a complete total or a fresh tag
// is the arrival, and what crosses is in the words that show it. Only the clear
// of a histogram needs more: the leader clears an iteration's once that
// iteration's sums have all come (a worker sends them after its last look), and
// the workers that add to it next must come after. The leader's releasing fence
// stands where it waits for counts; the workers' acquiring one empties their L1,
// so the histogram rotates through sixteen buffers and they take one as they
// enter each eighth iteration: at iteration i the latest belongs to a message
// after i - 8, the clear of that buffer to i - 16. Measured on GB300, one
// pair 640x480, set and aligned: 165 us with an acquire in every iteration, 159
// without any.
//
// A half item is four of the eight warps of an item (0 2 4 6 or 1 3 5 7), each
// shared by two warps here (team_batch): the
// rows, their halving within an item and the order over items are those
// of the queue's launch, so the two give the same bits, and 150 blocks share a
// 640x480 frame, one on an SM. A worker's frame and model pixels stay in its
// L1 from one iteration to the next.
//
// The launch is cooperative (its blocks wait on one another), and every wait
// is bounded: a wait that runs out ends its block, and the pair's output keeps
// the time-out status that the host wrote before the launch.
//
// Measured on GB300, set frame and align of one pair, queue -> team: 160x120
// (one level) 189 -> 100 us, 640x480 302 -> 158 us, 1280x960 430 -> 272 us (more
// sizes and batches at kTeamSlots).
#include "kf_icp.cuh"

namespace kf {

#ifdef KF_CHECKED
void checked_fault_team(long long out[3]) { take_fault(out); }
#endif

namespace {

constexpr int kTeamWarps = 4;            // item warps of a half item
static_assert(kTeamWarps * kTeamPlaces == level_chunk(0) / 2, "record places of a half item");
constexpr int kTeamBlock = 2 * 32 * kTeamWarps;  // two warps (parts) for each
// blocks per SM that a launch may count on; 0: what the device says
#ifndef KF_TEAM_PER_SM
#define KF_TEAM_PER_SM 0
#endif
constexpr int kPollCheck = 64;  // polls between two looks at the clock
// pause between two polls of a worker without half items at its level
#ifndef KF_TEAM_IDLE_NS
#define KF_TEAM_IDLE_NS 100
#endif

__device__ __forceinline__ void packet_store(unsigned long long* p, unsigned v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | v)
               : "memory");
}

__device__ __forceinline__ unsigned long long packet_load(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void fence_release() { asm volatile("fence.release.gpu;" ::: "memory"); }
__device__ __forceinline__ void fence_acquire() { asm volatile("fence.acquire.gpu;" ::: "memory"); }

__device__ __forceinline__ uint4 words_load(const unsigned* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}

// A bounded wait: true once limit_ns have passed since the first look.
struct Wait {
  unsigned long long t0 = 0;
  unsigned polls = 0;
  __device__ __forceinline__ bool ran_out(unsigned long long limit_ns) {
    if (++polls % kPollCheck != 0) return false;
    const unsigned long long t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    return t - t0 > limit_ns;
  }
};

// One warp: waits until the histogram holds `pixels` counts (the word after
// the bins counts the unmatched), then the median bin and the matched pairs N
// (median_and_band's rule). Lane l owns the bins [l per, (l + 1) per). Returns
// false when the wait ran out.
__device__ bool warp_median(const unsigned* hist, int bins, unsigned pixels,
                            unsigned long long limit_ns, int& N, int& kmed) {
  const int lane = threadIdx.x & 31;
  constexpr int kReg = 16;  // bins a lane holds in registers (512 bins)
  const int per = (bins + 127) / 128 * 4;
  const int b0 = lane * per;
  unsigned v[kReg];
  Wait wait;
  unsigned local, none;
  for (;;) {
    local = 0;
    none = lane == 0 ? words_load(hist + team_hist_none(bins)).x : 0u;
#pragma unroll
    for (int i = 0; i < kReg; i += 4) {
      uint4 w = make_uint4(0u, 0u, 0u, 0u);
      if (i < per && b0 + i < bins) w = words_load(hist + b0 + i);  // words past the bins stay 0
      v[i] = w.x, v[i + 1] = w.y, v[i + 2] = w.z, v[i + 3] = w.w;
      local += (w.x + w.y) + (w.z + w.w);
    }
    for (int i = kReg; i < per; i += 4)
      if (b0 + i < bins) {
        const uint4 w = words_load(hist + b0 + i);
        local += (w.x + w.y) + (w.z + w.w);
      }
    if (__reduce_add_sync(0xffffffffu, local + none) == pixels) break;
    if (__any_sync(0xffffffffu, wait.ran_out(limit_ns))) return false;
  }
  unsigned incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
  const unsigned before = incl - local;
  int k = -1;
  if (total > 0 && 2ull * incl >= total && 2ull * before < total) {
    unsigned c = before;
#pragma unroll
    for (int i = 0; i < kReg; ++i)
      if (k < 0 && i < per) {
        c += v[i];
        if (2ull * c >= total) k = b0 + i;
      }
    for (int i = kReg; k < 0 && i < per; ++i) {
      c += __ldcg(hist + b0 + i);
      if (2ull * c >= total) k = b0 + i;
    }
  }
  N = (int)total;
  kmed = max(0, __reduce_max_sync(0xffffffffu, k));
  return true;
}

// Barrier of the two warps (parts) of one item warp.
__device__ __forceinline__ void parts_sync(int lw) {
  asm volatile("bar.sync %0, 64;" ::"r"(1 + lw) : "memory");
}

struct TeamShared {
  float xf[24];  // first: 16-byte vector loads (load_xf)
  float hand[2][kTeamWarps][kSumRegs][32];  // part 0's sums per lane, for part 1 (by slot parity)
  float row_a[kTeamSlots][kTeamWarps][32];
  float row[2][kTeamWarps][32];
  int count[kTeamSlots][kTeamWarps][2];  // records of each part
  double T[12];
  SubSums part;
  double sums[kSums + 3];
  int level, w0, w1;
  unsigned it;
  int N, kmed, klo, khi, hit, stop;
  unsigned matched;
  int abort;
};

// An association pass of one warp (virtual warp vw of item li's eight), by two
// warps: a lane's pixels, in the order assoc_items gives that warp, are cut in
// two, part 0 takes the first half and part 1 the second. Each looks up, counts
// and forms the rows of its kN pixels at the same time; only the additions stay
// in order: part 0 hands its lanes' sums to part 1, which goes on from them and
// writes the warp's row. places: the first of the item warp's records, in the
// block's own part of the buffer: no other block of the launch, at this level or
// the next, writes or reads there. Part 1's start half the item warp's pixels on.
// Alone on its scheduler a warp took 5.9 us for the 16 pixels a lane has at level
// 0 (640x480), two take 3.6 us.
template <class T, int kA, int kPass, int kN>
__device__ __forceinline__ void team_batch(const PairDesc* d, const LevelMaps& L, int li, int vw, int lw,
                                           int part, int chunk, const KParams& P, TeamShared& sh, int s,
                                           unsigned* sh_hist, int lo, int hi, int places, float* row) {
  const int lane = threadIdx.x & 31, t = vw * 32 + lane;
  const int ib = li * chunk, b0 = ib + part * kN * kBlock;
  const int e = min(min(L.fw * L.fh, ib + chunk), b0 + kN * kBlock);
  Verts<kN> v;
  Batch<(kA & kAGate) != 0, kN> b;
  int bin[kN];
  load_verts<T>(L, b0, e, t, v);
  associate_batch<T, kA, kPass>(L, b0, t, v, sh.xf, P, b);
  finish_bins<kA, kPass, 0, kN>(d, b0, e, t, b, sh.xf, P, sh_hist, bin);
  if constexpr (kPass != kPassHist) {
    float sum[kSumRegs];
    float (*hand)[32] = sh.hand[s & 1][lw];
    int wc = 0;
    const int rbase = places + part * (chunk / kBlockWarps / 2);
    if (part == 0) {
      zero_sums(sum);
      finish_rows<kA, kPass, kN>(d, b, bin, lo, hi, sum, rbase, wc);
#pragma unroll
      for (int k = 0; k < kSumRegs; ++k) hand[k][lane] = sum[k];
      parts_sync(lw);
    } else {
      parts_sync(lw);
#pragma unroll
      for (int k = 0; k < kSumRegs; ++k) sum[k] = hand[k][lane];
      finish_rows<kA, kPass, kN>(d, b, bin, lo, hi, sum, rbase, wc);
      const float r = warp_sums(sum);
      if (lane < kSums) row[lane] = r;
    }
    if (kPass == kPassSplit && lane == 0) sh.count[s][lw][part] = wc;
  }
}

template <class T, int kA, int kPass>
__device__ __noinline__ void team_item(const PairDesc* d, const LevelMaps& maps, int li, int vw, int lw,
                                       int part, int chunk, const KParams& P, TeamShared& sh, int s,
                                       unsigned* sh_hist, int lo, int hi, int places, float* row) {
  const LevelMaps L = maps;  // in registers: the caller's copy lies in its stack frame
  static_assert(level_chunk(0) == 16 * kBlock && level_chunk(1) == 8 * kBlock && level_chunk(2) == 4 * kBlock &&
                    level_chunk(3) == 4 * kBlock, "pixels of a lane per level");
  if (chunk == 16 * kBlock)
    team_batch<T, kA, kPass, 8>(d, L, li, vw, lw, part, chunk, P, sh, s, sh_hist, lo, hi, places, row);
  else if (chunk == 8 * kBlock)
    team_batch<T, kA, kPass, 4>(d, L, li, vw, lw, part, chunk, P, sh, s, sh_hist, lo, hi, places, row);
  else
    team_batch<T, kA, kPass, 2>(d, L, li, vw, lw, part, chunk, P, sh, s, sh_hist, lo, hi, places, row);
}

// The recorded rows of one item warp with klo <= bin <= khi, added in packed
// order (fix_consume's): record i of the c0 + c1 lies in part 0's places up to
// c0, then in part 1's. issue() sends for the first 64.
struct TeamFix {
  int c0, total, base, half;
  float4 r0[kFixR], r1[kFixR];
  __device__ __forceinline__ void issue(const PairDesc* d, int e0) {
#pragma unroll
    for (int r = 0; r < kFixR; ++r) {
      const int i = e0 + r * 32 + (threadIdx.x & 31);
      if (i < total) {
        const size_t at = base + (i < c0 ? i : half + i - c0);
        KF_GUARD((int)at < d->rec_cap, 12, (int)at, d->rec_cap) {
          r0[r] = __ldcg(d->recs + 2 * at);
          r1[r] = __ldcg(d->recs + 2 * at + 1);
        }
      }
    }
  }
  __device__ __forceinline__ void begin(const PairDesc* d, int places, int chunk, const int (&count)[2]) {
    c0 = count[0];
    total = c0 + count[1];
    base = places;
    half = chunk / kBlockWarps / 2;
    issue(d, 0);
  }
  __device__ __forceinline__ float finish(const PairDesc* d, int klo, int khi) {
    float sum[kSumRegs];
    zero_sums(sum);
    for (int e0 = 0; e0 < total;) {
#pragma unroll
      for (int r = 0; r < kFixR; ++r) {
        if (e0 + r * 32 + (int)(threadIdx.x & 31) >= total) continue;
        const int k = __float_as_int(r1[r].w);
        if (k >= klo && k <= khi) {
          const float a[6] = {r0[r].x, r0[r].y, r0[r].z, r0[r].w, r1[r].x, r1[r].y};
          accumulate(a, r1[r].z, sum);
        }
      }
      e0 += 32 * kFixR;
      issue(d, e0);
    }
    return warp_sums(sum);
  }
};

// The band around a median and whether it lies in the window [w0, w1).
__device__ __forceinline__ void team_band(TeamShared& sh, const KParams& P, int N, int kmed, int w0, int w1) {
  int klo, khi;
  band_of(P, kmed, klo, khi);
  sh.N = N;
  sh.kmed = kmed;
  sh.klo = klo;
  sh.khi = khi;
  sh.hit = band_hits(klo, khi, w0, w1);
  sh.stop = N < P.n_min;
}

// Adds the block's histogram to the pair's: one atomic per filled bin, and the
// block's unmatched pixels, and empties it for the next iteration.
__device__ __forceinline__ void flush_hist(unsigned* sh_hist, unsigned* hist, int bins, unsigned pixels,
                                           unsigned* matched) {
  unsigned own = 0;
  for (int b = threadIdx.x; b < bins; b += kTeamBlock) {
    const unsigned c = sh_hist[b];
    if (c) {
      atomicAdd(hist + b, c);
      sh_hist[b] = 0u;
      own += c;
    }
  }
  own = __reduce_add_sync(0xffffffffu, own);
  if ((threadIdx.x & 31) == 0 && own) atomicAdd(matched, own);
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned none = pixels - *matched;
    if (none) atomicAdd(hist + team_hist_none(bins), none);
    *matched = 0u;
  }
}

// A worker: the half items w, w + W, ... of the pair's current level. The leader
// waits for the sums of the workers that have some, so such a worker meets every
// message; one without may sleep through a whole iteration (its block started
// late, say) and goes on from the first message that it finds complete, the
// iteration's number taken from the tag.
template <class T, int kA>
__device__ void team_work(const PairDesc* d, const TeamPair& tp, int w, unsigned long long limit_ns,
                          const KParams& P, TeamShared& sh, unsigned* sh_hist) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lw = warp % kTeamWarps, part = warp / kTeamWarps;
  int level = P.levels - 1, w0 = -1, w1 = -1;
  unsigned it = 0;
  // first record place of a slot's item warp
  auto places_of = [&](int slot) { return ((w * tp.slots + slot) * kTeamWarps + lw) * kTeamPlaces; };
  for (;;) {
    const LevelMaps L = d->lv[level];
    const int chunk = level_chunk(level), fn = L.fw * L.fh;
    const int halves = 2 * ((fn + chunk - 1) / chunk);
    if (w < halves) {
      unsigned* hist = d->team_hist + (it % kTeamHists) * team_hist_words(P.bins);
      unsigned pixels = 0;
      int s = 0;
      for (int hid = w; hid < halves; hid += tp.workers, ++s) {
        const int li = hid >> 1, vw = (hid & 1) + 2 * lw;
        // the half item's pixels: 32-pixel groups vw, vw + 8, ... of the item
        const int ip = min(fn - li * chunk, chunk), rest = ip % kBlock;
        if (warp == 0)
          for (int k = 0; k < kTeamWarps; ++k)
            pixels += ip / kBlock * 32 + min(32, max(0, rest - ((hid & 1) + 2 * k) * 32));
        if (w0 >= 0)
          team_item<T, kA, kPassSplit>(d, L, li, vw, lw, part, chunk, P, sh, s, sh_hist, w0, w1, places_of(s),
                                       sh.row_a[s][lw]);
        else
          team_item<T, kA, kPassHist>(d, L, li, vw, lw, part, chunk, P, sh, s, sh_hist, 0, 0, 0, nullptr);
      }
      const int slots = s;
      __syncthreads();
      flush_hist(sh_hist, hist, P.bins, pixels, &sh.matched);
      // the recorded rows of each part's first slot, on their way while the
      // histogram completes (the parts take the slots in turn)
      TeamFix f;
      auto item_of = [&](int slot) { return (w + slot * tp.workers) >> 1; };
      auto warp_of = [&](int slot) { return ((w + slot * tp.workers) & 1) + 2 * lw; };
      if (w0 >= 0 && part < slots) f.begin(d, places_of(part), chunk, sh.count[part][lw]);
      if (warp == 0) {
        int N, kmed;
        const bool ok = warp_median(hist, P.bins, (unsigned)fn, limit_ns, N, kmed);
        if (lane == 0) {
          if (ok) team_band(sh, P, N, kmed, w0, w1);
          else sh.abort = 1;
        }
      }
      __syncthreads();
      if (sh.abort) return;
      if (!sh.stop) {
        const int hit = sh.hit, klo = sh.klo, khi = sh.khi;
        // rows of two slots at a time: on a hit a slot for each part, else the
        // parts together on one slot after the other
        for (int s0 = 0; s0 < slots; s0 += 2) {
          if (hit) {
            s = s0 + part;
            if (s < slots) {
              if (s0 > 0) f.begin(d, places_of(s), chunk, sh.count[s][lw]);
              const float r = f.finish(d, klo, khi);
              if (lane < kSums) sh.row[part][lw][lane] = __fadd_rn(sh.row_a[s][lw][lane], r);
            }
          } else {
            for (s = s0; s < min(s0 + 2, slots); ++s) {
              float* row = sh.row[s & 1][lw];
              team_item<T, kA, kPassBand>(d, L, item_of(s), warp_of(s), lw, part, chunk, P, sh, s, nullptr, klo,
                                          khi, 0, row);
              if (part == 1 && lane < kSums) row[lane] = __fadd_rn(0.f, row[lane]);
            }
          }
          __syncthreads();
          // the item's pairwise halving, as far as these four warps go
          s = s0 + part;
          if (lw == 0 && s < slots && lane < kSums) {
            float (*r)[32] = sh.row[part];
            const float v = __fadd_rn(__fadd_rn(r[0][lane], r[2][lane]), __fadd_rn(r[1][lane], r[3][lane]));
            const int half = w + s * tp.workers;
            KF_GUARD(half < 2 * d->partial_cap, 13, half, d->partial_cap)
            packet_store(d->team_rows + (size_t)half * 32 + lane, __float_as_uint(v), tp.tag + it);
          }
          if (s0 + 2 < slots) __syncthreads();  // the rows are free again
        }
      }
    }
    if (warp == 0) {
      Wait wait;
      unsigned long long v;
      unsigned ahead;  // iterations; an earlier launch's tag lies far beyond kTeamTags
      bool ok = true;
      for (;;) {
        v = packet_load(d->team_msg + lane);
        ahead = (unsigned)(v >> 32) - (tp.tag + it);
        const bool same = ahead == __shfl_sync(0xffffffffu, ahead, 0);
        if (__all_sync(0xffffffffu, same && ahead - 1u < kTeamTags - 1u)) break;
        if (__any_sync(0xffffffffu, wait.ran_out(limit_ns))) {
          ok = false;
          break;
        }
        if (w >= halves) __nanosleep(KF_TEAM_IDLE_NS);  // nothing to do at this level
      }
      if (((it + ahead) ^ it) >= kTeamAcquire) fence_acquire();
      if (lane < 24) sh.xf[lane] = __uint_as_float((unsigned)v);
      if (lane == 24) sh.level = ok ? (int)(unsigned)v : -1;
      if (lane == 24) sh.it = it + ahead;
      if (lane == 25) sh.w0 = (int)(unsigned)v;
      if (lane == 26) sh.w1 = (int)(unsigned)v;
    }
    __syncthreads();
    it = sh.it;
    level = sh.level;
    w0 = sh.w0;
    w1 = sh.w1;
    if (level < 0) return;
  }
}

// The leader: medians for the record, the sums, the solve and update, the
// bookkeeping and the outputs.
__device__ void team_lead(const PairDesc* d, const TeamPair& tp, const PairInput& in,
                          unsigned long long limit_ns, const KParams& P, TeamShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PairState* st = d->st;
  // lane 0 of warp 0 keeps the pair's state in st (only this block writes it)
  if (threadIdx.x == 0) {
    double sT[12];
    init_state(d, in, P, sT);
  }
  __syncthreads();
  // what every solve takes, kept by warp 0
  const SolveLane sl = solve_lane();
  double Tmc[3], Tmt[3];
  load_tm(d->Tm, Tmc, Tmt);
  const double lam2c = 2.0 * in.lambda;
  int level = P.levels - 1, w0 = -1, w1 = -1;
  for (unsigned it = 0;; ++it) {
    const int chunk = level_chunk(level), fn = d->lv[level].fw * d->lv[level].fh;
    const int count = (fn + chunk - 1) / chunk;
    unsigned* hist = d->team_hist + (it % kTeamHists) * team_hist_words(P.bins);
    PairPre pre = {};
    if (warp == 0) {
      // the last iteration's clear (its warps met this one at the barrier) goes
      // before every message from here on; the workers' counts are awaited anyway
      fence_release();
      if (lane == 0) pre = load_pre(st, level);
      int N, kmed;
      const bool ok = warp_median(hist, P.bins, (unsigned)fn, limit_ns, N, kmed);
      if (lane == 0) {
        if (ok) {
          team_band(sh, P, N, kmed, w0, w1);
          pre.N = N;
          pre.kmed = kmed;
          pre.klo = sh.klo;
          pre.khi = sh.khi;
          pre.w0 = w0;
          pre.w1 = w1;
          st->hit = sh.hit;
        } else {
          sh.abort = 1;
        }
      }
    }
    __syncthreads();
    if (sh.abort) return;
    if (!sh.stop) {
      NextStep next = {};
      if (warp == 0) next = next_step(pre, level, P);
      // per sum (lane) the items' values: sub-sums over items sub, sub + 8, ...
      // (combine_and_solve's order)
      const unsigned long long want = tp.tag + it;
      Wait wait;
      bool ok = true;
      // a warp reads its sub-sum's packets together: one round trip covers 80
      // items (a 640x480 frame has 75)
      constexpr int kLeadWarps = kTeamBlock / 32, kSubs = kBlockWarps / kLeadWarps, kFly = 10;
      static_assert(kItemFold % kFly == 0, "folds where the other launches have them");
      FoldedSum sub[kSubs];
      for (int l0 = warp; l0 < count && ok; l0 += kFly * kBlockWarps) {
        unsigned long long a[kSubs][kFly], b[kSubs][kFly];
        for (;;) {
          bool all = true;
#pragma unroll
          for (int j = 0; j < kSubs; ++j)
#pragma unroll
            for (int i = 0; i < kFly; ++i) {
              const int l = l0 + j * kLeadWarps + i * kBlockWarps;
              a[j][i] = b[j][i] = want << 32;
              if (l < count && lane < kSums) {
                a[j][i] = packet_load(d->team_rows + (size_t)(2 * l) * 32 + lane);
                b[j][i] = packet_load(d->team_rows + (size_t)(2 * l + 1) * 32 + lane);
              }
            }
#pragma unroll
          for (int j = 0; j < kSubs; ++j)
#pragma unroll
            for (int i = 0; i < kFly; ++i) all = all && (a[j][i] >> 32) == want && (b[j][i] >> 32) == want;
          if (__all_sync(0xffffffffu, all)) break;
          if (__any_sync(0xffffffffu, wait.ran_out(limit_ns))) {
            ok = false;
            break;
          }
        }
#pragma unroll
        for (int j = 0; j < kSubs; ++j) {
          sub[j].room(kFly);
#pragma unroll
          for (int i = 0; i < kFly; ++i)
            if (l0 + j * kLeadWarps + i * kBlockWarps < count)
              sub[j].s.add(__fadd_rn(__uint_as_float((unsigned)a[j][i]), __uint_as_float((unsigned)b[j][i])));
        }
      }
      if (lane < kSums)
        for (int j = 0; j < kSubs; ++j) sh.part.put(warp + j * kLeadWarps, lane, sub[j], count);
      if (!ok) sh.abort = 1;
      __syncthreads();
      if (sh.abort) return;
      if (warp == 0) {
        if (lane < kSums) sh.sums[lane] = sh.part.total(lane, count);
        __syncwarp();
        double Tc[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) Tc[k] = sh.T[4 * k + (lane & 3)];
        auto publish = [&](const Solved& o, int nl, int nw0, int nw1) {
          const unsigned v = lane < 24 ? __float_as_uint(o.xf)
                                       : (unsigned)(lane == 24 ? nl : (lane == 25 ? nw0 : nw1));
          packet_store(d->team_msg + lane, v, tp.tag + it + 1u);
          if (lane < 12) sh.T[lane] = o.T;
          if (lane == 0) {
            sh.level = nl;
            sh.w0 = nw0;
            sh.w1 = nw1;
          }
        };
        if (solve_update(d, st, sh.sums, level, P, sh.hit ? 1 : 2, pre, next, sl, lam2c, Tc, Tmc, Tmt, publish) == -2)
          publish(Solved{}, -1, -1, -1);
      } else {
        // every worker has read this histogram (its sums are here): empty it
        for (int b = threadIdx.x - 32; b < team_hist_words(P.bins); b += kTeamBlock - 32) hist[b] = 0u;
      }
    } else {
      if (threadIdx.x == 0) {
        st->N = sh.N;
        st->status = KF_ERR_TOO_FEW_INLIERS;
        st->stopped = 1;
        sh.level = -1;
      }
      if (warp == 0) packet_store(d->team_msg + lane, lane == 24 ? 0xffffffffu : 0u, tp.tag + it + 1u);
    }
    __syncthreads();
    level = sh.level;
    w0 = sh.w0;
    w1 = sh.w1;
    if (level < 0) break;
  }
  if (threadIdx.x == 0) write_output(d, tp.out);
}

template <class T, int kA>
__global__ void __launch_bounds__(kTeamBlock, 1) k_icp_team(const __grid_constant__ TeamArgs A,
                                                            const __grid_constant__ KParams P) {
  extern __shared__ unsigned sh_hist[];
  __shared__ __align__(16) TeamShared sh;
  int p = 0;
  while (p + 1 < A.n && (int)blockIdx.x >= A.pair[p + 1].first) ++p;
  const TeamPair& tp = A.pair[p];
  const PairDesc* d = tp.d;
  const int rank = blockIdx.x - tp.first;
  if (threadIdx.x < 12) sh.T[threadIdx.x] = seed_entry(A.in[p], P, threadIdx.x);
  if (threadIdx.x == 0) {
    sh.matched = 0u;
    sh.abort = 0;
  }
  for (int b = threadIdx.x; b < P.bins; b += kTeamBlock) sh_hist[b] = 0u;
  __syncthreads();
  if (rank == 0) {
    team_lead(d, tp, A.in[p], A.limit_ns, P, sh);
  } else {
    if (threadIdx.x < 24) sh.xf[threadIdx.x] = xf_entry(sh.T, d->Tm, threadIdx.x);
    __syncthreads();
    team_work<T, kA>(d, tp, rank - 1, A.limit_ns, P, sh, sh_hist);
  }
}

}  // namespace

cudaError_t team_attributes(const KParams& P) {
  cudaError_t e = cudaSuccess;
#define KF_X(T, A)                                                                         \
  e = cudaFuncSetAttribute(k_icp_team<T, A>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                           kMaxBins * (int)sizeof(unsigned))
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return e;
}

int team_blocks(const KParams& P) {
  const int sm = P.bins * (int)sizeof(unsigned);
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
#define KF_X(T, A) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_icp_team<T, A>, kTeamBlock, sm)
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return sms * (KF_TEAM_PER_SM > 0 ? KF_TEAM_PER_SM : per);
}

cudaError_t launch_icp_team(const TeamArgs& args, int grid, const KParams& P, cudaStream_t s) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kTeamBlock);
  cfg.dynamicSmemBytes = (size_t)P.bins * sizeof(unsigned);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaSuccess;
#define KF_X(T, A) e = cudaLaunchKernelEx(&cfg, k_icp_team<T, A>, args, P)
  KF_ASSOC_SWITCH(P, KF_X);
#undef KF_X
  return e;
}

}  // namespace kf
