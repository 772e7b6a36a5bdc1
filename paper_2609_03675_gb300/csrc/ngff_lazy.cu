// The retention rule without forced retention (L_max = 0, Eq. 5's second term
// off). With no bound on t - r(t) the reference frame can lie any distance
// back, so the gap maps of the other selection kernels do not apply. The
// stream's state between pushes is {t, the open scene-change run} and two ring
// rows: slot 0 holds c_{t-1}, slot 1 holds c_{r(t)}.
//
// Pushes of at most kLazyWalkFrames frames (more of each of several streams,
// fewer of wide rows) whose rows fit shared memory (lazy_walk_kernel): one CTA
// per stream walks the rule in frame order.
//
// Larger pushes, in three launches:
//   lazy_next_kernel   which frame would follow frame r as a reference does
//     not depend on what came before r: it is the first t > r with
//     max(d_adj(t), d(c_t, c_r)) >= tau_h, or an earlier scene change. A warp
//     finds it for each r of a tile, 32 frames at a time, among the rows that
//     the CTA has staged in shared memory (adjacent distances on the way);
//   lazy_chain_kernel  one CTA per stream follows those links from the
//     stream's reference: within blocks of 32 frames by pointer doubling for
//     all entries at once, then one step per block. A link that the staged
//     rows did not settle (no keep for many frames) is scanned for by the
//     whole CTA, as far as the next scene change. Scene changes depend only on
//     the adjacent distances and are found first, by a scan of the twin
//     comparison's run;
//   lazy_emit_kernel   with every frame's reference known, scores and keep
//     codes, eight lanes per frame.
// Bound by latency, as the other selections are. A walk by one warp, a window
// of 32 frames at a time between keeps, took 145 us for 2048 frames with a
// keep every few frames (B = 32, scene changes on); the three launches take 24,
// and the whole push of those frames, 640x360, 227 instead of 348 us. Pushes of
// 8 frames of 448x448 take 5.8 instead of 10.3 us each from a graph.
#include <algorithm>

#include "ngff_common.cuh"

namespace cofie {
namespace {

// One launch up to where the serial walk passes the cost of two more. Which of
// the two is faster depends on how often frames are kept, which the host does
// not know (32 bins, us a push from a graph, walked / linked, with a keep every
// 4, 20 and 300 frames): 260 frames 24.7 / 14.4, 11.4 / 14.5 and 10.0 / 20.6,
// 400 35.7 / 15.6, 15.2 / 15.6 and 13.5 / 19.4, 500 45.5 / 16.0, 18.4 / 16.1 and
// 16.0 / 20.1. The walks of several streams run beside one another: 16 streams
// of 300 39.9 / 33.5, 24.0 / 33.8 and 22.2 / 56.2, 64 of 500 163.9 / 160.7, 136.8 /
// 161.8 and 134.8 / 204.2.
// With rows of more than 64 words a walk is slower and links are as fast (128
// bins, 260 frames 56.6 / 19.3, 24.7 / 19.2 and 21.2 / 28.7).
constexpr uint32_t kLazyWalkFrames = 384, kLazyWalkWideFrames = 256, kLazyWalkManyFrames = 512, kLazyMany = 4;
constexpr size_t kLazyWalkSmem = 200 * 1024;
constexpr uint32_t kWalkFew = 16;
constexpr int kLazyThreads = 256;
constexpr uint32_t kLazyWarps = kLazyThreads / 32;
constexpr uint32_t kStageWords = 16384;  // 64 KiB of rows per CTA of the next kernel
constexpr uint32_t kStageRows = 256;
static_assert((kStageWords + kMaxBins) * 4 <= kSpreadSmem, "the next kernel's limit");
constexpr int kLinkThreads = 1024;
constexpr uint32_t kLinkWarps = kLinkThreads / 32;
constexpr uint32_t kLinkBlocks = 128;              // blocks of 32 frames per pass of the chain kernel
constexpr uint32_t kLinkTile = 32 * kLinkBlocks;
constexpr uint32_t kPer = kLinkBlocks / kLinkWarps;  // blocks per warp
constexpr uint32_t kScanFrames = kLinkThreads / 8;   // frames per pass of an open link's scan, four times as many
constexpr uint32_t kScanNarrow = 64;                 // with rows of at most 64 words
constexpr uint32_t kUnknown = 0xffffffffu;         // no keep among the staged rows, but frames beyond them

__device__ __forceinline__ uint32_t word_dist(uint32_t x, uint32_t y, uint32_t kind) {
  return kind == 1 ? static_cast<uint32_t>(__popc(x ^ y)) : (x > y ? x - y : y - x);
}

// The distance numerator between two feature rows of B words, by one thread.
// With kVec4 (B % 4 == 0, sums of differences) 16-byte words from the rotated
// word `rot` on, so that lanes reading rows B words apart touch distinct banks.
template <bool kVec4>
__device__ __forceinline__ uint32_t row_dist(const uint32_t* x, const uint32_t* y, uint32_t B, uint32_t rot,
                                             uint32_t kind) {
  uint32_t s = 0;
  if (kVec4) {
    const uint4* x4 = reinterpret_cast<const uint4*>(x);
    const uint4* y4 = reinterpret_cast<const uint4*>(y);
    uint32_t q = rot;
#pragma unroll 8
    for (uint32_t i = 0; i < B / 4; ++i) {
      const uint4 u = x4[q], v = y4[q];
      s += word_dist(u.x, v.x, 0) + word_dist(u.y, v.y, 0) + word_dist(u.z, v.z, 0) + word_dist(u.w, v.w, 0);
      if (++q == B / 4) q = 0;
    }
  } else {
#pragma unroll 4
    for (uint32_t b = 0; b < B; ++b) s += word_dist(x[b], y[b], kind);
  }
  return s;
}

// The twin comparison's run as a monoid: a frame ends the open run (reset,
// the run restarts at sum 0 after it) or adds its adjacent numerator to it.
struct LzRun {
  uint32_t reset;
  unsigned long long sum;
};
__device__ __forceinline__ LzRun lz_cat(LzRun x, LzRun y) { return y.reset ? y : LzRun{x.reset, x.sum + y.sum}; }
__device__ __forceinline__ LzRun lz_shfl_up(LzRun v, uint32_t off) {
  return LzRun{__shfl_up_sync(0xffffffffu, v.reset, off), __shfl_up_sync(0xffffffffu, v.sum, off)};
}

// ---------------------------------------------------------- small pushes

// Row stride in shared memory: lanes that read the same word of consecutive
// rows touch distinct banks.
__host__ __device__ constexpr uint32_t walk_stride(uint32_t B, bool vec4) { return vec4 ? B + 4 : B + 1; }

// The distance of two staged rows over words part, part + parts, ... (16-byte
// words with kVec4).
template <bool kVec4>
__device__ __forceinline__ uint32_t walk_dist(const uint32_t* x, const uint32_t* y, uint32_t B, uint32_t part,
                                              uint32_t parts, uint32_t kind) {
  uint32_t d = 0;
  if (kVec4) {
#pragma unroll 8
    for (uint32_t q = part; q < B / 4; q += parts) {
      const uint4 u = reinterpret_cast<const uint4*>(x)[q], v = reinterpret_cast<const uint4*>(y)[q];
      d += word_dist(u.x, v.x, 0) + word_dist(u.y, v.y, 0) + word_dist(u.z, v.z, 0) + word_dist(u.w, v.w, 0);
    }
  } else {
#pragma unroll 4
    for (uint32_t b = part; b < B; b += parts) d += word_dist(x[b], y[b], kind);
  }
  return d;
}

// Shared memory: sprev, sref and the push's n rows, padded; per frame adj, the
// rule's distance max(d_adj, d_ref), a keep mask and a code.
//   n <= kWalkFew: the distances of every frame to every reference it may have
//     (the stream's, or an earlier frame) at once, a warp per frame, lanes
//     sharing out references and words; then one thread walks the frames;
//   more frames: the adjacent distances by all threads, then one warp goes by
//     windows: the reference stays until the next keep, so lane l scores frame
//     f + l against it, one ballot finds the first keep, the frames up to it
//     stand, and the next window starts after it. All pairs at once took 247
//     us for 20 pushes of 48 frames of 224x224, the windows 173.
template <bool kVec4>
__global__ void __launch_bounds__(kLazyThreads) lazy_walk_kernel(SegTable segs, SelectArgs a, uint32_t* __restrict__ feat,
                                                                 uint32_t* __restrict__ ring,
                                                                 StreamState* __restrict__ state) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t sfew[kWalkFew * kWalkFew];  // frame j's distance to reference i at [j][i]; i > 0 is frame i - 1
  __shared__ uint32_t s_last;
  pdl_trigger();  // the next push's first-stage kernel may be scheduled; it waits for this grid before its work
  pdl_wait();     // every device read follows
  const Segment& sg = segs.s[blockIdx.x];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t B = a.bins, n = sg.n, P = walk_stride(B, kVec4);
  if (n == 0) return;
  uint32_t* sprev = smem;
  uint32_t* sref = sprev + P;
  uint32_t* rows = sref + P;
  uint32_t* sadj = rows + n * P;
  uint32_t* sd = sadj + n;
  uint32_t* smask = sd + n;    // n <= kWalkFew: keep bit per reference
  uint32_t* scode = smask + n;
  uint32_t* ring_s = ring + static_cast<uint64_t>(sg.stream) * 2 * B;
  uint32_t* feat_s = feat + static_cast<uint64_t>(sg.row0) * B;
  const unsigned long long t0 = state[sg.stream].t;
  const unsigned long long acc0 = t0 > 0 ? state[sg.stream].acc : 0ull;
  if (kVec4) {
    const uint32_t nq = B / 4;
#pragma unroll 2
    for (uint32_t i = tid; i < (n + 2) * nq; i += kLazyThreads) {
      const uint32_t r = i / nq, q = i - r * nq;
      reinterpret_cast<uint4*>(smem + r * P)[q] = i < 2 * nq ? reinterpret_cast<const uint4*>(ring_s)[i]
                                                             : reinterpret_cast<const uint4*>(feat_s)[i - 2 * nq];
    }
  } else {
    for (uint32_t i = tid; i < (n + 2) * B; i += kLazyThreads) {
      const uint32_t r = i / B;
      smem[r * P + i - r * B] = i < 2 * B ? ring_s[i] : feat_s[i - 2 * B];
    }
  }
  __syncthreads();
  if (n <= kWalkFew) {
    const uint32_t refs = n == 1 ? 2u : 1u << (32 - __clz(n)), i = lane & (refs - 1);
    for (uint32_t j = warp; j < n; j += kLazyWarps) {
      // frame 0 takes the frame before it, sprev, as its reference 1
      const bool valid = i <= j || (j == 0 && i == 1);
      const uint32_t* y = !valid || i == 0 ? sref : (j == 0 ? sprev : rows + (i - 1) * P);
      uint32_t d = walk_dist<kVec4>(rows + j * P, y, B, lane / refs, 32 / refs, a.dist_kind);
      for (uint32_t o = refs; o < 32; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      const uint32_t adj = t0 + j == 0 ? 0u : __shfl_sync(0xffffffffu, d, j ? j : 1u);
      // fp32(max) / 2N >= tau exactly when max >= x_tau (the smallest such numerator)
      const uint32_t m = __ballot_sync(0xffffffffu, lane <= j && max(adj, d) >= a.x_tau);
      if (lane <= j) sfew[j * kWalkFew + i] = d;
      if (lane == 0) {
        sadj[j] = adj;
        smask[j] = m;
      }
    }
  } else {
    for (uint32_t j = tid; j < n; j += kLazyThreads)
      sadj[j] = t0 + j == 0 ? 0u : walk_dist<kVec4>(rows + j * P, j ? rows + (j - 1) * P : sprev, B, 0u, 1u, a.dist_kind);
  }
  __syncthreads();
  if (warp == 0) {
    // scene flags by twin comparison, 32 frames at a time: a cut (d_adj >= T_b)
    // or a low difference (d_adj < T_s) ends the run, others join it, with a
    // gradual change where its sum first reaches T_b
    unsigned long long acc = acc0;
    if (a.scd)
      for (uint32_t f = 0; f < n; f += 32) {
        const uint32_t j = f + lane;
        const bool in = j < n && t0 + j != 0;
        const unsigned long long adj = in ? sadj[j] : 0ull;
        LzRun x = !in ? LzRun{0u, 0ull} : (adj >= a.x_cut || adj < a.x_grad) ? LzRun{1u, 0ull} : LzRun{0u, adj};
#pragma unroll
        for (uint32_t off = 1; off < 32; off <<= 1) {
          if (off >= n) break;  // lanes past the push are left out
          const LzRun o = lz_shfl_up(x, off);
          if (lane >= off) x = lz_cat(o, x);
        }
        const unsigned long long run = x.reset ? x.sum : acc + x.sum;  // the run's sum at frame j
        if (j < n) scode[j] = in && (adj >= a.x_cut || (adj >= a.x_grad && run >= a.x_cut && run - adj < a.x_cut));
        acc = __shfl_sync(0xffffffffu, run, min(n - f, 32u) - 1);
      }
    if (lane == 0) {
      state[sg.stream].t = t0 + n;
      state[sg.stream].g = 1;
      state[sg.stream].acc = acc;
    }
    __syncwarp();
    if (n <= kWalkFew) {
      if (lane == 0) {
        uint32_t cur = 0;
        for (uint32_t j = 0; j < n; ++j) {
          const uint32_t d = max(sadj[j], sfew[j * kWalkFew + cur]);
          const bool first = t0 + j == 0, nov = (smask[j] >> cur) & 1u, scene = a.scd && scode[j];
          sd[j] = d;
          scode[j] = first ? 3 : (nov ? 1 : (scene ? 4 : 0));
          if (first || nov || scene) cur = j + 1;
        }
        s_last = cur;
      }
    } else {
      uint32_t cur = 0;  // the same in every lane
      for (uint32_t f = 0; f < n;) {
        const uint32_t j = f + lane;
        const bool in = j < n, first = t0 + j == 0;
        uint32_t d = 0;
        if (in) d = max(sadj[j], walk_dist<kVec4>(cur ? rows + (cur - 1) * P : sref, rows + j * P, B, 0u, 1u, a.dist_kind));
        const bool nov = d >= a.x_tau, scene = a.scd && in && scode[j];
        const uint32_t bal = __ballot_sync(0xffffffffu, in && (first || nov || scene));
        const uint32_t upto = bal ? static_cast<uint32_t>(__ffs(bal)) - 1 : 31u;  // the last lane whose result stands
        if (in && lane <= upto) {
          sd[j] = d;
          scode[j] = first ? 3 : (nov ? 1 : (scene ? 4 : 0));
        }
        if (bal) cur = f + upto + 1;
        f += upto + 1;
      }
      if (lane == 0) s_last = cur;
    }
  }
  __syncthreads();
  for (uint32_t base = 0; base < n; base += kLazyThreads) {  // warps stay whole: the record takes a ballot
    const uint32_t j = base + tid;
    uint32_t code = 0;
    if (j < n) {
      code = scode[j];
      if (sg.scores) sg.scores[j] = code == 3 ? 0.0f : __fdiv_rn(static_cast<float>(sd[j]), a.two_n);
      if (sg.keep) sg.keep[j] = static_cast<uint8_t>(code);
    }
    const uint32_t bits = __ballot_sync(0xffffffffu, code != 0);
    if (lane == 0 && a.record)
      record_bits(a.record + static_cast<uint64_t>(sg.stream) * a.rec_words, a.rec_words, t0 + base + 32 * warp, bits);
  }
  const uint32_t last = s_last;
  for (uint32_t b = tid; b < B; b += kLazyThreads) {
    ring_s[b] = rows[(n - 1) * P + b];
    if (last) ring_s[B + b] = rows[(last - 1) * P + b];
  }
  if (a.hist_out)
    for (uint32_t i = tid; i < n * B; i += kLazyThreads) {
      const uint32_t r = i / B;
      a.hist_out[i] = rows[r * P + i - r * B];
    }
  if (a.zero_hist)
    for (uint32_t i = tid; i < n * B; i += kLazyThreads) feat_s[i] = 0;
}

size_t lazy_walk_smem(uint32_t n, uint32_t bins, bool vec4) {
  return (static_cast<size_t>(n + 2) * walk_stride(bins, vec4) + 4 * n) * 4;
}

// ---------------------------------------------------------- larger pushes

// Tile k of a segment is its frames [k F, k F + F); the CTA stages rows
// k F - 1 .. k F + rows_max - 2 of the segment.
template <bool kVec4>
__global__ void __launch_bounds__(kLazyThreads) lazy_next_kernel(SegTable segs, SelectArgs a, LazyArgs z,
                                                                 const uint32_t* __restrict__ feat,
                                                                 const uint32_t* __restrict__ ring,
                                                                 const StreamState* __restrict__ state) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t sadj[kStageRows];
  pdl_trigger();
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t B = a.bins, F = z.tile;
  uint32_t seg = 0, k = blockIdx.x, tiles = (segs.s[0].n + F - 1) / F;
  while (k >= tiles && seg + 1 < segs.count) {
    k -= tiles;
    tiles = (segs.s[++seg].n + F - 1) / F;
  }
  const Segment& sg = segs.s[seg];
  const uint32_t n = sg.n, j0 = k * F, end = min(n, j0 + z.stage_rows - 1), fn = min(F, n - j0);
  if (!COFIE_BOUND(j0 < n && end - j0 < kStageRows)) return;
  pdl_wait();  // the rows of the first-stage kernel, and the ring and state that the last push left
  const unsigned long long t0 = state[sg.stream].t;
  const uint32_t* feat_s = feat + static_cast<uint64_t>(sg.row0) * B;
  const uint32_t* ring_s = ring + static_cast<uint64_t>(sg.stream) * 2 * B;
  // staged row i is frame j0 + i - 1; before the push's first frame comes the ring's slot 0
  uint32_t* rows = smem;
  uint32_t* sref = smem + z.stage_rows * B;  // the stream's reference (tile 0)
  const uint32_t m = end - j0 + 1;
  const auto source = [&](uint32_t r) { return j0 + r > 0 ? feat_s + static_cast<uint64_t>(j0 + r - 1) * B : ring_s; };
  if (kVec4) {
    const uint32_t nq = B / 4;
#pragma unroll 4
    for (uint32_t i = tid; i < m * nq; i += kLazyThreads) {
      const uint32_t r = i / nq;
      reinterpret_cast<uint4*>(rows)[i] = reinterpret_cast<const uint4*>(source(r))[i - r * nq];
    }
  } else {
    for (uint32_t i = tid; i < m * B; i += kLazyThreads) {
      const uint32_t r = i / B;
      rows[i] = source(r)[i - r * B];
    }
  }
  if (k == 0)
    for (uint32_t b = tid; b < B; b += kLazyThreads) sref[b] = ring_s[B + b];
  __syncthreads();
  const uint32_t rot = kVec4 ? lane % max(B / 4, 1u) : 0u;
  for (uint32_t i = tid; i + 1 < m; i += kLazyThreads) {  // the adjacent distance of frame j0 + i
    uint32_t d = row_dist<kVec4>(rows + (i + 1) * B, rows + i * B, B, rot, a.dist_kind);
    if (t0 + j0 + i == 0) d = 0;
    sadj[i] = d;
    if (i < fn) z.adj[sg.row0 + j0 + i] = d;
  }
  __syncthreads();
  // reference fn of tile 0 stands for the stream's reference, whose first successor may be frame 0
  const bool before = k == 0 && t0 > 0;
  for (uint32_t r = warp; r < fn + (before ? 1u : 0u); r += kLazyWarps) {
    const bool pre = r == fn;
    const uint32_t* ref = pre ? sref : rows + (r + 1) * B;
    uint32_t next = end < n ? kUnknown : n;
    for (uint32_t f = pre ? 0u : r + 1; j0 + f < end; f += 32) {
      const uint32_t fl = f + lane;
      bool keep = false;
      if (j0 + fl < end)  // fp32(max) / 2N >= tau exactly when max >= x_tau (the smallest such numerator)
        keep = max(sadj[fl], row_dist<kVec4>(rows + (fl + 1) * B, ref, B, rot, a.dist_kind)) >= a.x_tau;
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      if (bal) {
        next = j0 + f + __ffs(bal) - 1;
        break;
      }
    }
    if (lane == 0) (pre ? z.next_pre[seg] : z.next[sg.row0 + j0 + r]) = next;
  }
}

// kN * kScanFrames frames from f0 on, eight lanes per frame: those before
// `stop` whose distances reach the threshold lower *found. True in the lanes
// that found one. Bound by the latency of a pass, so passes are short (a keep
// is near more often than not) and rows are read in whole lines: stills of 64x64
// with 256 bins and scenes 80 frames apart, whose links all have to be scanned
// for, take 191 us for 4096 frames and 643 us for 16384 (walked by one warp 580
// and 2247 us; with a thread per row and every scan on to the push's end, past
// the scene changes, 3.6 and 86 ms).
template <bool kVec4, uint32_t kN>
__device__ __forceinline__ bool scan_pass(const uint32_t* feat_s, const uint32_t* adj, const uint32_t* ref, uint32_t f0,
                                          uint32_t stop, const SelectArgs& a, uint32_t* found) {
  const uint32_t sub = threadIdx.x & 7, B = a.bins;
  const uint32_t* row[kN];
  uint32_t d[kN], d_adj[kN];
#pragma unroll
  for (uint32_t u = 0; u < kN; ++u) {
    const uint32_t f = min(f0 + u * kScanFrames + (threadIdx.x >> 3), stop - 1);
    row[u] = feat_s + static_cast<uint64_t>(f) * B;
    d_adj[u] = adj[f];
    d[u] = 0;
  }
  if (kVec4) {
#pragma unroll(kN == 1 ? 8 : 1)
    for (uint32_t q = sub; q < B / 4; q += 8) {
      const uint4 v = reinterpret_cast<const uint4*>(ref)[q];
#pragma unroll
      for (uint32_t i = 0; i < kN; ++i) {
        const uint4 u = reinterpret_cast<const uint4*>(row[i])[q];
        d[i] += word_dist(u.x, v.x, 0) + word_dist(u.y, v.y, 0) + word_dist(u.z, v.z, 0) + word_dist(u.w, v.w, 0);
      }
    }
  } else {
#pragma unroll 4
    for (uint32_t b = sub; b < B; b += 8) {
#pragma unroll
      for (uint32_t i = 0; i < kN; ++i) d[i] += word_dist(row[i][b], ref[b], a.dist_kind);
    }
  }
  bool any = false;
#pragma unroll
  for (uint32_t u = 0; u < kN; ++u) {
#pragma unroll
    for (uint32_t o = 4; o > 0; o >>= 1) d[u] += __shfl_xor_sync(0xffffffffu, d[u], o);
    const uint32_t f = f0 + u * kScanFrames + (threadIdx.x >> 3);
    if (f < stop && max(d_adj[u], d[u]) >= a.x_tau) {
      any = true;
      if (sub == 0) atomicMin(found, f);
    }
  }
  return any;
}

template <bool kVec4>
__global__ void __launch_bounds__(kLinkThreads) lazy_chain_kernel(SegTable segs, SelectArgs a, LazyArgs z,
                                                                  const uint32_t* __restrict__ feat,
                                                                  uint32_t* __restrict__ ring,
                                                                  StreamState* __restrict__ state) {
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* hop = smem;                    // [kLinkTile] the first frame past the block that is kept, entering at this one
  uint32_t* visit = hop + kLinkTile;       // [kLinkTile] the block's frames that are kept, entering at this one
  uint32_t* kept = visit + kLinkTile;      // [kLinkBlocks] kept frames
  uint32_t* scenes = kept + kLinkBlocks;   // [kLinkBlocks] scene changes
  uint32_t* after = scenes + kLinkBlocks;  // [kLinkBlocks] the first scene change in a later block of the tile, or ~0
  uint32_t* before = after + kLinkBlocks;  // [kLinkBlocks] 1 + the last kept frame before the block, 0: the stream's reference
  __shared__ uint32_t breset[kLinkBlocks];
  __shared__ unsigned long long bsum[kLinkBlocks];
  __shared__ unsigned long long s_acc;
  __shared__ uint32_t s_at, s_last, s_start, s_stop, s_found;
  pdl_trigger();
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Segment& sg = segs.s[blockIdx.x];
  const uint32_t B = a.bins, n = sg.n, row0 = sg.row0;
  pdl_wait();
  if (n == 0) return;
  const unsigned long long t0 = state[sg.stream].t;
  const uint32_t* feat_s = feat + static_cast<uint64_t>(row0) * B;
  uint32_t* ring_s = ring + static_cast<uint64_t>(sg.stream) * 2 * B;
  uint32_t* old_ref = z.old_ref + static_cast<uint64_t>(blockIdx.x) * B;  // the emit kernel's copy
  for (uint32_t b = tid; b < B; b += kLinkThreads) old_ref[b] = ring_s[B + b];
  const auto resume = [&](uint32_t r) { return min(n, r / z.tile * z.tile + z.stage_rows - 1); };  // the first frame not staged with r
  if (tid == 0) {
    s_acc = t0 > 0 ? state[sg.stream].acc : 0ull;
    s_at = t0 > 0 ? z.next_pre[blockIdx.x] : 0u;  // the first kept frame (or kUnknown)
    s_last = 0;
  }
  uint32_t carried = 0;  // warp 0: 1 + the last frame kept before the tile
  for (uint32_t c0 = 0; c0 < n; c0 += kLinkTile) {
    const uint32_t m = min(kLinkTile, n - c0), c1 = c0 + m;
    uint32_t next[kPer], adj[kPer];
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const uint32_t f = 32 * (warp + i * kLinkWarps) + lane;
      next[i] = f < m ? z.next[row0 + c0 + f] : n;
      adj[i] = a.scd && f < m ? z.adj[row0 + c0 + f] : 0u;
    }
    __syncthreads();  // the arrays are free, s_acc and s_at are set
    if (a.scd) {
      // scene flags: frame f cuts (d_adj >= T_b: a scene change that ends the
      // run), joins the run (T_s <= d_adj < T_b: a scene change when the run's
      // sum first reaches T_b) or ends it; the stream's first frame is neither
      LzRun incl[kPer];
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const uint32_t blk = warp + i * kLinkWarps, f = 32 * blk + lane;
        incl[i] = f >= m || t0 + c0 + f == 0 ? LzRun{0u, 0ull}
                  : (adj[i] >= a.x_cut || adj[i] < a.x_grad) ? LzRun{1u, 0ull} : LzRun{0u, adj[i]};
#pragma unroll
        for (uint32_t off = 1; off < 32; off <<= 1) {
          const LzRun o = lz_shfl_up(incl[i], off);
          if (lane >= off) incl[i] = lz_cat(o, incl[i]);
        }
        if (lane == 31) {
          breset[blk] = incl[i].reset;
          bsum[blk] = incl[i].sum;
        }
      }
      __syncthreads();
      const unsigned long long carry = s_acc;
      __syncthreads();
      if (warp == 0) {  // exclusive scan of the block totals, kPer consecutive ones per lane
        LzRun t[kPer], run{0u, 0ull};
#pragma unroll
        for (uint32_t i = 0; i < kPer; ++i) {
          t[i] = run;
          run = lz_cat(run, LzRun{breset[kPer * lane + i], bsum[kPer * lane + i]});
        }
        LzRun w = run;
#pragma unroll
        for (uint32_t off = 1; off < 32; off <<= 1) {
          const LzRun o = lz_shfl_up(w, off);
          if (lane >= off) w = lz_cat(o, w);
        }
        LzRun pre = lz_shfl_up(w, 1);
        if (lane == 0) pre = LzRun{0u, 0ull};
        __syncwarp();
#pragma unroll
        for (uint32_t i = 0; i < kPer; ++i) {
          const LzRun x = lz_cat(pre, t[i]);
          breset[kPer * lane + i] = x.reset;
          bsum[kPer * lane + i] = x.sum;
        }
        if (lane == 31) s_acc = w.reset ? w.sum : carry + w.sum;
      }
      __syncthreads();
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const uint32_t blk = warp + i * kLinkWarps, f = 32 * blk + lane;
        const LzRun x = lz_cat(LzRun{breset[blk], bsum[blk]}, incl[i]);
        const unsigned long long r = x.reset ? x.sum : carry + x.sum;  // the run's sum at f
        const bool scene = f < m && t0 + c0 + f != 0 &&
                           (adj[i] >= a.x_cut || (adj[i] >= a.x_grad && r >= a.x_cut && r - adj[i] < a.x_cut));
        const uint32_t bal = __ballot_sync(0xffffffffu, scene);
        if (lane == 0) scenes[blk] = bal;
      }
    } else if (tid < kLinkBlocks) {
      scenes[tid] = 0;
    }
    __syncthreads();
    if (warp == 0) {  // the first scene change after each block: a suffix minimum
      uint32_t first = kUnknown, t[kPer];
#pragma unroll
      for (int i = kPer - 1; i >= 0; --i) {
        t[i] = first;
        const uint32_t b = kPer * lane + i;
        if (scenes[b]) first = c0 + 32 * b + __ffs(scenes[b]) - 1;
      }
#pragma unroll
      for (uint32_t off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_down_sync(0xffffffffu, first, off);
        if (lane + off < 32) first = min(first, o);
      }
      uint32_t later = __shfl_down_sync(0xffffffffu, first, 1);
      if (lane == 31) later = kUnknown;
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) after[kPer * lane + i] = min(t[i], later);
      // a keep due beyond an earlier tile gives way to a scene change before it
      if (lane == 0 && s_at != kUnknown) s_at = min(s_at, first);
    }
    if (tid >= 32 && tid < 32 + kLinkBlocks) kept[tid - 32] = 0;
    __syncthreads();
    // links: within the block by doubling, past it the terminal frame's link
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const uint32_t blk = warp + i * kLinkWarps, f = 32 * blk + lane;
      const uint32_t up = lane < 31 ? scenes[blk] & (0xfffffffeu << lane) : 0u;
      const uint32_t scene = up ? c0 + 32 * blk + __ffs(up) - 1 : after[blk];
      uint32_t nx = next[i];
      if (nx == kUnknown) {
        if (f < m && scene < resume(c0 + f)) nx = scene;
      } else {
        nx = min(nx, scene);
      }
      uint32_t p = nx < min(c1, c0 + 32 * blk + 32) ? (nx - c0) & 31u : lane, mask = 1u << lane;
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        mask |= __shfl_sync(0xffffffffu, mask, p);
        p = __shfl_sync(0xffffffffu, p, p);
      }
      hop[f] = __shfl_sync(0xffffffffu, nx, p);
      visit[f] = mask;
    }
    __syncthreads();
    // one step per block; a link still open is scanned for by the whole CTA, as
    // far as the first scene change or the tile's end: a reference without a
    // keep until there is scanned for on in the next tile
    for (;;) {
      if (tid == 0) {
        uint32_t r = s_at, last = s_last;
        while (r < c1) {  // kUnknown and n end the loop too
          const uint32_t blk = (r - c0) >> 5;
          kept[blk] |= visit[r - c0];
          last = c0 + 32 * blk + 32 - __clz(visit[r - c0]);  // 1 + the last frame kept in the block
          r = hop[r - c0];
        }
        s_at = r;
        s_last = last;
        if (r == kUnknown) {  // the reference is frame last - 1 (or the stream's, last = 0)
          const uint32_t from = last > c0 ? last - c0 : 0;  // local frames from here on
          uint32_t scene = kUnknown;
          if (from < m) {
            const uint32_t blk = from >> 5, up = scenes[blk] & (0xffffffffu << (from & 31));
            scene = up ? c0 + 32 * blk + __ffs(up) - 1 : after[blk];
          }
          // the first frame that was neither staged with it nor scanned in an earlier tile
          s_start = max(c0, last ? resume(last - 1) : min(n, z.stage_rows - 1));
          s_found = s_stop = min(scene, c1);
        }
      }
      __syncthreads();
      if (s_at != kUnknown) break;
      const uint32_t stop = s_stop;
      const uint32_t* ref = s_last ? feat_s + static_cast<uint64_t>(s_last - 1) * B : old_ref;
      const uint32_t per = B <= kScanNarrow ? 4 * kScanFrames : kScanFrames;
      for (uint32_t f0 = s_start; f0 < stop; f0 += per) {
        const bool keep = B <= kScanNarrow ? scan_pass<kVec4, 4>(feat_s, z.adj + row0, ref, f0, stop, a, &s_found)
                                           : scan_pass<kVec4, 1>(feat_s, z.adj + row0, ref, f0, stop, a, &s_found);
        if (__syncthreads_or(keep)) break;
      }
      const uint32_t found = s_found;
      __syncthreads();
      if (found == c1 && c1 < n) break;  // open still
      if (tid == 0) s_at = found;
    }
    __syncthreads();
    if (warp == 0) {  // the last kept frame before each block: a prefix maximum over blocks
      uint32_t run = 0, t[kPer];
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const uint32_t b = kPer * lane + i;
        t[i] = run;
        if (kept[b]) run = c0 + 32 * b + 32 - __clz(kept[b]);
      }
      uint32_t w = run;
#pragma unroll
      for (uint32_t off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w = max(w, o);
      }
      uint32_t pre = __shfl_up_sync(0xffffffffu, w, 1);
      if (lane == 0) pre = 0;
      pre = max(pre, carried);
      carried = max(carried, __shfl_sync(0xffffffffu, w, 31));
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) before[kPer * lane + i] = max(pre, t[i]);
    }
    __syncthreads();
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const uint32_t blk = warp + i * kLinkWarps, f = 32 * blk + lane, bits = kept[blk];
      const uint32_t below = bits & ((1u << lane) - 1u);
      const uint32_t ref1 = below ? c0 + 32 * blk + 32 - __clz(below) : before[blk];
      if (f < m) z.ref[row0 + c0 + f] = (ref1 << 1) | ((scenes[blk] >> lane) & 1u);
      if (lane == 0 && 32 * blk < m && a.record)
        record_bits(a.record + static_cast<uint64_t>(sg.stream) * a.rec_words, a.rec_words, t0 + c0 + 32 * blk, bits);
    }
  }
  __syncthreads();
  const uint32_t last = s_last;  // 1 + the reference's frame, 0: unchanged
  for (uint32_t b = tid; b < B; b += kLinkThreads) {
    ring_s[b] = feat_s[static_cast<uint64_t>(n - 1) * B + b];
    if (last) ring_s[B + b] = feat_s[static_cast<uint64_t>(last - 1) * B + b];
  }
  if (tid == 0) {
    z.first[blockIdx.x] = t0 == 0;
    state[sg.stream].t = t0 + n;
    state[sg.stream].g = 1;
    state[sg.stream].acc = s_acc;
  }
}

template <bool kVec4>
__global__ void __launch_bounds__(kLazyThreads) lazy_emit_kernel(SegTable segs, SelectArgs a, LazyArgs z,
                                                                 const uint32_t* __restrict__ feat) {
  const uint32_t row = blockIdx.x * (kLazyThreads / 8) + (threadIdx.x >> 3), sub = threadIdx.x & 7;
  pdl_wait();  // references; the distances of the kernel before that one
  uint32_t seg = 0;
  while (seg + 1 < segs.count && row >= segs.s[seg + 1].row0) ++seg;
  const Segment& sg = segs.s[seg];
  const uint32_t B = a.bins, j = row - sg.row0;
  uint32_t d = 0, code = 0;
  if (row < segs.rows) {
    code = z.ref[row];
    const uint32_t ref1 = code >> 1;
    const uint32_t* x = feat + static_cast<uint64_t>(row) * B;
    const uint32_t* y = ref1 ? feat + static_cast<uint64_t>(sg.row0 + ref1 - 1) * B : z.old_ref + static_cast<uint64_t>(seg) * B;
    if (kVec4) {
      for (uint32_t q = sub; q < B / 4; q += 8) {
        const uint4 u = reinterpret_cast<const uint4*>(x)[q], v = reinterpret_cast<const uint4*>(y)[q];
        d += word_dist(u.x, v.x, 0) + word_dist(u.y, v.y, 0) + word_dist(u.z, v.z, 0) + word_dist(u.w, v.w, 0);
      }
    } else {
      for (uint32_t b = sub; b < B; b += 8) d += word_dist(x[b], y[b], a.dist_kind);
    }
  }
#pragma unroll
  for (uint32_t o = 4; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if (row < segs.rows && sub == 0) {
    const bool first = j == 0 && z.first[seg];
    const float s = first ? 0.0f : __fdiv_rn(static_cast<float>(max(z.adj[row], d)), a.two_n);
    if (sg.scores) sg.scores[j] = s;
    if (sg.keep) sg.keep[j] = first ? 3 : (s >= a.tau ? 1 : ((code & 1u) ? 4 : 0));
  }
}

constexpr size_t kLinkSmem = (2 * kLinkTile + 4 * kLinkBlocks) * 4;

}  // namespace

bool lazy_walk_fits(uint32_t longest, uint32_t streams, uint32_t bins) {
  const uint32_t most = streams >= kLazyMany ? kLazyWalkManyFrames : (bins > 64 ? kLazyWalkWideFrames : kLazyWalkFrames);
  return longest <= most && lazy_walk_smem(longest, bins, true) <= kLazyWalkSmem;
}

// words of the larger pushes' scratch: adj, next, ref per frame, then next_pre, first and old_ref per segment
size_t lazy_scratch_words(uint32_t max_frames, uint32_t bins) {
  return 3 * static_cast<size_t>(max_frames) + kMaxSegs * (2 + static_cast<size_t>(bins));
}

cudaError_t lazy_prepare() {
  const int walk = kLazyWalkSmem, next = static_cast<int>(kSpreadSmem);
  cudaError_t e = cudaSuccess;
  const auto limit = [&](const auto k, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  limit(lazy_walk_kernel<true>, walk);
  limit(lazy_walk_kernel<false>, walk);
  limit(lazy_next_kernel<true>, next);
  limit(lazy_next_kernel<false>, next);
  limit(lazy_chain_kernel<true>, static_cast<int>(kLinkSmem));
  limit(lazy_chain_kernel<false>, static_cast<int>(kLinkSmem));
  return e;
}

cudaError_t launch_lazy_walk(const SegTable& segs, const SelectArgs& a, uint32_t* feat, uint32_t* ring, StreamState* state,
                             cudaStream_t st, bool pdl) {
  uint32_t longest = 0;
  for (uint32_t i = 0; i < segs.count; ++i) longest = std::max(longest, segs.s[i].n);
  const bool vec = a.bins % 4 == 0 && a.dist_kind == 0;
  const cudaError_t e = launch_dependent(pdl, vec ? lazy_walk_kernel<true> : lazy_walk_kernel<false>, dim3(segs.count),
                                         dim3(kLazyThreads), spread_smem(lazy_walk_smem(longest, a.bins, vec), segs.count, kMaxSegs), st,
                                         segs, a, feat, ring, state);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_lazy_select(const SegTable& segs, const SelectArgs& a, uint32_t* scratch, uint32_t max_frames, int num_sms,
                               const uint32_t* feat, uint32_t* ring, StreamState* state, cudaStream_t st, bool pdl) {
  LazyArgs z{};
  z.old_ref = scratch;  // first: 16-byte aligned rows
  z.adj = z.old_ref + kMaxSegs * a.bins;
  z.next = z.adj + max_frames;
  z.ref = z.next + max_frames;
  z.next_pre = z.ref + max_frames;
  z.first = z.next_pre + kMaxSegs;
  z.stage_rows = std::min(kStageRows, kStageWords / a.bins);
  // 32 frames per tile, fewer while the SMs are not full or where few rows are staged
  z.tile = 32;
  while (z.tile > 8 && (segs.rows < z.tile * static_cast<uint32_t>(num_sms) || z.stage_rows < 4 * z.tile)) z.tile /= 2;
  uint32_t tiles = 0;
  for (uint32_t i = 0; i < segs.count; ++i) tiles += (segs.s[i].n + z.tile - 1) / z.tile;
  const bool vec = a.bins % 4 == 0 && a.dist_kind == 0;
  const uint32_t sms = static_cast<uint32_t>(num_sms);
  const size_t rows = static_cast<size_t>(z.stage_rows + 1) * a.bins * 4, smem = tiles <= sms ? spread_smem(rows, tiles, sms) : rows;
  cudaError_t e = launch_dependent(pdl, vec ? lazy_next_kernel<true> : lazy_next_kernel<false>, dim3(tiles),
                                   dim3(kLazyThreads), smem, st, segs, a, z, feat, static_cast<const uint32_t*>(ring),
                                   static_cast<const StreamState*>(state));
  if (e == cudaSuccess)
    e = launch_dependent(true, vec ? lazy_chain_kernel<true> : lazy_chain_kernel<false>, dim3(segs.count),
                         dim3(kLinkThreads), kLinkSmem, st, segs, a, z, feat, ring, state);
  if (e == cudaSuccess)
    e = launch_dependent(true, vec ? lazy_emit_kernel<true> : lazy_emit_kernel<false>,
                         dim3((segs.rows + kLazyThreads / 8 - 1) / (kLazyThreads / 8)), dim3(kLazyThreads), 0, st, segs, a,
                         z, feat);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

uint32_t take_bounds_errors_lazy() { return take_local_bounds_errors(); }

}  // namespace cofie
