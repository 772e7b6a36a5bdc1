// Selection of larger pushes in one launch (CoFiE Sec. 3.2, Eqs. 2-5): novelty
// distances, the rule and the outputs of a push of any number of frames.
//
// The gap g = t - r(t) lies in [1, L_max] (Eq. 5's second term retains a frame
// whenever g reaches L_max), so a frame's keep decision is one bit per
// possible gap, and a run of frames is a map from the gap before it to the gap
// after it. The push is cut into tiles of `tile` frames of one stream. A CTA
// takes one tile:
//   1. the tile's histogram rows and the rows before them (this push's rows, or
//      the stream's ring) are copied into shared memory, for `lags` lags at a
//      time (all L_max unless the rows are too wide), and the windowed
//      distances L1[j][k-1] = sum_b |c_t - c_{t-k}| and keep bits computed
//      there, a warp per frame, lane = lag;
//   2. the tile's gap map is composed for every entry gap at once (thread =
//      entry gap), noting the gap before each frame, and published;
//   3. the entry gap follows from the stream's gap and the maps of the tiles
//      before this one, of which at most kLookBack are composed: a tile
//      further on takes the known exit gap of the tile kLookBack before it;
//   4. scores, keep codes and record bits are written. The stream's last tile
//      also stores the ring and the state. Rows that no later tile reads are
//      zeroed for the next push.
// Tiles are handed out by a ticket in stream order, so a CTA only ever waits
// for tiles that are already running: no co-residency is needed. Every wait is
// bounded; one that runs out sets an error bit and goes on with an arbitrary
// gap. The last CTA to finish returns tickets and flags to zero.
//
// Bound by latency: a push's tables are a few MB at most, in L2. This kernel
// took the place of three dependent launches, one for the distances, one
// single-CTA scan of the tables that it wrote and a memset of the rows: 4096
// frames of 224x224 (B = 32, L_max = 30) pushed in 116 instead of 135 us (107
// with the histogram kernel of now), 480 of 1280x720 (B = 256, L_max = 60) in 211
// instead of 236 us.
// With padded rows a warp reads the frame's word once for its 32 lags: 3000
// frames of 224x224 (B = 128, L_max = 120) 125 -> 106 us, 8 of 448x448 (L_max =
// 120) 7.8 -> 7.4 us each from a graph. Rows that do not fit at once, staged for
// some lags at a time: 1500 frames of 224x224, B = L_max = 256, 723 (rows read
// from L2 by every lane) -> 159 us.
#include <algorithm>

#include "ngff_common.cuh"

namespace cofie {
namespace {

constexpr int kChainThreads = 256;
constexpr uint32_t kChainWarps = kChainThreads / 32;
constexpr uint32_t kLookBack = 128;            // tiles whose maps a tile composes
constexpr size_t kChainSmemMax = 200 * 1024;   // a CTA's tables and staged rows
constexpr uint32_t kChainMaxTile = 32;

static_assert(kMaxLmax <= kChainThreads, "a thread per entry gap");
static_assert(kLookBack <= kChainThreads, "a thread per flag");

// A tile's flag: 0 nothing yet, 1 its map is published, (g << 2) | 3 also its
// exit gap g is known.
constexpr uint32_t kMapReady = 1u, kExitKnown = 3u;

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t flag_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void flag_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The flag once it has all bits of `want`, or 0 after timeout_ns.
__device__ __forceinline__ uint32_t flag_wait(const uint32_t* p, uint32_t want, uint64_t timeout_ns) {
  uint32_t v = flag_acquire(p);
  if ((v & want) == want) return v;
  const uint64_t t0 = now_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i) {
      v = flag_acquire(p);
      if ((v & want) == want) return v;
    }
    if (now_ns() - t0 > timeout_ns) return 0;
  }
}

// sum_b |x_b - y_b| by one thread (16-byte words with kVec4). x is the same row
// in every lane; staged rows are padded so that lanes reading the same word of
// consecutive rows y touch distinct banks.
template <bool kVec4>
__device__ __forceinline__ uint32_t row_l1(const uint32_t* x, const uint32_t* y, uint32_t B, uint32_t kind) {
  uint32_t d = 0;
  if (kVec4) {
    const uint4* x4 = reinterpret_cast<const uint4*>(x);
    const uint4* y4 = reinterpret_cast<const uint4*>(y);
#pragma unroll 8
    for (uint32_t q = 0; q < B / 4; ++q) {
      const uint4 u = x4[q], v = y4[q];
      d = __usad(u.x, v.x, d);
      d = __usad(u.y, v.y, d);
      d = __usad(u.z, v.z, d);
      d = __usad(u.w, v.w, d);
    }
  } else if (kind == 1) {  // Hamming distance of bit vectors (dHash)
    for (uint32_t b = 0; b < B; ++b) d += __popc(x[b] ^ y[b]);
  } else {
#pragma unroll 4
    for (uint32_t b = 0; b < B; ++b) d = __usad(x[b], y[b], d);
  }
  return d;
}

// Words from one staged row to the next.
__host__ __device__ constexpr uint32_t chain_stride(uint32_t bins, bool vec4) { return vec4 ? bins + 4 : bins | 1; }

// Shared memory, in words: [the rows that `lags` lags need][the tile's rows, which
// with all lags at once (lags = l_max) are the last of the rows before][l1]
// [masks][maps of kLookBack tiles][gap before each frame, by entry gap][the
// warps' composed maps]
struct ChainLayout {
  uint32_t own, l1, mask, maps, gaps, comp, words;
  __host__ __device__ ChainLayout(uint32_t tile, uint32_t l_max, uint32_t mask_words, uint32_t stride, uint32_t lags) {
    const uint32_t map_words = 8 * mask_words;  // 32 mask_words entries of one byte
    own = (lags == l_max ? lags : lags + tile) * stride;
    l1 = own + tile * stride;
    mask = l1 + tile * l_max;
    maps = mask + tile * mask_words;
    gaps = maps + kLookBack * map_words;
    comp = gaps + tile * map_words;
    words = comp + kChainWarps * map_words;
  }
};

// kAll: the rows of all lags at once, staged with the tile's in one pass.
template <bool kVec4, bool kAll>
__global__ void __launch_bounds__(kChainThreads) select_chain_kernel(SegTable segs, SelectArgs a, ChainArgs c,
                                                                     uint32_t* __restrict__ hist,
                                                                     uint32_t* __restrict__ ring,
                                                                     StreamState* __restrict__ state) {
  extern __shared__ __align__(16) uint32_t csm[];
  __shared__ uint32_t s_seg, s_k, s_base, s_entry, s_bad;
  __shared__ uint32_t s_flag0;
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t B = a.bins, L = a.l_max, W = a.mask_words, F = c.tile;
  const uint32_t stride = 32 * W;  // bytes of a map
  const uint32_t P = chain_stride(B, kVec4);
  const uint32_t K = kAll ? L : c.lags;  // lags staged at a time: L, or a multiple of 32
  const ChainLayout lay(F, L, W, P, K);
  uint32_t* before = csm;            // the rows that the lags at hand need
  uint32_t* own = csm + lay.own;     // row j of the tile
  uint32_t* l1 = csm + lay.l1;
  uint32_t* mask = csm + lay.mask;
  uint8_t* maps = reinterpret_cast<uint8_t*>(csm + lay.maps);
  uint8_t* gaps = reinterpret_cast<uint8_t*>(csm + lay.gaps);
  uint8_t* comp = reinterpret_cast<uint8_t*>(csm + lay.comp);

  pdl_trigger();  // the next push's first-stage kernel may be scheduled; it waits for this grid before its work
  pdl_wait();     // every device read follows: the histograms, and the state and counters the last push left
  if (tid == 0) {
    const uint32_t t = atomicAdd(&c.sync[0], 1u);
    uint32_t seg = 0, base = 0, n = (segs.s[0].n + F - 1) / F;
    while (t >= base + n && seg + 1 < segs.count) {
      base += n;
      n = (segs.s[++seg].n + F - 1) / F;
    }
    s_seg = seg;
    s_base = base;
    s_k = t - base;
    s_bad = 0;
  }
  __syncthreads();
  const Segment& sg = segs.s[s_seg];
  const uint32_t k_tile = s_k, base = s_base, n = sg.n, j0 = k_tile * F, n_tiles = (n + F - 1) / F;
  if (!COFIE_BOUND(j0 < n && base + k_tile < c.n_tiles)) return;
  const uint32_t fn = min(F, n - j0);
  const bool last_tile = k_tile + 1 == n_tiles;
  // the stream's state, read before this tile's map is published: the last tile
  // writes it once it has seen every map
  const unsigned long long t0 = state[sg.stream].t;
  const uint32_t g0 = state[sg.stream].g;
  const uint32_t t0_slot = static_cast<uint32_t>(t0 % L);  // ring slot of the push's first frame
  uint32_t* hist_s = hist + static_cast<uint64_t>(sg.row0) * B;
  uint32_t* ring_s = ring + static_cast<uint64_t>(sg.stream) * L * B;
  // the push's frame jj; frames before the push lie in the ring (slots of
  // frames that never were are read, not used)
  const auto row_of = [&](int32_t jj) -> const uint32_t* {
    if (jj >= 0) return hist_s + static_cast<uint64_t>(jj) * B;
    uint32_t slot = t0_slot + static_cast<uint32_t>(jj + static_cast<int32_t>(L));  // jj >= -L
    if (slot >= L) slot -= L;
    return ring_s + static_cast<uint64_t>(slot) * B;
  };
  // frames first, first + 1, ... into consecutive staged rows; those more than
  // L before the push are no frame's lag and left out
  const auto stage = [&](uint32_t* to, int32_t first, uint32_t rows) {
    const uint32_t per = kVec4 ? B / 4 : B;
#pragma unroll 4
    for (uint32_t i = tid; i < rows * per; i += kChainThreads) {
      const uint32_t r = i / per, q = i - r * per;
      const int32_t jj = first + static_cast<int32_t>(r);
      if (!kAll && jj < -static_cast<int32_t>(L)) continue;
      if (kVec4)
        reinterpret_cast<uint4*>(to + r * P)[q] = reinterpret_cast<const uint4*>(row_of(jj))[q];
      else
        to[r * P + q] = row_of(jj)[q];
    }
  };

  // 1. rows, distances, keep bits
  if (!kAll) stage(own, static_cast<int32_t>(j0), fn);
  for (uint32_t k0 = 0; k0 < (kAll ? 1u : L); k0 += K) {  // lags k0 + 1 .. k0 + K
    if (!kAll && k0 > 0) __syncthreads();   // the rows of the lags before have been read
    stage(before, static_cast<int32_t>(j0) - static_cast<int32_t>(k0 + K), kAll ? L + fn : K + fn - 1);
    __syncthreads();
    for (uint32_t j = warp; j < fn; j += kChainWarps) {
      const unsigned long long t = t0 + j0 + j;
      const uint32_t* ct = own + j * P;
      uint32_t l_adj = !kAll && k0 > 0 ? l1[j * L] : 0u;  // lag 1
      for (uint32_t w = kAll ? 0 : k0 / 32; kAll ? w < W : 32 * w < min(k0 + K, L); ++w) {
        const uint32_t k = 32 * w + lane + 1;
        const bool valid = k <= L && k <= t;
        uint32_t d = row_l1<kVec4>(ct, valid ? (kAll ? ct - k * P : before + (j + K - (k - k0)) * P) : ct, B, a.dist_kind);
        if (!valid) d = 0;
        if (w == 0) l_adj = __shfl_sync(0xffffffffu, d, 0);
        if (k <= L) l1[j * L + k - 1] = d;
        // fp32(max) / 2N >= tau exactly when max >= x_tau (the smallest such numerator)
        const bool keep = k <= L && (max(l_adj, d) >= a.x_tau || k >= L);
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) mask[j * W + w] = m;
      }
    }
  }
  if (a.hist_out) {  // before the map is published: later tiles clear this one's rows after that
    for (uint32_t i = tid; i < fn * B; i += kChainThreads) {
      const uint32_t r = i / B;
      a.hist_out[static_cast<uint64_t>(j0) * B + i] = own[r * P + i - r * B];
    }
  }
  __syncthreads();

  // 2. the tile's gap map (entry and exit gaps less one, in bytes)
  uint8_t* my_map = c.maps + static_cast<uint64_t>(base + k_tile) * stride;
  uint32_t exit_gap = 0;
  if (tid < L) {
    uint32_t g = tid;
    for (uint32_t j = 0; j < fn; ++j) {
      gaps[j * stride + tid] = static_cast<uint8_t>(g);
      const bool keep = (mask[j * W + (g >> 5)] >> (g & 31)) & 1u;
      g = (keep || t0 + j0 + j == 0) ? 0u : g + 1u;  // the stream's first frame restarts the gap
    }
    (void)COFIE_BOUND(g < L);
    exit_gap = g;
    if (!last_tile) __stcg(my_map + tid, static_cast<uint8_t>(g));
  }
  __syncthreads();
  if (tid == 0 && !last_tile) {
    __threadfence();
    flag_release(c.flags + base + k_tile, kMapReady);
  }

  // 3. the entry gap
  const uint32_t lo = k_tile > kLookBack ? k_tile - kLookBack : 0;  // the earliest tile looked at
  const uint32_t first = lo > 0 ? lo + 1 : 0;                       // the earliest whose map is composed
  const uint32_t m = k_tile - first;
  if (k_tile > 0) {
    if (tid < k_tile - lo) {
      const uint32_t v = flag_wait(c.flags + base + lo + tid, lo > 0 && tid == 0 ? kExitKnown : kMapReady, c.timeout_ns);
      if (v == 0) s_bad = 1;
      if (tid == 0) s_flag0 = v;
    }
    __syncthreads();
    const uint32_t* src = reinterpret_cast<const uint32_t*>(c.maps + static_cast<uint64_t>(base + first) * stride);
    for (uint32_t i = tid; i < m * (stride / 4); i += kChainThreads) reinterpret_cast<uint32_t*>(maps)[i] = __ldcg(src + i);
    __syncthreads();
    // a warp composes a run of maps for every entry gap, one thread chains the runs
    const uint32_t per = (m + kChainWarps - 1) / kChainWarps, a0 = min(warp * per, m), a1 = min(a0 + per, m);
    for (uint32_t e = lane; e < L; e += 32) {
      uint32_t g = e;
      for (uint32_t i = a0; i < a1; ++i) g = maps[i * stride + g];
      comp[warp * stride + e] = static_cast<uint8_t>(g);
    }
    __syncthreads();
  }
  if (tid == 0) {
    uint32_t g = lo > 0 ? s_flag0 >> 2 : g0;
    if (t0 == 0 && lo == 0) g = 1;
    if (g < 1 || g > L) g = L;  // the state only ever holds [1, L]
    --g;
    if (k_tile > 0)
      for (uint32_t w = 0; w < kChainWarps; ++w) g = comp[w * stride + g];
    if (s_bad) {
      atomicOr(c.err, kErrChainTimeout);
      g = L - 1;
    }
    s_entry = g;
  }
  __syncthreads();
  const uint32_t entry = s_entry;
  if (tid == entry) {  // this thread's exit gap is the tile's
    if (last_tile) {
      state[sg.stream].t = t0 + n;
      state[sg.stream].g = exit_gap + 1;
      if (t0 == 0) state[sg.stream].acc = 0;
    } else {
      flag_release(c.flags + base + k_tile, ((exit_gap + 1) << 2) | kExitKnown);
    }
  }

  // 4. outputs, the record, ring and state, and the rows cleared
  if (warp == 0) {
    const uint32_t j = lane;
    bool kept = false;
    if (j < fn) {
      float s = 0.0f;
      uint8_t code = 3;
      if (t0 + j0 + j != 0) {
        uint32_t g = gaps[j * stride + entry];
        if (!COFIE_BOUND(g < L)) g = 0;
        s = __fdiv_rn(static_cast<float>(max(l1[j * L], l1[j * L + g])), a.two_n);
        code = s >= a.tau ? 1 : (g + 1 >= L ? 2 : 0);
      }
      if (sg.scores) sg.scores[j0 + j] = s;
      if (sg.keep) sg.keep[j0 + j] = code;
      kept = code != 0;
    }
    const uint32_t bits = __ballot_sync(0xffffffffu, kept);
    if (lane == 0 && a.record)
      record_bits(a.record + static_cast<uint64_t>(sg.stream) * a.rec_words, a.rec_words, t0 + j0, bits);
  }
  if (last_tile) {  // every tile before this one has read the ring and the state: their flags were seen
    const uint32_t keep_n = min(n, L);
    for (uint32_t i = tid; i < keep_n * B; i += kChainThreads) {
      const uint32_t r = i / B, b = i - r * B, jj = n - keep_n + r;
      const uint32_t v = kAll ? before[(L + jj - j0) * P + b] : hist_s[static_cast<uint64_t>(jj) * B + b];
      ring_s[static_cast<uint64_t>((t0_slot + jj) % L) * B + b] = v;
    }
    __syncthreads();  // the rows below have been copied
  }
  if (a.zero_hist) {
    // tiles up to this one have read their rows, later ones read from L rows
    // before them on
    const uint32_t z0 = j0 > L ? j0 - L : 0, z1 = last_tile ? n : (j0 + F > L ? j0 + F - L : 0);
    for (uint64_t i = static_cast<uint64_t>(z0) * B + tid; i < static_cast<uint64_t>(z1) * B; i += kChainThreads) hist_s[i] = 0;
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();  // this CTA's flags are written before it counts as finished
    s_bad = atomicAdd(&c.sync[1], 1u) == c.n_tiles - 1;
    __threadfence();
  }
  __syncthreads();
  if (s_bad) {  // the last CTA: nobody waits any more
    for (uint32_t i = tid; i < c.n_tiles; i += kChainThreads) c.flags[i] = 0;
    if (tid < 2) c.sync[tid] = 0;
  }
}

// Frames per tile: as few as keep the grid at about one CTA per SM, so that a
// short push spreads over the SMs and a long one composes few maps.
uint32_t chain_tile(const SegTable& segs, int num_sms) {
  uint32_t tile = 8;
  while (tile < kChainMaxTile && segs.rows > tile * static_cast<uint32_t>(num_sms)) tile *= 2;
  return tile;
}

}  // namespace

// A tile's ticket, map and look-back are a fixed cost that pays where there are
// distances to share out or a long scan to cut up. Left to the window and scan
// kernels, of which the second takes a CTA per stream (us a push from a graph,
// tiles / window and scan):
//   one stream, at most 64 words of distances per frame (dHash with L_max up to
//     32, histograms with L_max = 1), while 8-frame tiles are at most one per
//     SM: 65 frames of 224x224, dHash, 13.4 / 12.0, 1000 of 64x48 22.9 / 19.6,
//     but 4096 34.5 / 43.3; of histograms only past 500 frames (L_max = 1, 32
//     bins: 130 frames 9.6 / 9.6, 1000 17.2 / 15.7);
//   several streams and many frames, whose scans run beside one another: 70
//     frames of each of 64 streams with 32 bins 38.4 / 32.5, 100 of 32 streams
//     26.9 / 23.0, but 100 of 4 streams 10.5 / 11.2 and 300 of 64 streams 95.2 /
//     106.5; with 256 bins and L_max = 1 140 of 32 streams 66.8 / 45.4, 100 of 8
//     17.3 / 20.4.
bool select_chain_takes(const SegTable& segs, uint32_t longest, const SelectArgs& a, int num_sms) {
  if (longest <= select_small_max()) return true;
  const uint32_t work = a.l_max * a.bins, rows = segs.rows;
  if (segs.count == 1) return work > 64 || rows > 8u * num_sms || (a.dist_kind != 1 && rows < 500);
  if (work <= 64) return rows < 500;
  return work > 1024 || rows < (a.bins <= 64 ? 800u : 3000u) || rows > 9000;
}

uint32_t chain_max_tiles(uint32_t max_frames) { return max_frames / 8 + kMaxSegs + 1; }

cudaError_t chain_prepare() {
  for (const auto k : {select_chain_kernel<true, true>, select_chain_kernel<false, true>, select_chain_kernel<true, false>,
                       select_chain_kernel<false, false>}) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kChainSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_select_chain(const SegTable& segs, const SelectArgs& a, ChainArgs c, int num_sms, uint32_t* hist,
                                uint32_t* ring, StreamState* state, cudaStream_t st, bool pdl) {
  c.tile = chain_tile(segs, num_sms);
  c.n_tiles = 0;
  for (uint32_t i = 0; i < segs.count; ++i) c.n_tiles += (segs.s[i].n + c.tile - 1) / c.tile;
  const bool vec = a.bins % 4 == 0 && a.dist_kind == 0;
  const uint32_t stride = chain_stride(a.bins, vec);
  const auto smem = [&](uint32_t lags) {
    return ChainLayout(c.tile, a.l_max, a.mask_words, stride, lags).words * sizeof(uint32_t);
  };
  c.lags = a.l_max;  // every row that a tile reads at once, or as many multiples of 32 lags as fit
  if (smem(c.lags) > kChainSmemMax) {
    c.lags = (a.l_max - 1) / 32 * 32;  // below l_max
    while (c.lags > 32 && smem(c.lags) > kChainSmemMax) c.lags -= 32;
  }
  const bool all = c.lags == a.l_max;
  const auto kernel = vec ? (all ? select_chain_kernel<true, true> : select_chain_kernel<true, false>)
                          : (all ? select_chain_kernel<false, true> : select_chain_kernel<false, false>);
  const uint32_t sms = static_cast<uint32_t>(num_sms);
  const size_t bytes = c.n_tiles <= sms ? spread_smem(smem(c.lags), c.n_tiles, sms) : smem(c.lags);
  const cudaError_t e = launch_dependent(pdl, kernel, dim3(c.n_tiles), dim3(kChainThreads), bytes, st, segs, a, c, hist, ring,
                                         state);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

uint32_t take_bounds_errors_chain() { return take_local_bounds_errors(); }

}  // namespace cofie
