// Kernels around the histograms: the spatial signals where the streaming
// kernel does not apply, the dHash bits from cell sums, the bounded-wait
// probe of the failure path, and the bin check over arbitrary pixels. They
// share K1's grayscale and bin functions (ngff_device.cuh).
#include <algorithm>

#include "ngff_device.cuh"

namespace cofie {
namespace {

// The spatial signals (low-res difference, dHash) where the bulk-copy kernel
// does not apply: a width that is no multiple of 16, frames that do not start
// on a 16-byte boundary, or no verified multiply-high for the grayscale
// division. CTA x of the grid sums one slice of one frame's pixels by cell.
// As in the generic histogram kernel a frame's pixels split into a prologue
// of fewer than 16 pixels, whole 16-pixel groups that start on a 16-byte
// boundary (three 128-bit loads, two dp2a per pixel) and an epilogue of fewer
// than 16. Groups take no notice of where image rows end: in row-major order
// the cell columns of a row, and the first column of the row below, are
// consecutive runs of pixels, so with columns of at least 16 pixels (kWide) a
// group meets at most one boundary, the end of a cell column or of the row,
// and is split there as the bulk-copy kernel splits its groups; narrower
// columns take a loop over the pixels. A thread's next group is
// 16 kAnyThreads pixels on, so its row and column advance by additions, and
// its cell row by comparison with the row where the next one starts.
//
// Bound by issue slots and load latency together: 208 instructions a warp for 32
// groups of 48 bytes keep 64 % of the issue slots busy, DRAM runs at 68 % of its
// peak, and over half of a warp's wait is for its loads, so the more warps there
// are to cover them, the nearer the kernel comes to DRAM's rate.
// Hence registers for six CTAs per SM and sums formed as the pixels are
// decoded, without arrays of prefix sums (four CTAs: 5 % slower over 600
// frames of 854x480; eight, which spill: 7 %). Lanes of a warp hold
// neighbouring groups, of which several fall in one cell; each cell is kept
// kCellCopies times, a lane adding to copy lane mod kCellCopies (4 and 16
// copies measured the same). Those 600 frames (738 MB) take 0.12 ms, 6.2 TB/s;
// the kernel this one replaced, a CTA per frame with byte loads and a division
// per pixel, took 0.79 ms.
constexpr int kAnyThreads = 256;
constexpr uint32_t kAnyGroups = 2048;    // 16-pixel groups per CTA, fewer for small launches
constexpr uint32_t kAnyGroupsMin = 256;
constexpr uint32_t kCellCopies = 8;

template <bool kDiv, bool kWide>
__global__ void __launch_bounds__(kAnyThreads, 6) cells_any_kernel(SegTable segs, FeatArgs fa, LumaConsts L,
                                                                uint32_t* __restrict__ cells) {
  __shared__ __align__(16) uint32_t cell[256 * kCellCopies];
  __shared__ uint32_t colstart[17];
  pdl_trigger();
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t row = blockIdx.x / fa.slices, slice = blockIdx.x - row * fa.slices;
  uint32_t seg = 0;
  while (seg + 1 < segs.count && row >= segs.s[seg + 1].row0) ++seg;
  const uint8_t* frame = segs.s[seg].frames + static_cast<uint64_t>(row - segs.s[seg].row0) * fa.frame_bytes;
  const uint32_t gh = fa.grid_h, gw = fa.grid_w, W = fa.width, H = fa.height, n_cells = gh * gw;
  const uint32_t gh_shift = 31 - __clz(gh);  // 8 or 16 cell rows
  for (uint32_t i = tid; i < n_cells * kCellCopies; i += kAnyThreads) cell[i] = 0;
  if (tid <= gw) colstart[tid] = static_cast<uint32_t>((static_cast<uint64_t>(tid) * W + gw - 1) / gw);
  // first 16-byte aligned pixel: 3 p = -(frame mod 16) mod 16, and 3 * 11 = 1 mod 16
  const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(frame) & 15u);
  const uint32_t p_a = min(((16u - mis) * 11u) & 15u, fa.npix);
  const uint32_t G = (fa.npix - p_a) / 16;
  const uint32_t g0 = slice * fa.slice_groups, g1 = min(g0 + fa.slice_groups, G);
  const uint8_t* base = frame + 3ull * p_a;
  // a programmatic dependent has its slice fetched into L2 while it waits (a
  // hint, as in the generic histogram kernel)
  if (fa.ahead && tid == 0 && g0 < g1)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + 48ull * g0), "r"(48 * (g1 - g0)) : "memory");
  pdl_wait();  // no frame is read and no cell written before the kernel before this one has completed
  __syncthreads();

  const auto floor_y = [&](uint32_t v) { return kDiv ? v / L.den : __umulhi(v, L.magic_y); };
  const auto add = [&](uint32_t c, uint32_t sum) {
    if (COFIE_BOUND(c < n_cells)) atomicAdd(&cell[c * kCellCopies + (lane & (kCellCopies - 1))], sum);
  };
  // first image row of the cell row after crow
  const auto next_cell_row = [&](uint32_t crow) { return ((crow + 1) * H + gh - 1) >> gh_shift; };

  if (g0 + tid < g1) {
    const uint32_t q = p_a + 16 * (g0 + tid);
    const uint32_t dr = 16 * kAnyThreads / W, dx = 16 * kAnyThreads - dr * W;
    uint32_t r = q / W, x = q - r * W;
    uint32_t crow = r * gh / H, row_end = next_cell_row(crow);
#pragma unroll 1
    for (uint32_t g = g0 + tid; g < g1; g += kAnyThreads) {
      const uint4* p = reinterpret_cast<const uint4*>(base + 48ull * g);
      const uint4 a = __ldcs(p), b = __ldcs(p + 1), c = __ldcs(p + 2);
      // cell column of x: m_col is below 2^32 gw / W by at most 1, so the
      // estimate is the column or one less
      uint32_t cx = __umulhi(x, fa.m_col);
      cx += x >= colstart[cx + 1];
      const uint32_t c0 = crow * gw + cx;
      const uint32_t w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
      if (kWide) {
        const uint32_t s = min(colstart[cx + 1] - x, 16u);  // pixels of the group before the boundary
        uint32_t lo = 0, sum = 0;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
          uint32_t v[4];
          luma4(w[3 * k], w[3 * k + 1], w[3 * k + 2], L, v[0], v[1], v[2], v[3]);
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i) {
            const uint32_t y = floor_y(v[i]);
            sum += y;
            if (4 * k + i < s) lo += y;
          }
        }
        add(c0, lo);
        // past the boundary: the next column, or the first one of the row below
        if (s < 16) add(cx + 1 < gw || r + 1 >= row_end ? c0 + 1 : crow * gw, sum - lo);
      } else {
        uint32_t acc = 0, ci = c0, xx = x, rr = r, cc = cx, cr = crow, end = row_end, nx = colstart[cx + 1];
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
          uint32_t v[4];
          luma4(w[3 * k], w[3 * k + 1], w[3 * k + 2], L, v[0], v[1], v[2], v[3]);
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i, ++xx) {
            if (xx == nx) {
              add(ci, acc);
              acc = 0;
              if (++cc == gw) {
                cc = xx = 0;
                if (++rr >= end) end = next_cell_row(++cr);
              }
              ci = cr * gw + cc;
              nx = colstart[cc + 1];
            }
            acc += floor_y(v[i]);
          }
        }
        add(ci, acc);
      }
      if (g + kAnyThreads < g1) {
        x += dx;
        r += dr;
        if (x >= W) {
          x -= W;
          ++r;
        }
        while (r >= row_end) row_end = next_cell_row(++crow);
      }
    }
  }
  // the ragged edges: prologue (first slice of the frame) and epilogue (last)
  const auto scalar = [&](uint32_t q) {
    const uint8_t* px = frame + 3ull * q;
    const uint32_t yv = (L.w[0] * px[0] + L.w[1] * px[1] + L.w[2] * px[2] + L.half) / L.den;
    const uint32_t y = q / W, x = q - y * W;
    add((y * gh / H) * gw + x * gw / W, yv);
  };
  if (slice == 0 && tid < p_a) scalar(tid);
  if (slice == fa.slices - 1 && p_a + 16 * G + tid < fa.npix) scalar(p_a + 16 * G + tid);
  __syncthreads();
  for (uint32_t i = tid; i < n_cells; i += kAnyThreads) {
    const uint4 u = reinterpret_cast<const uint4*>(cell)[2 * i], w = reinterpret_cast<const uint4*>(cell)[2 * i + 1];
    const uint32_t sum = u.x + u.y + u.z + u.w + w.x + w.y + w.z + w.w;
    if (sum && COFIE_BOUND(row < segs.rows)) atomicAdd(cells + static_cast<uint64_t>(row) * n_cells + i, sum);
  }
}

// dHash from the 8 x 9 cell sums the kernel before it accumulated (row-major,
// 72 per frame): bit (r, c) = [S(r, c) n(r, c + 1) > S(r, c + 1) n(r, c)], the
// comparison of the two cell means without division. The cell row is zeroed
// for the next push once read.
__global__ void __launch_bounds__(96) dhash_finish_kernel(uint32_t* __restrict__ cells, FeatArgs fa,
                                                          uint32_t* __restrict__ bits) {
  pdl_trigger();
  pdl_wait();  // the cell sums of the streaming kernel before it
  const uint32_t row = blockIdx.x, tid = threadIdx.x;
  uint32_t* c = cells + static_cast<uint64_t>(row) * 72;
  if (tid < 64) {
    const uint32_t r = tid / 8, k = tid % 8;
    const uint64_t sa = c[r * 9 + k], sb = c[r * 9 + k + 1];
    const uint64_t na = static_cast<uint64_t>(fa.row_h[r]) * fa.col_w[k];
    const uint64_t nb = static_cast<uint64_t>(fa.row_h[r]) * fa.col_w[k + 1];
    const uint32_t word = __ballot_sync(0xffffffffu, sa * nb > sb * na);
    if ((tid & 31) == 0) bits[static_cast<uint64_t>(row) * 2 + (tid >> 5)] = word;
  }
  __syncthreads();
  if (tid < 72) c[tid] = 0;
}

// Failure-path probe: one thread waits, with the pipeline's bounded wait, for
// an mbarrier phase that nothing completes; when the bound runs out it sets
// the consumer-timeout bit, exactly as a stalled K1 consumer would, and the
// kernel returns normally.
__global__ void wait_probe_kernel(uint64_t timeout_ns, uint32_t* __restrict__ err) {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t b = smem_u32(&bar);
  mbar_init(b, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (!mbar_wait_bounded(b, 0, timeout_ns)) atomicOr(err, kErrConsumerTimeout);
}

// Diagnostic: the fast kernel's per-pixel luma and bin functions applied to
// 4-pixel groups (12 bytes each), one bin index per pixel.
template <int kBin>
__global__ void debug_bins_kernel(const uint8_t* __restrict__ px, uint64_t n_groups, LumaConsts L,
                                  uint8_t* __restrict__ out) {
  for (uint64_t g = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; g < n_groups;
       g += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint8_t* q = px + 12 * g;
    uint32_t w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      w[k] = q[4 * k] | (q[4 * k + 1] << 8) | (q[4 * k + 2] << 16) | (static_cast<uint32_t>(q[4 * k + 3]) << 24);
    uint32_t v0, v1, v2, v3;
    luma4(w[0], w[1], w[2], L, v0, v1, v2, v3);
    out[4 * g + 0] = static_cast<uint8_t>(bin_of<kBin>(v0, L));
    out[4 * g + 1] = static_cast<uint8_t>(bin_of<kBin>(v1, L));
    out[4 * g + 2] = static_cast<uint8_t>(bin_of<kBin>(v2, L));
    out[4 * g + 3] = static_cast<uint8_t>(bin_of<kBin>(v3, L));
  }
}

}  // namespace

cudaError_t launch_dhash_finish(uint32_t* cells, uint32_t rows, const FeatArgs& fa, uint32_t* bits, cudaStream_t st,
                                bool pdl) {
  const cudaError_t e = launch_dependent(pdl, dhash_finish_kernel, dim3(rows), dim3(96), 0, st, cells, fa, bits);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_cells_any(const SegTable& segs, const FeatArgs& fa, const LumaConsts& lc, uint32_t* cells,
                             int num_sms, cudaStream_t st, bool pdl) {
  FeatArgs f = fa;
  const uint32_t groups = std::max(1u, fa.npix / 16);  // at least the whole groups, whatever the alignment
  const auto slices = [&](uint32_t per) { return (groups + per - 1) / per; };
  f.slice_groups = kAnyGroups;  // smaller slices until the grid has four CTAs for every SM
  while (f.slice_groups > kAnyGroupsMin && static_cast<uint64_t>(slices(f.slice_groups)) * segs.rows < 4ull * num_sms)
    f.slice_groups /= 2;
  f.slices = slices(f.slice_groups);
  f.slice_groups = ((groups + f.slices - 1) / f.slices + kAnyThreads - 1) / kAnyThreads * kAnyThreads;  // even slices
  f.slices = slices(f.slice_groups);
  const uint64_t ctas = static_cast<uint64_t>(f.slices) * segs.rows;
  if (ctas > 0x7fffffffull) return cudaErrorInvalidConfiguration;
  const bool wide = fa.width / fa.grid_w >= 16;
  // a programmatic dependent only while its CTAs leave room on the SMs that
  // the kernel before it still holds (as the generic histogram kernel)
  pdl = pdl && ctas <= 4ull * num_sms;
  f.ahead = pdl ? 1u : 0u;
  const auto kernel = fa.use_magic ? (wide ? cells_any_kernel<false, true> : cells_any_kernel<false, false>)
                                   : (wide ? cells_any_kernel<true, true> : cells_any_kernel<true, false>);
  const cudaError_t e = launch_dependent(pdl, kernel, dim3(static_cast<uint32_t>(ctas)), dim3(kAnyThreads), 0, st, segs,
                                         f, lc, cells);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_wait_probe(uint64_t timeout_ns, uint32_t* err, cudaStream_t st) {
  wait_probe_kernel<<<1, 1, 0, st>>>(timeout_ns, err);
  return cudaGetLastError();
}

cudaError_t launch_debug_bins(const uint8_t* px, uint64_t n_groups, const LumaConsts& lc, int bin_path,
                              uint8_t* bins_out, cudaStream_t st) {
  const int threads = 256;
  const uint64_t want = (n_groups + threads - 1) / threads;
  const int grid = static_cast<int>(want < 4096 ? (want ? want : 1) : 4096);
  if (bin_path == kBinFast)
    debug_bins_kernel<kBinFast><<<grid, threads, 0, st>>>(px, n_groups, lc, bins_out);
  else
    debug_bins_kernel<kBinTwoStep><<<grid, threads, 0, st>>>(px, n_groups, lc, bins_out);
  return cudaGetLastError();
}

uint32_t take_bounds_errors_features() { return take_local_bounds_errors(); }

}  // namespace cofie
