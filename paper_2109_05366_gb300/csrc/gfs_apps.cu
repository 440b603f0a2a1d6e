// Application-shaped consumers of the read path (the paper evaluates GPU
// applications that read their input files through GPUfs, Section 6.2):
//   gfs_rowdot     a row-major float32 matrix streamed by stripes of rows into
//                  per-row dot products with a resident vector;
//   gfs_histogram  an int32 array streamed into a histogram.
// Both gread their input in read_len pieces through the page cache, so every
// byte they consume came through the same path as the stride scan, and consume
// it where its pages lie (their sinks copy nothing); both also report checksums
// of the bytes they consumed.
#include <cuda_runtime.h>
#include <errno.h>

#include "gfs_device.cuh"
#include "gfs_host.h"

namespace gfs {
namespace {

constexpr uint32_t kThreads = 256;
constexpr uint32_t kSmemBins = 8192;  // histogram bins kept in shared memory (the heavy head of a Zipf law)

// Dot products of the rows of one gread (off: its first byte, whole rows) taken where
// their pages lie in the cache.  A warp takes consecutive rows, four at a time where
// they share a page, so that each load of the vector serves four rows; lane l takes the
// float4 columns l, l + 32, ... of a row in that order, whatever the pages.  A row cut
// by the end of a run of pages leaves its lanes' partial sums in `carry`, from where the
// next run goes on with them.
// Bound by HBM reads and the loads in flight.  Rows read from a gread buffer crossed HBM
// three times (out of the cache, into the buffer, back in): a cached 16384 x 8192 matrix
// took 303 us that way and takes 132 us in place.  (Two units a warp under way through
// shared memory: 130.  Checksums kept by row, with one 64-bit multiply-add a word: 152,
// a serial chain.)
struct RowdotSink {
  static constexpr bool kFar = false;
  static constexpr bool kArrive = true;
  // A row for every warp: with pieces of fewer rows most warps wait (first pass over a 2000 x
  // 8192 matrix in 64 KiB pages: 723 us in pieces of a page, 560 us so; 668 us through a buffer).
  __device__ __forceinline__ unsigned long long piece() const {
    const unsigned long long all = (kThreads / 32) * row_bytes;
    return all > dev::kPiece ? all : dev::kPiece;
  }
  const float4* vec;
  float* out;  // the gread's first row
  float4* carry;  // shared memory, 2 x 32; one half is read while the other is written
  unsigned long long off, row_bytes;
  uint32_t cols4, half;
  dev::Sums acc;

  // R whole rows that follow each other from p on (file offset o), all in one page.
  template <int R>
  __device__ __forceinline__ void rows_in_page(const uint8_t* p, unsigned long long o, uint32_t row,
                                               dev::Sums& part) const {
    constexpr int U = 8 / R;
    const uint32_t lane = threadIdx.x & 31u;
    float4 s[R];
#pragma unroll
    for (int i = 0; i < R; ++i) s[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t c = lane;
    for (; c + 32 * (U - 1) < cols4; c += 32 * U) {
      uint4 x[R][U];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u)
          x[i][u] = __ldcg(reinterpret_cast<const uint4*>(p + (size_t)i * row_bytes) + c + 32 * u);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float4 y = __ldg(vec + c + 32 * u);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          fma4(s[i], x[i][u], y);
          dev::sums_add16(part, x[i][u], o + (unsigned long long)i * row_bytes + 16ull * (c + 32 * u));
        }
      }
    }
    for (; c < cols4; c += 32) {
      const float4 y = __ldg(vec + c);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const uint4 x = __ldcg(reinterpret_cast<const uint4*>(p + (size_t)i * row_bytes) + c);
        fma4(s[i], x, y);
        dev::sums_add16(part, x, o + (unsigned long long)i * row_bytes + 16ull * c);
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) finish(s[i], row + (uint32_t)i);
  }

  // The part of row `row` that the view holds; pages may change inside it.
  __device__ __forceinline__ void row_any(const DevHandle& g, const dev::RunView& r, uint32_t row, dev::Sums& part) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long o = off + row * row_bytes, base = r.p << g.page_shift;
    const uint32_t c0 = r.lo > o ? (uint32_t)((r.lo - o) >> 4) : 0u;
    const uint32_t c1 = r.hi < o + row_bytes ? (uint32_t)((r.hi - o) >> 4) : cols4;
    float4 s = c0 ? carry[32 * half + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t c = c0 <= lane ? lane : lane + ((c0 - lane + 31u) & ~31u);
    for (; c < c1; c += 32 * 8) {
      uint4 x[8];
#pragma unroll
      for (uint32_t u = 0; u < 8; ++u)
        if (c + 32 * u < c1)
          x[u] = __ldcg(reinterpret_cast<const uint4*>(dev::run_at(g, r, o + 16ull * (c + 32 * u) - base)));
#pragma unroll
      for (uint32_t u = 0; u < 8; ++u)
        if (c + 32 * u < c1) {
          fma4(s, x[u], __ldg(vec + c + 32 * u));
          dev::sums_add16(part, x[u], o + 16ull * (c + 32 * u));
        }
    }
    if (c1 < cols4) carry[32 * (half ^ 1u) + lane] = s;
    else finish(s, row);
  }

  static __device__ __forceinline__ void fma4(float4& s, const uint4& x, const float4& y) {
    s.x = fmaf(__uint_as_float(x.x), y.x, s.x);
    s.y = fmaf(__uint_as_float(x.y), y.y, s.y);
    s.z = fmaf(__uint_as_float(x.z), y.z, s.z);
    s.w = fmaf(__uint_as_float(x.w), y.w, s.w);
  }
  __device__ __forceinline__ void finish(const float4& v, uint32_t row) const {
    float s = (v.x + v.y) + (v.z + v.w);
    for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(dev::kFull, s, d);
    if ((threadIdx.x & 31) == 0) out[row] = s;
  }

  __device__ __noinline__ void take(const DevHandle& g, const dev::RunView& r) {
    const uint32_t w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t first = (uint32_t)((r.lo - off) / row_bytes), last = (uint32_t)((r.hi - 1 - off) / row_bytes);
    const uint32_t per = (last - first + nw) / nw;  // rows a warp
    uint32_t row = first + w * per;
    const uint32_t stop = row + per < last + 1 ? row + per : last + 1;
    const unsigned long long base = r.p << g.page_shift;
    dev::Sums part{0ull, 0ull};
    while (row < stop) {
      const unsigned long long o = off + row * row_bytes;
      // whole rows from this one on that end before its page does
      uint32_t k = 0;
      if (o >= r.lo) {
        const unsigned long long page_end = (o | (g.page_size - 1u)) + 1;
        const unsigned long long lim = page_end < r.hi ? page_end : r.hi;
        while (k < 4 && row + k < stop && o + (k + 1) * row_bytes <= lim) ++k;
      }
      if (k == 0) {
        row_any(g, r, row, part);
        ++row;
        continue;
      }
      const uint8_t* p = dev::run_at(g, r, o - base);
      if (k == 4) rows_in_page<4>(p, o, row, part);
      else if (k >= 2) rows_in_page<2>(p, o, row, part);
      else rows_in_page<1>(p, o, row, part);
      row += k == 4 ? 4 : (k >= 2 ? 2 : 1);
    }
    half ^= 1u;
    acc.sum += part.sum;
    acc.hash += part.hash;
  }
};

// Block b reads stripes b, b + B, ...; a stripe is `stripe_rows` rows and is read
// in pieces of `rows_per_piece` rows.
__global__ void __launch_bounds__(kThreads, 2) k_rowdot(DevHandle g, int fid, uint32_t rows, uint32_t cols,
                                                     const float* __restrict__ vec, float* __restrict__ out,
                                                     uint32_t stripe_rows, uint32_t nstripes, uint32_t rows_per_piece,
                                                     unsigned long long* stripe_sum,
                                                     unsigned long long* stripe_hash, long long* status) {
  __shared__ float4 s_carry[64];
  const unsigned long long row_bytes = (unsigned long long)cols * 4;
  RowdotSink sink{reinterpret_cast<const float4*>(vec), out, s_carry, 0ull, row_bytes, cols / 4, 0u, {0ull, 0ull}};
  for (uint32_t st = blockIdx.x; st < nstripes; st += gridDim.x) {
    const uint32_t r0 = st * stripe_rows;
    const uint32_t r1 = rows - r0 > stripe_rows ? r0 + stripe_rows : rows;
    sink.acc = dev::Sums{0ull, 0ull};
    long long err = 0;
    for (uint32_t pr = r0, nr; pr < r1; pr += nr) {
      nr = rows_per_piece < r1 - pr ? rows_per_piece : r1 - pr;
      sink.off = (unsigned long long)pr * row_bytes;
      sink.out = out + pr;
      const long long n = dev::gread_impl(g, (int)blockIdx.x, fid, sink.off, nr * row_bytes, sink);
      if (n != (long long)(nr * row_bytes)) {
        err = n < 0 ? n : -5;
        break;
      }
    }
    dev::Sums acc = sink.acc;
    dev::block_sum2(acc.sum, acc.hash);
    if (threadIdx.x == 0) {
      stripe_sum[st] = acc.sum;
      stripe_hash[st] = acc.hash;
      if (err) atomicCAS((unsigned long long*)status, 0ull, (unsigned long long)err);
    }
    __syncthreads();
  }
  if (g.xfer != GFS_XFER_DMA)
    for (int i = 0; i < 4096; ++i)
      if (!dev::block_help(g, -1, true)) break;
}

// Counts the int32 values of a gread that starts at a multiple of 16, where their pages
// lie in the cache.  Bins below kSmemBins (the heavy head of a Zipf law) are counted in
// shared memory, the rest with one global atomic a value.  L2 adds to one address one after
// the other, so bins above kSmemBins that are hot are seen to: of every kSampled units a
// warp samples one.  Lanes that hold the same high bin there make it the warp's hot bin,
// counted in registers from then on; where several bins repeat at once, lanes that hold the
// same value add once (a match among the lanes, which does not pay otherwise).  64 MiB,
// cached, one atomic a value / so / always with the match: all 50000 10587 / 127 / 446 us,
// a tenth 50000 1194 / 270 / 505, 64 values from 8192 on 4161 / 2720 / 2686, Zipf law
// (s = 1.1) 193 / 195 / 378.  A last value of fewer than four bytes is not counted.
struct HistSink {
  static constexpr uint32_t kSampled = 8, kSeveral = 4, kOften = 8;
  static constexpr bool kFar = false;
  static constexpr bool kArrive = true;
  __device__ __forceinline__ uint32_t piece() const { return dev::kPiece; }
  enum Way { kPlain, kHot, kMatch };
  uint32_t* sh;
  uint32_t* hist;
  uint32_t nbins;
  uint32_t hot, hot_n;  // the warp's hot bin (0: none), and how often this lane met it
  unsigned long long bad;
  dev::Sums acc;

  __device__ __forceinline__ bool high(uint32_t v) const { return v >= kSmemBins && v < nbins; }
  // Whole warp: add what the lanes counted of the hot bin.
  __device__ __forceinline__ void flush() {
    const uint32_t n = __reduce_add_sync(dev::kFull, hot_n);
    if (n && (threadIdx.x & 31) == 0) atomicAdd(&hist[hot], n);
    hot_n = 0;
  }
  // Whole warp: look at x, one of the lanes' eight words each of a unit.  Returns the way of
  // counting it speaks for: a chance pair (a Zipf law has one a pass) speaks for none.
  __device__ __forceinline__ Way sample(const uint4* v, uint32_t x) {
    const bool h = high(x);
    const unsigned m = __ballot_sync(dev::kFull, h);
    unsigned same = 0;
    if (h) same = __match_any_sync(m, x);
    const unsigned again = __ballot_sync(dev::kFull, (same & (same - 1)) != 0u);
    if (again) {
      const uint32_t bin = __shfl_sync(dev::kFull, x, __ffs(again) - 1);
      const unsigned others = again & ~__ballot_sync(dev::kFull, x == bin);
      if (__popc(others) >= (int)kSeveral) return kMatch;
      uint32_t n = 0;
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) n += (v[k].x == bin) + (v[k].y == bin) + (v[k].z == bin) + (v[k].w == bin);
      if (bin != hot && __reduce_add_sync(dev::kFull, n) >= kOften) {
        flush();
        hot = bin;
      }
    }
    return hot ? kHot : kPlain;
  }
  // One value a lane.  kMatch: every lane of the warp calls it; `have`: it holds one.
  template <Way W>
  __device__ __forceinline__ void count(uint32_t v, bool have) {
    if (W != kMatch) {
      if (W == kHot && v == hot) ++hot_n;
      else if (v >= nbins) ++bad;
      else if (v < kSmemBins) atomicAdd(&sh[v], 1u);
      else atomicAdd(&hist[v], 1u);
      return;
    }
    if (have && v >= nbins) ++bad;
    if (have && v < kSmemBins && v < nbins) atomicAdd(&sh[v], 1u);
    const bool h = have && high(v);
    const unsigned m = __ballot_sync(dev::kFull, h);
    if (h) {
      const unsigned same = __match_any_sync(m, v);
      if ((threadIdx.x & 31) == (uint32_t)(__ffs(same) - 1)) atomicAdd(&hist[v], (uint32_t)__popc(same));
    }
  }
  // A lane's eight words of a unit, the first at file offset q, up to `end`.
  template <Way W>
  __device__ __forceinline__ void count_unit(const uint4* v, unsigned long long q, unsigned long long end) {
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k, q += 512) {
      count<W>(v[k].x, q + 4 <= end);
      count<W>(v[k].y, q + 8 <= end);
      count<W>(v[k].z, q + 12 <= end);
      count<W>(v[k].w, q + 16 <= end);
    }
  }
  __device__ __noinline__ void take(const DevHandle& g, const dev::RunView& r) {
    const uint32_t w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31u, units = dev::run_units(r);
    const unsigned long long end = r.hi & ~3ull;
    dev::Sums part{0ull, 0ull};
    uint32_t left = 0;
    Way way = kPlain;
    for (uint32_t u = w; u < units; u += nw) {
      const unsigned long long at = r.lo + ((unsigned long long)u << dev::kUnitShift), q = at + 16 * lane;
      uint4 v[8];
      dev::load_unit(g, r, at, v);
      dev::unit_sums(part, v, at);
      if (left == 0) {
        way = sample(v, v[0].x);
        if (way == kPlain) way = sample(v, v[4].z);
        left = kSampled;
      }
      --left;
      if (way == kMatch || at + (1u << dev::kUnitShift) > end) count_unit<kMatch>(v, q, end);
      else if (way == kHot) count_unit<kHot>(v, q, end);
      else count_unit<kPlain>(v, q, end);
    }
    acc.sum += part.sum;
    acc.hash += part.hash;
  }
};

// Block b reads pieces b, b + B, ... of the int32 file and counts values.
__global__ void __launch_bounds__(kThreads, 2) k_histogram(DevHandle g, int fid, unsigned long long size, uint32_t nbins,
                                                        uint32_t* __restrict__ hist, unsigned long long read_len,
                                                        unsigned long long* sums, long long* status) {
  __shared__ uint32_t sh[kSmemBins];
  for (uint32_t i = threadIdx.x; i < kSmemBins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const unsigned long long npieces = size / read_len + (size % read_len != 0);
  HistSink sink{sh, hist, nbins, 0u, 0u, 0ull, {0ull, 0ull}};
  for (unsigned long long pc = blockIdx.x; pc < npieces; pc += gridDim.x) {
    const long long n = dev::gread_impl(g, (int)blockIdx.x, fid, pc * read_len, read_len, sink);
    if (n < 0) {
      if (threadIdx.x == 0) atomicCAS((unsigned long long*)status, 0ull, (unsigned long long)n);
      break;
    }
  }
  sink.flush();
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < kSmemBins && i < nbins; i += blockDim.x)
    if (sh[i]) atomicAdd(&hist[i], sh[i]);
  unsigned long long total = sink.acc.sum, bad = sink.bad;
  dev::block_sum2(total, bad);
  if (threadIdx.x == 0) {
    atomicAdd(&sums[0], total);
    atomicAdd(&sums[1], bad);
  }
  if (g.xfer != GFS_XFER_DMA)
    for (int i = 0; i < 4096; ++i)
      if (!dev::block_help(g, -1, true)) break;
}

}  // namespace
}  // namespace gfs

using namespace gfs;

extern "C" int gfs_rowdot(gfs_ctx* ctx, int fid, uint32_t rows, uint32_t cols, const float* d_vec, float* d_out,
                          uint32_t stripe_rows, uint64_t read_len, uint32_t blocks, uint64_t* d_stripe_sum,
                          uint64_t* d_stripe_hash, int64_t* d_status, void* stream) {
  if (!ctx || !d_vec || !d_out || !d_stripe_sum || !d_stripe_hash || !d_status) return -EINVAL;
  if (fid < 0 || (size_t)fid >= ctx->files.size() || !ctx->files[fid].open) return -EBADF;
  if (rows == 0 || cols == 0 || cols % 4 || stripe_rows == 0 || blocks == 0) return -EINVAL;
  const uint64_t row_bytes = (uint64_t)cols * 4;
  if (read_len < row_bytes || read_len % row_bytes) return -EINVAL;  // pieces of whole rows
  if ((uint64_t)rows * row_bytes > ctx->files[fid].size) return -EINVAL;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return -ENODEV;
  const int rc = ensure_paper_state(ctx, blocks);
  if (rc) return rc;
  note_read(ctx, fid);
  DevHandle g = ctx->dev;
  g.reserve = frame_reserve(ctx, blocks, read_len);
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_status, 0, 8, s) != cudaSuccess) return -EINVAL;
  // a piece ends with its stripe: longer ones would not fit 32 bits, nor would their ends
  const uint32_t piece = (uint32_t)(read_len / row_bytes < stripe_rows ? read_len / row_bytes : stripe_rows);
  const uint32_t nstripes = rows / stripe_rows + (rows % stripe_rows != 0);
  k_rowdot<<<blocks, kThreads, 0, s>>>(g, fid, rows, cols, d_vec, d_out, stripe_rows, nstripes, piece,
                                       (unsigned long long*)d_stripe_sum, (unsigned long long*)d_stripe_hash, (long long*)d_status);
  return cudaGetLastError() == cudaSuccess ? 0 : -EINVAL;
}

extern "C" int gfs_histogram(gfs_ctx* ctx, int fid, uint32_t nbins, uint32_t* d_hist, uint64_t read_len,
                             uint32_t blocks, uint64_t* d_sums, int64_t* d_status, void* stream) {
  if (!ctx || !d_hist || !d_sums || !d_status) return -EINVAL;
  if (fid < 0 || (size_t)fid >= ctx->files.size() || !ctx->files[fid].open) return -EBADF;
  if (nbins == 0 || read_len == 0 || read_len % 16 || blocks == 0) return -EINVAL;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return -ENODEV;
  const int rc = ensure_paper_state(ctx, blocks);
  if (rc) return rc;
  note_read(ctx, fid);
  DevHandle g = ctx->dev;
  g.reserve = frame_reserve(ctx, blocks, read_len);
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_hist, 0, (size_t)nbins * 4, s) != cudaSuccess) return -EINVAL;
  if (cudaMemsetAsync(d_sums, 0, 16, s) != cudaSuccess) return -EINVAL;
  if (cudaMemsetAsync(d_status, 0, 8, s) != cudaSuccess) return -EINVAL;
  k_histogram<<<blocks, kThreads, 0, s>>>(g, fid, ctx->files[fid].size, nbins, d_hist, read_len,
                                          (unsigned long long*)d_sums, (long long*)d_status);
  return cudaGetLastError() == cudaSuccess ? 0 : -EINVAL;
}
