// Geometry: the synthetic np-Au stand-in (on the device; on the host with
// OpenMP for boxes that the device form does not take) and the derived integer
// structures on the device.
//
// The paper's own samples are grown from random 30 nm disks to a porosity of
// 0.70 (Sec. 2.1). Here the porous slab is a thresholded integer Gaussian
// random field with the requested porosity and correlation length; every
// solid cell touching gas is a catalytic node with b(x) active links
// (Appendix, after Eq. f_P_in). A caller mask may also mark inert solid
// (value 2): it bounces every array back and is never a node.
#include <omp.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "lbm_internal.h"

namespace lbm {

// ---------------------------------------------------------------------------
// Host: integer Gaussian random field and threshold
// ---------------------------------------------------------------------------
static int odd_box_width(double corr_len) {
  // nearest odd integer to sqrt(2 l^2 + 1): three box passes of width W have
  // variance 3 (W^2 - 1) / 12 ~ l^2 / 2, the Gaussian kernel of covariance
  // exp(-r^2 / (2 l^2))
  const double t = std::sqrt(2.0 * corr_len * corr_len + 1.0);
  int w = 1;
  double best = std::fabs(t - 1.0);
  for (int k = 3; k <= (int)t + 3; k += 2) {
    const double d = std::fabs(t - k);
    if (d < best) {  // strict: ties keep the smaller width
      best = d;
      w = k;
    }
  }
  return w;
}

// Periodic running-window sum of odd width W along one axis, exact in int64.
// Along x each row slides on its own; along y and z whole contiguous x-rows
// slide together, so every access walks memory in order.
static void box_axis(std::vector<int64_t> &v, std::vector<int64_t> &tmp, int nx, int ny, int nz, int axis, int W) {
  const int r = W / 2;
  const int64_t plane = (int64_t)nx * ny;
  if (axis == 0) {
#pragma omp parallel for schedule(static)
    for (int64_t row = 0; row < (int64_t)ny * nz; ++row) {
      const int64_t base = row * nx;
      auto at = [&](int k) { return v[base + ((k % nx) + nx) % nx]; };
      int64_t s = 0;
      for (int d = -r; d <= r; ++d) s += at(d);
      for (int k = 0; k < nx; ++k) {
        tmp[base + k] = s;
        s += at(k + r + 1) - at(k - r);
      }
    }
  } else {
    const int m = axis == 1 ? ny : nz;
    const int64_t stride = axis == 1 ? nx : plane;       // distance between successive lines
    const int64_t outer = axis == 1 ? nz : ny;            // independent groups
    const int64_t outer_stride = axis == 1 ? plane : nx;
#pragma omp parallel
    {
      std::vector<int64_t> acc(nx);
#pragma omp for schedule(static)
      for (int64_t o = 0; o < outer; ++o) {
        const int64_t base = o * outer_stride;
        auto row = [&](int k) { return &v[base + (int64_t)(((k % m) + m) % m) * stride]; };
        std::fill(acc.begin(), acc.end(), 0);
        for (int d = -r; d <= r; ++d) {
          const int64_t *p = row(d);
          for (int x = 0; x < nx; ++x) acc[x] += p[x];
        }
        for (int k = 0; k < m; ++k) {
          int64_t *out = &tmp[base + (int64_t)k * stride];
          for (int x = 0; x < nx; ++x) out[x] = acc[x];
          const int64_t *add = row(k + r + 1), *sub = row(k - r);
          for (int x = 0; x < nx; ++x) acc[x] += add[x] - sub[x];
        }
      }
    }
  }
  v.swap(tmp);
}

void grf_mask(int nx, int ny, int nz, int z0, int z1, double porosity, double corr_len, uint64_t seed,
              uint8_t *mask) {
  const int64_t n = (int64_t)nx * ny * nz, plane = (int64_t)nx * ny;
  std::vector<int64_t> v(n), tmp(n);
#pragma omp parallel for schedule(static)
  for (int64_t c = 0; c < n; ++c) {
    int64_t s = 0;
    for (uint64_t k = 0; k < 12; ++k) s += (int64_t)(splitmix64_next(seed ^ ((uint64_t)c * 12 + k)) >> 48);
    v[c] = s - 12 * 32768;
  }
  const int W = odd_box_width(corr_len);
  for (int axis = 0; axis < 3; ++axis)
    for (int pass = 0; pass < 3; ++pass) box_axis(v, tmp, nx, ny, nz, axis, W);
  std::vector<int64_t>().swap(tmp);

  std::memset(mask, 0, (size_t)n);
  const int64_t n_slab = plane * (z1 - z0);
  if (n_slab <= 0) return;
  const int64_t K = (int64_t)std::llrint(porosity * (double)n_slab);  // ties to even
  struct KV {
    int64_t v, i;
  };
  std::vector<KV> kv(n_slab);
#pragma omp parallel for schedule(static)
  for (int64_t k = 0; k < n_slab; ++k) {
    const int64_t c = (int64_t)z0 * plane + k;
    kv[k] = {v[c], c};
  }
  auto less = [](const KV &a, const KV &b) { return a.v < b.v || (a.v == b.v && a.i < b.i); };
  if (K > 0 && K < n_slab) std::nth_element(kv.begin(), kv.begin() + K, kv.end(), less);
#pragma omp parallel for schedule(static)
  for (int64_t k = 0; k < n_slab; ++k) mask[kv[k].i] = (k < K) ? 0 : 1;
}

double chord_length(int nx, int ny, int nz, int z0, int z1, const uint8_t *mask) {
  const int64_t plane = (int64_t)nx * ny;
  int64_t nf = 0, runs = 0;
#pragma omp parallel for reduction(+ : nf, runs) schedule(static)
  for (int z = z0; z < z1; ++z) {
    for (int y = 0; y < ny; ++y) {
      bool row_all = true;
      for (int x = 0; x < nx; ++x) {
        const int64_t c = z * plane + (int64_t)y * nx + x;
        if (mask[c]) {
          row_all = false;
          continue;
        }
        ++nf;
        runs += mask[c - x + (x == 0 ? nx - 1 : x - 1)];
        runs += mask[z * plane + (int64_t)(y == 0 ? ny - 1 : y - 1) * nx + x];
        runs += (z == z0) ? 1 : mask[c - plane];
      }
      runs += row_all;
    }
    for (int x = 0; x < nx; ++x) {
      bool col_all = true;
      for (int y = 0; y < ny && col_all; ++y) col_all = !mask[z * plane + (int64_t)y * nx + x];
      runs += col_all;
    }
  }
  if (nf == 0 || runs == 0) return 0.0;
  return 3.0 * (double)nf / (double)runs;
}

// ---------------------------------------------------------------------------
// Device: the same sample, bit for bit (whole numbers throughout)
// ---------------------------------------------------------------------------
//
// The field is kept as two 32-bit halves in two of the geometry's own arrays
// (its node-count and index arrays, written only afterwards), so a sample takes
// no device memory beyond the geometry's; the selection's histogram and the
// results use the neighbour masks' array. Per axis one launch: a block holds
// whole lines in shared memory and makes the three box passes there, so the
// field crosses memory once per axis in place (nine passes over two arrays
// otherwise), and the noise is formed in the first launch.
//
// Bound by latency and launches (15 of them) at ordinary sizes: a new
// 128x128x256 sample with its simulation and two fields takes 1.85 ms, 22 ms
// with the host's generator on 16 cores.
constexpr int kGenThreads = 256;
constexpr int kGenBins = 2048;  // of a selection pass: 11 bits of the key
constexpr int kGenValuePasses = 6, kGenIndexPasses = 3;
struct GenState {
  long long vmin, vmax;         // of the slab's values
  unsigned long long prefix;    // the threshold's leading bits found so far (value - vmin)
  unsigned long long nf, runs;  // chord length: fluid cells and fluid runs
  uint32_t rank;                // of the threshold among the cells that share the prefix
  uint32_t equal;               // how many those are
  uint32_t index;               // leading bits of the threshold's cell (ties: lower cell first)
  uint32_t done;                // blocks that have added to the histogram
};
// scratch in the neighbour masks' array: histogram, state, chunk hashes
constexpr int64_t kGenStateAt = kGenBins * sizeof(uint32_t);
constexpr int64_t kGenHashAt = kGenStateAt + 128;
static_assert(sizeof(GenState) <= 128, "room of the state");

// Lines per block along an axis of m cells: 32 (a full 128-byte row of each
// half) unless three blocks of them no longer fit an SM (72 KB each), then
// fewer, down to 8 (one 32-byte sector), and below that only where even a
// block alone on its SM (200 KB) holds no more; 0: a line too long, above
// 6,400 cells, which the host's passes take.
constexpr size_t gen_shared(int m, int lines) { return 2 * sizeof(int64_t) * (size_t)m * (lines + 1); }
static int gen_lines(int m) {
  int c = 32;
  while (c > 8 && gen_shared(m, c) > 72 * 1024) c /= 2;
  while (c > 0 && gen_shared(m, c) > 200 * 1024) c /= 2;
  return c;
}

__global__ void gen_init_kernel(uint32_t *hist, GenState *s, uint32_t rank, uint32_t n_slab) {
  for (int k = threadIdx.x; k < kGenBins; k += blockDim.x) hist[k] = 0;
  if (threadIdx.x == 0) {
    GenState v{};
    v.vmin = INT64_MAX;
    v.vmax = INT64_MIN;
    v.rank = rank;
    v.equal = n_slab;
    *s = v;
  }
}

// One axis: three periodic running sums of odd width W along lines of m
// cells; AXIS 0 forms the noise first, AXIS 2 also finds the smallest and
// largest value of the slab's cells. In shared memory cell k of line c lies at
// k (lines + 1) + c: lines side by side, so that neighbouring threads (lines)
// use different banks, the odd pitch doing the same for the x axis, whose
// loads run along a line.
template <int AXIS>
__global__ void __launch_bounds__(kGenThreads) gen_axis_kernel(uint32_t *lo, int32_t *hi, int nx, int ny, int nz,
                                                               int lines_log2, int W, uint64_t seed, int z0, int z1,
                                                               GenState *st) {
  extern __shared__ long long gen_sh[];
  const int C = 1 << lines_log2, pitch = C + 1;
  const int m = AXIS == 0 ? nx : AXIS == 1 ? ny : nz;
  const int64_t plane = (int64_t)nx * ny, n_lines = AXIS == 0 ? (int64_t)ny * nz : AXIS == 1 ? (int64_t)nx * nz : plane;
  const int64_t l0 = (int64_t)blockIdx.x << lines_log2;
  const int here = (int)(n_lines - l0 < C ? n_lines - l0 : C);
  auto cell = [&](int c, int k) -> int64_t {
    const int64_t l = l0 + c;
    if (AXIS == 0) return l * nx + k;
    if (AXIS == 1) return (int64_t)((uint32_t)l / (uint32_t)nx) * plane + (int64_t)k * nx + (uint32_t)l % (uint32_t)nx;
    return l + (int64_t)k * plane;
  };
  long long *a = gen_sh, *b = gen_sh + (int64_t)m * pitch;
  for (int e = threadIdx.x; e < m * C; e += kGenThreads) {
    const int c = AXIS == 0 ? e / m : e & (C - 1), k = AXIS == 0 ? e - c * m : e >> lines_log2;
    if (c >= here) continue;
    const int64_t i = cell(c, k);
    long long v;
    if (AXIS == 0) {
      v = -12 * 32768;
#pragma unroll
      for (uint64_t j = 0; j < 12; ++j) v += (long long)(splitmix64_next(seed ^ ((uint64_t)i * 12 + j)) >> 48);
    } else {
      v = (long long)(((unsigned long long)(uint32_t)hi[i] << 32) | lo[i]);
    }
    a[k * pitch + c] = v;
  }
  // each thread slides the window over one stretch of one line; a window of
  // more than a line takes in the whole line W / m times
  const int c = threadIdx.x & (C - 1), stretch = (m + (kGenThreads >> lines_log2) - 1) / (kGenThreads >> lines_log2);
  const int k0 = (threadIdx.x >> lines_log2) * stretch, k1 = k0 + stretch < m ? k0 + stretch : m;
  const int r = W / 2, whole = W / m, rest = W % m;
  for (int pass = 0; pass < 3; ++pass) {
    __syncthreads();
    if (k0 < k1 && c < here) {
      unsigned long long s = 0;
      if (whole > 0) {
        for (int k = 0; k < m; ++k) s += (unsigned long long)a[k * pitch + c];
        s *= (unsigned long long)whole;
      }
      int first = (int)(((int64_t)k0 - r) % m), next;  // the window's first cell
      first += first < 0 ? m : 0;
      next = first;
      for (int d = 0; d < rest; ++d) {
        s += (unsigned long long)a[next * pitch + c];
        next = next + 1 == m ? 0 : next + 1;
      }
      for (int k = k0; k < k1; ++k) {
        b[k * pitch + c] = (long long)s;
        s += (unsigned long long)a[next * pitch + c] - (unsigned long long)a[first * pitch + c];
        next = next + 1 == m ? 0 : next + 1;
        first = first + 1 == m ? 0 : first + 1;
      }
    }
    long long *t = a;
    a = b;
    b = t;
  }
  __syncthreads();
  long long vmin = INT64_MAX, vmax = INT64_MIN;
  for (int e = threadIdx.x; e < m * C; e += kGenThreads) {
    const int ce = AXIS == 0 ? e / m : e & (C - 1), k = AXIS == 0 ? e - ce * m : e >> lines_log2;
    if (ce >= here) continue;
    const int64_t i = cell(ce, k);
    const long long v = a[k * pitch + ce];
    lo[i] = (uint32_t)v;
    hi[i] = (int32_t)(v >> 32);
    if (AXIS == 2 && k >= z0 && k < z1) {
      vmin = v < vmin ? v : vmin;
      vmax = v > vmax ? v : vmax;
    }
  }
  if (AXIS == 2) {
    for (int o = 16; o > 0; o >>= 1) {
      const long long p = __shfl_xor_sync(0xffffffffu, vmin, o), q = __shfl_xor_sync(0xffffffffu, vmax, o);
      vmin = p < vmin ? p : vmin;
      vmax = q > vmax ? q : vmax;
    }
    if ((threadIdx.x & 31) == 0 && vmin <= vmax) {
      atomicMin(&st->vmin, vmin);
      atomicMax(&st->vmax, vmax);
    }
  }
}

// Pass `pass` of the radix selection of the cell of the given rank in (value,
// cell) order among the slab's n_slab cells (lo, hi: of the slab's first):
// counts the digit that follows the leading bits found so far over the cells
// that share them; the last block to finish takes the digit in which the rank
// falls. Six passes of up to 11 bits over the value's distance from the
// smallest one (those beyond the bits that the slab's range needs do nothing),
// then three over the cell number where several cells share the threshold's
// value.
__global__ void __launch_bounds__(kGenThreads) gen_select_kernel(const uint32_t *lo, const int32_t *hi, int64_t n_slab,
                                                                 int pass, uint32_t *hist, GenState *st) {
  __shared__ uint32_t sh[kGenBins];
  __shared__ uint32_t part[kGenThreads / 32];
  __shared__ bool last;
  const GenState s = *st;
  const unsigned long long range = (unsigned long long)s.vmax - (unsigned long long)s.vmin;
  const int bits = range ? 64 - __clzll((long long)range) : 0;
  const bool by_index = pass >= kGenValuePasses;
  int above, w;  // bits of the key above this pass's digit and in it
  if (by_index) {
    if (s.equal <= 1) return;
    const int q = pass - kGenValuePasses;  // 31 bits: 11, 10, 10
    above = q == 0 ? 0 : 1 + 10 * q;
    w = q == 0 ? 11 : 10;
  } else {
    above = 11 * pass;
    if (above >= bits) return;
    w = bits - above < 11 ? bits - above : 11;
  }
  const int shift = (by_index ? 31 : bits) - above - w;
  for (int k = threadIdx.x; k < kGenBins; k += kGenThreads) sh[k] = 0;
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * kGenThreads + threadIdx.x; i < n_slab; i += (int64_t)gridDim.x * kGenThreads) {
    const unsigned long long key =
        (((unsigned long long)(uint32_t)hi[i] << 32) | lo[i]) - (unsigned long long)s.vmin;
    uint32_t digit;
    bool mine;
    if (by_index) {
      mine = key == s.prefix && (uint32_t)((uint64_t)i >> (shift + w)) == s.index;
      digit = (uint32_t)((uint64_t)i >> shift) & ((1u << w) - 1u);
    } else {
      mine = above == 0 || (key >> (shift + w)) == s.prefix;
      digit = (uint32_t)(key >> shift) & ((1u << w) - 1u);
    }
    if (mine) atomicAdd(&sh[digit], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kGenBins; k += kGenThreads)
    if (sh[k]) atomicAdd(&hist[k], sh[k]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the bin that holds the rank: 8 bins per thread, scanned over the block
  constexpr int kPer = kGenBins / kGenThreads;
  uint32_t cnt[kPer], sum = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) sum += cnt[j] = __ldcg(&hist[threadIdx.x * kPer + j]);
  uint32_t before = sum;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t p = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += p;
  }
  if (lane == 31) part[wid] = before;
  __syncthreads();
  before -= sum;
  for (int q = 0; q < wid; ++q) before += part[q];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t bin = threadIdx.x * kPer + j;
    if (s.rank >= before && s.rank - before < cnt[j]) {
      if (by_index) st->index = (s.index << w) | bin;
      else st->prefix = (s.prefix << w) | bin;
      st->rank = s.rank - before;
      if (!by_index) st->equal = cnt[j];
    }
    before += cnt[j];
    hist[bin] = 0;
  }
  if (threadIdx.x == 0) st->done = 0;
}

// The slab's mask: fluid where (value, cell) lies below the threshold.
__global__ void gen_mask_kernel(const uint32_t *lo, const int32_t *hi, int64_t n_slab, const GenState *st, uint8_t *mask) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_slab) return;
  const unsigned long long key =
      (((unsigned long long)(uint32_t)hi[i] << 32) | lo[i]) - (unsigned long long)st->vmin;
  mask[i] = !(key < st->prefix || (key == st->prefix && (uint32_t)i < st->index));
}

// Fluid cells and fluid runs of the slab's planes (the chord length's two
// counts): one thread per cell, the rows along x and the columns along y that
// are fluid from end to end counted by their first cell's thread (most meet
// solid at once).
__global__ void __launch_bounds__(kGenThreads) gen_chord_kernel(const uint8_t *mask, int nx, int ny, int z0, int z1, GenState *st) {
  const int64_t plane = (int64_t)nx * ny, n = plane * (z1 - z0);
  unsigned nf = 0, runs = 0;
  for (int64_t i = (int64_t)blockIdx.x * kGenThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kGenThreads) {
    const int z = z0 + (int)((uint32_t)i / (uint32_t)plane);
    const int xy = (int)((uint32_t)i % (uint32_t)plane), y = xy / nx, x = xy - y * nx;
    const uint8_t *p = mask + (int64_t)z * plane + xy;
    if (*p) continue;
    ++nf;
    runs += p[x == 0 ? nx - 1 : -1] + p[y == 0 ? (int64_t)(ny - 1) * nx : -(int64_t)nx] + (z == z0 ? 1 : p[-plane]);
    if (x == 0) {
      int k = 1;
      while (k < nx && !p[k]) ++k;
      runs += k == nx;
    }
    if (y == 0) {
      int k = 1;
      while (k < ny && !p[(int64_t)k * nx]) ++k;
      runs += k == ny;
    }
  }
  nf = __reduce_add_sync(0xffffffffu, nf);
  runs = __reduce_add_sync(0xffffffffu, runs);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&st->nf, (unsigned long long)nf);
    atomicAdd(&st->runs, (unsigned long long)runs);
  }
}

// FNV-1a of a mask of 0s and 1s, in parallel: a byte b turns h into
// (h ^ b) P = (h + d) P with d = 0 for b = 0, and for b = 1 -1 or +1 by h's
// lowest bit, which (P being odd) the number of ones so far decides. So h after
// a chunk of N bytes is P^N h_0 + sum d_k P^(N - k), and a piece's share of the
// sum is known up to a sign: the parity of the ones before it. One block per
// piece of 64 KiB, 256 bytes a thread; out: the share with an even number of
// ones before the piece, and the piece's own parity.
__host__ __device__ inline unsigned long long fnv_power(uint32_t e) {
  unsigned long long r = 1, b = kFnvPrime;
  for (; e; e >>= 1, b *= b)
    if (e & 1u) r *= b;
  return r;
}
constexpr int kHashBytes = 256, kHashPiece = kGenThreads * kHashBytes;
static_assert(kHashChunk % kHashPiece == 0, "whole pieces per chunk");
__global__ void __launch_bounds__(kGenThreads) gen_hash_kernel(const uint8_t *mask, int64_t n, unsigned long long *out) {
  __shared__ uint32_t odd[kGenThreads / 32];
  __shared__ unsigned long long total[kGenThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t at = ((int64_t)blockIdx.x * kGenThreads + threadIdx.x) * kHashBytes;
  const int m = at >= n ? 0 : (n - at < kHashBytes ? (int)(n - at) : kHashBytes);
  const int64_t chunk_end = (at / kHashChunk + 1) * kHashChunk < n ? (at / kHashChunk + 1) * kHashChunk : n;
  unsigned long long s = 0;
  uint32_t ones = 0;
  for (int k = 0; k < m; ++k) {
    if (mask[at + k]) s += (ones++ & 1u) ? 1ull : ~0ull;
    s *= kFnvPrime;
  }
  const uint32_t ball = __ballot_sync(0xffffffffu, ones & 1u);
  if (lane == 0) odd[wid] = __popc(ball) & 1u;
  __syncthreads();
  uint32_t before = __popc(ball & ((1u << lane) - 1u)), all = 0;
  for (int q = 0; q < kGenThreads / 32; ++q) {
    before += q < wid ? odd[q] : 0u;
    all += odd[q];
  }
  unsigned long long h = m ? ((before & 1u) ? 0ull - s : s) * fnv_power((uint32_t)(chunk_end - at - m)) : 0ull;
  for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
  if (lane == 0) total[wid] = h;
  __syncthreads();
  if (threadIdx.x == 0) {
    h = 0;
    for (int q = 0; q < kGenThreads / 32; ++q) h += total[q];
    out[2 * blockIdx.x] = h;
    out[2 * blockIdx.x + 1] = all & 1u;
  }
}

bool sample_on_device(const lbm_geometry_desc *d) {
  const int64_t n = (int64_t)d->nx * d->ny * d->nz;
  const int64_t pieces = (n + kHashPiece - 1) / kHashPiece;
  return !d->mask && n * (int64_t)sizeof(uint32_t) >= kGenHashAt + 16 * pieces && gen_lines(d->nx) > 0 &&
         gen_lines(d->ny) > 0 && gen_lines(d->nz) > 0 &&
         (d->bc_z == LBM_BC_PERIODIC || (d->slab_z0 >= 2 && d->slab_z1 <= d->nz - 2));
}

cudaError_t generate_sample(lbm_geometry *g, double porosity, double corr_len, cudaStream_t st) {
  const int64_t n = g->n, plane = g->plane, n_slab = plane * (g->z1 - g->z0);
  uint32_t *lo = reinterpret_cast<uint32_t *>(g->idx);
  int32_t *hi = g->b;
  char *scratch = reinterpret_cast<char *>(g->nbm_dense);
  uint32_t *hist = reinterpret_cast<uint32_t *>(scratch);
  GenState *state = reinterpret_cast<GenState *>(scratch + kGenStateAt);
  unsigned long long *hash = reinterpret_cast<unsigned long long *>(scratch + kGenHashAt);
  const int W = odd_box_width(corr_len);
  const int64_t K = (int64_t)std::llrint(porosity * (double)n_slab);  // ties to even
  cudaError_t e = cudaMemsetAsync(g->mask, 0, (size_t)n, st);
  if (e != cudaSuccess) return e;
  gen_init_kernel<<<1, kGenThreads, 0, st>>>(hist, state, (uint32_t)K, (uint32_t)n_slab);
  const unsigned blocks = (unsigned)std::min<int64_t>((n_slab + kGenThreads - 1) / kGenThreads, 152 * 8);
  if (n_slab > 0 && K <= 0) {
    e = cudaMemsetAsync(g->mask + g->z0 * plane, 1, (size_t)n_slab, st);
  } else if (K < n_slab) {
    auto axis = [&](auto kernel, int m, int64_t lines) {
      const int c = gen_lines(m);
      const size_t bytes = gen_shared(m, c);
      int log2 = 0;
      while ((1 << log2) < c) ++log2;
      cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      if (r != cudaSuccess) return r;
      kernel<<<(unsigned)((lines + c - 1) / c), kGenThreads, bytes, st>>>(lo, hi, g->nx, g->ny, g->nz, log2, W, g->seed,
                                                                       g->z0, g->z1, state);
      return cudaGetLastError();
    };
    e = axis(gen_axis_kernel<0>, g->nx, (int64_t)g->ny * g->nz);
    if (e == cudaSuccess) e = axis(gen_axis_kernel<1>, g->ny, (int64_t)g->nx * g->nz);
    if (e == cudaSuccess) e = axis(gen_axis_kernel<2>, g->nz, plane);
    if (e != cudaSuccess) return e;
    const int64_t at = g->z0 * plane;
    for (int pass = 0; pass < kGenValuePasses + kGenIndexPasses; ++pass)
      gen_select_kernel<<<blocks, kGenThreads, 0, st>>>(lo + at, hi + at, n_slab, pass, hist, state);
    gen_mask_kernel<<<(unsigned)((n_slab + 255) / 256), 256, 0, st>>>(lo + at, hi + at, n_slab, state, g->mask + at);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  if (n_slab > 0) gen_chord_kernel<<<blocks, kGenThreads, 0, st>>>(g->mask, g->nx, g->ny, g->z0, g->z1, state);
  const int64_t pieces = (n + kHashPiece - 1) / kHashPiece;
  gen_hash_kernel<<<(unsigned)pieces, kGenThreads, 0, st>>>(g->mask, n, hash);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  std::vector<char> back((size_t)(kGenHashAt - kGenStateAt + 16 * pieces));
  if ((e = cudaMemcpyAsync(back.data(), scratch + kGenStateAt, back.size(), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  GenState s;
  std::memcpy(&s, back.data(), sizeof(s));
  g->delta = s.nf && s.runs ? 3.0 * (double)s.nf / (double)s.runs : 0.0;
  std::vector<uint64_t> share(2 * (size_t)pieces), chunk_hash;
  std::memcpy(share.data(), back.data() + (kGenHashAt - kGenStateAt), 8 * share.size());
  for (int64_t c = 0; c < n; c += kHashChunk) {
    uint64_t h = kFnvBasis * fnv_power((uint32_t)std::min(n - c, kHashChunk)), odd = 0;
    for (int64_t q = c / kHashPiece; q < std::min(pieces, (c + kHashChunk) / kHashPiece); ++q) {
      h += odd ? 0 - share[2 * q] : share[2 * q];
      odd ^= share[2 * q + 1];
    }
    chunk_hash.push_back(h);
  }
  g->mask_hash = hash_of_chunks(chunk_hash);
  return cudaSuccess;
}

// FNV-1a of the chunk hashes' bytes, in order.
uint64_t hash_of_chunks(const std::vector<uint64_t> &chunk_hash) {
  uint64_t h = kFnvBasis;
  for (uint64_t v : chunk_hash)
    for (int byte = 0; byte < 8; ++byte) h = (h ^ ((v >> (8 * byte)) & 0xffu)) * kFnvPrime;
  return h;
}

// ---------------------------------------------------------------------------
// Device: b(x), numbering, neighbour masks
// ---------------------------------------------------------------------------
struct GeoArgs {
  const uint8_t *mask;
  int32_t nx, ny, nz, per_z;
};

__device__ __forceinline__ int64_t geo_nbr(const GeoArgs &g, int x, int y, int z, int dx, int dy, int dz) {
  int xx = x + dx, yy = y + dy, zz = z + dz;
  xx = xx < 0 ? xx + g.nx : (xx >= g.nx ? xx - g.nx : xx);
  yy = yy < 0 ? yy + g.ny : (yy >= g.ny ? yy - g.ny : yy);
  if (zz < 0 || zz >= g.nz) {
    if (!g.per_z) return -1;
    zz = zz < 0 ? zz + g.nz : zz - g.nz;
  }
  return ((int64_t)zz * g.ny + yy) * g.nx + xx;
}

// b(c) for catalytic solid cells (fluid cells at c - c_j; 0 for inert solid),
// and the 18-bit masks: for fluid cells, bit i set when c + c_i is solid (the
// targets that bounce back or sputter); for solid cells, bit i set when
// c + c_i is fluid (the node's active outgoing links, from which the random
// sputtering matrix draws). Also counts fluid->catalytic links.
__global__ void classify_kernel(GeoArgs g, int32_t *b, uint32_t *nbm_dense, unsigned long long *n_links) {
  const int64_t n = (int64_t)g.nx * g.ny * g.nz;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int links = 0;
  if (c < n) {
    const int64_t plane = (int64_t)g.nx * g.ny;
    const int z = (int)(c / plane);
    const int y = (int)((c - z * plane) / g.nx);
    const int x = (int)(c - z * plane - (int64_t)y * g.nx);
    if (g.mask[c]) {
      int cnt = 0;
      uint32_t out = 0;
#pragma unroll
      for (int j = 1; j < kQ; ++j) {
        const int64_t s = geo_nbr(g, x, y, z, -cx(j), -cy(j), -cz(j));
        cnt += (s >= 0 && !g.mask[s]) ? 1 : 0;
        const int64_t t = geo_nbr(g, x, y, z, cx(j), cy(j), cz(j));
        if (t >= 0 && !g.mask[t]) out |= 1u << j;
      }
      b[c] = g.mask[c] == 1 ? cnt : 0;
      nbm_dense[c] = out;
    } else {
      uint32_t m = 0;
#pragma unroll
      for (int i = 1; i < kQ; ++i) {
        const int64_t t = geo_nbr(g, x, y, z, cx(i), cy(i), cz(i));
        if (t >= 0 && g.mask[t]) {
          m |= 1u << i;
          links += g.mask[t] == 1;
        }
      }
      b[c] = 0;
      nbm_dense[c] = m;
    }
  }
  // integer sum: order-independent
  for (int o = 16; o > 0; o >>= 1) links += __shfl_down_sync(0xffffffffu, links, o);
  if ((threadIdx.x & 31) == 0 && links) atomicAdd(n_links, (unsigned long long)links);
}

// per-plane counts of fluid cells and catalytic nodes: one block per plane
__global__ void plane_count_kernel(GeoArgs g, const int32_t *b, int64_t *fl_cnt, int64_t *node_cnt) {
  const int64_t plane = (int64_t)g.nx * g.ny;
  const int64_t base = (int64_t)blockIdx.x * plane;
  long long f = 0, s = 0;
  for (int64_t k = threadIdx.x; k < plane; k += blockDim.x) {
    const int64_t c = base + k;
    if (g.mask[c])
      s += b[c] > 0;
    else
      f += 1;
  }
  __shared__ long long shf[32], shs[32];
  for (int o = 16; o > 0; o >>= 1) {
    f += __shfl_down_sync(0xffffffffu, f, o);
    s += __shfl_down_sync(0xffffffffu, s, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    shf[wid] = f;
    shs[wid] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long tf = 0, ts = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      tf += shf[w];
      ts += shs[w];
    }
    fl_cnt[blockIdx.x] = tf;
    node_cnt[blockIdx.x] = ts;
  }
}

// Numbering, one block per plane, tiles of blockDim cells, ranks from a
// ballot/popc block scan:
//   - catalytic nodes in linear order;
//   - lattice entries of the fluid cells (fluid-only addressing): within each
//     plane first the cells with no solid neighbour, then the cells touching
//     a solid, each group in linear order. The second group then fills warps
//     of its own, and the warps of the first take the fast path, instead of
//     one wall cell sending its whole warp of 32 down the general one. (The
//     exported fluid index is the linear-order numbering, formed from the
//     mask on export.)
// pass 0 numbers the nodes and the first group, pass 1 the second group.
__global__ void number_kernel(GeoArgs g, const int32_t *b, const int64_t *fl_plane, const int64_t *node_plane,
                              int32_t *idx, int32_t *fcell, float *inv_b, int32_t *node_cell,
                              const uint32_t *nbm_dense, uint32_t *nbm_fluid) {
  const int64_t plane = (int64_t)g.nx * g.ny;
  const int64_t base = (int64_t)blockIdx.x * plane;
  int64_t fl_off = fl_plane[blockIdx.x], nd_off = node_plane[blockIdx.x];
  __shared__ int wf[32], ws[32];
  __shared__ int64_t tot_f, tot_s;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int pass = 0; pass < 2; ++pass) {
    for (int64_t t0 = 0; t0 < plane; t0 += blockDim.x) {
      const int64_t k = t0 + threadIdx.x;
      const bool in = k < plane;
      const int64_t c = base + k;
      const bool fl = in && !g.mask[c];
      const bool isf = fl && ((nbm_dense[c] != 0) == (pass == 1));
      const bool iss = pass == 0 && in && g.mask[c] && b[c] > 0;
      const unsigned bf = __ballot_sync(0xffffffffu, isf), bs = __ballot_sync(0xffffffffu, iss);
      const unsigned lt = (1u << lane) - 1u;
      if (lane == 0) {
        wf[wid] = __popc(bf);
        ws[wid] = __popc(bs);
      }
      __syncthreads();
      int pf = 0, ps = 0;
      for (int w = 0; w < wid; ++w) {
        pf += wf[w];
        ps += ws[w];
      }
      if (isf) {
        const int64_t r = fl_off + pf + __popc(bf & lt);
        idx[c] = (int32_t)r;
        fcell[r] = (int32_t)c;
        nbm_fluid[r] = nbm_dense[c];
      } else if (iss) {
        const int64_t r = nd_off + ps + __popc(bs & lt);
        idx[c] = (int32_t)r;
        inv_b[r] = 1.0f / (float)b[c];
        node_cell[r] = (int32_t)c;
      } else if (pass == 0 && in && g.mask[c]) {
        idx[c] = -1;
      }
      if (threadIdx.x == 0) {
        int sf = 0, ss = 0;
        for (int w = 0; w < nw; ++w) {
          sf += wf[w];
          ss += ws[w];
        }
        tot_f = sf;
        tot_s = ss;
      }
      __syncthreads();
      fl_off += tot_f;
      nd_off += tot_s;
      __syncthreads();
    }
  }
}

cudaError_t build_structures(lbm_geometry *g, cudaStream_t st) {
  GeoArgs ga{g->mask, g->nx, g->ny, g->nz, g->bc == LBM_BC_PERIODIC};
  const int64_t n = g->n;
  unsigned long long *d_links = (unsigned long long *)g->mem.alloc(sizeof(unsigned long long));
  int64_t *d_cnt = (int64_t *)g->mem.alloc(sizeof(int64_t) * 2 * g->nz);
  // the two counters go back to the allocator on every exit (stream-ordered)
  struct Scratch {
    lbm_geometry *g;
    unsigned long long *links;
    int64_t *cnt;
    ~Scratch() {
      g->mem.free(links, sizeof(unsigned long long));
      g->mem.free(cnt, sizeof(int64_t) * 2 * g->nz);
    }
  } scratch{g, d_links, d_cnt};
  if (!d_links || !d_cnt) return cudaErrorMemoryAllocation;
  cudaError_t e = cudaMemsetAsync(d_links, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  classify_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ga, g->b, g->nbm_dense, d_links);
  plane_count_kernel<<<g->nz, 512, 0, st>>>(ga, g->b, d_cnt, d_cnt + g->nz);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  std::vector<int64_t> cnt(2 * g->nz);
  unsigned long long links = 0;
  if ((e = cudaMemcpyAsync(cnt.data(), d_cnt, sizeof(int64_t) * 2 * g->nz, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(&links, d_links, sizeof(links), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  g->fl_plane_h = new int64_t[g->nz + 1];
  g->node_plane_h = new int64_t[g->nz + 1];
  g->fl_plane_h[0] = g->node_plane_h[0] = 0;
  for (int z = 0; z < g->nz; ++z) {
    g->fl_plane_h[z + 1] = g->fl_plane_h[z] + cnt[z];
    g->node_plane_h[z + 1] = g->node_plane_h[z] + cnt[g->nz + z];
  }
  g->n_fluid = g->fl_plane_h[g->nz];
  g->n_nodes = g->node_plane_h[g->nz];
  g->n_links = (int64_t)links;
  g->nbm_fluid = (uint32_t *)g->mem.alloc(sizeof(uint32_t) * std::max<int64_t>(g->n_fluid, 1));
  g->fcell = (int32_t *)g->mem.alloc(sizeof(int32_t) * std::max<int64_t>(g->n_fluid, 1));
  g->inv_b = (float *)g->mem.alloc(sizeof(float) * std::max<int64_t>(g->n_nodes, 1));
  g->node_cell = (int32_t *)g->mem.alloc(sizeof(int32_t) * std::max<int64_t>(g->n_nodes, 1));
  g->fl_plane_d = (int64_t *)g->mem.alloc(sizeof(int64_t) * (g->nz + 1));
  g->node_plane_d = (int64_t *)g->mem.alloc(sizeof(int64_t) * (g->nz + 1));
  g->cell_plane_d = (int64_t *)g->mem.alloc(sizeof(int64_t) * (g->nz + 1));
  if (!g->nbm_fluid || !g->fcell || !g->inv_b || !g->node_cell || !g->fl_plane_d || !g->node_plane_d || !g->cell_plane_d)
    return cudaErrorMemoryAllocation;
  std::vector<int64_t> cp(g->nz + 1);
  for (int z = 0; z <= g->nz; ++z) cp[z] = (int64_t)z * g->plane;
  if ((e = cudaMemcpyAsync(g->fl_plane_d, g->fl_plane_h, sizeof(int64_t) * (g->nz + 1), cudaMemcpyHostToDevice,
                           st)) != cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(g->node_plane_d, g->node_plane_h, sizeof(int64_t) * (g->nz + 1), cudaMemcpyHostToDevice,
                           st)) != cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(g->cell_plane_d, cp.data(), sizeof(int64_t) * (g->nz + 1), cudaMemcpyHostToDevice, st)) !=
      cudaSuccess)
    return e;
  number_kernel<<<g->nz, 1024, 0, st>>>(ga, g->b, g->fl_plane_d, g->node_plane_d, g->idx, g->fcell, g->inv_b,
                                        g->node_cell, g->nbm_dense, g->nbm_fluid);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return cudaStreamSynchronize(st);
}

}  // namespace lbm
