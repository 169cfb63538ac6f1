// Exactly rounded float GROUP BY sums (AGG_FLAG_EXACT_SUM), and the error of
// the strategy's sums against them (AGG_FLAG_SUM_ERROR).
//
// Float sums built with atomics depend on the order in which rows arrive.
// With this flag every group's SUM is the exact real sum of its rows rounded
// once to float64 (to nearest, ties to even) and AVG is that sum divided by
// the count, so the result is the same bit for bit for every strategy, grid
// and run (the deterministic float GROUP BY mode). It runs after a strategy
// has produced the groups (keys ascending, counts, MIN/MAX):
//   exact_span   the lowest and highest exponent among the nonzero values,
//                and whether any value is not finite (one read-back);
//   exact_add    every row adds its value, an integer number of units of the
//                column's lowest exponent, to its group's digits (integer
//                additions: the order is free). Groups whose digits fit one
//                block's shared memory are added there, found through a hash
//                table of the result keys; more groups are found by binary
//                search over the result keys and added with 64-bit atomics;
//   exact_round  per group, carry propagation and one rounding.
// The digits per group cover only the column's exponent span (plus 32 bits
// for the row count), so a column of similar magnitudes needs a handful.
#include <algorithm>
#include <climits>
#include <mutex>

#include "exact.cuh"
#include "groupby.cuh"

namespace agg {

constexpr int kExactThreads = 256;

template <int DT>
__device__ __forceinline__ ExactParts parts_of(const void* vals, int64_t i) {
  if (DT == AGG_F32) return exact_parts_f32(__float_as_uint(((const float*)vals)[i]));
  return exact_parts_f64((uint64_t)__double_as_longlong(((const double*)vals)[i]));
}

// span[0] = lowest lsb exponent, span[1] = highest, span[2] = nonfinite rows.
// Eight loads in flight a thread: the pass is bound by memory (2^25 float32
// rows: 40 -> 35 us).
template <int DT>
__global__ void __launch_bounds__(kExactThreads) exact_span(const void* __restrict__ vals, int64_t n,
                                                            int* __restrict__ span) {
  constexpr int kLoads = 8;
  constexpr int kInf = DT == AGG_F32 ? 0xFF : 0x7FF;
  constexpr int kLsb0 = DT == AGG_F32 ? 150 : 1075;  // lsb exponent = exponent field (1 for subnormals) - kLsb0
  int lo = INT_MAX, hi = INT_MIN;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += kLoads * stride) {
    int e[kLoads];
    bool zero[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int64_t j = i + u * stride;
      if (DT == AGG_F32) {
        const uint32_t b = j < n ? ((const uint32_t*)vals)[j] : 0u;
        e[u] = (int)((b >> 23) & 0xFFu);
        zero[u] = (b << 1) == 0u;
      } else {
        const uint64_t b = j < n ? ((const uint64_t*)vals)[j] : 0ull;
        e[u] = (int)((b >> 52) & 0x7FFu);
        zero[u] = (b << 1) == 0ull;
      }
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      if (zero[u]) continue;
      lo = min(lo, max(e[u], 1));
      hi = max(hi, max(e[u], 1));
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0 && lo != INT_MAX) {
    if (lo != kInf) atomicMin(&span[0], lo - kLsb0);
    atomicMax(&span[1], hi - kLsb0);
    if (hi == kInf) atomicOr(&span[2], 1);
  }
}

template <int DT>
__global__ void __launch_bounds__(kExactThreads) exact_add(const uint32_t* __restrict__ keys,
                                                           const void* __restrict__ vals, int64_t n,
                                                           const uint32_t* __restrict__ gkeys, int64_t d,
                                                           const uint32_t* __restrict__ index,
                                                           unsigned long long* __restrict__ acc, int D, int base) {
  const uint32_t k0 = gkeys[0], range = gkeys[d - 1] - k0;
  const int shift = max(0, 16 - (int)__clz((int)range));
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const ExactParts p = parts_of<DT>(vals, i);
    if (p.mant == 0) continue;
    const uint32_t key = keys[i];
    const uint32_t part = (key - k0) >> shift;
    int64_t lo = index[part], len = index[part + 1] - lo;  // the group: the last result key <= key (it is present)
    while (len > 1) {
      const int64_t half = len >> 1;
      if (__ldg(&gkeys[lo + half]) <= key) lo += half;
      len -= half;
    }
    const int pos = p.lsb - base;  // >= 0
    const int q = pos / kDigitBits;
    int64_t c[3];
    exact_chunks(p.mant, pos - q * kDigitBits, c);
    unsigned long long* w = acc + (size_t)lo * (size_t)D + (size_t)q;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (c[k] != 0) atomicAdd(&w[k], (unsigned long long)(p.neg ? -c[k] : c[k]));
  }
}

// Groups added in shared memory. A block holds a hash table of the d result
// keys (buckets of 4 slots, at most half full, with each key's group number)
// and for every group W words of 32 bits, digits of 16 bits: a value adds at
// most 65535 to each of 3 (float32) or 5 (float64) neighbouring digits, with
// native shared atomics that return nothing. After kExactIters iterations the block
// carries the digits into their 16 bits; the last two digits hold the growth
// of 2^32 rows. Few groups get several copies of their words, one per lane
// class, so that a warp's rows of one group do not serialise. Against 64-bit
// atomics in HBM after a binary search: 2^25 float32 rows over 4096 keys 2100
// -> 153 us; bound by the shared-memory wavefronts of the lookup and the
// three updates (30 a warp and 32 rows).
constexpr int kExactSmemThreads = 1024;
constexpr int kExactRows = 4;                                                  // rows a thread adds per iteration
constexpr int kExactIters = 32767 / (kExactSmemThreads * kExactRows);          // iterations between two carries
constexpr int kExactDigits(bool f64) { return f64 ? 5 : 3; }

__device__ __forceinline__ uint32_t exact_home(uint32_t key, int shift) {
  return ((key ^ (key >> 15)) * 0x9E3779B1u) >> shift;
}

// Carry every word group's digits: words k * stride + i, k < W.
__device__ __forceinline__ void exact_settle(uint32_t* dig, int words, int stride, int W) {
  for (int i = threadIdx.x; i < words; i += blockDim.x) {
    int c = 0;
    for (int k = 0; k < W - 1; ++k) {
      const int v = (int)dig[k * stride + i] + c;
      dig[k * stride + i] = (uint32_t)v & 0xFFFFu;
      c = v >> 16;
    }
    dig[(W - 1) * stride + i] += (uint32_t)c;
  }
}

// acc: d x W signed 64-bit words (digits of 16 bits), zero at the start.
// copies (a power of two): words of one digit are (group * copies + copy).
template <int DT>
__global__ void __launch_bounds__(kExactSmemThreads, 1)
    exact_add_shared(const uint32_t* __restrict__ keys, const void* __restrict__ vals, int64_t n,
                     const uint32_t* __restrict__ gkeys, int d, int slots, int copies, int W, int base,
                     unsigned long long* __restrict__ acc) {
  extern __shared__ __align__(16) uint32_t sm[];
  constexpr int kDig = kExactDigits(DT == AGG_F64);
  uint32_t* tkey = sm;                          // key + 1, 0 = empty
  const int words = d * copies;
  const int stride = words;
  uint32_t* dig = sm + slots;                   // W x stride
  uint16_t* tidx = (uint16_t*)(dig + W * stride);
  const int shift = __clz(slots) + 1;           // 32 - log2(slots)
  for (int i = threadIdx.x; i < slots + W * stride; i += blockDim.x) sm[i] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    const uint32_t key = gkeys[i];
    if (key == 0xFFFFFFFFu) continue;           // the last group: found without the table
    uint32_t h = exact_home(key, shift) & ~3u;
    for (int p = 0; p < slots; ++p) {           // at most half the slots are taken
      const uint32_t at = (h + (uint32_t)p) & (uint32_t)(slots - 1);
      if (atomicCAS(&tkey[at], 0u, key + 1) == 0u) {
        tidx[at] = (uint16_t)i;
        break;
      }
    }
  }
  __syncthreads();
  const int copy = (int)threadIdx.x & (copies - 1);
  const int64_t span = (int64_t)gridDim.x * kExactSmemThreads * kExactRows;
  int it = 0;
  for (int64_t r0 = (int64_t)blockIdx.x * kExactSmemThreads * kExactRows; r0 < n; r0 += span) {
    uint32_t key[kExactRows];
    uint64_t bits[kExactRows];
#pragma unroll
    for (int u = 0; u < kExactRows; ++u) {
      const int64_t j = r0 + u * kExactSmemThreads + threadIdx.x;
      key[u] = j < n ? keys[j] : 0u;
      if (DT == AGG_F32) bits[u] = j < n ? ((const uint32_t*)vals)[j] : 0u;
      else bits[u] = j < n ? ((const uint64_t*)vals)[j] : 0ull;  // rows past the end are zeros: nothing to add
    }
    uint4 q[kExactRows];
#pragma unroll
    for (int u = 0; u < kExactRows; ++u) q[u] = *(const uint4*)&tkey[exact_home(key[u], shift) & ~3u];
#pragma unroll
    for (int u = 0; u < kExactRows; ++u) {
      const ExactParts p = DT == AGG_F32 ? exact_parts_f32((uint32_t)bits[u]) : exact_parts_f64(bits[u]);
      if (p.mant == 0) continue;
      const uint32_t k1 = key[u] + 1;
      uint32_t b = exact_home(key[u], shift) & ~3u;
      int g = d - 1;
      if (k1 != 0u) {
        uint4 x = q[u];
        for (int t = 0; t < slots; t += 4) {  // the key is in the table: a few buckets at most
          const int s = x.x == k1 ? 0 : x.y == k1 ? 1 : x.z == k1 ? 2 : x.w == k1 ? 3 : -1;
          if (s >= 0) {
            b += (uint32_t)s;
            break;
          }
          b = (b + 4) & (uint32_t)(slots - 1);
          x = *(const uint4*)&tkey[b];
        }
        g = tidx[b];
      }
      const int pos = p.lsb - base;  // >= 0
      const int r = pos & 15;
      uint32_t* w = dig + (pos >> 4) * stride + g * copies + copy;
      const uint64_t lo = p.mant << r;
      const uint32_t hi = DT == AGG_F64 && r ? (uint32_t)(p.mant >> (64 - r)) : 0u;
#pragma unroll
      for (int k = 0; k < kDig; ++k) {
        const uint32_t v = k < 4 ? (uint32_t)(lo >> (16 * k)) & 0xFFFFu : hi;
        atomicAdd(&w[k * stride], p.neg ? 0u - v : v);
      }
    }
    if (++it == kExactIters) {
      it = 0;
      __syncthreads();
      exact_settle(dig, words, stride, W);
      __syncthreads();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < d * W; i += blockDim.x) {
    const int g = i / W, k = i - g * W;
    int64_t v = 0;
    for (int c = 0; c < copies; ++c) v += (int)dig[k * stride + g * copies + c];
    if (v != 0) atomicAdd(&acc[(size_t)g * W + k], (unsigned long long)v);
  }
}

// First group of each of 65536 equal parts of the result keys' range (and one
// past the last), so that exact_add's search starts from a short interval.
__global__ void __launch_bounds__(kExactThreads) exact_index(const uint32_t* __restrict__ gkeys, int64_t d,
                                                             uint32_t* __restrict__ index) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t > 65536u) return;
  const uint32_t k0 = gkeys[0], range = gkeys[d - 1] - k0;
  const int shift = max(0, 16 - (int)__clz((int)range));  // (key - k0) >> shift < 65536
  const uint64_t want = ((uint64_t)t << shift) + k0;      // the first key of part t
  int64_t lo = 0, hi = d;                                 // first group with key >= want
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (gkeys[mid] < want) lo = mid + 1;
    else hi = mid;
  }
  index[t] = (uint32_t)lo;
}

// replace: write the exact sum (and avg) over the result's; err (nullable):
// the distance of the sum the result keeps from the exact one.
__global__ void __launch_bounds__(kExactThreads) exact_round_groups(const unsigned long long* __restrict__ acc,
                                                                    int64_t d, int D, int base, int digit_bits,
                                                                    const int64_t* __restrict__ count,
                                                                    double* __restrict__ sum,
                                                                    double* __restrict__ avg, bool replace,
                                                                    double* __restrict__ err) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= d) return;
  int64_t a[kMaxDigits];
  int used = D;
  if (digit_bits == kDigitBits) {
    for (int k = 0; k < D; ++k) a[k] = (int64_t)acc[(size_t)g * D + k];
  } else {  // digits of 16 bits in signed 64-bit words, regrouped
    used = (16 * D + 48) / kDigitBits + 2;  // a word is below 2^48 in magnitude
    for (int k = 0; k < used; ++k) a[k] = 0;
    for (int k = 0; k < D; ++k) {
      const int64_t v = (int64_t)acc[(size_t)g * D + k];
      const int q = 16 * k / kDigitBits, r = 16 * k - q * kDigitBits;
      const int64_t h = v >> kDigitBits;  // floor, so the rest is in [0, 2^28)
      a[q] += (v - h * (int64_t(1) << kDigitBits)) * (int64_t(1) << r);
      a[q + 1] += h * (int64_t(1) << r);
    }
  }
  const double s = exact_round(a, used, base);
  if (err) err[g] = replace ? 0.0 : fabs(sum[g] - s);
  if (!replace) return;
  sum[g] = s;
  if (avg) avg[g] = count[g] ? s / (double)count[g] : __longlong_as_double(0x7ff8000000000000ll);
}

// Exactly rounded sums of a finished float GROUP BY result: with replace, they
// replace the result's sums (and averages); with report, g->sum_err receives
// |kept sum - exact sum| per group. keys/vals: the query's device columns.
agg_status exact_fp_sums(const uint32_t* keys, const void* vals, int64_t n, int vdt, uint32_t ops,
                         agg_groups* g, cudaStream_t s, bool replace, bool report) {
  const int64_t d = g->num_groups;
  if (d == 0 || n == 0) return AGG_OK;
  double* err = nullptr;
  if (report) {
    if (dev_malloc_async((void**)&err, (size_t)d * 8, s) != cudaSuccess) {
      set_error("sum errors: cannot allocate %lld bytes", (long long)d * 8);
      return AGG_ERR_OOM;
    }
    ((GroupsPriv*)g->priv)->extra = err;  // freed with the result from here on
    g->sum_err = err;
  }
  const DeviceInfo& di = device_info();
  const int grid = di.sm_count * 8;
  PhaseTimer pt(AGG_PHASE_FINALIZE, s);
  agg_status st = AGG_OK;
  char* scr = (char*)stream_scratch(s, 4096 + 256, &st);
  if (!scr) return st;
  int* span_dev = (int*)(scr + 4096);  // transient, past the scan's ticket and the sketch's features
  const int init[3] = {INT_MAX, INT_MIN, 0};
  AGG_CUDA_TRY(cudaMemcpyAsync(span_dev, init, sizeof(init), cudaMemcpyHostToDevice, s));
  if (vdt == AGG_F32) exact_span<AGG_F32><<<grid, kExactThreads, 0, s>>>(vals, n, span_dev);
  else exact_span<AGG_F64><<<grid, kExactThreads, 0, s>>>(vals, n, span_dev);
  note_launch();
  AGG_CUDA_TRY(cudaGetLastError());
  int span[3];
  AGG_CUDA_TRY(cudaMemcpyAsync(span, span_dev, sizeof(span), cudaMemcpyDeviceToHost, s));
  AGG_CUDA_TRY(cudaStreamSynchronize(s));
  AGG_CHECK_ARG(span[2] == 0, "exact float sums need finite values (the column holds an infinity or NaN)");
  const int mant_bits = vdt == AGG_F32 ? 24 : 53;
  int base = 0, D = 1;
  if (span[0] != INT_MAX) {
    base = span[0];
    const int bits = span[1] - span[0] + mant_bits + 33;  // sum of < 2^32 rows, and a sign
    D = (bits + kDigitBits - 1) / kDigitBits + 2;
  }
  if (D > kMaxDigits) {
    set_error("exact float sums: %d digits exceed %d", D, kMaxDigits);
    return AGG_ERR_INVALID;
  }
  // In shared memory when a block holds every group's words and the table of
  // keys (up to about 4096 groups of an ordinary column).
  const bool f64 = vdt == AGG_F64;
  const int W = (span[0] != INT_MAX ? (span[1] - span[0] + mant_bits + 15) / 16 : 0) + 3;  // value digits, growth
  const int64_t slots = std::max<int64_t>(64, next_pow2(2 * d));
  int copies = 32;
  auto smem_bytes = [&](int c) { return (size_t)slots * 6 + (size_t)d * c * W * 4 + 64; };
  while (copies > 1 && smem_bytes(copies) > ((size_t)96 << 10)) copies >>= 1;
  // A group of few rows is cheaper added in HBM than merged from every block
  // (300 K rows over 3000 keys: the whole call 283 us in HBM, 336 us shared).
  const bool shared = n >= 256 * d && d <= 65535 && W <= 16 &&
                      smem_bytes(copies) <= (size_t)di.smem_per_block_optin - 1024;
  if (shared) D = W;
  void* acc = nullptr;
  const size_t index_b = shared ? 0 : (65537 * 4 + 255) & ~size_t(255);
  const size_t bytes = (size_t)d * (size_t)D * 8 + index_b;
  if (dev_malloc_async(&acc, bytes, s) != cudaSuccess) {
    set_error("exact float sums: cannot allocate %zu bytes of digits", bytes);
    return AGG_ERR_OOM;
  }
  unsigned long long* words = (unsigned long long*)((char*)acc + index_b);
  uint32_t* index = (uint32_t*)acc;
  cudaError_t e = cudaMemsetAsync(acc, 0, bytes, s);
  if (e == cudaSuccess && span[0] != INT_MAX) {
    if (shared) {
      const size_t sm = smem_bytes(copies);
      const void* fn = f64 ? (const void*)exact_add_shared<AGG_F64> : (const void*)exact_add_shared<AGG_F32>;
      static std::mutex mu;  // the shared-memory limit is set per device, to the most a block may have
      static bool ready[64] = {};
      {
        std::lock_guard<std::mutex> lk(mu);
        const int dev = di.device;
        if (dev >= 64 || !ready[dev]) {
          const int most = di.smem_per_block_optin - 1024;
          e = cudaFuncSetAttribute(exact_add_shared<AGG_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
          if (e == cudaSuccess)
            e = cudaFuncSetAttribute(exact_add_shared<AGG_F64>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
          if (e == cudaSuccess && dev < 64) ready[dev] = true;
        }
      }
      const int64_t per = (int64_t)kExactSmemThreads * kExactRows;
      const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(di.sm_count, (n + per - 1) / per));
      int dd = (int)d, sl = (int)slots;
      const uint32_t* gk = g->keys;
      void* args[] = {(void*)&keys, (void*)&vals, (void*)&n, (void*)&gk, &dd, &sl, &copies, &D, &base, &words};
      if (e == cudaSuccess) e = cudaLaunchKernel(fn, dim3((unsigned)blocks), dim3(kExactSmemThreads), args, sm, s);
      note_launch();
    } else {
      exact_index<<<65537 / kExactThreads + 1, kExactThreads, 0, s>>>(g->keys, d, index);
      if (f64)
        exact_add<AGG_F64><<<grid, kExactThreads, 0, s>>>(keys, vals, n, g->keys, d, index, words, D, base);
      else
        exact_add<AGG_F32><<<grid, kExactThreads, 0, s>>>(keys, vals, n, g->keys, d, index, words, D, base);
      note_launch(2);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) {
    const int rgrid = (int)((d + kExactThreads - 1) / kExactThreads);
    exact_round_groups<<<rgrid, kExactThreads, 0, s>>>(words, d, D, base, shared ? 16 : kDigitBits, g->count,
                                                       (double*)g->sum, (ops & AGG_AVG) ? g->avg : nullptr,
                                                       replace, err);
    note_launch();
    e = cudaGetLastError();
  }
  cudaFreeAsync(acc, s);
  if (e != cudaSuccess) {
    set_error("exact float sums: %s", cudaGetErrorString(e));
    return AGG_ERR_CUDA;
  }
  AGG_CUDA_TRY(cudaStreamSynchronize(s));
  return AGG_OK;
}

}  // namespace agg
