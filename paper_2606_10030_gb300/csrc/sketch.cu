// Key sketch: 16 features of a strided sample of m = min(n, 4096)
// keys, computed by one block. The strategy selectors (the rule and the MLP)
// read them; the global table is sized from the GEE distinct-count estimate
// (Charikar, Chaudhuri, Motwani and Narasayya, PODS 2000).
#include <cmath>
#include <cstdint>

#include "groupby.cuh"

namespace agg {

constexpr int kSketchThreads = 1024;
constexpr int kSketchSlots = 2 * kSketchSample;  // hash slots for the sample (load <= 1/2)
constexpr size_t kSketchSmem = (size_t)kSketchSlots * 8 + (kSketchSample + 1) * 4 + 64 * 4;

// One block. The sample's keys are counted in a shared-memory hash table
// (key + 1, 0 = empty; the key 0xFFFFFFFF has a counter of its own), their
// counts histogrammed, and the 32 largest counts read off the histogram from
// the top by one warp. The block is one chain of latencies in front of every
// GROUP BY call (37-51 thousand clocks when the sums and quotients ran in
// float64, 13 thousand of them in the slope alone): sums are 64-bit integers in
// fixed point, the entropy is summed over the histogram's counts, quotients
// of integers below 2^24 are float32 (correctly rounded, as their float64
// quotient rounded to float32 is: it is never close enough to a tie), and two
// float64 divisions remain. 18-22 -> 9-14 us.
// The sample: row p_j = (offset + j * (n / m)) mod n for j < m, and the row
// after it (for the adjacent-repeat feature).
__device__ __forceinline__ int64_t sample_row(int64_t n, int m, uint64_t offset, int j) {
  const int64_t stride = m > 0 ? n / m : 1;
  const uint64_t off = n > 0 ? offset % (uint64_t)n : 0;
  const uint64_t q = off + (uint64_t)j * (uint64_t)stride;  // < 2n
  return (int64_t)(q >= (uint64_t)n ? q - (uint64_t)n : q);
}

// Gathers the sampled keys (pre[j]) and whether their successor repeats them
// (pre[kSketchSample + j]) with many blocks: one block issuing 8192 scattered loads is bound by its
// own load queue.
__global__ void sketch_gather(const uint32_t* __restrict__ keys, int64_t n, uint64_t offset,
                              int64_t stride, int m, uint32_t* __restrict__ pre) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const uint64_t q = offset + (uint64_t)j * (uint64_t)stride;  // sample_row, its divisions done on the host
  const int64_t p = (int64_t)(q >= (uint64_t)n ? q - (uint64_t)n : q);
  const uint32_t k = keys[p];
  pre[j] = k;
  pre[kSketchSample + j] = p + 1 < n && keys[p + 1] == k ? 1u : 0u;
}

// pre: the gathered sample (sketch_gather), or null to load it here.
__device__ void sketch_block(const uint32_t* __restrict__ keys, int64_t n, int vbytes, int nops, int fp,
                             int slot_bytes, uint64_t offset, double smem_bytes, double l2_bytes,
                             float* __restrict__ feat, const uint32_t* __restrict__ pre) {
  extern __shared__ __align__(16) unsigned char sm[];
  uint32_t* slot = (uint32_t*)sm;                                // kSketchSlots
  uint32_t* cnt = slot + kSketchSlots;                           // kSketchSlots
  uint32_t* hist = cnt + kSketchSlots;                           // kSketchSample + 1
  uint32_t* top = hist + kSketchSample + 1;                      // 32 (+ pad)
  __shared__ long long s_ent[kSketchThreads / 32];
  __shared__ unsigned int s_d, s_f1, s_f2, s_adj, s_kmin, s_kmax, s_maxc, s_ones;
  const int tid = threadIdx.x;
  for (int i = tid; i < 2 * kSketchSlots / 4; i += kSketchThreads) ((uint4*)slot)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i <= kSketchSample; i += kSketchThreads) hist[i] = 0;
  if (tid == 0) {
    s_d = s_f1 = s_f2 = s_adj = s_maxc = s_ones = 0;
    s_kmin = 0xFFFFFFFFu;
    s_kmax = 0;
  }
  const int m = (int)(n < kSketchSample ? n : kSketchSample);
  __syncthreads();
  constexpr int kPer = kSketchSample / kSketchThreads;  // sampled keys per thread
  uint32_t kk[kPer], adj[kPer];
  bool have[kPer];
#pragma unroll
  for (int u = 0; u < kPer; ++u) {  // issue every load before using any
    const int j = tid + u * kSketchThreads;
    have[u] = j < m;
    kk[u] = 0;
    adj[u] = 0;
    if (have[u]) {
      if (pre) {
        kk[u] = pre[j];
        adj[u] = pre[kSketchSample + j];
      } else {
        const int64_t p = sample_row(n, m, offset, j);
        kk[u] = keys[p];
        if (p + 1 < n) adj[u] = keys[p + 1] == kk[u] ? 1u : 0u;
      }
    }
  }
  {  // key range and adjacent repeats: reduced per warp, one atomic each per warp
    uint32_t lmin = 0xFFFFFFFFu, lmax = 0, ladj = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (!have[u]) continue;
      lmin = min(lmin, kk[u]);
      lmax = max(lmax, kk[u]);
      ladj += adj[u];
    }
    lmin = __reduce_min_sync(0xffffffffu, lmin);
    lmax = __reduce_max_sync(0xffffffffu, lmax);
    ladj = __reduce_add_sync(0xffffffffu, ladj);
    if ((tid & 31) == 0) {
      atomicMin(&s_kmin, lmin);
      atomicMax(&s_kmax, lmax);
      if (ladj) atomicAdd(&s_adj, ladj);
    }
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    if (!have[u]) continue;
    const uint32_t k1 = kk[u] + 1;
    if (k1 == 0u) {
      atomicAdd(&s_ones, 1u);
      continue;
    }
    uint32_t h = fmix32(kk[u]) & (kSketchSlots - 1);
    for (;;) {  // at most m < kSketchSlots occupied slots: an empty or matching one exists
      uint32_t cur = *(volatile uint32_t*)&slot[h];
      if (cur == 0) cur = atomicCAS(&slot[h], 0u, k1);
      if (cur == 0 || cur == k1) break;
      h = (h + 1) & (kSketchSlots - 1);
    }
    atomicAdd(&cnt[h], 1u);
  }
  __syncthreads();
  {
    uint32_t ld = 0, lf1 = 0, lf2 = 0, lmaxc = 0;
    for (int i = tid; i < kSketchSlots; i += kSketchThreads) {
      const uint32_t c = cnt[i];
      ld += c ? 1u : 0u;
      lf1 += c == 1 ? 1u : 0u;
      lf2 += c == 2 ? 1u : 0u;
      lmaxc = max(lmaxc, c);
      if (c > 2) atomicAdd(&hist[c], 1u);  // the many keys seen once or twice are counted per warp
    }
    if (tid == 0 && s_ones) {  // the key 0xFFFFFFFF
      const uint32_t c = s_ones;
      ld += 1u;
      lf1 += c == 1 ? 1u : 0u;
      lf2 += c == 2 ? 1u : 0u;
      lmaxc = max(lmaxc, c);
      if (c > 2) atomicAdd(&hist[c], 1u);
    }
    ld = __reduce_add_sync(0xffffffffu, ld);
    lf1 = __reduce_add_sync(0xffffffffu, lf1);
    lf2 = __reduce_add_sync(0xffffffffu, lf2);
    lmaxc = __reduce_max_sync(0xffffffffu, lmaxc);
    if ((tid & 31) == 0) {
      if (ld) atomicAdd(&s_d, ld);
      if (lf1) atomicAdd(&s_f1, lf1);
      if (lf2) atomicAdd(&s_f2, lf2);
      if (lmaxc) atomicMax(&s_maxc, lmaxc);
    }
  }
  __syncthreads();
  // entropy: -sum over counts c of hist[c] (c / m) ln(c / m), in units of 2^-40
  const float mf = (float)(m > 0 ? m : 1);
  {
    long long e = 0;
    for (int c = tid; c <= (int)s_maxc; c += kSketchThreads) {
      const uint32_t k = c == 1 ? s_f1 : c == 2 ? s_f2 : c > 2 ? hist[c] : 0u;
      if (k == 0) continue;
      const float p = (float)c / mf;
      e -= (long long)k * __float2ll_rn(p * logf(p) * 0x1p40f);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0) s_ent[tid >> 5] = e;
    if (tid == 0 && m > 0) {
      hist[1] = s_f1;
      hist[2] = s_f2;
    }
  }
  __syncthreads();
  if (tid >= 32) return;  // one warp from here on
  const int R = (int)(s_d < 32 ? s_d : 32);
  {  // the R largest counts, in descending order
    const int lane = tid;
    int got = 0;
    for (int base = (int)s_maxc; base >= 1 && got < R; base -= 32) {
      const int c = base - lane;
      const uint32_t v = c >= 1 ? hist[c] : 0u;
      uint32_t b = __ballot_sync(0xffffffffu, v != 0);
      while (b && got < R) {
        const int src = __ffs(b) - 1;
        b &= b - 1;
        const int mult = (int)__shfl_sync(0xffffffffu, v, src);
        const int take = mult < R - got ? mult : R - got;
        if (lane < take) top[got + lane] = (uint32_t)(base - src);
        got += take;
      }
    }
  }
  __syncwarp();
  // Least-squares slope of log(count) on log(rank) over the R largest counts:
  // lane r - 1 takes rank r. The logarithms (float32, at most 8.4, 0 or at
  // least 0.69) are exact multiples of 2^-24, so the sums of their products are
  // exact 64-bit integers.
  long long sx, sy, sxx, sxy;
  long long ent = tid < kSketchThreads / 32 ? s_ent[tid] : 0;
  {
    const int r = tid + 1;
    const bool in = r <= R;
    const int x = in ? __float2int_rn(logf((float)r) * 0x1p24f) : 0;
    const int y = in ? __float2int_rn(logf((float)top[r - 1]) * 0x1p24f) : 0;
    sx = x;
    sy = y;
    sxx = (long long)x * x;
    sxy = (long long)x * y;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
      sxx += __shfl_xor_sync(0xffffffffu, sxx, o);
      sxy += __shfl_xor_sync(0xffffffffu, sxy, o);
      ent += __shfl_xor_sync(0xffffffffu, ent, o);
    }
  }
  if (tid != 0) return;
  const float d = (float)s_d, f1 = (float)s_f1, f2 = (float)s_f2;
  float* f = feat;
  f[F_LOG2N] = n > 0 ? log2f((float)n) : 0.f;
  f[F_VBYTES] = (float)vbytes;
  f[F_NOPS] = (float)nops;
  f[F_FP] = (float)fp;
  if (m == 0) {
    for (int i = F_DISTINCT; i < F_COUNT; ++i) f[i] = 0.f;
    return;
  }
  f[F_DISTINCT] = d / mf;
  f[F_F1] = f1 / mf;
  f[F_F2] = f2 / mf;
  f[F_TOP1] = (float)top[0] / mf;
  uint32_t top8 = 0;
  for (int r = 0; r < 8 && r < R; ++r) top8 += top[r];
  f[F_TOP8] = (float)top8 / mf;
  // R sxy - sx sy and R sxx - sx sx in 128 bits, rounded once each
  f[F_SLOPE] = R >= 2 ? (float)((double)((__int128)R * sxy - (__int128)sx * sy) /
                                (double)((__int128)R * sxx - (__int128)sx * sx))
                      : 0.f;
  f[F_ENTROPY] = m > 1 ? (float)((double)ent * 0x1p-40 / (double)logf(mf)) : 0.f;
  f[F_ADJ_EQ] = (float)s_adj / mf;
  // float32 from here on: the features are float32, and float64 library
  // calls on one thread are slow on GB300's narrow float64 pipe
  float gee = sqrtf((float)n / mf) * f1 + (d - f1);
  if (gee < 1.f) gee = 1.f;
  if (gee > (float)n) gee = (float)n;
  f[F_LOG2_GEE] = log2f(gee);
  const float tbytes = 2.f * gee * (float)slot_bytes;
  f[F_SMEM_RATIO] = log2f(1.f + tbytes / (float)smem_bytes);
  f[F_L2_RATIO] = log2f(1.f + tbytes / (float)l2_bytes);
  f[F_LOG2_RANGE] = log2f((float)(s_kmax - s_kmin) + 1.f);
}

__global__ void __launch_bounds__(kSketchThreads) sketch_kernel(const uint32_t* __restrict__ keys, int64_t n,
                                                                int vbytes, int nops, int fp, int slot_bytes,
                                                                uint64_t offset, double smem_bytes, double l2_bytes,
                                                                float* __restrict__ feat,
                                                                const uint32_t* __restrict__ pre) {
  sketch_block(keys, n, vbytes, nops, fp, slot_bytes, offset, smem_bytes, l2_bytes, feat, pre);
}

// One block per query of a batch.
__global__ void __launch_bounds__(kSketchThreads) sketch_batch_kernel(const SketchJob* __restrict__ jobs,
                                                                      double smem_bytes, double l2_bytes,
                                                                      float* __restrict__ feat) {
  const SketchJob j = jobs[blockIdx.x];
  sketch_block(j.keys, j.n, j.vbytes, j.nops, j.fp, j.slot_bytes, j.offset, smem_bytes, l2_bytes,
               feat + (size_t)blockIdx.x * F_COUNT, nullptr);
}

agg_status sketch_batch_launch(const SketchJob* jobs_dev, int nq, float* feat_dev, cudaStream_t s) {
  const DeviceInfo& di = device_info();
  static bool attr_set[64] = {};
  if (di.device >= 0 && di.device < 64 && !attr_set[di.device]) {
    AGG_CUDA_TRY(
        cudaFuncSetAttribute(sketch_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSketchSmem));
    attr_set[di.device] = true;
  }
  if (nq <= 0) return AGG_OK;
  PhaseTimer pt(AGG_PHASE_SKETCH, s);
  sketch_batch_kernel<<<nq, kSketchThreads, kSketchSmem, s>>>(jobs_dev, (double)di.smem_per_block_optin,
                                                              (double)di.l2_bytes, feat_dev);
  note_launch();
  AGG_CUDA_TRY(cudaGetLastError());
  return AGG_OK;
}

agg_status sketch_launch(const uint32_t* keys, int64_t n, int vdt, uint32_t ops, uint64_t offset, float* feat_dev,
                         cudaStream_t s) {
  const DeviceInfo& di = device_info();
  static bool attr_set[64] = {};
  if (di.device >= 0 && di.device < 64 && !attr_set[di.device]) {
    AGG_CUDA_TRY(cudaFuncSetAttribute(sketch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSketchSmem));
    attr_set[di.device] = true;
  }
  // the gathered sample sits at 64 KiB of the stream scratch (transient; the
  // scratch block is at least 1 MiB, so this request never moves it)
  agg_status st = AGG_OK;
  char* scr = (char*)stream_scratch(s, (size_t)96 << 10, &st);
  if (!scr) return st;
  uint32_t* pre = (uint32_t*)(scr + ((size_t)64 << 10));
  PhaseTimer pt(AGG_PHASE_SKETCH, s);
  const int m = (int)(n < kSketchSample ? n : kSketchSample);
  if (m > 0) {
    const int64_t stride = n / m;
    sketch_gather<<<(m + 255) / 256, 256, 0, s>>>(keys, n, offset % (uint64_t)n, stride, m, pre);
    note_launch();
  }
  note_launch();
  sketch_kernel<<<1, kSketchThreads, kSketchSmem, s>>>(keys, n, (int)dtype_size(vdt), __builtin_popcount(ops),
                                             dtype_is_fp(vdt) ? 1 : 0, gslot_bytes(ops_minmax(ops)), offset,
                                             (double)di.smem_per_block_optin, (double)di.l2_bytes, feat_dev, pre);
  AGG_CUDA_TRY(cudaGetLastError());
  return AGG_OK;
}

}  // namespace agg

using namespace agg;

extern "C" agg_status agg_sketch(const uint32_t* keys_dev, int64_t n, agg_dtype vdtype, uint32_t ops,
                                 uint64_t sample_offset, float* features_dev, void* stream) {
  clear_error();
  AGG_CHECK_ARG(dtype_valid(vdtype), "invalid dtype %d", (int)vdtype);
  AGG_CHECK_ARG(ops != 0 && (ops & ~(uint32_t)AGG_ALL) == 0, "invalid ops mask 0x%x", ops);
  AGG_CHECK_ARG(n >= 0, "invalid row count");
  AGG_CHECK_ARG(n == 0 || keys_dev != nullptr, "null key pointer");
  AGG_CHECK_ARG(features_dev != nullptr, "null features pointer");
  return sketch_launch(keys_dev, n, vdtype, ops, sample_offset, features_dev, (cudaStream_t)stream);
}
