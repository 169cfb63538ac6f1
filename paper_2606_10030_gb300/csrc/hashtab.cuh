// Device side of the hash GROUP BY (build and finalisation), shared by the
// single-query driver (groupby.cu) and the batched persistent kernel
// (batch.cu): slot layouts, shared- and global-table probing and updates, the
// build kernel and the finalise kernels.
//
// Build. Every row is folded (the aggregate() of Fig. 4) into the slot of its
// key in an open-addressing hash table (MurmurHash3 fmix32, linear probing,
// bounded probe count):
//   SMEM    each block owns a table in shared memory and updates it with
//           shared-memory atomics; rows whose key finds no slot within the
//           probe bound go straight to the global table ("spill"); at the end
//           the block merges its table into the global one.
//   GLOBAL  every row updates the global table in HBM with L2 atomics.
// Keys are stored as key + 1 so that an all-zero table is empty; the key
// 0xFFFFFFFF has its own side slot after the main slots. All global
// accumulators start at zero: count and sum add, MIN is kept as the
// complement of an order-preserving image and MAX as the image, both updated
// with atomicMax; float sums in the global table are float64 (L2 atomic adds:
// a per-block or per-warp compensated float32 partial, or a single row, is
// merged into a float64 accumulator; the float64 additions run in the L2's
// atomic units, not on the SM's narrow float64 pipe).
#pragma once

#include <cstring>

#include "groupby.cuh"
#include "quotient.cuh"

namespace agg {

// ---------------------------------------------------------------------------
// Value traits: order-preserving 64-bit image of a value.
// ---------------------------------------------------------------------------
template <int DT> struct GV;
template <> struct GV<AGG_I32> {
  using T = int32_t;
  __device__ static uint64_t img(T v) { return img_i64((int64_t)v); }
};
template <> struct GV<AGG_I64> {
  using T = int64_t;
  __device__ static uint64_t img(T v) { return img_i64(v); }
};
template <> struct GV<AGG_U32> {
  using T = uint32_t;
  __device__ static uint64_t img(T v) { return img_i64((int64_t)v); }
};
template <> struct GV<AGG_F32> {
  using T = float;
  __device__ static uint64_t img(T v) { return (uint64_t)img_f32(v); }
};
template <> struct GV<AGG_F64> {
  using T = double;
  __device__ static uint64_t img(T v) { return img_f64(v); }
};

template <bool MM> struct GSlot;
template <> struct __align__(16) GSlot<false> {
  uint32_t key1;
  uint32_t cnt;
  unsigned long long sum;
};
template <> struct __align__(32) GSlot<true> {
  uint32_t key1;
  uint32_t cnt;
  unsigned long long sum;
  unsigned long long minc;
  unsigned long long mx;
};

constexpr int kGlobalProbe = 128;
constexpr int kStatusFull = 1;

struct BuildArgs {
  const uint32_t* keys;
  const void* vals;
  int64_t n;
  int64_t head;        // rows before the 16-byte aligned body (vector path)
  void* table;         // GSlot[mask + 2]
  uint32_t mask;       // main slots - 1 (main slots a power of two)
  int gshift;          // home slot = fmix32(key) >> gshift (top bits: 32 - log2(main slots))
  int smem_slots;      // S (power of two) for SMEM, else 0
  int* status;
  unsigned long long* progress;  // [0] rows gone through, [1] rows that found no slot, counted
                                 // when a full table stopped the build (or null)
  uint32_t* block_fails;         // this block's count of rows that found no slot (shared memory, or null)
};

// Global slot of key (insert if absent); -1 if no slot within the probe bound.
// The home slot is taken from the top bits of the hash, so keys whose hash
// shares its top bits (one partition of a hash-partitioned input) live in one
// contiguous region of the table.
template <bool MM>
__device__ __forceinline__ int64_t g_slot(GSlot<MM>* tab, uint32_t mask, int shift, uint32_t key,
                                          int max_probe = kGlobalProbe) {
  if (key == 0xFFFFFFFFu) return (int64_t)mask + 1;
  const uint32_t k1 = key + 1;
  uint32_t h = fmix32(key) >> shift;
#pragma unroll 1
  for (int p = 0; p < max_probe; ++p) {
    uint32_t cur = *(volatile uint32_t*)&tab[h].key1;
    if (cur == k1) return h;
    if (cur == 0) {
      uint32_t old = atomicCAS(&tab[h].key1, 0u, k1);
      if (old == 0u || old == k1) return h;
    }
    h = (h + 1) & mask;
  }
  return -1;
}

// Order-preserving image of a value in its own width.
template <int DT> struct SImg { using U = uint32_t; };
template <> struct SImg<AGG_I64> { using U = unsigned long long; };
template <> struct SImg<AGG_F64> { using U = unsigned long long; };

template <int DT>
__device__ __forceinline__ typename SImg<DT>::U s_img(typename GV<DT>::T v) {
  if (DT == AGG_I32) return (uint32_t)(int32_t)v ^ 0x80000000u;
  if (DT == AGG_U32) return (uint32_t)v;
  if (DT == AGG_F32) return img_f32((float)v);
  if (DT == AGG_I64) return (unsigned long long)img_i64((int64_t)v);
  return (unsigned long long)img_f64((double)v);
}
// shared image -> the 64-bit image kept in the global table (GV<DT>::img)
template <int DT>
__device__ __forceinline__ uint64_t g_img_of(typename SImg<DT>::U m) {
  if (DT == AGG_I32) return img_i64((int64_t)(int32_t)((uint32_t)m ^ 0x80000000u));
  if (DT == AGG_U32) return img_i64((int64_t)(uint32_t)m);
  return (uint64_t)m;
}

// Count rows that found no global slot in the block's shared counter.
__device__ __forceinline__ void note_fail(const BuildArgs& a, uint32_t rows) {
  *(volatile int*)a.status = kStatusFull;
  if (a.block_fails) atomicAdd(a.block_fails, rows);
}

// What a row, a warp or a block adds to a group: rows, sum (int64 bits, or
// float64 bits for floats), complement of the minimum's image, image of the
// maximum (MM only).
struct GPart {
  uint32_t key, cnt;
  unsigned long long sum, nmn, mx;
};

template <int DT, bool MM>
__device__ __forceinline__ GPart g_part_of(uint32_t key, typename GV<DT>::T v) {
  GPart p;
  p.key = key;
  p.cnt = 1;
  if (DT == AGG_F32 || DT == AGG_F64) p.sum = (unsigned long long)__double_as_longlong((double)v);
  else p.sum = (unsigned long long)(int64_t)v;
  if (MM) {
    p.mx = GV<DT>::img(v);
    p.nmn = ~p.mx;
  }
  return p;
}

// Add the N parts marked in parts to their global slots. The keys' home slots
// (and, with MIN/MAX, their extremes) are all read before any is used, so a
// thread waits once for N slots: the builds that send many rows here, and the
// merge of a tile's table, were bound by that latency. An extreme's atomic is
// issued only when the value read does not already cover it (extremes only
// move outwards, so a stale reading is harmless). Once a part of this block
// found the table full, the others probe only kShortProbe slots: the build is
// redone, and the rows folded before the block notices should not each walk
// the whole probe bound.
constexpr int kShortProbe = 8;

template <int DT, bool MM, int N>
__device__ __forceinline__ void g_merge(const BuildArgs& a, const GPart (&p)[N], uint32_t parts) {
  GSlot<MM>* tab = (GSlot<MM>*)a.table;
  uint32_t h[N], cur[N];
  ulonglong2 ext[N];
#pragma unroll
  for (int r = 0; r < N; ++r) {
    h[r] = fmix32(p[r].key) >> a.gshift;
    cur[r] = 0u;
    ext[r] = make_ulonglong2(0, 0);
    if ((parts >> r) & 1u) {
      cur[r] = *(volatile uint32_t*)&tab[h[r]].key1;
      if constexpr (MM) ext[r] = __ldcg((const ulonglong2*)&tab[h[r]].minc);
    }
  }
#pragma unroll
  for (int r = 0; r < N; ++r) {
    if (!((parts >> r) & 1u)) continue;
    int64_t g = h[r];
    if (cur[r] != p[r].key + 1 || p[r].key == 0xFFFFFFFFu) {
      const bool met_full = a.block_fails && *(volatile uint32_t*)a.block_fails != 0;
      g = g_slot<MM>(tab, a.mask, a.gshift, p[r].key, met_full ? kShortProbe : kGlobalProbe);
      if (g < 0) {
        note_fail(a, p[r].cnt);
        continue;
      }
      if constexpr (MM) ext[r] = __ldcg((const ulonglong2*)&tab[g].minc);
    }
    GSlot<MM>& s = tab[g];
    atomicAdd(&s.cnt, p[r].cnt);
    if (DT == AGG_F32 || DT == AGG_F64) atomicAdd((double*)&s.sum, __longlong_as_double((long long)p[r].sum));
    else atomicAdd(&s.sum, p[r].sum);
    if constexpr (MM) {
      if (p[r].nmn > ext[r].x) atomicMax(&s.minc, p[r].nmn);
      if (p[r].mx > ext[r].y) atomicMax(&s.mx, p[r].mx);
    }
  }
}

template <int DT>
struct Partial4 {  // partial aggregate of rows with one key
  uint32_t cnt;
  unsigned long long isum;  // integer sum mod 2^64
  float fs, fc;             // float32: compensated pair
  double ds;                // float64 sum
  typename SImg<DT>::U mn, mx;
};

template <int DT, bool MM>
__device__ __forceinline__ Partial4<DT> partial_of(const typename GV<DT>::T (&v)[4], uint32_t take) {
  Partial4<DT> p;
  p.cnt = 0;
  p.isum = 0;
  p.fs = 0.f;
  p.fc = 0.f;
  p.ds = 0.0;
  p.mn = (typename SImg<DT>::U) ~(typename SImg<DT>::U)0;
  p.mx = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if (!((take >> r) & 1u)) continue;
    p.cnt += 1;
    if (DT == AGG_F32) {
      float t, e;
      two_sum(p.fs, (float)v[r], t, e);
      p.fs = t;
      p.fc += e;
    } else if (DT == AGG_F64) {
      p.ds += (double)v[r];
    } else {
      p.isum += (unsigned long long)(int64_t)v[r];
    }
    if (MM) {
      const typename SImg<DT>::U m = s_img<DT>(v[r]);
      p.mn = min(p.mn, m);
      p.mx = max(p.mx, m);
    }
  }
  return p;
}

template <int DT, bool MM>
__device__ __forceinline__ void warp_reduce_partial(Partial4<DT>& p) {
  if (DT == AGG_I32 || DT == AGG_U32 || DT == AGG_I64) {
    // integers: warp reductions of 32-bit words. The sum mod 2^64 from the
    // low word's two 16-bit halves (each total below 2^21) and the high word
    // (mod 2^32); a 64-bit minimum from the high words' minimum, then the low
    // words of the lanes holding it (likewise the maximum).
    constexpr unsigned kAll = 0xffffffffu;
    p.cnt = __reduce_add_sync(kAll, p.cnt);
    const uint32_t lo = (uint32_t)p.isum;
    const uint32_t s0 = __reduce_add_sync(kAll, lo & 0xFFFFu);
    const uint32_t s1 = __reduce_add_sync(kAll, lo >> 16);
    const uint32_t sh = __reduce_add_sync(kAll, (uint32_t)(p.isum >> 32));
    p.isum = ((unsigned long long)sh << 32) + ((unsigned long long)s1 << 16) + (unsigned long long)s0;
    if (MM) {
      if (sizeof(p.mn) == 4) {
        p.mn = __reduce_min_sync(kAll, (uint32_t)p.mn);
        p.mx = __reduce_max_sync(kAll, (uint32_t)p.mx);
      } else {
        const uint64_t mn = (uint64_t)p.mn, mx = (uint64_t)p.mx;
        const uint32_t mnh = __reduce_min_sync(kAll, (uint32_t)(mn >> 32));
        const uint32_t mnl = __reduce_min_sync(kAll, (uint32_t)(mn >> 32) == mnh ? (uint32_t)mn : 0xFFFFFFFFu);
        const uint32_t mxh = __reduce_max_sync(kAll, (uint32_t)(mx >> 32));
        const uint32_t mxl = __reduce_max_sync(kAll, (uint32_t)(mx >> 32) == mxh ? (uint32_t)mx : 0u);
        p.mn = (typename SImg<DT>::U)(((uint64_t)mnh << 32) | mnl);
        p.mx = (typename SImg<DT>::U)(((uint64_t)mxh << 32) | mxl);
      }
    }
    return;
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    p.cnt += __shfl_xor_sync(0xffffffffu, p.cnt, o);
    if (DT == AGG_F32) {
      const float s2 = __shfl_xor_sync(0xffffffffu, p.fs, o), c2 = __shfl_xor_sync(0xffffffffu, p.fc, o);
      float t, e;
      two_sum(p.fs, s2, t, e);
      p.fs = t;
      p.fc += c2 + e;
    } else if (DT == AGG_F64) {
      p.ds += __shfl_xor_sync(0xffffffffu, p.ds, o);
    } else {
      p.isum += __shfl_xor_sync(0xffffffffu, p.isum, o);
    }
    if (MM) {
      p.mn = min(p.mn, __shfl_xor_sync(0xffffffffu, p.mn, o));
      p.mx = max(p.mx, __shfl_xor_sync(0xffffffffu, p.mx, o));
    }
  }
}

// The warp reduces the rows marked in take (a 4-bit mask per lane; all of
// one key) and lane 0 folds the partial into the global table.
template <int DT, bool MM>
__device__ __forceinline__ void g_fold_warp_key(const BuildArgs& a, uint32_t key, const typename GV<DT>::T (&v)[4],
                                                uint32_t take) {
  Partial4<DT> p = partial_of<DT, MM>(v, take);
  warp_reduce_partial<DT, MM>(p);
  if ((threadIdx.x & 31) != 0) return;
  GPart g[1];
  g[0].key = key;
  g[0].cnt = p.cnt;
  if (DT == AGG_F32) g[0].sum = (unsigned long long)__double_as_longlong((double)p.fs + (double)p.fc);
  else if (DT == AGG_F64) g[0].sum = (unsigned long long)__double_as_longlong(p.ds);
  else g[0].sum = p.isum;
  if (MM) {
    g[0].nmn = ~g_img_of<DT>(p.mn);
    g[0].mx = g_img_of<DT>(p.mx);
  }
  g_merge<DT, MM, 1>(a, g, 1u);
}

template <class T>
__device__ __forceinline__ void unpack4(const uint4& lo, const uint4& hi, T* v) {
  if (sizeof(T) == 4) {
    uint32_t w[4] = {lo.x, lo.y, lo.z, lo.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t x = w[i];
      memcpy(&v[i], &x, 4);
    }
  } else {
    uint64_t w[4] = {((uint64_t)lo.y << 32) | lo.x, ((uint64_t)lo.w << 32) | lo.z, ((uint64_t)hi.y << 32) | hi.x,
                     ((uint64_t)hi.w << 32) | hi.z};
#pragma unroll
    for (int i = 0; i < 4; ++i) memcpy(&v[i], &w[i], 8);
  }
}

// Per-block counts reported after a build: when a full table stopped it, the
// rows the block went through and those that found no slot are added to
// a.progress, from which the host sizes the next table. Call after a barrier
// that follows every thread's count_seen.
struct BlockCounts {
  uint32_t seen, fails;
};

__device__ __forceinline__ void report_counts(const BuildArgs& a, const BlockCounts& c) {
  if (threadIdx.x != 0 || a.progress == nullptr || *(volatile int*)a.status == 0) return;
  atomicAdd(&a.progress[0], (unsigned long long)c.seen);
  atomicAdd(&a.progress[1], (unsigned long long)c.fails);
}

// ---------------------------------------------------------------------------
// Shared-memory table of a block: S slots (a power of two in [64, kP]), a side
// slot for the key 0xFFFFFFFF and 16 scratch slots whose contents nobody reads
// (rows that fold nothing update those instead of being predicated off), as
// planes of one 32-bit word a slot, so that 32 lanes on random slots spread
// over the 32 banks. The planes lie at compile-time distances: a slot is named
// by the shared address of its key word, and every update is one instruction
// with an immediate offset.
//
// What bounds it: shared-memory wavefronts, then warp instructions. The earlier
// fold (generic pointers, one row at a time, an out-of-line lookup for every
// key outside its home bucket, predicated and branched updates, carries added
// separately) took 175 instructions and 39 wavefronts a warp and 32 rows on int64
// SUM/COUNT/MIN/MAX over 1024 keys; four rows folded phase by phase (lookups,
// sum updates, extremes) with unconditional updates take 76 and 32 (L1 pipe 89 %
// busy, issue 46 %). Builds: 2^26 int64 rows over 1024 keys 0.412 -> 0.284 ms;
// 2^28 float32 rows over 14 M keys (partitioned) 3.41 -> 2.48 ms; 2^30 int64 rows
// over 2^16 keys (partitioned) 6.51 -> 5.38 ms; 16 M float64 rows over 2^20 keys
// (partitioned) 0.47 -> 0.33 ms. Every update but those of rows outside the window
// is a native 32-bit shared atomic:
//   count   low half of the cnt word; its high half counts, for integers, the
//           carries out of the sum's low word (one atomic adds the row and its
//           carry) and, for floats, the negative rows (below). A block folds at
//           most kEpochRows rows before the halves are moved to wide words.
//   sum     integers: the value relative to a base (int32: biased to unsigned;
//           int64: the block's window, see below) in words w0, w1; the low
//           word's atomic returns the previous value, so the adding thread
//           sees its own carry. w1 is touched only by values outside the
//           window. float32 and float64: a fixed-point number (64 and 96 bits)
//           in units of the lowest bit the window's lowest exponent can have,
//           exact for every value whose exponent lies in the window (24 and 27
//           binades); negative rows add their one's complement, and the high
//           half of the cnt word counts the +1s they owe. Float atomics would
//           be compare-and-swap loops (float32 6.6, float64 9.4 clocks a row).
//           Other finite values, infinities and NaN take the word fb: a
//           compensated float32 pair or a float64, updated with those loops.
//   MIN/MAX an adjacent pair of 32-bit words in one 8-byte read: the minimum
//           as the maximum of the complements, so that an empty table is all
//           zeros; an update is issued only for a value that moves one. 4-byte
//           types: the order-preserving image. int64: the offset in the
//           window, other values on a pair of 64-bit images (mm64). float64: a
//           pair of 64-bit images.
// The window of a block or tile comes from 32 of its rows: int64: 2^32 values
// from a base that holds the sampled range (aligned to 2^32 when the samples
// share their high word, else centred); floats: up to 3 binades above the
// largest exponent sampled (of 512 rows more when the 32 are zeros).
// ---------------------------------------------------------------------------
constexpr uint32_t kMiss = 0xFFFFFFFFu;  // no slot (yet)
constexpr int64_t kEpochRows = 65532;    // rows a block folds between two moves of the cnt halves (a multiple of 4)
constexpr int kScratchSlots = 16;

constexpr bool is_f32(int dt) { return dt == AGG_F32; }
constexpr bool is_f64(int dt) { return dt == AGG_F64; }
constexpr bool is_float(int dt) { return dt == AGG_F32 || dt == AGG_F64; }
constexpr bool is_wide(int dt) { return dt == AGG_I64 || dt == AGG_F64; }

// Planes of a table. WIDE: for blocks of more than kEpochRows rows (one block
// a SM, up to 4096 slots); else two blocks a SM (float64 sums of 4096 slots
// just fit twice).
template <int DT, bool MM, bool WIDE>
struct Lay {
  static constexpr int kP = MM && (!WIDE || is_f64(DT)) ? 2048 : 4096;  // most slots
  static constexpr int kStride = (kP + 4 + kScratchSlots) * 4;          // bytes of a plane (a multiple of 16)
  static constexpr int kKey = 0;
  static constexpr int kMM64 = kStride;                                            // four words a slot
  static constexpr int kMM = kMM64 + (MM && is_wide(DT) ? 4 * kStride : 0);        // two words a slot (not float64)
  static constexpr int kFb = kMM + (MM && !is_f64(DT) ? 2 * kStride : 0);          // two words a slot
  static constexpr int kCnt = kFb + (is_float(DT) ? 2 * kStride : 0);
  static constexpr int kW0 = kCnt + kStride;
  static constexpr int kW1 = kW0 + kStride;
  static constexpr int kW2 = kW1 + kStride;                                        // float64
  static constexpr int kCnt32 = kW2 + (is_f64(DT) ? kStride : 0);                  // WIDE: count
  static constexpr int kTop = kCnt32 + (WIDE ? kStride : 0);                       // WIDE floats: wide top word
  static constexpr int kBytes = kTop + (WIDE && is_float(DT) ? kStride : 0);
};

// Shared memory of a block's table, and its most slots.
inline size_t stab_bytes_dt(int dt, bool mm, bool wide) {
#define AGG_SB(D)                                                                  \
  case D:                                                                          \
    return wide ? (mm ? Lay<D, true, true>::kBytes : Lay<D, false, true>::kBytes) \
                : (mm ? Lay<D, true, false>::kBytes : Lay<D, false, false>::kBytes);
  switch (dt) { AGG_SB(AGG_I32) AGG_SB(AGG_I64) AGG_SB(AGG_U32) AGG_SB(AGG_F32) AGG_SB(AGG_F64) }
#undef AGG_SB
  return 0;
}
inline int stab_max_slots(int dt, bool mm, bool wide) { return mm && (!wide || dt == AGG_F64) ? 2048 : 4096; }

// Shared-memory accesses at a + OFF.
template <int OFF>
__device__ __forceinline__ uint32_t sm_ld(uint32_t a) {
  uint32_t v;
  asm volatile("ld.volatile.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
  return v;
}
template <int OFF>
__device__ __forceinline__ uint2 sm_ld2(uint32_t a) {
  uint2 v;
  asm volatile("ld.volatile.shared.v2.u32 {%0,%1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(a), "n"(OFF));
  return v;
}
template <int OFF>
__device__ __forceinline__ uint4 sm_ld4(uint32_t a) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0,%1,%2,%3}, [%4+%5];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a), "n"(OFF));
  return v;
}
template <int OFF>
__device__ __forceinline__ ulonglong2 sm_ld2_64(uint32_t a) {
  ulonglong2 v;
  asm volatile("ld.volatile.shared.v2.u64 {%0,%1}, [%2+%3];" : "=l"(v.x), "=l"(v.y) : "r"(a), "n"(OFF));
  return v;
}
template <int OFF>
__device__ __forceinline__ void sm_st2_64(uint32_t a, unsigned long long x, unsigned long long y) {
  asm volatile("st.volatile.shared.v2.u64 [%0+%3], {%1,%2};" ::"r"(a), "l"(x), "l"(y), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ void sm_st2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.volatile.shared.v2.u32 [%0+%3], {%1,%2};" ::"r"(a), "r"(x), "r"(y), "n"(OFF));
}
// 64-bit maxima (a compare-and-swap loop), issued only where v exceeds cur.
template <int OFF>
__device__ __forceinline__ void sm_raise64(uint32_t a, unsigned long long v, unsigned long long cur) {
  if (v > cur) asm volatile("red.shared.max.u64 [%0+%2], %1;" ::"r"(a), "l"(v), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ void sm_st(uint32_t a, uint32_t v) {
  asm volatile("st.volatile.shared.u32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF));
}
template <int OFF>
__device__ __forceinline__ uint32_t sm_add_ret(uint32_t a, uint32_t v) {
  uint32_t o;
  asm volatile("atom.shared.add.u32 %0, [%1+%3], %2;" : "=r"(o) : "r"(a), "r"(v), "n"(OFF));
  return o;
}
template <int OFF>
__device__ __forceinline__ void sm_add(uint32_t a, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF));
}
// max of the word with v, issued only where v exceeds cur (a value read before)
template <int OFF>
__device__ __forceinline__ void sm_raise(uint32_t a, uint32_t v, uint32_t cur) {
  asm volatile("{.reg .pred q; setp.gt.u32 q, %1, %2; @q red.shared.max.u32 [%0+%3], %1;}" ::"r"(a), "r"(v), "r"(cur),
               "n"(OFF));
}
__device__ __forceinline__ uint32_t sm_cas(uint32_t a, uint32_t cmp, uint32_t v) {
  uint32_t o;
  asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(o) : "r"(a), "r"(cmp), "r"(v));
  return o;
}

// Block window (shared memory, one per block).
struct Window {
  unsigned long long base;  // int64: image of the first value of the 2^32-value window
  int ebase;                // floats: exponent field of the lowest exact binade
};

template <int DT, bool MM, bool WIDE>
struct STab {
  using L = Lay<DT, MM, WIDE>;
  uint32_t b0;              // shared address of the key plane
  uint32_t mask;            // 4 S - 16: byte offsets of the buckets
  int shift;                // a key's hash >> shift, masked, is its bucket's byte offset
  unsigned long long base;  // window (int64)
  int ebase;                // window (floats)
  __device__ __forceinline__ void init(const void* smem, int S) {
    b0 = (uint32_t)__cvta_generic_to_shared(smem);
    mask = 4u * (uint32_t)S - 16u;
    shift = __clz(S) - 1;  // 30 - log2(S)
  }
  __device__ __forceinline__ void set_window(const Window& w) {
    base = w.base;
    ebase = w.ebase;
  }
  __device__ __forceinline__ uint32_t side() const { return b0 + 4 * L::kP; }
  __device__ __forceinline__ uint32_t scratch() const { return b0 + 4 * L::kP + 16 + 4 * (threadIdx.x & (kScratchSlots - 1)); }
  // Bucket (address of its first key word): a multiplicative hash (the golden
  // ratio's odd multiplier) of the key folded once; the table tolerates a poor
  // hash (rows without a slot spill to the global table).
  __device__ __forceinline__ uint32_t bucket(uint32_t key) const {
    return b0 + ((((key ^ (key >> 15)) * 0x9E3779B1u) >> shift) & mask);
  }
  // The slot of the next bucket after the one at a.
  __device__ __forceinline__ uint32_t next(uint32_t a) const { return b0 + ((a - b0 + 16) & mask); }
  // An empty table is all zeros.
  __device__ __forceinline__ void clear() const {
    clear_plane<L::kKey, 1>();
    if (MM) {
      if (is_wide(DT)) clear_plane<L::kMM64, 4>();
      if (!is_f64(DT)) clear_plane<L::kMM, 2>();
    }
    if (is_float(DT)) clear_plane<L::kFb, 2>();
    clear_plane<L::kCnt, 1>();
    clear_plane<L::kW0, 1>();
    clear_plane<L::kW1, 1>();
    if (is_f64(DT)) clear_plane<L::kW2, 1>();
    if (WIDE) {
      clear_plane<L::kCnt32, 1>();
      if (is_float(DT)) clear_plane<L::kTop, 1>();
    }
  }

 private:
  // The S slots and the side slot of a plane of WORDS words a slot.
  template <int OFF, int WORDS>
  __device__ __forceinline__ void clear_plane() const {
    const uint32_t n = (mask + 16) * WORDS;
    for (uint32_t i = 16 * threadIdx.x; i < n; i += 16 * blockDim.x) zero16(b0 + OFF + i);
    if (threadIdx.x == 0) zero16(b0 + OFF + 4 * WORDS * L::kP);
  }
  __device__ static __forceinline__ void zero16(uint32_t a) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(a), "r"(0u));
  }
};

__device__ __forceinline__ uint32_t s_match(const uint4& q, uint32_t k1, uint32_t b) {
  uint32_t j = q.x == k1 ? b : kMiss;
  j = q.y == k1 ? b + 4 : j;
  j = q.z == k1 ? b + 8 : j;
  return q.w == k1 ? b + 12 : j;
}

// Slot of a key (given as key + 1): its home bucket or the next one, inserting
// the key in the first empty slot, or kMiss when both are full (the row then
// goes to the global table). Each failed claim means that a slot filled, so 8
// claims and 2 full buckets end the loop.
template <class TAB>
__device__ __forceinline__ uint32_t s_place(uint32_t k1, const TAB& t) {
  uint32_t b = t.bucket(k1 - 1);
  bool second = false;
#pragma unroll 1
  for (int tries = 0; tries < 10; ++tries) {
    const uint4 q = sm_ld4<0>(b);
    const uint32_t j = s_match(q, k1, b);
    if (j != kMiss) return j;
    const uint32_t e = s_match(q, 0u, b);
    if (e != kMiss) {
      const uint32_t old = sm_cas(e, 0u, k1);
      if (old == 0u || old == k1) return e;
    } else {
      if (second) break;
      second = true;
      b = t.next(b);
    }
  }
  return kMiss;
}

// A value in the table's terms: the sum's words (e0, e1, e2; floats in one's
// complement with neg = 0x10000 when negative), whether the window holds it
// (ok), and the word the MIN/MAX pair compares (m).
template <int DT>
struct Enc {
  uint32_t e0, e1, e2, neg, m;
  bool ok;
};

template <int DT, class TAB>
__device__ __forceinline__ Enc<DT> s_enc(const TAB& t, typename GV<DT>::T v) {
  Enc<DT> e;
  e.e1 = e.e2 = e.neg = 0u;
  e.ok = true;
  if constexpr (DT == AGG_I32) {
    e.e0 = (uint32_t)v ^ 0x80000000u;
    e.m = e.e0;
  } else if constexpr (DT == AGG_U32) {
    e.e0 = v;
    e.m = v;
  } else if constexpr (DT == AGG_I64) {
    const uint64_t u = img_i64(v) - t.base;
    e.e0 = (uint32_t)u;
    e.e1 = (uint32_t)(u >> 32);
    e.m = e.e0;
    e.ok = e.e1 == 0u;
  } else if constexpr (DT == AGG_F32) {
    const uint32_t b = __float_as_uint(v);
    const uint32_t s = (uint32_t)((int32_t)b >> 31);
    const uint32_t sh = ((b >> 23) & 0xFFu) - (uint32_t)t.ebase;
    const uint32_t mant = (b & 0x007FFFFFu) | 0x00800000u;
    e.ok = sh < 24u;  // a window's ebase is at least 1: zero and subnormals are not ok
    e.e0 = (mant << (sh & 31u)) ^ s;
    e.e1 = __funnelshift_l(mant, 0u, sh) ^ s;
    e.neg = s & 0x10000u;
    e.m = b ^ (s | 0x80000000u);
  } else {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const uint32_t bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    const uint32_t s = (uint32_t)((int32_t)bh >> 31);
    const uint32_t sh = ((bh >> 20) & 0x7FFu) - (uint32_t)t.ebase;
    const uint32_t mh = (bh & 0x000FFFFFu) | 0x00100000u;
    e.ok = sh < 27u;
    e.e0 = (bl << (sh & 31u)) ^ s;
    e.e1 = __funnelshift_l(bl, mh, sh) ^ s;
    e.e2 = __funnelshift_l(mh, 0u, sh) ^ s;
    e.neg = s & 0x10000u;
    e.m = bh ^ (s | 0x80000000u);  // the image's high word
  }
  return e;
}

// Sum of a float the window does not hold (zeros add nothing), into the fb words at a.
template <int DT>
__device__ __forceinline__ void s_add_other(uint32_t a, typename GV<DT>::T v) {
  if (v == typename GV<DT>::T(0)) return;
  if constexpr (DT == AGG_F32) {
    float old, sum, err;
    asm volatile("atom.shared.add.f32 %0, [%1], %2;" : "=f"(old) : "r"(a), "f"(v));
    two_sum(old, v, sum, err);
    if (err != 0.f) asm volatile("red.shared.add.f32 [%0+4], %1;" ::"r"(a), "f"(err));
  } else if constexpr (DT == AGG_F64) {
    asm volatile("red.shared.add.f64 [%0], %1;" ::"r"(a), "d"(v));
  }
}

// MIN/MAX of image m on the 64-bit pair at a (int64 values outside the window).
static __device__ __noinline__ void s_mm64(uint32_t a, uint64_t m) {
  const ulonglong2 q = sm_ld2_64<0>(a);
  sm_raise64<0>(a, ~m, q.x);
  sm_raise64<8>(a, m, q.y);
}

// Fold the N rows marked in rows (N-bit mask; ALL: every row).
template <int DT, bool MM, int N, bool ALL, class TAB>
__device__ __forceinline__ void s_fold(const BuildArgs& a, const TAB& t, const uint32_t (&key)[N],
                                       const typename GV<DT>::T (&val)[N], uint32_t rows) {
  using L = typename TAB::L;
  uint32_t j[N];
  uint32_t spilled = 0u;  // rows without a slot: folded into the global table below
  {
    uint32_t b[N];
    uint4 q[N];
    uint32_t kmax = 0u;
#pragma unroll
    for (int r = 0; r < N; ++r) {
      b[r] = t.bucket(key[r]);
      q[r] = sm_ld4<0>(b[r]);
      kmax = max(kmax, key[r]);
    }
    bool miss = false;
#pragma unroll
    for (int r = 0; r < N; ++r) {
      j[r] = s_match(q[r], key[r] + 1, b[r]);
      if (!ALL) j[r] = ((rows >> r) & 1u) ? j[r] : t.scratch();
      miss |= j[r] == kMiss;
    }
    // Keys outside their home bucket, new keys, and the key 0xFFFFFFFF (its key
    // word would be an empty slot's): the home bucket again, then the next one;
    // a new key claims the first of them with room (all rows' claims in flight
    // together: a column of many keys has some such row in every warp), and
    // lost races are settled one row at a time.
    if (miss || kmax == 0xFFFFFFFFu) {
      uint32_t old[N];
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (key[r] == 0xFFFFFFFFu && (ALL || ((rows >> r) & 1u))) j[r] = t.side();
        old[r] = 0u;
        if (j[r] != kMiss) continue;
        uint32_t b = t.bucket(key[r]);
        uint4 q = sm_ld4<0>(b);
        j[r] = s_match(q, key[r] + 1, b);
        uint32_t e = s_match(q, 0u, b);
        if (j[r] == kMiss && e == kMiss) {
          b = t.next(b);
          q = sm_ld4<0>(b);
          j[r] = s_match(q, key[r] + 1, b);
          e = s_match(q, 0u, b);
        }
        if (j[r] == kMiss) {
          if (e != kMiss) {
            j[r] = e;
            old[r] = sm_cas(e, 0u, key[r] + 1);
          } else {
            j[r] = t.scratch();
            spilled |= 1u << r;
          }
        }
      }
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (old[r] == 0u || old[r] == key[r] + 1) continue;
        j[r] = s_place(key[r] + 1, t);
        if (j[r] == kMiss) {
          spilled |= 1u << r;
          j[r] = t.scratch();
        }
      }
    }
  }
  Enc<DT> e[N];
  uint32_t old[N], js[N];  // js: where the sum goes (a float outside the window adds to fb instead)
  bool other = false;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    e[r] = s_enc<DT>(t, val[r]);
    other |= !e[r].ok;
    js[r] = !is_float(DT) || e[r].ok ? j[r] : t.scratch();
    old[r] = sm_add_ret<L::kW0>(js[r], e[r].e0);
  }
  uint2 ext[N];
  if constexpr (MM && DT != AGG_F64) {
#pragma unroll
    for (int r = 0; r < N; ++r) ext[r] = sm_ld2<L::kMM>(j[r] + (j[r] - t.b0));
  }
  if constexpr (is_float(DT)) {
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const uint32_t c = (uint32_t)(old[r] + e[r].e0) < old[r] ? 1u : 0u;
      e[r].e1 += c;
      if constexpr (is_f64(DT)) {
        // e1 + c wraps only to 0, which carries by itself and adds nothing
        e[r].e2 += e[r].e1 < c ? 1u : 0u;
        old[r] = sm_add_ret<L::kW1>(js[r], e[r].e1);
      } else {
        sm_add<L::kW1>(js[r], e[r].e1);
      }
    }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      sm_add<L::kCnt>(j[r], 1u + (e[r].ok ? e[r].neg : 0u));
      if constexpr (is_f64(DT)) sm_add<L::kW2>(js[r], e[r].e2 + ((uint32_t)(old[r] + e[r].e1) < old[r] ? 1u : 0u));
    }
  } else {
#pragma unroll
    for (int r = 0; r < N; ++r) sm_add<L::kCnt>(j[r], (uint32_t)(old[r] + e[r].e0) < old[r] ? 0x10001u : 1u);
  }
  if (DT != AGG_I32 && DT != AGG_U32 && other) {  // rows outside the window
#pragma unroll
    for (int r = 0; r < N; ++r) {
      if (e[r].ok) continue;
      if constexpr (is_float(DT)) {
        s_add_other<DT>(j[r] + (j[r] - t.b0) + L::kFb, val[r]);
      } else {
        sm_add<L::kW1>(j[r], e[r].e1);
        if (MM) s_mm64(t.b0 + L::kMM64 + 4 * (j[r] - t.b0), GV<DT>::img(val[r]));
        ext[r] = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);  // the window's pair stays as it is
      }
    }
  }
  if constexpr (MM) {
    if constexpr (DT == AGG_F64) {
      ulonglong2 x[N];
#pragma unroll
      for (int r = 0; r < N; ++r) x[r] = sm_ld2_64<L::kMM64>(t.b0 + 4 * (j[r] - t.b0));
#pragma unroll
      for (int r = 0; r < N; ++r) {
        const uint64_t m = GV<DT>::img(val[r]);
        sm_raise64<L::kMM64>(t.b0 + 4 * (j[r] - t.b0), ~m, x[r].x);
        sm_raise64<L::kMM64 + 8>(t.b0 + 4 * (j[r] - t.b0), m, x[r].y);
      }
    } else {
#pragma unroll
      for (int r = 0; r < N; ++r) {
        sm_raise<L::kMM>(j[r] + (j[r] - t.b0), ~e[r].m, ext[r].x);
        sm_raise<L::kMM + 4>(j[r] + (j[r] - t.b0), e[r].m, ext[r].y);
      }
    }
  }
  if (spilled != 0u) {
    GPart g[N];
#pragma unroll
    for (int r = 0; r < N; ++r) g[r] = g_part_of<DT, MM>(key[r], val[r]);
    g_merge<DT, MM, N>(a, g, spilled);
  }
}

// ---------------------------------------------------------------------------
// Frequent keys: when at least kDominantRows of the 128 rows a warp holds
// carry one key (hot keys of a skewed, partitioned or clustered input, or a
// column with a handful of keys), the warp reduces those rows with warp
// reductions and one lane applies the partial aggregate; the remaining rows
// take the per-row path. This removes the same-slot atomic conflicts that
// frequent keys cause.
// ---------------------------------------------------------------------------
constexpr int kDominantRows = 16; // rows of one key (of 128) that make a reduced update pay
constexpr int kDominantOther = 4; // of floats outside the window (compare-and-swap updates)
                                  // (above 8 keys: 30 keys, float32 294 us with 4, 337 with 16)
constexpr int kMaxWarpKeys = 8;   // keys reduced per warp and quad of rows, at most

// a2:a1:a0 += v
__device__ __forceinline__ void add96(uint32_t& a0, uint32_t& a1, uint32_t& a2, uint32_t v) {
  asm("{add.cc.u32 %0, %0, %3; addc.cc.u32 %1, %1, 0; addc.u32 %2, %2, 0;}" : "+r"(a0), "+r"(a1), "+r"(a2) : "r"(v));
}

// The fixed-point sum top:w1:w0 (float64) or top:w0 (float32) of a window as a
// float64. float32: one rounding (both words are float64 integers). float64: the
// magnitude's low word is rounded, then the whole, each to 2^-53 of the sum (of
// the two's complement itself, a small negative sum's low word lies just below
// 2^64 and would be rounded to multiples of 2^11 units); a single value has no
// bits below its word's 53 and is exact. Then an exact scaling.
template <int DT>
__device__ __forceinline__ double fixed_to_double(int ebase, int64_t top, uint32_t w1, uint32_t w0) {
  if (DT == AGG_F32) {
    const double s = __hiloint2double((ebase - 150 + 1023) << 20, 0);
    return fma((double)top, 4294967296.0, (double)w0) * s;
  }
  const uint64_t neg = (uint64_t)(top >> 63);  // all ones for a negative sum
  uint64_t lo = (((uint64_t)w1 << 32) | w0) ^ neg;
  uint64_t hi = (uint64_t)top ^ neg;
  lo -= neg;
  hi += neg != 0 && lo == 0 ? 1u : 0u;
  const double d = fma((double)hi, 18446744073709551616.0, (double)lo);
  const int k = (ebase - 1075) / 2;  // in two steps, so that neither factor leaves the normal range
  const double m = d * __hiloint2double((k + 1023) << 20, 0) * __hiloint2double((ebase - 1075 - k + 1023) << 20, 0);
  return neg != 0 ? -m : m;
}

// What a row's value exceeds its sum term by (mod 2^64).
template <int DT>
__device__ __forceinline__ unsigned long long int_base(unsigned long long window) {
  return DT == AGG_I32 ? 0xFFFFFFFF80000000ull : DT == AGG_I64 ? window ^ 0x8000000000000000ull : 0ull;
}

// Warp sums mod 2^32 with the bits above returned in hi (each lane's halves
// total below 2^21).
__device__ __forceinline__ void warp_add32(uint32_t v, uint32_t& lo, uint32_t& carry) {
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, v & 0xFFFFu);
  const uint32_t s1 = __reduce_add_sync(0xffffffffu, v >> 16);
  const uint64_t s = ((uint64_t)s1 << 16) + s0;
  lo = (uint32_t)s;
  carry = (uint32_t)(s >> 32);
}

// The warp reduces the rows marked in take (a 4-bit mask a lane; all of one
// key, floats all zero or in the window) and lane 0 adds them to the key's slot.
template <int DT, bool MM, class TAB>
__device__ __forceinline__ void s_fold_warp_key(const BuildArgs& a, const TAB& t, uint32_t key,
                                                const typename GV<DT>::T (&v)[4], uint32_t take) {
  using L = typename TAB::L;
  constexpr unsigned kAll = 0xffffffffu;
  uint32_t c0 = 0, c1 = 0, c2 = 0;  // this lane's sum words (floats: two's complement)
  uint32_t mn32 = 0xFFFFFFFFu, mx32 = 0u;
  uint64_t mn = ~0ull, mx = 0ull;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if (!((take >> r) & 1u)) continue;
    const Enc<DT> e = s_enc<DT>(t, v[r]);
    if (!is_float(DT) || e.ok) {  // zeros add nothing
      asm("{add.cc.u32 %0, %0, %3; addc.cc.u32 %1, %1, %4; addc.u32 %2, %2, %5;}"
          : "+r"(c0), "+r"(c1), "+r"(c2)
          : "r"(e.e0), "r"(e.e1), "r"(e.e2));
      if (is_float(DT)) add96(c0, c1, c2, e.neg >> 16);  // the +1 of a negative row's two's complement
    }
    if (MM) {
      if (is_wide(DT)) {
        const uint64_t m = GV<DT>::img(v[r]);
        mn = min(mn, m);
        mx = max(mx, m);
      } else {
        mn32 = min(mn32, e.m);
        mx32 = max(mx32, e.m);
      }
    }
  }
  const uint32_t cnt = __reduce_add_sync(kAll, (uint32_t)__popc(take));
  uint32_t w0, w1, w2 = 0, k0, k1 = 0;
  warp_add32(c0, w0, k0);
  if (is_f64(DT)) {
    warp_add32(c1, w1, k1);
    w1 += k0;
    k1 += w1 < k0 ? 1u : 0u;
    w2 = __reduce_add_sync(kAll, c2) + k1;
  } else {
    w1 = __reduce_add_sync(kAll, c1) + k0;
  }
  if (MM) {
    if (is_wide(DT)) {  // the high words' minimum, then the low words of the lanes holding it
      const uint32_t nh = __reduce_min_sync(kAll, (uint32_t)(mn >> 32));
      const uint32_t nl = __reduce_min_sync(kAll, (uint32_t)(mn >> 32) == nh ? (uint32_t)mn : 0xFFFFFFFFu);
      const uint32_t xh = __reduce_max_sync(kAll, (uint32_t)(mx >> 32));
      const uint32_t xl = __reduce_max_sync(kAll, (uint32_t)(mx >> 32) == xh ? (uint32_t)mx : 0u);
      mn = ((uint64_t)nh << 32) | nl;
      mx = ((uint64_t)xh << 32) | xl;
    } else {
      mn32 = __reduce_min_sync(kAll, mn32);
      mx32 = __reduce_max_sync(kAll, mx32);
    }
  }
  if ((threadIdx.x & 31) != 0) return;
  uint32_t j = t.side();
  if (key != 0xFFFFFFFFu) {
    j = s_place(key + 1, t);
  }
  if (j == kMiss) {  // no slot: the partial goes to the global table
    GPart g[1];
    g[0].key = key;
    g[0].cnt = cnt;
    if constexpr (is_float(DT))
      g[0].sum = (unsigned long long)__double_as_longlong(fixed_to_double<DT>(t.ebase, (int32_t)(is_f64(DT) ? w2 : w1), w1, w0));
    else
      g[0].sum = (((unsigned long long)w1 << 32) | w0) + cnt * int_base<DT>(t.base);
    if (MM) {
      g[0].nmn = ~(is_wide(DT) ? mn : g_img_of<DT>((typename SImg<DT>::U)mn32));
      g[0].mx = is_wide(DT) ? mx : g_img_of<DT>((typename SImg<DT>::U)mx32);
    }
    g_merge<DT, MM, 1>(a, g, 1u);
    return;
  }
  const uint32_t old = sm_add_ret<L::kW0>(j, w0);
  const uint32_t c = (uint32_t)(old + w0) < old ? 1u : 0u;
  if constexpr (is_float(DT)) {
    sm_add<L::kCnt>(j, cnt);
    w1 += c;
    if constexpr (is_f64(DT)) {
      w2 += w1 < c ? 1u : 0u;
      const uint32_t old1 = sm_add_ret<L::kW1>(j, w1);
      sm_add<L::kW2>(j, w2 + ((uint32_t)(old1 + w1) < old1 ? 1u : 0u));
    } else {
      sm_add<L::kW1>(j, w1);
    }
  } else {
    sm_add<L::kCnt>(j, cnt + (c << 16));
    if (w1 != 0u) sm_add<L::kW1>(j, w1);
  }
  if constexpr (MM) {
    if constexpr (is_wide(DT)) {
      const uint32_t jw = t.b0 + L::kMM64 + 4 * (j - t.b0);
      if (DT == AGG_F64 || (uint32_t)((mn - t.base) >> 32) != 0u || (uint32_t)((mx - t.base) >> 32) != 0u) {
        const ulonglong2 q = sm_ld2_64<0>(jw);
        sm_raise64<0>(jw, ~mn, q.x);
        sm_raise64<8>(jw, mx, q.y);
        return;
      }
      mn32 = (uint32_t)(mn - t.base);
      mx32 = (uint32_t)(mx - t.base);
    }
    const uint32_t jm = j + (j - t.b0);
    const uint2 q = sm_ld2<L::kMM>(jm);
    sm_raise<L::kMM>(jm, ~mn32, q.x);
    sm_raise<L::kMM + 4>(jm, mx32, q.y);
  }
}

// The same for a key with floats outside the window: all of its rows as a
// compensated float32 pair or a float64 sum, into the slot's fb words. (Row by row,
// they are compare-and-swap loops on one address. 2^24 rows with exponents uniform
// over 60 binades, SUM/COUNT: of 8 keys, float32 664 us, 306 so, float64 1621 and
// 828; of 10^6 skewed keys, float32 1362 and 748, float64 5003 and 945.)
template <int DT, bool MM>
__device__ __noinline__ Partial4<DT> s_other_partial(typename GV<DT>::T v0, typename GV<DT>::T v1,
                                                     typename GV<DT>::T v2, typename GV<DT>::T v3, uint32_t take) {
  const typename GV<DT>::T v[4] = {v0, v1, v2, v3};
  Partial4<DT> p = partial_of<DT, MM>(v, take);
  warp_reduce_partial<DT, MM>(p);
  return p;
}

template <int DT, bool MM, class TAB>
__device__ __forceinline__ void s_fold_warp_other(const BuildArgs& a, const TAB& t, uint32_t key,
                                                  const typename GV<DT>::T (&v)[4], uint32_t take) {
  using L = typename TAB::L;
  const Partial4<DT> p = s_other_partial<DT, MM>(v[0], v[1], v[2], v[3], take);
  if ((threadIdx.x & 31) != 0) return;
  const uint32_t j = key == 0xFFFFFFFFu ? t.side() : s_place(key + 1, t);
  if (j == kMiss) {
    GPart g[1];
    g[0].key = key;
    g[0].cnt = p.cnt;
    g[0].sum = (unsigned long long)__double_as_longlong(is_f32(DT) ? (double)p.fs + (double)p.fc : p.ds);
    if (MM) {
      g[0].nmn = ~g_img_of<DT>(p.mn);
      g[0].mx = g_img_of<DT>(p.mx);
    }
    g_merge<DT, MM, 1>(a, g, 1u);
    return;
  }
  sm_add<L::kCnt>(j, p.cnt);
  const uint32_t jf = j + (j - t.b0) + L::kFb;
  if constexpr (is_f32(DT)) {
    s_add_other<DT>(jf, p.fs);
    if (p.fc != 0.f) asm volatile("red.shared.add.f32 [%0+4], %1;" ::"r"(jf), "f"(p.fc));
    if constexpr (MM) {
      const uint32_t jm = j + (j - t.b0);
      const uint2 q = sm_ld2<L::kMM>(jm);
      sm_raise<L::kMM>(jm, ~p.mn, q.x);
      sm_raise<L::kMM + 4>(jm, p.mx, q.y);
    }
  } else {
    s_add_other<DT>(jf, p.ds);
    if constexpr (MM) {
      const uint32_t jw = t.b0 + L::kMM64 + 4 * (j - t.b0);
      const ulonglong2 q = sm_ld2_64<0>(jw);
      sm_raise64<0>(jw, ~(uint64_t)p.mn, q.x);
      sm_raise64<8>(jw, (uint64_t)p.mx, q.y);
    }
  }
}

// The window of rows [0, n) of vals, from 32 of them (called by one whole warp).
template <int DT>
__device__ __forceinline__ void s_window(const typename GV<DT>::T* vals, int64_t n, Window* w) {
  const int lane = threadIdx.x & 31;
  const int64_t r = n > 32 ? (int64_t)lane * (n / 32) : min((int64_t)lane, n - 1);
  if constexpr (DT == AGG_I64) {
    uint64_t mn = n > 0 ? img_i64(vals[r]) : 0ull, mx = mn;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      mn = min(mn, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)mn, o));
      mx = max(mx, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)mx, o));
    }
    const uint64_t range = mx - mn, span = uint64_t(1) << 32;
    uint64_t b = mn & ~0xFFFFFFFFull;
    if ((mn >> 32) != (mx >> 32) && range < span) {
      const uint64_t margin = (span - range) / 2;
      b = mn > margin ? mn - margin : 0;
      b = min(b, (uint64_t)(0 - span));  // the window ends at 2^64 at most
    }
    if (lane == 0) w->base = b;
  } else if constexpr (is_float(DT)) {
    constexpr uint32_t kInf = is_f32(DT) ? 0xFFu : 0x7FFu;
    auto exponent = [&](int64_t i) -> uint32_t {
      uint32_t e;
      if constexpr (is_f32(DT)) e = (__float_as_uint(vals[i]) >> 23) & 0xFFu;
      else e = (uint32_t)((uint64_t)__double_as_longlong(vals[i]) >> 52) & 0x7FFu;
      return e == kInf ? 0u : e;
    };
    uint32_t e = __reduce_max_sync(0xffffffffu, n > 0 ? exponent(r) : 0u);
    if (e == 0u && n > 32) {  // zeros only: a column of few other values shows one among 512 rows more
      constexpr int kMore = 16;
      const int64_t step = max(n / (32 * kMore), (int64_t)1);
      uint32_t x[kMore];
#pragma unroll
      for (int u = 0; u < kMore; ++u) x[u] = exponent(min((lane * kMore + u) * step + step / 2, n - 1));
#pragma unroll
      for (int u = 0; u < kMore; ++u) e = max(e, x[u]);
      e = __reduce_max_sync(0xffffffffu, e);
    }
    const int top = (int)e + 3;
    if (lane == 0) w->ebase = max(1, min(top, (int)kInf - 1) - (is_f32(DT) ? 23 : 26));
  }
}

// Move the halves of the cnt words to the wide count, the carries into the sum
// and, for floats, the top word's upper part to the wide top word (blocks of
// more than kEpochRows rows; all threads, between two barriers).
template <int DT, bool MM>
__device__ __forceinline__ void s_settle(const STab<DT, MM, true>& t) {
  using L = Lay<DT, MM, true>;
  const int S = (int)(t.mask / 4) + 4;
  for (int i = threadIdx.x; i <= S; i += blockDim.x) {
    const uint32_t j = t.b0 + 4 * (i == S ? L::kP : i);
    const uint32_t w = sm_ld<L::kCnt>(j);
    if (w == 0) continue;
    sm_st<L::kCnt>(j, 0u);
    sm_st<L::kCnt32>(j, sm_ld<L::kCnt32>(j) + (w & 0xFFFFu));
    if constexpr (is_float(DT)) {
      uint32_t a0 = sm_ld<L::kW0>(j), a1 = sm_ld<L::kW1>(j), a2 = is_f64(DT) ? sm_ld<L::kW2>(j) : 0u;
      add96(a0, a1, a2, w >> 16);
      const int32_t h = (int32_t)(is_f64(DT) ? a2 : a1);
      sm_st<L::kTop>(j, sm_ld<L::kTop>(j) + (uint32_t)(h >> 16));
      sm_st<L::kW0>(j, a0);
      if (is_f64(DT)) sm_st<L::kW1>(j, a1);
      sm_st<is_f64(DT) ? L::kW2 : L::kW1>(j, (uint32_t)h & 0xFFFFu);
    } else {
      sm_st<L::kW1>(j, sm_ld<L::kW1>(j) + (w >> 16));
    }
  }
}

// Merge a block's shared table into the global table (after a barrier). CLEAR:
// and leave it empty.
template <int DT, bool MM, bool WIDE, bool CLEAR>
__device__ __forceinline__ void s_flush(const BuildArgs& a, const STab<DT, MM, WIDE>& t) {
  using L = Lay<DT, MM, WIDE>;
  constexpr int N = MM ? 2 : 4;  // slots a thread merges at once
  const int S = (int)(t.mask / 4) + 4;
  for (int i0 = threadIdx.x; i0 <= S; i0 += N * blockDim.x) {
    GPart g[N];
    uint32_t parts = 0u;
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int i = i0 + r * (int)blockDim.x;
      g[r].key = 0u;
      if (i > S) continue;
      const uint32_t j = t.b0 + 4 * (i == S ? L::kP : i);
      const uint32_t w = sm_ld<L::kCnt>(j);
      const uint32_t c = (w & 0xFFFFu) + (WIDE ? sm_ld<L::kCnt32>(j) : 0u);
      if (c == 0) continue;
      parts |= 1u << r;
      g[r].key = i == S ? 0xFFFFFFFFu : sm_ld<L::kKey>(j) - 1;
      g[r].cnt = c;
      uint32_t a0 = sm_ld<L::kW0>(j), a1 = sm_ld<L::kW1>(j);
      if (CLEAR) {
        sm_st<L::kKey>(j, 0u);
        sm_st<L::kCnt>(j, 0u);
        sm_st<L::kW0>(j, 0u);
        sm_st<L::kW1>(j, 0u);
      }
      if constexpr (is_float(DT)) {
        uint32_t a2 = is_f64(DT) ? sm_ld<L::kW2>(j) : 0u;
        if (CLEAR && is_f64(DT)) sm_st<L::kW2>(j, 0u);
        add96(a0, a1, a2, w >> 16);
        int64_t top = (int32_t)(is_f64(DT) ? a2 : a1);
        if (WIDE) top += (int64_t)(int32_t)sm_ld<L::kTop>(j) * 65536;
        double d = fixed_to_double<DT>(t.ebase, top, a1, a0);
        const uint2 f = sm_ld2<L::kFb>(j + (j - t.b0));
        if (f.x | f.y) {
          if (CLEAR) sm_st2<L::kFb>(j + (j - t.b0), 0u, 0u);
          if (DT == AGG_F32) d += (double)__uint_as_float(f.x) + (double)__uint_as_float(f.y);
          else d += __hiloint2double((int)f.y, (int)f.x);
        }
        g[r].sum = (unsigned long long)__double_as_longlong(d);
      } else {
        g[r].sum = (((unsigned long long)a1 << 32) | a0) + ((unsigned long long)(w >> 16) << 32) +
                   c * int_base<DT>(t.base);
      }
      if constexpr (MM) {
        g[r].nmn = 0;  // complement of the minimum's image, image of the maximum
        g[r].mx = 0;
        if (is_wide(DT)) {
          const ulonglong2 q = sm_ld2_64<L::kMM64>(t.b0 + 4 * (j - t.b0));
          if (CLEAR && (q.x | q.y)) sm_st2_64<L::kMM64>(t.b0 + 4 * (j - t.b0), 0ull, 0ull);
          g[r].nmn = q.x;
          g[r].mx = q.y;
        }
        if (DT != AGG_F64) {
          const uint2 q = sm_ld2<L::kMM>(j + (j - t.b0));
          if (CLEAR) sm_st2<L::kMM>(j + (j - t.b0), 0u, 0u);
          if (DT == AGG_I64) {
            if (q.x | q.y) {  // the window's pair took a row
              g[r].nmn = max(g[r].nmn, ~(t.base + (uint32_t)~q.x));
              g[r].mx = max(g[r].mx, t.base + q.y);
            }
          } else {
            g[r].nmn = ~g_img_of<DT>((typename SImg<DT>::U)(uint32_t)~q.x);
            g[r].mx = g_img_of<DT>((typename SImg<DT>::U)q.y);
          }
        }
      }
    }
    if (parts) g_merge<DT, MM, N>(a, g, parts);
  }
}

// Rows [0, a.n) of a column (SMEM: folded into the shared table t, else into
// the global table) by the block whose thread 0 is thread `first` of nthreads.
// VEC: 16-byte vector loads of 4 keys and 4 values per quad, QPI quads per
// thread per iteration (all loads issued before any row is folded): 4 or 8
// rows a thread per iteration, the autotuner's items-per-thread axis. WIDE
// (shared table): any number of rows, else at most kEpochRows.
// MULTI: up to kMaxWarpKeys frequent keys per warp and quad of rows get a
// reduced update (columns with a handful of keys or hot keys); without it
// every row takes the per-row path.
// Returns the number of rows this thread went through (the vector body's).
template <int DT, bool MM, bool SMEM, bool VEC, bool MULTI, int QPI, bool WIDE>
__device__ __forceinline__ uint32_t build_rows(const BuildArgs& a, const STab<DT, MM, WIDE>& t, int64_t first,
                                               int64_t nthreads) {
  using T = typename GV<DT>::T;
  const uint32_t* keys = a.keys;
  const T* vals = (const T*)a.vals;
  const int64_t tid = first + threadIdx.x;
  auto fold1 = [&](bool ok, int64_t i) {
    if (!ok) return;
    const uint32_t k1[1] = {keys[i]};
    const T v1[1] = {vals[i]};
    if constexpr (SMEM) {
      s_fold<DT, MM, 1, true>(a, t, k1, v1, 1u);
    } else {
      const GPart g[1] = {g_part_of<DT, MM>(k1[0], v1[0])};
      g_merge<DT, MM, 1>(a, g, 1u);
    }
  };
  auto fold4_global = [&](const uint32_t (&key)[4], const T (&val)[4], uint32_t rows) {
    GPart g[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) g[r] = g_part_of<DT, MM>(key[r], val[r]);
    g_merge<DT, MM, 4>(a, g, rows);
  };
  // iterations between two settlings of the cnt words (the head and tail rows are at most 6)
  const int per_epoch = (int)((kEpochRows - 6) / ((int64_t)blockDim.x * (VEC ? 4 * QPI : 1)));
  constexpr bool kEpochs = SMEM && WIDE;
  int it = 0;
  if (VEC) {
    using I = int;  // a column has fewer than 2^30 quads
    const I nq = (I)((a.n - a.head) / 4), step = (I)nthreads;  // full quads of rows
    const int64_t tail0 = a.head + (int64_t)nq * 4;
    fold1(tid < a.head, tid);
    fold1(tid < a.n - tail0, tail0 + tid);
    const uint4* kq = (const uint4*)(keys + a.head);
    const uint4* vq = (const uint4*)(vals + a.head);
    constexpr int VPQ = sizeof(T) == 4 ? 1 : 2;  // 16-byte value vectors per quad
    // All warps of the block take the same iterations (the settling has a
    // barrier) and all lanes of a warp every warp-wide operation; lanes past
    // the end have no rows.
    for (I qb = (I)first; qb < nq; qb += QPI * step) {
      const I q = qb + (I)threadIdx.x;
      uint4 kk[QPI], va[QPI], vb[QPI];
#pragma unroll
      for (int u = 0; u < QPI; ++u) {  // issue every load of the iteration first
        const I qu = q + u * step;
        const bool has = qu < nq;
        kk[u] = has ? ld_stream_v4(kq + qu) : make_uint4(0, 0, 0, 0);
        va[u] = has ? ld_stream_v4(vq + (int64_t)qu * VPQ) : make_uint4(0, 0, 0, 0);
        vb[u] = (has && VPQ == 2) ? ld_stream_v4(vq + (int64_t)qu * VPQ + 1) : va[u];
      }
#pragma unroll
      for (int u = 0; u < QPI; ++u) {
        const bool has = q + u * step < nq;
        const uint32_t key[4] = {kk[u].x, kk[u].y, kk[u].z, kk[u].w};
        T val[4];
        unpack4<T>(va[u], vb[u], val);
        if constexpr (MULTI) {
          // Frequent keys among the warp's 128 rows go through one reduced
          // update each: first the key of lane 0's first row; while a key had
          // at least kDominantRows rows, the next candidate is the first row of a
          // key not yet looked at. The remaining rows take the per-row path.
          uint32_t rem = has ? 0xFu : 0u;  // this lane's rows not yet folded, of keys not looked at
          uint32_t late = 0u;              // of them, those of a key looked at
          uint32_t k0 = __shfl_sync(0xffffffffu, key[0], 0);
#pragma unroll 1
          for (int w = 0; w < kMaxWarpKeys; ++w) {
            uint32_t take = 0;
#pragma unroll
            for (int r = 0; r < 4; ++r) take |= (((rem >> r) & 1u) && key[r] == k0) ? (1u << r) : 0u;
            const uint32_t n = __reduce_add_sync(0xffffffffu, (unsigned)__popc(take));
            if constexpr (SMEM && is_float(DT)) {
              // few rows outside the window (and not zero) take the per-row path; more
              // of them, and the key's rows are all summed as floats
              if (n < (uint32_t)kDominantOther) break;
              uint32_t in = take;
#pragma unroll
              for (int r = 0; r < 4; ++r) in &= s_enc<DT>(t, val[r]).ok || val[r] == T(0) ? 0xFu : ~(1u << r);
              if (__popc(__ballot_sync(0xffffffffu, take != in)) >= kDominantOther) {  // that many lanes
                s_fold_warp_other<DT, MM>(a, t, k0, val, take);
                rem &= ~take;
              } else {
                if (n < (uint32_t)kDominantRows) break;
                s_fold_warp_key<DT, MM>(a, t, k0, val, in);
                rem &= ~take;
                late |= take & ~in;
              }
            } else {
              if (n < (uint32_t)kDominantRows) break;
              if constexpr (SMEM) s_fold_warp_key<DT, MM>(a, t, k0, val, take);
              else g_fold_warp_key<DT, MM>(a, k0, val, take);
              rem &= ~take;
            }
            if (w + 1 == kMaxWarpKeys) break;
            const uint32_t lanes = __ballot_sync(0xffffffffu, rem != 0u);
            if (lanes == 0u) break;
            uint32_t next = key[3];  // this lane's first row of a key not yet looked at
            if (rem & 4u) next = key[2];
            if (rem & 2u) next = key[1];
            if (rem & 1u) next = key[0];
            k0 = __shfl_sync(0xffffffffu, next, __ffs(lanes) - 1);
          }
          rem |= late;
          if (rem != 0u) {
            if constexpr (SMEM) s_fold<DT, MM, 4, false>(a, t, key, val, rem);
            else fold4_global(key, val, rem);
          }
        } else if (has) {
          if constexpr (SMEM) s_fold<DT, MM, 4, true>(a, t, key, val, 0xFu);
          else fold4_global(key, val, 0xFu);
        }
      }
      ++it;
      if constexpr (kEpochs) {
        if (it % per_epoch == 0) {
          // a full table: the build is redone (one thread's reading, so the block leaves together)
          if (__syncthreads_or(threadIdx.x == 0 ? *(volatile int*)a.status : 0)) break;
          s_settle(t);
          __syncthreads();
        }
      } else if ((it & 15) == 0 &&
                 __shfl_sync(0xffffffffu, (threadIdx.x & 31) == 0 ? *(volatile int*)a.status : 0, 0)) {
        break;  // the whole warp leaves
      }
    }
    return (uint32_t)it * 4u * QPI;
  } else {
    for (int64_t b = first; b < a.n; b += nthreads) {
      fold1(b + threadIdx.x < a.n, b + threadIdx.x);
      ++it;
      if constexpr (kEpochs) {
        if (it % per_epoch == 0) {
          if (__syncthreads_or(threadIdx.x == 0 ? *(volatile int*)a.status : 0)) break;
          s_settle(t);
          __syncthreads();
        }
      } else if ((it & 63) == 0 && *(volatile int*)a.status) {
        break;
      }
    }
    return (uint32_t)it;
  }
}

// The build kernel of one query: grid-stride over all rows. 64 registers; one quad
// a turn spills nothing but 8 to 44 bytes for int64 and float64 MIN/MAX with
// frequent keys, two quads (on request) up to 164.
template <int DT, bool MM, bool SMEM, bool VEC, bool MULTI, int QPI = 1>
__global__ void __launch_bounds__(1024, 1) gb_build(BuildArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockCounts s_cnt;
  __shared__ Window s_win;
  if (threadIdx.x == 0) s_cnt = BlockCounts{0u, 0u};
  a.block_fails = &s_cnt.fails;
  STab<DT, MM, true> t;
  if (SMEM) {
    if (threadIdx.x < 32) s_window<DT>((const typename GV<DT>::T*)a.vals, a.n, &s_win);
    t.init(smem, a.smem_slots);
    t.clear();
  }
  __syncthreads();
  if (SMEM) t.set_window(s_win);
  const uint32_t seen = build_rows<DT, MM, SMEM, VEC, MULTI, QPI, true>(
      a, t, (int64_t)blockIdx.x * blockDim.x, (int64_t)gridDim.x * blockDim.x);
  atomicAdd(&s_cnt.seen, seen);
  if (SMEM) {
    __syncthreads();
    s_flush<DT, MM, true, false>(a, t);
  }
  __syncthreads();
  report_counts(a, s_cnt);
}

// Tile-queue build for hash-partitioned input: blocks pull tiles of up to
// 65532 rows in order from a counter, so all blocks work on neighbouring partitions and the
// table region they update stays in L2; each tile clears its shared table
// first and merges it into the global table at the end. With a tile list
// (rows partitioned chunk by chunk), tile t is the row range tiles[t] =
// (first row, rows), *ntiles of them, listed partition by partition. 64 registers;
// one quad a turn spills 24 to 68 bytes, 120 for float64 MIN/MAX, two quads (on
// request) 36 to 252.
constexpr int64_t kPartTileRows = int64_t(1) << 16;
// A tile never needs its cnt words settled.
constexpr int64_t kTileRowsMax = kEpochRows;
constexpr int kTileThreads = 512;  // at most: two blocks a SM of 64 registers a thread

template <int DT, bool MM, bool VEC, int QPI = 1>
__global__ void __launch_bounds__(kTileThreads, 2) gb_build_tiles(BuildArgs a, unsigned long long* next_tile,
                                                        int64_t tile_rows, const longlong2* tiles,
                                                        const unsigned long long* ntiles) {
  using T = typename GV<DT>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int64_t s_t;
  __shared__ BlockCounts s_cnt;
  __shared__ Window s_win;
  if (threadIdx.x == 0) s_cnt = BlockCounts{0u, 0u};
  a.block_fails = &s_cnt.fails;
  STab<DT, MM, false> t;
  t.init(smem, a.smem_slots);
  // one window for all of the block's tiles: their values come from one column
  // (with a tile list only the listed rows hold data: the first tile's)
  if (threadIdx.x < 32) {
    const longlong2 w = !tiles ? make_longlong2(0, a.n) : *ntiles ? tiles[0] : make_longlong2(0, 0);
    s_window<DT>((const T*)a.vals + w.x, w.y, &s_win);
  }
  t.clear();
  // The next tile's number is fetched while the current tile is folded. No new
  // tile once the table is full (the build is redone with a larger one).
  if (threadIdx.x == 0) s_t = *(volatile int*)a.status ? -1 : (int64_t)atomicAdd(next_tile, 1ull);
  __syncthreads();
  t.set_window(s_win);
  for (;;) {
    const int64_t tl = s_t;
    int64_t r0, rows;
    if (tiles) {
      if (tl < 0 || tl >= (int64_t)*ntiles) break;
      const longlong2 x = tiles[tl];
      r0 = x.x;
      rows = x.y;
    } else {
      r0 = tl * tile_rows;
      if (tl < 0 || r0 >= a.n) break;
      rows = min(tile_rows, a.n - r0);
    }
    BuildArgs b = a;
    b.keys = a.keys + r0;
    b.vals = (const T*)a.vals + r0;
    b.n = rows;
    b.head = min((int64_t)((-r0) & 3), rows);  // rows before the next 16-byte boundary of the keys
    int64_t next = 0;
    if (threadIdx.x == 0) next = *(volatile int*)a.status ? -1 : (int64_t)atomicAdd(next_tile, 1ull);
    atomicAdd(&s_cnt.seen, build_rows<DT, MM, true, VEC, true, QPI, false>(b, t, 0, blockDim.x));
    __syncthreads();
    if (threadIdx.x == 0) s_t = next;
    s_flush<DT, MM, false, true>(b, t);
    __syncthreads();
  }
  report_counts(a, s_cnt);
}

// ---------------------------------------------------------------------------
// Finalise.
// ---------------------------------------------------------------------------
struct OutArrays {
  uint32_t* keys;
  int64_t* count;
  unsigned long long* sum;
  unsigned long long* min;
  unsigned long long* max;
  double* avg;  // null: neither SUM nor AVG asked for
  int64_t* d;   // number of groups (device)
};

template <int DT, bool MM>
__device__ __forceinline__ void write_group(const OutArrays& o, int64_t i, uint32_t key, const GSlot<MM>& s) {
  const uint32_t c = s.cnt;
  o.keys[i] = key;
  o.count[i] = c;
  const unsigned long long sv = s.sum;
  o.sum[i] = sv;
  if (o.avg)
    o.avg[i] = average(DT == AGG_F32 || DT == AGG_F64 ? sv : float64_bits_of((long long)sv), c);
  if (MM) {
    const GSlot<true>& w = (const GSlot<true>&)s;
    const uint64_t mn = ~w.minc, mx = w.mx;
    if (DT == AGG_F32) {
      o.min[i] = (unsigned long long)__double_as_longlong((double)f32_of_img((uint32_t)mn));
      o.max[i] = (unsigned long long)__double_as_longlong((double)f32_of_img((uint32_t)mx));
    } else if (DT == AGG_F64) {
      o.min[i] = (unsigned long long)__double_as_longlong(f64_of_img(mn));
      o.max[i] = (unsigned long long)__double_as_longlong(f64_of_img(mx));
    } else {
      o.min[i] = (unsigned long long)i64_of_img(mn);
      o.max[i] = (unsigned long long)i64_of_img(mx);
    }
  }
}

template <bool MM>
__device__ __forceinline__ bool occupied(const GSlot<MM>* tab, uint32_t mask, int64_t j) {
  return j <= (int64_t)mask ? tab[j].key1 != 0 : tab[j].cnt != 0;
}

template <bool MM>
__device__ __forceinline__ uint32_t key_of(const GSlot<MM>* tab, uint32_t mask, int64_t j) {
  return j <= (int64_t)mask ? tab[j].key1 - 1 : 0xFFFFFFFFu;
}

// Small tables (at most kSmallSlots slots): one kernel. Every block loads the
// keys of all slots into shared memory (an empty slot as 0xFFFFFFFF, which no
// key exceeds) and writes each of its slots' groups at the key's rank, the
// number of smaller keys; keys are distinct, so the ranks are a permutation
// and the output is in ascending key order. Medium tables (at most kRankSlots
// slots) are compacted first and ranked among the d keys found: d^2 compares
// over the whole GPU cost less than the 20 launches of a radix sort (3000 keys
// in 8192 slots: 31 us with the compaction, 125 us sorted).
constexpr int kSmallSlots = 4097;
constexpr int kRankSlots = 32769;
constexpr int kRankThreads = 512;
constexpr int kRankSplit = 8;                         // threads counting one key's rank
constexpr int kRankKeys = kRankThreads / kRankSplit;  // keys ranked per block

// The number of sk[0 .. d) below key, sk padded with 0xFFFFFFFF to a multiple
// of 4; kRankSplit neighbouring lanes count every kRankSplit-th group of four
// and add their counts with shuffles.
__device__ __forceinline__ int rank_of(const uint32_t* sk, int d, uint32_t key, int part) {
  int rank = 0;
#pragma unroll 4
  for (int t = 4 * part; t < d; t += 4 * kRankSplit) {
    const uint4 q = *(const uint4*)&sk[t];
    rank += (q.x < key) + (q.y < key) + (q.z < key) + (q.w < key);
  }
#pragma unroll
  for (int m = 1; m < kRankSplit; m <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, m);
  return rank;
}

template <int DT, bool MM>
__global__ void __launch_bounds__(kRankThreads) gb_rank_small(const GSlot<MM>* tab, uint32_t mask, OutArrays o) {
  __shared__ __align__(16) uint32_t sk[kSmallSlots + 7];
  const int n = (int)mask + 1;  // main slots; the side slot's key exceeds all of theirs
  const bool side = tab[n].cnt != 0;
  int occ = 0;
  for (int t = threadIdx.x; t < ((n + 3) & ~3); t += kRankThreads) {
    const uint32_t k1 = t < n ? tab[t].key1 : 0u;
    sk[t] = k1 - 1;
    occ += k1 ? 1 : 0;
  }
  if (blockIdx.x == 0) {  // the number of groups
    const int c = __syncthreads_count(occ & 1) + 2 * __syncthreads_count(occ & 2 ? 1 : 0) +
                  4 * __syncthreads_count(occ & 4 ? 1 : 0) + 8 * __syncthreads_count(occ & 8 ? 1 : 0);
    if (threadIdx.x == 0) *o.d = c + (side ? 1 : 0);
  } else {
    __syncthreads();
  }
  const int i = blockIdx.x * kRankKeys + (int)threadIdx.x / kRankSplit;
  const int part = (int)threadIdx.x % kRankSplit;
  const bool have = i < n ? sk[i] != 0xFFFFFFFFu : i == n && side;
  const uint32_t key = i < n ? sk[i] : 0xFFFFFFFFu;
  const int rank = rank_of(sk, n, key, part);
  if (have && part == 0) write_group<DT, MM>(o, rank, key, tab[i]);
}

template <int DT, bool MM>
__global__ void __launch_bounds__(kRankThreads) gb_rank_gather(const GSlot<MM>* tab, const uint32_t* ckeys,
                                                               const uint32_t* cslot, OutArrays o) {
  extern __shared__ __align__(16) uint32_t sk[];
  const int d = (int)*(const unsigned long long*)o.d;
  if (blockIdx.x * kRankKeys >= d) return;
  for (int t = threadIdx.x; t < ((d + 3) & ~3); t += kRankThreads) sk[t] = t < d ? ckeys[t] : 0xFFFFFFFFu;
  __syncthreads();
  const int i = blockIdx.x * kRankKeys + (int)threadIdx.x / kRankSplit;
  const int part = (int)threadIdx.x % kRankSplit;
  const uint32_t key = i < d ? sk[i] : 0u;
  const int rank = rank_of(sk, d, key, part);
  if (i < d && part == 0) write_group<DT, MM>(o, rank, key, tab[cslot[i]]);
}

// Large tables: compact occupied slots into (key, slot) pairs.
// PER slots per thread per run of the compaction (1 for small tables, whose
// few slots are best spread over all threads; 8 for large ones, all loaded
// before the first is looked at: 33 M slots of 16 bytes 197 us one by one, 100
// us so, 5.4 TB/s).
template <bool MM, int kCompactPer = 8>
__global__ void gb_compact(const GSlot<MM>* tab, uint32_t mask, uint32_t* okeys, uint32_t* oslot,
                           unsigned long long* counter) {
  // each block takes runs of kCompactPer * blockDim.x slots and reserves its
  // output range with one atomic per run (order within a run: warp, then lane)
  __shared__ uint32_t s_warp[32];
  __shared__ unsigned long long s_base;
  const int64_t nslots = (int64_t)mask + 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const int64_t span = (int64_t)kCompactPer * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * span; base < nslots; base += (int64_t)gridDim.x * span) {
    uint32_t k1[kCompactPer];  // key + 1; of the last slot, the key 2^32 - 1, the count; 0: empty
    uint32_t b[kCompactPer];
    uint32_t wtot = 0;
#pragma unroll
    for (int i = 0; i < kCompactPer; ++i) {  // all loads before the first use
      const int64_t j = base + (int64_t)i * blockDim.x + threadIdx.x;
      k1[i] = j < nslots ? *(j <= (int64_t)mask ? &tab[j].key1 : &tab[j].cnt) : 0u;
    }
#pragma unroll
    for (int i = 0; i < kCompactPer; ++i) {
      b[i] = __ballot_sync(0xffffffffu, k1[i] != 0);
      wtot += __popc(b[i]);
    }
    if (lane == 0) s_warp[warp] = wtot;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t t = 0;
      for (int w = 0; w < nw; ++w) {
        const uint32_t c = s_warp[w];
        s_warp[w] = t;
        t += c;
      }
      s_base = t ? atomicAdd(counter, (unsigned long long)t) : 0ull;
    }
    __syncthreads();
    unsigned long long pos = s_base + s_warp[warp];
#pragma unroll
    for (int i = 0; i < kCompactPer; ++i) {
      if (k1[i] != 0) {
        const int64_t j = base + (int64_t)i * blockDim.x + threadIdx.x;
        const unsigned long long p = pos + __popc(b[i] & lt);
        okeys[p] = j <= (int64_t)mask ? k1[i] - 1 : 0xFFFFFFFFu;
        oslot[p] = (uint32_t)j;
      }
      pos += __popc(b[i]);
    }
    __syncthreads();  // s_warp and s_base are rewritten by the next run
  }
}

// A slot per thread and turn is bound by the latency of one random access:
// 502 us for 14 M groups of 16 bytes, 371 us with kGatherSlots in flight a
// thread, each read whole (1.0 GB of rows written and sectors read: 2.8 TB/s).
constexpr int kGatherThreads = 256;
constexpr int kGatherSlots = 4;
template <int DT, bool MM>
__global__ void __launch_bounds__(kGatherThreads) gb_gather(const GSlot<MM>* __restrict__ tab,
                                                            const uint32_t* __restrict__ skeys,
                                                            const uint32_t* __restrict__ sslot, OutArrays o,
                                                            int64_t cap) {
  const int64_t d = min((int64_t)*(const unsigned long long*)o.d, cap);
  constexpr int64_t kTurn = kGatherThreads * kGatherSlots;
  for (int64_t base = (int64_t)blockIdx.x * kTurn; base < d; base += (int64_t)gridDim.x * kTurn) {
    uint32_t key[kGatherSlots], slot[kGatherSlots];
    GSlot<MM> g[kGatherSlots];
#pragma unroll
    for (int u = 0; u < kGatherSlots; ++u) {
      const int64_t i = base + u * kGatherThreads + threadIdx.x;
      key[u] = i < d ? skeys[i] : 0u;
      slot[u] = i < d ? sslot[i] : 0u;
    }
#pragma unroll
    for (int u = 0; u < kGatherSlots; ++u) {  // slot 0 exists: its row is dropped below
      const uint4* q = (const uint4*)&tab[slot[u]];
#pragma unroll
      for (int h = 0; h < (int)(sizeof(GSlot<MM>) / 16); ++h) ((uint4*)&g[u])[h] = __ldg(q + h);
    }
#pragma unroll
    for (int u = 0; u < kGatherSlots; ++u) {
      const int64_t i = base + u * kGatherThreads + threadIdx.x;
      if (i < d) write_group<DT, MM>(o, i, key[u], g[u]);
    }
  }
}


}  // namespace agg
