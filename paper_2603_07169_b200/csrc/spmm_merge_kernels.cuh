// nnz-balanced CSR SpMM: Y = alpha * A * B + beta * Y, B (n x k) and Y (m x k) row-major
// (paper, Appendix C, Table 6, task 13, with alpha/beta).
//
// The work list is the merge of the m row-end markers with the nnz nonzeros, cut into equal shares of `witems` items per WARP,
// whatever rows they belong to: neither long rows nor empty ones unbalance it, and Y of the empty rows is written by the same
// pass.  A warp walks its nonzeros one after another with all 32 lanes along k, so the end of a row is one warp-uniform branch
// and no sum is ever combined across lanes.
#pragma once
#include "common.cuh"

namespace b200sp {

__device__ __forceinline__ float bf16_lo(unsigned w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(unsigned w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ unsigned bf16_pair(float a, float b) {
  return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(a)) | ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}

// V consecutive stored values as one load / store, converted to FP32 only when consumed.
template <typename T, int V> struct Piece;
template <> struct Piece<float, 1> {
  typedef float raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[1]) { o[0] = b; }
  static __device__ __forceinline__ raw pack(const float (&o)[1]) { return o[0]; }
};
template <> struct Piece<float, 2> {
  typedef float2 raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[2]) { o[0] = b.x; o[1] = b.y; }
  static __device__ __forceinline__ raw pack(const float (&o)[2]) { return make_float2(o[0], o[1]); }
};
template <> struct Piece<float, 4> {
  typedef float4 raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[4]) { o[0] = b.x; o[1] = b.y; o[2] = b.z; o[3] = b.w; }
  static __device__ __forceinline__ raw pack(const float (&o)[4]) { return make_float4(o[0], o[1], o[2], o[3]); }
};
template <> struct Piece<bf16_t, 1> {
  typedef bf16_t raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[1]) { o[0] = to_f32(b); }
  static __device__ __forceinline__ raw pack(const float (&o)[1]) { return __bfloat16_as_ushort(__float2bfloat16_rn(o[0])); }
};
template <> struct Piece<bf16_t, 2> {
  typedef unsigned raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[2]) { o[0] = bf16_lo(b); o[1] = bf16_hi(b); }
  static __device__ __forceinline__ raw pack(const float (&o)[2]) { return bf16_pair(o[0], o[1]); }
};
template <> struct Piece<bf16_t, 4> {
  typedef uint2 raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[4]) { o[0] = bf16_lo(b.x); o[1] = bf16_hi(b.x); o[2] = bf16_lo(b.y); o[3] = bf16_hi(b.y); }
  static __device__ __forceinline__ raw pack(const float (&o)[4]) { return make_uint2(bf16_pair(o[0], o[1]), bf16_pair(o[2], o[3])); }
};
template <> struct Piece<bf16_t, 8> {
  typedef uint4 raw;
  static __device__ __forceinline__ void widen(raw b, float (&o)[8]) {
    o[0] = bf16_lo(b.x); o[1] = bf16_hi(b.x); o[2] = bf16_lo(b.y); o[3] = bf16_hi(b.y);
    o[4] = bf16_lo(b.z); o[5] = bf16_hi(b.z); o[6] = bf16_lo(b.w); o[7] = bf16_hi(b.w);
  }
  static __device__ __forceinline__ raw pack(const float (&o)[8]) {
    return make_uint4(bf16_pair(o[0], o[1]), bf16_pair(o[2], o[3]), bf16_pair(o[4], o[5]), bf16_pair(o[6], o[7]));
  }
};

// acc += v * b.  BF16 pairs by the mixed-precision FMA of sm_100 (BF16 factors, FP32 addend and result, one rounding; v is a widened BF16
// value): the same value as fmaf on the widened factors without the widening (100 columns of 2^18 rows of 32: 198 -> 173 us).
__device__ __forceinline__ void mixed_fma(unsigned w, float v, float& a0, float& a1) {
  asm("{ .reg .b16 lo, hi;\n\t"
      "mov.b32 {lo, hi}, %3;\n\t"
      "fma.rn.f32.bf16 %0, %2, lo, %0;\n\t"
      "fma.rn.f32.bf16 %1, %2, hi, %1; }"
      : "+f"(a0), "+f"(a1) : "h"((unsigned short)(__float_as_uint(v) >> 16)), "r"(w));
}
template <typename T, int V>
__device__ __forceinline__ void piece_fma(const typename Piece<T, V>::raw& b, float v, float (&acc)[V]) {
  if constexpr (sizeof(T) == 2 && V == 2) {
    mixed_fma(b, v, acc[0], acc[1]);
  } else if constexpr (sizeof(T) == 2 && V == 4) {
    mixed_fma(b.x, v, acc[0], acc[1]);
    mixed_fma(b.y, v, acc[2], acc[3]);
  } else if constexpr (sizeof(T) == 2 && V == 8) {
    mixed_fma(b.x, v, acc[0], acc[1]);
    mixed_fma(b.y, v, acc[2], acc[3]);
    mixed_fma(b.z, v, acc[4], acc[5]);
    mixed_fma(b.w, v, acc[6], acc[7]);
  } else {
    float w[V];
    Piece<T, V>::widen(b, w);
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] = fmaf(v, w[i], acc[i]);
  }
}

template <typename T, int V>
__device__ __forceinline__ void piece_store(T* yp, const float (&acc)[V], float alpha, float beta) {
  typedef typename Piece<T, V>::raw raw;
  float out[V];
#pragma unroll
  for (int j = 0; j < V; ++j) out[j] = alpha * acc[j];
  if (beta != 0.0f) {
    float old[V];
    Piece<T, V>::widen(*(const raw*)yp, old);
#pragma unroll
    for (int j = 0; j < V; ++j) out[j] += beta * old[j];
  }
  *(raw*)yp = Piece<T, V>::pack(out);
}

// The same with Y's old values already here.
template <typename T, int V>
__device__ __forceinline__ void piece_store(T* yp, const float (&acc)[V], float alpha, float beta, const typename Piece<T, V>::raw& old) {
  float out[V];
  Piece<T, V>::widen(old, out);
#pragma unroll
  for (int j = 0; j < V; ++j) out[j] = alpha * acc[j] + beta * out[j];
  *(typename Piece<T, V>::raw*)yp = Piece<T, V>::pack(out);
}

// N consecutive words of shared memory (N 2, 4 or 8; aligned to 4 N or 16 bytes) with vector loads
template <int N, typename W>
__device__ __forceinline__ void lds_group(const W* p, W (&o)[N]) {
  if constexpr (N >= 4) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const int4 t = *(const int4*)(p + i);
      o[i] = *(const W*)&t.x; o[i + 1] = *(const W*)&t.y; o[i + 2] = *(const W*)&t.z; o[i + 3] = *(const W*)&t.w;
    }
  } else {
    const int2 t = *(const int2*)p;
    o[0] = *(const W*)&t.x; o[1] = *(const W*)&t.y;
  }
}

// A value that is the same in all lanes, made known as such: branches on it need no reconvergence code.
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xFFFFFFFFu, v, 0); }

// 4-byte asynchronous copy global -> shared of which the first `bytes` (2 or 4) are read and the rest is zero
__device__ __forceinline__ void cp_async4(void* dst, const void* src, int bytes = 4) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int kMergeWarps = 8;       // warps per CTA of spmm_merge_kernel
constexpr int kMergeWarpItems = 128; // most merge items per share
constexpr int kMergeShares = 4;      // most consecutive shares per warp

// Nonzeros whose loads of B (J each) are in flight per warp: 8 loads, 16 where a nonzero takes four of them (100,000 uneven rows, k = 127
// FP32: 84 us against 89 us with 8; with one or two loads per nonzero 16 in flight are slower).
template <int V, int J>
constexpr int kMergeUnroll = J >= 4 ? (V >= 4 ? 2 : 4) : 8 / J;

// Resident CTAs per SM that the registers are capped for, by the registers the loads in flight and the sums take: warps resident, not
// loads per warp, hide the latency (R-MAT 2^22, k = 64 FP32: 828 us with 6 CTAs, 854 us with 5), as long as little spills.  (Two or four
// nonzeros per step on half or quarter warps, 16 bytes per lane, measured 905 us: the sums of the halves at every row end cost more.)
template <typename T, int V, int J>
constexpr int merge_ctas() {
  constexpr int need = kMergeUnroll<V, J> * J * ((V * (int)sizeof(T) + 3) / 4) + 2 * V * J;
  return need <= 20 ? 6 : need <= 24 ? 5 : need <= 40 ? 4 : 3;
}

// Forms whose registers are full without Y's old values asked for ahead (bytes spilled, and us on 150,000 uneven rows of 11, without / with them):
// four loads of one column (FP32 0 / 68 bytes, k = 127 187 / 248 us; BF16 42 / 86 bytes, 168 / 218 us) and two of eight BF16 columns
// (52 / 300 bytes, k = 264 190 / 306 us, k = 512 285 / 410 us).  Where two loads of one or two BF16 columns spill some 40 bytes for them the wait
// saved is still worth more (k = 63 83.5 / 80.1 us, k = 66 86.5 / 83.8 us).
template <typename T, int V, int J>
constexpr bool kMergeNoRoom = (V == 1 && J == 4) || (sizeof(T) == 2 && V == 8 && J == 2);

// What a warp keeps in shared memory of one share: its columns, its values and the ends of its rows, and room to read a group ahead.
template <typename T> struct MergeStage;
template <> struct MergeStage<float> {
  int col[kMergeWarpItems + 8];
  float val[kMergeWarpItems + 8];
  int end[kMergeWarpItems + 4];
};
template <> struct MergeStage<bf16_t> {
  int col[kMergeWarpItems + 8];
  unsigned raw[kMergeWarpItems / 2 + 4];      // the 4-byte words that hold the values, as stored
  int end[kMergeWarpItems + 4];
};

// A warp takes `shares` consecutive shares; the (col, val) pairs and row ends of the next one arrive in shared memory (cp.async)
// while it walks the current one.  Lane l holds columns slice * 32 * V * J + 32 * V * j + l * V + (0 .. V-1), j < J, of the current
// row in FP32 registers (acc: products of the current share; tot: of the row's earlier shares); U nonzeros, U J loads of B, are
// in flight.  A warp leaves two partial sums in shared memory: `head` for a first row that began before its shares, `carry` for
// the row it leaves unfinished; after one barrier the warp that holds a row's end adds the carries of the warps before it in
// order, and what crosses the CTA's own ends goes to tile_tail / tile_carry and is finished by spmm_merge_fixup_kernel.  No
// chain is longer than kMergeWarpItems products + kMergeShares + kMergeWarps partial sums + the tiles' terms.
// split[i]: row ends before item i * witems.
// MODE 0: beta == 0.  1: beta != 0; Y's old values of a row are asked for when the row before it ends, not when it ends itself (50,000 uneven
// rows of 11, k = 128 FP32: 37.1 -> 34.0 us; 30,000 of 12, k = 256 48.8 -> 41.8 us; two rows ahead, in a second set of registers: 41.2 us for the
// former).  Not in kMergeNoRoom's forms, which have no registers left for them.
// 2: beta != 0 and empty rows, which are listed apart (see below); the listing costs 2-5 % where there are none, and old values asked for
// ahead cost it more than they save (R-MAT 2^20, k = 64 FP32 303 / 442 us).
// none: what mode 2 multiplies the old values of an empty row by.
template <typename T, int V, int J, int MODE>
__global__ void __launch_bounds__(kMergeWarps * 32, (merge_ctas<T, V, J>()))
spmm_merge_kernel(int m, int nnz, int k, int tiles, int witems, int shares, const int* __restrict__ split, const int* __restrict__ row_ptr,
                  const int* __restrict__ col_idx, const T* __restrict__ vals, const T* __restrict__ B, T* __restrict__ Y,
                  float* __restrict__ tile_carry, float* __restrict__ tile_tail, int2* __restrict__ tile_row, float alpha, float beta, float none) {
  constexpr int U = kMergeUnroll<V, J>, KS = 32 * V * J;
  constexpr bool LIST = MODE == 2, AHEAD = MODE == 1 && !kMergeNoRoom<T, V, J>;
  typedef typename Piece<T, V>::raw raw;
  __shared__ __align__(16) MergeStage<T> stage_s[kMergeWarps][2];
  __shared__ __align__(16) float wide_s[sizeof(T) == 2 ? kMergeWarps : 1][sizeof(T) == 2 ? kMergeWarpItems + 8 : 4];   // BF16: the current share's values widened
  __shared__ unsigned char empty_s[LIST ? kMergeWarps : 1][LIST ? kMergeWarpItems : 4];
  __shared__ float head_s[kMergeWarps][KS];
  __shared__ int first_s[2];                                 // the tile's first row and where it starts, -1 when inside the tile
  static_assert(sizeof(stage_s[0]) >= KS * sizeof(float), "a warp's carry takes the place of its stages");
  auto carry_s = [&](int w) { return reinterpret_cast<float*>(&stage_s[w][0]); };
  grid_dependency_wait();
  const int slice = blockIdx.x / tiles, t = blockIdx.x - slice * tiles;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const long long total = (long long)m + nnz;
  const int last = (int)((total + witems - 1) / witems);
  const int s0 = (int)min(((long long)t * kMergeWarps + warp) * shares, (long long)last), s1 = min(s0 + shares, last);
  const int r_first = uniform(__ldg(split + s0));
  int r_lo = r_first, r_hi = uniform(__ldg(split + min(s0 + 1, last)));
  const int start0 = uniform(__ldg(row_ptr + r_first));      // start of the first row (nnz when there is none)
  const int p_first = (int)(min((long long)s0 * witems, total) - r_first);
  bool head = start0 < p_first;                              // the current row began before this warp's shares

  // copies of share s (rows r0 .. r1 end in it) into stage st
  auto fetch = [&](int s, int r0, int r1, MergeStage<T>& st) {
    const int p0 = (int)((long long)s * witems - r0), cnt = (int)(min((long long)(s + 1) * witems, total) - r1) - p0, rows = r1 - r0;
#pragma unroll
    for (int i = 0; i < kMergeWarpItems; i += 32) {
      if (i + lane < cnt) {
        cp_async4(&st.col[i + lane], col_idx + p0 + i + lane);
        if constexpr (sizeof(T) == 4) cp_async4(&st.val[i + lane], vals + p0 + i + lane);
      }
      if (i + lane < rows) cp_async4(&st.end[i + lane], row_ptr + r0 + 1 + i + lane);
    }
    if constexpr (sizeof(T) == 2) {
      const int w0 = p0 & ~1, words = (p0 + cnt - w0 + 1) >> 1;
#pragma unroll
      for (int i = 0; i < kMergeWarpItems / 2 + 32; i += 32)
        if (i + lane < words) cp_async4(&st.raw[i + lane], vals + w0 + 2 * (i + lane), min(4, 2 * (nnz - w0 - 2 * (i + lane))));
    }
    if (lane < U) st.col[cnt + lane] = 0;                    // read ahead of the end, never multiplied
    if (!LIST && lane == 0) st.end[rows] = (int)((unsigned)p0 + 0x100000u);   // no end inside this share
  };

  const int col0 = slice * KS + lane * V;
  bool on[J];
  float acc[J][V], tot[J][V];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    on[j] = col0 + 32 * V * j < k;
#pragma unroll
    for (int i = 0; i < V; ++i) { acc[j][i] = 0.0f; tot[j][i] = 0.0f; }
  }
  const char* const Bc = (const char*)(B + col0);
  const int row_bytes = k * (int)sizeof(T);
  T* yrow = Y + (long long)r_first * k + col0;
  int begin = start0;                                        // start of the current row
  raw old[AHEAD ? J : 1];                                    // Y's old values of the current row
  auto ask_old = [&]() {
#pragma unroll
    for (int j = 0; j < (AHEAD ? J : 0); ++j) if (on[j]) old[j] = *(const raw*)(yrow + 32 * V * j);
  };
  if (AHEAD && r_first < m) ask_old();
  // rows empty_s[warp][0 .. count) of the share whose first row is at ys: y = none * y over the slice's columns
  auto scale_rows = [&](T* ys, int count) {
    const int width = min(KS, k - slice * KS);
    const bool wide = V * sizeof(T) < 16 && k * (int)sizeof(T) % 16 == 0;       // 16 bytes a lane where the rows allow it
    const int per = wide ? 16 / (int)sizeof(T) : V;
    int lanes = 32;                                          // lanes to a row: a power of two
    while (lanes > 1 && (lanes / 2) * per >= width) lanes /= 2;
    const int sub = lane / lanes, step = 32 / lanes;
    for (int c = (lane & (lanes - 1)) * per; c < width; c += lanes * per) {
      T* const yc = ys + slice * KS + c;
#pragma unroll 4
      for (int i = sub; i < count; i += step) {
        T* const y = yc + (long long)empty_s[warp][i] * k;
        if (wide) {
          float zero[16 / sizeof(T)];
#pragma unroll
          for (int x = 0; x < 16 / (int)sizeof(T); ++x) zero[x] = 0.0f;
          piece_store<T, 16 / (int)sizeof(T)>(y, zero, 0.0f, none);
        } else {
          float zero[V];
#pragma unroll
          for (int x = 0; x < V; ++x) zero[x] = 0.0f;
          piece_store<T, V>(y, zero, 0.0f, none);
        }
      }
    }
  };

  if (s0 < s1) fetch(s0, r_lo, r_hi, stage_s[warp][0]);
  cp_async_commit();
  int r_next = uniform(__ldg(split + min(s0 + 2, last)));
  for (int s = s0; s < s1; ++s) {
    const int cur = (s - s0) & 1;
    if (s + 1 < s1) fetch(s + 1, r_hi, r_next, stage_s[warp][cur ^ 1]);
    cp_async_commit();
    const int r_after = __ldg(split + min(s + 3, last));
    cp_async_wait<1>();
    __syncwarp();
    MergeStage<T>& st = stage_s[warp][cur];
    const int p0 = (int)((long long)s * witems - r_lo), cnt = (int)(min((long long)(s + 1) * witems, total) - r_hi) - p0, rows = r_hi - r_lo;
    const float* vls;
    if constexpr (sizeof(T) == 2) {
      const bf16_t* const raw_v = (const bf16_t*)st.raw + (p0 & 1);
#pragma unroll
      for (int i = 0; i < kMergeWarpItems; i += 32) if (i + lane < cnt) wide_s[warp][i + lane] = to_f32(raw_v[i + lane]);
      __syncwarp();
      vls = wide_s[warp];
    } else {
      vls = st.val;
    }
    int listed = rows, empties = 0;
    if constexpr (LIST) {
      listed = 0;
      // The rows of the share that have nonzeros, in order, written over the ends: (number among the share's rows) << 8 | (nonzero before
      // which it ends).  The others are listed apart and scaled (set to zero) at once, as many lanes to a row as it has pieces and several
      // rows in flight: one by one between the others, each would cost the walk a wait for its old values.
      for (int i0 = 0; i0 < rows; i0 += 32) {
        const int i = i0 + lane;
        const int e = i < rows ? st.end[i] : 0;
        int before = __shfl_up_sync(0xFFFFFFFFu, e, 1);
        if (lane == 0) before = begin;
        begin = __shfl_sync(0xFFFFFFFFu, e, min(31, rows - 1 - i0));
        const bool full = i < rows && e != before, empty = i < rows && e == before;
        const unsigned fulls = __ballot_sync(0xFFFFFFFFu, full), empty_rows = __ballot_sync(0xFFFFFFFFu, empty), below = (1u << lane) - 1u;
        if (full) st.end[listed + __popc(fulls & below)] = (i << 8) | (e - p0);     // (behind what has been read: the list is never ahead of i)
        if (empty) empty_s[warp][empties + __popc(empty_rows & below)] = (unsigned char)i;
        listed += __popc(fulls);
        empties += __popc(empty_rows);
        __syncwarp();
      }
      if (lane == 0) st.end[listed] = 0xFF;                    // no end inside this share
      __syncwarp();
    }
    T* const ys = LIST ? Y + (long long)r_lo * k : nullptr;
    if constexpr (LIST) { if (empties > 0) scale_rows(ys, empties); }
    // the current row ends before nonzero `end` of the share
    auto share_end = [&](int j) { return LIST ? uniform(st.end[j]) : (int)((unsigned)uniform(st.end[j]) - (unsigned)p0); };
    int j_row = 0, row = share_end(0), end = LIST ? row & 0xFF : row;
    // the current row has been added up to its end: stored, or left as the warp's head when it began earlier
    auto finish_row = [&]() {
#pragma unroll
      for (int j = 0; j < J; ++j)
#pragma unroll
        for (int i = 0; i < V; ++i) { acc[j][i] += tot[j][i]; tot[j][i] = 0.0f; }
      if (head) {
        head = false;
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
          for (int i = 0; i < V; ++i) head_s[warp][32 * V * j + lane * V + i] = acc[j][i];
      } else {
        T* const yp = LIST ? ys + (long long)(row >> 8) * k + col0 : yrow;
#pragma unroll
        for (int j = 0; j < J; ++j)
          if (on[j]) {
            if constexpr (AHEAD) piece_store<T, V>(yp + 32 * V * j, acc[j], alpha, beta, old[j]);
            else piece_store<T, V>(yp + 32 * V * j, acc[j], alpha, MODE ? beta : 0.0f);
          }
      }
#pragma unroll
      for (int j = 0; j < J; ++j)
#pragma unroll
        for (int i = 0; i < V; ++i) acc[j][i] = 0.0f;
      row = share_end(++j_row);
      end = LIST ? row & 0xFF : row;
      if constexpr (!LIST) yrow += k;
      if (AHEAD && r_lo + j_row < m) ask_old();
    };
    for (int q = 0; q < cnt; q += U) {
      int c[U];
      float v[U];
      raw b[U][J];
      lds_group<U>(st.col + q, c);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int j = 0; j < J; ++j) if (on[j]) b[u][j] = __ldg((const raw*)(Bc + (long long)c[u] * row_bytes) + 32 * j);
      lds_group<U>(vls + q, v);
      if (q + U > cnt) {                                     // the last, partly filled group: (0, 0) instead of what was read ahead
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (q + u >= cnt) {
            v[u] = 0.0f;
#pragma unroll
            for (int j = 0; j < J; ++j) b[u][j] = raw();
          }
      }
      if (end >= q + U) {                                    // no row ends inside this group
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int j = 0; j < J; ++j) piece_fma<T, V>(b[u][j], v[u], acc[j]);
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if constexpr (LIST) { if (end == q + u) finish_row(); }
          else while (end == q + u) finish_row();
#pragma unroll
          for (int j = 0; j < J; ++j) piece_fma<T, V>(b[u][j], v[u], acc[j]);
        }
      }
    }
    while (j_row < listed) finish_row();                     // the row (rows) that end with the share
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
      for (int i = 0; i < V; ++i) { tot[j][i] += acc[j][i]; acc[j][i] = 0.0f; }
    __syncwarp();                                            // every lane is done with the stage: the next copies may land in it
    r_lo = r_hi; r_hi = r_next; r_next = uniform(r_after);
  }
#pragma unroll
  for (int j = 0; j < J; ++j)
#pragma unroll
    for (int i = 0; i < V; ++i) carry_s(warp)[32 * V * j + lane * V + i] = tot[j][i];   // zero when the shares end with a row
  if (warp == 0 && lane == 0) { first_s[0] = r_first; first_s[1] = start0 < p_first ? start0 : -1; }
  __syncthreads();

  // (r_lo is now the number of row ends before this warp's end)
  // Merge items are counted in 32 bits (m + nnz < 2^32): three divisions in 64 bits would be calls, and spills in the loop above.
  const unsigned region = (unsigned)(witems * shares);
  const long long slot = ((long long)slice * tiles + t) * KS;
  if (start0 < p_first && r_lo > r_first) {                  // complete the row that ends here: the carries before it, in order, then the head
    const int ws = (int)(((unsigned)start0 + (unsigned)r_first) / region) - t * kMergeWarps;   // the warp that holds the row's start
#pragma unroll
    for (int j = 0; j < J; ++j) {
      float s[V];
#pragma unroll
      for (int i = 0; i < V; ++i) s[i] = 0.0f;
      for (int w = ws > 0 ? ws : 0; w < warp; ++w)
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] += carry_s(w)[32 * V * j + lane * V + i];
#pragma unroll
      for (int i = 0; i < V; ++i) s[i] += head_s[warp][32 * V * j + lane * V + i];
      if (ws >= 0) { if (on[j]) piece_store<T, V>(Y + (long long)r_first * k + col0 + 32 * V * j, s, alpha, beta); }
      else {
#pragma unroll
        for (int i = 0; i < V; ++i) tile_tail[slot + 32 * V * j + lane * V + i] = s[i];
      }
    }
  }
  if (warp == kMergeWarps - 1) {                             // what the tile leaves unfinished
    if (slice == 0 && lane == 0) {                           // and for the fix-up: the row that it completes for earlier tiles, and the first of them
      const int r = first_s[0], rs = first_s[1];
      tile_row[t] = rs >= 0 && r_lo > r ? make_int2(r, (int)(((unsigned)rs + (unsigned)r) / (region * kMergeWarps))) : make_int2(-1, 0);
    }
    int ws = kMergeWarps;
    if (r_lo < m) ws = (int)(((unsigned)__ldg(row_ptr + r_lo) + (unsigned)r_lo) / region) - t * kMergeWarps;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      float s[V];
#pragma unroll
      for (int i = 0; i < V; ++i) s[i] = 0.0f;
      for (int w = ws > 0 ? ws : 0; w < kMergeWarps; ++w)
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] += carry_s(w)[32 * V * j + lane * V + i];
#pragma unroll
      for (int i = 0; i < V; ++i) tile_carry[slot + 32 * V * j + lane * V + i] = s[i];
    }
  }
}

// Finishes the rows that a tile boundary of spmm_merge_kernel cut: the row's value is tile_carry[first .. t-1] + tile_tail[t], the carries
// added in trees of 16 whose sums form a chain; `lanes` threads per (slice, tile), fixed order.  Latency-bound: which row and from which
// tile on comes from the tile itself (tile_row), so that only one load stands before those of the partial sums.
template <typename T>
__global__ void __launch_bounds__(256)
spmm_merge_fixup_kernel(int k, int tiles, int slices, int ks, int lanes, const int2* __restrict__ tile_row, const float* __restrict__ tile_carry,
                        const float* __restrict__ tile_tail, T* __restrict__ Y, float alpha, float beta) {
  grid_dependency_wait();
  const long long id = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / lanes;
  const int lane = threadIdx.x & (lanes - 1);
  if (id >= (long long)slices * tiles) return;
  const int slice = (int)(id / tiles), t = (int)(id - (long long)slice * tiles);
  const int2 row = __ldg(tile_row + t);
  if (row.x < 0) return;                                     // no row that began in an earlier tile ends in this one
  for (int c = lane; c < ks && slice * ks + c < k; c += lanes) {
    const float* const cp = tile_carry + (long long)slice * tiles * ks + c;
    const float tail = tile_tail[((long long)slice * tiles + t) * ks + c];
    float acc = 0.0f;
    for (int u = row.y; u < t; u += 16) {
      float part[16];
#pragma unroll
      for (int v = 0; v < 16; ++v) part[v] = u + v < t ? cp[(long long)(u + v) * ks] : 0.0f;
#pragma unroll
      for (int w = 8; w > 0; w >>= 1)
#pragma unroll
        for (int v = 0; v < w; ++v) part[v] += part[v + w];
      acc += part[0];
    }
    epilogue_store(Y, (long long)row.x * k + slice * ks + c, acc + tail, alpha, beta);
  }
}

}  // namespace b200sp
