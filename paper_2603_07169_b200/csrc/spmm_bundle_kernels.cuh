// nnz-balanced CSR SpMM for narrow rows of B: rows of about equal length side by side in a warp.
// Y = alpha * A * B + beta * Y, B (n x k) and Y (m x k) row-major (paper, Appendix C, Table 6, task 13, with alpha/beta).
//
// The list of row ends and nonzeros is cut into equal regions per WARP, as for spmm_merge_kernel.  There a warp takes one nonzero at a time with all
// lanes along k, so a row of B of 128 bytes is 32 loads of 4 bytes, and what L1 takes per load instruction (about 4 cycles, and 1.5 per line) bounds
// it.  Here LANES lanes of 16 bytes hold a row of B and a warp takes G = 32 / LANES rows of A at a time.  It sorts the pieces of rows in its
// region by length (32 at a time, in registers) and walks G of about the same length side by side, so that the ends of G rows are one step and the
// columns and values of four nonzeros of each cost four loads of shared memory.  Pieces longer than kBundleLong are walked by all groups together.
// Bound by latency in calls of a wave or two, else by the wait for lines of B and by L1's data pipe, which a line keeps for two cycles (R-MAT 2^20, k = 64 BF16: 57 %
// busy, 9 warp instructions a nonzero instead of 15; 162 us by spmm_merge_kernel, 106 us).
#pragma once
#include "spmm_merge_kernels.cuh"

namespace b200sp {

constexpr int kBundleLong = 32;      // longer pieces of rows are split over the lane groups
// Resident CTAs per SM: 4 loads of 16 bytes per lane in flight, and more warps rather than more loads (R-MAT 2^22, k = 64 FP32: 968 us with 4 CTAs, 824 with 5, 797 with 6;
// 8 loads and 3 CTAs 990 us).  Some forms spill a little for it (FP32 at six with beta == 0 and 8 or 16 lanes 20 bytes stored and up to 64 loaded a thread, BF16 at five
// with narrow ragged rows up to 32 / 48); BF16, with eight sums a lane, spills much more at six.
template <typename T> constexpr int kBundleCtas = sizeof(T) == 4 ? 6 : 5;
// Most merge items per warp: no lane adds more than 128 products of a long piece in one chain, and the shared memory of the resident warps leaves L1 room
// for what is in flight (320 items: 27 KB a CTA).
constexpr int bundle_most(int lanes) { return lanes >= 32 ? 128 : lanes == 16 ? 256 : 320; }

// Shared memory of a warp: (col, val) pairs, the pieces of its rows (one for two items at most, and the row left unfinished) and the empty ones of 32 rows.
__host__ __device__ constexpr int bundle_bytes(int region) { return (region + 8) * 8 + (region / 2 + 8) * 4 + 32; }

// Y's VEC columns of a lane, YV to a store; `left` columns up to k.  old: their values before (BETA).
template <typename T, int VEC, int YV, bool BETA>
__device__ __forceinline__ void bundle_store(T* yp, int left, const float (&acc)[VEC], float alpha, float beta, const typename Piece<T, YV>::raw (&old)[BETA ? VEC / YV : 1]) {
#pragma unroll
  for (int i = 0; i < VEC / YV; ++i)
    if (YV == VEC || i * YV < left) {
      float a[YV];
#pragma unroll
      for (int j = 0; j < YV; ++j) a[j] = alpha * acc[i * YV + j];
      if (BETA) {
        float o[YV];
        Piece<T, YV>::widen(old[i], o);
#pragma unroll
        for (int j = 0; j < YV; ++j) a[j] += beta * o[j];
      }
      *((typename Piece<T, YV>::raw*)yp + i) = Piece<T, YV>::pack(a);
    }
}

// Y's VEC columns of a lane in a row without nonzeros.  none: the factor of its old values (BETA), or what it gets.  A parameter of the kernel, which takes no
// register; alpha * 0 would (R-MAT 2^17, k = 63 FP32, beta = 1: 84 / 116 us).
template <typename T, int VEC, int YV, bool BETA>
__device__ __forceinline__ void bundle_store_empty(T* yp, int left, float none, const typename Piece<T, YV>::raw (&old)[BETA ? VEC / YV : 1]) {
  float acc[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) acc[j] = BETA ? 0.0f : none;
  bundle_store<T, VEC, YV, BETA>(yp, left, acc, BETA ? 0.0f : 1.0f, none, old);
}

// The same over `count` elements by a warp: whole rows, whatever their width, in pieces of 16 bytes but for what lies before the first boundary of
// 16 bytes and after the last.
template <typename T, bool BETA>
__device__ __forceinline__ void bundle_empty_span(T* y, int count, int lane, float none) {
  constexpr int VEC = 16 / sizeof(T);
  typedef typename Piece<T, VEC>::raw raw;
  const int before = min(count, (int)((16u - ((unsigned)(uintptr_t)y & 15u)) & 15u) / (int)sizeof(T));
  const int pieces = (count - before) / VEC, after = count - before - pieces * VEC;
  T* const body = y + before;
  for (int p = lane; p < pieces; p += 4 * 32) {
    raw old[4][1];
    if constexpr (BETA) {
#pragma unroll
      for (int u = 0; u < 4; ++u) if (p + 32 * u < pieces) old[u][0] = *((const raw*)body + p + 32 * u);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) if (p + 32 * u < pieces) bundle_store_empty<T, VEC, VEC, BETA>(body + (p + 32 * u) * VEC, VEC, none, old[u]);
  }
  T* const at = lane < before ? y + lane : body + pieces * VEC + (lane - before);
  if (lane < before + after) {
    typename Piece<T, 1>::raw old_1[1];
    if constexpr (BETA) old_1[0] = *at;
    bundle_store_empty<T, 1, 1, BETA>(at, 1, none, old_1);
  }
}

// Rows without nonzeros are written as others are, by the lanes that hold a piece of B, several rows at a time; BF16 of ragged width above 32 columns apart, where
// a lane has columns one or two at a time to store: consecutive empty rows of so many bytes of Y are one span, whatever k is, and with odd k a warp takes shorter runs
// row by row.  40,000 rows of 20 and 100,000 empty ones, by lanes / so: k = 127 293 / 45 us, k = 63 146 / 26 us, k = 50 and beta = 1 56 / 35 us.  R-MAT 2^17, beta = 1: k = 63
// 140 / 75 us, k = 50 56 / 54 us (61 us with k = 50 row by row).  FP32 spills for it (R-MAT 2^17, k = 63, beta = 1 84 / 95 us).
constexpr int kBundleSpan = 512, kBundleSpanByLanes = 2048;

// A tile is kMergeWarps regions, one per warp.  What crosses the ends of a region goes to head_s / carry_s and is put together inside the tile after one
// barrier; what crosses the ends of the tile goes to tile_carry / tile_tail and is finished by spmm_merge_fixup_kernel, as for spmm_merge_kernel: fixed order, no
// atomics.  split[i]: row ends before item i * per.
template <typename T, int LANES, int YV, bool BETA>
__global__ void __launch_bounds__(kMergeWarps * 32, kBundleCtas<T>)
spmm_bundle_kernel(int m, int nnz, int k, int row_bytes, int region, const int* __restrict__ split, int per, const int* __restrict__ row_ptr,
                   const int* __restrict__ col_idx, const T* __restrict__ vals, const T* __restrict__ B, T* __restrict__ Y,
                   float* __restrict__ tile_carry, float* __restrict__ tile_tail, int2* __restrict__ tile_row, float alpha, float beta, float none) {
  constexpr int VEC = 16 / sizeof(T), G = 32 / LANES, KS = LANES * VEC, NY = VEC / YV, U = 4;   // U: loads of B in flight per lane
  constexpr bool BY_WARP = NY >= 8 && LANES >= 8;             // empty rows apart from others: see kBundleSpan
  typedef typename Piece<T, VEC>::raw raw;
  typedef typename Piece<T, YV>::raw yraw;
  extern __shared__ __align__(16) unsigned char bundle_smem[];
  __shared__ float head_s[kMergeWarps][KS], carry_s[kMergeWarps][KS];
  __shared__ int first_s[2];                                 // the tile's first row and where it starts, -1 when inside the tile
  // Before anything is read, also where B is a padded copy and only B comes from the kernel before this one: that kernel has waited for the stream's earlier
  // work, but what it then sees is promised to it alone, not to the kernel that it lets start.
  grid_dependency_wait();
  const int t = blockIdx.x;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31, g = lane / LANES, l = lane % LANES;
  unsigned char* const mine = bundle_smem + warp * bundle_bytes(region);
  int2* const pair = (int2*)mine;
  unsigned* const list = (unsigned*)(pair + region + 8);
  unsigned char* const empty_rows = (unsigned char*)(list + region / 2 + 8);

  const long long total = (long long)m + nnz;
  // Row ends before item x: split[] has them for every `per` items, the rest is counted.  Within the bounds that the split points keep, and ends within the
  // region below: whatever ascending row_ptr holds, a region's nonzeros lie in [0, nnz).
  auto row_ends = [&](long long x) {
    const int at = (int)((unsigned)x / (unsigned)per);
    const int r0 = __ldg(split + at);
    if (x == (long long)at * per || x >= total) return x >= total ? m : r0;
    const int r1 = __ldg(split + at + 1);
    int n = 0;
    for (int j = r0 + lane; __any_sync(0xFFFFFFFFu, j < r1); j += 32)
      n += __popc(__ballot_sync(0xFFFFFFFFu, j < r1 && (unsigned)__ldg(row_ptr + j + 1) + (unsigned)j < (unsigned)x));
    return min(max(r0 + n, (int)max(x - nnz, 0LL)), (int)min(x, (long long)m));
  };
  const long long x0 = min(((long long)t * kMergeWarps + warp) * region, total), x1 = min(x0 + region, total);
  const int r_lo = uniform(row_ends(x0)), r_hi = uniform(row_ends(x1));
  const int p0 = (int)(x0 - r_lo), p1 = (int)(x1 - r_hi);
  const int cnt = p1 - p0, rows = r_hi - r_lo;
  auto row_end = [&](int i) { return i < rows ? min(max(__ldg(row_ptr + r_lo + 1 + i) - p0, 0), cnt) : cnt; };
  int e_next = row_end(lane);                                // ends of 32 rows
  if constexpr (sizeof(T) == 4) {
    for (int i = lane; i < cnt; i += 32) {
      cp_async4(&pair[i].x, col_idx + p0 + i);
      cp_async4(&pair[i].y, vals + p0 + i);
    }
    cp_async_commit();
  } else {
#pragma unroll 4
    for (int i = lane; i < cnt; i += 32) pair[i] = make_int2(__ldg(col_idx + p0 + i), (int)((unsigned)__ldg(vals + p0 + i) << 16));
  }
  const int start0 = uniform(__ldg(row_ptr + r_lo));         // start of the first row (nnz when there is none)
  const bool head = start0 < p0;                             // the first row began before this warp's region
  for (int c = lane; c < KS; c += 32) { head_s[warp][c] = 0.0f; carry_s[warp][c] = 0.0f; }
  const int col0 = l * VEC, left = k - col0;
  const bool on = left > 0;
  const char* const Bc = (const char*)(B + (on ? col0 : 0));     // lanes past k read what lane 0 reads
  T* const Yc = Y + (long long)r_lo * k + col0;

  auto ask_old = [&](const T* yp, yraw (&old)[BETA ? NY : 1]) {
#pragma unroll
    for (int i = 0; i < (BETA ? NY : 0); ++i) if (YV == VEC || i * YV < left) old[i] = *((const yraw*)yp + i);
  };
  // Pieces of rows: length << 20 | row of the region << 10 | first nonzero.  Piece `rows`: of the row left unfinished.  Rows without nonzeros are
  // written on the way.
  int listed = 0, before0 = 0;
  for (int i0 = 0; i0 <= rows; i0 += 32) {
    const int i = i0 + lane, e = e_next;
    e_next = row_end(i + 32);
    int before = __shfl_up_sync(0xFFFFFFFFu, e, 1);
    if (lane == 0) before = before0;
    before0 = __shfl_sync(0xFFFFFFFFu, e, 31);
    const bool full = i <= rows && e > before, vacant = i < rows && e == before && !(head && i == 0);
    const unsigned fulls = __ballot_sync(0xFFFFFFFFu, full), vacants = __ballot_sync(0xFFFFFFFFu, vacant), below = (1u << lane) - 1u;
    if (full) list[listed + __popc(fulls & below)] = ((unsigned)(e - before) << 20) | (unsigned)(i << 10) | (unsigned)before;
    listed += __popc(fulls);
    if (vacants) {
      unsigned apart = vacants;                                   // without long runs of empty rows, which are written as one span
      if constexpr (sizeof(T) == 2 && YV != VEC && LANES >= 8) {
        constexpr int LEAST = (BY_WARP ? kBundleSpan : kBundleSpanByLanes) / (int)sizeof(T);
        if (__popc(vacants) * k >= LEAST)
          for (unsigned rest = vacants; rest;) {
            const int first = __ffs(rest) - 1, run = __ffs(~(rest >> first)) - 1, count = run < 0 ? 32 : run;
            const unsigned these = (count == 32 ? ~0u : (1u << count) - 1u) << first;
            rest &= ~these;
            if (count * k >= LEAST) {
              apart &= ~these;
              bundle_empty_span<T, BETA>(Y + (long long)(r_lo + i0 + first) * k, count * k, lane, none);
            }
          }
      }
      if ((apart >> lane) & 1u) empty_rows[__popc(apart & below)] = (unsigned char)lane;
      __syncwarp();
      const int empties = __popc(apart);
      if constexpr (BY_WARP) {
        constexpr int NC = KS / 32, R = 8 / NC;
        T* const y0 = Y + (long long)(r_lo + i0) * k + lane;
        for (int j = 0; j < empties; j += R) {
          yraw old[R][NC][1];
          T* yp[R];
#pragma unroll
          for (int u = 0; u < R; ++u) {
            yp[u] = y0 + (long long)empty_rows[min(j + u, empties - 1)] * k;
#pragma unroll
            for (int c = 0; c < (BETA ? NC : 0); ++c)
              if (j + u < empties && lane + 32 * c < k) old[u][c][0] = *(const yraw*)(yp[u] + 32 * c);
          }
#pragma unroll
          for (int u = 0; u < R; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c)
              if (j + u < empties && lane + 32 * c < k) bundle_store_empty<T, 1, 1, BETA>(yp[u] + 32 * c, 1, none, old[u][c]);
        }
      } else {
        T* const y0 = Yc + (long long)i0 * k;
        for (int j = g; j < empties; j += 4 * G) {
          yraw old[4][BETA ? NY : 1];
          T* yp[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            yp[u] = y0 + (long long)empty_rows[min(j + u * G, empties - 1)] * k;
            if constexpr (BETA) { if (j + u * G < empties && on) ask_old(yp[u], old[u]); }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (j + u * G < empties && on) bundle_store_empty<T, VEC, YV, BETA>(yp[u], left, none, old[u]);
        }
      }
      __syncwarp();
    }
  }
  if constexpr (sizeof(T) == 4) cp_async_wait<0>();
  __syncwarp();
  for (int j0 = 0; j0 < listed; j0 += 32) {
    // 32 pieces sorted by length, the longest first
    unsigned key = j0 + lane < listed ? list[j0 + lane] : 0u;
#pragma unroll
    for (int size = 2; size <= 32; size *= 2)
#pragma unroll
      for (int d = size / 2; d > 0; d /= 2) {
        const unsigned other = __shfl_xor_sync(0xFFFFFFFFu, key, d);
        key = ((lane & size) == 0) == ((lane & d) == 0) ? max(key, other) : min(key, other);
      }
    const int full = __popc(__ballot_sync(0xFFFFFFFFu, key != 0u)), longs = __popc(__ballot_sync(0xFFFFFFFFu, (key >> 20) > kBundleLong));
    for (int e = 0; e < full; e += e < longs ? 1 : G) {
      const bool joint = e < longs;                            // a long piece: a part of it for every group
      unsigned piece = __shfl_sync(0xFFFFFFFFu, key, joint ? e : min(e + g, 31));
      int len = (int)(piece >> 20);
      if (joint) {
        const int part = (len + G - 1) / G;
        len = max(0, min(part, len - g * part));
        piece += g * part;
      } else if (e + g > 31) {
        len = 0;
      }
      const int i = (int)(piece >> 10) & 1023;
      const bool holds_sum = joint ? g == 0 : len != 0;
      yraw old[BETA ? NY : 1];
      if constexpr (BETA) { if (on && holds_sum && i < rows) ask_old(Yc + (long long)i * k, old); }
      float acc[VEC];
#pragma unroll
      for (int j = 0; j < VEC; ++j) acc[j] = 0.0f;
      const int2* pp = pair + (piece & 1023u);
#pragma unroll 1
      for (; len >= U; len -= U, pp += U) {
        int2 a[U];
        raw b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = pp[u];
#pragma unroll
        for (int u = 0; u < U; ++u) b[u] = __ldg((const raw*)(Bc + (long long)a[u].x * row_bytes));
#pragma unroll
        for (int u = 0; u < U; ++u) piece_fma<T, VEC>(b[u], __int_as_float(a[u].y), acc);
      }
      if (len > 0) {                                         // the last one to three; loads without a nonzero read the last row of B again, and zeros take their place
        int2 a[U - 1];
        raw b[U - 1];
#pragma unroll
        for (int u = 0; u < U - 1; ++u) a[u] = pp[min(u, len - 1)];
#pragma unroll
        for (int u = 0; u < U - 1; ++u) b[u] = __ldg((const raw*)(Bc + (long long)a[u].x * row_bytes));
#pragma unroll
        for (int u = 0; u < U - 1; ++u) {
          uint4 w = *(const uint4*)&b[u];
          if (u >= len) { w = make_uint4(0, 0, 0, 0); a[u].y = 0; }
          piece_fma<T, VEC>(*(const raw*)&w, __int_as_float(a[u].y), acc);
        }
      }
      if (joint) {
#pragma unroll
        for (int d = LANES; d < 32; d *= 2)
#pragma unroll
          for (int j = 0; j < VEC; ++j) acc[j] += __shfl_xor_sync(0xFFFFFFFFu, acc[j], d);
      }
      if (holds_sum) {                                         // to Y, or the head of a row that began earlier, or the carry of a row left unfinished
        if (i == rows || (i == 0 && head)) {
          float* const to = i == rows ? carry_s[warp] : head_s[warp];
#pragma unroll
          for (int j = 0; j < VEC; ++j) to[l * VEC + j] = acc[j];
        } else if (on) {
          bundle_store<T, VEC, YV, BETA>(Yc + (long long)i * k, left, acc, alpha, beta, old);
        }
      }
      __syncwarp();
    }
  }
  if (warp == 0 && lane == 0) { first_s[0] = r_lo; first_s[1] = head ? start0 : -1; }
  __syncthreads();

  // Merge items are counted in 32 bits (m + nnz < 2^32).
  const long long slot = (long long)t * KS;
  if (head && rows > 0) {                                    // complete the row that ends here: the carries before it, in order, then the head
    const int ws = (int)(((unsigned)start0 + (unsigned)r_lo) / (unsigned)region) - t * kMergeWarps;   // the warp that holds the row's start
    for (int c = lane; c < KS; c += 32) {
      float s = 0.0f;
      for (int w = ws > 0 ? ws : 0; w < warp; ++w) s += carry_s[w][c];
      s += head_s[warp][c];
      if (ws >= 0) { if (c < k) epilogue_store(Y, (long long)r_lo * k + c, s, alpha, beta); }
      else tile_tail[slot + c] = s;
    }
  }
  if (warp == kMergeWarps - 1) {                             // what the tile leaves unfinished
    if (lane == 0) {                                         // and for the fix-up: the row that it completes for earlier tiles, and the first of them
      const int r = first_s[0], rs = first_s[1];
      tile_row[t] = rs >= 0 && r_hi > r ? make_int2(r, (int)(((unsigned)rs + (unsigned)r) / ((unsigned)region * kMergeWarps))) : make_int2(-1, 0);
    }
    int ws = kMergeWarps;
    if (r_hi < m) ws = (int)(((unsigned)__ldg(row_ptr + r_hi) + (unsigned)r_hi) / (unsigned)region) - t * kMergeWarps;
    for (int c = lane; c < KS; c += 32) {
      float s = 0.0f;
      for (int w = ws > 0 ? ws : 0; w < kMergeWarps; ++w) s += carry_s[w][c];
      tile_carry[slot + c] = s;
    }
  }
}

// Rows of B (k elements each) copied into rows of `pitch` 4-byte words (a multiple of 16 bytes), zeros behind column k, so that lanes can read 16 bytes of
// any row.  A warp takes a row at a time, a word per lane, four rows in flight; pairs of 16-bit elements that no word of B holds (odd k) by two loads.
// Latency-bound (120,007 rows of 50 BF16 6.9 us; 4, 8 or 16 consecutive pieces in flight 0.1 to 30 us slower or 0.5 faster).
template <typename T>
__global__ void __launch_bounds__(256) spmm_pad_rows_kernel(int n, int k, int pitch, const T* __restrict__ B, unsigned* __restrict__ P) {
  grid_dependency_wait();
  const int lane = threadIdx.x & 31, warps = gridDim.x * 8;
  auto word = [&](int r, int w) -> unsigned {
    if (r >= n) return 0u;
    if constexpr (sizeof(T) == 4) {
      return w < k ? __float_as_uint(__ldg(B + (long long)r * k + w)) : 0u;
    } else {
      const T* const at = B + (long long)r * k + 2 * w;
      if ((k & 1) == 0) return 2 * w < k ? __ldg((const unsigned*)at) : 0u;
      return (2 * w < k ? (unsigned)__ldg(at) : 0u) | (2 * w + 1 < k ? (unsigned)__ldg(at + 1) << 16 : 0u);
    }
  };
  for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < n; r += 4 * warps)
    for (int w = lane; w < pitch; w += 32) {
      unsigned v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = word(min(r + u * warps, n), w);
#pragma unroll
      for (int u = 0; u < 4; ++u) if (r + u * warps < n) P[(long long)(r + u * warps) * pitch + w] = v[u];
    }
}

}  // namespace b200sp
