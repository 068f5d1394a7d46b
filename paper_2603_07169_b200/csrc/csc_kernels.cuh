// CSC SpMV by products (paper, Appendix C, Table 6, task 10, with alpha/beta): y = alpha * A * x + beta * y, A given by columns.
//
// In CSC order the product vals[p] * x[col(p)] needs no gather: vals is a stream and x is read in order.  What is random is the way
// from there to the rows.  Permuting the values into row order and running the CSR kernel pays two random accesses of four bytes per
// nonzero (a value, then an entry of x); here the products make the way once, and in runs instead of one by one:
//   pass 1  a CTA computes the products of a TILE of consecutive CSC entries into shared memory and writes them out sorted by
//           BUCKET (a range of rows that holds about C nonzeros), so that what goes to one bucket is a run of consecutive words;
//   pass 2  a CTA reads the products of its bucket, which are contiguous, puts them into row order in shared memory and adds
//           the rows up.
// The pattern alone decides all of these places; they are computed once per pattern (kernels csc_*_plan below) and kept in
// 16-bit form: per nonzero 2 bytes of column (from the tile's first), 2 of source place in the tile and 2 of place in the bucket.
// The sum of a row is added in CSC order of its entries on every run.
#pragma once
#include "format_kernels.cuh"
#include "spmv_kernels.cuh"

namespace b200sp {

constexpr int kCscThreads = 512;
constexpr int kCscSlack = 1024;        // a bucket holds at most C + kCscSlack nonzeros: rows of at most that many
constexpr int kCscMaxTile = 32768;
constexpr int kCscMaxBuckets = 4096;
constexpr int kCscShortRow = 32;       // rows of at most this many products are added by one thread

__device__ __forceinline__ unsigned ld_stream_u16(const unsigned short* p) {
  unsigned short v;
  asm("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_stream_u2(const unsigned short* p) {
  uint2 v;
  asm("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// Pass 1.  Slot j of the tile's output (sorted by bucket) takes the product of the tile's entry src[j] & 0x7FFF; bit 15 marks the
// first slot of a run.  run_before[chunk]: runs that begin before the chunk of 32 slots; run r of the tile goes to slot + run_shift[r].
// Bound by memory (14 bytes of streams per FP32 nonzero) and by how long the runs are that it writes: tiles as large as shared memory
// takes, one CTA per SM, and W chunks' places fetched ahead.
template <typename T, int TILE, int THREADS>
__global__ void __launch_bounds__(THREADS)
csc_products_kernel(int nnz, int runs_per_tile, const T* __restrict__ vals, const T* __restrict__ x, const unsigned short* __restrict__ dcol,
                    const int* __restrict__ tile_col, const unsigned short* __restrict__ src, const unsigned short* __restrict__ run_before,
                    const int* __restrict__ run_shift, float* __restrict__ prod) {
  constexpr int Q = TILE / (THREADS * 4);        // groups of four entries per thread, all in flight
  constexpr int W = Q < 4 ? 4 : Q;               // chunks of 32 slots per warp and batch; the next batch is in flight
  extern __shared__ __align__(16) unsigned char csc_smem[];
  float* const prod_s = (float*)csc_smem;
  int* const shift_s = (int*)(csc_smem + TILE * sizeof(float));
  grid_dependency_wait();
  const int t = blockIdx.x, p0 = t * TILE, cnt = min(TILE, nnz - p0), tid = threadIdx.x, lane = tid & 31;
  const T* const xt = x + __ldg(tile_col + t);
  unsigned s[2][W];                              // source places of the warp's next chunks, this batch of W and the next one
  int before[2];                                 // lane w: runs before the batch's chunk w
  auto places = [&](int j0, unsigned (&sw)[W], int& bw) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int j = j0 + w * THREADS + lane;     // (warps take chunks in turn)
      sw[w] = j < cnt ? ld_stream_u16(src + p0 + j) : 0u;
    }
    bw = lane < W && j0 + lane * THREADS < cnt ? (int)ld_stream_u16(run_before + ((p0 + j0 + lane * THREADS) >> 5)) : 0;
  };
  places(tid & ~31, s[0], before[0]);
  for (int r = tid; r < runs_per_tile; r += THREADS) shift_s[r] = ld_stream_i1(run_shift + (long long)t * runs_per_tile + r);
  if (cnt == TILE) {
    float v[Q][4];
    uint2 d[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int i = (q * THREADS + tid) * 4;
      ld_stream_vals4(vals + p0 + i, v[q]);
      d[q] = ld_stream_u2(dcol + p0 + i);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      *(float4*)(prod_s + (q * THREADS + tid) * 4) =
          make_float4(v[q][0] * ld_gather(xt + (d[q].x & 0xFFFFu)), v[q][1] * ld_gather(xt + (d[q].x >> 16)),
                      v[q][2] * ld_gather(xt + (d[q].y & 0xFFFFu)), v[q][3] * ld_gather(xt + (d[q].y >> 16)));
  } else {
    for (int i = tid; i < cnt; i += THREADS) prod_s[i] = ld_stream_val1(vals + p0 + i) * ld_gather(xt + dcol[p0 + i]);
  }
  __syncthreads();
  const unsigned upto = 0xFFFFFFFFu >> (31 - lane);
  auto write = [&](int j0, const unsigned (&sw)[W], int bw) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int j = j0 + w * THREADS + lane;
      const unsigned firsts = __ballot_sync(0xFFFFFFFFu, sw[w] >> 15);
      const int run = __shfl_sync(0xFFFFFFFFu, bw, w) + __popc(firsts & upto) - 1;
      if (j < cnt) prod[p0 + j + shift_s[run]] = prod_s[sw[w] & 0x7FFFu];
    }
  };
  constexpr int STEP = W * THREADS;
  for (int j0 = tid & ~31; j0 < cnt; j0 += 2 * STEP) {
    if (j0 + STEP < cnt) places(j0 + STEP, s[1], before[1]);
    write(j0, s[0], before[0]);
    if (j0 + STEP < cnt) {
      if (j0 + 2 * STEP < cnt) places(j0 + 2 * STEP, s[0], before[0]);
      write(j0 + STEP, s[1], before[1]);
    }
  }
}

// Pass 2.  Rows bucket_row[b] .. bucket_row[b + 1] of bucket b; its product i belongs at place dst[i] of the bucket's nonzeros in row order.
template <typename T>
__global__ void __launch_bounds__(kCscThreads)
csc_bucket_sums_kernel(int cap, const int* __restrict__ bucket_row, const int* __restrict__ bucket_start, const int* __restrict__ row_ptr, const float* __restrict__ prod,
                       const unsigned short* __restrict__ dst, T* __restrict__ y, float alpha, float beta) {
  extern __shared__ __align__(16) unsigned char csc_smem[];
  float* const prod_s = (float*)csc_smem;
  int* const long_rows = (int*)(prod_s + pad_index(cap) + 1);
  __shared__ int n_long;
  grid_dependency_wait();
  const int tid = threadIdx.x;
  const int r0 = __ldg(bucket_row + blockIdx.x), r1 = __ldg(bucket_row + blockIdx.x + 1);
  const int s0 = __ldg(bucket_start + blockIdx.x), cnt = __ldg(bucket_start + blockIdx.x + 1) - s0;
  if (tid == 0) n_long = 0;
  for (int i0 = tid; i0 < cnt; i0 += 8 * kCscThreads) {
    unsigned at[8];
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + u * kCscThreads;
      at[u] = i < cnt ? ld_stream_u16(dst + s0 + i) : 0u;
      v[u] = i < cnt ? __ldcg(prod + s0 + i) : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) if (i0 + u * kCscThreads < cnt) prod_s[pad_index(at[u])] = v[u];
  }
  int rs = 0, re = 0;                            // the thread's first row: its bounds are asked for before the barrier
  if (r0 + tid < r1) { rs = __ldg(row_ptr + r0 + tid) - s0; re = __ldg(row_ptr + r0 + tid + 1) - s0; }
  __syncthreads();
  for (int r = r0 + tid; r < r1;) {
    if (re - rs <= kCscShortRow) {
      float acc = 0.0f;
      for (int q = rs; q < re; ++q) acc += prod_s[pad_index(q)];
      epilogue_store(y, r, acc, alpha, beta);
    } else {
      long_rows[atomicAdd(&n_long, 1)] = r;      // order of the list does not affect any value
    }
    r += kCscThreads;
    if (r < r1) { rs = __ldg(row_ptr + r) - s0; re = __ldg(row_ptr + r + 1) - s0; }
  }
  __syncthreads();
  const int lane = tid & 31;
  for (int i = tid >> 5; i < n_long; i += kCscThreads / 32) {
    const int r = long_rows[i];
    rs = __ldg(row_ptr + r) - s0;
    re = __ldg(row_ptr + r + 1) - s0;
    float acc = 0.0f;
    for (int q = rs + lane; q < re; q += 32) acc += prod_s[pad_index(q)];
    acc = warp_sum(acc);
    if (lane == 0) epilogue_store(y, r, acc, alpha, beta);
  }
}

// ---- the places, once per pattern -------------------------------------------------------------------------------------------------
// bucket of a row that has nonzeros: row_ptr[row] >> log2(C).  bucket_row[b]: first row with row_ptr >= b C; bucket_row[buckets] = m; bucket_start: their row_ptr.
__global__ void __launch_bounds__(256) csc_bucket_rows_plan(const int* __restrict__ row_ptr, int m, int buckets, int shift, int* __restrict__ bucket_row,
                                                            int* __restrict__ bucket_start) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > buckets) return;
  int lo = 0, hi = m;
  if (b == buckets) lo = m;
  else while (lo < hi) { const int mid = (lo + hi) >> 1; if ((long long)row_ptr[mid] < ((long long)b << shift)) lo = mid + 1; else hi = mid; }
  bucket_row[b] = lo;
  bucket_start[b] = row_ptr[lo];
}

// Most nonzeros of a bucket -> stat[0]; widest range of columns of a tile -> stat[1]; most rows of a bucket -> stat[2]; tile_col[t]: the column
// of the tile's first entry.
__global__ void __launch_bounds__(256) csc_extents_plan(const int* __restrict__ row_ptr, const int* __restrict__ bucket_row, int buckets,
                                                        const int* __restrict__ col_ptr, int n, int nnz, int tile, int tiles,
                                                        int* __restrict__ tile_col, int* __restrict__ stat) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < buckets) {
    atomicMax(stat, row_ptr[bucket_row[i + 1]] - row_ptr[bucket_row[i]]);
    atomicMax(stat + 2, bucket_row[i + 1] - bucket_row[i]);
  }
  if (i < tiles) {
    auto column = [&](int p) {                   // the last j with col_ptr[j] <= p
      int lo = 0, hi = n;
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (col_ptr[mid + 1] <= p) lo = mid + 1; else hi = mid; }
      return lo;
    };
    const long long end = (long long)(i + 1) * tile;
    const int first = column(i * tile), last = column((int)(end < nnz ? end : nnz) - 1);
    tile_col[i] = first;
    atomicMax(stat + 1, last - first);
  }
}

// count[t * buckets + b]: entries of tile t in bucket b.  One CTA per tile.
__global__ void __launch_bounds__(512) csc_tile_counts_plan(const int* __restrict__ row_idx, const int* __restrict__ row_ptr, int nnz, int tile,
                                                            int shift, int buckets, int* __restrict__ count) {
  extern __shared__ int csc_hist[];
  for (int b = threadIdx.x; b < buckets; b += 512) csc_hist[b] = 0;
  __syncthreads();
  const int p0 = blockIdx.x * tile, p1 = p0 + min(tile, nnz - p0);
  for (int p = p0 + threadIdx.x; p < p1; p += 512) atomicAdd(&csc_hist[__ldg(row_ptr + row_idx[p]) >> shift], 1);
  __syncthreads();
  for (int b = threadIdx.x; b < buckets; b += 512) count[(long long)blockIdx.x * buckets + b] = csc_hist[b];
}

// count -> where tile t's run in bucket b begins: the bucket's first nonzero + the counts of the tiles before t.  CTA: 32 buckets x 32
// parts of the tiles.
__global__ void __launch_bounds__(1024) csc_run_starts_plan(const int* __restrict__ row_ptr, const int* __restrict__ bucket_row, int buckets, int tiles,
                                                            int* __restrict__ count) {
  __shared__ int s_sum[32][33];
  const int bx = threadIdx.x & 31, part = threadIdx.x >> 5, b = blockIdx.x * 32 + bx;
  const int per = (tiles + 31) / 32, t0 = min(tiles, part * per), t1 = min(tiles, t0 + per);
  int sum = 0;
  if (b < buckets)
#pragma unroll 8
    for (int t = t0; t < t1; ++t) sum += count[(long long)t * buckets + b];
  s_sum[part][bx] = sum;
  __syncthreads();
  if (b >= buckets) return;
  int run = row_ptr[bucket_row[b]];
  for (int q = 0; q < part; ++q) run += s_sum[q][bx];
#pragma unroll 8
  for (int t = t0; t < t1; ++t) {
    const int c = count[(long long)t * buckets + b];
    count[(long long)t * buckets + b] = run;
    run += c;
  }
}

// Exclusive sum over the block of one int per thread (1024 threads); s: 33 ints.
__device__ __forceinline__ int block_exclusive_sum(int v, int* s, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += u; }
  __syncthreads();
  if (lane == 31) s[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = s[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xFFFFFFFFu, w, o); if (lane >= o) w += u; }
    s[lane] = w;
  }
  __syncthreads();
  if (total) *total = s[31];
  return (warp ? s[warp - 1] : 0) + incl - v;
}

// The slots of a tile: src, run_before, run_shift (see pass 1), the columns, and position[i]: the CSC position of product i of the buffer.  One
// CTA of 1024 threads per tile.  The order inside a run is arbitrary: pass 2 undoes it.
// start: where the tile's run in each bucket begins; on return the shifts of its runs, one after another.
// Dynamic shared memory: 3 * buckets ints, then tile 16-bit words.
__global__ void __launch_bounds__(1024) csc_tile_slots_plan(const int* __restrict__ row_idx, const int* __restrict__ row_ptr, const int* __restrict__ col_ptr,
                                                            const int* __restrict__ tile_col, int n, int nnz, int tile, int shift, int buckets,
                                                            unsigned short* __restrict__ src, unsigned short* __restrict__ run_before, int* start,
                                                            unsigned short* __restrict__ dcol, int* __restrict__ position) {
  extern __shared__ int csc_slots_smem[];
  __shared__ int s_scan[33];
  int* const cursor = csc_slots_smem;            // counts, then the next free slot of each run
  int* const first = cursor + buckets;           // first slot of each run
  int* const shift_s = first + buckets;
  unsigned short* const src_s = (unsigned short*)(shift_s + buckets);
  const int t = blockIdx.x, p0 = t * tile, cnt = min(tile, nnz - p0), tid = threadIdx.x;
  for (int b = tid; b < buckets; b += 1024) cursor[b] = 0;
  __syncthreads();
  for (int i = tid; i < cnt; i += 1024) atomicAdd(&cursor[__ldg(row_ptr + row_idx[p0 + i]) >> shift], 1);
  __syncthreads();
  int slots = 0, runs = 0;
  for (int b0 = 0; b0 < buckets; b0 += 1024) {
    const int b = b0 + tid, c = b < buckets ? cursor[b] : 0;
    const int begin = c > 0 ? start[(long long)t * buckets + b] : 0;   // read before the sums below synchronise, written after
    int total_c, total_r;
    const int j = slots + block_exclusive_sum(c, s_scan, &total_c);
    const int r = runs + block_exclusive_sum(c > 0, s_scan, &total_r);
    if (b < buckets) {
      const int to = begin - (p0 + j);
      cursor[b] = j; first[b] = j; shift_s[b] = to;
      if (c > 0) start[(long long)t * buckets + r] = to;
    }
    slots += total_c; runs += total_r;
  }
  __syncthreads();
  const int c0 = tile_col[t], c1 = t + 1 < gridDim.x ? tile_col[t + 1] : n - 1;
  for (int i = tid; i < cnt; i += 1024) {
    const int p = p0 + i, b = __ldg(row_ptr + row_idx[p]) >> shift;
    const int j = atomicAdd(&cursor[b], 1);
    src_s[j] = (unsigned short)(i | (j == first[b] ? 0x8000 : 0));
    position[p0 + j + shift_s[b]] = p;
    int lo = c0, hi = c1;                        // the last column with col_ptr <= p
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldg(col_ptr + mid + 1) <= p) lo = mid + 1; else hi = mid; }
    dcol[p] = (unsigned short)(lo - c0);
  }
  __syncthreads();
  const int lane = tid & 31;
  int before = 0;
  for (int k0 = 0; k0 < cnt; k0 += 32768) {      // 1024 chunks of 32 slots at a time: thread k counts the runs that begin in chunk k
    int mine = 0;
    for (int w = 0; w < 32; ++w) {               // warp w' looks at its 32 chunks one after another
      const int j = k0 + ((tid >> 5) * 32 + w) * 32 + lane;
      const unsigned s = j < cnt ? src_s[j] : 0u;
      const unsigned firsts = __ballot_sync(0xFFFFFFFFu, s >> 15);
      if (j < cnt) src[p0 + j] = (unsigned short)s;
      if (w == lane) mine = __popc(firsts);
    }
    int total;
    const int r = before + block_exclusive_sum(mine, s_scan, &total);
    if (k0 + tid * 32 < cnt) run_before[(p0 + k0) / 32 + tid] = (unsigned short)r;
    before += total;
  }
}

// dst: the place of the bucket's product i in row order, the entries of a row in the order of their CSC positions.  One CTA per bucket.
// The positions go to their rows' ranges in shared memory in any order (slots claimed with atomics, on counters in shared memory
// where the bucket has at most cap rows); an entry's place in its row is the number of smaller ones there.  Dynamic shared memory:
// cap ints, cap pairs of 16 bits, cap ints.
__global__ void __launch_bounds__(1024) csc_bucket_places_plan(int cap, const int* __restrict__ bucket_row, const int* __restrict__ bucket_start,
                                                               const int* __restrict__ row_ptr, const int* __restrict__ row_idx,
                                                               const int* __restrict__ position, int* __restrict__ fill, unsigned short* __restrict__ dst) {
  extern __shared__ int csc_places_smem[];
  int* const key_s = csc_places_smem;
  ushort2* const row_s = (ushort2*)(key_s + cap);            // of product i: its row's range among the bucket's nonzeros
  int* const claimed_s = (int*)(row_s + cap);
  const int r0 = bucket_row[blockIdx.x], rows = bucket_row[blockIdx.x + 1] - r0;
  const int s0 = bucket_start[blockIdx.x], cnt = bucket_start[blockIdx.x + 1] - s0;
  const bool few = rows <= cap;
  if (few) for (int i = threadIdx.x; i < rows; i += 1024) claimed_s[i] = 0;
  __syncthreads();
#pragma unroll 4
  for (int i = threadIdx.x; i < cnt; i += 1024) {
    const int p = position[s0 + i], r = row_idx[p];
    const int rs = __ldg(row_ptr + r) - s0, re = __ldg(row_ptr + r + 1) - s0;
    key_s[rs + (few ? atomicAdd(claimed_s + (r - r0), 1) : atomicAdd(fill + r, 1))] = p;
    row_s[i] = make_ushort2((unsigned short)rs, (unsigned short)re);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += 1024) {
    const int p = position[s0 + i], rs = row_s[i].x, re = row_s[i].y;
    int place = rs;
#pragma unroll 4
    for (int q = rs; q < re; ++q) place += key_s[q] < p;
    dst[s0 + i] = (unsigned short)place;
  }
}

}  // namespace b200sp
