// Host side of libb200sp.so: the COO, CSC and ELL front ends (row offsets, transpose plan, ELL launches).
// One of the pieces of the single translation unit b200sp.cu; include/b200sp.h states the contract of every entry point.
#pragma once
#include "host_spmm.cuh"
#include "format_kernels.cuh"
#include "csc_kernels.cuh"

// ---- COO front end: row offsets from sorted row indices, then the CSR path ----
struct CooEntry { int32_t* row_ptr = nullptr; };
static std::map<std::tuple<int, const void*, int64_t, int64_t, int64_t>, CooEntry> g_coo_cache;

static int coo_row_ptr(const int32_t** out, int64_t m, int64_t n, int64_t nnz, const int32_t* row_idx, cudaStream_t stream) {
  DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != B200SP_OK) return rc;
  int d = 0;
  CU(cudaGetDevice(&d));
  const auto key = std::make_tuple(d, (const void*)row_idx, m, n, nnz);
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    auto it = g_coo_cache.find(key);
    if (it != g_coo_cache.end()) { *out = it->second.row_ptr; return B200SP_OK; }
  }
  int32_t* rp = nullptr;
  int* d_bad = nullptr;
  int h_bad = 0;
  CU(cudaMalloc(&rp, (size_t)(m + 1) * sizeof(int32_t)));
  cudaError_t e = cudaMalloc(&d_bad, sizeof(int));
  if (e == cudaSuccess) e = cudaMemsetAsync(d_bad, 0, sizeof(int), stream);
  if (e == cudaSuccess) {
    const long long work = (m + 1 > nnz ? m + 1 : nnz);
    long long blocks = (work + 255) / 256;
    if (blocks > (long long)dev->sms * 16) blocks = (long long)dev->sms * 16;
    coo_row_ptr_kernel<<<(unsigned)blocks, 256, 0, stream>>>(row_idx, (int)nnz, (int)m, rp, d_bad);
    g_launches++;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h_bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (d_bad) cudaFree(d_bad);
  if (e != cudaSuccess) { cudaFree(rp); return cuda_fail(e, "COO row offsets"); }
  if (h_bad) { cudaFree(rp); return B200SP_ERR_UNSUPPORTED; }   // entries not sorted by row, or a row index out of range
  std::lock_guard<std::mutex> lock(g_mutex);
  auto ins = g_coo_cache.emplace(key, CooEntry{rp});
  if (!ins.second) { cudaFree(rp); rp = ins.first->second.row_ptr; }
  *out = rp;
  return B200SP_OK;
}

// ---- CSC front end: a transpose plan built on the device (see format_kernels.cuh and csc_kernels.cuh) ----
// Per pattern: row offsets; for SpMV the places of the products (csc_kernels.cuh); for SpMM, and for SpMV where those do not apply, the
// CSC positions and columns in row-major order and room for the permuted values.  The last two are built on first use.
struct CscEntry {
  void* block = nullptr;
  int32_t* row_ptr = nullptr;
  int32_t* fill = nullptr;            // m + 2 counters, for building the parts below
  struct Csr { void* block = nullptr; int32_t* perm = nullptr; int32_t* col = nullptr; void* vals_t = nullptr; } csr;
  void* prod_block = nullptr;
  bool prod_tried = false;
  int bucket_rows = 0;                // most rows of a bucket, once counted
  int tile = 0, tiles = 0, buckets = 0, cap = 0;
  int *bucket_row = nullptr, *bucket_start = nullptr, *tile_col = nullptr, *run_shift = nullptr;
  unsigned short *src = nullptr, *dst = nullptr, *dcol = nullptr, *run_before = nullptr;
  float* prod = nullptr;
};
static std::map<std::tuple<int, const void*, const void*, int64_t, int64_t, int64_t>, CscEntry> g_csc_cache;
static std::mutex g_csc_build;      // one thread at a time adds parts to an entry

static void csc_free(CscEntry& e) {
  for (void* b : {e.block, e.csr.block, e.prod_block}) if (b) cudaFree(b);
  e = CscEntry();
}

static int csc_plan(CscEntry** out, int64_t m, int64_t n, int64_t nnz, const int32_t* col_ptr, const int32_t* row_idx, cudaStream_t stream) {
  DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != B200SP_OK) return rc;
  int d = 0;
  CU(cudaGetDevice(&d));
  const auto key = std::make_tuple(d, (const void*)col_ptr, (const void*)row_idx, m, n, nnz);
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    auto it = g_csc_cache.find(key);
    if (it != g_csc_cache.end()) { *out = &it->second; return B200SP_OK; }
  }
  if (stream_captures(stream)) return B200SP_ERR_UNSUPPORTED;    // the check of the pattern is read back
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t blocks = (size_t)((m + 1 + kScanBlock - 1) / kScanBlock);
  const size_t o_rp = 0, o_fill = o_rp + up(((size_t)m + 2) * 4), o_bs = o_fill + up(((size_t)m + 2) * 4), o_bad = o_bs + up((blocks + 1) * 4), total = o_bad + 256;
  CscEntry e;
  rc = pool_alloc(dev, &e.block, total, stream);
  if (rc != B200SP_OK) return rc;
  char* base = (char*)e.block;
  e.row_ptr = (int32_t*)(base + o_rp);
  e.fill = (int32_t*)(base + o_fill);
  int* fill = e.fill;
  int* bsum = (int*)(base + o_bs);
  int* d_bad = (int*)(base + o_bad);
  int h_bad = 0;
  auto fail = [&](int code) { cudaFreeAsync(e.block, stream); cudaStreamSynchronize(stream); return code; };
#define CUF(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return fail(cuda_fail(e_, #call)); } while (0)
  const unsigned wide = (unsigned)(dev->sms * 16);
  auto grid_for = [&](int64_t work) { long long b = (work + 255) / 256; if (b < 1) b = 1; return (unsigned)(b > (long long)wide ? wide : b); };
  CUF(cudaMemsetAsync(d_bad, 0, sizeof(int), stream));
  CUF(cudaMemsetAsync(fill, 0, ((size_t)m + 2) * 4, stream));
  csc_check_kernel<<<grid_for(nnz > n ? nnz : n), 256, 0, stream>>>(col_ptr, row_idx, (int)m, (int)n, (int)nnz, d_bad);
  g_launches++;
  CUF(cudaGetLastError());
  CUF(cudaMemcpyAsync(&h_bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, stream));
  CUF(cudaStreamSynchronize(stream));                          // nothing below may index with an unchecked row number
  if (h_bad) return fail(B200SP_ERR_BAD_CSR);
  if (nnz > 0) csc_count_rows_kernel<<<grid_for(nnz), 256, 0, stream>>>(row_idx, (long long)nnz, fill);
  // exclusive scan of the m + 1 counts (the last one is zero) -> row offsets, row_ptr[m] = nnz
  scan_block_sums_kernel<<<(unsigned)blocks, 256, 0, stream>>>(fill, (long long)m + 1, bsum);
  plan_compact_scan_kernel<<<1, 1024, 0, stream>>>(bsum, (int)blocks);
  scan_apply_kernel<<<(unsigned)blocks, 256, 0, stream>>>(fill, (long long)m + 1, bsum, e.row_ptr);
  g_launches += 4;
  CUF(cudaGetLastError());
  CUF(cudaStreamSynchronize(stream));
#undef CUF
  std::lock_guard<std::mutex> lock(g_mutex);
  auto ins = g_csc_cache.emplace(key, e);
  if (!ins.second) cudaFreeAsync(e.block, stream);
  *out = &ins.first->second;
  return B200SP_OK;
}

// CSC positions and columns in row-major order and room for the permuted values: what the CSR kernels need.  Built for the one call when the
// stream is captured.
static int csc_csr_part(CscEntry* e, CscEntry::Csr* out, CallBlock* own, int64_t m, int64_t n, int64_t nnz, const int32_t* col_ptr,
                        const int32_t* row_idx, cudaStream_t stream, DeviceInfo* dev) {
  std::lock_guard<std::mutex> lock(g_csc_build);
  if (e->csr.block) { *out = e->csr; return B200SP_OK; }
  const size_t bytes = ((size_t)(nnz > 0 ? nnz : 1) * 4 + 255) & ~(size_t)255;
  char* blk = nullptr;
  const int rc = pool_alloc(dev, (void**)&blk, 3 * bytes, stream);
  if (rc != B200SP_OK) return rc;
  int* perm = (int*)blk;
  int* col = (int*)(blk + bytes);
  if (nnz > 0) {
    long long blocks = (nnz + 255) / 256;
    if (blocks > (long long)dev->sms * 16) blocks = (long long)dev->sms * 16;
    cudaError_t err = cudaMemsetAsync(e->fill, 0, ((size_t)m + 2) * 4, stream);
    if (err == cudaSuccess) {
      csc_place_kernel<<<(unsigned)blocks, 256, 0, stream>>>(row_idx, (long long)nnz, e->row_ptr, e->fill, perm);
      csc_sort_rows_kernel<<<(unsigned)((m + 255) / 256), 256, 0, stream>>>((int)m, e->row_ptr, perm);
      csc_cols_kernel<<<(unsigned)blocks, 256, 0, stream>>>((long long)nnz, (int)n, col_ptr, perm, col);
      g_launches += 3;
      err = cudaGetLastError();
    }
    if (err != cudaSuccess) { cudaFreeAsync(blk, stream); return cuda_fail(err, "CSC row-major order"); }
  }
  *out = {blk, perm, col, blk + 2 * bytes};
  if (stream_captures(stream)) own->take(blk, stream);
  else e->csr = *out;
  return B200SP_OK;
}

// Most rows of one bucket for which the products pay.  Buckets are cut by nonzeros, so one may hold any number of empty rows, and its CTA
// walks them 512 at a time, 0.28 us a step (0.43 us where y is read), while the CSR kernels spread them over the GPU.  Where both take
// the same time, FP32 and BF16 alike (beta = 0 / beta != 0): 262,144 nonzeros 12,000 / 8,600 rows, 2^20 16,500 / 9,700, 2^22 36,000 / 24,000,
// 6.2 M (R-MAT) 33,000 / 20,000, 2^24 110,000 / 66,000, 27 M (R-MAT) more than 49,000 / 65,000; 2000 nonzeros in 2^22 rows 2278 us by products,
// 27 us by the CSR kernels.
static int64_t csc_most_bucket_rows(int64_t nnz, float beta) {
  const int64_t rows = std::min(4096 + nnz / 16, 12000 + nnz / 300);
  return beta == 0.0f ? rows : rows * 2 / 3;
}


// Entries of a tile and, as a power of two, nonzeros of a bucket of the products.
// Sizes: below 7.3 M nonzeros tiles of 2048, 4096 or 8192 entries, so that every SM gets several that overlap, and buckets of as many nonzeros (8192 from 3.8 M
// on: 4.3 M 24.0 / 21.5 us, 4.7 M 25.3 / 22.3 us); else one tile of 24576 .. 32768 entries per SM and round (96 .. 128 KB of products), the size that leaves
// the least of the last round idle (4.9 M nonzeros in two rounds of 24576 31.3 us, in tiles of 8192 26.5 us; 6.9 M 40.9 / 35.6 us; but 8 M in two
// rounds of 28672 38.9 us, in tiles of 8192 43.7 us), and buckets of 8192 nonzeros, 16384 above 2^25.  A run (a tile's products for one bucket) then averages
// tile * C / nnz = 3.5 .. 55 words: 2^24 nonzeros take 78 us, 81 us with tiles of 32768, 84 us with two tiles of 16384 per SM, 90 us with buckets of 16384.
// Below 4.8 M buckets of 8192 only where a row has one nonzero or more on average, two below 4.2 M: what a CTA walks of empty rows doubles with its bucket (buckets of
// 4096 / 8192: 3.9 M nonzeros in as many rows 31.9 / 33.9 us, in 7.8 M rows 45.8 / 49.4 us, 4.3 M in 8.6 M rows 50.1 / 51.1 us; but 4.8 M in as many rows 39.6 / 37.0 us).
struct CscSizes { int tile, shift; };
static CscSizes csc_sizes(int64_t m, int64_t nnz, int64_t sms) {
  CscSizes s;
  s.tile = nnz < sms * 4 * 2048 ? 2048 : nnz < sms * 8 * 4096 ? 4096 : 8192;
  if (nnz >= sms * 6 * 8192) {
    int64_t best = INT64_MAX;
    for (int t : {32768, 28672, 24576}) {
      const int64_t time = (((nnz + t - 1) / t + sms - 1) / sms) * t;     // rounds of one tile per SM
      if (time < best) { best = time; s.tile = t; }
    }
  }
  const bool larger = nnz >= sms * 8 * 4096 || (nnz >= sms * 25 * 1024 && nnz >= (nnz >= sms * 28 * 1024 ? m : 2 * m));
  s.shift = nnz < sms * 4 * 2048 ? 11 : !larger ? 12 : nnz <= ((int64_t)1 << 25) ? 13 : 14;
  return s;
}

// The places of the products of csc_kernels.cuh with tiles and buckets of the given sizes; leaves e->prod_block null where they do not apply: a row of more than
// kCscSlack nonzeros, a tile over more than 65536 columns or a bucket of more than most_rows rows.  Synchronises the stream.
static int csc_places(CscEntry* e, int64_t m, int64_t n, int64_t nnz, const int32_t* col_ptr, const int32_t* row_idx, int tile, int shift, int64_t most_rows,
                      cudaStream_t stream, DeviceInfo* dev) {
  const int tiles = (int)((nnz + tile - 1) / tile), buckets = (int)(((nnz - 1) >> shift) + 1), cap = (1 << shift) + kCscSlack;
  if (buckets > kCscMaxBuckets) { e->prod_tried = true; return B200SP_OK; }
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t nz = (size_t)tiles * tile;
  const size_t o_src = 0, o_dst = o_src + up(nz * 2), o_dcol = o_dst + up(nz * 2), o_before = o_dcol + up(nz * 2), o_shift = o_before + up(nz / 32 * 2),
               o_brow = o_shift + up((size_t)tiles * buckets * 4), o_bstart = o_brow + up((size_t)(buckets + 1) * 4), o_tcol = o_bstart + up((size_t)(buckets + 1) * 4), o_prod = o_tcol + up((size_t)tiles * 4),
               total = o_prod + up(nz * 4);
  char* blk = nullptr;
  const int rc = pool_alloc(dev, (void**)&blk, total, stream);
  if (rc != B200SP_OK) return rc;
  auto fail = [&](int code) { cudaFreeAsync(blk, stream); cudaStreamSynchronize(stream); return code; };
#define CUP(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return fail(cuda_fail(e_, #call)); } while (0)
  int* stat = (int*)(blk + o_before);            // not needed yet
  int* count = (int*)(blk + o_shift);            // counts, then starts, then shifts of the runs
  int* place = (int*)(blk + o_prod);             // the products' CSC positions; the products come later
  int* brow = (int*)(blk + o_brow);
  int* tcol = (int*)(blk + o_tcol);
  int h[3] = {0, 0, 0};
  CUP(cudaMemsetAsync(stat, 0, sizeof h, stream));
  csc_bucket_rows_plan<<<(buckets + 1 + 255) / 256, 256, 0, stream>>>(e->row_ptr, (int)m, buckets, shift, brow, (int*)(blk + o_bstart));
  const int wider = buckets > tiles ? buckets : tiles;
  csc_extents_plan<<<(wider + 255) / 256, 256, 0, stream>>>(e->row_ptr, brow, buckets, col_ptr, (int)n, (int)nnz, tile, tiles, tcol, stat);
  g_launches += 2;
  CUP(cudaGetLastError());
  CUP(cudaMemcpyAsync(h, stat, sizeof h, cudaMemcpyDeviceToHost, stream));
  CUP(cudaStreamSynchronize(stream));
  e->bucket_rows = h[2];
  e->prod_tried = h[0] > cap || h[1] > 65535;
  if (e->prod_tried || e->bucket_rows > most_rows) return fail(B200SP_OK);
  const size_t slots_smem = (size_t)buckets * 12 + (size_t)tile * 2;
  CUP(cudaFuncSetAttribute(csc_tile_slots_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, kCscMaxBuckets * 12 + kCscMaxTile * 2));
  csc_tile_counts_plan<<<tiles, 512, (size_t)buckets * 4, stream>>>(row_idx, e->row_ptr, (int)nnz, tile, shift, buckets, count);
  csc_run_starts_plan<<<(buckets + 31) / 32, 1024, 0, stream>>>(e->row_ptr, brow, buckets, tiles, count);
  csc_tile_slots_plan<<<tiles, 1024, slots_smem, stream>>>(row_idx, e->row_ptr, col_ptr, tcol, (int)n, (int)nnz, tile, shift, buckets,
                                                          (unsigned short*)(blk + o_src), (unsigned short*)(blk + o_before), count,
                                                          (unsigned short*)(blk + o_dcol), place);
  CUP(cudaMemsetAsync(e->fill, 0, ((size_t)m + 2) * 4, stream));
  CUP(cudaFuncSetAttribute(csc_bucket_places_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, ((1 << 14) + kCscSlack) * 12));
  csc_bucket_places_plan<<<buckets, 1024, (size_t)cap * 12, stream>>>(cap, brow, (const int*)(blk + o_bstart), e->row_ptr, row_idx, place, e->fill,
                                                                    (unsigned short*)(blk + o_dst));
  g_launches += 4;
  CUP(cudaGetLastError());
#undef CUP
  e->tile = tile; e->tiles = tiles; e->buckets = buckets; e->cap = cap;
  e->bucket_row = brow; e->bucket_start = (int*)(blk + o_bstart); e->tile_col = tcol; e->run_shift = (int*)(blk + o_shift);
  e->src = (unsigned short*)(blk + o_src); e->dst = (unsigned short*)(blk + o_dst); e->dcol = (unsigned short*)(blk + o_dcol);
  e->run_before = (unsigned short*)(blk + o_before);
  e->prod = (float*)(blk + o_prod);
  e->prod_block = blk;
  e->prod_tried = true;
  return B200SP_OK;
}

// The same with the sizes that csc_sizes names, and with buckets of 4096 below 4.8 M nonzeros where those of 8192 do not apply or hold more rows than pay with
// beta != 0 (4.8 M nonzeros in 12 M rows, beta = 0.5 82 / 113 us by products / by the CSR kernels).  Nothing is done while the stream is captured (the limits are read
// back).  Above 2^26 nonzeros, and where the places do not apply, SpMV takes the CSR kernels.
static int csc_product_part(CscEntry* e, int64_t m, int64_t n, int64_t nnz, const int32_t* col_ptr, const int32_t* row_idx, int64_t most_rows,
                            cudaStream_t stream, DeviceInfo* dev) {
  std::lock_guard<std::mutex> lock(g_csc_build);
  if (e->prod_tried || e->bucket_rows > most_rows || stream_captures(stream)) return B200SP_OK;
  if (nnz <= 0 || nnz > ((int64_t)1 << 26)) { e->prod_tried = true; return B200SP_OK; }
  const CscSizes sizes = csc_sizes(m, nnz, dev->sms);
  const bool smaller = sizes.shift == 13 && nnz < (int64_t)dev->sms * 8 * 4096;
  int rc = csc_places(e, m, n, nnz, col_ptr, row_idx, sizes.tile, sizes.shift, smaller ? csc_most_bucket_rows(nnz, 1.0f) : most_rows, stream, dev);
  if (rc == B200SP_OK && smaller && !e->prod_block) rc = csc_places(e, m, n, nnz, col_ptr, row_idx, sizes.tile, 12, most_rows, stream, dev);
  return rc;
}

// Gives back the memory of the places, in stream order (the calls of a pattern do not overlap); the next SpMV builds them again.
static bool csc_drop_products(CscEntry* e, cudaStream_t stream) {
  std::lock_guard<std::mutex> lock(g_csc_build);
  if (!e->prod_block || stream_captures(stream)) return false;
  if (cudaFreeAsync(e->prod_block, stream) != cudaSuccess) { (void)cudaGetLastError(); return false; }
  e->prod_block = nullptr;
  e->prod_tried = false;
  return true;
}

template <typename T, int TILE, int THREADS>
static int launch_csc_products(const CscEntry* e, int64_t nnz, const T* vals, const T* x, cudaStream_t stream, DeviceInfo* dev) {
  auto kernel = csc_products_kernel<T, TILE, THREADS>;
  const size_t smem = (size_t)e->tile * 4 + (size_t)e->buckets * 4;
  CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCscMaxTile * 4 + kCscMaxBuckets * 4));
  tl_pdl_kernel = true;
  return launch_smem(kernel, dim3((unsigned)e->tiles), dim3(THREADS), smem, stream, nullptr, 0, dev, (int)nnz, e->buckets, vals, x,
                     (const unsigned short*)e->dcol, (const int*)e->tile_col, (const unsigned short*)e->src, (const unsigned short*)e->run_before,
                     (const int*)e->run_shift, e->prod);
}

// SpMV by products: two launches.
template <typename T>
static int run_csc_products(const CscEntry* e, int64_t nnz, const T* vals, const T* x, T* y, float alpha, float beta, cudaStream_t stream, DeviceInfo* dev) {
  int rc;
  switch (e->tile) {
    case 2048: rc = launch_csc_products<T, 2048, 512>(e, nnz, vals, x, stream, dev); break;
    case 4096: rc = launch_csc_products<T, 4096, 512>(e, nnz, vals, x, stream, dev); break;
    case 8192: rc = launch_csc_products<T, 8192, 512>(e, nnz, vals, x, stream, dev); break;
    case 24576: rc = launch_csc_products<T, 24576, 1024>(e, nnz, vals, x, stream, dev); break;
    case 28672: rc = launch_csc_products<T, 28672, 1024>(e, nnz, vals, x, stream, dev); break;
    default: rc = launch_csc_products<T, 32768, 1024>(e, nnz, vals, x, stream, dev); break;
  }
  if (rc != B200SP_OK) return rc;
  auto kernel = csc_bucket_sums_kernel<T>;
  const size_t smem = (size_t)(e->cap + e->cap / 32 + 2) * 4 + (size_t)(e->cap / (kCscShortRow + 1) + 1) * 4;
  CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
  tl_pdl_kernel = true;
  return launch_smem(kernel, dim3((unsigned)e->buckets), dim3(kCscThreads), smem, stream, nullptr, 0, dev, e->cap, (const int*)e->bucket_row,
                     (const int*)e->bucket_start, (const int*)e->row_ptr, (const float*)e->prod, (const unsigned short*)e->dst, y, alpha, beta);
}

// SpMM in a capture before any plan of the row offsets exists (the pattern has only been used for SpMV): the statistics cannot be read back,
// and the nnz-balanced kernel needs none.
template <typename T, int VEC>
static int csc_spmm_without_plan(int64_t m, int64_t n, int64_t nnz, int64_t k, const int32_t* row_ptr, const int32_t* col, const T* vals, const void* B,
                                 void* Y, float alpha, float beta, int dtype, cudaStream_t stream, DeviceInfo* dev) {
  b200sp_plan p;
  CU(cudaGetDevice(&p.device));
  p.row_ptr = row_ptr;
  p.info.m = m; p.info.n = n; p.info.nnz = nnz;
  const int rc = check_common(&p, col, vals, B, Y, dtype);
  if (rc != B200SP_OK) return rc;
  if (k >= ((int64_t)1 << 31) || m * k >= ((int64_t)1 << 40)) return B200SP_ERR_INVALID_ARG;
  if (alpha == 0.0f || nnz == 0) return run_scale<T>((long long)m * k, (T*)Y, beta, stream, dev);
  if (!spmm_offsets_fit(k, (int)sizeof(T))) return B200SP_ERR_UNSUPPORTED;
  return run_spmm_merge<T, VEC>(&p, (int)k, col, vals, (const T*)B, (T*)Y, alpha, beta, stream, dev);
}

static int csc_call(bool is_mm, int64_t m, int64_t n, int64_t nnz, int64_t k, const int32_t* col_ptr, const int32_t* row_idx, const void* vals,
                    const void* in, void* out, float alpha, float beta, int dtype, void* stream_v) {
  int rc = check_sizes(m, n, nnz);
  if (rc != B200SP_OK) return rc;
  if (dtype != B200SP_F32 && dtype != B200SP_BF16) return B200SP_ERR_INVALID_ARG;
  if (k <= 0) return B200SP_ERR_INVALID_ARG;
  if (!col_ptr || (nnz > 0 && (!row_idx || !vals))) return B200SP_ERR_INVALID_ARG;
  if (m == 0) return B200SP_OK;
  DeviceInfo* dev = nullptr;
  rc = device_info(&dev);
  if (rc != B200SP_OK) return rc;
  cudaStream_t stream = (cudaStream_t)stream_v;
  CscEntry* entry = nullptr;
  rc = csc_plan(&entry, m, n, nnz, col_ptr, row_idx, stream);
  if (rc != B200SP_OK) return rc;
  if (!is_mm && nnz > 0 && alpha != 0.0f && in && out && aligned16(vals) && aligned16(in) && aligned16(out)) {
    const int64_t most_rows = csc_most_bucket_rows(nnz, beta);
    rc = csc_product_part(entry, m, n, nnz, col_ptr, row_idx, most_rows, stream, dev);
    if (rc != B200SP_OK && rc != B200SP_ERR_ALLOC) return rc;   // without memory for the places: the CSR kernels
    if (entry->prod_block && (entry->bucket_rows <= most_rows || (!entry->csr.block && stream_captures(stream))))
      return dtype == B200SP_F32 ? run_csc_products<float>(entry, nnz, (const float*)vals, (const float*)in, (float*)out, alpha, beta, stream, dev)
                                 : run_csc_products<bf16_t>(entry, nnz, (const bf16_t*)vals, (const bf16_t*)in, (bf16_t*)out, alpha, beta, stream, dev);
  }
  CscEntry::Csr e;
  CallBlock own;
  rc = csc_csr_part(entry, &e, &own, m, n, nnz, col_ptr, row_idx, stream, dev);
  if (rc == B200SP_ERR_ALLOC && csc_drop_products(entry, stream)) rc = csc_csr_part(entry, &e, &own, m, n, nnz, col_ptr, row_idx, stream, dev);
  if (rc != B200SP_OK) return rc;
  if (nnz > 0) {
    long long blocks = (nnz + 255) / 256;
    if (blocks > (long long)dev->sms * 16) blocks = (long long)dev->sms * 16;
    rc = dtype == B200SP_F32
             ? launch(csc_permute_vals_kernel<float>, dim3((unsigned)blocks), dim3(256), stream, nullptr, 0, dev, (long long)nnz, (const int*)e.perm, (const float*)vals, (float*)e.vals_t)
             : launch(csc_permute_vals_kernel<bf16_t>, dim3((unsigned)blocks), dim3(256), stream, nullptr, 0, dev, (long long)nnz, (const int*)e.perm, (const bf16_t*)vals, (bf16_t*)e.vals_t);
    if (rc != B200SP_OK) return rc;
  }
  int d = 0;
  CU(cudaGetDevice(&d));
  if (is_mm && own.block && !cache_find(std::make_tuple(d, (const void*)entry->row_ptr, m, n, nnz)))
    return dtype == B200SP_F32 ? csc_spmm_without_plan<float, 4>(m, n, nnz, k, entry->row_ptr, e.col, (const float*)e.vals_t, in, out, alpha, beta, dtype, stream, dev)
                               : csc_spmm_without_plan<bf16_t, 8>(m, n, nnz, k, entry->row_ptr, e.col, (const bf16_t*)e.vals_t, in, out, alpha, beta, dtype, stream, dev);
  return is_mm ? spmm_csr(m, n, nnz, k, entry->row_ptr, e.col, e.vals_t, in, out, alpha, beta, dtype, stream_v)
               : spmv_csr(m, n, nnz, entry->row_ptr, e.col, e.vals_t, in, out, alpha, beta, dtype, stream_v);
}

// ---- ELL front end ----
static int check_ell(int64_t m, int64_t n, int64_t width, const void* col_ids, const void* vals, const void* in, const void* out, int dtype) {
  if (m < 0 || n < 0 || width < 0 || n >= ((int64_t)1 << 31) || m >= ((int64_t)1 << 31) - 1 || width >= ((int64_t)1 << 31)) return B200SP_ERR_INVALID_ARG;
  if (m * width >= ((int64_t)1 << 31)) return B200SP_ERR_INVALID_ARG;
  if (dtype != B200SP_F32 && dtype != B200SP_BF16) return B200SP_ERR_INVALID_ARG;
  if (m > 0 && !out) return B200SP_ERR_INVALID_ARG;
  if (m * width > 0 && (!col_ids || !vals || !in)) return B200SP_ERR_INVALID_ARG;
  if (!aligned16(col_ids) || !aligned16(vals) || !aligned16(in) || !aligned16(out)) return B200SP_ERR_INVALID_ARG;
  return B200SP_OK;
}

template <typename T, int LPR, int VECW>
static int launch_ell_spmv(int64_t m, int width, const int32_t* col_ids, const T* vals, const T* x, T* y, float alpha, float beta,
                           cudaStream_t stream, DeviceInfo* dev) {
  constexpr int THREADS = 128;
  const long long blocks = (m * LPR + THREADS - 1) / THREADS;
  if (blocks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  tl_pdl_kernel = true;
  return launch(spmv_ell_kernel<T, LPR, VECW, THREADS>, dim3((unsigned)blocks), dim3(THREADS), stream, nullptr, 0, dev, (int)m, width, col_ids,
                vals, x, y, alpha, beta);
}

template <typename T>
static int run_ell_spmv(int64_t m, int width, const int32_t* col_ids, const T* vals, const T* x, T* y, float alpha, float beta,
                        cudaStream_t stream, DeviceInfo* dev) {
  if (m == 0) return B200SP_OK;
  if (alpha == 0.0f || width == 0) return run_scale<T>(m, y, beta, stream, dev);
  if (width % 4 != 0 && width <= kRowMaxLen)   // odd widths (stencils): the staged row-direct kernel with implicit row offsets
    return launch_row_direct_ell<T>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  if (width % 4 == 0) {   // 128-bit loads: lanes per row = largest power of two not above width / 4 (at most 32)
    const int q = width / 4;
    if (q >= 32) return launch_ell_spmv<T, 32, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
    if (q >= 16) return launch_ell_spmv<T, 16, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
    if (q >= 8) return launch_ell_spmv<T, 8, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
    if (q >= 4) return launch_ell_spmv<T, 4, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
    if (q >= 2) return launch_ell_spmv<T, 2, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
    return launch_ell_spmv<T, 1, 4>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  }
  if (width >= 32) return launch_ell_spmv<T, 16, 1>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  if (width >= 12) return launch_ell_spmv<T, 8, 1>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  if (width >= 6) return launch_ell_spmv<T, 4, 1>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  if (width >= 3) return launch_ell_spmv<T, 2, 1>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
  return launch_ell_spmv<T, 1, 1>(m, width, col_ids, vals, x, y, alpha, beta, stream, dev);
}

template <typename T, int VEC>
static int run_ell_spmm(int64_t m, int width, int k, const int32_t* col_ids, const T* vals, const T* B, T* Y, float alpha, float beta,
                        cudaStream_t stream, DeviceInfo* dev) {
  if (m == 0) return B200SP_OK;
  if (alpha == 0.0f || width == 0) return run_scale<T>((long long)m * k, Y, beta, stream, dev);
  if (k % VEC == 0) {
    constexpr int KS = 8 * VEC, GROUPS = kSpmmThreads / 8;
    const int slices = (k - 1) / KS + 1;
    const int row_blocks = (int)((m + GROUPS - 1) / GROUPS);
    if ((long long)slices * row_blocks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
    return launch(spmm_ell_slice_kernel<T, VEC, kSpmmThreads>, dim3((unsigned)(slices * row_blocks)), dim3(kSpmmThreads), stream, nullptr, 0, dev,
                  (int)m, k, width, row_blocks, col_ids, vals, B, Y, alpha, beta);
  }
  const long long blocks = ((long long)m * k + 255) / 256;
  if (blocks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  return launch(spmm_ell_entry_kernel<T>, dim3((unsigned)blocks), dim3(256), stream, nullptr, 0, dev, (long long)m, k, width, col_ids, vals, B, Y,
                alpha, beta);
}

