// Host side of libb200sp.so: SpMM kernel selection and launches.
// One of the pieces of the single translation unit b200sp.cu; include/b200sp.h states the contract of every entry point.
#pragma once
#include "host_spmv.cuh"
#include "spmm_kernels.cuh"
#include "spmm_bstage_kernels.cuh"
#include "spmm_merge_kernels.cuh"
#include "spmm_bundle_kernels.cuh"
#include "format_kernels.cuh"

namespace {

// Rows of at most kLongRow nonzeros by one lane group each; longer rows by a CTA per (row, 8 * VEC columns).
template <typename T, int VEC, int LANES, int NCH>
int launch_spmm(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                cudaStream_t stream, DeviceInfo* dev) {
  const b200sp_plan_info_t& I = p->info;
  constexpr int GROUPS = kSpmmThreads / LANES;
  const unsigned grid = (unsigned)((I.m + GROUPS - 1) / GROUPS);
  b200sp_plan::RowLists lists;
  CallBlock own_lists;
  int rc = plan_row_lists(p, &lists, &own_lists, stream, dev);
  if (rc != B200SP_OK) return rc;
  tl_pdl_kernel = true;
  rc = launch(spmm_row_group_kernel<T, VEC, LANES, NCH, kSpmmThreads>, dim3(grid), dim3(kSpmmThreads), stream, B,
                  (size_t)I.n * k * sizeof(T), dev, (int)I.m, k, p->row_ptr, col_idx, vals, B, Y, alpha, beta, kLongRow);
  if (rc != B200SP_OK || p->num_long == 0) return rc;
  const long long ctas = (long long)((k - 1) / (8 * VEC) + 1) * p->num_long;
  if (ctas >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  tl_pdl_kernel = true;
  return launch(spmm_long_row_kernel<T, VEC, kSpmmThreads>, dim3((unsigned)ctas), dim3(kSpmmThreads), stream, nullptr, 0, dev, k, p->num_long,
                lists.longer, p->row_ptr, col_idx, vals, B, Y, alpha, beta);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn tensor_map_encoder() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!tried) {
    tried = true;
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
    else
      (void)cudaGetLastError();
  }
  return fn;
}

// B slice in shared memory: used when A has few enough columns and every row of B is re-used often enough.
template <typename T, int VEC, int LANES, int THREADS = 1024>
int launch_spmm_bstage(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                       cudaStream_t stream, DeviceInfo* dev, EncodeTiledFn encode) {
  const b200sp_plan_info_t& I = p->info;
  constexpr int KS = LANES * VEC, ROW_BYTES = LANES * 16;
  const int box_rows = I.n < 256 ? (int)I.n : 256;
  const int boxes = (int)((I.n + box_rows - 1) / box_rows);
  const size_t bslice = (((size_t)boxes * box_rows * ROW_BYTES) + 127) & ~(size_t)127;
  // what the slice of B leaves of the SM's shared memory is split among the warps as staging buffers for their (col, val) pairs
  const size_t limit = (size_t)kSmemPerSm - 2048;
  int capw = 0;
  if (g_opt.bstage_stage_a && bslice < limit) {
    const size_t per_warp = (limit - bslice) / (THREADS / 32);
    const long long entries = (long long)(per_warp / (4 + sizeof(T))) & ~7LL;
    if (entries >= 72) capw = (int)(entries > 4096 ? 4096 : entries) - 4;
  }
  const size_t smem = bslice + (capw > 0 ? (size_t)(THREADS / 32) * (capw + 4) * (4 + sizeof(T)) : 0);
  CUtensorMap map;
  const cuuint64_t gdim[2] = {(cuuint64_t)k, (cuuint64_t)I.n};
  const cuuint64_t gstride[1] = {(cuuint64_t)k * sizeof(T)};
  const cuuint32_t box[2] = {(cuuint32_t)KS, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult cr = encode(&map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<T*>(B), gdim,
                             gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) return B200SP_ERR_UNSUPPORTED;
  auto kernel = spmm_bstage_kernel<T, VEC, LANES, THREADS>;
  static bool configured[64] = {};
  if (!configured[p->device]) {
    CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm - 2048));
    configured[p->device] = true;
  }
  const int slices = (k - 1) / KS + 1;
  const int per_cta = g_opt.bstage_nnz > 0 ? g_opt.bstage_nnz : 131072;
  long long chunks = (I.nnz + per_cta - 1) / per_cta;   // a given number of nonzeros per CTA ...
  const long long fill = (2LL * dev->sms + slices - 1) / slices;   // ... but at least two CTAs per SM over the grid
  if (chunks < fill) chunks = fill;
  if (chunks > I.m) chunks = I.m;
  if (chunks < 1) chunks = 1;
  const int rows_per_chunk = (int)((I.m + chunks - 1) / chunks);
  const int row_chunks = (int)((I.m + rows_per_chunk - 1) / rows_per_chunk);
  if ((long long)slices * row_chunks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  int rc = ensure_err_flag(dev);
  if (rc != B200SP_OK) return rc;
  tl_pdl_kernel = true;
  return launch_smem(kernel, dim3((unsigned)(slices * row_chunks)), dim3(THREADS), smem, stream, nullptr, 0, dev, map, (int)I.m, (int)I.n,
                     k, row_chunks, rows_per_chunk, box_rows, (int)bslice, capw, p->row_ptr, col_idx, vals, Y, alpha, beta, dev->err_flag,
                     g_opt.spin_limit, g_opt.debug_no_copies);
}

// Exclusive scan of `count` ints in place; bsum: (count + kScanBlock - 1) / kScanBlock + 1 ints of scratch.  Three launches.
int device_scan_in_place(int* data, long long count, int* bsum, cudaStream_t stream) {
  const long long blocks = (count + kScanBlock - 1) / kScanBlock;
  if (blocks < 1 || blocks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  scan_block_sums_kernel<<<(unsigned)blocks, 256, 0, stream>>>(data, count, bsum);
  plan_compact_scan_kernel<<<1, 1024, 0, stream>>>(bsum, (int)blocks);
  scan_apply_kernel<<<(unsigned)blocks, 256, 0, stream>>>(data, count, bsum, data);
  g_launches += 3;
  CU(cudaGetLastError());
  return B200SP_OK;
}

// The processing order of spmm_bstage_quads_kernel (see plan_kernels.cuh), built once per plan and lane-group width, on the
// device and in stream order: no synchronisation.  B200SP_ERR_UNSUPPORTED when the positions would not fit 32 bits.
int plan_quad_order(b200sp_plan* p, int gpw, b200sp_plan::QuadOrder* out, CallBlock* own, cudaStream_t stream, DeviceInfo* dev) {
  static_assert(kLongRow == 1024, "quad_key() assumes rows of at most 1024 nonzeros");
  b200sp_plan::QuadOrder& Q = p->quad[gpw == 4 ? 0 : gpw == 8 ? 1 : 2];   // rows per warp: 4, 8 or 16
  std::lock_guard<std::mutex> lock(p->build);
  if (Q.block) { *out = Q; return B200SP_OK; }
  const b200sp_plan_info_t& I = p->info;
  const long long listed = I.m - p->num_long;
  const long long blocks = (listed + gpw - 1) / gpw;
  if ((I.nnz + 3 * I.m) / 4 + (long long)(kLongRow / 4 + 2) * gpw >= (1LL << 31) - 64 || blocks < 1) return B200SP_ERR_UNSUPPORTED;
  long long rows_per_blk = (I.m + 65535) / 65536;
  if (rows_per_blk < 256) rows_per_blk = 256;
  rows_per_blk = (rows_per_blk + 31) / 32 * 32;
  const long long nblk = (I.m + rows_per_blk - 1) / rows_per_blk;
  const long long slots = blocks * gpw, table = (long long)kQuadKeys * nblk;
  const long long scan_len = table > blocks + 1 ? table : blocks + 1;
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t o_row = 0, o_len = up((size_t)slots * 4), o_pos = o_len + up((size_t)slots * 4), keep = o_pos + up((size_t)(blocks + 1) * 4);
  void* blk = nullptr;
  void* tmp = nullptr;      // the histogram table and the scan's block sums: only needed while the order is built
  int rc = pool_alloc(dev, &blk, keep, stream);
  if (rc != B200SP_OK) return rc;
  rc = pool_alloc(dev, &tmp, up((size_t)table * 4) + up((size_t)(scan_len / kScanBlock + 2) * 4), stream);
  if (rc != B200SP_OK) { cudaFreeAsync(blk, stream); return rc; }
  int* row_of = (int*)((char*)blk + o_row);
  int* len_of = (int*)((char*)blk + o_len);
  int* pos = (int*)((char*)blk + o_pos);
  int* hist = (int*)tmp;
  int* bsum = (int*)((char*)tmp + up((size_t)table * 4));
  auto fail = [&](int code) { cudaFreeAsync(tmp, stream); cudaFreeAsync(blk, stream); return code; };
#define CUQ(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return fail(cuda_fail(e_, #call)); } while (0)
  CUQ(cudaMemsetAsync(row_of, 0xFF, (size_t)slots * 4, stream));      // unused slots: row -1, length 0
  CUQ(cudaMemsetAsync(len_of, 0, (size_t)slots * 4, stream));
  const unsigned grid = (unsigned)((nblk + 3) / 4);
  quad_order_hist_kernel<<<grid, 128, 0, stream>>>(p->row_ptr, (int)I.m, (int)rows_per_blk, (int)nblk, hist);
  g_launches++;
  CUQ(cudaGetLastError());
  rc = device_scan_in_place(hist, table, bsum, stream);
  if (rc != B200SP_OK) return fail(rc);
  quad_order_scatter_kernel<<<grid, 128, 0, stream>>>(p->row_ptr, (int)I.m, (int)rows_per_blk, (int)nblk, hist, row_of, len_of);
  quad_order_block_quads_kernel<<<(unsigned)((blocks + 1 + 255) / 256), 256, 0, stream>>>(len_of, (int)blocks, gpw, pos);
  g_launches += 2;
  CUQ(cudaGetLastError());
  rc = device_scan_in_place(pos, blocks + 1, bsum, stream);
  if (rc != B200SP_OK) return fail(rc);
  CUQ(cudaFreeAsync(tmp, stream));
#undef CUQ
  *out = {blk, row_of, len_of, pos, (int)blocks};
  if (stream_captures(stream)) own->take(blk, stream);
  else Q = *out;
  return B200SP_OK;
}

// The same with the rows in the plan's sorted order and A re-laid once per call into padded quads (spmm_bstage_prep_kernel),
// which the main kernel's warps fetch with bulk copies; rows longer than kLongRow by spmm_long_row_kernel.
template <typename T, int VEC, int SLICE_LANES, int PIECES, bool OLD, int THREADS>
int launch_spmm_bstage_quads_as(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                             cudaStream_t stream, DeviceInfo* dev, EncodeTiledFn encode) {
  const b200sp_plan_info_t& I = p->info;
  constexpr int LANES = SLICE_LANES / PIECES;
  static_assert(LANES == 2 || LANES == 4 || LANES == 8, "one order of the rows for each");
  constexpr int KS = SLICE_LANES * VEC, ROW_BYTES = SLICE_LANES * 16, GPW = 32 / LANES, WARPS = THREADS / 32;
  const int box_rows = I.n < 256 ? (int)I.n : 256;
  const int boxes = (int)((I.n + box_rows - 1) / box_rows);
  const size_t bslice = (((size_t)boxes * box_rows * ROW_BYTES) + 127) & ~(size_t)127;
  // what the slice of B leaves of the SM's shared memory is split among the warps as buffers for their blocks' quads
  // (four 16-bit offsets and four values each)
  constexpr size_t QUAD_BYTES = 8 + 4 * sizeof(T);
  const size_t limit = (size_t)kSmemPerSm - 2048 - 32 * WARPS;
  int capq = 0;
  if (g_opt.bstage_stage_a && bslice < limit) {
    const size_t quads = (limit - bslice) / WARPS / QUAD_BYTES;
    capq = (int)(quads > 2048 ? 2048 : quads) & ~1;
    if (capq < 2 * GPW) capq = 0;
  }
  const size_t smem = bslice + (((size_t)WARPS * capq * QUAD_BYTES + 15) & ~(size_t)15);
  CUtensorMap map;
  const cuuint64_t gdim[2] = {(cuuint64_t)k, (cuuint64_t)I.n};
  const cuuint64_t gstride[1] = {(cuuint64_t)k * sizeof(T)};
  const cuuint32_t box[2] = {(cuuint32_t)KS, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult cr = encode(&map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<T*>(B), gdim,
                             gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) return B200SP_ERR_UNSUPPORTED;
  b200sp_plan::QuadOrder Q;
  CallBlock own_order;
  b200sp_plan::RowLists lists;
  CallBlock own_lists;
  int rc = plan_quad_order(p, GPW, &Q, &own_order, stream, dev);
  if (rc == B200SP_OK) rc = plan_row_lists(p, &lists, &own_lists, stream, dev);
  if (rc != B200SP_OK) return rc;
  auto kernel = spmm_bstage_quads_kernel<T, VEC, LANES, PIECES, OLD, THREADS>;
  static bool configured[64] = {};
  if (!configured[p->device]) {
    CU(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm - 2048));
    configured[p->device] = true;
  }
  const int slices = (k - 1) / KS + 1;
  const int blocks = Q.blocks;
  const long long most = (blocks + WARPS - 1) / WARPS;   // a block per warp at least
  long long chunks;
  if (g_opt.bstage_nnz > 0) {
    chunks = (I.nnz + g_opt.bstage_nnz - 1) / g_opt.bstage_nnz;   // a given number of nonzeros per CTA ...
    const long long fill = (2LL * dev->sms + slices - 1) / slices;   // ... but at least two CTAs per SM over the grid
    if (chunks < fill) chunks = fill;
  } else {
    // One CTA per SM is resident and all CTAs take the same time (each gets the same mix of rows), so the kernel lasts
    // ceil(CTAs / SMs) rounds of (nonzeros per CTA + the fetch of the slice of B, about 4096 nonzeros' worth): the chunk
    // count with the smallest product, among those that leave a CTA at least 8192 nonzeros (or one chunk).
    chunks = 1;
    double best = 0.0;
    for (long long c = 1; c <= 4096 && c <= most && (c == 1 || I.nnz / c >= 8192); ++c) {
      const double rounds = (double)((slices * c + dev->sms - 1) / dev->sms);
      const double cost = rounds * ((double)I.nnz / (double)c + 4096.0);
      if (c == 1 || cost < best) { best = cost; chunks = c; }
    }
  }
  if (chunks > most) chunks = most;
  if (chunks < 1) chunks = 1;
  const int row_chunks = (int)chunks;
  if ((long long)slices * row_chunks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  rc = ensure_err_flag(dev);
  if (rc != B200SP_OK) return rc;
  // the per-call copy of A: at most the rows' quads plus (kLongRow / 4 + 2) * GPW of padding where the length changes along the list
  const size_t entries = (((size_t)((I.nnz + 3 * I.m) / 4) + (size_t)(kLongRow / 4 + 2) * GPW) * 4 + 15) & ~(size_t)7;
  void* scratch = nullptr;
  const long long slots = (long long)blocks * GPW;
  // 64-byte rows of the slice: the copy of A changes the order of a block's rows to have fewer bank conflicts, if there are slices and rows enough
  // to pay for it (2^14 rows of 20: 8 slices 18.5 us without, 19.5 us with; 16 slices 27.5 / 27.7; 256 slices 276 / 258; 2^15 rows, 32 slices
  // 85.1 / 83.0; 2^11 rows, 32 slices 12.1 / 12.6; 11,782 rows, 33 slices 46.0 / 46.7)
  const bool reorder = ROW_BYTES == 64 && slices >= 24 && (long long)slices * I.m >= (1 << 19);
  rc = pool_alloc(dev, &scratch, entries * (2 + sizeof(T)) + (reorder ? (size_t)slots * 8 : 0), stream);
  if (rc != B200SP_OK) return rc;
  unsigned short* qoff = (unsigned short*)scratch;       // entries 16-bit offsets, then entries values (16-byte aligned: entries is a multiple of 8)
  T* qval = (T*)((char*)scratch + entries * 2);
  int* const new_row = reorder ? (int*)((char*)scratch + entries * (2 + sizeof(T))) : nullptr;
  int* const new_len = reorder ? new_row + slots : nullptr;
  tl_pdl_kernel = true;
  rc = launch(spmm_bstage_prep_kernel<T, ROW_BYTES>, dim3((unsigned)((slots * 8 + 255) / 256)), dim3(256), stream, nullptr, 0, dev, (int)slots, GPW,
              Q.row, Q.pos, p->row_ptr, col_idx, vals, qoff, qval, (int)reorder, new_row, new_len);
  if (rc == B200SP_OK) {
    tl_pdl_kernel = true;
    rc = launch_smem(kernel, dim3((unsigned)(slices * row_chunks)), dim3(THREADS), smem, stream, nullptr, 0, dev, map, (int)I.n, k, row_chunks,
                     blocks, box_rows, (int)bslice, capq, (const int*)(reorder ? new_row : Q.row), (const int*)(reorder ? new_len : Q.len), Q.pos,
                     (const unsigned short*)qoff, (const T*)qval, Y, alpha, beta, dev->err_flag, g_opt.spin_limit, g_opt.debug_no_copies);
  }
  const cudaError_t e = cudaFreeAsync(scratch, stream);
  if (e != cudaSuccess && rc == B200SP_OK) rc = cuda_fail(e, "cudaFreeAsync");
  if (rc == B200SP_OK && p->num_long > 0) {
    const long long ctas = (long long)((k - 1) / (8 * VEC) + 1) * p->num_long;
    if (ctas >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
    tl_pdl_kernel = true;
    rc = launch(spmm_long_row_kernel<T, VEC, kSpmmThreads>, dim3((unsigned)ctas), dim3(kSpmmThreads), stream, nullptr, 0, dev, k, p->num_long,
                lists.longer, p->row_ptr, col_idx, vals, B, Y, alpha, beta);
  }
  return rc;
}

// Pieces of 16 bytes per lane and row: two where the slice has at least 64 bytes a row and the warps of all SMs get a step at least (half as
// many reads of A and half as many address instructions per product).  2^16 rows of 20 x 4096 FP32 1017 us with two, 1092 us with one; 2^14 rows
// of 10 (128-byte slices) 156 / 203 us; but 2^10 rows x 256 columns, 1024 steps, 12.1 / 10.8 us.  BF16 with 16 columns a lane wants
// 80 registers: 768 threads (512 threads 285 us, 768 threads 270 us on 2^16 rows x 2048 columns, one piece 308 us).  With beta != 0 the old
// values of Y take registers too and the CTAs are smaller (640 threads BF16: 186 us, 704 197, 768 203, one piece 197, 2^14 rows x 4096), which
// pays from some ten steps a warp on (2^14 rows of 20 x 1024 BF16 56.4 / 60.2 us; 11,782 x 1048, eight steps, 46.7 / 45.6 us).
template <typename T, int VEC, int SLICE_LANES, int THREADS>
int launch_spmm_bstage_quads(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                             cudaStream_t stream, DeviceInfo* dev, EncodeTiledFn encode) {
  if constexpr (SLICE_LANES >= 4 && THREADS == 1024) {
    const long long slices = (k - 1) / (SLICE_LANES * VEC) + 1, steps = (p->info.m * SLICE_LANES / 64 + 1) * slices;
    if (beta == 0.0f && steps >= 32LL * dev->sms)
      return launch_spmm_bstage_quads_as<T, VEC, SLICE_LANES, 2, false, sizeof(T) == 2 ? 768 : 1024>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);
    if (beta != 0.0f && steps >= 192LL * dev->sms)
      return launch_spmm_bstage_quads_as<T, VEC, SLICE_LANES, 2, true, sizeof(T) == 2 ? 640 : 768>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);
  }
  return launch_spmm_bstage_quads_as<T, VEC, SLICE_LANES, 1, false, THREADS>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);
}

// Column ranges for the k-sliced kernel: how many, and the per-row cut positions (computed once per col_idx; one small
// kernel and one synchronisation of the stream).  Returns 1 in *ranges when the ranges do not apply: B's slice fits L2,
// the rows' columns are not in ascending order, or the switch says so.
int spmm_column_ranges(b200sp_plan* p, const int32_t* col_idx, int slice_bytes, cudaStream_t stream, DeviceInfo* dev, int* ranges) {
  const b200sp_plan_info_t& I = p->info;
  *ranges = 1;
  int want = g_opt.spmm_ranges;
  if (want == 0) {
    // a range of B (n / ranges rows of slice_bytes) should take at most this share of L2: the L2 of this part keeps a line
    // read by all SMs in both of its halves, and the streams of A and Y pass through it as well
    const double budget = 0.3 * (double)dev->l2_bytes;
    want = (int)(((double)I.n * slice_bytes + budget - 1) / budget);
    if (want > 8) want = 8;
  }
  if (want <= 1 || I.n < want || I.m < 1) return B200SP_OK;
  if (p->cuts_col_idx == (const void*)col_idx && p->cuts_ranges == want) { if (p->cols_sorted) *ranges = want; return B200SP_OK; }
  if (p->cuts_block) { CU(cudaFreeAsync(p->cuts_block, stream)); p->cuts_block = nullptr; p->cuts_ranges = 0; p->cuts_col_idx = nullptr; }
  const size_t bytes = (size_t)(want - 1) * (size_t)I.m * 4 + 256;
  void* blk = nullptr;
  int rc = pool_alloc(dev, &blk, bytes, stream);
  if (rc != B200SP_OK) return rc;
  int* flag = (int*)((char*)blk + (size_t)(want - 1) * (size_t)I.m * 4);
  int h = 0;
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), stream);
  if (e == cudaSuccess) {
    spmm_range_cuts_kernel<<<(unsigned)((I.m + 255) / 256), 256, 0, stream>>>((int)I.m, (int)I.n, want, p->row_ptr, col_idx, (int*)blk, flag);
    g_launches++;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) { cudaFreeAsync(blk, stream); return cuda_fail(e, "column ranges"); }
  p->cuts_block = blk;
  p->cuts_col_idx = col_idx;
  p->cuts_ranges = want;
  p->cols_sorted = h == 0;
  if (p->cols_sorted) *ranges = want;
  return B200SP_OK;
}

bool spmm_rows_are_uneven(const b200sp_plan_info_t& I) {
  if (I.nnz <= 0 || I.m <= 0) return false;
  const int64_t nonempty = I.m - I.bin_rows[0];
  const double mean = (double)I.nnz / (double)(nonempty > 0 ? nonempty : 1);
  return (I.bin_nnz[4] + I.bin_nnz[5]) * 20 >= I.nnz      // 5 % or more of the nonzeros sit in rows longer than 128
         || I.bin_rows[0] * 4 >= I.m                        // a quarter or more of the rows are empty
         || (double)I.max_row_len > 4.0 * mean + 8.0;       // or the longest row is far above the mean
}

// Uneven rows and few columns: whether the kernels by rows are faster than shares, by a model of both times in us.  A warp of the nnz-balanced
// kernel takes a nonzero at a time however few columns there are, so its time is that of the rows + nonzeros.  By rows a nonzero costs less
// the fewer lanes hold its row, more where the rows of a warp differ (spread: mean length over the nonzeros, by length bins, over the mean
// length), and the longest row walked by one lane group is a chain; rows of 129-1024 nonzeros (aligned k) and longer ones are launches apart.
// Constants: least squares over log-normal rows (means 4 .. 40, sigma 0.7 .. 1.2, 5000 .. 2 M rows) and even rows with a few long ones, both
// dtypes, beta = 0 and 1, 1268 points (rms error 0.2 in the logarithm).  Of the 444 that go by rows 8 are slower by 5 % than by shares, by 10 % at
// most; of those that go by shares 104 are slower by 5 % than by rows.  By rows / shares in us: 600,000 log-normal rows of 12, FP32 k = 2
// 76 / 116, k = 3 91 / 117, k = 8 155 / 117, BF16 k = 2 89 / 135, k = 16 142 / 136; 20,011 rows of 10, k = 2 21.5 / 10.6; 600,000 rows of 8 and one of
// 3000, k = 2 41 / 89, k = 8 49 / 90; R-MAT 2^20 (spread above 30) k = 2 359 / 140, k = 16 465 / 146.
bool spmm_uneven_by_rows(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  const int vec = 16 / elem_bytes;
  if (k > (k % vec == 0 ? 4 * vec : 16) || I.bin_rows[0] * 4 >= I.m) return false;
  const double m = 1e-6 * (double)I.m, nnz = 1e-6 * (double)I.nnz;
  double squares = 0.0;
  for (int j = 1; j < B200SP_NUM_BINS; ++j)
    if (I.bin_rows[j] > 0) squares += (double)I.bin_nnz[j] * (double)I.bin_nnz[j] / (double)I.bin_rows[j];
  const double spread = squares * (double)I.m / ((double)I.nnz * (double)I.nnz);
  if (spread > (k % vec == 0 && k > 2 * vec ? 1.5 : 2.6) || (I.bin_rows[4] > 0 && I.bin_rows[5] > 0)) return false;
  const int longest = I.max_row_len, medium = I.bin_rows[4] > 0 ? longest : 0;
  const int shortest = longest <= 128 ? longest : 128;
  double rows;
  if (k % vec == 0) {
    rows = std::max(nnz * (4.4 + 3.2 * (double)(k / vec)) * (1.0 + 0.34 * (spread - 1.0)), 0.09 * shortest) + 0.09 * medium;
  } else {
    int lanes = 2;
    while (lanes < k) lanes *= 2;
    rows = std::max(nnz * (3.9 + 1.15 * lanes) * (1.0 + 0.77 * (spread - 1.0)), 0.088 * std::max(shortest, medium)) * (elem_bytes == 4 ? 1.0 : 1.2);
  }
  rows += 5.0 + (longest > 1024 ? 0.005 * longest : 0.0);
  const double shares = 8.6 + nnz * (elem_bytes == 4 ? 11.8 : 14.3) + m * (beta != 0.0f ? 75.0 : 40.0);
  return 1.05 * rows < shares;
}

// The nnz-balanced kernel counts the bytes of a row of B, and columns past k up to a slice, in 32 bits.
bool spmm_offsets_fit(int64_t k, int elem_bytes) { return k <= (INT32_MAX - 2048) / elem_bytes; }

// Whether SpMM goes by equal shares (spmm_merge_kernel): uneven rows (see above), and k that is no multiple of 16 bytes unless it is so narrow
// that a lane per column and a group of lanes per row lose little (100,000 rows of 13: k = 13 18 us by rows, 27 us by shares; k = 23 35 / 27 us;
// k = 50 47 / 35 us FP32, 42 / 34 us BF16).
bool spmm_by_shares(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  if (!spmm_offsets_fit(k, elem_bytes) || !g_opt.spmm_sliced) return false;
  if (g_opt.spmm_flat != 2) return g_opt.spmm_flat == 1;
  if (k % (16 / elem_bytes) != 0 && k > 16) return true;
  return spmm_rows_are_uneven(I) && !spmm_uneven_by_rows(I, k, elem_bytes, beta);
}

// Even rows of A, BF16, rows of B in whole 32-byte pieces and at least 64 columns of them (narrower slices, 16 / 32 bytes a lane on 2^18 rows: k = 32
// 31.8 / 33.6 us, k = 16 24.1 / 26.6 us): whether four lanes a row with 32 bytes of B per load (spmm_slice_wide_kernel) are faster than eight with 16
// and staged pairs.  Per nonzero they are; what they lose by are single steps, which rows take up to a multiple of four nonzeros at both ends
// ("quads": no row does), and half as many warps where few blocks are left.  Times: 16 / 32 bytes a lane, us; waves: blocks over those resident.
// - Other rows than quads only while a slice of B takes less than half of L2, where loads do not wait for memory (rows of 13, k = 64: 350,000 of them
//   78.1 / 74.5, 450,000 102.9 / 100.6, 550,000 130 / 132, 2^20 286 / 303; rows of 6, 550,000 86.0 / 88.4; but 2^20 rows of 16, k = 128 514 / 491).
// - Other rows than quads of up to 25 nonzeros: the shorter ones from a quarter of a wave on (8000 of 5 to 15, k = 64 5.1 / 5.2; 20,000 9.6 / 7.4),
//   and those of less than 5 and mixed lengths up to three waves (100,000 of 2 to 6, k = 64 16.2 / 14.8, k = 128 31.3 / 32.2).
// - Of 26 to 32: where the blocks are one wave or many (20,000 of 20 to 36, k = 64 16.5 / 14.3, k = 128 18.5 / 20.2; 100,000, k = 192 103 / 99).
// - Rows of more than 32, whose pairs the staged kernel's warps read from memory as well: quads, and rows of clearly different lengths, except where
//   blocks wait for a second or a third wave (k = 128, 26,000 rows of 64 32.1 / 36.8, 16,000 23.8 / 21.5, 54,000 59.4 / 53.8; 20,000 of 64 to 128,
//   k = 192 65.4 / 71.5, 100,000 282 / 247); not others of one length (20,000 of 33, k = 256 31.5 / 35.3, of 65 53.9 / 61.5).
bool spmm_wide_pieces(const b200sp_plan_info_t& I, int64_t k, int sms, int64_t l2_bytes) {
  const bool equal = I.min_row_len == I.max_row_len, quads = equal && I.max_row_len % 4 == 0;
  if (!quads && (double)I.n * 128.0 > 0.45 * (double)l2_bytes) return false;
  const double mean = I.m > 0 ? (double)I.nnz / (double)I.m : 0.0;
  const double waves = (double)((k + 63) / 64) * (double)((I.m + 31) / 32) / (8.0 * sms);      // 64 columns, 32 rows a block; eight of them per SM
  if (quads && I.max_row_len <= 32) return true;
  if (!quads && mean <= 25.0) return (waves >= 0.25 || mean >= 20.0) && (equal || mean >= 5.0 || waves <= 3.0);
  if (!quads && mean <= 32.0) return waves <= 1.0 || waves >= 4.0;
  return (quads || 2 * I.max_row_len >= 3 * I.min_row_len) && (waves <= 1.0 || waves >= 2.6);
}

// alpha * 0 + beta * y for rows without nonzeros as one number: the factor of y, or the value itself with beta == 0.
float spmm_none(float alpha, float beta) { return beta == 0.0f ? alpha * 0.0f : std::isfinite(alpha) ? beta : std::numeric_limits<float>::quiet_NaN(); }

template <typename T, int V, int J, int MODE>
int launch_spmm_merge_as(b200sp_plan* p, const b200sp_plan::Shares& work, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                      cudaStream_t stream, DeviceInfo* dev) {
  const b200sp_plan_info_t& I = p->info;
  constexpr int KS = 32 * V * J;
  const int witems = work.witems;
  auto kernel = spmm_merge_kernel<T, V, J, MODE>;
  static int per_sm[64] = {};   // per instantiation and device: resident CTAs
  if (!per_sm[p->device]) {
    int nb = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kMergeWarps * 32, 0));
    per_sm[p->device] = nb > 0 ? nb : 1;
  }
  // Shares per warp, by a model of the time: a wave of resident warps costs their items and about 40 more (what a warp does before its first
  // and after its last nonzero); the last of several waves is, on average, a third full, and a single wave has nothing to fill in behind
  // its slower warps.  40,000 rows of 20, k = 256 FP32 with a fresh plan: 131 us with two shares (one wave), 149 us with one (1.8 waves);
  // 100,000 rows of 12, k = 127: 84 us with one (1.7 waves), 94 us with two; 155,787 rows of 12, k = 96: 80 us with two, 84 us with one.
  int shares = 1;
  {
    const double resident = (double)per_sm[p->device] * dev->sms * kMergeWarps, total = (double)(I.m + I.nnz) / witems;
    double best = 0.0;
    for (int s = 1; s <= kMergeShares; ++s) {
      const double waves = total / (s * resident), cost = (s * witems + 40.0) * (waves > 0.95 ? waves + 0.35 : 1.15);
      if (s == 1 || cost < best) { best = cost; shares = s; }
    }
  }
  const long long per_tile = (long long)witems * shares * kMergeWarps;
  const int tiles = (int)((I.m + I.nnz + per_tile - 1) / per_tile);
  const int slices = (k - 1) / KS + 1;
  if ((long long)slices * tiles >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
  // per-call scratch: what each tile leaves unfinished and what it finishes for an earlier tile, KS floats per (slice, tile)
  float* scratch = nullptr;
  const size_t per = (size_t)slices * tiles * KS;
  int rc = pool_alloc(dev, (void**)&scratch, 2 * per * sizeof(float) + (size_t)tiles * sizeof(int2), stream);
  int2* const tile_row = (int2*)(scratch + 2 * per);
  if (rc != B200SP_OK) return rc;
  tl_pdl_kernel = true;
  rc = launch(kernel, dim3((unsigned)(slices * tiles)), dim3(kMergeWarps * 32), stream, B, (size_t)I.n * k * sizeof(T), dev,
              (int)I.m, (int)I.nnz, k, tiles, witems, shares, work.split, p->row_ptr, col_idx, vals, B, Y, scratch, scratch + per, tile_row, alpha, beta, spmm_none(alpha, beta));
  if (rc == B200SP_OK && tiles > 1) {
    tl_pdl_kernel = true;
    const int lanes = KS >= 128 ? 128 : KS;      // a power of two
    rc = launch(spmm_merge_fixup_kernel<T>, dim3((unsigned)(((long long)slices * tiles * lanes + 255) / 256)), dim3(256), stream, nullptr, 0, dev, k,
                tiles, slices, KS, lanes, (const int2*)tile_row, (const float*)scratch, (const float*)(scratch + per), Y, alpha, beta);
  }
  const cudaError_t e = cudaFreeAsync(scratch, stream);
  if (e != cudaSuccess && rc == B200SP_OK) rc = cuda_fail(e, "cudaFreeAsync");
  return rc;
}

// beta != 0 and one row in sixteen or more without nonzeros: these are listed and scaled apart (R-MAT 2^21, k = 64 BF16, 61 % empty: 458 us
// against 657 us; with beta == 0 the listing costs as much as it saves).  Otherwise Y's old values are asked for a row ahead.
template <typename T, int V, int J>
int launch_spmm_merge(b200sp_plan* p, const b200sp_plan::Shares& work, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                      cudaStream_t stream, DeviceInfo* dev) {
  if (beta == 0.0f) return launch_spmm_merge_as<T, V, J, 0>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  return p->info.bin_rows[0] * 16 >= p->info.m ? launch_spmm_merge_as<T, V, J, 2>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev)
                                               : launch_spmm_merge_as<T, V, J, 1>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
}

// nnz-balanced SpMM (spmm_merge_kernel), any k.  The widest pieces (16 bytes per lane at most) that k allows, narrowed while half as
// wide a piece still covers all of k with one load; then as many loads per nonzero as it takes (at most 4) before k is cut into slices.
template <typename T, int VMAX>
int run_spmm_merge(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
                   cudaStream_t stream, DeviceInfo* dev) {
  int v = 1;
  while (v < VMAX && k % (2 * v) == 0 && 32 * v < k) v *= 2;
  b200sp_plan::Shares work;
  CallBlock own_work;
  const int rc = plan_shares(p, &work, &own_work, stream, dev);
  if (rc != B200SP_OK) return rc;
  const int loads = (k - 1) / (32 * v) + 1;
#define B200SP_MERGE_J(V)                                                                                                   \
  do {                                                                                                                      \
    if (loads == 1) return launch_spmm_merge<T, V, 1>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev);                 \
    if (loads == 2) return launch_spmm_merge<T, V, 2>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev);                 \
    return launch_spmm_merge<T, V, (V * sizeof(T) >= 16 ? 2 : 4)>(p, work, k, col_idx, vals, B, Y, alpha, beta, stream, dev);     \
  } while (0)
  if (v == 1) B200SP_MERGE_J(1);
  if (v == 2) B200SP_MERGE_J(2);
  if (v == 4) B200SP_MERGE_J(4);
  if constexpr (VMAX == 8) { if (v == 8) B200SP_MERGE_J(8); }
  return B200SP_ERR_UNSUPPORTED;
#undef B200SP_MERGE_J
}

// Merge items per warp of spmm_bundle_kernel: one wave of resident warps where that takes no more than `most`, else as few waves as that allows, all of them
// full; small matrices fewer warps instead of very short regions.
int bundle_region(int64_t items, int sms, int ctas, int most) {
  const int64_t resident = (int64_t)ctas * kMergeWarps * sms, waves = (items + resident * most - 1) / (resident * most);
  int64_t region = (items + resident * waves - 1) / (resident * waves);
  if (region < most && region < 128) region = std::min((int64_t)std::min(most, 128), std::max((int64_t)24, items / (20 * sms)));
  return (int)((region + 7) / 8 * 8);
}

template <typename T, int LANES, int YV, bool BETA>
int launch_spmm_bundle_as(b200sp_plan* p, const b200sp_plan::Shares& work, int k, int row_bytes, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha,
                          float beta, cudaStream_t stream, DeviceInfo* dev) {
  const b200sp_plan_info_t& I = p->info;
  constexpr int KS = LANES * (16 / (int)sizeof(T)), CTAS = kBundleCtas<T>;
  const int region = bundle_region(I.m + I.nnz, dev->sms, CTAS, bundle_most(LANES));
  const long long per_tile = (long long)region * kMergeWarps;
  const int tiles = (int)((I.m + I.nnz + per_tile - 1) / per_tile);
  float* scratch = nullptr;                      // what each tile leaves unfinished and what it finishes for an earlier tile
  const size_t per = (size_t)tiles * KS;
  int rc = pool_alloc(dev, (void**)&scratch, 2 * per * sizeof(float) + (size_t)tiles * sizeof(int2), stream);
  if (rc != B200SP_OK) return rc;
  int2* const tile_row = (int2*)(scratch + 2 * per);
  tl_pdl_kernel = true;
  rc = launch_smem(spmm_bundle_kernel<T, LANES, YV, BETA>, dim3((unsigned)tiles), dim3(kMergeWarps * 32), (size_t)kMergeWarps * bundle_bytes(region), stream, B,
                   (size_t)I.n * row_bytes, dev, (int)I.m, (int)I.nnz, k, row_bytes, region, work.split, work.witems, p->row_ptr, col_idx, vals, B, Y, scratch,
                   scratch + per, tile_row, alpha, beta, spmm_none(alpha, beta));
  if (rc == B200SP_OK && tiles > 1) {
    tl_pdl_kernel = true;
    const int lanes = KS >= 128 ? 128 : KS;      // a power of two
    rc = launch(spmm_merge_fixup_kernel<T>, dim3((unsigned)(((long long)tiles * lanes + 255) / 256)), dim3(256), stream, nullptr, 0, dev, k, tiles, 1, KS, lanes,
                (const int2*)tile_row, (const float*)scratch, (const float*)(scratch + per), Y, alpha, beta);
  }
  const cudaError_t e = cudaFreeAsync(scratch, stream);
  if (e != cudaSuccess && rc == B200SP_OK) rc = cuda_fail(e, "cudaFreeAsync");
  return rc;
}

// Bytes of a row of the padded copy of B: whole lines (32-byte steps measured the same to 10 % more and less).
int64_t spmm_padded_row(int64_t k, int elem_bytes) { return (k * elem_bytes + 127) / 128 * 128; }

// Columns of Y per store: all of a lane's where k is a multiple of 16 bytes; else B is copied into padded rows first (one kernel and n rows of memory from the
// pool) and Y is written by pairs (even k) or one by one.
template <typename T, int YV>
int run_spmm_bundle(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta, cudaStream_t stream, DeviceInfo* dev) {
  constexpr int VEC = 16 / (int)sizeof(T);
  b200sp_plan::Shares work;
  CallBlock own_work;
  int rc = plan_shares(p, &work, &own_work, stream, dev);
  if (rc != B200SP_OK) return rc;
  T* padded = nullptr;
  int row_bytes = k * (int)sizeof(T);
  if (YV != VEC) {
    row_bytes = (int)spmm_padded_row(k, (int)sizeof(T));
    rc = pool_alloc(dev, (void**)&padded, (size_t)p->info.n * row_bytes, stream);
    if (rc != B200SP_OK) return rc;
    const long long blocks = (p->info.n + 31) / 32;
    tl_pdl_kernel = true;
    rc = launch(spmm_pad_rows_kernel<T>, dim3((unsigned)(blocks < dev->sms * 8 ? blocks : dev->sms * 8)), dim3(256), stream, nullptr, 0, dev, (int)p->info.n, k,
                row_bytes / 4, B, (unsigned*)padded);
    B = padded;
  }
  if (rc == B200SP_OK) {
    const int pieces = (k + VEC - 1) / VEC;
#define B200SP_BUNDLE(L)                                                                                                                       \
    rc = beta == 0.0f ? launch_spmm_bundle_as<T, L, YV, false>(p, work, k, row_bytes, col_idx, vals, B, Y, alpha, beta, stream, dev)               \
                      : launch_spmm_bundle_as<T, L, YV, true>(p, work, k, row_bytes, col_idx, vals, B, Y, alpha, beta, stream, dev)
    if (pieces <= 4) B200SP_BUNDLE(4);
    else if (pieces <= 8) B200SP_BUNDLE(8);
    else if (pieces <= 16) B200SP_BUNDLE(16);
    else if constexpr (sizeof(T) == 4 && YV == VEC) B200SP_BUNDLE(32);
    else rc = B200SP_ERR_UNSUPPORTED;
#undef B200SP_BUNDLE
  }
  if (padded) { const cudaError_t e = cudaFreeAsync(padded, stream); if (e != cudaSuccess && rc == B200SP_OK) rc = cuda_fail(e, "cudaFreeAsync"); }
  return rc;
}

// Of the calls that go by shares with k no multiple of 16 bytes, those that spmm_bundle_kernel takes, with a padded copy of B: where spmm_merge_kernel loads single elements (odd k) or pairs of BF16, and B is read often enough, rows are long enough and the copy is small enough for it to pay:
// a row of the copy takes 128 bytes at least, and one that does not fit L2 beside the rest is read from memory.  Lines drawn over 3027 calls that a laxer rule takes
// (log-normal rows of 4 to 24, 25,000 to 800,000 of them, half to twice as many columns; the same with 12 % of the rows empty; R-MAT 2^16 to 2^21 with hubs packed and spread;
// k = 2 .. 127): those taken are 1.34 times as fast as by shares, ten slower by more than 3 %, one of them by 12 %; those left would be 0.99.  By shares / side by side, us:
// - BF16, odd k above 32, which by shares takes two loads of one element or more a nonzero: from 350,000 items, rows of seven and five reads of a row of B on, over copies of
//   any size (50,000 rows of 14, n = 100,000, k = 33 24 / 14; 200,000 rows of 4, n = 100,000, k = 63 43 / 56: single stores of Y).
// - beta != 0 and a sixteenth of the rows empty, which spmm_merge_kernel lists first: seven reads (R-MAT 2^18, k = 50 BF16 179 / 78; k = 17 FP32 138 / 66), up to 16 columns only
//   while the copy takes less than a quarter of L2 (R-MAT 2^19, k = 3 BF16 95 / 106).
// - beta == 0 and a quarter of the rows empty: BF16, eight reads, from 1 M items on, 2 M with more stores a row (R-MAT 2^18, k = 50 BF16 67 / 58, k = 127 153 / 138; 2^17 32 / 36 and
//   79 / 92); not FP32 above 16 columns (R-MAT 2^17, k = 63 50 / 72), nor copies of more than a quarter of L2 (R-MAT 2^19, k = 50 95 / 102) but for odd k above 32.
// - Odd k of 17 to 31, one load a nonzero by shares and up to eight stores a row here: with beta == 0 only small copies read 15 times (100,000 rows of 24, k = 17 FP32 44 / 38;
//   100,000 of 14 26 / 28).
// - The rest: ten reads (beta != 0: eight) while the copy takes less than a quarter of L2 (200,000 rows of 9, n = 200,000, k = 50 BF16 42.3 / 44.9; n = 100,000 43 / 39), beyond that 16,
//   or 12 where a nonzero takes two loads by shares (400,000 rows of 14, k = 63 FP32 233 / 163); from 450,000, 600,000 or 900,000 items on.
bool spmm_by_padded_bundles(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  const int64_t items = I.m + I.nnz, vec = 16 / elem_bytes, copy = I.n * spmm_padded_row(k, elem_bytes);
  const bool bf16 = elem_bytes == 2, odd = k % 2 != 0, one_load = k <= (odd ? 32 : 64), small = copy <= 36000000;
  if ((k + vec - 1) / vec > 16 || (!odd && (!bf16 || k % 4 != 2))) return false;
  auto reads = [&](int64_t times) { return I.nnz >= times * I.n; };
  const bool mostly = beta == 0.0f && I.bin_rows[0] * 4 >= I.m;             // a quarter of the rows or more are empty, and only written
  if (bf16 && odd && k > 32) return mostly ? reads(8) && items >= (k > 40 ? 2000000 : 1000000) : reads(5) && I.nnz >= 7 * I.m && items >= 350000;
  if (beta != 0.0f && I.bin_rows[0] * 16 >= I.m) return reads(7) && items >= 450000 && (k > 16 || !odd || small);
  if (odd && k > 16 && k <= 32 && beta == 0.0f) return !mostly && reads(15) && copy <= 16000000 && items >= 1000000;
  if (mostly) return reads(8) && small && items >= (odd || k > 64 ? 2000000 : 1000000) && (bf16 || k <= 16);
  if (items < (!bf16 && one_load ? 900000 : !bf16 || one_load ? 600000 : 450000)) return false;
  return reads(small ? (beta != 0.0f ? 8 : 10) : one_load || beta != 0.0f ? 16 : 12);
}

// Of the calls that go by shares, those whose rows of B are narrow for spmm_merge_kernel go to spmm_bundle_kernel.  Times: shares / bundles, us.
// - k a multiple of 16 bytes, up to eight pieces of 16 bytes a row of B, four rows or more side by side, from 250,000 items on (four pieces) or 350,000 (BF16) or
//   600,000 (FP32): 250,000 log-normal rows of 8, BF16 k = 64 46 / 35, FP32 k = 16 64 / 41; R-MAT 2^20, BF16 k = 64 162 / 106, FP32 k = 32 152 / 122.
//   Below that the few regions are as long as before and start later (25,000 rows of 5, FP32 k = 32 9.0 / 10.7).
// - Nine to sixteen pieces, two rows side by side: FP32 gains less from loads twice as wide than it loses at the ends of rows (R-MAT 2^22, k = 64 759 / 797).  BF16 gains by what is
//   left of the last wave by shares, from 800,000 items on up to 1.4 M (beta != 0 2.5 M, a sixteenth of the rows empty 3 M; 100,000 rows of 8, k = 128 1.11 times as fast, beta = 1 1.21
//   times; 124,000 rows of 4, k = 128 25.0 / 28.5, 320,000 57.3 / 61.3, 1,000,000 of 8 252 / 280), and where a quarter of the rows is empty from 1 M on (R-MAT 2^18 1.14 times).
// - beta != 0 and a sixteenth of the rows empty, which spmm_merge_kernel lists first: up to eight pieces from 150,000 items on, 60,000 where it is a quarter (R-MAT 2^20, FP32 k = 32 1.56
//   times as fast, 2^13 1.09 times; 7000 rows of 14, 12 % empty 0.94 times); up to 16 from 450,000, 60,000 (BF16 120,000) where it is a quarter (R-MAT 2^20, FP32 k = 64 303 / 240, 2^14 13.9 / 12.3,
//   BF16 k = 128 1.19 times as fast; 20,000 rows of 14, 12 % empty, k = 48 0.87 times; 600,000, k = 72 BF16 310 / 337), and up to 32 pieces of FP32 only then, from 250,000 on (R-MAT 2^15, k = 128 50 / 36; 2^14 17.4 / 19.7).
bool spmm_by_bundles(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  const int64_t items = I.m + I.nnz, vec = 16 / elem_bytes, pieces = (k + vec - 1) / vec;
  if (k % vec != 0) return spmm_by_padded_bundles(I, k, elem_bytes, beta);
  const bool bf16 = elem_bytes == 2, some = I.bin_rows[0] * 16 >= I.m, many = I.bin_rows[0] * 4 >= I.m;      // rows without nonzeros
  if (beta != 0.0f && some) {
    if (pieces <= 8) return items >= (many ? 60000 : 150000);
    if (pieces <= 16) return items >= (!many ? 450000 : bf16 ? 120000 : 60000) && (many || !bf16 || items <= 6000000);
    return !bf16 && pieces <= 32 && many && items >= 250000;
  }
  if (pieces <= 8) return items >= (pieces <= 4 ? 250000 : bf16 ? 350000 : 600000);
  if (!bf16 || pieces > 16) return false;
  return many ? items >= 1000000 : items >= 800000 && items <= (some ? 3000000 : beta != 0.0f ? 2500000 : 1400000);
}

// Rows all of one length of 5 to 13 that is no multiple of four, k a multiple of 16 bytes and five to sixteen pieces of them a row of B: by rows they take single
// steps at both ends of nearly every row, side by side only at one.  What that gains goes with the last steps that the length leaves (5 and 7 most, 10 and 13 least), with the
// number of items, and with what the call would take by rows: BF16 whose rows of B are whole pieces of 32 bytes has a faster kernel there (spmm_slice_wide_kernel).
// 7 lengths, 10 widths, 0.8 to 9 M items, half to twice as many columns as rows, beta = 0 and 1; least number of items, and by rows / side by side in us on both sides of it:
// - FP32, up to eight pieces: 2 M, 5 M for rows of 10 and more (k = 32: 190,000 rows of 10 56 / 56, 96,000 25 / 35); more pieces: 780,000 for rows of 5 and 7, 1.4 M for 6, 9 and 11, 3 M
//   for 10 and 13 (k = 36: 57,000 rows of 13 20 / 27, 114,000 of 6 22 / 28; 8 M nonzeros in rows of 6, k = 64 466 / 373).
// - BF16, k no multiple of 16, up to eight pieces: 1 M, 5 M for rows of 10 and 13; more: 780,000 (k = 72: 111,500 rows of 6 1.19 times as fast).
// - BF16, k a multiple of 16, up to eight pieces: 1 M for rows of 5, 6 and 7, 3 M for 9 and 11, 8 M for 10 and 13 (k = 64: 150,000 rows of 13, beta = 1 31 / 37; 131,072 of 7 23.5 / 18.2; rows
//   of 6 gain from 2 M on and lose up to 14 % at 1 M); more: 780,000 for 5 and 7, 1 M for 6, 9 and 11, 1.5 M for 10 and 13 and these with beta == 0 only (k = 128: 131,072 rows of 7 41.9 / 28.6,
//   364,000 of 13 and beta = 1 163 / 172).
// Not rows of 21 (FP32 k = 64 192 / 201), fewer (70,000 rows of 6, BF16 k = 64 9.4 / 13.4) or wider (k = 128 FP32, rows of 13 241 / 254).
// Where a switch asks for one of the kernels by rows they stay by rows.
bool spmm_even_by_bundles(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  const int64_t items = I.m + I.nnz, vec = 16 / elem_bytes, pieces = k / vec;
  const int length = I.max_row_len;
  if (!g_opt.spmm_sliced || g_opt.spmm_flat != 2 || g_opt.spmm_stage_a != 2 || g_opt.spmm_ranges != 1) return false;
  if (I.min_row_len != length || length % 4 == 0 || length < 5 || length > 13 || k % vec != 0 || pieces < 5 || pieces > 16) return false;
  const bool most = length == 5 || length == 7, least = length == 10 || length == 13, wide = elem_bytes == 2 && k % 16 == 0;
  if (elem_bytes == 4) return items >= (pieces <= 8 ? (length < 10 ? 2000000 : 5000000) : most ? 780000 : least ? 3000000 : 1400000);
  if (!wide) return items >= (pieces > 8 ? 780000 : least ? 5000000 : 1000000);
  if (pieces <= 8) return items >= (length <= 7 ? 1000000 : least ? 8000000 : 3000000);
  return items >= (most ? 780000 : least ? 1500000 : 1000000) && (!least || beta == 0.0f);
}

// Whether spmm_bundle_kernel takes a call with k > 1 columns under the present switches.
bool spmm_side_by_side(const b200sp_plan_info_t& I, int64_t k, int elem_bytes, float beta) {
  return spmm_by_shares(I, k, elem_bytes, beta) ? spmm_by_bundles(I, k, elem_bytes, beta) : spmm_even_by_bundles(I, k, elem_bytes, beta);
}

template <typename T, int VEC>
int run_spmm(b200sp_plan* p, int k, const int32_t* col_idx, const T* vals, const T* B, T* Y, float alpha, float beta,
             cudaStream_t stream, DeviceInfo* dev) {
  const b200sp_plan_info_t& I = p->info;
  if (I.m == 0) return B200SP_OK;
  if (alpha == 0.0f || I.nnz == 0) return run_scale<T>((long long)I.m * k, Y, beta, stream, dev);
  if (k == 1) return run_spmv<T>(p, col_idx, vals, B, Y, alpha, beta, stream, dev);   // one column: the SpMV kernels
  if (k % VEC == 0 && g_opt.spmm_bstage && I.nnz >= 4 * I.n && ((size_t)k * sizeof(T)) % 16 == 0) {
    // widest slice of B (128, 64 or 32 bytes per row) whose n rows fit in one SM's shared memory
    const size_t budget = (size_t)kSmemPerSm - 4096;
    const size_t n_pad = (size_t)((I.n + 255) / 256) * 256;
    EncodeTiledFn encode = tensor_map_encoder();
    if (encode && n_pad * 32 <= budget) {
      int rc;
#define B200SP_BSTAGE(FN)                                                                                                                  \
  do {                                                                                                                                     \
    if (g_opt.bstage_threads == 256) {                                                                                                     \
      if (n_pad * 128 <= budget) rc = FN<T, VEC, 8, 256>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                     \
      else if (n_pad * 64 <= budget) rc = FN<T, VEC, 4, 256>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                 \
      else rc = FN<T, VEC, 2, 256>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                                           \
    } else if (g_opt.bstage_threads == 512) {                                                                                              \
      if (n_pad * 128 <= budget) rc = FN<T, VEC, 8, 512>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                     \
      else if (n_pad * 64 <= budget) rc = FN<T, VEC, 4, 512>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                 \
      else rc = FN<T, VEC, 2, 512>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                                           \
    } else {                                                                                                                               \
      if (n_pad * 128 <= budget) rc = FN<T, VEC, 8, 1024>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                    \
      else if (n_pad * 64 <= budget) rc = FN<T, VEC, 4, 1024>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                \
      else rc = FN<T, VEC, 2, 1024>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev, encode);                                          \
    }                                                                                                                                      \
  } while (0)
      if (g_opt.bstage_quads) B200SP_BSTAGE(launch_spmm_bstage_quads);
      else B200SP_BSTAGE(launch_spmm_bstage);
#undef B200SP_BSTAGE
      if (rc != B200SP_ERR_UNSUPPORTED) return rc;   // unsupported shape for the tensor map: fall through to the sliced kernel
    }
  }
  if (spmm_side_by_side(I, k, (int)sizeof(T), beta)) {
    const int rc = k % VEC == 0 ? run_spmm_bundle<T, VEC>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev)
                   : sizeof(T) == 2 && k % 2 == 0 ? run_spmm_bundle<T, sizeof(T) == 2 ? 2 : 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev)
                                : run_spmm_bundle<T, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    if (rc != B200SP_ERR_ALLOC) return rc;       // (nothing that writes Y is launched then)
  }
  if (spmm_by_shares(I, k, (int)sizeof(T), beta)) {
    const int rc = run_spmm_merge<T, VEC>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    if (rc != B200SP_ERR_UNSUPPORTED && rc != B200SP_ERR_ALLOC) return rc;   // without its scratch (nothing is launched then) by rows, which need none
  }
  if (k % VEC == 0 && g_opt.spmm_sliced) {
    // lanes per row: eight (a 128-byte slice) unless k is narrower than that
    const int vecs_k = k / VEC;
    const int lanes = vecs_k >= 8 ? 8 : (vecs_k > 2 ? 4 : vecs_k);
    const int KS = lanes * VEC, GROUPS = kSpmmThreads / lanes;
    const int slices = (k - 1) / KS + 1;
    const int row_blocks = (int)((I.m + GROUPS - 1) / GROUPS);
    if ((long long)slices * row_blocks >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
    b200sp_plan::RowLists lists;
    CallBlock own_lists;
    int rc = plan_row_lists(p, &lists, &own_lists, stream, dev);
    if (rc != B200SP_OK) return rc;
    const int mid_blocks = (p->num_medium + GROUPS - 1) / GROUPS;
    const bool wide = sizeof(T) == 2 && lanes == 8 && g_opt.spmm_stage_a == 2 && k % 16 == 0 && ((uintptr_t)B & 31) == 0 && spmm_wide_pieces(I, k, dev->sms, dev->l2_bytes);
    int ranges = 1;
    if (lanes == 8) {
      rc = spmm_column_ranges(p, col_idx, 8 * 16, stream, dev, &ranges);
      if (rc != B200SP_OK) return rc;
    }
    if (ranges > 1) {
      // one launch per column range; FP32 partial sums for BF16 storage come from the pool and go back in stream order
      float* partial = nullptr;
      if (sizeof(T) == 2) {
        rc = pool_alloc(dev, (void**)&partial, (size_t)I.m * (size_t)k * sizeof(float), stream);
        if (rc != B200SP_OK) return rc;
      }
      for (int r = 0; r < ranges && rc == B200SP_OK; ++r) {
        tl_pdl_kernel = true;
        rc = launch(spmm_slice_range_kernel<T, VEC, kSpmmThreads, 8>, dim3((unsigned)(slices * row_blocks)), dim3(kSpmmThreads), stream, nullptr, 0,
                    dev, (int)I.m, k, row_blocks, r, ranges, (const int*)p->cuts_block, p->row_ptr, col_idx, vals, B, Y, partial, alpha, beta,
                    kMediumRow);
      }
      if (partial) { const cudaError_t e = cudaFreeAsync(partial, stream); if (e != cudaSuccess && rc == B200SP_OK) rc = cuda_fail(e, "cudaFreeAsync"); }
      if (rc == B200SP_OK && p->num_medium > 0) {
        tl_pdl_kernel = true;
        rc = launch(spmm_medium_row_kernel<T, VEC, kSpmmThreads, 8>, dim3((unsigned)(slices * mid_blocks)), dim3(kSpmmThreads), stream,
                    nullptr, 0, dev, p->num_medium, lists.medium, k, mid_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, beta);
      }
    } else if (wide) {
      if constexpr (sizeof(T) == 2) {
        constexpr int THREADS = 128;
        static_assert(THREADS / 4 == kSpmmThreads / 8, "the same rows per block as the kernels with eight lanes a row");
        tl_pdl_kernel = true;
        rc = launch(spmm_slice_wide_kernel<THREADS>, dim3((unsigned)(slices * row_blocks)), dim3(THREADS), stream, B, (size_t)I.n * k * sizeof(T), dev, (int)I.m,
                    k, row_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, beta, kMediumRow);
        if (rc == B200SP_OK && p->num_medium > 0) {
          tl_pdl_kernel = true;
          rc = launch(spmm_medium_row_kernel<T, VEC, kSpmmThreads, 8>, dim3((unsigned)(slices * mid_blocks)), dim3(kSpmmThreads), stream, nullptr, 0, dev,
                      p->num_medium, lists.medium, k, mid_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, beta);
        }
      }
    } else
    // rows of at most kMediumRow nonzeros: the register-capped kernel; kMediumRow + 1 .. kLongRow: the same scheme with
    // blocked sums over the plan's list of such rows; longer rows: a CTA per (row, slice)
#define B200SP_SLICE_LAUNCH(L)                                                                                                      \
    tl_pdl_kernel = true;                                                                                                           \
    if ((g_opt.spmm_stage_a == 1 || (g_opt.spmm_stage_a == 2 && sizeof(T) == 2)) && L > 1)                                          \
      rc = launch(spmm_slice_staged_kernel<T, VEC, kSpmmThreads, (L > 1 ? L : 2), kSpmmStageCap>, dim3((unsigned)(slices * row_blocks)),  \
                  dim3(kSpmmThreads), stream, B, (size_t)I.n * k * sizeof(T), dev, (int)I.m, (int)I.nnz, k, row_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, \
                  beta, kMediumRow);                                                                                                \
    else                                                                                                                            \
      rc = launch(spmm_slice_kernel<T, VEC, kSpmmThreads, L>, dim3((unsigned)(slices * row_blocks)), dim3(kSpmmThreads), stream, B,       \
                  (size_t)I.n * k * sizeof(T), dev, (int)I.m, k, row_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, beta, kMediumRow);                          \
    if (rc == B200SP_OK && p->num_medium > 0) {                                                                                     \
      tl_pdl_kernel = true;                                                                                                         \
      rc = launch(spmm_medium_row_kernel<T, VEC, kSpmmThreads, L>, dim3((unsigned)(slices * mid_blocks)), dim3(kSpmmThreads), stream, \
                  nullptr, 0, dev, p->num_medium, lists.medium, k, mid_blocks, p->row_ptr, col_idx, vals, B, Y, alpha, beta); \
    }
    if (lanes == 8) { B200SP_SLICE_LAUNCH(8); }
    else if (lanes == 4) { B200SP_SLICE_LAUNCH(4); }
    else if (lanes == 2) { B200SP_SLICE_LAUNCH(2); }
    else { B200SP_SLICE_LAUNCH(1); }
#undef B200SP_SLICE_LAUNCH
    if (rc != B200SP_OK || p->num_long == 0) return rc;
    const long long ctas = (long long)((k - 1) / (8 * VEC) + 1) * p->num_long;
    if (ctas >= (1LL << 31)) return B200SP_ERR_UNSUPPORTED;
    tl_pdl_kernel = true;
    return launch(spmm_long_row_kernel<T, VEC, kSpmmThreads>, dim3((unsigned)ctas), dim3(kSpmmThreads), stream, nullptr, 0,
                  dev, k, p->num_long, lists.longer, p->row_ptr, col_idx, vals, B, Y, alpha, beta);
  }
  if (k % VEC != 0) {  // ragged k: scalar lanes
    if (k <= 2) return launch_spmm<T, 1, 2, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    if (k <= 4) return launch_spmm<T, 1, 4, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    if (k <= 8) return launch_spmm<T, 1, 8, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    if (k <= 16) return launch_spmm<T, 1, 16, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
    return launch_spmm<T, 1, 32, 2>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  }
  const int vecs = k / VEC;  // vector columns per row
  if (vecs <= 4) return launch_spmm<T, VEC, 4, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  if (vecs <= 8) return launch_spmm<T, VEC, 8, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  if (vecs <= 16) return launch_spmm<T, VEC, 16, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  if (vecs <= 32) return launch_spmm<T, VEC, 32, 1>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
  return launch_spmm<T, VEC, 32, 2>(p, k, col_idx, vals, B, Y, alpha, beta, stream, dev);
}

}  // namespace
