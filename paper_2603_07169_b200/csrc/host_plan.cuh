// Host side of libb200sp.so: the plan pass (row statistics, bins, splits, medium- and long-row lists) and the plan cache.
// One of the pieces of the single translation unit b200sp.cu; include/b200sp.h states the contract of every entry point.
#pragma once
#include "host_runtime.cuh"
#include "plan_kernels.cuh"
#include "spmm_merge_kernels.cuh"

namespace {

// Plans cached by the one-shot entry points, keyed on (device, row_ptr address, m, n, nnz).  The address may be a device
// pointer (spmv_csr, spmm_csr) or a host pointer (spmv_csr_host, spmm_csr_host); the two never collide in a unified
// address space.  At most kCacheCap plans are kept: the least recently used one is dropped when another is added.
typedef std::tuple<int, const void*, int64_t, int64_t, int64_t> PlanKey;
struct CachedPlan { b200sp_plan* plan = nullptr; uint64_t stamp = 0; };
std::map<PlanKey, CachedPlan> g_cache;
uint64_t g_cache_clock = 0;
constexpr size_t kCacheCap = 1024;

// Frees a plan.  With stream_ordered the block goes back to the pool in the order of `stream` (the caller
// knows that every kernel that used the plan ran there); otherwise the device is synchronised first.
int plan_free(b200sp_plan* p, bool stream_ordered = false, cudaStream_t stream = nullptr) {
  if (!p) return B200SP_OK;
  int rc = B200SP_OK;
  void* const blocks[] = {p->block, p->cuts_block, p->compact_block, p->shares.block, p->quad[0].block, p->quad[1].block, p->quad[2].block,
                          p->lists.block};
  bool any = false;
  for (void* b : blocks) any |= b != nullptr;
  if (any) {
    cudaError_t e = cudaSuccess;
    int cur = p->device;
    if (!stream_ordered) {
      e = cudaGetDevice(&cur);
      if (e == cudaSuccess && cur != p->device) e = cudaSetDevice(p->device);
      if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    for (void* b : blocks)
      if (b && e == cudaSuccess) e = stream_ordered ? cudaFreeAsync(b, stream) : cudaFree(b);
    if (cur != p->device) cudaSetDevice(cur);
    if (e != cudaSuccess) rc = cuda_fail(e, "freeing a plan");
  }
  delete p;
  return rc;
}

// The list of the rows that have nonzeros (their numbers and their offsets), built on the device in stream order and kept with
// the plan: used by the merge-tile SpMV kernel under the switch "merge_empty".  Needs
// info.bin_rows[0] (the number of empty rows).  No synchronisation.
int plan_compact_rows(b200sp_plan* p, cudaStream_t stream, DeviceInfo* dev) {
  if (p->compact_block) return B200SP_OK;
  b200sp_plan_info_t& I = p->info;
  const int64_t m = I.m, mc = m - I.bin_rows[0];
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const int blocks = (int)((m + kCompactBlock - 1) / kCompactBlock);
  const size_t o_id = 0, o_rp = o_id + up((size_t)(mc + 1) * 4), o_bc = o_rp + up((size_t)(mc + 1) * 4), total = o_bc + up((size_t)(blocks + 1) * 4);
  void* blk = nullptr;
  int rc = pool_alloc(dev, &blk, total, stream);
  if (rc != B200SP_OK) return rc;
  char* b2 = (char*)blk;
  int32_t* row_id = (int32_t*)(b2 + o_id);
  int32_t* row_ptr_c = (int32_t*)(b2 + o_rp);
  int* d_bc = (int*)(b2 + o_bc);
  plan_compact_count_kernel<<<blocks, 256, 0, stream>>>(p->row_ptr, (int)m, d_bc);
  plan_compact_scan_kernel<<<1, 1024, 0, stream>>>(d_bc, blocks);
  plan_compact_write_kernel<<<blocks, 256, 0, stream>>>(p->row_ptr, (int)m, (int)I.nnz, d_bc, row_id, row_ptr_c);
  g_launches += 3;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { cudaFreeAsync(blk, stream); return cuda_fail(e, "list of non-empty rows"); }
  p->compact_block = blk;
  p->compact_row_id = row_id;
  p->compact_row_ptr = row_ptr_c;
  p->compact_rows = (int)mc;
  I.scratch_bytes += (int64_t)total;
  return B200SP_OK;
}

// Pinned host memory for the results of plan passes, one slot per pass in flight; a pass holds its slot (and the accumulators of
// the same index in g_plan_slots) from before its launch until its results have been read.
struct PlanSlots {
  std::mutex mutex;
  std::condition_variable freed;
  PlanStats* host = nullptr;
  std::vector<int> idle;
} g_slots;

int plan_slot_take(int* slot) {
  std::unique_lock<std::mutex> lock(g_slots.mutex);
  if (!g_slots.host) {
    CU(cudaHostAlloc((void**)&g_slots.host, kPlanSlots * sizeof(PlanStats), cudaHostAllocPortable | cudaHostAllocMapped));
    for (int i = kPlanSlots - 1; i >= 0; --i) g_slots.idle.push_back(i);
  }
  g_slots.freed.wait(lock, [] { return !g_slots.idle.empty(); });
  *slot = g_slots.idle.back();
  g_slots.idle.pop_back();
  return B200SP_OK;
}

void plan_slot_give(int slot) {
  { std::lock_guard<std::mutex> lock(g_slots.mutex); g_slots.idle.push_back(slot); }
  g_slots.freed.notify_one();
}

// Merge items per share of the nnz-balanced SpMM kernel: 128, fewer for small problems (20,011 rows, 220,121 items, k = 128 with a fresh
// plan: 64 us with shares of 56 and 64, 71 us with 32, 70 us with 128).
int spmm_share_items(const b200sp_plan_info_t& I, const DeviceInfo* dev) {
  const int64_t w = (I.m + I.nnz + (int64_t)dev->sms * 24 - 1) / ((int64_t)dev->sms * 24);
  return w >= kMergeWarpItems ? kMergeWarpItems : w <= 32 ? 32 : (int)((w + 7) / 8 * 8);
}

// The lists of rows of kMediumRow + 1 .. kLongRow and of more than kLongRow nonzeros, built on the device in stream order on the
// first SpMM call that needs them; their lengths are known from the plan pass.
int plan_row_lists(b200sp_plan* p, b200sp_plan::RowLists* out, CallBlock* own, cudaStream_t stream, DeviceInfo* dev) {
  if (p->num_medium + p->num_long == 0) return B200SP_OK;
  std::lock_guard<std::mutex> lock(p->build);
  if (!p->lists.block) {
    const size_t n_mid = (size_t)p->num_medium, n_long = (size_t)p->num_long;
    int* blk = nullptr;
    const int rc = pool_alloc(dev, (void**)&blk, (4 + n_mid + n_long) * sizeof(int32_t), stream);
    if (rc != B200SP_OK) return rc;
    cudaError_t e = cudaMemsetAsync(blk, 0, 2 * sizeof(int), stream);
    if (e == cudaSuccess) {
      const int blocks = (int)((p->info.m + 255) / 256);
      plan_row_lists_kernel<<<blocks < dev->sms * 8 ? blocks : dev->sms * 8, 256, 0, stream>>>(
          p->row_ptr, (int)p->info.m, kMediumRow, kLongRow, (int)n_mid, (int)n_long, blk + 4, blk + 4 + n_mid, blk);
      g_launches++;
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) { cudaFreeAsync(blk, stream); return cuda_fail(e, "lists of medium and long rows"); }
    *out = {blk, blk + 4, blk + 4 + n_mid};
    if (stream_captures(stream)) { own->take(blk, stream); return B200SP_OK; }
    p->lists = *out;
  }
  *out = p->lists;
  return B200SP_OK;
}

// The shares of the nnz-balanced SpMM kernel: with the plan pass for small matrices, else by a small kernel in stream order on the first
// SpMM call that needs them.
int plan_shares(b200sp_plan* p, b200sp_plan::Shares* out, CallBlock* own, cudaStream_t stream, DeviceInfo* dev) {
  std::lock_guard<std::mutex> lock(p->build);
  if (!p->shares.split) {
    const b200sp_plan_info_t& I = p->info;
    const int w = spmm_share_items(I, dev);
    const long long shares = (I.m + I.nnz + w - 1) / w;
    int* blk = nullptr;
    int rc = pool_alloc(dev, (void**)&blk, (size_t)(shares + 1) * sizeof(int32_t), stream);
    if (rc != B200SP_OK) return rc;
    rc = launch(plan_merge_split_kernel, dim3((unsigned)((shares + 1 + 255) / 256)), dim3(256), stream, nullptr, 0, dev, p->row_ptr, (int)I.m,
                (int)I.nnz, w, (int)shares, blk);
    if (rc != B200SP_OK) { cudaFreeAsync(blk, stream); return rc; }
    *out = {blk, blk, w};
    if (stream_captures(stream)) { own->take(blk, stream); return B200SP_OK; }
    p->shares = *out;
  }
  *out = p->shares;
  return B200SP_OK;
}

// Lanes per row of the sub-warp kernel: by the mean row length, raised so that no lane adds more than kSubwarpChain terms in sequence.
int subwarp_lanes(int64_t m, int64_t nnz, int max_len) {
  const double mean = m > 0 ? (double)nnz / (double)m : 0.0;
  int lpr = g_opt.sub_lanes;
  if (lpr <= 0) lpr = mean <= 3 ? 1 : mean <= 6 ? 2 : mean <= 12 ? 4 : mean <= 24 ? 8 : mean <= 64 ? 16 : 32;
  while (lpr < 32 && ((long long)max_len + lpr - 1) / lpr > kSubwarpChain) lpr *= 2;
  return lpr;
}

int plan_build(b200sp_plan** out, int64_t m, int64_t n, int64_t nnz, const int32_t* row_ptr, cudaStream_t stream) {
  DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != B200SP_OK) return rc;
  b200sp_plan* p = new b200sp_plan();
  CU(cudaGetDevice(&p->device));
  p->row_ptr = row_ptr;
  b200sp_plan_info_t& I = p->info;
  I.m = m; I.n = n; I.nnz = nnz;
  // SpMV tiles of 1024 items instead of 2048 below 12 M: more CTAs (R-MAT 2^17 10.4 / 11.5 us, 2^18 15.9 / 16.5 us, 2^19 23.7 / 25.4 us,
  // 2^20 40.6 / 42.2 us; equal from 2^21 on)
  const int items = !g_opt.merge_items_set && m + nnz < 12000000 ? 1024 : g_opt.merge_items;
  I.spmv_tile_items = items;
  I.spmv_tiles = (int32_t)((m + nnz + items - 1) / items);
  I.spmv_kernel = g_opt.spmv_kernel >= 0 ? g_opt.spmv_kernel : 0;
  if (m == 0) { *out = p; return B200SP_OK; }
  if (stream_captures(stream)) { delete p; return B200SP_ERR_UNSUPPORTED; }   // the statistics are read back

  // one block from the pool: the probe's counters, split points, carries, tails; for small matrices also the shares of the
  // nnz-balanced SpMM kernel, which then cost no launch of their own (large ones search them on first use)
  const size_t nt = (size_t)I.spmv_tiles;
  const int witems = spmm_share_items(I, dev);
  const long long shares = (m + nnz + witems - 1) / witems;
  const bool with_shares = shares <= 65536;   // (m + nnz <= 2^23)
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t o_split = 256, o_carry = o_split + up((nt + 1) * 4), o_tail = o_carry + up((nt + 1) * 4), o_share = o_tail + up((nt + 1) * 4),
               total = o_share + (with_shares ? up((size_t)(shares + 1) * 4) : 0);
  auto fail = [&](int code) { plan_free(p, true, stream); cudaStreamSynchronize(stream); return code; };
#define CUP(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return fail(cuda_fail(e_, #call)); } while (0)
  rc = pool_alloc(dev, &p->block, total, stream);
  if (rc != B200SP_OK) { delete p; return rc; }
  char* base = (char*)p->block;
  p->probe_out = (unsigned long long*)base;   // two probe counters
  p->split_row = (int32_t*)(base + o_split);
  p->carry = (float*)(base + o_carry);
  p->tail = (float*)(base + o_tail);
  int32_t* const share_split = (int32_t*)(base + o_share);
  if (with_shares) p->shares = {nullptr, share_split, witems};
  I.scratch_bytes = (int64_t)total;
  int slot = 0;
  rc = plan_slot_take(&slot);
  if (rc != B200SP_OK) return fail(rc);
  PlanStats h;
  {
    const SplitRule tile_rule = split_rule(items, (unsigned)nt + 1), share_rule = split_rule(witems, with_shares ? (unsigned)shares + 1 : 0);
    // The rows write their split points themselves, or every split point is searched.  Rows: up to 2^17 of them (plan_pass_kernel), while a block's
    // 256 rows hold few, which it writes alone however many blocks there are (creating a plan, search / rows, us: 8 rows of 2 x 10^8 nonzeros
    // 22 / 204, 200 of 30,000 17 / 33, 500 of 2000 18 / 19; but 2^17 of 16,000, 8 to a row, 38 / 24, 30,000 of 50,000, 24 to a row, 30 / 24).
    const long long splits = (long long)tile_rule.count + share_rule.count;
    const bool by_rows = m <= (1 << 17) && splits <= (m >= (1 << 14) ? 32 : 8) * m;
    const long long work = by_rows || m > splits ? m : splits, blocks = (work + 255) / 256;
    rc = launch(by_rows ? plan_pass_kernel<false> : plan_pass_kernel<true>, dim3((unsigned)(by_rows || blocks < dev->sms * 8 ? blocks : dev->sms * 8)), dim3(256),
                stream, nullptr, 0, dev, row_ptr, (int)m, (int)nnz, slot, g_slots.host + slot, tile_rule, p->split_row, share_rule, share_split);
    const cudaError_t e = cudaStreamSynchronize(stream);
    h = g_slots.host[slot];
    if (e == cudaSuccess) plan_slot_give(slot);   // only a finished pass (or none) has left its slot to the next; an error here means a lost device
    if (rc != B200SP_OK) return fail(rc);
    if (e != cudaSuccess) return fail(cuda_fail(e, "plan pass"));
  }
  if (!h.bad) { p->num_medium = (int)h.bin_rows[4]; p->num_long = (int)h.bin_rows[5]; }
  // Many rows without nonzeros (a quarter or more): the merge list is built over the rows that have nonzeros only, and the
  // split points are searched again over that list.
  if (!h.bad && g_opt.merge_empty && nnz > 0 && (int64_t)h.bin_rows[0] * 4 >= m) {
    for (int j = 0; j < B200SP_NUM_BINS; ++j) I.bin_rows[j] = (int64_t)h.bin_rows[j];
    rc = plan_compact_rows(p, stream, dev);
    if (rc != B200SP_OK) return fail(rc);
    const int64_t mc = p->compact_rows;
    const size_t ntc = (size_t)((mc + nnz + items - 1) / items);     // fewer items, fewer tiles: the arrays sized above suffice
    plan_merge_split_kernel<<<(unsigned)((ntc + 1 + 255) / 256), 256, 0, stream>>>(p->compact_row_ptr, (int)mc, (int)nnz, items, (int)ntc, p->split_row);
    g_launches++;
    CUP(cudaGetLastError());
    CUP(cudaStreamSynchronize(stream));
    p->merge_compact = true;
    I.spmv_tiles = (int32_t)ntc;
  }
#undef CUP
  if (h.bad) { plan_free(p, true, stream); cudaStreamSynchronize(stream); return B200SP_ERR_BAD_CSR; }
  I.min_row_len = h.min_len; I.max_row_len = h.max_len;
  for (int j = 0; j < B200SP_NUM_BINS; ++j) { I.bin_rows[j] = (int64_t)h.bin_rows[j]; I.bin_nnz[j] = (int64_t)h.bin_nnz[j]; }
  // Kernel choice from the row statistics: when every row is short and the mean is not far below the
  // maximum, a thread per row wastes little and rows never need splitting -> row-direct kernel.
  // Anything with long or very uneven rows goes to the merge-tile kernel.
  const bool row_direct_ok = nnz > 0 && h.max_len <= kRowMaxLen && aligned16(row_ptr) &&
                             (h.max_len <= 8 || nnz * 4 >= (int64_t)h.max_len * m);
  // Rows all of one length 4, 8, ..., 128: sub-warp-per-row kernel with 128-bit loads and no shared memory.
  const bool uniform_ok = nnz > 0 && h.min_len == h.max_len && h.max_len >= 4 && h.max_len <= 128 && (h.max_len & (h.max_len - 1)) == 0;
  const bool row_direct_possible = nnz > 0 && h.max_len <= kRowMaxLen && aligned16(row_ptr);
  int choice = uniform_ok ? 2 : (row_direct_ok ? 1 : 0);
  // Small problems (launch-latency regime): one sub-warp per row, no scratch, maximum spread over the SMs -- unless the
  // rows are uniform (the uniform-row kernel is as flat) or the row-direct kernel would still get a tile for every SM.
  // A lane that adds more than some 40 products in sequence makes the launch wait for it (0.27 us for two): the merge-tile kernel with its
  // second launch is then faster (R-MAT 2^14 / 2^15 / 2^16: 7.5 / 9.3 / 17.7 us by sub-warps, 6.5 / 7.3 / 7.8 us by tiles).
  const int sub = subwarp_lanes(m, nnz, h.max_len);
  if (nnz > 0 && nnz <= kSmallNnz && (h.max_len + sub - 1) / sub <= 40 && !uniform_ok && !(row_direct_ok && m >= (int64_t)kRowThreads * dev->sms)) choice = 3;
  if (g_opt.spmv_kernel == 3) choice = h.max_len <= 32 * kSubwarpChain ? 3 : 0;
  if (g_opt.spmv_kernel == 0) choice = 0;
  if (g_opt.spmv_kernel == 1) choice = row_direct_possible ? 1 : 0;
  if (g_opt.spmv_kernel == 2) choice = uniform_ok ? 2 : (row_direct_ok ? 1 : 0);
  I.spmv_kernel = choice;
  if (g_opt.log) {
    static const char* const kname[4] = {"merge-tile", "row-direct", "uniform-row", "sub-warp"};
    fprintf(stderr, "b200sp plan: m=%lld n=%lld nnz=%lld rows by length 0|1-4|5-32|33-128|129-1024|>1024 = %lld|%lld|%lld|%lld|%lld|%lld min=%d max=%d "
                    "spmv kernel=%s tiles=%d x %d items%s scratch=%lld bytes\n",
            (long long)m, (long long)n, (long long)nnz, (long long)I.bin_rows[0], (long long)I.bin_rows[1], (long long)I.bin_rows[2], (long long)I.bin_rows[3],
            (long long)I.bin_rows[4], (long long)I.bin_rows[5], I.min_row_len, I.max_row_len, kname[choice & 3], I.spmv_tiles, I.spmv_tile_items,
            p->merge_compact ? " (non-empty rows only)" : "", (long long)I.scratch_bytes);
  }
  *out = p;
  return B200SP_OK;
}

int check_common(const b200sp_plan* p, const void* col_idx, const void* vals, const void* dense_in, const void* dense_out, int dtype) {
  if (!p) return B200SP_ERR_INVALID_ARG;
  if (dtype != B200SP_F32 && dtype != B200SP_BF16) return B200SP_ERR_INVALID_ARG;
  const b200sp_plan_info_t& I = p->info;
  if (I.nnz > 0 && (!col_idx || !vals || !dense_in)) return B200SP_ERR_INVALID_ARG;
  if (I.m > 0 && !dense_out) return B200SP_ERR_INVALID_ARG;
  if (!aligned16(col_idx) || !aligned16(vals) || !aligned16(dense_in) || !aligned16(dense_out)) return B200SP_ERR_INVALID_ARG;
  int cur = 0;
  CU(cudaGetDevice(&cur));
  if (I.m > 0 && cur != p->device) return B200SP_ERR_INVALID_ARG;   // a plan belongs to the device it was created on
  return B200SP_OK;
}

// Looks `key` up; a hit refreshes its stamp.  The caller holds no lock.
b200sp_plan* cache_find(const PlanKey& key) {
  std::lock_guard<std::mutex> lock(g_mutex);
  auto it = g_cache.find(key);
  if (it == g_cache.end()) return nullptr;
  it->second.stamp = ++g_cache_clock;
  return it->second.plan;
}

// Adds a plan under `key` (or returns the one another thread added first) and drops the least recently used
// plan beyond the cap.  Dropping synchronises the device of the dropped plan.
b200sp_plan* cache_insert(const PlanKey& key, b200sp_plan* p) {
  b200sp_plan* victim = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    auto ins = g_cache.emplace(key, CachedPlan{p, ++g_cache_clock});
    if (!ins.second) { victim = p; p = ins.first->second.plan; }
    else if (g_cache.size() > kCacheCap) {
      auto oldest = g_cache.end();
      for (auto it = g_cache.begin(); it != g_cache.end(); ++it)
        if (it->second.plan != p && (oldest == g_cache.end() || it->second.stamp < oldest->second.stamp)) oldest = it;
      if (oldest != g_cache.end()) { victim = oldest->second.plan; g_cache.erase(oldest); }
    }
  }
  if (victim) plan_free(victim);
  return p;
}

int get_cached_plan(b200sp_plan** out, int64_t m, int64_t n, int64_t nnz, const int32_t* row_ptr, cudaStream_t stream) {
  int dev = 0;
  CU(cudaGetDevice(&dev));
  const PlanKey key = std::make_tuple(dev, (const void*)row_ptr, m, n, nnz);
  if (b200sp_plan* hit = cache_find(key)) { *out = hit; return B200SP_OK; }
  b200sp_plan* p = nullptr;
  int rc = b200sp_plan_create(&p, m, n, nnz, row_ptr, stream);
  if (rc != B200SP_OK) return rc;
  *out = cache_insert(key, p);
  return B200SP_OK;
}

}  // namespace
