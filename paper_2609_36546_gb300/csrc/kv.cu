// Append of newly computed tokens' K/V rows into a paged cache (Sec. 3.2.3:
// the proposer's decode extends its own cache by one token per step, the
// verifier's prefill writes the span's tokens into its cache; each happens
// before the attention that reads them).
//
// One warp per new token: its K and V head rows (a 128-wide bf16 head row is
// 16 pieces of 16 bytes) are contiguous in the inputs, and each head row is a
// contiguous 256-byte run of a page slot.  A few microseconds of latency bound
// the launch (a step moves a few MB), so a lane's loads, up to eight, are in
// flight while the warp looks the token's request up in one or two rounds of
// probes and follows the page table, once per token.  Spans of 8 of 256 requests,
// us a call: 6.6, with a thread and a bisection per 16-byte piece 8.2; of 16 of
// 300: 8.2 and 14.9; of 24 of 768: 25.5 and 43.1; small appends the same (6.4).
// Every write is bounds-checked against the request offsets, the sequence
// length, the page table and the pool; a bad entry is recorded in the device
// error word and skipped.  One launch takes up to IPD_MAX_BATCHES appends
// (caches and request batches), so a step's appends cost one launch.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "common.cuh"

IPD_DECLARE_ERROR_WORD(g_kv_err);

namespace {

constexpr int kPieces = 16;  // 16-byte pieces per 128-wide bf16 row
constexpr int kAppendThreads = 128;
constexpr int kAppendWarps = kAppendThreads / 32;
constexpr int kAppendLoads = 8;  // pieces of a lane in flight (a token of 8 KV heads)

// One append (one cache, one batch of requests) of a launch.
struct AppendDev {
  uint16_t *k_pages, *v_pages;
  const uint16_t *k_new, *v_new;
  const int32_t *cu_new, *seq_len, *page_table;
  long long num_pages;
  int total_new, hkv, max_pages, num_reqs;
};

struct AppendParams {
  AppendDev d[IPD_MAX_BATCHES];
  long long end[IPD_MAX_BATCHES];  // inclusive prefix of total_new over the appends
  int n;
};

__global__ void __launch_bounds__(kAppendThreads) kv_append_kernel(
    const __grid_constant__ AppendParams P) {
  const long long total = P.end[P.n - 1];
  const int lane = threadIdx.x & 31;
  for (long long u0 = (long long)blockIdx.x * kAppendWarps + (threadIdx.x >> 5); u0 < total;
       u0 += (long long)gridDim.x * kAppendWarps) {
    int di = 0;
    while (di + 1 < P.n && u0 >= P.end[di]) ++di;
    const AppendDev &D = P.d[di];
    const int tok = (int)(u0 - (di > 0 ? P.end[di - 1] : 0));
    const int half = D.hkv * kPieces, n = 2 * half;  // pieces of K, of K and V
    const uint4 *ks = reinterpret_cast<const uint4 *>(D.k_new) + (size_t)tok * half;
    const uint4 *vs = reinterpret_cast<const uint4 *>(D.v_new) + (size_t)tok * half;
    uint4 v[kAppendLoads];
    auto load = [&](int p0) {
#pragma unroll
      for (int j = 0; j < kAppendLoads; ++j) {
        const int p = p0 + 32 * j + lane;
        if (p < n) v[j] = p < half ? ks[p] : vs[p - half];
      }
    };
    load(0);
    // a row that no request's offsets cover is not written
    if (tok < D.cu_new[0] || tok >= D.cu_new[D.num_reqs]) {
      if (lane == 0) ipd_set_error(&g_kv_err, IPD_DEVERR_SPAN);
      continue;
    }
    const int r = warp_find_request(D.cu_new, D.num_reqs, tok);
    const int first = D.cu_new[r], len = D.seq_len[r];
    const int pos = len - (D.cu_new[r + 1] - first) + (tok - first);  // absolute position of the row
    if (pos < 0 || pos >= len || (pos >> 4) >= D.max_pages) {
      if (lane == 0) ipd_set_error(&g_kv_err, IPD_DEVERR_SEQ_LEN);
      continue;
    }
    const int page = D.page_table[(size_t)r * D.max_pages + (pos >> 4)];
    if (page < 0 || page >= D.num_pages) {
      if (lane == 0) ipd_set_error(&g_kv_err, IPD_DEVERR_PAGE_ID);
      continue;
    }
    // head 0's row of the slot; head h's is 16 rows further per head
    const size_t slot = ((size_t)page * D.hkv * 16 + (pos & 15)) * kPieces;
    uint4 *kd = reinterpret_cast<uint4 *>(D.k_pages) + slot;
    uint4 *vd = reinterpret_cast<uint4 *>(D.v_pages) + slot;
    for (int p0 = 0; p0 < n; p0 += 32 * kAppendLoads) {
      if (p0 > 0) load(p0);
#pragma unroll
      for (int j = 0; j < kAppendLoads; ++j) {
        const int p = p0 + 32 * j + lane;
        if (p >= n) break;
        const int q = p < half ? p : p - half;
        (p < half ? kd : vd)[(size_t)(q / kPieces) * 16 * kPieces + q % kPieces] = v[j];
      }
    }
  }
}

// Host validation of one append; fills its device descriptor.  IPD_OK with
// total_new == 0 for an append with no rows.
int check_append(const ipd_kv_append_desc &a, AppendDev *d) {
  if (a.num_reqs < 0 || a.total_new < 0 || a.num_pages < 0 || a.num_kv_heads < 1 ||
      a.max_pages < 1)
    return IPD_ERR_INVALID_ARG;
  if (a.page_size != 16 || a.head_dim != 128) return IPD_ERR_UNSUPPORTED;
  *d = AppendDev{};
  if (a.total_new == 0) return IPD_OK;
  if (a.num_reqs == 0 || !a.k_pages || !a.v_pages || !a.k_new || !a.v_new || !a.cu_new ||
      !a.seq_len || !a.page_table)
    return IPD_ERR_INVALID_ARG;
  if (((uintptr_t)a.k_pages | (uintptr_t)a.v_pages | (uintptr_t)a.k_new | (uintptr_t)a.v_new) &
      15)
    return IPD_ERR_INVALID_ARG;
  *d = AppendDev{a.k_pages, a.v_pages, a.k_new, a.v_new, a.cu_new, a.seq_len, a.page_table,
                 a.num_pages, a.total_new, a.num_kv_heads, a.max_pages, a.num_reqs};
  return IPD_OK;
}

int launch_appends(const ipd_kv_append_desc *descs, int n, ipd_stream_t stream) {
  if (n < 0 || n > IPD_MAX_BATCHES || (n > 0 && !descs)) return IPD_ERR_INVALID_ARG;
  AppendParams P;
  memset(&P, 0, sizeof(P));
  long long total = 0;
  for (int i = 0; i < n; ++i) {
    AppendDev d;
    const int st = check_append(descs[i], &d);
    if (st != IPD_OK) return st;
    if (d.total_new == 0) continue;  // nothing to write: not part of the launch
    P.d[P.n] = d;
    total += d.total_new;
    P.end[P.n] = total;
    ++P.n;
  }
  if (P.n == 0) return IPD_OK;
  const long long blocks = (total + kAppendWarps - 1) / kAppendWarps;
  const int grid = (int)(blocks < 8192 ? blocks : 8192);
  kv_append_kernel<<<grid, kAppendThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(P);
  if (cudaGetLastError() != cudaSuccess) return IPD_ERR_CUDA;
  return IPD_OK;
}

}  // namespace

extern "C" __attribute__((visibility("hidden"))) unsigned int ipd_internal_take_kv_error() {
  unsigned int v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_kv_err, sizeof(v)) != cudaSuccess) return 0xffffffffu;
  if (cudaMemcpyToSymbol(g_kv_err, &z, sizeof(z)) != cudaSuccess) return 0xffffffffu;
  return v;
}

extern "C" int ipd_kv_append(uint16_t *k_pages, uint16_t *v_pages, int64_t num_pages,
                             int num_kv_heads, int page_size, int head_dim,
                             const uint16_t *k_new, const uint16_t *v_new, const int32_t *cu_new,
                             const int32_t *seq_len, const int32_t *page_table, int max_pages,
                             int num_reqs, int total_new, ipd_stream_t stream) {
  const ipd_kv_append_desc a{k_pages, v_pages, num_pages, num_kv_heads, page_size, head_dim,
                             k_new,   v_new,   cu_new,    seq_len,      page_table, max_pages,
                             num_reqs, total_new};
  return launch_appends(&a, 1, stream);
}

extern "C" int ipd_kv_append_many(const ipd_kv_append_desc *appends, int n,
                                  ipd_stream_t stream) {
  return launch_appends(appends, n, stream);
}
