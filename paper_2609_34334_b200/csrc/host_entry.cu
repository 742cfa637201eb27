// The pipelined hoccl_host_allreduce on the automatic direct schedule: how the vectors cross PCIe (paper Sec. 3.3.1, chunk pipelining,
// applied to that link) and which sums run on what has arrived.
#include <cuda.h>

#include <cmath>

#include "comm.h"

namespace hoccl {

// The sums of bytes [a, b) of the vector: one segment per ring chunk the range touches (the order of the adds is the chunk's), stored
// to every dst.
static RGroup range_sums(int R, const char* const* src, char* const* dst, int ndst, size_t a, size_t b, size_t chunk, int piece) {
  RGroup g;
  g.kind = OP_CHAIN;
  g.piece = piece;
  g.phase = PHASE_RS;
  g.chain_dep = -1;
  for (size_t at = a; at < b;) {
    const int owner = (int)(at / chunk);
    Seg s = {};
    s.bytes = std::min<size_t>(std::min(b, (size_t)(owner + 1) * chunk) - at, kMaxChainSegBytes);
    for (int j = 1; j <= R; j++) s.ops.push_back(src[(owner + j) % R] + at);
    s.dst = dst[0] + at;
    if (ndst > 1)
      for (int d = 0; d < ndst; d++) s.dsts.push_back(dst[d] + at);
    g.segs.push_back(std::move(s));
    at += g.segs.back().bytes;
  }
  return g;
}

// Host all-reduce whose sums read the ranks' staging buffers in place: no schedule over ring chunks is left, so a piece is one
// contiguous range of the vector (one plain copy per rank and direction instead of a 2-D copy and one for the shorter last chunk),
// the sum writes it once, and every rank's result is copied out of that one buffer.
// Pieces: with np equal pieces the two directions overlap in all but one piece each, (1 + 1 / np) S R / 50 GB/s, and every copy costs
// 6 to 9 us beside one of the other direction, np R of them; so the best np grows with the root of S (1 up to 1 MiB per rank, 3 at 4 MiB,
// 5 at 16 MiB).  Measured over 8 ranks against 8 pieces of every ring chunk: 64 KiB per rank 122 -> 89 us, 1 MiB 403 -> 380, 4 MiB 1372 ->
// 1087, 8 MiB 2120 -> 2060; over 3 ranks 64 KiB 74 -> 38, 1 MiB 243 -> 150, 16 MiB 1541 -> 1460.
// Size from which the 2-D pieces of the staged form serve (kHostInPlaceBytes), in place against staged, ms, 8 ranks, bytes of all ranks
// together: whole chunks 40 MB 1.33 / 1.37, 60 MB 1.91 / 1.86, 70 MB 2.06 / 2.06, 80 MB 2.36 / 2.39, 100 MB 2.86 / 2.74, 134 MB 3.72 / 3.54,
// 200 MB 5.23 / 4.99.  The line lies where the two cross; the rule looks at the size only.  Chunks of unequal length add a copy per rank and
// direction to every 2-D piece and nothing to a contiguous one: 70 MB 2.03 / 2.45, 80 MB 2.33 / 2.69, 134 MB 3.72 / 4.35, 200 MB 5.18 / 5.94 (3
// ranks, 200 MB: 5.20 / 5.31), so for them the line costs up to 0.8 ms.
size_t host_pieces(const hoccl_comm* c, size_t S, double unit) {
  if (c->host_pieces_set) return (size_t)c->host_pieces;
  return std::min<size_t>(32, std::max<size_t>(1, (size_t)(std::sqrt((double)S / unit) + 0.5)));
}
hoccl_result_t run_host_in_place(hoccl_comm* c, const Call& call, std::vector<uint64_t>&& key, cudaStream_t user, double t0) {
  const int R = c->R;
  Plan P;
  P.kind = PLAN_ALLREDUCE;
  P.R = R;
  P.dtype = call.dtype;
  P.elem = dtype_size(call.dtype);
  const size_t S = call.count * P.elem, chunk = (call.count + R - 1) / R * P.elem;
  const size_t np = host_pieces(c, S, 600e3);
  const size_t piece = ((S + np - 1) / np + 4095) & ~(size_t)4095;
  GraphEntry entry;
  entry.key = std::move(key);
  std::vector<RGroup> groups;
  char* result = (char*)call.recv[0];
  for (size_t a = 0; a < S; a += piece) {
    const size_t b = std::min(S, a + piece);
    groups.push_back(range_sums(R, (const char* const*)call.send, &result, 1, a, b, chunk, (int)groups.size()));
    entry.h2d.emplace_back();
    entry.d2h.emplace_back();
    for (int r = 0; r < R; r++) {
      entry.h2d.back().push_back(HostCopy{(char*)call.send[r] + a, (char*)call.h_send[r] + a, b - a, b - a, 1});
      entry.d2h.back().push_back(HostCopy{result + a, (char*)call.h_recv[r] + a, b - a, b - a, 1});
    }
  }
  entry.n_pieces = (long)groups.size();
  entry.piece_exec.assign(groups.size(), nullptr);
  for (size_t p = 0; p < groups.size(); p++) {
    const hoccl_result_t rc = build_graph(c, P, groups, &entry, (int)p, &entry.piece_exec[p]);
    if (rc != HOCCL_OK) {
      destroy_entry(&entry);
      return rc;
    }
  }
  return launch_entry(c, cache_put(c, std::move(entry)), user, t0);
}

// Whether a kernel can access the `bytes` bytes at `host`, and where it finds them: host memory that CUDA allocated or registered as
// one range.  Asked at every call; memory can change hands between two calls.
static bool device_view(const void* host, size_t bytes, char** out) {
  using Fn = CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
  static const Fn query = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &qr) != cudaSuccess || qr != cudaDriverEntryPointSuccess) fn = nullptr;
    return reinterpret_cast<Fn>(fn);
  }();
  if (!query) return false;
  unsigned type = 0, managed = 0;
  CUdeviceptr dev = 0, start = 0;
  size_t size = 0;
  CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* values[] = {&type, &managed, &dev, &start, &size};
  if (query(5, what, values, (CUdeviceptr)(uintptr_t)host) != CUDA_SUCCESS) return false;   // an address CUDA does not know reads as type 0
  const uintptr_t at = (uintptr_t)host;
  if (type != CU_MEMORYTYPE_HOST || managed || !dev || !start || at < (uintptr_t)start || bytes > size || at - (uintptr_t)start > size - bytes) return false;
  *out = (char*)(uintptr_t)dev;
  return true;
}

// The sums run on the host buffers themselves: loads and stores of the summing CTAs cross PCIe, both directions busy from the first
// vector to the last, one launch and no copy to wait for.  PCIe bounds it: 40 GB/s each way (52 for loads or stores alone, driver copies both ways
// at once 49.7; two CTAs already reach 39), so driver copies are ahead once their fixed costs (6 to 9 us per copy, one piece in and one piece out
// that overlap nothing) fade.  Us, 8 CTAs, against the piecewise forms: 8 ranks 64 KiB per rank 20 / 81, 1 MiB 229 / 470, 4 MiB 870 /
// 1140, 8 MiB 1750 / 2090, 11.7 MiB 2450 / 3080, 25 MiB 5150 / 5240, 40 MiB 8280 / 8050; 3 ranks 1 MiB 91 / 195; 16 ranks 1 MiB 465 / 750.
// Driver copies inbound with SM stores outbound came out behind both (8 MiB 2100 in 3 pieces): a copy beside stores takes 17 us to start.
// Within kHostInPlaceBytes it needs every buffer to be one range that CUDA pinned or registered, one 16-byte phase for all of
// them (element-wise accesses would cross the link one by one), and "host_pieces" left alone.
bool host_direct_applies(const hoccl_comm* c, const Call& call, const OptionsOut& opt, HostViews* v) {
  const size_t S = call.count * dtype_size(call.dtype);
  if (!(opt.plan_kind & PLAN_FLAG_RS_DIRECT) || c->rs_direct != 2 || c->R < 2 || opt.executor != EXEC_GRAPH || c->host_pieces_set ||
      (size_t)c->R * S > kHostInPlaceBytes)
    return false;
  for (int r = 0; r < c->R; r++) {
    char* p = nullptr;
    if (!device_view(call.h_send[r], S, &p)) return false;
    v->send[r] = p;
    if (!device_view(call.h_recv[r], S, &v->recv[r])) return false;
    if ((((uintptr_t)v->send[r] ^ (uintptr_t)v->send[0]) | ((uintptr_t)v->recv[r] ^ (uintptr_t)v->send[0])) & 15) return false;
  }
  return true;
}

hoccl_result_t run_host_direct(hoccl_comm* c, const Call& call, const HostViews& v, cudaStream_t user, double t0) {
  Plan P;
  P.kind = PLAN_ALLREDUCE;
  P.R = c->R;
  P.dtype = call.dtype;
  P.elem = dtype_size(call.dtype);
  const size_t S = call.count * P.elem, chunk = (call.count + c->R - 1) / c->R * P.elem;
  c->stats = hoccl_stats_t{};
  CU_TRY(c, cudaSetDevice(c->device));
  for (const KernelLaunch& k : kernel_launches(c, P, range_sums(c->R, v.send, v.recv, c->R, 0, S, chunk, 0))) {
    const hoccl_result_t rc = launch_sum_kernel(c, k, user);
    if (rc != HOCCL_OK) return rc;
    c->stats.n_sum_launches++;
  }
  c->stats.n_pieces = 1;
  c->stats.max_sum_ctas = c->sum_ctas;
  c->stats.host_launch_us = now_us() - t0;
  return HOCCL_OK;
}

}  // namespace hoccl
