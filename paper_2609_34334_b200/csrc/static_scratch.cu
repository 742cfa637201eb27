// hoccl_allreduce_static: the ring all-reduce for callers that are not allowed to allocate.
//
// Some users of this library run where device allocation is off limits: a communication thread that
// works beside training kernels and must never trigger the device-wide synchronisation an allocation
// can imply, or a process whose device memory is handed out once by a static memory planner so that no
// byte is left to ask for.  They cannot attach scratch to a communicator either, because they have none
// to give.  For them the ring's inbox and partial slots live in the fixed array below, which is part of
// the library image: every GPU that loads the library holds it from module load until the process ends.
//
// Nothing here calls cudaMalloc, cudaFree, or creates streams, events or graphs: the whole schedule is
// issued as kernel launches on the caller's stream in the planner's (topological) order.
//
// Buffers that share their address modulo 16 (the usual case) do not need the scratch at all: the chain sum reads every rank's
// contribution where it lies, as the communicator's automatic schedule does, and one launch of moves, or the sum itself, brings
// the result to every rank (6 ranks of 500,009 fp32: 123 us as a ring of 15 launches, 17 us as two).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "../../include/hoccl.h"
#include "kernels.cuh"
#include "plan.h"

using namespace hoccl;

namespace {

// The scratch itself.  In host code this name is only a handle for the runtime's symbol table, not a
// device address: its address on a given device comes from cudaGetSymbolAddress (see scratch_base).
static __device__ __align__(256) unsigned char g_static_scratch[HOCCL_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
constexpr int kStaticSumCtas = 8;    // same SM budget for sums as the communicator's default
constexpr int kStaticCopyCtas = 32;    // of the ring's copies, which run between its sums
constexpr int kStaticMoveCtas = 148;   // of the one launch of moves behind the sums: the whole GPU, as the communicator's short moves (6 ranks of
                                       // 500,009 fp32 21.4 us on 32 CTAs, 16.7; of 8 MiB 80.7 and 58.5)
std::mutex g_mu;
void* g_base[kMaxDevices] = {};

// Device address of the array on the CURRENT device; looked up once per device.
cudaError_t scratch_base(int device, void** out) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_base[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_base[device] = p;
  }
  *out = g_base[device];
  return cudaSuccess;
}

// The all-reduce in one or two launches for buffers of one 16-byte phase.  q: elements of a full ring chunk.
cudaError_t read_in_place(const void* const* send, void* const* recv, size_t count, size_t q, int dtype, size_t e, int R, cudaStream_t st) {
  const bool store_all = (size_t)R * count * e <= (size_t)kStaticSumCtas * kStoreAllBytesPerCta;
  if (store_all) {
    StoreAllArgs a;
    int grid = 0, threads = 0;
    const void* fn = store_all_entry(R, dtype, kStaticSumCtas, count, &a, &grid, &threads);
    if (fn) {
      a.phase = (unsigned)((uintptr_t)send[0] & 15);
      for (int r = 0; r < R; r++) {
        a.x[r] = send[r];
        a.y[r] = recv[r];
      }
      return launch_in_order(fn, grid, threads, &a, st);
    }
  }
  ChainBatch b;
  MoveBatch m;
  b.dtype = dtype;
  b.nseg = b.nptr = 0;
  m.nseg = m.ndst_total = 0;
  cudaError_t err = cudaSuccess;
  // all sums first: a chunk is final before any move of it is issued
  for (int c = 0; c < R && err == cudaSuccess; c++) {
    const size_t lo = std::min((size_t)c * q, count), n = std::min(lo + q, count) - lo;
    if (!n) continue;
    const void* ops[64];
    void* dsts[64];
    for (int j = 1; j <= R; j++) ops[j - 1] = (const char*)send[(c + j) % R] + lo * e;
    for (int r = 0; r < R; r++) dsts[r] = (char*)recv[(c + r) % R] + lo * e;   // the owner's first
    const int ndst = store_all ? R : 1;
    if (!add_chain_seg(&b, ops, R, dsts, ndst, (unsigned long long)n)) {
      err = launch_chain(b, kStaticSumCtas, st);
      b.nseg = b.nptr = 0;
      add_chain_seg(&b, ops, R, dsts, ndst, (unsigned long long)n);
    }
  }
  if (err == cudaSuccess) err = launch_chain(b, kStaticSumCtas, st);
  for (int c = 0; c < R && !store_all && err == cudaSuccess; c++) {
    const size_t lo = std::min((size_t)c * q, count), n = std::min(lo + q, count) - lo;
    if (!n) continue;
    void* dsts[64];
    for (int k = 1; k < R; k++) dsts[k - 1] = (char*)recv[(c + k) % R] + lo * e;
    if (!add_move_seg(&m, (const char*)recv[c] + lo * e, dsts, R - 1, (unsigned long long)(n * e))) {
      err = launch_moves(&m, kStaticMoveCtas, st);
      m.nseg = m.ndst_total = 0;
      add_move_seg(&m, (const char*)recv[c] + lo * e, dsts, R - 1, (unsigned long long)(n * e));
    }
  }
  return err == cudaSuccess ? launch_moves(&m, kStaticMoveCtas, st) : err;
}

bool overlap(const char* a, size_t an, const char* b, size_t bn) { return an && bn && a < b + bn && b < a + an; }

}  // namespace

extern "C" hoccl_result_t hoccl_allreduce_static(const void* const* send, void* const* recv, size_t count, hoccl_dtype_t dtype,
                                                 hoccl_op_t op, int R, hoccl_stream_t stream) {
  if (!send || !recv || R < 1 || R > 64) return HOCCL_ERR_INVALID_ARG;
  if (op != HOCCL_SUM) return HOCCL_ERR_UNSUPPORTED;
  const size_t e = dtype_size((int)dtype);
  if (e == 0) return HOCCL_ERR_UNSUPPORTED;
  const size_t bytes = count * e;
  int n_in = 0;
  for (int r = 0; r < R; r++) {
    if (!send[r] || !recv[r]) return HOCCL_ERR_INVALID_ARG;
    if (((uintptr_t)send[r] % e) || ((uintptr_t)recv[r] % e)) return HOCCL_ERR_INVALID_ARG;
    if (send[r] == recv[r]) n_in++;
    else if (overlap((const char*)send[r], bytes, (const char*)recv[r], bytes)) return HOCCL_ERR_INVALID_ARG;
  }
  if (n_in != 0 && n_in != R) return HOCCL_ERR_INVALID_ARG;
  for (int a = 0; a < R; a++)
    for (int b = a + 1; b < R; b++) {
      const char *sa = (const char*)send[a], *sb = (const char*)send[b], *da = (const char*)recv[a], *db = (const char*)recv[b];
      if (overlap(sa, bytes, sb, bytes) || overlap(da, bytes, db, bytes) || overlap(sa, bytes, db, bytes) || overlap(da, bytes, sb, bytes))
        return HOCCL_ERR_INVALID_ARG;
    }
  if (count == 0) return HOCCL_OK;

  if (R > 1) {
    const size_t q = (count + R - 1) / R;
    if (2 * (size_t)R * ((q * e + 16 + 255) / 256 * 256) > (size_t)HOCCL_STATIC_SCRATCH_BYTES) return HOCCL_ERR_SCRATCH;
    bool one_phase = true;
    for (int r = 0; r < R; r++) one_phase = one_phase && !((((uintptr_t)send[r] ^ (uintptr_t)send[0]) | ((uintptr_t)recv[r] ^ (uintptr_t)send[0])) & 15);
    if (one_phase)
      return read_in_place(send, recv, count, q, (int)dtype, e, R, (cudaStream_t)stream) == cudaSuccess ? HOCCL_OK : HOCCL_ERR_CUDA;
  }

  // one piece per ring chunk: the schedule runs on one stream, so pieces would buy nothing
  Plan P;
  unsigned char align[64];
  for (int r = 0; r < R; r++) align[r] = (unsigned char)((uintptr_t)send[r] & 15);
  if (!build_plan(&P, PLAN_ALLREDUCE, R, count, (int)dtype, n_in == R, (size_t)1 << 40, 1, align)) return HOCCL_ERR_INVALID_ARG;
  const size_t need = 2 * (size_t)R * P.slot_bytes;
  if (need > (size_t)HOCCL_STATIC_SCRATCH_BYTES) return HOCCL_ERR_SCRATCH;   // beyond the fixed maximum

  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= kMaxDevices) return HOCCL_ERR_CUDA;
  void* base = nullptr;
  if (P.slot_bytes && scratch_base(device, &base) != cudaSuccess) return HOCCL_ERR_CUDA;
  char* inbox0 = (char*)base;
  char* partial0 = inbox0 + (size_t)R * P.slot_bytes;
  auto addr = [&](int buf, int rank, uint64_t off) -> char* {
    switch (buf) {
      case BUF_SEND: return (char*)send[rank] + off;
      case BUF_RECV: return (char*)recv[rank] + off;
      case BUF_INBOX: return inbox0 + (size_t)rank * P.slot_bytes + off;
      default: return partial0 + (size_t)rank * P.slot_bytes + off;
    }
  };
  cudaStream_t st = (cudaStream_t)stream;
  // Groups are stored in a topological order of the plan's DAG; on a single stream that order is a valid schedule.
  for (const PlanGroup& g : P.groups) {
    for (int first = 0; first < g.num_ops; first += kMaxSegs) {
      const int n = std::min(kMaxSegs, g.num_ops - first);
      cudaError_t err;
      if (g.kind == OP_SUM) {
        SumBatch b;
        b.nseg = n;
        b.dtype = (int)dtype;
        for (int i = 0; i < n; i++) {
          const PlanOp& o = P.ops[g.first_op + first + i];
          b.seg[i] = SumSeg{addr(o.src_buf, o.rank, o.src_off), addr(o.local_buf, o.rank, o.local_off), addr(o.dst_buf, o.rank, o.dst_off),
                            (unsigned long long)(o.bytes / e)};
        }
        err = launch_sum(b, kStaticSumCtas, st);
      } else {
        CopyBatch b;
        b.nseg = n;
        b.pad = 0;
        for (int i = 0; i < n; i++) {
          const PlanOp& o = P.ops[g.first_op + first + i];
          b.seg[i] = CopySeg{addr(o.src_buf, o.rank, o.src_off), addr(o.dst_buf, o.dst_rank, o.dst_off), (unsigned long long)o.bytes};
        }
        err = launch_copy(b, kStaticCopyCtas, st);
      }
      if (err != cudaSuccess) return HOCCL_ERR_CUDA;
    }
  }
  return HOCCL_OK;
}
