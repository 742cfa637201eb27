// Shared internals of libhoccl: the communicator object and small helpers used by the executors, the point-to-point
// path, the pattern executor and the C ABI.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstring>
#include <deque>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "../../include/hoccl.h"
#include "../../include/hoccl_diag.h"
#include "kernels.cuh"
#include "plan.h"
#include "options.h"
#include "proxy.h"
#include "sched.h"

namespace hoccl {

constexpr int kMaxRanks = 64;
constexpr int kMaxLanes = 8;
constexpr size_t kGraphCacheCap = 48;

inline double now_us() {
  return std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

struct Seg {
  const char* src;    // MOVE: source; SUM: inbox
  const char* local;  // SUM only
  char* dst;
  uint64_t bytes;
  uint64_t host_off = 0;  // HOCCL_PATH_CE_HOST: where this move bounces in the pinned host staging
  int nsrc = 1;           // OP_CHAIN: inbox operands at src + j * src_stride
  uint64_t src_stride = 0;
  // OP_CHAIN that reads the contributions where they lie (see contributions() in exec.cu): all operands in the order of addition, the owner's
  // last; and, if the sum stores the result for every rank, all destinations (otherwise `dst`)
  std::vector<const void*> ops;
  std::vector<void*> dsts;
  bool host_first = true; // HOCCL_PATH_CE_HOST: this move issues the outbound copy into host_off (false: another move of the group did)
};

// One kernel launch of a schedule: the batch is its only parameter, by value.  The kernel is one that launch_in_order may start.
struct KernelLaunch {
  const void* fn = nullptr;
  int grid = 0, threads = 0;
  std::vector<char> args;
  double bytes = 0;   // algorithmic bytes
  long moves = 0;     // MOVE operations it carries (0: a sum)
  int priority = 0;   // of the launch; 0: the stream's
};

struct RGroup {
  int kind;
  int piece;
  int phase = 0;   // plan phase of the group (reduce-scatter, all-gather, own chunk, all-to-all stage)
  std::vector<Seg> segs;
  std::vector<int> deps;
  int chain_dep;
  std::vector<KernelLaunch> ready;   // if not empty, the launches that carry out the group (instead of batches built from segs)
  long ctas = 0;        // moves on the move kernel: its CTAs, 0 = "copy_ctas"
  bool beside = false;  // sums: driver copies of another piece run beside them
  bool edges = false;   // copy route: the ends of driver copies, carried by a copy-kernel launch (see trim_driver_copies)
};

struct Post {
  bool is_send;
  void* buf;
  size_t count;
  int dtype;
  cudaStream_t stream;
  cudaEvent_t at_post;   // recorded on `stream` when the post was made: the move waits for this point, not for later work
};

// One host <-> staging copy of the pipelined host all-reduce: `rows` rows of `width` bytes at `pitch` (rows == 1: plain).
struct HostCopy {
  char* dev;
  char* host;
  size_t pitch, width, rows;
};

struct GraphEntry {
  std::vector<uint64_t> key;
  cudaGraphExec_t exec = nullptr;
  std::vector<KernelLaunch> launches;   // the same work as `exec`, for a call of a burst (see launch_entry)
  double est_us = 0;                    // what they take, roughly: 1.5 (sums) or 2.5 us (moves) each, HBM, 90 GB/s per summing and 45 per moving CTA
  uint64_t last_use = 0;
  long n_moves = 0, n_move_launches = 0, n_sum_launches = 0, n_pieces = 0, n_order_launches = 0;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_events;  // owned; only with profile = 1
  std::vector<double> prof_bytes;
  bool prof_pending = false;  // replayed since the profile events were last read
  // pipelined host all-reduce: one graph per piece, and the host copies in front of and behind each of them
  std::vector<cudaGraphExec_t> piece_exec;
  std::vector<std::vector<HostCopy>> h2d, d2h;   // [piece]
  // "ce_overlap" setting: per piece three graphs (the reduce-scatter's moves, the sum, the all-gather's moves) that run on three
  // internal streams, so that one piece's driver copies overlap another piece's sum (inside ONE graph they never did)
  std::vector<cudaGraphExec_t> part_exec;   // [piece * 3 + part], null where a part is empty
  std::vector<std::vector<KernelLaunch>> part_sums;   // [piece]: the sums as launches instead of a graph (Layout::sums_by_launch)
  // "fused" setting: the whole plan as one cooperative kernel instead of a graph (exec stays null)
  std::vector<char> ring_args;  // a RingArgsSmall or RingArgsLarge, by value
  bool ring_large = false;
  int ring_grid = 0, ring_threads = 0;
  bool ring_has_sum = false;
  // "roles" setting: the direct schedule as one cooperative kernel with summing and moving CTAs (exec stays null)
  char* roles_tab = nullptr;    // owned device memory: the segment tables of this call signature
  std::vector<char> roles_args; // a RolesArgs, by value
  const void* roles_fn = nullptr;
  int roles_grid = 0, roles_sum_ctas = 0;
  size_t roles_smem = 0;        // dynamic shared memory of the launch = size of the tables
};

}  // namespace hoccl

struct hoccl_comm {
  int R = 0, device = 0, num_sms = 0;
  hoccl_path_t path = HOCCL_PATH_CE;
  long sum_ctas = 8, copy_ctas = 8, piece_bytes = 4 << 20, max_pieces = 8, lanes = 4, use_graph = 1, profile = 0, p2p_split = 1, ce_sub_bytes = 0,
       handshake = 0, watchdog_ms = 10000, onepass = 0, forward = 0, fused = 0, host_pieces = 8, ag_direct = 2, order_kernels = 1, rs_direct = 2,
       ce_small_bytes = 8 << 20, ce_small_ctas = 148, p2p_strict = 0, ce_overlap = -1, model_gpus_per_node = 0, model_rdma_sub_bytes = 0, roles = 0, piece_grade = -1,
       roles_missing = 0 /* self-test only: summing CTAs wait for this many movers that do not exist */;
  bool piece_bytes_set = false;  // the caller chose a piece size: no automatic choice
  bool host_pieces_set = false;  // the same for "host_pieces"
  hoccl::Proxy* proxy = nullptr;
  cudaStream_t lane[hoccl::kMaxLanes] = {};
  cudaStream_t sum_stream = nullptr;
  int sum_priority = 0;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_next = 0;
  void* scratch = nullptr;
  size_t scratch_bytes = 0;
  void* staging = nullptr;
  size_t staging_bytes = 0;
  unsigned* ring_bar = nullptr;  // "fused" setting: three device words of the grid barrier (library owned, 16 bytes)
  int* ring_err = nullptr;       // mapped pinned host word the ring kernel sets when a barrier wait ran out
  int* ring_err_dev = nullptr;   // the same word as the device sees it
  char* roles_ctl = nullptr;     // "roles" setting: control words and per-piece counters of the roles kernel (library owned, 1 KiB)
  int* roles_err = nullptr;      // mapped pinned host word the roles kernel sets when a wait ran out
  int* roles_err_dev = nullptr;
  char* host_staging = nullptr;  // pinned host memory of the CE_HOST path
  size_t host_staging_bytes = 0;
  std::map<std::pair<int, int>, std::deque<hoccl::Post>> pending;
  std::vector<cudaEvent_t> post_events;   // free list of the events that mark parked posts
  int n_pending = 0;
  unsigned p2p_rr = 0;
  std::vector<hoccl::GraphEntry> cache;
  uint64_t use_counter = 0;
  hoccl_stats_t stats = {};
  std::string cuda_err;
  // profile accumulation
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_pool;   // timing events of the stream executor
  std::vector<std::pair<std::pair<cudaEvent_t, cudaEvent_t>, double>> prof_open;  // recorded, not yet read
  double prof_ms = 0, prof_bytes = 0;
  long prof_n = 0;
  double prof_copy_ms = 0, prof_copy_bytes = 0;   // copy_kernel launches (graph executor)
  long prof_copy_n = 0;
};

namespace hoccl {

inline hoccl_result_t cuda_fail(hoccl_comm* c, cudaError_t e, const char* what) {
  if (c) {
    c->cuda_err = std::string(what) + ": " + cudaGetErrorString(e);
  }
  return HOCCL_ERR_CUDA;
}

#define CU_TRY(c, call)                                   \
  do {                                                    \
    cudaError_t e__ = (call);                             \
    if (e__ != cudaSuccess) return cuda_fail(c, e__, #call); \
  } while (0)

inline cudaEvent_t next_event(hoccl_comm* c) {
  if (c->ev_next == c->ev_pool.size()) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    c->ev_pool.push_back(e);
  }
  return c->ev_pool[c->ev_next++];
}

inline bool ranges_overlap(const char* a, size_t an, const char* b, size_t bn) {
  if (an == 0 || bn == 0) return false;
  return a < b + bn && b < a + an;
}

struct Call {
  int kind;  // PlanKind
  size_t count;
  int dtype;
  bool in_place;
  size_t send_bytes, recv_bytes;
  const void* const* send;
  void* const* recv;
  // hoccl_host_allreduce, pipelined form: the caller's HOST buffers; send/recv then point into the device staging and
  // the graph carries, per piece, the host-to-device copies in front of the ring and the device-to-host copies behind it
  const void* const* h_send = nullptr;
  void* const* h_recv = nullptr;
};

// A call laid out: its plan, and the plan's groups over the call's addresses.
struct Layout {
  Plan plan;
  std::vector<RGroup> groups;
  size_t host_need = 0;   // bytes of pinned host staging the moves bounce through (HOCCL_PATH_CE_HOST)
  bool overlap = false;   // copy route: the pieces' parts run on three internal streams
  bool sums_by_launch = false;   // of those the sums go out as launches, not as graphs
  // inspect_call only: per group, the CTAs of its largest kernel launch (0 = driver copies); per piece, copy_chains
  std::vector<int> ctas, chains;
};

// What a driver copy inside one device does at once, as timed on B200: a copy of 1 MiB or more whose destination does not start on a
// 128-byte line or whose length is not a multiple of 4 KiB takes 4 us more than a whole one (8 MiB 8.3 against 4.3 us, 64 MiB 28.7
// against 24.6), one whose ends differ modulo 4 runs at half the rate.
constexpr size_t kDriverLine = 128, kDriverPage = 4096, kDriverWhole = 1 << 20, kDriverShort = 4 << 20;
inline bool bad_for_driver(const char* src, const char* dst, size_t bytes) {
  return bytes >= kDriverWhole && (bytes % kDriverPage || (uintptr_t)dst % kDriverLine || (((uintptr_t)src ^ (uintptr_t)dst) & 15));
}

// "ce_small_ctas" from which a launch of the move kernel carries copies no slower than the driver does; from kWideMoves on the rules of the
// callers hold as they were measured, with 148.  A CTA copies 46 GB/s (one store per load; all-gathers 58), driver copies side by side whole ones at
// 3.1 TB/s, with odd ends at 1.4, with ends that differ modulo 4 at 0.65, and none in less than 0.5 us.  Us in driver copies / on 16 / 32 / 64 CTAs: all-gather of
// 64 MiB per rank over 8 ranks, whole 174 / 555 / 279 / 141, 16 bytes short per block 371 / 558 / 281 / 142, 2 bytes out of phase 816 / 559 / 282 / 144;
// all-to-all of 16 MiB over 8 ranks 51 / 175 / 89 / 49, of 64 MiB 16 bytes short 384 / 722 / 362 / 190; over 64 ranks in blocks of 280 KB 1884 / 1673 / 919 / 579.
constexpr long kWideMoves = 128;
inline double kernel_ahead_from(const char* src, const char* dst, size_t bytes) {
  const double copies = bad_for_driver(src, dst, bytes) ? ((((uintptr_t)src ^ (uintptr_t)dst) & 3) ? 16 : 32) : 64;
  return std::max(1.0, std::min((double)bytes / 20e3, copies));
}

// The move route of one call: the communicator shows it for the call only.
struct RouteGuard {
  hoccl_comm* c;
  hoccl_path_t path;
  long ctas;
  RouteGuard(hoccl_comm* comm, hoccl_path_t p, long n) : c(comm), path(comm->path), ctas(comm->copy_ctas) {
    c->path = p;
    c->copy_ctas = n;
  }
  ~RouteGuard() {
    c->path = path;
    c->copy_ctas = ctas;
  }
};

struct Tally {
  long moves = 0, move_launches = 0, sum_launches = 0;
};

// exec.cu
// The kernel launches that carry out one group: its sums, or (SM route) its moves.
std::vector<KernelLaunch> kernel_launches(const hoccl_comm* c, const Plan& P, const RGroup& g);
cudaError_t launch_kernel(const KernelLaunch& k, cudaStream_t stream);
hoccl_result_t launch_sum_kernel(hoccl_comm* c, const KernelLaunch& k, cudaStream_t stream);   // ... between two events if "profile" is set
template <class Batch>
inline KernelLaunch make_launch(const Batch& b, const void* fn, long grid, int threads, double bytes, long moves) {
  KernelLaunch k;
  k.fn = fn;
  k.grid = (int)grid;
  k.threads = threads;
  k.args.assign(reinterpret_cast<const char*>(&b), reinterpret_cast<const char*>(&b) + sizeof(b));
  k.bytes = bytes;
  k.moves = moves;
  return k;
}
// The launches of the move kernel that carry out a group of moves, prepared for `ctas` CTAs: moves with one source, one length and one
// 16-byte phase of the destination share a segment (one read, one store per destination).
std::vector<MoveBatch> pack_moves(const RGroup& g, int ctas);
// The same sharing as the roles kernel takes it over, in batches of its own.  Returns false (and leaves *out empty) if no source
// repeats: plain copies are used then.  bytes_out[i] = HBM bytes of batch i (reads + writes), moves_out[i] = moves it carries.
bool build_fan_batches(const RGroup& g, std::vector<FanBatch>* out, std::vector<double>* bytes_out, std::vector<long>* moves_out);
// graph.cu
// Fills entry->launches and est_us if the groups are at most kMaxChainLaunches kernels, each waiting for the one before it.  (Inside a graph a
// kernel follows another in 0.65 us, so longer chains, and calls with something to overlap, lose nothing there.)
constexpr size_t kMaxChainLaunches = 3;
// They stay in the groups (`ready`) for the graph that is built of them next: made twice they cost a first call up to 45 us of 240 (16 ranks).
void add_launches(const hoccl_comm* c, const Plan& P, std::vector<RGroup>* groups, GraphEntry* entry);
// In how many chains the copies of this piece's all-gather run beside the next piece's sum; 0: all at once.
constexpr size_t kMaxCopyChains = 6;
size_t copy_chains(const hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, int piece);
// part < 0: every group (of `only_piece`, if that is >= 0); part 0 / 1 / 2: only the reduce-scatter's MOVE groups / the SUM and
// CHAIN groups / the remaining MOVE groups; dependencies on groups outside the part are left to the caller (events).
// *out_exec stays null when nothing falls into the selection.
hoccl_result_t build_graph(hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, GraphEntry* entry, int only_piece,
                           cudaGraphExec_t* out_exec, int part = -1);
void add_host_copies(const Plan& P, int p, char* dev, char* host, std::vector<HostCopy>* out);
cudaError_t enqueue_host_copy(const HostCopy& hc, bool to_device, cudaStream_t s);
// ring_host.cu
hoccl_result_t build_ring(hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, GraphEntry* entry);
// roles.cu
hoccl_result_t build_roles(hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, GraphEntry* entry);
hoccl_result_t launch_roles(hoccl_comm* c, GraphEntry* entry, cudaStream_t stream);
// exec.cu
hoccl_result_t run_collective(hoccl_comm* c, Call* call, cudaStream_t user);
// What run_collective would run for this call, and the signature its graph would be cached under; nothing is enqueued.
hoccl_result_t inspect_call(hoccl_comm* c, Call* call, Layout* out, std::vector<uint64_t>* key);
hoccl_result_t run_streams(hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, cudaStream_t user, Tally* tally);
// HOCCL_OK if the communicator's settings fit together for such a call (see options.h); nothing is enqueued
hoccl_result_t check_options(hoccl_comm* c, int kind, size_t count, int dtype);
hoccl_result_t ensure_proxy(hoccl_comm* c);
void harvest_profile(hoccl_comm* c);
void destroy_entry(GraphEntry* e);
GraphEntry* cache_put(hoccl_comm* c, GraphEntry&& entry);
hoccl_result_t build_pattern_graph_modelled(hoccl_comm* c, const Schedule& S, const void* const* send, const size_t* sdispls,
                                            void* const* recv, const size_t* rdispls, size_t e, char* out_stage, char* in_stage,
                                            const std::vector<uint64_t>& flow_stage_off, size_t chunk_bytes, size_t rdma_sub,
                                            GraphEntry* entry);
hoccl_result_t ring_barrier_selftest(hoccl_comm* c, void* dst, const void* src, size_t bytes, cudaStream_t stream);
// Replays a cached graph into the caller's stream (directly, or through the CPU proxy in handshake mode).
hoccl_result_t launch_entry(hoccl_comm* c, GraphEntry* hit, cudaStream_t user, double t0);
// host_entry.cu: the pipelined hoccl_host_allreduce on the automatic direct schedule
constexpr size_t kHostInPlaceBytes = 72000000;   // R * S up to which its sums store for every rank; above, launches of moves do (see host_entry.cu)
// The caller's host buffers as kernels see them.
struct HostViews {
  const char* send[kMaxRanks];
  char* recv[kMaxRanks];
};
bool host_direct_applies(const hoccl_comm* c, const Call& call, const OptionsOut& opt, HostViews* views);
hoccl_result_t run_host_direct(hoccl_comm* c, const Call& call, const HostViews& views, cudaStream_t user, double t0);
size_t host_pieces(const hoccl_comm* c, size_t S, double unit);
hoccl_result_t run_host_in_place(hoccl_comm* c, const Call& call, std::vector<uint64_t>&& key, cudaStream_t user, double t0);
// p2p.cu
hoccl_result_t p2p_post(hoccl_comm* c, bool is_send, void* buf, size_t count, int dtype, int src, int dst, cudaStream_t stream);

}  // namespace hoccl
