// libhoccl: how a collective call is executed (the graphs themselves are built in graph.cu, the one-kernel form in ring_host.cu).
//
// A collective call = plan (host, plan.cpp) -> resolve the plan's buffer offsets against the caller's
// pointers -> issue.  Two issue engines consume the same plan and give the same bits:
//   * graph executor (default): the plan's group DAG becomes an explicit CUDA graph (memcpy nodes for
//     moves on the copy route, kernel nodes for sums and SM copies), instantiated once per distinct
//     call signature, cached, and replayed with one cudaGraphLaunch into the caller's stream.  A graph
//     launch is stream ordered, which is exactly the operator-level ordering the paper's stream
//     manager provides (Sec. 3.2), and it removes the per-operation host cost that the paper reports
//     as its launch overhead (Sec. 5 "CPU launch overhead").
//   * stream executor: internal move lanes plus one sum stream, ordered with CUDA events
//     (fork from the caller's stream, join back into it).
// SUM launches are chained (one at a time) so that the SM budget for sums is global, not per piece.
#include <climits>
#include <cmath>
#include <tuple>

#include "comm.h"
#include "options.h"

namespace hoccl {

hoccl_result_t validate(hoccl_comm* c, Call* call) {
  const int R = c->R;
  const size_t e = dtype_size(call->dtype);
  if (!call->send || !call->recv) return HOCCL_ERR_INVALID_ARG;
  for (int r = 0; r < R; r++) {
    if (!call->send[r] || !call->recv[r]) return HOCCL_ERR_INVALID_ARG;
    if (((uintptr_t)call->send[r] % e) || ((uintptr_t)call->recv[r] % e)) return HOCCL_ERR_INVALID_ARG;
  }
  // in-place forms
  int n_in = 0;
  for (int r = 0; r < R; r++) {
    const char* s = (const char*)call->send[r];
    const char* d = (const char*)call->recv[r];
    bool in;
    if (call->kind == PLAN_ALLREDUCE) in = (s == d);
    else if (call->kind == PLAN_REDUCE_SCATTER) in = (d == s + (size_t)r * call->count * e);
    else if (call->kind == PLAN_ALLTOALL) in = false;   // no in-place form: any overlap of send[r] and recv[r] is an error
    else in = (s == d + (size_t)r * call->count * e);
    if (in) n_in++;
    else if (ranges_overlap(s, call->send_bytes, d, call->recv_bytes)) return HOCCL_ERR_INVALID_ARG;
  }
  if (n_in != 0 && n_in != R) return HOCCL_ERR_INVALID_ARG;
  call->in_place = (n_in == R);
  // buffers of different ranks must be disjoint
  for (int a = 0; a < R; a++)
    for (int b = a + 1; b < R; b++) {
      const char *sa = (const char*)call->send[a], *sb = (const char*)call->send[b];
      const char *da = (const char*)call->recv[a], *db = (const char*)call->recv[b];
      if (ranges_overlap(sa, call->send_bytes, sb, call->send_bytes) || ranges_overlap(da, call->recv_bytes, db, call->recv_bytes) ||
          ranges_overlap(sa, call->send_bytes, db, call->recv_bytes) || ranges_overlap(da, call->recv_bytes, sb, call->send_bytes))
        return HOCCL_ERR_INVALID_ARG;
    }
  return HOCCL_OK;
}

// Host-bounce path: moves of one group with the same source and length get the same place in the host staging; the first
// of them (host_first = true) carries the outbound copy, the others only their inbound copy behind it.  Recomputes *host_need.
static void share_host_legs(std::vector<RGroup>* groups, size_t* host_need) {
  *host_need = 0;
  for (RGroup& g : *groups) {
    if (g.kind != OP_MOVE) continue;
    std::map<std::pair<const char*, uint64_t>, size_t> first_of;   // (source, bytes) -> index of the seg that owns the staging
    for (size_t i = 0; i < g.segs.size(); i++) {
      Seg& s = g.segs[i];
      auto it = first_of.find({s.src, s.bytes});
      if (it == first_of.end()) {
        first_of.emplace(std::make_pair(s.src, s.bytes), i);
        s.host_off = *host_need;
        s.host_first = true;
        *host_need += (s.bytes + 255) / 256 * 256;
      } else {
        s.host_off = g.segs[it->second].host_off;
        s.host_first = false;
      }
    }
  }
}

constexpr size_t kGradeInPlace = 4 << 20;   // ring chunk from which pieces are graded on the SM path when contributions are read in place

// How the direct reduce-scatter's contributions reach the owner's sum.
enum Contributions {
  STAGED = 0,      // moved into the owner's inbox slots first (the plan as it is)
  READ_IN_PLACE,   // the sum reads them where they lie: the plan's moves into the inbox fall away
  READ_AND_STORE   // ... and it stores the result for every rank: the all-gather's moves fall away too
};

// All ranks live in one device's memory, so a sum can read the other ranks' contributions without a copy of them.  Staging
// them costs 2 (R - 1) bytes of traffic per output byte and buys nothing for the sum, which reads R operands either way.
// Only the automatic schedule does this: "rs_direct" = 1 keeps the staged form that a rank-local owner needs.
//   * The send buffers have to share their 16-byte phase.  (Inbox slots are placed so that the operands always do; contributions
//     that do not would be summed element by element.)
//   * The host-bounce path keeps its moves: that no SM takes part in them is what it is chosen for.  The host entry keeps them for
//     long vectors (see host_pieces).
//   * It needs the scratch of the staged form all the same, although it touches none of it: whether the addresses of a call permit it is
//     known at the call, and the staged form of the same schedule is what runs when they do not.
// The sum stores for all ranks on the SM route (on the copy route the all-gather's moves are the driver's) when its grid is the
// whole GPU, or when the message is so short that the second launch and not the stores decide: a CTA stores ~60 GB/s, so R S
// bytes over n CTAs take R S / (60 n) ns against ~2.5 us for a launch of its own and the wider copy grid.  Measured, one kernel
// against two, 8-CTA sums and 148 copy CTAs: R = 8 bf16 4 KiB per rank 3.0 / 6.2 us, 384 KiB 10.3 / 12.3, 512 KiB 14.4 / 12.4;
// R = 4 fp32 512 KiB 8.2 / 10.3, 1 MiB 14.4 / 12.4; R = 2 bf16 1 MiB 8.3 / 9.0, 2 MiB 14.4 / 12.4: the line lies at R S = 3 MiB.
static Contributions contributions(const hoccl_comm* c, const Call& call, const OptionsOut& opt, size_t S) {
  if (!(opt.plan_kind & PLAN_FLAG_RS_DIRECT) || c->rs_direct != 2 || c->R < 2 || c->path == HOCCL_PATH_CE_HOST ||
      (call.h_send && (size_t)c->R * S > kHostInPlaceBytes))
    return STAGED;
  if (opt.executor != EXEC_GRAPH && opt.executor != EXEC_STREAMS && opt.executor != EXEC_PROXY) return STAGED;
  const uintptr_t phase = (uintptr_t)call.send[0] & 15;
  bool recv_too = true;
  for (int r = 0; r < c->R; r++) {
    if (((uintptr_t)call.send[r] & 15) != phase) return STAGED;
    recv_too = recv_too && ((uintptr_t)call.recv[r] & 15) == phase;
  }
  if (call.kind == PLAN_ALLREDUCE && c->path == HOCCL_PATH_SM && (opt.plan_kind & PLAN_FLAG_AG_DIRECT) && recv_too &&
      (c->sum_ctas >= 128 || (size_t)c->R * S <= (size_t)c->sum_ctas * kStoreAllBytesPerCta))
    return READ_AND_STORE;
  return READ_IN_PLACE;
}

// Copy route, contributions read in place: the all-gather's copies keep what the driver does at once and their ends (less than 128 bytes
// in front, less than 4 KiB behind) go to one launch of the copy kernel per piece, "copy_ctas" CTAs, instead of a second pass per copy.
// The ends take over what their copy waited for.  That is all they need only while no copy waits for another copy: in a ring
// all-gather a step forwards what the step before it has written, ends included, so its copies stay whole.
static void trim_driver_copies(std::vector<RGroup>* groups) {
  const size_t n = groups->size();
  for (const RGroup& g : *groups)
    for (int d : g.deps)
      if (g.kind == OP_MOVE && (*groups)[(size_t)d].kind == OP_MOVE) return;
  for (size_t g = 0; g < n; g++) {
    if ((*groups)[g].kind != OP_MOVE) continue;
    RGroup ends = (*groups)[g];
    ends.segs.clear();
    ends.edges = true;
    for (Seg& s : (*groups)[g].segs) {
      if (s.bytes < kDriverWhole) continue;
      const uint64_t head = (kDriverLine - (uintptr_t)s.dst % kDriverLine) % kDriverLine;
      const uint64_t body = (s.bytes - head) / kDriverPage * kDriverPage, tail = s.bytes - head - body;
      if (head == 0 && tail == 0) continue;
      Seg e = s;
      e.bytes = head;
      if (head) ends.segs.push_back(e);
      e.src += head + body;
      e.dst += head + body;
      e.bytes = tail;
      if (tail) ends.segs.push_back(e);
      s.src += head;
      s.dst += head;
      s.bytes = body;
    }
    if (ends.segs.empty()) continue;
    // the ends of a piece's stages wait for the same sum: one group
    if (groups->size() > n && groups->back().piece == ends.piece && groups->back().deps == ends.deps)
      groups->back().segs.insert(groups->back().segs.end(), ends.segs.begin(), ends.segs.end());
    else
      groups->push_back(std::move(ends));
  }
}

// Turns plan offsets into addresses (the plan already places pieces inside the scratch slots).
void resolve(hoccl_comm* c, const Plan& P, const Call& call, Contributions how, std::vector<RGroup>* out, size_t* host_need) {
  *host_need = 0;
  const int R = P.R;
  char* inbox0 = (char*)c->scratch;
  const size_t inbox_bytes = (size_t)P.inbox_slots * P.slot_bytes;   // one rank's inbox: 1 slot, or R-1 for the direct reduce-scatter
  char* partial0 = inbox0 + (size_t)R * inbox_bytes;
  auto addr = [&](int buf, int rank, int chunk, uint64_t off) -> char* {
    (void)chunk;
    switch (buf) {
      case BUF_SEND: return (char*)call.send[rank] + off;
      case BUF_RECV: return (char*)call.recv[rank] + off;
      case BUF_INBOX: return inbox0 + (size_t)rank * inbox_bytes + off;
      default: return partial0 + (size_t)rank * P.slot_bytes + off;
    }
  };
  out->clear();
  out->resize(P.groups.size());
  for (size_t g = 0; g < P.groups.size(); g++) {
    const PlanGroup& pg = P.groups[g];
    RGroup& rg = (*out)[g];
    rg.kind = pg.kind;
    rg.piece = pg.piece;
    rg.phase = pg.phase;
    rg.deps = pg.deps;
    rg.chain_dep = pg.chain_dep;
    for (int i = 0; i < pg.num_ops; i++) {
      const PlanOp& op = P.ops[pg.first_op + i];
      Seg s;
      s.bytes = op.bytes;
      if (op.kind == OP_MOVE) {
        s.src = addr(op.src_buf, op.rank, op.chunk, op.src_off);
        s.dst = addr(op.dst_buf, op.dst_rank, op.chunk, op.dst_off);
        s.local = nullptr;
      } else {
        s.src = addr(op.src_buf, op.rank, op.chunk, op.src_off);
        s.local = addr(op.local_buf, op.rank, op.chunk, op.local_off);
        s.dst = addr(op.dst_buf, op.dst_rank, op.chunk, op.dst_off);  // dst_rank == rank except in the forward variant
        s.nsrc = op.nsrc;
        s.src_stride = op.src_stride;
        if (op.kind == OP_CHAIN && how != STAGED) {
          for (int j = 1; j <= R; j++) s.ops.push_back((const char*)call.send[(op.rank + j) % R] + op.local_off);
          if (how == READ_AND_STORE)
            for (int r = 0; r < R; r++) s.dsts.push_back((char*)call.recv[r] + op.dst_off);
        }
      }
      if (op.kind == OP_MOVE && c->path == HOCCL_PATH_CE_HOST) {
        s.host_off = *host_need;
        *host_need += (s.bytes + 255) / 256 * 256;
      }
      rg.segs.push_back(s);
      if (op.kind == OP_CHAIN) {   // the chain kernels use 32-bit offsets inside a segment
        while (rg.segs.back().bytes > kMaxChainSegBytes) {
          Seg& head = rg.segs.back();
          Seg rest = head;
          head.bytes = kMaxChainSegBytes;
          rest.bytes -= kMaxChainSegBytes;
          rest.src += kMaxChainSegBytes;
          rest.local += kMaxChainSegBytes;
          rest.dst += kMaxChainSegBytes;
          for (const void*& p : rest.ops) p = (const char*)p + kMaxChainSegBytes;
          for (void*& p : rest.dsts) p = (char*)p + kMaxChainSegBytes;
          rg.segs.push_back(rest);
        }
      }
    }
  }
  if (how != STAGED) {   // the moves the sums do themselves
    std::vector<RGroup> kept;
    std::vector<int> remap(out->size(), -1);
    for (size_t g = 0; g < out->size(); g++) {
      RGroup& cur = (*out)[g];
      if (cur.kind == OP_MOVE && (how == READ_AND_STORE || cur.phase == PHASE_RS)) continue;
      std::vector<int> deps;
      for (int d : cur.deps)
        if (remap[d] >= 0) deps.push_back(remap[d]);
      cur.deps.swap(deps);
      if (cur.chain_dep >= 0) cur.chain_dep = remap[cur.chain_dep];
      remap[g] = (int)kept.size();
      kept.push_back(std::move(cur));
    }
    out->swap(kept);
    if (how == READ_AND_STORE && out->size() == 1) {   // a short message: the kernel without tables
      StoreAllArgs a;
      int grid = 0, threads = 0;
      const void* fn = store_all_entry(R, P.dtype, (int)c->sum_ctas, call.count, &a, &grid, &threads);
      if (fn) {
        a.phase = (unsigned)((uintptr_t)call.send[0] & 15);
        for (int r = 0; r < R; r++) {
          a.x[r] = call.send[r];
          a.y[r] = call.recv[r];
        }
        out->front().ready.push_back(make_launch(a, fn, grid, threads, 2.0 * R * (double)call.count * (double)P.elem, 0));
      }
    }
    if (c->path == HOCCL_PATH_CE && c->ce_small_bytes > 0) trim_driver_copies(out);
  }
  // SM path: the stages of an all-to-all are independent (disjoint blocks, no dependencies), so their moves go into as few
  // batched launches as the segment table allows instead of one launch per stage
  if (c->path == HOCCL_PATH_SM && P.kind == PLAN_ALLTOALL && out->size() > 1) {
    bool independent = true;
    for (const RGroup& g : *out) independent = independent && g.deps.empty() && g.kind == OP_MOVE;
    if (independent) {
      RGroup all = (*out)[0];
      for (size_t g = 1; g < out->size(); g++) all.segs.insert(all.segs.end(), (*out)[g].segs.begin(), (*out)[g].segs.end());
      out->assign(1, all);
    }
  }
  // SM path, direct all-gather: its stages (the trailing MOVE groups of a piece, nothing depends on them) wait for the same
  // thing, so consecutive ones with equal dependencies become one group = one batched launch (or one phase of the ring kernel).
  // Host-bounce path: the same merge lets the moves of a group that read the same bytes share ONE outbound copy into the
  // host staging (see share_host_legs): a chunk crosses PCIe once outbound and R-1 times inbound instead of R-1 times each way.
  if ((c->path == HOCCL_PATH_SM || c->path == HOCCL_PATH_CE_HOST) && P.ag_direct && P.kind != PLAN_ALLTOALL) {
    std::vector<char> has_user(out->size(), 0);
    for (const RGroup& g : *out) {
      for (int d : g.deps) has_user[d] = 1;
      if (g.chain_dep >= 0) has_user[g.chain_dep] = 1;
    }
    std::vector<RGroup> merged;
    std::vector<int> remap(out->size(), -1);
    for (size_t g = 0; g < out->size(); g++) {
      RGroup& cur = (*out)[g];
      for (int& d : cur.deps) d = remap[d];
      if (cur.chain_dep >= 0) cur.chain_dep = remap[cur.chain_dep];
      const bool tail_move = cur.kind == OP_MOVE && !has_user[g] && cur.phase != PHASE_RS;
      if (tail_move && !merged.empty() && g > 0 && remap[g - 1] == (int)merged.size() - 1 && merged.back().kind == OP_MOVE &&
          !has_user[g - 1] && merged.back().phase != PHASE_RS && merged.back().piece == cur.piece && merged.back().deps == cur.deps) {
        merged.back().segs.insert(merged.back().segs.end(), cur.segs.begin(), cur.segs.end());
        remap[g] = (int)merged.size() - 1;
      } else {
        merged.push_back(cur);
        remap[g] = (int)merged.size() - 1;
      }
    }
    out->swap(merged);
    if (c->path == HOCCL_PATH_CE_HOST) share_host_legs(out, host_need);
  }
}

namespace {
// Moves of a group with the same source, the same length and the same 16-byte phase of the destination.
struct MoveClass {
  const char* src;
  size_t bytes;
  std::vector<void*> dsts;
};
}  // namespace

// *repeats: whether some source goes to more than one destination of a class.
static std::vector<MoveClass> move_classes(const RGroup& g, bool* repeats) {
  std::vector<MoveClass> classes;
  std::map<std::tuple<const char*, size_t, unsigned>, size_t> index;
  *repeats = false;
  for (const Seg& s : g.segs) {
    auto key = std::make_tuple((const char*)s.src, (size_t)s.bytes, (unsigned)((uintptr_t)s.dst & 15));
    auto it = index.find(key);
    if (it == index.end()) {
      index.emplace(key, classes.size());
      classes.push_back(MoveClass{s.src, s.bytes, {s.dst}});
    } else {
      classes[it->second].dsts.push_back(s.dst);
      *repeats = true;
    }
  }
  return classes;
}

bool build_fan_batches(const RGroup& g, std::vector<FanBatch>* out, std::vector<double>* bytes_out, std::vector<long>* moves_out) {
  out->clear();
  bytes_out->clear();
  moves_out->clear();
  if (g.kind != OP_MOVE) return false;
  bool repeats = false;
  const std::vector<MoveClass> classes = move_classes(g, &repeats);
  if (!repeats) return false;
  FanBatch cur;
  cur.nseg = 0;
  cur.ndst_total = 0;
  double cur_bytes = 0;
  long cur_moves = 0;
  auto flush = [&]() {
    if (cur.nseg == 0) return;
    out->push_back(cur);
    bytes_out->push_back(cur_bytes);
    moves_out->push_back(cur_moves);
    cur.nseg = 0;
    cur.ndst_total = 0;
    cur_bytes = 0;
    cur_moves = 0;
  };
  for (const MoveClass& cl : classes) {
    size_t done = 0;
    while (done < cl.dsts.size()) {   // a class with more destinations than a batch holds is cut
      if (cur.nseg == kMaxSegs || cur.ndst_total == kMaxFanDsts) flush();
      const size_t n = std::min<size_t>(cl.dsts.size() - done, (size_t)(kMaxFanDsts - cur.ndst_total));
      cur.seg[cur.nseg++] = FanSeg{cl.src, (unsigned long long)cl.bytes, cur.ndst_total, (int)n};
      for (size_t i = 0; i < n; i++) cur.dst[cur.ndst_total++] = cl.dsts[done + i];
      cur_bytes += (double)cl.bytes * (1.0 + (double)n);
      cur_moves += (long)n;
      done += n;
    }
  }
  flush();
  return true;
}

// Fills *b with chain segments of g from `first` on; returns how many fitted.
static size_t fill_chain_batch(const RGroup& g, size_t first, int dtype, size_t elem, ChainBatch* b) {
  b->nseg = 0;
  b->nptr = 0;
  b->dtype = dtype;
  size_t i = first;
  for (; i < g.segs.size(); i++) {
    const Seg& s = g.segs[i];
    const void* ops[kMaxRanks];
    int nops = 0;
    if (!s.ops.empty()) {
      for (const void* p : s.ops) ops[nops++] = p;
    } else {
      for (int j = 0; j < s.nsrc; j++) ops[nops++] = s.src + (size_t)j * s.src_stride;
      ops[nops++] = s.local;
    }
    void* one = s.dst;
    void* const* dsts = s.dsts.empty() ? &one : s.dsts.data();
    const int ndst = s.dsts.empty() ? 1 : (int)s.dsts.size();
    if (!add_chain_seg(b, ops, nops, dsts, ndst, (unsigned long long)(s.bytes / elem))) break;
  }
  return i - first;
}

std::vector<MoveBatch> pack_moves(const RGroup& g, int ctas) {
  std::vector<MoveBatch> out;
  MoveBatch b;
  b.nseg = b.ndst_total = 0;
  auto flush = [&]() {
    if (b.nseg == 0) return;
    prepare_move_batch(&b, ctas);
    out.push_back(b);
    b.nseg = b.ndst_total = 0;
  };
  bool repeats = false;
  for (const MoveClass& cl : move_classes(g, &repeats))
    for (size_t done = 0; done < cl.dsts.size();) {
      const size_t n = std::min<size_t>(cl.dsts.size() - done, (size_t)kMaxRanks);
      for (size_t at = 0; at < cl.bytes; at += kMaxMoveSegBytes) {
        const size_t len = std::min<size_t>(kMaxMoveSegBytes, cl.bytes - at);
        std::vector<void*> dsts(cl.dsts.begin() + done, cl.dsts.begin() + done + n);
        for (void*& d : dsts) d = (char*)d + at;
        if (!add_move_seg(&b, cl.src + at, dsts.data(), (int)n, len)) {
          flush();
          add_move_seg(&b, cl.src + at, dsts.data(), (int)n, len);
        }
      }
      done += n;
    }
  flush();
  return out;
}

static std::vector<KernelLaunch> move_launches(const hoccl_comm* c, const RGroup& g) {
  std::vector<KernelLaunch> out;
  const int ctas = (int)(g.ctas ? g.ctas : c->copy_ctas);
  for (const MoveBatch& b : pack_moves(g, ctas)) {
    double bytes = 0;
    for (int k = 0; k < b.nseg; k++) bytes += (1.0 + (double)b.seg[k].ndst) * (double)b.seg[k].bytes;
    int threads = 0, grid = 0;
    MoveBatchSmall small;
    const bool fits = shrink_move_batch(b, &small);
    const void* fn = move_kernel_entry(b, ctas, fits, &threads, &grid);
    out.push_back(fits ? make_launch(small, fn, grid, threads, bytes, b.ndst_total) : make_launch(b, fn, grid, threads, bytes, b.ndst_total));
  }
  return out;
}

std::vector<KernelLaunch> kernel_launches(const hoccl_comm* c, const Plan& P, const RGroup& g) {
  if (!g.ready.empty()) return g.ready;
  std::vector<KernelLaunch> out;
  int threads = 0;
  if (g.kind == OP_CHAIN) {
    for (size_t first = 0; first < g.segs.size();) {
      ChainBatch b;
      const size_t n = fill_chain_batch(g, first, P.dtype, P.elem, &b);
      b.walk = g.beside ? 1 : 0;
      prepare_chain_batch(&b, (int)c->sum_ctas);
      double bytes = 0;
      for (int i = 0; i < b.nseg; i++) bytes += (double)(b.seg[i].nops + b.seg[i].ndst) * (double)b.seg[i].n * (double)P.elem;
      int grid = 0;
      const void* fn = chain_kernel_entry(b, (int)c->sum_ctas, &threads, &grid);
      out.push_back(make_launch(b, fn, grid, threads, bytes, 0));
      first += n;
    }
    return out;
  }
  if (g.kind == OP_SUM) {
    for (size_t first = 0; first < g.segs.size(); first += kMaxSegs) {
      SumBatch b;
      b.nseg = (int)std::min<size_t>(kMaxSegs, g.segs.size() - first);
      b.dtype = P.dtype;
      double bytes = 0;
      for (int i = 0; i < b.nseg; i++) {
        const Seg& s = g.segs[first + i];
        b.seg[i] = SumSeg{s.src, s.local, s.dst, (unsigned long long)(s.bytes / P.elem)};
        bytes += 3.0 * (double)s.bytes;
      }
      prepare_sum_batch(&b, (int)c->sum_ctas);
      const void* fn = sum_kernel_entry(P.dtype, (int)c->sum_ctas, &threads);
      out.push_back(make_launch(b, fn, c->sum_ctas, threads, bytes, 0));
    }
    return out;
  }
  return move_launches(c, g);
}

cudaError_t launch_kernel(const KernelLaunch& k, cudaStream_t stream) {
  return launch_in_order(k.fn, k.grid, k.threads, const_cast<char*>(k.args.data()), stream, k.priority);
}

hoccl_result_t launch_sum_kernel(hoccl_comm* c, const KernelLaunch& k, cudaStream_t s) {
  std::pair<cudaEvent_t, cudaEvent_t> pe{nullptr, nullptr};
  if (c->profile) {
    if (c->prof_pool.empty()) {
      cudaEvent_t a, z;
      CU_TRY(c, cudaEventCreate(&a));
      CU_TRY(c, cudaEventCreate(&z));
      pe = {a, z};
    } else {
      pe = c->prof_pool.back();
      c->prof_pool.pop_back();
    }
    CU_TRY(c, cudaEventRecord(pe.first, s));
  }
  CU_TRY(c, launch_kernel(k, s));
  if (c->profile) {
    CU_TRY(c, cudaEventRecord(pe.second, s));
    c->prof_open.push_back({pe, k.bytes});
  }
  return HOCCL_OK;
}

// ------------------------------------------------------------------ stream executor -------------
hoccl_result_t run_streams(hoccl_comm* c, const Plan& P, const std::vector<RGroup>& groups, cudaStream_t user, Tally* tally) {
  const int lanes = (int)std::max<long>(1, std::min<long>(c->lanes, kMaxLanes));
  c->ev_next = 0;
  std::vector<cudaStream_t> where(groups.size(), nullptr);
  std::vector<cudaEvent_t> done(groups.size(), nullptr);
  std::vector<char> lane_used(lanes, 0);
  bool sum_used = false;
  cudaEvent_t fork = next_event(c);
  if (!fork) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
  CU_TRY(c, cudaEventRecord(fork, user));
  auto touch = [&](cudaStream_t s, char* used) -> cudaError_t {
    if (*used) return cudaSuccess;
    *used = 1;
    return cudaStreamWaitEvent(s, fork, 0);
  };
  int move_rr = 0;
  for (size_t g = 0; g < groups.size(); g++) {
    const RGroup& rg = groups[g];
    cudaStream_t s;
    if (rg.kind != OP_MOVE) {
      s = c->sum_stream;
      char u = sum_used ? 1 : 0;
      CU_TRY(c, touch(s, &u));
      sum_used = true;
    } else {
      int l = c->path == HOCCL_PATH_SM ? 0 : move_rr++ % lanes;   // SM copies share one lane: global CTA budget
      s = c->lane[l];
      CU_TRY(c, touch(s, &lane_used[l]));
    }
    where[g] = s;
    for (int d : rg.deps)
      if (where[d] != s) CU_TRY(c, cudaStreamWaitEvent(s, done[d], 0));
    // chain_dep needs no event here: every SUM is on the one sum stream
    if (rg.kind != OP_MOVE) {
      for (const KernelLaunch& k : kernel_launches(c, P, rg)) {
        const hoccl_result_t lrc = launch_sum_kernel(c, k, s);
        if (lrc != HOCCL_OK) return lrc;
        tally->sum_launches++;
      }
    } else if (c->path == HOCCL_PATH_CE && !rg.edges) {
      for (const Seg& sg : rg.segs) {
        CU_TRY(c, cudaMemcpyAsync(sg.dst, sg.src, sg.bytes, cudaMemcpyDeviceToDevice, s));
        tally->moves++;
      }
    } else if (c->path == HOCCL_PATH_CE_HOST) {
      // two copy-engine legs through pinned host memory: no SM takes part in the move
      for (const Seg& sg : rg.segs) {
        // a seg that shares another seg's outbound copy comes after it in the same group, hence later on this stream
        if (sg.host_first) CU_TRY(c, cudaMemcpyAsync(c->host_staging + sg.host_off, sg.src, sg.bytes, cudaMemcpyDeviceToHost, s));
        CU_TRY(c, cudaMemcpyAsync(sg.dst, c->host_staging + sg.host_off, sg.bytes, cudaMemcpyHostToDevice, s));
        tally->moves++;
      }
    } else {
      for (const KernelLaunch& k : kernel_launches(c, P, rg)) {
        CU_TRY(c, launch_kernel(k, s));
        if (!rg.edges) tally->moves += k.moves;
        tally->move_launches++;
      }
    }
    cudaEvent_t ev = next_event(c);
    if (!ev) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
    CU_TRY(c, cudaEventRecord(ev, s));
    done[g] = ev;
  }
  // join: the caller's stream waits for every internal stream that was used
  for (int l = 0; l < lanes; l++)
    if (lane_used[l]) {
      cudaEvent_t ev = next_event(c);
      if (!ev) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
      CU_TRY(c, cudaEventRecord(ev, c->lane[l]));
      CU_TRY(c, cudaStreamWaitEvent(user, ev, 0));
    }
  if (sum_used) {
    cudaEvent_t ev = next_event(c);
    if (!ev) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
    CU_TRY(c, cudaEventRecord(ev, c->sum_stream));
    CU_TRY(c, cudaStreamWaitEvent(user, ev, 0));
  }
  return HOCCL_OK;
}

std::vector<uint64_t> make_key(hoccl_comm* c, const Call& call) {
  std::vector<uint64_t> k;
  k.reserve(27 + 2 * c->R);
  k.push_back((uint64_t)call.kind);
  k.push_back((uint64_t)call.count);
  k.push_back((uint64_t)call.dtype);
  k.push_back((uint64_t)c->path);
  k.push_back((uint64_t)c->sum_ctas);
  k.push_back((uint64_t)c->copy_ctas);
  k.push_back((uint64_t)c->piece_bytes);
  k.push_back((uint64_t)c->piece_bytes_set);
  k.push_back((uint64_t)c->max_pieces);
  k.push_back((uint64_t)c->profile);
  k.push_back((uint64_t)c->ce_sub_bytes);
  k.push_back((uint64_t)(c->ce_small_bytes > 0));   // whether driver copies leave their ends to the copy kernel
  k.push_back((uint64_t)c->forward);
  k.push_back((uint64_t)c->ag_direct);
  k.push_back((uint64_t)c->order_kernels);
  k.push_back((uint64_t)c->rs_direct);
  k.push_back((uint64_t)c->ce_overlap);
  k.push_back((uint64_t)(c->fused && c->path == HOCCL_PATH_SM && !c->handshake));
  k.push_back((uint64_t)c->handshake);   // an entry of handshake mode has no launches of its own and its graph is on the device before the proxy meets it
  k.push_back((uint64_t)c->roles);
  k.push_back((uint64_t)c->piece_grade);
  k.push_back((uint64_t)c->roles_missing);
  k.push_back((uint64_t)(uintptr_t)c->scratch);
  k.push_back((uint64_t)c->scratch_bytes);
  k.push_back((uint64_t)(uintptr_t)c->host_staging);
  k.push_back((uint64_t)c->host_staging_bytes);
  for (int r = 0; r < c->R; r++) {
    k.push_back((uint64_t)(uintptr_t)call.send[r]);
    k.push_back((uint64_t)(uintptr_t)call.recv[r]);
  }
  k.push_back(call.h_send ? (uint64_t)c->host_pieces * 2 + (c->host_pieces_set ? 1 : 0) : 0);
  if (call.h_send)
    for (int r = 0; r < c->R; r++) {
      k.push_back((uint64_t)(uintptr_t)call.h_send[r]);
      k.push_back((uint64_t)(uintptr_t)call.h_recv[r]);
    }
  return k;
}

// reads back the profile events of finished work (the caller has synchronised)
void harvest_profile(hoccl_comm* c) {
  for (auto& rec : c->prof_open) {
    float ms = 0;
    if (cudaEventElapsedTime(&ms, rec.first.first, rec.first.second) == cudaSuccess) {
      c->prof_ms += ms;
      c->prof_bytes += rec.second;
      c->prof_n++;
    }
    c->prof_pool.push_back(rec.first);
  }
  c->prof_open.clear();
  // cached graphs keep their own events; a replay overwrites them, so only the latest replay is readable
  for (auto& e : c->cache) {
    if (!e.prof_pending) continue;
    e.prof_pending = false;
    for (size_t i = 0; i < e.prof_events.size(); i++) {
      float ms = 0;
      if (cudaEventElapsedTime(&ms, e.prof_events[i].first, e.prof_events[i].second) == cudaSuccess) {
        if (e.prof_bytes[i] < 0) {
          c->prof_copy_ms += ms;
          c->prof_copy_bytes -= e.prof_bytes[i];
          c->prof_copy_n++;
        } else {
          c->prof_ms += ms;
          c->prof_bytes += e.prof_bytes[i];
          c->prof_n++;
        }
      }
    }
  }
}

// The CPU proxy of the handshake mode is created on first use.
hoccl_result_t ensure_proxy(hoccl_comm* c) {
  if (c->proxy) {
    c->proxy->set_watchdog_ms(c->watchdog_ms);
    return HOCCL_OK;
  }
  Proxy* p = new Proxy(c->device, c->watchdog_ms);
  cudaError_t e = p->init();
  if (e != cudaSuccess) {
    delete p;
    return cuda_fail(c, e, "proxy init (stream memory operations)");
  }
  c->proxy = p;
  return HOCCL_OK;
}

// What this thread last put on a stream: the stream, when the call returned, and when by estimate the device is through with it.  Only a
// hint which of two equal ways a call takes; a stream that died and whose handle came back misleads it for one call.
struct Burst {
  cudaStream_t stream = nullptr;
  double returned = 0, busy_until = 0;
};
static thread_local Burst t_burst;
constexpr double kBurstGapUs = 5;   // a Python caller's loop leaves about 2 us between calls; waiting for the device in between takes 7 or more

// Replays a cached entry into the caller's stream (directly, or through the CPU proxy in handshake mode: an entry of that mode has no launches).
hoccl_result_t launch_entry(hoccl_comm* c, GraphEntry* hit, cudaStream_t user, double t0) {
  hit->last_use = ++c->use_counter;
  // A short chain of kernels goes out as a graph or as launches (see launch_in_order).  A graph costs the host less (0.9 us against 1.6 to 2.4
  // per launch) and reaches an idle device 1.6 us earlier; behind other work launches start up to 2 us earlier.  Whether there is
  // work in front cannot be asked for less (cudaStreamQuery 0.3 us if there is, 1.6 if not).  So: launches if the call follows the one before
  // it at once, on the same stream, and takes the device longer than the host, or is one launch of 3.5 us or more and the calls before it did (a shorter
  // one takes two steps of 2.048 us as a graph, 4.1, and what the host needs as a launch, up to 5.6: all-reduce of 4 ranks, 147 KB, est. 3.1, 4.1 / 4.7-5.6,
  // 200 KB, est. 3.7, 6.2 / 3.6; all-gather of 4 ranks est. 2.7 3.9 / 4.7, est. 3.6 4.1 / 3.65); otherwise the graph.  Us of a call
  // in a burst as graphs / as launches, R = 8 bf16: all-reduce 4 KiB per rank 3.6 / 4.9, 96 KiB 4.10 / 4.52, 128 KiB 6.15 / 4.55, 384 KiB
  // 10.25 / 9.1, 1 MiB with 8 + 40 CTAs 17.0 / 14.35; 148 CTAs 512 KiB 4.10 / 4.85, 1 MiB 6.14 / 4.85; all-to-all 512 KiB 4.10 / 4.80, 1 MiB
  // 6.15 / 4.80; two launches, R = 16, all-to-all 512 KiB 8.19 / 8.56, 2 MiB 20.5 / 18.3.  The line: the estimate against 1.8 + 2.2 per launch.
  Burst& last = t_burst;
  const bool follows = last.stream == user && t0 - last.returned < kBurstGapUs;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;   // a capture is refused by the graph launch, in a burst or not
  const size_t n = hit->launches.size();
  const bool behind = n && follows && ((n == 1 && hit->est_us >= 3.5 && t0 < last.busy_until) || hit->est_us >= 1.8 + 2.2 * (double)n) &&
                      cudaStreamIsCapturing(user, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone;
  last.busy_until = (follows ? std::max(t0, last.busy_until) : t0) + hit->est_us;
  struct Returns {   // on every way out
    Burst& last;
    cudaStream_t s;
    double at;   // 0: not read yet (a reading of the clock is 1 % of a short call)
    ~Returns() {
      last.stream = s;
      last.returned = at != 0 ? at : now_us();
    }
  } returns{last, user, 0};
  if (!hit->ring_args.empty()) {
    if (hit->ring_large)
      CU_TRY(c, launch_ring(*reinterpret_cast<const RingArgsLarge*>(hit->ring_args.data()), hit->ring_grid, hit->ring_threads, user));
    else
      CU_TRY(c, launch_ring(*reinterpret_cast<const RingArgsSmall*>(hit->ring_args.data()), hit->ring_grid, hit->ring_threads, user));
    c->stats.n_pieces = hit->n_pieces;
    c->stats.n_moves = hit->n_moves;
    c->stats.n_move_launches = 1;
    c->stats.n_sum_launches = 0;
    c->stats.max_copy_ctas = hit->ring_grid;
    c->stats.max_sum_ctas = hit->ring_has_sum ? hit->ring_grid : 0;
    c->stats.host_launch_us = now_us() - t0;
    return HOCCL_OK;
  }
  if (hit->roles_fn) {
    hoccl_result_t rrc = launch_roles(c, hit, user);
    if (rrc != HOCCL_OK) return rrc;
    c->stats.n_pieces = hit->n_pieces;
    c->stats.n_moves = hit->n_moves;
    c->stats.n_move_launches = 1;
    c->stats.n_sum_launches = 0;
    c->stats.max_copy_ctas = hit->roles_grid - hit->roles_sum_ctas;
    c->stats.max_sum_ctas = hit->roles_sum_ctas;
    c->stats.host_launch_us = now_us() - t0;
    return HOCCL_OK;
  }
  if (!hit->part_exec.empty()) {
    // Copy route with overlap: the reduce-scatter's moves of every piece on one internal stream, the sums on the sum stream
    // (one at a time: the SM budget stays global), the all-gather's moves on a second internal stream; events carry the
    // per-piece dependencies between them.
    cudaStream_t rs = c->lane[0], sm = c->sum_stream, ag = c->lane[1];
    c->ev_next = 0;
    cudaEvent_t fork = next_event(c);
    if (!fork) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
    CU_TRY(c, cudaEventRecord(fork, user));
    CU_TRY(c, cudaStreamWaitEvent(rs, fork, 0));
    CU_TRY(c, cudaStreamWaitEvent(sm, fork, 0));
    CU_TRY(c, cudaStreamWaitEvent(ag, fork, 0));
    const size_t np = hit->part_exec.size() / 3;
    for (size_t p = 0; p < np; p++) {
      cudaGraphExec_t g_rs = hit->part_exec[3 * p], g_sum = hit->part_exec[3 * p + 1], g_ag = hit->part_exec[3 * p + 2];
      if (g_rs) {
        CU_TRY(c, cudaGraphLaunch(g_rs, rs));
        cudaEvent_t moved = next_event(c);
        if (!moved) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
        CU_TRY(c, cudaEventRecord(moved, rs));
        CU_TRY(c, cudaStreamWaitEvent(sm, moved, 0));
      }
      if (g_sum) CU_TRY(c, cudaGraphLaunch(g_sum, sm));
      if (!hit->part_sums.empty())
        for (const KernelLaunch& k : hit->part_sums[p]) CU_TRY(c, launch_kernel(k, sm));
      if (g_ag) {
        cudaEvent_t summed = next_event(c);
        if (!summed) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
        CU_TRY(c, cudaEventRecord(summed, sm));
        CU_TRY(c, cudaStreamWaitEvent(ag, summed, 0));
        CU_TRY(c, cudaGraphLaunch(g_ag, ag));
      }
    }
    for (cudaStream_t s : {rs, sm, ag}) {
      cudaEvent_t done = next_event(c);
      if (!done) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
      CU_TRY(c, cudaEventRecord(done, s));
      CU_TRY(c, cudaStreamWaitEvent(user, done, 0));
    }
  } else if (!hit->piece_exec.empty()) {
    // Pipelined host all-reduce: the inbound copies run on one internal stream, the outbound copies on another, and the
    // caller's stream runs the ring piece by piece as each piece arrives; PCIe carries both directions at once.
    cudaStream_t in = c->lane[0], out = c->lane[1];
    c->ev_next = 0;
    cudaEvent_t fork = next_event(c);
    if (!fork) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
    CU_TRY(c, cudaEventRecord(fork, user));
    CU_TRY(c, cudaStreamWaitEvent(in, fork, 0));
    CU_TRY(c, cudaStreamWaitEvent(out, fork, 0));
    const size_t np = hit->piece_exec.size();
    std::vector<cudaEvent_t> arrived(np, nullptr);
    for (size_t p = 0; p < np; p++) {
      for (const HostCopy& hc : hit->h2d[p]) CU_TRY(c, enqueue_host_copy(hc, true, in));
      arrived[p] = next_event(c);
      if (!arrived[p]) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
      CU_TRY(c, cudaEventRecord(arrived[p], in));
    }
    for (size_t p = 0; p < np; p++) {
      CU_TRY(c, cudaStreamWaitEvent(user, arrived[p], 0));
      if (hit->piece_exec[p]) CU_TRY(c, cudaGraphLaunch(hit->piece_exec[p], user));
      cudaEvent_t reduced = next_event(c);
      if (!reduced) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
      CU_TRY(c, cudaEventRecord(reduced, user));
      CU_TRY(c, cudaStreamWaitEvent(out, reduced, 0));
      for (const HostCopy& hc : hit->d2h[p]) CU_TRY(c, enqueue_host_copy(hc, false, out));
    }
    cudaEvent_t done = next_event(c);
    if (!done) return cuda_fail(c, cudaErrorMemoryAllocation, "event pool");
    CU_TRY(c, cudaEventRecord(done, out));
    CU_TRY(c, cudaStreamWaitEvent(user, done, 0));
  } else if (behind) {
    for (const KernelLaunch& k : hit->launches) CU_TRY(c, launch_kernel(k, user));
  } else if (c->handshake) {
    // paper Sec. 3.2: the stream hands itself to the CPU proxy, which runs the schedule and hands it back
    ProxyTask t;
    t.kind = ProxyTask::GRAPH;
    t.exec = hit->exec;
    CU_TRY(c, c->proxy->submit(user, t));
  } else {
    CU_TRY(c, cudaGraphLaunch(hit->exec, user));
  }
  hit->prof_pending = !hit->prof_events.empty();
  c->stats.n_pieces = hit->n_pieces;
  c->stats.n_moves = hit->n_moves;
  c->stats.n_move_launches = hit->n_move_launches;
  c->stats.n_sum_launches = hit->n_sum_launches;
  c->stats.n_order_launches = hit->n_order_launches;
  c->stats.max_sum_ctas = hit->n_sum_launches ? c->sum_ctas : 0;
  c->stats.max_copy_ctas = hit->n_move_launches ? c->copy_ctas : 0;
  returns.at = now_us();
  c->stats.host_launch_us = returns.at - t0;
  return HOCCL_OK;
}

static OptionsIn options_of(hoccl_comm* c, int kind, size_t count, int dtype, bool host_call) {
  return OptionsIn{kind, c->R, count, dtype, (int)c->path, c->onepass, c->forward, c->fused, c->rs_direct, c->ag_direct,
                   c->handshake, c->use_graph, c->ce_small_bytes, c->ce_small_ctas, c->copy_ctas, c->scratch ? c->scratch_bytes : 0,
                   host_call ? 1 : 0, c->roles};
}

hoccl_result_t check_options(hoccl_comm* c, int kind, size_t count, int dtype) {
  OptionsOut o;
  return resolve_options(options_of(c, kind, count, dtype, false), &o);
}

// Whether an all-gather or all-to-all is better not left to driver copies.  Such a call runs on the move kernel at any size, like a
// small one.
//   * Some block is a copy the driver does badly (see kDriverLine): 64 MiB per rank over 8 ranks, blocks 16 bytes short of whole: all-gather
//     372 us in driver copies, 96 on the kernel, all-to-all 384 and 164; two bytes out of phase 818 and 99, 838 and 171.
//   * The blocks of an all-to-all are short, or few: 64 MiB per rank over 2 ranks 46.7 and 41.0 us, over 4 88 and 81.5.  Long whole blocks between more
//     ranks stay with the driver, 5 % behind at 64 MiB (8 ranks 172 and 164), 1 % at 256 MiB (655 and 650).
//   * An all-gather: the kernel reads a block once, driver copies once per destination (64 MiB per rank over 2 ranks 45 and 31 us, over 8 150 and
//     96; 256 MiB over 8 572 and 345).  Both take the whole GPU.
//     Beside a loop of 8192^3 bf16 GEMMs a call of 25 MiB per rank over 8 ranks costs the GEMMs (median and quartiles) and takes meanwhile: all-gather
//     25 us (5 to 37) and 0.13 ms, in driver copies 22 (4 to 37) and 0.24 ms; all-to-all 14 (-10 to 40) and 0.33 ms, 11 (-18 to 31) and 0.28 ms.
// With "ce_small_ctas" below 128 only where that many CTAs keep up with the driver (kernel_ahead_from); long whole blocks of an all-to-all then stay
// with it between any number of ranks (64 MiB over 2 ranks 45.7 us, on 64 CTAs 48.5, 96 46.4; over 4 88, 93, 91).
static bool blocks_bad_for_driver(const hoccl_comm* c, const Call& call) {
  const size_t block = call.count * dtype_size(call.dtype);
  const bool wide = c->ce_small_ctas >= kWideMoves, few = block < kDriverShort || call.kind == PLAN_ALLGATHER;
  if (wide && (few || c->R <= 4)) return true;
  bool bad = false;
  double ahead = 0;   // the mean of 1 / kernel_ahead_from
  for (int u = 0; u < c->R; u++)
    for (int v = 0; v < c->R; v++) {
      const char* src = (const char*)call.send[u] + (call.kind == PLAN_ALLTOALL ? (size_t)v * block : 0);
      const char* dst = (const char*)call.recv[v] + (size_t)u * block;
      bad = bad || bad_for_driver(src, dst, block);
      if (wide && bad) return true;
      ahead += 1 / kernel_ahead_from(src, dst, block) / ((double)c->R * c->R);
    }
  return !wide && (few || bad) && (double)c->ce_small_ctas * ahead >= 1;
}

// An all-reduce whose sums read the contributions in place and whose ring chunks the driver copies badly (not whole pages on 128-byte lines), or
// are short copies: its all-gather runs on the move kernel too, which reads a chunk once for all ranks.  Us in driver copies with their ends on the
// kernel / on the kernel alone, bf16: R = 8, 16 MiB per rank 149.5 / 137.5, 64 MiB 554 / 527; R = 3, 32 MiB 174 / 155; R = 5, 32 MiB 221 / 203; R = 6, 64 MiB
// 456 / 445; R = 16, 19 MiB 352 / 290, 64 MiB 1072 / 887.  A loop of 8192^3 GEMMs loses less to it as well (8 ranks, 64 MiB 97 us per
// call, in driver copies 175).  Only with "ce_small_ctas" >= 128: on fewer it is even at best, R = 8 64 MiB driver 521 us, 8 CTAs 1027, 16 624, 40 515, 64 527;
// R = 3 32 MiB 157, 216, 172, 165, 165 (148: 145).  Whole chunks stay with the driver, whose copies run beside the next piece's sum: 8 ranks 40 MiB 335 us,
// 320 on the kernel.  So do ragged ones of 1 to 1.17 MiB, 80 MB for all ranks, though the kernel is ahead of them too (8 ranks of 8.5 MB 85 / 72, of
// 9.6 MB 92 / 80): they keep the form with trimmed copies, whose layout and signature are checked at these sizes.
static bool chunks_bad_for_driver(const hoccl_comm* c, const Call& call) {
  const size_t S = call.count * dtype_size(call.dtype), chunk = (call.count + c->R - 1) / c->R * dtype_size(call.dtype);
  if (chunk >= kDriverWhole && chunk < ((size_t)1200 << 10) && (size_t)c->R * S < 80000000) return false;
  bool bad = chunk < kDriverWhole || chunk % kDriverPage || S % kDriverPage;
  for (int v = 0; v < c->R; v++) bad = bad || (uintptr_t)call.recv[v] % kDriverLine;
  return bad;
}

// How the communicator's settings combine for this call (options.h); a contradictory combination is refused here.
static hoccl_result_t call_options(hoccl_comm* c, const Call& call, OptionsOut* opt) {
  OptionsIn oin = options_of(c, call.kind, call.count, call.dtype, call.h_send != nullptr);
  const bool may_switch = c->path == HOCCL_PATH_CE && c->ce_small_bytes > 0;
  if (may_switch && (call.kind == PLAN_ALLGATHER || call.kind == PLAN_ALLTOALL) && blocks_bad_for_driver(c, call)) oin.ce_small_bytes = LONG_MAX;
  const hoccl_result_t rc = resolve_options(oin, opt);
  if (rc == HOCCL_OK && may_switch && call.kind == PLAN_ALLREDUCE && opt->path == HOCCL_PATH_CE && opt->executor == EXEC_GRAPH && c->ag_direct == 2 &&
      c->ce_overlap < 0 && !c->piece_bytes_set && c->sum_ctas < 64 && c->ce_small_ctas >= kWideMoves && !call.h_send && chunks_bad_for_driver(c, call) &&
      contributions(c, call, *opt, call.count * dtype_size(call.dtype)) == READ_IN_PLACE) {
    oin.ce_small_bytes = LONG_MAX;
    return resolve_options(oin, opt);
  }
  return rc;
}

// CTAs of an all-gather that runs beside a SUM under a CTA budget: stores at 2.4 TB/s, which the sum does not feel (beside 64 it loses
// 2 %; 24 do not finish in time).  25 MiB per rank over 8 ranks in three pieces 206.8 us with 24, 207.0 with 40, 208.7 with 64.
constexpr long kBesideSums = 40;

// A step of the ring, by bytes of all ranks, whose whole-GPU moves are one CTA per SM that walks its tiles: what it reads the step before has just
// written to L2, so there is nothing for a CTA per tile to hide, only more of them to start.  Us, bf16, a CTA per tile / the walk: all-gather 8 ranks 2 MiB 20.4 /
// 18.4, 12 MiB 37.0 / 35.7, 25 MiB 59.4 / 59.3, 32 MiB 71.3 / 76.9, 64 MiB 136 / 146, 16 ranks 0.8 MiB 33.6 / 34.6, 12 MiB 70.4 / 67.5, 25 MiB 110.7 / 107.9, 32
// MiB 133 / 139; all-reduce 16 ranks 2 MiB 112.7 / 107.5, 25 MiB 351 / 342, 8 ranks 0.5 MiB 44.0 / 45.1, 25 MiB 167.5 / 164.0.
constexpr size_t kRingWalkFrom = 1280 << 10, kRingWalkTo = (size_t)28 << 20;

// Pure host work, nothing is enqueued.  The communicator shows the call's route (RouteGuard).
static hoccl_result_t lay_out(hoccl_comm* c, const Call& call, const OptionsOut& opt, Contributions how, Layout* out) {
  const bool fused = opt.executor == EXEC_ONE_KERNEL, roles = opt.executor == EXEC_ROLES;
  Plan& P = out->plan;
  unsigned char align[kMaxRanks];
  for (int r = 0; r < c->R; r++) align[r] = (unsigned char)((uintptr_t)call.send[r] & 15);
  const int plan_kind = opt.plan_kind;
  // Piece size: the caller's if set.  Otherwise: on the SM path under CTA budgets a reduction is cut into at least two
  // pieces (the copy kernel of one piece then overlaps the sum kernel of the other: measured 1.6x on a 3 MiB chunk with
  // 8 + 8 CTAs) of at most 4 MiB.  That does not pay with driver copies (they take the whole GPU and never overlap a sum:
  // every extra copy only adds its start-up) nor with whole-GPU grids (two kernels then share the same SMs), so the
  // copy route and the SM path with 128 CTAs or more for both kernels keep whole chunks up to 256 MiB (measured, R = 8,
  // bf16, 64 MiB to 1 GiB per rank: 7-15 % faster than 4 MiB pieces on the copy route with 8-CTA sums, 19-33 % with
  // 148-CTA sums, 3-14 % on the whole-GPU SM path).
  size_t piece_bytes = (size_t)c->piece_bytes;
  int max_pieces = (int)c->max_pieces;
  const bool reduction = call.kind == PLAN_ALLREDUCE || call.kind == PLAN_REDUCE_SCATTER;
  const size_t ring_chunk = (call.kind == PLAN_ALLREDUCE ? (call.count + c->R - 1) / c->R : call.count) * dtype_size(call.dtype);
  // the staged form of the direct schedule: 5 pieces at 25 MiB per rank (8 ranks 5.23 ms; 8 pieces 5.27), 4 at 16 MiB (3.58; 3.81)
  const size_t host_np = call.h_send && (opt.plan_kind & PLAN_FLAG_RS_DIRECT) ? host_pieces(c, call.count * dtype_size(call.dtype), 1e6) : (size_t)c->host_pieces;
  const bool sum_only = how == READ_AND_STORE || (how == READ_IN_PLACE && call.kind == PLAN_REDUCE_SCATTER);   // no moves at all
  // Copy route with overlap ("ce_overlap"): the direct schedule cut into pieces whose three parts run on three internal
  // streams (see launch_entry).  Automatic (-1): 2 pieces from 2 MiB per ring chunk, from 4 MiB on pieces of about 4 MiB, at
  // least 4 and at most 32 of them; below that the ~30 us of host time per call and the extra copies cost more than the overlap
  // gives (measured on B200, R = 8, bf16, 8-CTA sums: 25 MiB per rank 0.290 -> 0.280 ms with 2 pieces; 40 MiB 0.468 -> 0.421 with
  // 4; 256 MiB 2.97 -> 2.44 with 8; 1 GiB 11.8 -> 9.72 with 8, 9.52 with 32).
  long overlap_pieces = c->ce_overlap;
  if (overlap_pieces < 0) {
    // (whole-GPU sums are short: beside them more than 8 pieces only add copies; 1 GiB per rank 6.34 ms with 8, 6.80 with 32)
    const size_t most = c->sum_ctas >= 64 ? 8 : 32;
    overlap_pieces = ring_chunk >= ((size_t)4 << 20) ? (long)std::min<size_t>(most, std::max<size_t>(4, ring_chunk >> 22))
                                                     : ring_chunk >= ((size_t)2 << 20) ? 2 : 0;
    // With the contributions read in place only the all-gather's copies are left to hide behind the sums.  np equal pieces leave
    // 1 / np of them exposed and cost 5.4 us each (drain and refill of the sums, launches, events), so np is the root of the copies' time over 5.4 us,
    // in pieces of 1.25 MiB or more.  Us in 1 / 2 / 3 / 4 / 6 / 8 / 12 pieces, bf16, 8-CTA sums (in brackets what the rule takes): R = 2, 64 MiB 242 / 241 /
    // 243 / 244 / 254 / 262 / 273 (2), 256 MiB 958 / 937 / 922 / 920 / 927 / 932 / 941 (4); R = 3, 64 MiB 304 / 295 / 292 / 297 / 308 (2); R = 4, 32 MiB
    // 175 / 176 / 179 / 180 / 187 (2), 64 MiB 357 / 338 / 334 / 335 / 340 / 353 / 356 (3), 256 MiB 1410 / 1345 / 1307 / 1293 / 1283 / 1283 / 1282 (6);
    // R = 6, 64 MiB 488 / 451 / 445 / 444 / 461 / 465 (4); R = 8, 40 MiB - / 337 / 332 / 335 (4), 64 MiB 602 / 544 / 526 / 523 / 535 / 558 (5), 256 MiB 2370 /
    // 2220 / 2150 / 2105 / 2060 / 2047 / 2015 (10); R = 16, 64 MiB 1127 / 983 / 941 / 933 / 1032 (3).  Chunks above 8 MiB are cut in two at least,
    // which costs two ranks up to 5 % (32 MiB 123 whole, 128 in two).  (148-CTA sums: 16 MiB 0.056 ms whole, 0.076 in 2, 64 MiB 0.244 / 0.225, 0.262 in 6.)
    if (how == READ_IN_PLACE) {
      if (c->sum_ctas >= 64) {
        overlap_pieces = (long)std::min<size_t>(8, ring_chunk >> 22);
      } else {
        const double copies_us = 2.0 * (c->R - 1) * (double)ring_chunk * c->R / 6.2e6;
        const size_t np = std::min((size_t)std::sqrt(copies_us / 5.4), ring_chunk / ((size_t)1280 << 10));
        overlap_pieces = (long)std::min<size_t>(32, std::max<size_t>(ring_chunk > ((size_t)8 << 20) ? 2 : 0, np));
      }
    }
  }
  const bool overlap = overlap_pieces > 1 && c->path == HOCCL_PATH_CE && opt.executor == EXEC_GRAPH && !call.h_send &&
                       (plan_kind & PLAN_FLAG_RS_DIRECT) && c->R > 1 && !c->piece_bytes_set && !sum_only;
  // Sums under a CTA budget with the all-gather on a whole-GPU grid of the move kernel: the pieces follow the rule above with 5 us per piece and
  // (R stores per vector read) the move kernel's R S bytes; the all-gathers of all pieces but the last run on kBesideSums CTAs.  Us
  // whole / in two / in three, bf16: R = 8, 10 MiB per rank 86.6 / 87.2 / 90.2 (1), 16 MiB 139.4 / 135.0 / 135.2 (2), 25 MiB 216.8 / 208.0 / 207.0 (2);
  // R = 4, 10 MiB 54.3 / 58.5 / 61.8 (1), 16 MiB 84.8 / 88.9 / 89.2 (1).
  const bool beside = how == READ_IN_PLACE && call.kind == PLAN_ALLREDUCE && c->path == HOCCL_PATH_SM && opt.executor == EXEC_GRAPH &&
                      (plan_kind & PLAN_FLAG_AG_DIRECT) && c->sum_ctas < 64 && c->copy_ctas >= 128 && !c->piece_bytes_set && !call.h_send;
  if (sum_only && !c->piece_bytes_set && !call.h_send) {   // nothing to overlap
    piece_bytes = (size_t)1 << 60;
    max_pieces = 1;
  } else if (beside) {
    max_pieces = (int)std::min<size_t>(32, std::max<size_t>(ring_chunk > ((size_t)8 << 20) ? 2 : 1, (size_t)std::sqrt((double)c->R * (double)call.send_bytes / 6e6 / 5.0)));
    piece_bytes = std::max<size_t>((size_t)64 << 10, ((ring_chunk + max_pieces - 1) / max_pieces + 1023) / 1024 * 1024);
  } else if (overlap) {
    max_pieces = (int)overlap_pieces;
    piece_bytes = std::max<size_t>((size_t)64 << 10, ((ring_chunk + max_pieces - 1) / max_pieces + 1023) / 1024 * 1024);
  } else if (!c->piece_bytes_set && c->path == HOCCL_PATH_SM && opt.executor == EXEC_GRAPH && !call.h_send && reduction &&
             (plan_kind & PLAN_FLAG_RS_DIRECT) && c->sum_ctas < 64 && c->copy_ctas < 128 && ring_chunk >= ((size_t)1 << 20)) {
    // SM path, direct schedule under CTA budgets: pieces of an eighth of a ring chunk, between 640 KiB and 2 MiB, issued as a
    // software pipeline (see build_graph): a piece's copies run beside another piece's chain sum (measured, 8-CTA sums and
    // 40 copy CTAs: 40 MiB per rank 0.46 ms with 2 pieces, 0.41 with 4, 0.38 with 8, 0.45 with 10; 25 MiB 0.30 / 0.26 / 0.245 /
    // 0.29 ms with 2 / 4 / 5 / 7 pieces; 256 MiB 2.92 / 2.57 / 2.40 / 2.32 ms with 2 / 4 / 8 / 16 pieces)
    // With the contributions read in place: a sixth of a chunk, between 1 and 3.25 MiB, from 4 MiB per chunk on (32 MiB per rank
    // 0.271 ms, 40 MiB 0.329, 64 MiB 0.508, 128 MiB 1.010, 256 MiB 1.978; an eighth: 0.282 / 0.336 / 0.519 / 1.016 / 1.986).
    if (how == READ_IN_PLACE && ring_chunk >= kGradeInPlace)
      piece_bytes = std::min<size_t>((size_t)3328 << 10, std::max<size_t>((size_t)1 << 20, (ring_chunk / 6 + 1023) / 1024 * 1024));
    else
      piece_bytes = std::min<size_t>((size_t)2 << 20, std::max<size_t>((size_t)640 << 10, (ring_chunk / 8 + 1023) / 1024 * 1024));
    max_pieces = 64;
  } else if (call.h_send) {   // pipelined host all-reduce: host_pieces pieces per chunk, whatever the chunk size
    const size_t q = (call.count + c->R - 1) / c->R;
    const size_t chunk = q * dtype_size(call.dtype);
    max_pieces = (int)host_np;
    piece_bytes = std::max<size_t>((size_t)64 << 10, ((chunk + max_pieces - 1) / max_pieces + 1023) / 1024 * 1024);
  } else if (roles) {
    // the piece rule of the graph form of the same schedule (above): both forms measured best with the same pieces
    if (!c->piece_bytes_set)
      piece_bytes = std::min<size_t>((size_t)2 << 20, std::max<size_t>((size_t)640 << 10, (ring_chunk / 8 + 1023) / 1024 * 1024));
    max_pieces = 64;   // (when the tables of that many pieces do not fit into shared memory the graph form runs the plan)
  } else if (fused) {   // one kernel walks the steps in order; whole chunks measured faster than pieces (fewer barriers and tails)
    piece_bytes = (size_t)1 << 60;
    max_pieces = 1;
  } else if (!c->piece_bytes_set && reduction &&
             (c->path == HOCCL_PATH_CE || (c->path == HOCCL_PATH_SM && std::min(c->sum_ctas, c->copy_ctas) >= 128))) {
    // "whole" stops at 256 MiB: several concurrent driver copies of 512 MiB each ran at half speed (R = 2, 1 GiB per rank)
    piece_bytes = (size_t)256 << 20;
  } else if (!c->piece_bytes_set && c->path == HOCCL_PATH_SM && std::max(c->sum_ctas, c->copy_ctas) < 64 &&
      (call.kind == PLAN_ALLREDUCE || call.kind == PLAN_REDUCE_SCATTER)) {
    const size_t q = call.kind == PLAN_ALLREDUCE ? (call.count + c->R - 1) / c->R : call.count;
    const size_t chunk = q * dtype_size(call.dtype);
    if (chunk >= ((size_t)1 << 20)) piece_bytes = std::min(piece_bytes, (chunk / 2 + 1023) / 1024 * 1024);
  }
  // graded pieces ("piece_grade"; -1 = automatic): measured on B200 (R = 8, bf16, 8-CTA sums) they gain 1-5 % from 64 MiB per rank
  // on (256 MiB: copy route 2.46 -> 2.44 ms, SM path 8 + 40 CTAs 2.32 -> 2.27, roles kernel 2.32 -> 2.25) and lose below (40 MiB
  // buckets: copy route 0.423 -> 0.444 ms, SM path 0.380 -> 0.431: the small outer pieces cost more in fixed time per piece than
  // their shorter fill saves), so automatic means: from 8 MiB per ring chunk, under a SUM budget (with whole-GPU sums the outer
  // pieces' moves are no longer what is exposed: 256 MiB per rank, copy route, 148-CTA sums 1.51 -> 1.53 ms)
  // (with the contributions read in place the SM path gains from 4 MiB per ring chunk on: 40 MiB per rank in 5 pieces 0.340 -> 0.329)
  const size_t grade_from = how == READ_IN_PLACE && c->path == HOCCL_PATH_SM ? kGradeInPlace : (size_t)8 << 20;
  const bool graded = reduction && !call.h_send && !fused && (plan_kind & PLAN_FLAG_RS_DIRECT) &&
                      (c->piece_grade == 1 || (c->piece_grade < 0 && !beside && ring_chunk >= grade_from && c->sum_ctas < 64));
  if (!build_plan(&P, plan_kind | (graded ? PLAN_FLAG_GRADED : 0), c->R, call.count, call.dtype, call.in_place, piece_bytes, max_pieces, align))
    return HOCCL_ERR_INVALID_ARG;
  if (P.slot_bytes) {
    size_t need = P.scratch_need();
    if (!c->scratch || c->scratch_bytes < need) return HOCCL_ERR_SCRATCH;
    // scratch must not overlap any rank buffer
    for (int r = 0; r < c->R; r++)
      if (ranges_overlap((const char*)c->scratch, need, (const char*)call.send[r], call.send_bytes) ||
          ranges_overlap((const char*)c->scratch, need, (const char*)call.recv[r], call.recv_bytes))
        return HOCCL_ERR_INVALID_ARG;
  }
  out->overlap = overlap && P.pieces > 1;   // with one piece there is nothing to overlap
  resolve(c, P, call, how, &out->groups, &out->host_need);
  // A sum that is launched starts on time behind another piece's (see launch_in_order).  That helps where the sums are the longer part and run back
  // to back, on few CTAs with the contributions read in place; sums of the whole GPU take the SMs that another piece's copies were waiting for,
  // and staged ones wait for copies of their own.  Us as launches / as graphs, bf16: 8 SUM CTAs R = 8 40 MiB 333 / 340, 256 MiB 2028 / 2046, R = 16
  // 256 MiB 3644 / 3672; 148 R = 2 128 MiB 142 / 121, R = 8 40 MiB in 4 pieces 159.9 / 157.9; staged, 148, R = 2 175 / 165, R = 4 64 MiB 186.5 / 183.2, R = 8 40 MiB 255 / 244,
  // 256 MiB 1543 / 1512; staged, 8, R = 8 40 MiB 417.5 / 412.6.
  out->sums_by_launch = out->overlap && !c->profile && how != STAGED && c->sum_ctas < 64;
  for (RGroup& g : out->groups) {
    if (g.kind == OP_MOVE && c->path == HOCCL_PATH_SM && c->copy_ctas >= kAllSms && call.kind != PLAN_ALLTOALL && g.phase != PHASE_OWN &&
        !(plan_kind & (g.phase == PHASE_RS ? PLAN_FLAG_RS_DIRECT : PLAN_FLAG_AG_DIRECT))) {
      size_t bytes = 0;
      for (const Seg& s : g.segs) bytes += s.bytes;
      if (bytes >= kRingWalkFrom && bytes <= kRingWalkTo) g.ctas = kAllSms - 1;
    }
    if (beside && g.kind == OP_MOVE && g.piece + 1 < P.pieces) g.ctas = kBesideSums;
    // the first piece's sum has nothing beside it unless the next piece's contributions are copied meanwhile
    if (out->overlap && g.kind == OP_CHAIN) g.beside = g.piece > 0 || how == STAGED;
  }
  return HOCCL_OK;
}

hoccl_result_t inspect_call(hoccl_comm* c, Call* call, Layout* out, std::vector<uint64_t>* key) {
  OptionsOut opt;
  hoccl_result_t rc = call_options(c, *call, &opt);
  if (rc != HOCCL_OK) return rc;
  if (opt.executor == EXEC_ONEPASS || call->h_send) return HOCCL_ERR_UNSUPPORTED;
  RouteGuard guard(c, (hoccl_path_t)opt.path, opt.copy_ctas);
  *key = make_key(c, *call);
  rc = validate(c, call);
  if (rc != HOCCL_OK || call->count == 0) return rc;
  rc = lay_out(c, *call, opt, contributions(c, *call, opt, call->count * dtype_size(call->dtype)), out);
  for (const RGroup& g : out->groups) {
    out->ctas.push_back(0);
    if (g.kind == OP_MOVE && c->path != HOCCL_PATH_SM && !g.edges) continue;
    for (const KernelLaunch& k : kernel_launches(c, out->plan, g)) out->ctas.back() = std::max(out->ctas.back(), k.grid);
  }
  for (int p = 0; p < out->plan.pieces; p++) out->chains.push_back(out->overlap ? (int)copy_chains(c, out->plan, out->groups, p) : 0);
  return rc;
}

hoccl_result_t run_collective(hoccl_comm* c, Call* call, cudaStream_t user) {
  const double t0 = now_us();
  if (!c) return HOCCL_ERR_INVALID_ARG;
  if (dtype_size(call->dtype) == 0) return HOCCL_ERR_UNSUPPORTED;
  if (!call->send || !call->recv) return HOCCL_ERR_INVALID_ARG;
  OptionsOut opt;
  {
    hoccl_result_t orc = call_options(c, *call, &opt);
    if (orc != HOCCL_OK) return orc;
  }
  // a small message on the copy route runs on the copy kernel's route: the communicator shows that route for this call only
  RouteGuard guard(c, (hoccl_path_t)opt.path, opt.copy_ctas);
  if (call->h_send && call->count != 0) {
    HostViews views;
    if (host_direct_applies(c, *call, opt, &views)) {
      const hoccl_result_t vrc = validate(c, call);
      return vrc == HOCCL_OK ? run_host_direct(c, *call, views, user, t0) : vrc;
    }
  }
  const bool onepass_case = opt.executor == EXEC_ONEPASS;
  const bool fused = opt.executor == EXEC_ONE_KERNEL;
  const bool roles = opt.executor == EXEC_ROLES;
  const bool graphs = opt.executor != EXEC_STREAMS && !onepass_case;
  std::vector<uint64_t> key;
  if (graphs && call->count != 0) {
    // Fast path: a call whose signature (operation, count, dtype, every pointer, every setting that shapes the graph)
    // was seen before was validated and planned then; replaying its graph is all that is left to do.
    key = make_key(c, *call);
    for (auto& e : c->cache)
      if (e.key == key) {
        c->stats = hoccl_stats_t{};
        c->stats.graph_hit = 1;
        CU_TRY(c, cudaSetDevice(c->device));
        if (c->handshake) {
          hoccl_result_t prc = ensure_proxy(c);
          if (prc != HOCCL_OK) return prc;
        }
        return launch_entry(c, &e, user, t0);
      }
  }
  hoccl_result_t rc = validate(c, call);
  if (rc != HOCCL_OK) return rc;
  c->stats = hoccl_stats_t{};
  if (call->count == 0) return HOCCL_OK;
  CU_TRY(c, cudaSetDevice(c->device));

  if (onepass_case) {
    // comparison point: the whole reduction in one kernel, same order and rounding as the ring, no moves, no scratch
    OnePassArgs a;
    a.R = c->R;
    a.dtype = call->dtype;
    a.write_all = call->kind == PLAN_ALLREDUCE ? 1 : 0;
    a.pad = 0;
    if (call->kind == PLAN_ALLREDUCE) {
      a.count = call->count;
      a.q = (call->count + (size_t)c->R - 1) / (size_t)c->R;
    } else {
      a.count = (unsigned long long)call->count * c->R;
      a.q = call->count;
    }
    for (int r = 0; r < c->R; r++) {
      a.x[r] = call->send[r];
      a.y[r] = call->recv[r];
    }
    CU_TRY(c, launch_onepass(a, (int)c->sum_ctas, user));
    c->stats.n_sum_launches = 1;
    c->stats.max_sum_ctas = c->sum_ctas;
    c->stats.n_pieces = 1;
    c->stats.host_launch_us = now_us() - t0;
    return HOCCL_OK;
  }
  const Contributions how = contributions(c, *call, opt, call->count * dtype_size(call->dtype));
  if (call->h_send && how != STAGED) return run_host_in_place(c, *call, std::move(key), user, t0);
  Layout lay;
  rc = lay_out(c, *call, opt, how, &lay);
  if (rc != HOCCL_OK) return rc;
  const Plan& P = lay.plan;
  const std::vector<RGroup>& groups = lay.groups;
  c->stats.n_pieces = P.pieces;
  c->stats.max_sum_ctas = 0;
  if (c->path == HOCCL_PATH_CE_HOST && (!c->host_staging || lay.host_need > c->host_staging_bytes)) return HOCCL_ERR_SCRATCH;
  if (graphs) {
    if (c->handshake) {
      // Driver copies share a hardware queue with the copies the parked stream has queued behind its hand-over; a copy
      // issued by the proxy can end up behind them and never start (observed).  Kernels do not have that problem.
      // (Checked before the cache lookup; the proxy is created on first use.)
      rc = ensure_proxy(c);
      if (rc != HOCCL_OK) return rc;
    }
    GraphEntry entry;
    entry.key = key;
    entry.n_pieces = P.pieces;
    if (call->h_send) {
      entry.piece_exec.assign(P.pieces, nullptr);
      entry.h2d.resize(P.pieces);
      entry.d2h.resize(P.pieces);
      for (int p = 0; p < P.pieces; p++) {
        for (int r = 0; r < c->R; r++) {
          add_host_copies(P, p, (char*)call->send[r], (char*)call->h_send[r], &entry.h2d[p]);
          add_host_copies(P, p, (char*)call->recv[r], (char*)call->h_recv[r], &entry.d2h[p]);
        }
        bool any = false;
        for (const PlanGroup& pg : P.groups) any = any || pg.piece == p;
        if (!any) continue;   // e.g. one rank copying in place: nothing to run between the copies
        rc = build_graph(c, P, groups, &entry, p, &entry.piece_exec[p]);
        if (rc != HOCCL_OK) {
          destroy_entry(&entry);   // the pieces built so far, and any profile events
          return rc;
        }
      }
    } else if (lay.overlap) {
      entry.part_exec.assign((size_t)P.pieces * 3, nullptr);
      if (lay.sums_by_launch) {
        entry.part_sums.resize((size_t)P.pieces);
        for (const RGroup& g : groups)
          if (g.kind != OP_MOVE)
            for (KernelLaunch& k : kernel_launches(c, P, g)) {
              entry.part_sums[(size_t)g.piece].push_back(std::move(k));
              entry.n_sum_launches++;
            }
      }
      for (int p = 0; p < P.pieces && rc == HOCCL_OK; p++)
        for (int part = 0; part < 3 && rc == HOCCL_OK; part++)
          if (part != 1 || !lay.sums_by_launch) rc = build_graph(c, P, groups, &entry, p, &entry.part_exec[(size_t)p * 3 + part], part);
      if (rc != HOCCL_OK) {
        destroy_entry(&entry);
        return rc;
      }
    } else {
      rc = fused ? build_ring(c, P, groups, &entry) : roles ? build_roles(c, P, groups, &entry) : HOCCL_ERR_UNSUPPORTED;
      // not asked for, too many ranks for one launch (fused), or more CTAs than can be resident together (roles)
      if (rc == HOCCL_ERR_UNSUPPORTED) {
        add_launches(c, P, &lay.groups, &entry);
        rc = build_graph(c, P, groups, &entry, -1, &entry.exec);
      }
      if (rc != HOCCL_OK) {
        destroy_entry(&entry);
        return rc;
      }
    }
    // handshake mode: place the graph on the device now; the proxy must not meet first-launch work later
    if (c->handshake) {
      cudaError_t ue = cudaGraphUpload(entry.exec, c->proxy->work_stream());
      if (ue != cudaSuccess) {
        destroy_entry(&entry);
        return cuda_fail(c, ue, "cudaGraphUpload");
      }
    }
    return launch_entry(c, cache_put(c, std::move(entry)), user, t0);
  }
  Tally tally;
  rc = run_streams(c, P, groups, user, &tally);
  if (rc != HOCCL_OK) return rc;
  c->stats.n_moves = tally.moves;
  c->stats.n_move_launches = tally.move_launches;
  c->stats.n_sum_launches = tally.sum_launches;
  c->stats.max_sum_ctas = tally.sum_launches ? c->sum_ctas : 0;
  c->stats.max_copy_ctas = tally.move_launches ? c->copy_ctas : 0;
  c->stats.host_launch_us = now_us() - t0;
  return HOCCL_OK;
}

}  // namespace hoccl
