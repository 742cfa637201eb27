// sm_100a kernels of libhoccl.
//
// sum2_kernel  - the one arithmetic step of the ring reduce-scatter (the paper has none: Sec. 4
//                "Limitations" leaves reductions to SM-side execution): per element one binary32
//                add of the arrived partial and the local contribution, rounded to nearest even
//                into the I/O dtype.  HBM bound: 2 reads + 1 write per element and one add.
// copy_kernel  - SM-driven byte copy with a CTA budget: the comparison path for moves (the paper's
//                "NCCL under an SM budget", Sec. 5 "Baselines").
// Both are batched: one launch serves all ranks of a ring step through a segment table, and the
// segments are flattened into one index space (by the host, which passes the prefix sums along with the
// table: the kernels have no set-up phase and no barrier) so that a small CTA budget stays balanced.  Loads and
// stores are 16-byte vectors, fully coalesced (consecutive threads touch consecutive vectors);
// segments whose three addresses are not congruent modulo 16 fall back to element-wise accesses.
// The sum streams CTA-contiguous tiles (blockDim x 4 vectors per operand) with all of a tile's loads in
// flight before the first add.  No shared-memory or bulk-copy staging: one SM's memory port carries about
// 123 GB/s of mixed 2:1 read/write traffic whatever issues it (bulk loads + bulk stores measured the same),
// stores are capped at 32 B/clk per SM, and the register version already reaches 116 GB/s per SM.
#include "kernels.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "device_common.cuh"

namespace hoccl {

namespace {

template <int DT, int U, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) sum2_kernel(const __grid_constant__ SumBatch batch) {
  using T = Traits<DT>;
  const Flat& f = batch.flat;   // filled on the host for this kernel variant: no set-up phase, no barrier
  const int nseg = batch.nseg;
  wait_for_stream();
  if (batch.smid_out != nullptr && threadIdx.x == 0) {
    unsigned id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    batch.smid_out[blockIdx.x] = id;
  }
  const unsigned long long total = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long gt = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;

  // ---- vector body, tile by tile: a tile is a contiguous run of U * blockDim vectors of one segment; the
  // CTA streams it with U loads per operand in flight per thread (thread t takes vectors t, t+B, t+2B, ...).
  {
    const unsigned long long T_all = f.tpre[nseg];
    const unsigned tile_v = U * blockDim.x;
    int k = 0;
    for (unsigned long long t = blockIdx.x; t < T_all; t += gridDim.x) {
      while (t >= f.tpre[k + 1]) k++;
      const unsigned long long first = (t - f.tpre[k]) * tile_v;          // first vector of the tile in segment k
      const unsigned long long left = f.nvec[k] - first;
      const unsigned n_here = left < tile_v ? (unsigned)left : tile_v;
      const size_t h = (size_t)f.head[k] * T::E;
      const uint4* a = reinterpret_cast<const uint4*>(static_cast<const char*>(batch.seg[k].inbox) + h) + first;
      const uint4* b = reinterpret_cast<const uint4*>(static_cast<const char*>(batch.seg[k].local) + h) + first;
      uint4* o = reinterpret_cast<uint4*>(static_cast<char*>(batch.seg[k].out) + h) + first;
      uint4 va[U], vb[U];
      if (n_here == tile_v) {
#pragma unroll
        for (int u = 0; u < U; u++) {
          va[u] = __ldcs(a + threadIdx.x + u * blockDim.x);
          vb[u] = __ldcs(b + threadIdx.x + u * blockDim.x);
        }
#pragma unroll
        for (int u = 0; u < U; u++) o[threadIdx.x + u * blockDim.x] = T::add_vec(va[u], vb[u]);
      } else {
#pragma unroll
        for (int u = 0; u < U; u++) {
          const unsigned i = threadIdx.x + u * blockDim.x;
          if (i < n_here) {
            va[u] = __ldcs(a + i);
            vb[u] = __ldcs(b + i);
          }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const unsigned i = threadIdx.x + u * blockDim.x;
          if (i < n_here) o[i] = T::add_vec(va[u], vb[u]);
        }
      }
    }
  }
  // ---- element-wise items: heads, tails and segments without a common 16-byte phase
  {
    const unsigned long long S = f.spre[nseg];
    int k = 0;
    for (unsigned long long j = gt; j < S; j += total) {
      while (j >= f.spre[k + 1]) k++;
      unsigned long long i = j - f.spre[k];
      if (i >= f.head[k]) i += f.nvec[k] * T::VE;
      T::add_scalar(batch.seg[k].inbox, batch.seg[k].local, batch.seg[k].out, i);
    }
  }
}

template <int U, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) copy_kernel(const __grid_constant__ CopyBatch batch) {
  const Flat& f = batch.flat;
  const int nseg = batch.nseg;
  if (batch.smid_out != nullptr && threadIdx.x == 0) {
    unsigned id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    batch.smid_out[blockIdx.x] = id;
  }
  const unsigned long long total = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long gt = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  {
    const unsigned long long T_all = f.tpre[nseg];
    const unsigned tile_v = U * blockDim.x;
    int k = 0;
    for (unsigned long long t = blockIdx.x; t < T_all; t += gridDim.x) {
      while (t >= f.tpre[k + 1]) k++;
      const unsigned long long first = (t - f.tpre[k]) * tile_v;
      const unsigned long long left = f.nvec[k] - first;
      const unsigned n_here = left < tile_v ? (unsigned)left : tile_v;
      const uint4* a = reinterpret_cast<const uint4*>(static_cast<const char*>(batch.seg[k].src) + f.head[k]) + first;
      uint4* o = reinterpret_cast<uint4*>(static_cast<char*>(batch.seg[k].dst) + f.head[k]) + first;
      uint4 va[U];
      if (n_here == tile_v) {
#pragma unroll
        for (int u = 0; u < U; u++) va[u] = __ldcs(a + threadIdx.x + u * blockDim.x);
#pragma unroll
        for (int u = 0; u < U; u++) o[threadIdx.x + u * blockDim.x] = va[u];
      } else {
#pragma unroll
        for (int u = 0; u < U; u++) {
          const unsigned i = threadIdx.x + u * blockDim.x;
          if (i < n_here) va[u] = __ldcs(a + i);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
          const unsigned i = threadIdx.x + u * blockDim.x;
          if (i < n_here) o[i] = va[u];
        }
      }
    }
  }
  {
    const unsigned long long S = f.spre[nseg];
    int k = 0;
    for (unsigned long long j = gt; j < S; j += total) {
      while (j >= f.spre[k + 1]) k++;
      unsigned long long i = j - f.spre[k];
      if (i >= f.head[k]) i += f.nvec[k] * 16;
      static_cast<unsigned char*>(batch.seg[k].dst)[i] = static_cast<const unsigned char*>(batch.seg[k].src)[i];
    }
  }
}

__device__ __forceinline__ float scalar_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ unsigned short scalar_add(unsigned short a, unsigned short b) {   // bf16
  return __bfloat16_as_ushort(__float2bfloat16_rn(__fadd_rn(__uint_as_float((uint32_t)a << 16), __uint_as_float((uint32_t)b << 16))));
}

// One element of a chain segment, element-wise: the same adds in the same order as the vector bodies.  NOPS > 0: the operand count.  Eight
// loads of an element are in flight together (one after the other they cost ~0.7 us each).
template <int DT, int NOPS>
__device__ __forceinline__ void chain_scalar(const ChainBatch& b, const ChainSeg& sg, unsigned long long i) {
  using V = typename std::conditional<DT == 0, float, unsigned short>::type;
  constexpr int N = NOPS ? NOPS : 8;
  void* const* op = b.ptr + sg.first_ptr;
  const int nops = NOPS ? NOPS : sg.nops;
  V acc = V();
  for (int q0 = 0; q0 < nops; q0 += N) {
    V x[N];
#pragma unroll
    for (int q = 0; q < N; q++)
      if (NOPS || q0 + q < nops) x[q] = static_cast<const V*>(op[q0 + q])[i];
#pragma unroll
    for (int q = 0; q < N; q++)
      if (NOPS || q0 + q < nops) acc = q0 + q == 0 ? x[q] : scalar_add(acc, x[q]);
  }
  for (int d = 0; d < sg.ndst; d++) static_cast<V*>(op[nops + d])[i] = acc;
}

// Element-wise items of a launch: heads, tails and segments without a common 16-byte phase.
template <int DT, int NOPS>
__device__ __forceinline__ void chain_scalar_items(const ChainBatch& batch) {
  using T = Traits<DT>;
  const Flat& f = batch.flat;
  const unsigned long long total = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long S = f.spre[batch.nseg];
  int k = 0;
  for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < S; j += total) {
    while (j >= f.spre[k + 1]) k++;
    unsigned long long i = j - f.spre[k];
    if (i >= f.head[k]) i += f.nvec[k] * T::VE;
    chain_scalar<DT, NOPS>(batch, batch.seg[k], i);
  }
}

template <int DT>
__device__ __forceinline__ uint4 chain_add(uint4 a, uint4 b) {
  return DT == 1 ? add_vec_bf16_native(a, b) : Traits<DT>::add_vec(a, b);
}

template <class Batch>
__device__ __forceinline__ void report_sm(const Batch& batch) {
  if (batch.smid_out != nullptr && threadIdx.x == 0) {
    unsigned id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    batch.smid_out[blockIdx.x] = id;
  }
}

// Chain sum for any number of operands and destinations: one 16-byte vector per thread and tile; the operands are loaded in batches of up
// to 8 before they are added, so up to 8 x 16 KiB are in flight per CTA.  It serves what the compiled forms below do not (see
// chain_variant): more than 16 operands, mixed counts, and from 9 operands on sums that store for every rank on fewer than 148 CTAs and
// one destination on 128 to 147.  With 148 CTAs and 64 MiB per rank: 9 operands 108 us (6.2 TB/s), 12 139 (6.3), 16 175 (6.5).
template <int DT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) chain_kernel(const __grid_constant__ ChainBatch batch) {
  using T = Traits<DT>;
  const Flat& f = batch.flat;
  const unsigned long long T_all = f.tpre[batch.nseg];
  int k = 0;
  wait_for_stream();
  report_sm(batch);
  for (unsigned long long t = blockIdx.x; t < T_all; t += gridDim.x) {
    while (t >= f.tpre[k + 1]) k++;
    const unsigned long long v = (t - f.tpre[k]) * blockDim.x + threadIdx.x;   // vector of segment k
    if (v >= f.nvec[k]) continue;
    const ChainSeg& sg = batch.seg[k];
    void* const* op = batch.ptr + sg.first_ptr;
    const size_t off = (size_t)f.head[k] * T::E + (size_t)v * 16;
    uint4 acc;
    for (int j0 = 0; j0 < sg.nops; j0 += 8) {
      uint4 buf[8];
#pragma unroll
      for (int j = 0; j < 8; j++)
        if (j0 + j < sg.nops) buf[j] = __ldcs(reinterpret_cast<const uint4*>(static_cast<const char*>(op[j0 + j]) + off));
#pragma unroll
      for (int j = 0; j < 8; j++)
        if (j0 + j < sg.nops) acc = (j0 + j == 0) ? buf[j] : chain_add<DT>(acc, buf[j]);
    }
    for (int d = 0; d < sg.ndst; d++) *reinterpret_cast<uint4*>(static_cast<char*>(op[sg.nops + d]) + off) = acc;
  }
  chain_scalar_items<DT, 0>(batch);
}

// Software-pipelined form of the chain sum for a compile-time operand count NOPS that all segments of the launch share, one
// destination each.  Under a CTA budget the chain sum is bound by the bytes one SM keeps in flight: a load takes
// the better part of a microsecond to come back, so a thread that loads a tile, adds it, stores it and only then loads the
// next one leaves the memory port idle most of the time.  Here every thread keeps P tiles in registers: the loads of tile
// t + P - 1 are issued before the adds and the store of tile t, so P - 1 to P tiles of NOPS x 16 bytes per thread are in
// flight all the time.  That only works when the steady state is straight-line code: with a branch or a segment look-up
// between the loads and the adds the compiler waits for every outstanding load at the join (measured: 89 GB/s per SM, the
// rate of ONE tile in flight, whatever P).  So a CTA takes a CONTIGUOUS range of the flattened tile space, walks it segment
// by segment, and inside a segment the full tiles run through a loop whose body has no branch: unconditional loads, adds,
// store (measured: 163 GB/s per SM for 8 operands with P = 3 and 512 threads, against 111 for chain_kernel).  The ragged
// last tile of a segment and ranges shorter than P tiles take a plain guarded path.  The order of the adds and their
// rounding are those of chain_kernel.  Tiles are THREADS vectors.  The operand pointers are the same for all threads and a
// thread's offset fits 32 bits (kMaxChainSegBytes), which keeps the NOPS + 1 addresses out of the per-thread registers.
template <int DT, int NOPS, int P, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) chain_pipe_kernel(const __grid_constant__ ChainBatch batch) {
  using T = Traits<DT>;
  const Flat& f = batch.flat;
  const int nseg = batch.nseg;
  {
    const unsigned long long T_all = f.tpre[nseg];
    // this CTA's share of the flattened tile space: [A, B)
    const unsigned long long A = T_all / gridDim.x * blockIdx.x + min((unsigned long long)blockIdx.x, T_all % gridDim.x);
    const unsigned long long B = A + T_all / gridDim.x + (blockIdx.x < T_all % gridDim.x ? 1 : 0);
    int k = 0;
    while (k < nseg && f.tpre[k + 1] <= A) k++;
    wait_for_stream();
    report_sm(batch);
    for (; k < nseg && f.tpre[k] < B; k++) {
      const unsigned a = (unsigned)((A > f.tpre[k] ? A : f.tpre[k]) - f.tpre[k]);                 // tiles [a, b) of segment k
      const unsigned b = (unsigned)((B < f.tpre[k + 1] ? B : f.tpre[k + 1]) - f.tpre[k]);
      const unsigned nvec = (unsigned)f.nvec[k];
      const unsigned bf = b < nvec / THREADS ? b : nvec / THREADS;                                // full tiles end here
      const char* src[NOPS];
#pragma unroll
      for (int q = 0; q < NOPS; q++) src[q] = static_cast<const char*>(batch.ptr[batch.seg[k].first_ptr + q]);
      char* out = static_cast<char*>(batch.ptr[batch.seg[k].first_ptr + NOPS]);
      const unsigned off0 = f.head[k] * T::E + threadIdx.x * 16;
      uint4 buf[P][NOPS];
      auto load = [&](uint4(&bb)[NOPS], unsigned t) {
        const unsigned o = off0 + t * (THREADS * 16);
#pragma unroll
        for (int q = 0; q < NOPS; q++) bb[q] = __ldcs(reinterpret_cast<const uint4*>(src[q] + o));
      };
      auto finish = [&](const uint4(&bb)[NOPS], unsigned t) {
        uint4 acc = bb[0];
#pragma unroll
        for (int q = 1; q < NOPS; q++) acc = chain_add<DT>(acc, bb[q]);
        *reinterpret_cast<uint4*>(out + (off0 + t * (THREADS * 16))) = acc;
      };
      unsigned i = a;
      if (bf > a && bf - a >= (unsigned)P) {
#pragma unroll
        for (int p = 0; p < P - 1; p++) load(buf[p], i + p);
        for (; i + 2 * P - 1 <= bf; i += P) {   // steady state: no branch between a tile's loads and the adds of an older tile
#pragma unroll
          for (int p = 0; p < P; p++) {
            load(buf[(p + P - 1) % P], i + p + P - 1);
            finish(buf[p], i + p);
          }
        }
#pragma unroll
        for (int p = 0; p < P - 1; p++) finish(buf[p], i + p);
        i += P - 1;
      }
      for (; i < bf; i++) {   // what is left of the full tiles
        load(buf[0], i);
        finish(buf[0], i);
      }
      if (i < b && i * THREADS + threadIdx.x < nvec) {   // the ragged last tile of the segment
        load(buf[0], i);
        finish(buf[0], i);
      }
    }
  }
  chain_scalar_items<DT, NOPS>(batch);
}

// The same for 9 to 16 operands, which do not fit a thread's registers P at a time: a tile is two steps of NA and NOPS - NA operands,
// the accumulator is carried from the first to the second, and P steps of loads are in flight.  chain_kernel, which loads 8
// operands, waits, adds and only then loads the rest, ran at 75 (9 operands) to 133 GB/s per SM (16) with 8 CTAs (64 MiB per
// rank: 910 and 1051 us, now 526 and 838).
template <int DT, int NOPS, int P, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) chain_pipe2_kernel(const __grid_constant__ ChainBatch batch) {
  using T = Traits<DT>;
  constexpr int NA = (NOPS + 1) / 2, NB = NOPS - NA;
  constexpr int STEPS = P % 2 ? 2 * P : P;             // steps of one round: whole tiles, and every buffer back in its place
  constexpr int AHEAD = (P - 2) / 2 + 1;               // tiles the prologue touches
  const Flat& f = batch.flat;
  const int nseg = batch.nseg;
  {
    const unsigned long long T_all = f.tpre[nseg];
    const unsigned long long A = T_all / gridDim.x * blockIdx.x + min((unsigned long long)blockIdx.x, T_all % gridDim.x);
    const unsigned long long B = A + T_all / gridDim.x + (blockIdx.x < T_all % gridDim.x ? 1 : 0);
    int k = 0;
    while (k < nseg && f.tpre[k + 1] <= A) k++;
    wait_for_stream();
    report_sm(batch);
    for (; k < nseg && f.tpre[k] < B; k++) {
      const unsigned a = (unsigned)((A > f.tpre[k] ? A : f.tpre[k]) - f.tpre[k]);   // tiles [a, b) of segment k
      const unsigned b = (unsigned)((B < f.tpre[k + 1] ? B : f.tpre[k + 1]) - f.tpre[k]);
      const unsigned nvec = (unsigned)f.nvec[k];
      const unsigned bf = b < nvec / THREADS ? b : nvec / THREADS;                  // full tiles end here
      const char* src[NOPS];
#pragma unroll
      for (int q = 0; q < NOPS; q++) src[q] = static_cast<const char*>(batch.ptr[batch.seg[k].first_ptr + q]);
      char* out = static_cast<char*>(batch.ptr[batch.seg[k].first_ptr + NOPS]);
      const unsigned off0 = f.head[k] * T::E + threadIdx.x * 16;
      uint4 buf[P][NA], acc;
      auto load = [&](uint4(&bb)[NA], unsigned t, int h) {   // step h of tile t
        const unsigned o = off0 + t * (THREADS * 16);
#pragma unroll
        for (int q = 0; q < NA; q++)
          if (h == 0 || q < NB) bb[q] = __ldcs(reinterpret_cast<const uint4*>(src[(h ? NA : 0) + (h && q >= NB ? 0 : q)] + o));
      };
      auto consume = [&](const uint4(&bb)[NA], unsigned t, int h) {
        if (h == 0) {
          acc = bb[0];
#pragma unroll
          for (int q = 1; q < NA; q++) acc = chain_add<DT>(acc, bb[q]);
        } else {
#pragma unroll
          for (int q = 0; q < NB; q++) acc = chain_add<DT>(acc, bb[q]);
          *reinterpret_cast<uint4*>(out + (off0 + t * (THREADS * 16))) = acc;
        }
      };
      unsigned i = a;
      if (bf > a && bf - a >= (unsigned)AHEAD) {
#pragma unroll
        for (int s = 0; s < P - 1; s++) load(buf[s], i + s / 2, s % 2);
        for (; i + (STEPS + P - 2) / 2 < bf; i += STEPS / 2) {   // steady state: straight-line code, as above
#pragma unroll
          for (int s = 0; s < STEPS; s++) {
            load(buf[(s + P - 1) % P], i + (s + P - 1) / 2, (s + P - 1) % 2);
            consume(buf[s % P], i + s / 2, s % 2);
          }
        }
#pragma unroll
        for (int s = 0; s < P - 1; s++) consume(buf[s], i + s / 2, s % 2);
        if ((P - 1) % 2) {   // the last tile the prologue touched has its first step only
          load(buf[P - 1], i + (P - 2) / 2, 1);
          consume(buf[P - 1], i + (P - 2) / 2, 1);
        }
        i += AHEAD;
      }
      for (; i < b; i++) {   // what is left: full tiles and the ragged last one
        if (i * THREADS + threadIdx.x >= nvec) break;
        load(buf[0], i, 0);
        load(buf[1], i, 1);
        consume(buf[0], i, 0);
        consume(buf[1], i, 1);
      }
    }
  }
  chain_scalar_items<DT, NOPS>(batch);
}

// Whole-GPU sums, and the sum that carries the all-gather too: NOPS operands are read once, the result is stored to NDST
// destinations (1, or NOPS: one per rank).  That is what the collective cannot do without; bound by HBM with a whole-GPU grid, which has a CTA
// per tile (R = 8, 64 MiB fp32, every rank: 163.8 us, 6.56 TB/s; 170 with one CTA per SM that walks the tiles).
// A tile is U x THREADS vectors, so U x NOPS loads are in flight per thread before the first add.
template <int DT, int NOPS, int NDST, int U, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) chain_fan_kernel(const __grid_constant__ ChainBatch batch) {
  using T = Traits<DT>;
  const Flat& f = batch.flat;
  // tile t of the flattened space belongs to CTA t mod grid; a walk goes segment by segment, so that the NOPS + NDST pointers are loaded
  // once per segment and not once per tile (one CTA per SM, R = 8, 64 MiB fp32, tiles of 384 vectors: 194 us with a look-up per tile, 171 without)
  const unsigned long long T_all = f.tpre[batch.nseg];
  int k = 0;
  wait_for_stream();
  report_sm(batch);
  for (unsigned long long at = blockIdx.x; at < T_all;) {
    while (at >= f.tpre[k + 1]) k++;
    const unsigned tiles = (unsigned)(f.tpre[k + 1] - f.tpre[k]);
    const char* src[NOPS];
    char* dst[NDST];
#pragma unroll
    for (int q = 0; q < NOPS; q++) src[q] = static_cast<const char*>(batch.ptr[batch.seg[k].first_ptr + q]);
#pragma unroll
    for (int d = 0; d < NDST; d++) dst[d] = static_cast<char*>(batch.ptr[batch.seg[k].first_ptr + NOPS + d]);
    const unsigned nvec = (unsigned)f.nvec[k], head = f.head[k] * T::E;
    unsigned t = (unsigned)(at - f.tpre[k]);
    for (; t < tiles; t += gridDim.x) {
      const unsigned v0 = t * (U * THREADS) + threadIdx.x;   // first vector of this thread
      const unsigned off = head + v0 * 16;
      auto finish = [&](const uint4(&bb)[NOPS], int u) {
        uint4 acc = bb[0];
#pragma unroll
        for (int q = 1; q < NOPS; q++) acc = chain_add<DT>(acc, bb[q]);
#pragma unroll
        for (int d = 0; d < NDST; d++) *reinterpret_cast<uint4*>(dst[d] + (off + u * (THREADS * 16))) = acc;
      };
      uint4 buf[U][NOPS];
      if (v0 + (U - 1) * THREADS < nvec) {
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
          for (int q = 0; q < NOPS; q++) buf[u][q] = __ldcs(reinterpret_cast<const uint4*>(src[q] + (off + u * (THREADS * 16))));
#pragma unroll
        for (int u = 0; u < U; u++) finish(buf[u], u);
      } else {
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (v0 + u * THREADS >= nvec) break;
#pragma unroll
          for (int q = 0; q < NOPS; q++) buf[u][q] = __ldcs(reinterpret_cast<const uint4*>(src[q] + (off + u * (THREADS * 16))));
          finish(buf[u], u);
        }
      }
    }
    at = f.tpre[k] + t;
  }
  chain_scalar_items<DT, NOPS>(batch);
}

// See StoreAllArgs.  Latency bound: one fetch of parameters, one round trip of loads, one of stores.  Us per call in a burst, against chain_kernel's tables
// and 8 operands at a time: 16 ranks bf16 on 8 CTAs 4 KiB per rank 6.1 -> 4.1, 8.1 KiB (heads and tails) 10.25 -> 4.15, 192 KiB 12.3 -> 9.5; 9 ranks fp32 64
// KiB 8.2 -> 4.4; whole GPU 16 ranks 1 MiB 10.2 -> 5.0, 8 ranks 1 MiB (chain_fan_kernel) 6.1 -> 4.1.
// SPLIT: several chunks per CTA.  A form of its own: with both in one, three divisions by arguments stand before the first load instead of one, and
// calls that just end within a step of 2.048 us (see launch_in_order) need two (2 ranks bf16 16 KiB 2.4 us a call in a burst, 4.1 so).
template <int DT, int NOPS, int THREADS, bool SPLIT>
__global__ void __launch_bounds__(THREADS, 1) store_all_kernel(const __grid_constant__ StoreAllArgs a) {
  using T = Traits<DT>;
  const unsigned width = SPLIT ? THREADS / a.groups : THREADS, group = SPLIT ? threadIdx.x / width : 0, tid = threadIdx.x - group * width;
  const unsigned c = SPLIT ? blockIdx.x * a.groups + group : blockIdx.x / a.parts, part = SPLIT ? 0 : blockIdx.x - c * a.parts;
  wait_for_stream();
  if (SPLIT && c >= NOPS) return;   // the last CTA of a grid that the chunks do not fill
  const char* src[NOPS];
#pragma unroll
  for (int j = 0; j < NOPS; j++) src[j] = static_cast<const char*>(a.x[(c + 1 + j) % NOPS]);
  const unsigned lo = min(c * a.q, a.count), n = min(a.q, a.count - lo);      // elements [lo, lo + n)
  const unsigned at = lo * T::E;                                              // byte offset of the chunk
  const unsigned head = min(((16u - ((a.phase + at) & 15u)) & 15u) / T::E, n), nvec = (n - head) / T::VE;
  const unsigned per = (nvec + a.parts - 1) / a.parts, v1 = min(nvec, (part + 1) * per);
  constexpr int U = NOPS <= 4 ? 4 : NOPS <= 8 ? 2 : 1;   // vectors of a thread in flight
  for (unsigned v = part * per + tid; v < v1; v += U * width) {
    uint4 buf[U][NOPS];
#pragma unroll
    for (int u = 0; u < U; u++)
      if (v + u * width < v1) {
#pragma unroll
        for (int j = 0; j < NOPS; j++) buf[u][j] = __ldcs(reinterpret_cast<const uint4*>(src[j] + (at + head * T::E + (v + u * width) * 16)));
      }
#pragma unroll
    for (int u = 0; u < U; u++)
      if (v + u * width < v1) {
        uint4 acc = buf[u][0];
#pragma unroll
        for (int j = 1; j < NOPS; j++) acc = chain_add<DT>(acc, buf[u][j]);
#pragma unroll
        for (int r = 0; r < NOPS; r++) *reinterpret_cast<uint4*>(static_cast<char*>(a.y[r]) + (at + head * T::E + (v + u * width) * 16)) = acc;
      }
  }
  // head and tail, element by element
  const unsigned ns = n - nvec * T::VE;
  if (part == a.parts - 1 && tid < ns) {
    using V = typename std::conditional<DT == 0, float, unsigned short>::type;
    const unsigned i = lo + (tid < head ? tid : tid + nvec * T::VE);
    V x[NOPS];
#pragma unroll
    for (int j = 0; j < NOPS; j++) x[j] = reinterpret_cast<const V*>(src[j])[i];
#pragma unroll
    for (int j = 1; j < NOPS; j++) x[0] = scalar_add(x[0], x[j]);
#pragma unroll
    for (int r = 0; r < NOPS; r++) static_cast<V*>(a.y[r])[i] = x[0];
  }
}

// The 16 bytes that start `sh` bytes into the 32 bytes lo, hi; sh (0..15) is the same for all threads.
__device__ __forceinline__ uint4 bytes_at(uint4 lo, uint4 hi, unsigned sh) {
  uint32_t w0 = lo.x, w1 = lo.y, w2 = lo.z, w3 = lo.w, w4 = hi.x, w5 = hi.y, w6 = hi.z, w7 = hi.w;
  if (sh & 8) {
    w0 = w2;
    w1 = w3;
    w2 = w4;
    w3 = w5;
    w4 = w6;
    w5 = w7;
  }
  if (sh & 4) {
    w0 = w1;
    w1 = w2;
    w2 = w3;
    w3 = w4;
    w4 = w5;
  }
  const unsigned b = (sh & 3) * 8;
  return make_uint4(__funnelshift_r(w0, w1, b), __funnelshift_r(w1, w2, b), __funnelshift_r(w2, w3, b), __funnelshift_r(w3, w4, b));
}

// Segment of item t: the largest k with pre[k] <= t (pre is non-decreasing, pre[n] > t).
__device__ __forceinline__ int find_segment(const unsigned* pre, int n, unsigned t) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] <= t) lo = mid;
    else hi = mid;
  }
  return lo;
}

// The moves of a launch: copies and fan-outs (one read, ndst stores) of any phase and length, the tile walk of copy_kernel with the
// tile chosen for the launch.  In phase it is HBM bound with a whole-GPU grid and bound by the SM's stores (62 GB/s) under a CTA
// budget.  Out of phase a byte-wise copy ran at a tenth of that (8 chunks of 500,014 bytes to 8 ranks each: 37 us of a 38 us
// all-gather, now 10); here a thread loads the two aligned vectors that hold its 16 bytes (the second is its neighbour's first, an
// L1 hit), shifts them into place and stores aligned vectors.
template <int U, int THREADS, class Batch>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 6 : 1) move_kernel(const __grid_constant__ Batch batch) {
  constexpr int H = U < 4 ? U : 4;
  const int nseg = batch.nseg;
  const unsigned T_all = batch.tpre[nseg], tile_u = batch.tile_u;
  int k = blockIdx.x < T_all ? find_segment(batch.tpre, nseg, blockIdx.x) : 0;
  wait_for_stream();
  if (blockIdx.x < T_all) {
    for (unsigned t = blockIdx.x; t < T_all; t += gridDim.x) {
      while (t >= batch.tpre[k + 1]) k++;
      const MoveSeg& sg = batch.seg[k];
      const unsigned first = (t - batch.tpre[k]) * (tile_u * THREADS) + threadIdx.x;
      const unsigned tile_end = (t - batch.tpre[k] + 1) * (tile_u * THREADS), end = tile_end < sg.nvec ? tile_end : sg.nvec;
      const char* s = static_cast<const char*>(sg.src) + sg.head;
      const unsigned sh = (unsigned)(uintptr_t)s & 15;
      const uint4* a = reinterpret_cast<const uint4*>(s - sh) + first;
      uint4 v[U];
      if (sh == 0 && tile_u == U && tile_end <= sg.nvec) {   // a whole tile: no bounds between its loads
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = __ldcs(a + u * THREADS);
        for (int d = 0; d < sg.ndst; d++) {
          uint4* o = reinterpret_cast<uint4*>(static_cast<char*>(batch.dst[sg.first_dst + d]) + sg.head) + first;
#pragma unroll
          for (int u = 0; u < U; u++) o[u * THREADS] = v[u];
        }
        continue;
      }
      if (sh == 0) {
#pragma unroll
        for (int u = 0; u < U; u++)
          if (first + u * THREADS < end) v[u] = __ldcs(a + u * THREADS);
      } else {
#pragma unroll
        for (int h = 0; h < U; h += H) {   // H pairs in flight
          uint4 hi[H];
#pragma unroll
          for (int u = 0; u < H; u++)
            if (first + (h + u) * THREADS < end) {
              v[h + u] = a[(h + u) * THREADS];
              hi[u] = a[(h + u) * THREADS + 1];
            }
#pragma unroll
          for (int u = 0; u < H; u++) v[h + u] = bytes_at(v[h + u], hi[u], sh);
        }
      }
      for (int d = 0; d < sg.ndst; d++) {
        uint4* o = reinterpret_cast<uint4*>(static_cast<char*>(batch.dst[sg.first_dst + d]) + sg.head) + first;
#pragma unroll
        for (int u = 0; u < U; u++)
          if (first + u * THREADS < end) o[u * THREADS] = v[u];
      }
    }
  }
  const unsigned S = batch.spre[nseg], j0 = blockIdx.x * THREADS + threadIdx.x;
  if (j0 < S) {
    k = find_segment(batch.spre, nseg, j0);
    for (unsigned j = j0; j < S; j += gridDim.x * THREADS) {
      while (j >= batch.spre[k + 1]) k++;
      const MoveSeg& sg = batch.seg[k];
      unsigned long long i = j - batch.spre[k];
      if (i >= sg.head) i += (unsigned long long)sg.nvec * 16;
      const unsigned char v = static_cast<const unsigned char*>(sg.src)[i];
      for (int d = 0; d < sg.ndst; d++) static_cast<unsigned char*>(batch.dst[sg.first_dst + d])[i] = v;
    }
  }
}

// ---- one-pass ring reduction (comparison point) -------------------------------------------------------------------
template <int DT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) onepass_kernel(const __grid_constant__ OnePassArgs a) {
  using T = Traits<DT>;
  __shared__ unsigned long long tpre[kMaxOnePassRanks + 1], spre[kMaxOnePassRanks + 1], lo_s[kMaxOnePassRanks], nvec_s[kMaxOnePassRanks];
  __shared__ int vec_ok;
  const int R = a.R;
  if (threadIdx.x == 0) {
    bool ok = ((a.q * T::E) % 16) == 0;
    for (int r = 0; r < R; r++) ok = ok && (((uintptr_t)a.x[r] | (uintptr_t)a.y[r]) & 15) == 0;
    vec_ok = ok ? 1 : 0;
    unsigned long long t = 0, sc = 0;
    tpre[0] = 0;
    spre[0] = 0;
    for (int c = 0; c < R; c++) {
      unsigned long long lo = (unsigned long long)c * a.q, hi = lo + a.q;
      if (lo > a.count) lo = a.count;
      if (hi > a.count) hi = a.count;
      const unsigned long long len = hi - lo;
      const unsigned long long nv = ok ? len / T::VE : 0;
      lo_s[c] = lo;
      nvec_s[c] = nv;
      t += (nv + blockDim.x - 1) / blockDim.x;
      tpre[c + 1] = t;
      sc += len - nv * T::VE;
      spre[c + 1] = sc;
    }
  }
  __syncthreads();
  // vector part: one 16-byte vector per thread and tile, the R operands loaded in batches of 8 before they are added
  {
    int c = 0;
    for (unsigned long long t = blockIdx.x; t < tpre[R]; t += gridDim.x) {
      while (t >= tpre[c + 1]) c++;
      const unsigned long long v = (t - tpre[c]) * blockDim.x + threadIdx.x;
      if (v >= nvec_s[c]) continue;
      const size_t byte_off = (size_t)(lo_s[c] + v * T::VE) * T::E;
      uint4 acc;
      for (int k0 = 1; k0 <= R; k0 += 8) {
        uint4 buf[8];
#pragma unroll
        for (int j = 0; j < 8; j++)
          if (k0 + j <= R) buf[j] = __ldcs(reinterpret_cast<const uint4*>(static_cast<const char*>(a.x[(c + k0 + j) % R]) + byte_off));
#pragma unroll
        for (int j = 0; j < 8; j++)
          if (k0 + j <= R) acc = (k0 + j == 1) ? buf[j] : T::add_vec(acc, buf[j]);
      }
      if (a.write_all) {
        for (int r = 0; r < R; r++) *reinterpret_cast<uint4*>(static_cast<char*>(a.y[r]) + byte_off) = acc;
      } else {
        *reinterpret_cast<uint4*>(static_cast<char*>(a.y[c]) + (size_t)v * 16) = acc;
      }
    }
  }
  // element-wise part: chunk tails, or everything when a buffer or the chunk size is not 16-byte aligned
  {
    const unsigned long long total = (unsigned long long)gridDim.x * blockDim.x;
    int c = 0;
    for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < spre[R]; j += total) {
      while (j >= spre[c + 1]) c++;
      const unsigned long long local = nvec_s[c] * T::VE + (j - spre[c]);   // element inside chunk c
      const unsigned long long i = lo_s[c] + local;
      if (DT == 0) {
        float acc = static_cast<const float*>(a.x[(c + 1) % R])[i];
        for (int k = 2; k <= R; k++) acc = __fadd_rn(acc, static_cast<const float*>(a.x[(c + k) % R])[i]);
        if (a.write_all) {
          for (int r = 0; r < R; r++) static_cast<float*>(a.y[r])[i] = acc;
        } else {
          static_cast<float*>(a.y[c])[local] = acc;
        }
      } else {
        unsigned short acc = static_cast<const unsigned short*>(a.x[(c + 1) % R])[i];
        for (int k = 2; k <= R; k++) {
          float s = __fadd_rn(__uint_as_float((uint32_t)acc << 16),
                              __uint_as_float((uint32_t) static_cast<const unsigned short*>(a.x[(c + k) % R])[i] << 16));
          acc = __bfloat16_as_ushort(__float2bfloat16_rn(s));
        }
        if (a.write_all) {
          for (int r = 0; r < R; r++) static_cast<unsigned short*>(a.y[r])[i] = acc;
        } else {
          static_cast<unsigned short*>(a.y[c])[local] = acc;
        }
      }
    }
  }
}

// ---- memory-port probe: what one SM can read, or write, when it does nothing else ---------------------------------
// mode 0: every thread streams 16-byte loads (8 in flight) over its share of the buffer and folds them into one word
// that is stored once; mode 1: every thread streams 16-byte stores.  Same tile walk as the copy kernel.
template <int MODE>
__global__ void __launch_bounds__(1024, 1) port_probe_kernel(uint4* buf, unsigned long long nvec, unsigned int* sink) {
  constexpr int U = 8;
  const unsigned long long tile = (unsigned long long)U * 1024, ntiles = nvec / tile;
  uint4 acc = make_uint4(0, 0, 0, 0);
  for (unsigned long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    uint4* p = buf + t * tile + threadIdx.x;
    if (MODE == 0) {
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; u++) v[u] = __ldcs(p + u * 1024);
#pragma unroll
      for (int u = 0; u < U; u++) {
        acc.x ^= v[u].x;
        acc.y ^= v[u].y;
        acc.z ^= v[u].z;
        acc.w ^= v[u].w;
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; u++) p[u * 1024] = make_uint4((unsigned)t, u, threadIdx.x, 0);
    }
  }
  if (MODE == 0 && (acc.x ^ acc.y ^ acc.z ^ acc.w) == 0x9e3779b9u) *sink = 1;   // keeps the loads alive
}

// Self-test: add.rn.bf16x2 against the reference add (binary32 add of the widened operands, rounded to nearest even into
// bf16) for every pair of bf16 bit patterns.  Block a handles all b; counts[0] = value mismatches, counts[1] = pairs where
// both are NaN with different payloads.
__global__ void bf16_add_selftest_kernel(unsigned long long* counts) {
  const uint32_t a = blockIdx.x;
  unsigned long long nb = 0, np = 0;
  for (uint32_t b = threadIdx.x * 2; b < 65536; b += blockDim.x * 2) {
    const uint32_t A = a | (a << 16), B = b | ((b + 1) << 16);
    const uint32_t r = add_bf16x2(A, B), h = add_bf16x2_native(A, B);
    for (int l = 0; l < 2; l++) {
      const uint32_t rr = (r >> (16 * l)) & 0xffffu, hh = (h >> (16 * l)) & 0xffffu;
      if (rr != hh) {
        if ((rr & 0x7fffu) > 0x7f80u && (hh & 0x7fffu) > 0x7f80u) np++;
        else nb++;
      }
    }
  }
  if (nb) atomicAdd(&counts[0], nb);
  if (np) atomicAdd(&counts[1], np);
}

// Does nothing: a graph node that only orders (see build_graph).
__global__ void graph_root_kernel() {}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Every CTA keeps its thread slots for `ns` nanoseconds and then returns.  Bounded by construction:
// the loop only reads the global timer; a second cap on the iteration count guards against a stuck timer.
__global__ void __launch_bounds__(kThreads, 2) occupy_kernel(unsigned long long ns) {
  const unsigned long long t0 = global_ns();
  for (unsigned it = 0; it < (1u << 26); it++) {
    if (global_ns() - t0 >= ns) break;
    __nanosleep(256);
  }
}

}  // namespace

// Launch shapes (measured on B200, 256 MiB operands).  SUM: 1024 threads x 4 vectors per operand in flight give 116 GB/s
// per SM under a small budget (the mixed read/write ceiling of one SM's memory port is ~123 GB/s) and reach 6.1 TB/s
// (0.93 of the measured HBM peak) from 64 CTAs on; with 128 CTAs and more, 512 threads x 4 are a little faster
// (6.35 against 6.1-6.2 TB/s).  Copy: 1024 threads x 8 vectors below 128 CTAs (5.5 TB/s at 64 CTAs); from 128 CTAs on
// 512 x 4: on 256 MiB operands the two are equal there, but the four times smaller tile (32 KiB) balances the few-MB
// chunks of a ring step over the grid (gradient bucket, whole GPU: 0.201 against 0.213 ms per step).
static bool wide_grid(int ctas) { return ctas >= 128; }
static bool wide_copy_grid(int ctas) { return ctas >= 128; }
static bool whole_gpu(int ctas) { return ctas >= kAllSms; }   // a CTA per tile, see kMoveShapes

// Host side of the flattened view (same split as the device helper; tile = 4 x threads vectors for the sum, 8 x 1024 or
// 4 x 512 for the copy: the shapes launch_sum / launch_copy pick for `ctas`).
static void fill_flat(Flat* f, int nseg, unsigned long long tile_v, const unsigned* head, const unsigned long long* nvec,
                      const unsigned long long* nscalar) {
  unsigned long long t = 0, sc = 0;
  f->tpre[0] = 0;
  f->spre[0] = 0;
  for (int k = 0; k < nseg; k++) {
    f->head[k] = head[k];
    f->nvec[k] = nvec[k];
    t += (nvec[k] + tile_v - 1) / tile_v;
    sc += nscalar[k];
    f->tpre[k + 1] = t;
    f->spre[k + 1] = sc;
  }
}

void prepare_sum_batch(SumBatch* b, int ctas) {
  const int E = b->dtype == 0 ? 4 : 2, VE = 16 / E;
  const unsigned long long tile_v = 4ull * (wide_grid(ctas) ? 512 : 1024);
  unsigned head[kMaxSegs];
  unsigned long long nvec[kMaxSegs], nscalar[kMaxSegs];
  for (int k = 0; k < b->nseg; k++) {
    const SumSeg& s = b->seg[k];
    const unsigned ma = (unsigned)((uintptr_t)s.inbox & 15), mb = (unsigned)((uintptr_t)s.local & 15), mo = (unsigned)((uintptr_t)s.out & 15);
    split_segment(s.n, ma, ma == mb && mb == mo, E, VE, &head[k], &nvec[k], &nscalar[k]);
  }
  fill_flat(&b->flat, b->nseg, tile_v, head, nvec, nscalar);
}

void prepare_copy_batch(CopyBatch* b, int ctas) {
  const unsigned long long tile_v = wide_copy_grid(ctas) ? 4ull * 512 : 8ull * 1024;
  unsigned head[kMaxSegs];
  unsigned long long nvec[kMaxSegs], nscalar[kMaxSegs];
  for (int k = 0; k < b->nseg; k++) {
    const CopySeg& s = b->seg[k];
    const unsigned ms = (unsigned)((uintptr_t)s.src & 15), md = (unsigned)((uintptr_t)s.dst & 15);
    split_segment(s.bytes, ms, ms == md, 1, 16, &head[k], &nvec[k], &nscalar[k]);
  }
  fill_flat(&b->flat, b->nseg, tile_v, head, nvec, nscalar);
}

// Which chain kernel serves a batch.  The compiled forms need one operand count for the whole launch (the usual case: R) and one
// destination (below 128 CTAs chain_pipe_kernel for 2 to 8 operands and chain_pipe2_kernel for 9 to 16, from 128 on chain_fan_kernel for 2 to
// 8) or as many as operands (chain_fan_kernel, 2 to 8).  chain_pipe_kernel against chain_kernel, measured on
// B200 (8 operands, 25 MiB each, bf16): 163 against 111 GB/s per SM with 8 CTAs, 158 / 107 with 16, 138 / 99 with 32,
// 113 / 89 with 48, 88 / 80 with 64, 59 / 58 with 96; from 128 CTAs on chain_fan_kernel with one destination (64 MiB per rank 94 us,
// 6.4 TB/s).  Variants with the same
// or more bytes in flight (P = 2 with 640 threads, P = 4 with 384, P = 4 and 6 with 256) end at the same 159-163 GB/s per
// SM with 8 CTAs: that is the SM's memory port at 8 reads : 1 write, no longer the bytes in flight.
struct ChainVariant {
  const void* fn;
  int threads;
  int tile;      // vectors of a tile
};
template <int DT, int NOPS, int P, int THREADS>
static ChainVariant pipe_of() {
  return {reinterpret_cast<const void*>(&chain_pipe_kernel<DT, NOPS, P, THREADS>), THREADS, THREADS};
}
template <int DT, int NOPS, int P, int THREADS>
static ChainVariant pipe2_of() {
  return {reinterpret_cast<const void*>(&chain_pipe2_kernel<DT, NOPS, P, THREADS>), THREADS, THREADS};
}
template <int DT, int NOPS, int U, int THREADS>
static ChainVariant fan_of() {
  return {reinterpret_cast<const void*>(&chain_fan_kernel<DT, NOPS, NOPS, U, THREADS>), THREADS, U * THREADS};
}
template <int DT, int NOPS, int U, int THREADS>
static ChainVariant wide_of() {
  return {reinterpret_cast<const void*>(&chain_fan_kernel<DT, NOPS, 1, U, THREADS>), THREADS, U * THREADS};
}
template <int DT>
static ChainVariant chain_pipe_variant(int nops) {
  // P x NOPS vectors per thread: 16 to 24, i.e. 128 to 192 KiB per SM with 512 threads
  switch (nops) {
    case 2: return pipe_of<DT, 2, 8, 512>();
    case 3: return pipe_of<DT, 3, 6, 512>();
    case 4: return pipe_of<DT, 4, 5, 512>();
    case 5: return pipe_of<DT, 5, 4, 512>();
    case 6: return pipe_of<DT, 6, 3, 512>();
    case 7: return pipe_of<DT, 7, 3, 512>();
    case 8: return pipe_of<DT, 8, 3, 512>();
    case 9: return pipe2_of<DT, 9, 4, 512>();
    case 10: return pipe2_of<DT, 10, 4, 512>();
    case 11: return pipe2_of<DT, 11, 4, 512>();
    case 12: return pipe2_of<DT, 12, 4, 512>();
    case 13: return pipe2_of<DT, 13, 3, 512>();
    case 14: return pipe2_of<DT, 14, 3, 512>();
    case 15: return pipe2_of<DT, 15, 3, 512>();
    case 16: return pipe2_of<DT, 16, 3, 512>();
    default: return {nullptr, 0, 0};
  }
}
template <int DT>
static ChainVariant chain_wide_variant(int nops) {
  // One destination, whole-GPU grids.  The mix is read heavy and takes 60 to 80 KiB of loads in flight per SM; what chain_kernel
  // lost with few operands was the look-up per tile (R = 2, 256 MiB per rank: 152 us, now 126).
  switch (nops) {
    case 2: return wide_of<DT, 2, 4, 512>();
    case 3: return wide_of<DT, 3, 2, 768>();
    case 4: return wide_of<DT, 4, 2, 640>();
    case 5: return wide_of<DT, 5, 2, 448>();
    case 6: return wide_of<DT, 6, 2, 384>();
    case 7: return wide_of<DT, 7, 1, 640>();
    case 8: return wide_of<DT, 8, 1, 640>();
    default: return {nullptr, 0, 0};
  }
}
template <int DT>
static ChainVariant chain_fan_variant(int nops, int ctas) {
  // Whole-GPU grids: 42 to 50 KiB of loads in flight per SM.  More of them make it slower (the reads then come in longer bursts
  // between the writes): 8 operands of 64 MiB to 8 destinations 5.85 TB/s with 128 KiB, 6.02 with 64, 6.26 with 48, 6.11 with 40; 4
  // and 4 5.90 with 64, 6.13 with 48; 2 and 2 of 256 MiB 5.85 with 64, 6.27 with 48.
  if (wide_grid(ctas)) {
    switch (nops) {
      case 2: return fan_of<DT, 2, 4, 384>();
      case 3: return fan_of<DT, 3, 2, 448>();
      case 4: return fan_of<DT, 4, 2, 384>();
      case 5: return fan_of<DT, 5, 2, 320>();
      case 6: return fan_of<DT, 6, 1, 448>();
      case 7: return fan_of<DT, 7, 1, 416>();
      case 8: return fan_of<DT, 8, 1, 384>();
      default: return {nullptr, 0, 0};
    }
  }
  // Few CTAs serve short messages only: U x NOPS loads per thread, 8 to 16
  switch (nops) {
    case 2: return fan_of<DT, 2, 4, 512>();
    case 3: return fan_of<DT, 3, 4, 512>();
    case 4: return fan_of<DT, 4, 2, 512>();
    case 5: return fan_of<DT, 5, 2, 512>();
    case 6: return fan_of<DT, 6, 2, 512>();
    case 7: return fan_of<DT, 7, 2, 512>();
    case 8: return fan_of<DT, 8, 2, 512>();
    default: return {nullptr, 0, 0};
  }
}
// The whole GPU, a CTA per tile (see kMoveShapes; the walk above stays between 128 CTAs and all SMs).  Us, 64 MiB per rank bf16 (32 for 3 and 6), walk / CTA
// per tile: sums that store for every rank R = 2 (128 MiB) 89 / 80.2, 4 86 / 80.5, 8 171 / 163.8; one destination R = 8 94 / 88.1, 3 24 / 20.7.  Tiles of
// 128 to 512 vectors are within 3 %, but for 2 and 3 operands with one destination, which want two vectors per thread (R = 2, 128 MiB 59.4, 67.0 with one).
// 9 to 16 operands, against chain_kernel: every rank R = 9 bf16 32 MiB 99.6 / 95.2, 16 167.9 / 165.7; reduce-scatter + all-gather R = 9 fp32 32 MiB 114 / 103,
// 4 MiB 17.6 / 15.2, R = 16 bf16 0.28 MiB 14.4 / 12.3.  Beside a loop of 8192^3 GEMMs the walk (140 CTAs) is the gentler one for long sums: all-reduce that
// stores for every rank, R = 8 256 MiB 996 us a call and 770 lost to the GEMMs, 1210 and 254 with the walk; 40 MiB 176 and 74, 192 and 56.
template <int DT, int N>
static ChainVariant chain_tile_variant(int nops, bool fan) {
  if constexpr (N > 16) return {nullptr, 0, 0};
  else if (nops != N) return chain_tile_variant<DT, N + 1>(nops, fan);
  else return fan ? fan_of<DT, N, N <= 3 ? 2 : 1, 256>() : wide_of<DT, N, N <= 3 ? 2 : 1, 256>();
}
// A whole-GPU sum with driver copies of another piece beside it: one CTA per SM that walks the tiles, as between 128 CTAs and all SMs.  A CTA per tile
// takes every slot that comes free and the copies wait.  Us of an all-reduce on the copy route, 148 SUM CTAs, bf16, a CTA per tile / the walk from the second
// piece on: R = 8 40 MiB in 4 pieces 164.6 / 157.9, 1 GiB in 8 3945 / 3858; R = 4 64 MiB 128.0 / 125.1; R = 2 128 MiB 144.5 / 121.0; staged, R = 8 40 MiB 250.8 / 244.1,
// R = 2 128 MiB 174.9 / 165.1.  Nine operands and more have no compiled walk, and chain_kernel's tables cost more than the crowding (R = 16, 256 MiB 2070 /
// 2084).
static bool chain_walks(const ChainBatch& b) { return b.walk && b.nseg > 0 && b.seg[0].nops <= 8; }
static ChainVariant chain_variant(const ChainBatch& b, int ctas) {
  ChainVariant plain{b.dtype == 0 ? reinterpret_cast<const void*>(&chain_kernel<0, 1024>) : reinterpret_cast<const void*>(&chain_kernel<1, 1024>), 1024, 1024};
  if (b.nseg <= 0) return plain;
  const int nops = b.seg[0].nops, ndst = b.seg[0].ndst;
  for (int k = 1; k < b.nseg; k++)
    if (b.seg[k].nops != nops || b.seg[k].ndst != ndst) return plain;
  ChainVariant v = plain;
  if (whole_gpu(ctas) && !chain_walks(b) && (ndst == 1 || ndst == nops)) v = b.dtype == 0 ? chain_tile_variant<0, 2>(nops, ndst != 1) : chain_tile_variant<1, 2>(nops, ndst != 1);
  else if (ndst == 1 && !wide_grid(ctas)) v = b.dtype == 0 ? chain_pipe_variant<0>(nops) : chain_pipe_variant<1>(nops);
  else if (ndst == 1) v = b.dtype == 0 ? chain_wide_variant<0>(nops) : chain_wide_variant<1>(nops);
  else if (ndst == nops) v = b.dtype == 0 ? chain_fan_variant<0>(nops, ctas) : chain_fan_variant<1>(nops, ctas);
  return v.fn ? v : plain;
}

void prepare_chain_batch(ChainBatch* b, int ctas) {
  const int E = b->dtype == 0 ? 4 : 2, VE = 16 / E;
  const unsigned long long tile_v = (unsigned long long)chain_variant(*b, ctas).tile;
  unsigned head[kMaxSegs];
  unsigned long long nvec[kMaxSegs], nscalar[kMaxSegs];
  for (int k = 0; k < b->nseg; k++) {
    const ChainSeg& s = b->seg[k];
    const unsigned phase = (unsigned)((uintptr_t)b->ptr[s.first_ptr] & 15);
    bool same = true;
    for (int q = 1; q < s.nops + s.ndst; q++) same = same && ((unsigned)((uintptr_t)b->ptr[s.first_ptr + q] & 15) == phase);
    split_segment(s.n, phase, same, E, VE, &head[k], &nvec[k], &nscalar[k]);
    // Start the body of a long segment on a 128-byte line where all operands have one together: a warp's 512 bytes then touch four
    // lines of each operand, not five (40 MiB per rank over 8 ranks in ragged chunks: 406 -> 351 us with the loads of an element-wise
    // item in flight together).
    const unsigned line = (unsigned)((uintptr_t)b->ptr[s.first_ptr] & 127);
    for (int q = 1; q < s.nops; q++) same = same && ((unsigned)((uintptr_t)b->ptr[s.first_ptr + q] & 127) == line);
    if (same && nvec[k] >= 4096 && line % E == 0) {
      head[k] = ((128 - line) & 127) / E;
      nvec[k] = (s.n - head[k]) / VE;
      nscalar[k] = s.n - nvec[k] * VE;
    }
  }
  fill_flat(&b->flat, b->nseg, tile_v, head, nvec, nscalar);
}

template <int DT, int R>
static const void* store_all_from(int r, bool split) {
  if constexpr (R > kMaxStoreAllRanks) return nullptr;
  else if (r != R) return store_all_from<DT, R + 1>(r, split);
  else return split ? reinterpret_cast<const void*>(&store_all_kernel<DT, R, 512, true>) : reinterpret_cast<const void*>(&store_all_kernel<DT, R, 512, false>);
}
static const void* store_all_of(int R, int dtype, bool split) { return dtype == 0 ? store_all_from<0, 2>(R, split) : store_all_from<1, 2>(R, split); }
const void* store_all_entry(int R, int dtype, int ctas, unsigned long long count, StoreAllArgs* a, int* grid, int* threads) {
  const void* fn = store_all_of(R, dtype, ctas < R);
  if (!fn || count > (1ull << 28)) return nullptr;   // 32-bit byte offsets
  a->count = (unsigned)count;
  a->q = (unsigned)((count + R - 1) / R);
  const unsigned vecs = a->q / (dtype == 0 ? 4 : 8);
  a->groups = a->parts = 1;
  if (ctas < R) {   // fewer CTAs than chunks: a CTA's warps are split between chunks
    while ((int)a->groups * ctas < R) a->groups *= 2;
    if (a->groups > 16) return nullptr;
    *grid = (R + (int)a->groups - 1) / (int)a->groups;
  } else {   // no more CTAs than have a round of vectors each
    a->parts = std::max(1u, std::min((unsigned)(ctas / R), (vecs + 511) / 512));
    *grid = R * (int)a->parts;
  }
  *threads = 512;
  if (wide_grid(ctas) && vecs > a->parts * 512u) return nullptr;   // from a second round on chain_fan_kernel's shapes are the better ones
  // CTAs that the chunks do not divide among themselves stay idle: fine while latency decides, not when the stores do
  if (*grid < ctas && vecs > a->parts * (1024u / a->groups)) return nullptr;
  return fn;
}

bool add_chain_seg(ChainBatch* b, const void* const* ops, int nops, void* const* dsts, int ndst, unsigned long long n) {
  if (b->nseg == kMaxSegs || b->nptr + nops + ndst > kMaxChainPtrs) return false;
  ChainSeg& s = b->seg[b->nseg++];
  s = ChainSeg{n, b->nptr, nops, ndst, 0};
  for (int q = 0; q < nops; q++) b->ptr[b->nptr++] = const_cast<void*>(ops[q]);
  for (int d = 0; d < ndst; d++) b->ptr[b->nptr++] = dsts[d];
  return true;
}

cudaError_t launch_in_order(const void* fn, int grid, int threads, void* args, cudaStream_t stream, int priority) {
  cudaStreamCaptureStatus capture;
  const cudaError_t e = cudaStreamIsCapturing(stream, &capture);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = stream;
  cfg.attrs = attr;
  if (capture == cudaStreamCaptureStatusNone) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (priority) {
    attr[cfg.numAttrs].id = cudaLaunchAttributePriority;
    attr[cfg.numAttrs++].val.priority = priority;
  }
  void* params[1] = {args};
  return cudaLaunchKernelExC(&cfg, fn, params);
}

cudaError_t launch_chain(const ChainBatch& batch, int ctas, cudaStream_t stream) {
  if (batch.nseg <= 0) return cudaSuccess;
  ChainBatch b = batch;
  prepare_chain_batch(&b, ctas);
  int threads = 0, grid = 0;
  const void* fn = chain_kernel_entry(b, ctas, &threads, &grid);
  return launch_in_order(fn, grid, threads, &b, stream);
}

void prepare_fan_batch(FanBatch* b, int ctas) {
  const unsigned long long tile_v = wide_copy_grid(ctas) ? 4ull * 512 : 8ull * 1024;
  unsigned head[kMaxSegs];
  unsigned long long nvec[kMaxSegs], nscalar[kMaxSegs];
  for (int k = 0; k < b->nseg; k++) {
    const FanSeg& s = b->seg[k];
    const unsigned ms = (unsigned)((uintptr_t)s.src & 15);
    bool same = true;
    for (int d = 0; d < s.ndst; d++) same = same && ((unsigned)((uintptr_t)b->dst[s.first_dst + d] & 15) == ms);
    split_segment(s.bytes, ms, same, 1, 16, &head[k], &nvec[k], &nscalar[k]);
  }
  fill_flat(&b->flat, b->nseg, tile_v, head, nvec, nscalar);
}

bool add_move_seg(MoveBatch* b, const void* src, void* const* dsts, int ndst, unsigned long long bytes) {
  if (b->nseg == MoveBatch::kSegs || b->ndst_total + ndst > MoveBatch::kDsts) return false;
  MoveSeg& s = b->seg[b->nseg++];
  s.src = src;
  s.bytes = bytes;
  s.first_dst = b->ndst_total;
  s.ndst = ndst;
  for (int d = 0; d < ndst; d++) b->dst[b->ndst_total++] = dsts[d];
  return true;
}

// Launch shape: a thread keeps up to u vectors.  Under a CTA budget 8 x 1024 (the bytes in flight per SM decide).  On the whole GPU a CTA
// per tile, in small CTAs: they drift apart, so that some load while others store; CTAs that walk many tiles, one per SM, go through the two
// phases together.  TB/s at 8 MiB per segment, 2 x 256 or (stored four times and more) 1 x 256 with a CTA per tile against the best
// walk: copies 6.81 / 6.25 (4 x 704), 1:3 6.37 / 5.94 (4 x 384), 1:7 6.46 / 5.80 (1 x 448); 512 KiB 5.60 / 5.32, 4.29 / 3.22, 5.08 / 4.41.  Larger and smaller
// tiles (1 to 16 x 128 to 512) are within 3 % of these.  Between 128 CTAs and all SMs the walk stays, in its own shapes: it wants little in
// flight per SM, the less the more often a vector is stored, 44 KiB for copies (4 x 704 6.2 TB/s, 8 x 1024 4.2), 7 for one read stored 7 times.
// (Who comes between: steps of the ring whose bytes are in L2, see kRingWalkFrom, and budgets of 128 to 147, a caller's own choice.)
struct MoveShape {
  int u, threads;
};
static constexpr MoveShape kMoveShapes[] = {{8, 1024}, {4, 704}, {2, 704}, {4, 384}, {2, 384}, {1, 448}, {2, 256}, {1, 256}};
static int move_shape(const MoveBatch& b, int ctas) {
  if (!wide_copy_grid(ctas)) return 0;
  const int per_seg = b.nseg > 0 ? (b.ndst_total + b.nseg / 2) / b.nseg : 1;   // stores per load, rounded
  if (whole_gpu(ctas)) return per_seg <= 3 ? 6 : 7;
  for (int k = 0; k < b.nseg; k++)   // out of phase every vector is loaded twice: the shape for copies
    if (((uintptr_t)b.seg[k].src ^ (uintptr_t)b.dst[b.seg[k].first_dst]) & 15) return 1;
  return per_seg <= 1 ? 1 : per_seg == 2 ? 2 : per_seg == 3 ? 3 : per_seg <= 5 ? 4 : 5;
}
template <class Batch>
static const void* move_entry(int shape) {
  switch (shape) {
    case 1: return reinterpret_cast<const void*>(&move_kernel<4, 704, Batch>);
    case 2: return reinterpret_cast<const void*>(&move_kernel<2, 704, Batch>);
    case 3: return reinterpret_cast<const void*>(&move_kernel<4, 384, Batch>);
    case 4: return reinterpret_cast<const void*>(&move_kernel<2, 384, Batch>);
    case 5: return reinterpret_cast<const void*>(&move_kernel<1, 448, Batch>);
    case 6: return reinterpret_cast<const void*>(&move_kernel<2, 256, Batch>);
    case 7: return reinterpret_cast<const void*>(&move_kernel<1, 256, Batch>);
    default: return reinterpret_cast<const void*>(&move_kernel<8, 1024, Batch>);
  }
}

void prepare_move_batch(MoveBatch* b, int ctas) {
  const MoveShape shape = kMoveShapes[move_shape(*b, ctas)];
  const unsigned threads = (unsigned)shape.threads, most_u = (unsigned)shape.u;
  b->spre[0] = 0;
  for (int k = 0; k < b->nseg; k++) {
    MoveSeg& s = b->seg[k];
    const unsigned long long at = (uintptr_t)s.src & 15;
    // destination on a 128-byte line if the segment is long (a warp's 512 bytes then touch four lines, not five), on a vector if not
    const unsigned long long grid = s.bytes >= kMoveLineBytes ? 128 : 16;
    unsigned long long head = (grid - ((uintptr_t)b->dst[s.first_dst] & (grid - 1))) & (grid - 1);
    const unsigned long long sh = (at + head) & 15;                                // where a vector starts inside the source's
    if (head < sh) head += 16;                 // the first aligned vector of the source must not start in front of it
    const unsigned long long reach = sh ? 32 - sh : 16;   // source bytes from the start of a vector to the end of what it loads
    unsigned long long nvec = 0;
    if (s.bytes >= head + reach) nvec = (s.bytes - head - reach) / 16 + 1;
    else head = 0;
    s.head = (unsigned)head;
    s.nvec = (unsigned)nvec;
    b->spre[k + 1] = b->spre[k] + (unsigned)(s.bytes - nvec * 16);
  }
  // Tiles of a whole-GPU launch: the shape's, one vector per thread where that gives fewer than two per SM.  Of a walk: as large as
  // a thread's registers hold (a tile's loads are in flight together), smaller where that would leave CTAs
  // without a tile or with one more than others.  In units of one vector per thread stored once, a tile costs its stores and ~3 for
  // the loads to come back; the grid runs ceil(tiles / ctas) of them one after another.
  double best = 0;
  if (whole_gpu(ctas)) {
    unsigned long long tiles = 0;
    for (int k = 0; k < b->nseg; k++) tiles += (b->seg[k].nvec + most_u * threads - 1) / (most_u * threads);
    b->tile_u = tiles < 2 * kAllSms ? 1 : most_u;
  } else for (unsigned u = most_u; u >= 1; u /= 2) {
    unsigned long long tiles = 0;
    for (int k = 0; k < b->nseg; k++) tiles += (b->seg[k].nvec + u * threads - 1) / (u * threads);
    const double per_tile = 3.0 + (double)u * b->ndst_total / (b->nseg > 0 ? b->nseg : 1);
    const double cost = (double)((tiles + ctas - 1) / ctas) * per_tile;
    if (u == most_u || cost < best) {
      best = cost;
      b->tile_u = u;
    }
  }
  b->tpre[0] = 0;
  for (int k = 0; k < b->nseg; k++) b->tpre[k + 1] = b->tpre[k] + (b->seg[k].nvec + b->tile_u * threads - 1) / (b->tile_u * threads);
}

bool shrink_move_batch(const MoveBatch& b, MoveBatchSmall* o) {
  if (b.nseg > MoveBatchSmall::kSegs || b.ndst_total > MoveBatchSmall::kDsts) return false;
  o->nseg = b.nseg;
  o->ndst_total = b.ndst_total;
  o->tile_u = b.tile_u;
  std::copy(b.seg, b.seg + b.nseg, o->seg);
  std::copy(b.dst, b.dst + b.ndst_total, o->dst);
  std::copy(b.tpre, b.tpre + b.nseg + 1, o->tpre);
  std::copy(b.spre, b.spre + b.nseg + 1, o->spre);
  return true;
}

const void* move_kernel_entry(const MoveBatch& b, int ctas, bool small, int* threads, int* grid) {
  const int shape = move_shape(b, ctas);
  *threads = kMoveShapes[shape].threads;
  *grid = whole_gpu(ctas) ? (int)std::max(b.tpre[b.nseg], std::min(8u * (unsigned)ctas, (b.spre[b.nseg] + *threads - 1) / *threads)) : ctas;
  return small ? move_entry<MoveBatchSmall>(shape) : move_entry<MoveBatch>(shape);
}

cudaError_t launch_moves(MoveBatch* b, int ctas, cudaStream_t stream) {
  if (b->nseg <= 0) return cudaSuccess;
  prepare_move_batch(b, ctas);
  MoveBatchSmall small;
  const bool fits = shrink_move_batch(*b, &small);
  int threads = 0, grid = 0;
  const void* fn = move_kernel_entry(*b, ctas, fits, &threads, &grid);
  return launch_in_order(fn, grid, threads, fits ? static_cast<void*>(&small) : static_cast<void*>(b), stream);
}

cudaError_t launch_move(const void* src, void* dst, unsigned long long bytes, int ctas, cudaStream_t stream) {
  // One long copy in phase leaves nothing to choose: copy_kernel's plain tile walk is 0.5 to 0.8 % faster there (waves of 42.8 MB
  // messages on 40 CTAs, three communicators at once: 98.7 -> 98.0 us).  Below 16 MB its tiles leave CTAs without work.
  if (!whole_gpu(ctas) && bytes >= (16ull << 20) && (((uintptr_t)src ^ (uintptr_t)dst) & 15) == 0 && ((uintptr_t)dst & 127) == 0) {
    CopyBatch cb;
    cb.nseg = 1;
    cb.pad = 0;
    cb.seg[0] = CopySeg{src, dst, bytes};
    return launch_copy(cb, ctas, stream);
  }
  MoveBatch b;
  b.nseg = b.ndst_total = 0;
  for (unsigned long long at = 0; at < bytes; at += kMaxMoveSegBytes) {
    void* d = static_cast<char*>(dst) + at;
    add_move_seg(&b, static_cast<const char*>(src) + at, &d, 1, std::min(kMaxMoveSegBytes, bytes - at));
  }
  return launch_moves(&b, ctas, stream);
}

cudaError_t launch_sum(const SumBatch& batch, int ctas, cudaStream_t stream) {
  if (batch.nseg <= 0) return cudaSuccess;
  SumBatch b = batch;
  prepare_sum_batch(&b, ctas);
  if (b.dtype == 0) {
    if (wide_grid(ctas)) sum2_kernel<0, 4, 512><<<ctas, 512, 0, stream>>>(b);
    else sum2_kernel<0, 4, 1024><<<ctas, 1024, 0, stream>>>(b);
  } else {
    if (wide_grid(ctas)) sum2_kernel<1, 4, 512><<<ctas, 512, 0, stream>>>(b);
    else sum2_kernel<1, 4, 1024><<<ctas, 1024, 0, stream>>>(b);
  }
  return cudaGetLastError();
}

cudaError_t launch_copy(const CopyBatch& batch, int ctas, cudaStream_t stream) {
  if (batch.nseg <= 0) return cudaSuccess;
  CopyBatch b = batch;
  prepare_copy_batch(&b, ctas);
  if (wide_copy_grid(ctas)) copy_kernel<4, 512><<<ctas, 512, 0, stream>>>(b);
  else copy_kernel<8, 1024><<<ctas, 1024, 0, stream>>>(b);
  return cudaGetLastError();
}

cudaError_t launch_port_probe(int mode, void* buf, unsigned long long bytes, int ctas, unsigned int* sink, cudaStream_t stream) {
  if (mode == 0) port_probe_kernel<0><<<ctas, 1024, 0, stream>>>(static_cast<uint4*>(buf), bytes / 16, sink);
  else port_probe_kernel<1><<<ctas, 1024, 0, stream>>>(static_cast<uint4*>(buf), bytes / 16, sink);
  return cudaGetLastError();
}

cudaError_t launch_onepass(const OnePassArgs& args, int ctas, cudaStream_t stream) {
  if (args.count == 0) return cudaSuccess;
  // more threads under a CTA budget: the loads in flight per SM set the rate there
  if (wide_grid(ctas)) {
    if (args.dtype == 0) onepass_kernel<0, 512><<<ctas, 512, 0, stream>>>(args);
    else onepass_kernel<1, 512><<<ctas, 512, 0, stream>>>(args);
  } else {
    if (args.dtype == 0) onepass_kernel<0, 1024><<<ctas, 1024, 0, stream>>>(args);
    else onepass_kernel<1, 1024><<<ctas, 1024, 0, stream>>>(args);
  }
  return cudaGetLastError();
}

const void* sum_kernel_entry(int dtype, int ctas, int* threads) {
  *threads = wide_grid(ctas) ? 512 : 1024;
  if (dtype == 0)
    return wide_grid(ctas) ? reinterpret_cast<const void*>(&sum2_kernel<0, 4, 512>) : reinterpret_cast<const void*>(&sum2_kernel<0, 4, 1024>);
  return wide_grid(ctas) ? reinterpret_cast<const void*>(&sum2_kernel<1, 4, 512>) : reinterpret_cast<const void*>(&sum2_kernel<1, 4, 1024>);
}
const void* copy_kernel_entry(int ctas, int* threads) {
  *threads = wide_copy_grid(ctas) ? 512 : 1024;
  return wide_copy_grid(ctas) ? reinterpret_cast<const void*>(&copy_kernel<4, 512>) : reinterpret_cast<const void*>(&copy_kernel<8, 1024>);
}
cudaError_t launch_bf16_add_selftest(unsigned long long* counts, cudaStream_t stream) {
  bf16_add_selftest_kernel<<<65536, 256, 0, stream>>>(counts);
  return cudaGetLastError();
}
const void* chain_kernel_entry(const ChainBatch& batch, int ctas, int* threads, int* grid) {
  const ChainVariant v = chain_variant(batch, ctas);
  const Flat& f = batch.flat;
  *threads = v.threads;
  *grid = whole_gpu(ctas) && !chain_walks(batch) ? (int)std::max(f.tpre[batch.nseg], std::min(8ull * (unsigned)ctas, (f.spre[batch.nseg] + v.threads - 1) / v.threads)) : ctas;
  return v.fn;
}
const void* graph_root_kernel_entry() { return reinterpret_cast<const void*>(&graph_root_kernel); }
// The kernels that the rules of this file may pick for a call, asked from the rules themselves: one CTA count on each side of every line between
// launch shapes (wide_grid, whole_gpu), every operand count, one destination or one per operand.
static std::vector<const void*> dispatched_kernels() {
  std::vector<const void*> fns = {reinterpret_cast<const void*>(&occupy_kernel),           reinterpret_cast<const void*>(&graph_root_kernel),
                                  reinterpret_cast<const void*>(&onepass_kernel<0, 512>),  reinterpret_cast<const void*>(&onepass_kernel<1, 512>),
                                  reinterpret_cast<const void*>(&onepass_kernel<0, 1024>), reinterpret_cast<const void*>(&onepass_kernel<1, 1024>)};
  for (int ctas : {1, kAllSms - 1, kAllSms}) {
    int threads = 0;
    fns.push_back(copy_kernel_entry(ctas, &threads));
    for (int dtype = 0; dtype < 2; dtype++) {
      fns.push_back(sum_kernel_entry(dtype, ctas, &threads));
      for (int nops = 2; nops <= kMaxChainSrcs + 1; nops++)
        for (int ndst : {1, nops}) {
          ChainBatch b;
          b.nseg = 1;
          b.dtype = dtype;
          b.seg[0] = ChainSeg{0, 0, nops, ndst, 0};
          fns.push_back(chain_variant(b, ctas).fn);
        }
    }
  }
  for (int R = 2; R <= kMaxStoreAllRanks; R++)
    for (int form = 0; form < 4; form++) fns.push_back(store_all_of(R, form & 1, form & 2));
  for (int shape = 0; shape < (int)(sizeof(kMoveShapes) / sizeof(kMoveShapes[0])); shape++)
    for (const void* f : {move_entry<MoveBatch>(shape), move_entry<MoveBatchSmall>(shape)}) fns.push_back(f);
  std::sort(fns.begin(), fns.end());
  fns.erase(std::unique(fns.begin(), fns.end()), fns.end());
  return fns;
}
// Forces the module that holds these kernels to be loaded now.  Loading a kernel on first launch can synchronise the
// device; that must never happen while a stream is parked in a hand-over that only the launching thread can finish.
cudaError_t preload_kernels() {
  for (const void* f : dispatched_kernels()) {
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
bool is_preloaded(const void* fn) {
  const std::vector<const void*> fns = dispatched_kernels();
  return std::find(fns.begin(), fns.end(), fn) != fns.end();
}

cudaError_t launch_occupy_all_sms(unsigned long long ns, int num_sms, cudaStream_t stream, int* ctas_out) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, occupy_kernel, kThreads, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int ctas = per_sm * num_sms;
  if (ctas_out) *ctas_out = ctas;
  occupy_kernel<<<ctas, kThreads, 0, stream>>>(ns);
  return cudaGetLastError();
}

}  // namespace hoccl
