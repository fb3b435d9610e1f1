// Stage 3c: fused deinterleave + scatter (Section 3.5).  Each staged record
// holds a neuron's gate, up and transposed-down rows back to back; the kernel
// writes the three rows to the slot the delta step assigned, in the three
// projection-specific resident buffers.  Pure 16-byte coalesced copies.
//
// k_pull_rows does the same straight from the pinned record store, records addressed by neuron ID:
// transfer and placement in one kernel, for several layers a launch.
#include <cuda_bf16.h>

#include <algorithm>

#include "np_device.cuh"
#include "np_internal.h"

namespace npi {
using namespace npd;

constexpr int kScatterThreads = 256;

__global__ void __launch_bounds__(kScatterThreads) k_deinterleave_scatter(
    const uint4* __restrict__ src, const int32_t* __restrict__ slots, const int32_t* __restrict__ count_ptr, int first,
    int max_rows, uint4* __restrict__ gate, uint4* __restrict__ up, uint4* __restrict__ downT,
    int row_chunks /* D*2/16 */, int C, int32_t* status, int check) {
  int n = *count_ptr - first;  // rows of this chunk
  if (n > max_rows) n = max_rows;
  for (int r = blockIdx.x; r < n; r += gridDim.x) {
    const int slot = slots[first + r];
    if (check && (slot < 0 || slot >= C)) {
      if (threadIdx.x == 0) atomicOr(status, kStatBadSlot);
      continue;
    }
    const uint4* s = src + (size_t)r * 3 * row_chunks;
    const size_t dst = (size_t)slot * row_chunks;
    // up to 4 loads in flight per thread per projection
    for (int c0 = threadIdx.x; c0 < row_chunks; c0 += kScatterThreads * 4) {
      uint4 g[4], u[4], d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j * kScatterThreads;
        if (c < row_chunks) {
          g[j] = ldg_stream(s + c);
          u[j] = ldg_stream(s + row_chunks + c);
          d[j] = ldg_stream(s + 2 * row_chunks + c);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j * kScatterThreads;
        if (c < row_chunks) {
          gate[dst + c] = g[j];
          up[dst + c] = u[j];
          downT[dst + c] = d[j];
        }
      }
    }
  }
}

// 8-bit records (int8 gate | up | downT rows, three fp32 scales, padding): the rows are
// dequantised on their way into the resident buffers, w = bf16_rn(float(q) * scale), so only
// half the bytes of a bf16 record cross PCIe or sit in staging.  A thread turns 16 bytes of one
// row into 32 bytes of bf16.
__device__ __forceinline__ uint32_t dequant2(uint32_t q4, int shift, float scale) {
  const float a = (float)(int)(signed char)((q4 >> shift) & 0xffu) * scale;
  const float b = (float)(int)(signed char)((q4 >> (shift + 8)) & 0xffu) * scale;
  const uint32_t lo = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a));
  const uint32_t hi = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b));
  return lo | (hi << 16);
}

template <bool kFromStore>
__global__ void __launch_bounds__(kScatterThreads) k_dequant_scatter(
    const unsigned char* __restrict__ src, const int32_t* __restrict__ ids, const int32_t* __restrict__ slots,
    const int32_t* __restrict__ count_ptr, int first, int max_rows, uint4* __restrict__ gate,
    uint4* __restrict__ up, uint4* __restrict__ downT, int D, size_t rec_bytes, int M, int C, int dst_pitch,
    int32_t* status, int check) {
  // count_ptr == NULL: exactly max_rows rows (the dense prefix is dequantised once, at start-up)
  int n = count_ptr ? *count_ptr - first : max_rows;
  if (n > max_rows) n = max_rows;
  const int q_chunks = D >> 4;  // 16-byte pieces of one int8 row
  for (int r = blockIdx.x; r < n; r += gridDim.x) {
    const int slot = slots[first + r];
    size_t rec;
    if (kFromStore) {
      const int id = ids[first + r];
      if (check && (id < 0 || id >= M)) {
        if (threadIdx.x == 0) atomicOr(status, kStatBadNeuron);
        continue;
      }
      rec = (size_t)id;
    } else {
      rec = (size_t)r;
    }
    if (check && (slot < 0 || slot >= C)) {
      if (threadIdx.x == 0) atomicOr(status, kStatBadSlot);
      continue;
    }
    const unsigned char* s = src + rec * rec_bytes;
    const float* scales = reinterpret_cast<const float*>(s + (size_t)3 * D);
    const size_t dst = (size_t)slot * dst_pitch;  // uint4 units from one slot's row to the next
    // up to four loads of a thread are issued before the first is converted
    for (int c0 = threadIdx.x; c0 < 3 * q_chunks; c0 += kScatterThreads * 4) {
      uint4 q[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j * kScatterThreads;
        if (c < 3 * q_chunks) {
          const int p = c / q_chunks, cc = c - p * q_chunks;
          q[j] = ldg_stream(s + (size_t)p * D + (size_t)cc * 16);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j * kScatterThreads;
        if (c < 3 * q_chunks) {
          const int p = c / q_chunks, cc = c - p * q_chunks;
          const float scale = __ldg(scales + p);
          uint4 lo, hi;
          lo.x = dequant2(q[j].x, 0, scale);
          lo.y = dequant2(q[j].x, 16, scale);
          lo.z = dequant2(q[j].y, 0, scale);
          lo.w = dequant2(q[j].y, 16, scale);
          hi.x = dequant2(q[j].z, 0, scale);
          hi.y = dequant2(q[j].z, 16, scale);
          hi.z = dequant2(q[j].w, 0, scale);
          hi.w = dequant2(q[j].w, 16, scale);
          uint4* row = p == 0 ? gate : (p == 1 ? up : downT);
          row[dst + 2 * cc] = lo;
          row[dst + 2 * cc + 1] = hi;
        }
      }
    }
  }
}

cudaError_t launch_scatter(const Dims& d, const void* src, const int32_t* slots, const int32_t* count_ptr, int first,
                           int max_rows, void* gate_l, void* up_l, void* downT_l, int32_t* status, int check,
                           cudaStream_t s, int sm_count) {
  if (max_rows <= 0) return cudaSuccess;
  const int blocks = std::min(max_rows, sm_count * 8);
  if (d.rec_int8)
    k_dequant_scatter<false><<<blocks, kScatterThreads, 0, s>>>(
        static_cast<const unsigned char*>(src), nullptr, slots, count_ptr, first, max_rows, static_cast<uint4*>(gate_l),
        static_cast<uint4*>(up_l), static_cast<uint4*>(downT_l), d.D, d.rec_bytes, d.M, d.C, (d.D >> 4) * 2, status, check);
  else
    k_deinterleave_scatter<<<blocks, kScatterThreads, 0, s>>>(
        static_cast<const uint4*>(src), slots, count_ptr, first, max_rows, static_cast<uint4*>(gate_l),
        static_cast<uint4*>(up_l), static_cast<uint4*>(downT_l), d.D * 2 / 16, d.C, status, check);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Transfer and placement in one: the incoming rows of several layers, read by neuron ID from the pinned store.
//
// What bounds it is the host link, and in front of that the reads in flight: 128-byte lines, 512 bytes a warp instruction,
// about 4.5 us each.  The 147 MB of incoming rows of a 7B-shaped step, one context on its own (one contiguous copy of the
// same bytes: 55.1 GB/s; the store's size, 8.7 GB or an eighth of that, makes no difference):
//
//   two SMs of 1024 threads, six loads per lane, pieces of 384 units in rounds   44.4 GB/s    301 steps/s
//   the same with eight loads per lane                                           49.6         332
//   three SMs, six / eight loads                                                 46.9 / 50.0  316 / 337
//   four / six SMs, six loads                                                    48.1 / 49.0  324 / 330
//   two SMs, six loads, pieces of one round                                      50.1         337
//
// A piece of a record is what one round of a warp's loads takes, all pieces of a record alike and whole 128-byte lines from
// the line the record starts in, so that no round is nearly empty; the next piece's layer and list entry are read while
// the rows are on their way.  More in flight than this gives nothing alone, and where two contexts pull at a time (51 GB/s
// together) it only delays what else crosses the link: seven or eight loads per lane cost three stacks of 20 layers that
// select and step in turn 2 to 3 %.  Every further SM is one less for the resident MLP kernels, which are launched
// narrower while rows are on their way (kPullReserve; two pulls fit).  Packing the records with the host's cores and
// copying the packed parts gives 40 to 47 GB/s depending on the host (304 to 317 steps/s; the packing reads and writes
// every byte in host memory beside the copy's own reads), and a copy call per record 4.8.  A kernel on all SMs, small
// enough to fit beside the resident blocks, was no faster, and the resident kernels lost 7 % by giving up the registers.
//
// 8-bit records: a lane's dequantising adds to the trip of its loads.  Two SMs read 27 GB/s (361 steps/s), four 47 (606;
// eight loads per lane 597): they take four (pull_blocks on where they do not).
// ---------------------------------------------------------------------------------------
constexpr int kPullThreads = 1024;
constexpr int kPullLoads = 6;  // loads a lane has in flight

struct PullArgs {
  const char* store;        // device alias of the pinned store
  const int32_t* ids;       // [L][C]
  const int32_t* slots;     // [L][C]
  const int32_t* counters;  // [L][NP_N_COUNTERS]
  char* gate;               // first sparse layer of each row buffer
  char* up;
  char* downT;
  int32_t* status;
  size_t rec_bytes;
  int l_begin, l_end, dense, D, M, C, Lp, check;
  int pieces, piece;  // pieces of a record, 16-byte units of a piece
};

template <bool kInt8>
__global__ void __launch_bounds__(kPullThreads) k_pull_rows(PullArgs a) {
  constexpr int U = kPullLoads;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (kPullThreads / 32);
  const int row_units = kInt8 ? a.D >> 4 : a.D >> 3;             // 16-byte units of a source row
  const int pieces = a.pieces;
  // pieces of a layer: the lanes hold 32 layers' counts, read at once (a launch without rows is as long as these reads)
  int base = a.l_begin, held = 0;
  auto read_counts = [&] {
    held = base + lane < a.l_end ? min(max(a.counters[(size_t)(base + lane) * NP_N_COUNTERS + NP_CNT_DELTA], 0), a.C) * pieces : 0;
  };
  auto pieces_of = [&](int l) {
    if (l - base >= 32) {
      base = l;
      read_counts();
    }
    return __shfl_sync(0xffffffffu, held, l - base);
  };
  read_counts();
  // this warp's pieces are every nw-th of all layers' in a row: i counts from the start of layer l
  int l = a.l_begin, total = pieces_of(l), id = 0, slot = 0;
  int i = blockIdx.x * (kPullThreads / 32) + (threadIdx.x >> 5);
  auto settle = [&] {  // to the layer that holds piece i, and its list entry
    while (i >= total) {
      i -= total;
      if (++l == a.l_end) return;
      total = pieces_of(l);
    }
    id = a.ids[(size_t)l * a.C + i / pieces];
    slot = a.slots[(size_t)l * a.C + i / pieces];
  };
  settle();
  while (l < a.l_end) {
    const int p = i % pieces;
    if (a.check && (id < 0 || id >= a.M || slot < 0 || slot >= a.C)) {
      if (lane == 0) atomicOr(a.status, id < 0 || id >= a.M ? kStatBadNeuron : kStatBadSlot);
      i += nw;
      settle();
      continue;
    }
    const char* rec = a.store + ((size_t)(l % a.Lp) * a.M + id) * a.rec_bytes;
    const size_t dst = ((size_t)(l - a.dense) * a.C + slot) * a.D * 2;
    const int mis = (int)((reinterpret_cast<uintptr_t>(rec) >> 4) & 7);  // units between the line's start and the record
    const int end = min((p + 1) * a.piece - mis, 3 * row_units);
    const int v0 = p * a.piece - mis + lane;
    float sc[3];
    if (kInt8) {
      const uint4 s4 = ldg_stream(rec + (size_t)3 * a.D);
      sc[0] = __uint_as_float(s4.x), sc[1] = __uint_as_float(s4.y), sc[2] = __uint_as_float(s4.z);
    }
    uint4 x[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int v = v0 + 32 * j;
      if (v >= 0 && v < end) x[j] = ldg_stream(rec + (size_t)v * 16);
    }
    i += nw;
    settle();  // the next piece's list entry comes while the rows are on their way
#pragma unroll
    for (int j = 0; j < U; ++j) {
      int v = v0 + 32 * j;
      if (v >= 0 && v < end) {
        char* row = a.gate;
        float scale = kInt8 ? sc[0] : 0.f;
        if (v >= row_units) {
          v -= row_units;
          row = a.up;
          if (kInt8) scale = sc[1];
          if (v >= row_units) {
            v -= row_units;
            row = a.downT;
            if (kInt8) scale = sc[2];
          }
        }
        if (kInt8) {
          uint4* o = reinterpret_cast<uint4*>(row + dst) + 2 * v;
          o[0] = make_uint4(dequant2(x[j].x, 0, scale), dequant2(x[j].x, 16, scale), dequant2(x[j].y, 0, scale), dequant2(x[j].y, 16, scale));
          o[1] = make_uint4(dequant2(x[j].z, 0, scale), dequant2(x[j].z, 16, scale), dequant2(x[j].w, 0, scale), dequant2(x[j].w, 16, scale));
        } else {
          reinterpret_cast<uint4*>(row + dst)[v] = x[j];
        }
      }
    }
  }
}

cudaError_t launch_pull(const Dims& d, const Tables& t, const char* store_dev, void* gate, void* up, void* downT, int l_begin,
                        int l_end, int blocks, int check, cudaStream_t s) {
  PullArgs a;
  a.store = store_dev;
  a.ids = t.delta_ids;
  a.slots = t.delta_slots;
  a.counters = t.counters;
  a.gate = static_cast<char*>(gate);
  a.up = static_cast<char*>(up);
  a.downT = static_cast<char*>(downT);
  a.status = t.status;
  a.rec_bytes = d.rec_bytes;
  a.l_begin = l_begin;
  a.l_end = l_end;
  a.dense = d.dense;
  a.D = d.D;
  a.M = d.M;
  a.C = d.C;
  a.Lp = d.Lp;
  a.check = check;
  // whole lines, and no more units than one round of a warp's loads; a record starts up to `mis` units into its first line
  const int units = 3 * d.D / (d.rec_int8 ? 16 : 8), most = 32 * kPullLoads;
  const int mis = d.rec_bytes % 128 == 0 ? (int)((reinterpret_cast<uintptr_t>(store_dev) >> 4) & 7) : 7;
  a.pieces = (units + mis + most - 1) / most;
  a.piece = ((units + mis + a.pieces - 1) / a.pieces + 7) & ~7;
  if (d.rec_int8) k_pull_rows<true><<<blocks, kPullThreads, 0, s>>>(a);
  else k_pull_rows<false><<<blocks, kPullThreads, 0, s>>>(a);
  return cudaGetLastError();
}

// Start-up only: the 8-bit records of one dense layer, read from the pinned store, become whole
// bf16 records [M][gate | up | downT][D] in the dense buffer (slot = neuron, rows three times
// as far apart as in a slot buffer).
cudaError_t launch_dequant_dense_layer(const Dims& d, const void* store_l, const int32_t* identity, void* dense_l,
                                       int32_t* status, cudaStream_t s, int sm_count) {
  const size_t row_bytes = (size_t)d.D * 2;
  char* base = static_cast<char*>(dense_l);
  const int blocks = std::min(d.M, sm_count * 8);
  k_dequant_scatter<true><<<blocks, kScatterThreads, 0, s>>>(
      static_cast<const unsigned char*>(store_l), identity, identity, nullptr, 0, d.M,
      reinterpret_cast<uint4*>(base), reinterpret_cast<uint4*>(base + row_bytes),
      reinterpret_cast<uint4*>(base + 2 * row_bytes), d.D, d.rec_bytes, d.M, d.M, 3 * (d.D >> 4) * 2, status, 1);
  return cudaGetLastError();
}

}  // namespace npi
