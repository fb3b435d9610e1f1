// Stage 4 over a run of consecutive layers in ONE resident kernel for two to sixteen sequences:
//
//   x_{l+1}[b] = x_l[b] + sum_{i in act_l} silu(gate_l[s_i].n_l[b]) * (up_l[s_i].n_l[b]) * downT_l[s_i],
//   n_l[b] = x_l[b] / sqrt(mean(x_l[b]^2) + 1e-6)
//
// (Section 3.4 through the slot map; every sequence computes over the union of the active rows.)
//
// A layer of the 7B shape is 58 MB at sixteen sequences (8.8 us of HBM time) and 34 MB at two (5.3 us), so the two
// kernels per layer this replaces (23.4 us per layer at sixteen, 17.4 at two) were bound by what lies between them:
// launches, x re-read and re-split by every block, dot products and outputs reduced through global memory, a ring that
// starts empty in every kernel.  Here the rows stream through one ring across phases and layers, and what is left on
// the path from x_l to x_{l+1} is the tensor-core work, one exchange per sixteen rows that hides behind the next
// sixteen, and one hand-over of x per layer.
//
// Partition.  The grid is Q column slices x R row groups (Q: slices of at most kMaxNk K blocks of 16; R = SMs / Q).
// Block (r, q) owns the rows of row group r and slice q of the columns: the K range of its dot products is the column
// range of its outputs, so of x it only ever needs slice q.
//
//   up     Eight consumer warps.  A tile is 8 gate and 8 up pieces (the 16 rows of an MMA, mma.sync m16n8k16, bf16 x
//          bf16 -> fp32).  The K blocks are dealt to the warps, and a warp keeps the B operand of its K blocks -- x as
//          three truncated bf16 terms, exact to 2^-24 -- in registers for the whole layer: x costs no shared memory,
//          which all goes to rows in flight, and an A fragment read from shared memory serves all sequences (a tile read
//          once per group of eight sequences kept shared memory busy for two thirds of the MMAs' time).
//   chunk  Sixteen rows (two up tiles, one down tile).  Two groups of exchange warps take the chunks in turn: they add
//          the consumers' partial dot products, trade them with the other slices of the row group through (value, stamp)
//          words in global memory (one store, polled by the readers: no fence, no counter), form the activations and
//          leave them as A fragments of the down phase.  The consumers are in the next chunk meanwhile.
//   down   The activations' three terms are the rows of the MMA (NSG = 2: one MMA per term over 16 sequences; NSG = 1:
//          terms 0 and 1 of 8 sequences in one MMA, term 2 in a second), 16 records its K, 8 output columns its N.  A
//          warp keeps the accumulators of its columns over the layer and then adds them to x with 16-byte reductions.
//
// x lives in global memory in tiles of 8 columns, [D / 8][8 NSG sequences][8] fp32, so that both the fragment loads and
// the reductions of a warp are contiguous.  It is updated in place: block (r, q) may add once all R blocks of slice q
// have read x_l, and may read x_{l+1} once all R have added.  Two counters per slice say so (they only grow; the host
// tracks their value); a warp of its own waits on them.
//
// Every wait is bounded (np_pipe.cuh); once one has run out the block records kStatTimeout and skips all later waits except
// those for its ring (np_ring.h).
#include <algorithm>

#include "np_device.cuh"
#include "np_internal.h"
#include "np_pipe.cuh"

namespace npi {
namespace chain_batch {
using namespace npd;

constexpr int kWarps = 8;             // consumer warps
constexpr int kThreads = 512;         // warps 8..15: producer, synchroniser, four exchange warps, two spare (a warpgroup
                                      // changes its register share as a whole)
constexpr int kConsumerRegs = 168;    // 256 x 168 + 256 x 88 = 512 x 128, what the block is launched with
constexpr int kOtherRegs = 88;
constexpr int kProducer = 8, kSync = 9, kExch0 = 10;
constexpr int kExchGroups = 2, kExchWarps = 2;  // groups that take the chunks in turn, warps per group
constexpr int kChunk = 16;            // rows of a chunk
constexpr int kMaxNk = 80;            // most K blocks of a slice (1280 columns)
constexpr int kMaxSlots = 16;         // ring slots
constexpr int kMaxLayers = 64;        // layers per launch
constexpr int kMaxQ = 8;
constexpr int kPad = 16;              // bytes between pieces in shared memory: ldmatrix rows fall into different banks
constexpr int kCntStride = 32;        // one 128-byte line per counter
// 64-bit words a block publishes per chunk: pairs (gate, up) per row and sequence, then the sums of squares, a copy per
// exchange warp: a warp only ever polls words of its counterpart in the other blocks, so a word is not written again
// before the warps that poll it are done with it (a warp publishes a chunk after it has finished its previous one).
constexpr int kAreaWords = 2 * kChunk * 16 + kExchWarps * 16;

struct KArgs {
  const unsigned char* gate;  // layer 0 of each buffer (dense layers: the three rows of layer 0's first record)
  const unsigned char* up;
  const unsigned char* downT;
  const int32_t* slots;       // active_slots [L][C] (dense layers: not read, row i is record i)
  const int32_t* counters;    // [L][NP_N_COUNTERS]
  float* x;                   // [D / 8][8 NSG][8]
  unsigned int* cnt;          // [2][kMaxQ][kCntStride]: blocks that have read x_l; warps that have added MLP_l
  unsigned long long* xch;    // [grid][2 kExchGroups][kAreaWords]
  int32_t* status;
  size_t layer_bytes, row_pitch;
  unsigned int read_base, add_base, seq_base;
  int l_begin, l_end, B, D, C, check, Q, dense_rows;
  int ng;                     // ring slots
  int max_rows;               // most rows a block can have in a layer
  uint32_t slot_bytes;
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// fp32 -> three truncated bf16 terms (v = t0 + t1 + t2 up to 2^-24 |v|), as fp32 bit patterns with a zero low half
__device__ __forceinline__ void split3(float v, uint32_t (&t)[3]) {
  t[0] = __float_as_uint(v) & 0xffff0000u;
  const float r1 = v - __uint_as_float(t[0]);
  t[1] = __float_as_uint(r1) & 0xffff0000u;
  const float r2 = r1 - __uint_as_float(t[1]);
  t[2] = __float_as_uint(r2) & 0xffff0000u;
}
__device__ __forceinline__ uint32_t pack2(uint32_t first, uint32_t second) { return __byte_perm(first, second, 0x7632); }

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ unsigned long long stamped(float v, unsigned int stamp) {
  return ((unsigned long long)stamp << 32) | (unsigned long long)__float_as_uint(v);
}
__device__ __forceinline__ void ld_relaxed_v2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void st_relaxed_v2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// A warp's wait, by all lanes or by lane 0.  The latter parts the warp and brings it together again, some 300 cycles where the phase
// is long complete, so the barriers on the way of x are waited for by all lanes (sixteen sequences of 1024 columns 83 us per 12 layers,
// 90 with lane 0's waits; two of the 7B shape 319 per 32 and 337).  The waits inside the up phase's loop are lane 0's: by all lanes
// they cost the widest rows more than they give the others (13B shape, eight sequences, 581 us per 40 layers against 560).  (The polls of
// the exchange's words still end lane by lane.)
__device__ __forceinline__ void all_wait(uint64_t* bar, uint32_t parity, volatile int* ok, int32_t* status) {
  npp::wait_or_flag(bar, parity, ok, status);
  __syncwarp();
}
__device__ __forceinline__ void warp_wait(uint64_t* bar, uint32_t parity, volatile int* ok, int32_t* status, int lane) {
  if (lane == 0) npp::wait_or_flag(bar, parity, ok, status);
  __syncwarp();
}
// Whether the phase of that parity is complete, without waiting.  The consumers ask early and look at the answer when they
// need it: asked at the point of use, the answer's way back is idle time of the tensor pipe (a warp per scheduler computes
// while the other one waits, and both wait for the same tile).
__device__ __forceinline__ uint32_t mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(npp::smem_addr(bar)), "r"(parity)
      : "memory");
  return ok;
}
// one lane: until the counter at `p` has reached `target` (modulo 2^32)
__device__ __forceinline__ void wait_count(const unsigned int* p, unsigned int target, volatile int* ok, int32_t* status) {
  if (!*ok) return;
  for (uint32_t spin = 0; spin < npp::kSpinLimit; ++spin) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if ((int)(v - target) >= 0) return;
  }
  *ok = 0;
  atomicOr(status, npp::kStatTimeout);
}

// Exchange of one chunk by the kExchWarps * 32 threads of a group (t: this thread's index): sums of this block's partial
// dot products, the other slices' sums, activations.  A thread's pairs (row, sequence) all belong to one sequence.
template <int NSG>
__device__ __forceinline__ void exchange_chunk(const KArgs& a, const float4* part, const float* ssq_part, uint16_t* hs, int t, int rows,
                                               int q, int r, unsigned int area, unsigned int stamp, uint64_t* part_empty, int lane,
                                               volatile int* ok) {
  constexpr int NS = 8 * NSG, NT = kExchWarps * 32;
  constexpr int NPAIR = kChunk * NS / NT;  // pairs of a thread
  constexpr int PB = 2, PQ = 4;            // pairs and slices whose words are polled together
  const int seq = t & (NS - 1), row0 = t / NS;
  constexpr int row_step = NT / NS;
  const bool live = seq < a.B;
  float g[NPAIR], u[NPAIR], ss = 0.f;
  const float2* p2 = reinterpret_cast<const float2*>(part);
#pragma unroll
  for (int k = 0; k < kWarps; ++k) ss += ssq_part[k * 16 + seq];
#pragma unroll
  for (int i = 0; i < NPAIR; ++i) {
    const int row = row0 + i * row_step;
    g[i] = u[i] = 0.f;
    const float2* p = p2 + ((size_t)((row >> 3) * NSG + (seq >> 3)) * kWarps * 32 + (row & 7) * 4 + ((seq & 7) >> 1)) * 2 + (seq & 1);
#pragma unroll
    for (int k = 0; k < kWarps; ++k) {
      const float2 v = p[k * 64];
      g[i] += v.x;
      u[i] += v.y;
    }
  }
  const int Q = a.Q;
  const int ss_word = 2 * kChunk * 16 + (t >> 5) * 16;  // this warp's copy of the sums of squares
  if (Q > 1) {
    unsigned long long* mine = a.xch + ((size_t)blockIdx.x * (2 * kExchGroups) + area) * kAreaWords;
#pragma unroll
    for (int i = 0; i < NPAIR; ++i)
      if (live && row0 + i * row_step < rows) st_relaxed_v2(mine + 2 * (t + i * NT), stamped(g[i], stamp), stamped(u[i], stamp));
    if (lane < NS) st_relaxed(mine + ss_word + lane, stamped(ss, stamp));
  }
  __syncwarp();
  if (lane == 0) npp::mbar_arrive(part_empty);  // the partial sums have been read
  if (Q > 1) {
    const unsigned long long* base = a.xch + ((size_t)r * Q * (2 * kExchGroups) + area) * kAreaWords;
    constexpr size_t peer = (size_t)(2 * kExchGroups) * kAreaWords;
    const unsigned long long mark = (unsigned long long)stamp << 32;
    const float own_ss = ss;
#pragma unroll
    for (int i0 = 0; i0 < NPAIR; i0 += PB) {
      float gs[PB], us[PB];  // sums in slice order, the same in every block of the row group
#pragma unroll
      for (int i = 0; i < PB; ++i) gs[i] = us[i] = 0.f;
      if (i0 == 0) ss = 0.f;
      for (int qb = 0; qb < Q; qb += PQ) {
        unsigned long long wg[PB][PQ], wu[PB][PQ], ws[PQ];
        bool done = !*ok;
        uint32_t spin = 0;
        do {  // every load of the round is issued before any is looked at
          unsigned int bad = 0;
#pragma unroll
          for (int k = 0; k < PQ; ++k) {
            const int qq = qb + k;
#pragma unroll
            for (int i = 0; i < PB; ++i) {
              wg[i][k] = wu[i][k] = mark;
              if (qq < Q && qq != q && live && row0 + (i0 + i) * row_step < rows)
                ld_relaxed_v2(base + qq * peer + 2 * (t + (i0 + i) * NT), wg[i][k], wu[i][k]);
            }
            ws[k] = mark;
            if (i0 == 0 && qq < Q && qq != q && live) ws[k] = ld_relaxed(base + qq * peer + ss_word + seq);
          }
#pragma unroll
          for (int k = 0; k < PQ; ++k) {
#pragma unroll
            for (int i = 0; i < PB; ++i) bad |= ((unsigned int)(wg[i][k] >> 32) ^ stamp) | ((unsigned int)(wu[i][k] >> 32) ^ stamp);
            bad |= (unsigned int)(ws[k] >> 32) ^ stamp;
          }
          done = done || bad == 0;
        } while (!done && ++spin < npp::kSpinLimit);
        if (!done && *ok) {
          *ok = 0;
          atomicOr(a.status, npp::kStatTimeout);
        }
#pragma unroll
        for (int k = 0; k < PQ; ++k) {
          const bool own = qb + k == q;  // slices past Q add the zero under the mark
#pragma unroll
          for (int i = 0; i < PB; ++i) {
            gs[i] += own ? g[i0 + i] : __uint_as_float((unsigned int)wg[i][k]);
            us[i] += own ? u[i0 + i] : __uint_as_float((unsigned int)wu[i][k]);
          }
          if (i0 == 0) ss += own ? own_ss : __uint_as_float((unsigned int)ws[k]);
        }
      }
#pragma unroll
      for (int i = 0; i < PB; ++i) {
        g[i0 + i] = gs[i];
        u[i0 + i] = us[i];
      }
    }
  }
  const float inv = rsqrtf(ss / (float)a.D + kRmsEps);
#pragma unroll
  for (int i = 0; i < NPAIR; ++i) {
    const int row = row0 + i * row_step;
    const float gs = g[i] * inv, us = u[i] * inv;
    const float h = live && row < rows ? gs / (1.f + __expf(-gs)) * us : 0.f;  // rows and sequences that pad a tile: zero
    uint32_t tr[3];
    split3(h, tr);
    // A fragment of m16n8k16: element (m, k) is half k & 1 of register (m >> 3) + 2 (k >> 3) of lane 4 (m & 7) + (k & 7) / 2
    const int fl = (seq & 7) * 4 + ((row & 7) >> 1), half = row & 1, rk = 2 * (row >> 3);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      // NSG = 2: tile e holds term e of 16 sequences; NSG = 1: tile 0 holds terms 0 | 1 of 8 sequences, tile 1 term 2
      const int tile = NSG == 2 ? e : e >> 1, reg = (NSG == 2 ? seq >> 3 : e & 1) + rk;
      hs[((tile * 32 + fl) * 4 + reg) * 2 + half] = (uint16_t)(tr[e] >> 16);
    }
  }
}

// acc += h . down of one chunk over PN pairs of 8-column tiles: pairs pair0, pair0 + kWarps, ... of the slice.  `bp`: the
// lane's ldmatrix address of the tile's first pair.  Pairs past the slice's end are computed and never looked at.
template <int NSG, int PN>
__device__ __forceinline__ void down_mma(float (&acc)[2 * PN][4], const uint16_t* hc, uint32_t bp, int pair0, int nk, int lane) {
  constexpr int HT = NSG == 2 ? 3 : 2;
  uint32_t hf[HT][4];
#pragma unroll
  for (int e = 0; e < HT; ++e) {
    const uint4 v = *reinterpret_cast<const uint4*>(hc + ((size_t)e * 32 + lane) * 8);
    hf[e][0] = v.x;
    hf[e][1] = NSG == 1 && e == 1 ? 0u : v.y;
    hf[e][2] = v.z;
    hf[e][3] = NSG == 1 && e == 1 ? 0u : v.w;
  }
#pragma unroll
  for (int p0 = 0; p0 < PN; p0 += 4) {
    uint32_t bf[4][4];
#pragma unroll
    for (int p = 0; p < 4 && p0 + p < PN; ++p) {
      const int pair = pair0 + (p0 + p) * kWarps;
      ldmatrix_x4_trans(bf[p], bp + (pair < nk ? (uint32_t)pair * 32u : 0u));
    }
#pragma unroll
    for (int e = 0; e < HT; ++e)
#pragma unroll
      for (int p = 0; p < 4 && p0 + p < PN; ++p) {
        mma_bf16(acc[2 * (p0 + p)], hf[e], bf[p][0], bf[p][1]);
        mma_bf16(acc[2 * (p0 + p) + 1], hf[e], bf[p][2], bf[p][3]);
      }
  }
}

// x += acc for the same pairs
template <int NSG, int PN>
__device__ __forceinline__ void down_reds(const float (&acc)[2 * PN][4], float* xs, int pair0, int nk, int B, int lane) {
  constexpr int NS = 8 * NSG;
  const int g8 = lane >> 2, t4 = lane & 3;
  const bool odd = t4 & 1;
#pragma unroll
  for (int p = 0; p < PN; ++p) {
    const int pair = pair0 + p * kWarps;
    if (pair >= nk) break;
    float* tile = xs + (size_t)pair * 2 * NS * 8;
    if (NSG == 2) {
      // rows g8 / g8 + 8 = sequences; even lanes end up with four columns of sequence g8, odd lanes of 8 + g8
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float* v = acc[2 * p + j];
        const float ra = __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[2], 1), rb = __shfl_xor_sync(0xffffffffu, odd ? v[1] : v[3], 1);
        const int seq = odd ? 8 + g8 : g8;
        float* dst = tile + (size_t)j * NS * 8 + seq * 8 + (t4 >> 1) * 4;
        const float o0 = odd ? ra : v[0], o1 = odd ? rb : v[1], o2 = odd ? v[2] : ra, o3 = odd ? v[3] : rb;
        if (seq < B) red_add_v4(dst, o0, o1, o2, o3);
      }
    } else {
      // rows g8 and g8 + 8 belong to one sequence; even lanes take the pair's first tile, odd lanes its second
      const float a0 = acc[2 * p][0] + acc[2 * p][2], a1 = acc[2 * p][1] + acc[2 * p][3];
      const float b0 = acc[2 * p + 1][0] + acc[2 * p + 1][2], b1 = acc[2 * p + 1][1] + acc[2 * p + 1][3];
      const float ra = __shfl_xor_sync(0xffffffffu, odd ? a0 : b0, 1), rb = __shfl_xor_sync(0xffffffffu, odd ? a1 : b1, 1);
      float* dst = tile + (size_t)(odd ? 1 : 0) * NS * 8 + g8 * 8 + (t4 >> 1) * 4;
      const float o0 = odd ? ra : a0, o1 = odd ? rb : a1, o2 = odd ? b0 : ra, o3 = odd ? b1 : rb;
      if (g8 < B) red_add_v4(dst, o0, o1, o2, o3);
    }
  }
}

// NSG: groups of eight sequences.  NP: pairs of 8-column output tiles per warp (= 16-wide K blocks per eight warps).
template <int NSG, int NP>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_batch(KArgs a) {
  extern __shared__ __align__(128) unsigned char csm[];
  __shared__ __align__(8) uint64_t full_bar[kMaxSlots], empty_bar[kMaxSlots];
  __shared__ __align__(8) uint64_t part_full[2], part_empty[2];
  __shared__ __align__(8) uint64_t x_ready, x_read, may_add;
  __shared__ float ssq_part[kWarps * 16];
  __shared__ int s_ok[2];  // no wait has run out; the ring was given up
  __shared__ unsigned int s_act[kExchGroups * kExchWarps];  // chunks each exchange warp has finished, ever growing
  __shared__ int lay_rb[kMaxLayers], lay_n[kMaxLayers], lay_pre[kMaxLayers + 1];

  constexpr int NS = 8 * NSG;
  constexpr int kPart = 2 * NSG * kWarps * 32;          // float4 of a chunk's partial dot products
  constexpr int HT = NSG == 2 ? 3 : 2;                  // A tiles per chunk
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int Q = a.Q, R = gridDim.x / Q;
  const int q = blockIdx.x % Q, r = blockIdx.x / Q;
  const int nkt = a.D >> 4;                             // K blocks of a whole row; slice q takes [k0, k0 + nk) of them
  const int k0 = nkt * q / Q, nk = nkt * (q + 1) / Q - k0;
  const uint32_t piece_bytes = (uint32_t)nk * 32u, pstride = piece_bytes + kPad;
  const int nl = a.l_end - a.l_begin;
  const int max_chunks = (a.max_rows + kChunk - 1) / kChunk;
  // dynamic shared memory: ring | partial dot products, two chunks | activations of a layer | slots
  float4* part = reinterpret_cast<float4*>(csm + (size_t)a.ng * a.slot_bytes);           // [2][2 tiles][NSG][8 warps][32]
  uint16_t* hs = reinterpret_cast<uint16_t*>(part + 2 * kPart);                // [max_chunks][HT][32][4] words
  uint16_t* slot_cache = hs + (size_t)max_chunks * HT * 256;
  volatile int* ok = s_ok;
  unsigned int* cnt_read = a.cnt + (size_t)q * kCntStride;
  unsigned int* cnt_add = a.cnt + (size_t)(kMaxQ + q) * kCntStride;

  if (tid < nl) {
    int n = a.dense_rows > 0 ? a.dense_rows : a.counters[(size_t)(a.l_begin + tid) * NP_N_COUNTERS + NP_CNT_ACTIVE];
    if (a.check && a.dense_rows == 0 && (n < 0 || n > a.C)) {
      atomicOr(a.status, kStatBadCount);
      n = 0;
    }
    const int rb = (int)(((long long)n * r) / R), re = (int)(((long long)n * (r + 1)) / R);
    lay_rb[tid] = rb;
    lay_n[tid] = min(re - rb, a.max_rows);
  }
  if (tid == 0) {
    for (int s = 0; s < a.ng; ++s) {
      npp::mbar_init(&full_bar[s], 1);
      npp::mbar_init(&empty_bar[s], kWarps);
    }
    for (int i = 0; i < 2; ++i) {
      npp::mbar_init(&part_full[i], kWarps);
      npp::mbar_init(&part_empty[i], kExchWarps);
    }
    npp::mbar_init(&x_ready, 1);
    npp::mbar_init(&x_read, kWarps);
    npp::mbar_init(&may_add, 1);
    npp::fence_barrier_init();
    s_ok[0] = 1, s_ok[1] = 0;
    for (int i = 0; i < kExchGroups * kExchWarps; ++i) s_act[i] = 0;
  }
  // The tiles are read whole: rows that no copy fills meet zero activations, so what they hold must be finite.
  for (uint32_t i = tid; i < (uint32_t)a.ng * a.slot_bytes / 16; i += kThreads) reinterpret_cast<uint4*>(csm)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (tid == 0) {
    lay_pre[0] = 0;
    for (int i = 0; i < nl; ++i) lay_pre[i + 1] = lay_pre[i] + lay_n[i];
  }
  npp::fence_proxy_async();  // the zeros precede the bulk copies into the same bytes
  __syncthreads();
  if (a.dense_rows == 0) {
    for (int li = 0; li < nl; ++li) {
      for (int i = tid; i < lay_n[li]; i += kThreads) {
        int slot = a.slots[(size_t)(a.l_begin + li) * a.C + lay_rb[li] + i];
        if (a.check && (slot < 0 || slot >= a.C)) {
          atomicOr(a.status, kStatBadSlot);
          slot = 0;
        }
        slot_cache[lay_pre[li] + i] = (uint16_t)slot;
      }
    }
  }
  __syncthreads();

  if (wid >= kWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (wid == kProducer) {
      // ---- producer: gate|up tiles of a layer (8 records), its down tiles (16), the next layer's, in the order of use ----
      int slot = 0;
      uint32_t par = 0;
      const uint64_t pol = npp::policy_evict_first();  // a row is read once per token
      const size_t qoff = (size_t)k0 * 32;
      for (int li = 0; li < nl; ++li) {
        const int nrows = lay_n[li];
        const size_t lbase = (size_t)(a.l_begin + li) * a.layer_bytes + qoff;
        for (int pass = 0; pass < 2; ++pass) {
          const int step = pass == 0 ? 8 : 16;
          for (int r0 = 0; r0 < nrows; r0 += step) {
            const int n = min(step, nrows - r0);
            npp::ring_wait(&empty_bar[slot], par ^ 1u, ok, a.status);
            if (lane == 0) npp::mbar_expect_tx(&full_bar[slot], (uint32_t)(pass == 0 ? 2 * n : n) * piece_bytes);
            __syncwarp();
            const int i = pass == 0 ? (lane & 7) : lane;
            if (lane < 16 && i < n) {
              const int row = r0 + i;
              const size_t rec = a.dense_rows > 0 ? (size_t)(lay_rb[li] + row) : (size_t)slot_cache[lay_pre[li] + row];
              const unsigned char* src = (pass == 0 ? (lane < 8 ? a.gate : a.up) : a.downT) + lbase + rec * a.row_pitch;
              npp::bulk_g2s_stream(csm + (size_t)slot * a.slot_bytes + (size_t)lane * pstride, src, piece_bytes, &full_bar[slot], pol);
            }
            __syncwarp();
            if (++slot == a.ng) {
              slot = 0;
              par ^= 1u;
            }
          }
        }
      }
      uint32_t patience = npp::kSpinLimit;
      if (lane == 0) npp::drain_ring(full_bar, a.ng, slot, par, patience);  // nobody leaves before the copies have landed
    } else if (wid == kSync) {
      // ---- synchroniser: the two counters of the slice ----
      if (lane == 0) {
        for (int li = 0; li < nl; ++li) {
          if (li > 0) wait_count(cnt_add, a.add_base + (unsigned int)li * (unsigned int)(R * kWarps), ok, a.status);
          npp::mbar_arrive(&x_ready);
          npp::wait_or_flag(&x_read, (uint32_t)li & 1u, ok, a.status);
          asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt_read) : "memory");
          wait_count(cnt_read, a.read_base + (unsigned int)(li + 1) * (unsigned int)R, ok, a.status);
          npp::mbar_arrive(&may_add);
        }
      }
    } else if (wid < kExch0 + kExchGroups * kExchWarps) {
      const int e = (wid - kExch0) / kExchWarps, t = ((wid - kExch0) % kExchWarps) * 32 + lane;
      unsigned int nx = 0;  // chunks so far
      for (int li = 0; li < nl; ++li) {
        const int nrows = lay_n[li], nch = (nrows + kChunk - 1) / kChunk;
        for (int c = 0; c < nch; ++c) {
          const unsigned int n = nx + (unsigned int)c;
          if (n % kExchGroups != (unsigned int)e) continue;
          const unsigned int buf = n & 1u, use = n >> 1, turn = n / kExchGroups;
          all_wait(&part_full[buf], use & 1u, ok, a.status);
          const unsigned int area = (unsigned int)e * 2u + (turn & 1u), stamp = a.seq_base + 1u + n;
          const float4* pt = part + (size_t)buf * kPart;
          uint16_t* hc = hs + (size_t)c * HT * 256;
          const int rows = min(kChunk, nrows - c * kChunk);
          exchange_chunk<NSG>(a, pt, ssq_part, hc, t, rows, q, r, area, stamp, &part_empty[buf], lane, ok);
          __syncwarp();
          if (lane == 0) {
            __threadfence_block();
            *const_cast<volatile unsigned int*>(&s_act[wid - kExch0]) = turn + 1u;
          }
        }
        nx += (unsigned int)nch;
      }
    }
    return;
  }

  // =========================== consumer warps ===========================
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsumerRegs));
  const int g8 = lane >> 2, t4 = lane & 3;
  const uint32_t ring = npp::smem_addr(csm);
  const uint32_t up_off = (uint32_t)(lane & 15) * pstride + (uint32_t)(lane >> 4) * 16u;
  // transposed loads: matrices 0 / 1 = records 0-7 / 8-15 of an 8-column tile, 2 / 3 = the same of the next tile
  const uint32_t dn_off = (uint32_t)((lane & 7) + ((lane >> 3) & 1) * 8) * pstride + (uint32_t)(lane >> 4) * 16u;
  float* xs = a.x + (size_t)k0 * 2 * NS * 8;  // this slice's tiles: 2 NS 8 floats per K block
  int slot = 0;
  uint32_t par = 0;
  unsigned int nx = 0;  // chunks so far
  auto next_slot = [&] {
    if (++slot == a.ng) {
      slot = 0;
      par ^= 1u;
    }
  };

  for (int li = 0; li < nl; ++li) {
    const int nrows = lay_n[li], n_up = (nrows + 7) >> 3, nch = (nrows + kChunk - 1) / kChunk;
    // ---- x_l: this warp's K blocks wid, wid + 8, ..., straight into B fragments ----
    uint32_t xb[NP][NSG][3][2];
    {
      all_wait(&x_ready, (uint32_t)li & 1u, ok, a.status);
      float2 lo[NP][NSG], hi[NP][NSG];
      const float* xp = xs + (size_t)g8 * 8 + 2 * t4;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int kb = wid + i * kWarps;
#pragma unroll
        for (int sg = 0; sg < NSG; ++sg) {
          lo[i][sg] = hi[i][sg] = make_float2(0.f, 0.f);
          if (kb < nk) {
            lo[i][sg] = __ldcg(reinterpret_cast<const float2*>(xp + ((size_t)kb * 2 * NS + sg * 8) * 8));
            hi[i][sg] = __ldcg(reinterpret_cast<const float2*>(xp + ((size_t)(kb * 2 + 1) * NS + sg * 8) * 8));
          }
        }
      }
      float ss[NSG];
#pragma unroll
      for (int sg = 0; sg < NSG; ++sg) {
        ss[sg] = 0.f;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const float2 l2 = lo[i][sg], h2 = hi[i][sg];
          ss[sg] += l2.x * l2.x + l2.y * l2.y + h2.x * h2.x + h2.y * h2.y;
          uint32_t s0[3], s1[3], s2[3], s3[3];
          split3(l2.x, s0);
          split3(l2.y, s1);
          split3(h2.x, s2);
          split3(h2.y, s3);
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            xb[i][sg][e][0] = pack2(s0[e], s1[e]);
            xb[i][sg][e][1] = pack2(s2[e], s3[e]);
          }
        }
        ss[sg] += __shfl_xor_sync(0xffffffffu, ss[sg], 1);
        ss[sg] += __shfl_xor_sync(0xffffffffu, ss[sg], 2);
        if (t4 == 0) ssq_part[wid * 16 + sg * 8 + g8] = ss[sg];
      }
      __syncwarp();
      if (lane == 0) npp::mbar_arrive(&x_read);
    }
    // ---- up: partial dot products of the slice, a tile of 8 records at a time ----
    uint32_t rdy = mbar_test(&full_bar[slot], par);
    for (int t = 0; t < n_up; ++t) {
      const unsigned int n = nx + (unsigned int)(t >> 1), buf = n & 1u;
      if (!__all_sync(0xffffffffu, rdy)) {
        if (lane == 0) npp::ring_wait(&full_bar[slot], par, ok, a.status);
        __syncwarp();
      }
      const uint32_t ap = ring + (uint32_t)slot * a.slot_bytes + up_off;
      uint64_t* const done_bar = &empty_bar[slot];
      next_slot();
      rdy = mbar_test(&full_bar[slot], par);  // the next tile's
      const uint32_t room = (t & 1) || n < 2 ? 1u : mbar_test(&part_empty[buf], ((n >> 1) - 1u) & 1u);
      float c[NSG][3][4];
#pragma unroll
      for (int sg = 0; sg < NSG; ++sg)
#pragma unroll
        for (int e = 0; e < 3; ++e) c[sg][e][0] = c[sg][e][1] = c[sg][e][2] = c[sg][e][3] = 0.f;
#pragma unroll
      for (int i0 = 0; i0 < NP; i0 += 4) {
        uint32_t af[4][4];
#pragma unroll
        for (int i = 0; i < 4 && i0 + i < NP; ++i) {
          const int kb = wid + (i0 + i) * kWarps;  // past the slice's end: x is zero, any of the row's bytes do
          ldmatrix_x4(af[i], ap + (kb < nk ? (uint32_t)kb * 32u : 0u));
        }
#pragma unroll
        for (int i = 0; i < 4 && i0 + i < NP; ++i)
#pragma unroll
          for (int e = 0; e < 3; ++e)
#pragma unroll
            for (int sg = 0; sg < NSG; ++sg) mma_bf16(c[sg][e], af[i], xb[i0 + i][sg][e][0], xb[i0 + i][sg][e][1]);
      }
      __syncwarp();
      if (lane == 0) npp::mbar_arrive(done_bar);
      if (!__all_sync(0xffffffffu, room)) warp_wait(&part_empty[buf], ((n >> 1) - 1u) & 1u, ok, a.status, lane);
      // rows g8 (gate of record g8) and g8 + 8 (its up), sequences 8 sg + 2 t4, + 1
#pragma unroll
      for (int sg = 0; sg < NSG; ++sg)
        part[(size_t)buf * kPart + (size_t)(((t & 1) * NSG + sg) * kWarps + wid) * 32 + lane] =
            make_float4(c[sg][0][0] + c[sg][1][0] + c[sg][2][0], c[sg][0][2] + c[sg][1][2] + c[sg][2][2],
                        c[sg][0][1] + c[sg][1][1] + c[sg][2][1], c[sg][0][3] + c[sg][1][3] + c[sg][2][3]);
      if ((t & 1) || t == n_up - 1) {
        __syncwarp();
        if (lane == 0) npp::mbar_arrive(&part_full[buf]);
      }
    }
    // ---- down: y[sequences][columns] += h . down, this warp's 16-column pairs wid, wid + 8, ... ----
    // A chunk is ready when both exchange warps of its group have left its activations and its rows have landed.
    auto acts_there = [&](unsigned int n) {
      const volatile unsigned int* done = &s_act[(n % kExchGroups) * kExchWarps];
      const unsigned int target = n / kExchGroups + 1u;
      bool there = true;
#pragma unroll
      for (int w = 0; w < kExchWarps; ++w) there = there && (int)(done[w] - target) >= 0;  // one may be a chunk ahead
      return there;
    };
    auto chunk_wait = [&](int c, int sl, uint32_t pr) {
      const unsigned int n = nx + (unsigned int)c;
      if (!__all_sync(0xffffffffu, acts_there(n))) {
        bool done = false;  // the same in all lanes
#pragma unroll 1
        for (uint32_t spin = 0; spin < npp::kSpinLimit * 16u && !done; ++spin) done = __all_sync(0xffffffffu, acts_there(n) || !*ok);
        if (!done) {
          *ok = 0;
          atomicOr(a.status, npp::kStatTimeout);
        }
        __syncwarp();
      }
      __threadfence_block();
      if (!__all_sync(0xffffffffu, mbar_test(&full_bar[sl], pr))) {
        npp::ring_wait(&full_bar[sl], pr, ok, a.status);
        __syncwarp();
      }
    };
    {
      float acc[2 * NP][4];
#pragma unroll
      for (int j = 0; j < 2 * NP; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
      for (int c = 0; c < nch; ++c) {
        chunk_wait(c, slot, par);
        down_mma<NSG, NP>(acc, hs + (size_t)c * HT * 256, ring + (uint32_t)slot * a.slot_bytes + dn_off, wid, nk, lane);
        __syncwarp();
        if (lane == 0) npp::mbar_arrive(&empty_bar[slot]);
        next_slot();
      }
      // x += y in place, once every block of the slice has read x_l
      all_wait(&may_add, (uint32_t)li & 1u, ok, a.status);
      if (nrows > 0) down_reds<NSG, NP>(acc, xs, wid, nk, a.B, lane);
    }
    nx += (unsigned int)nch;
    __syncwarp();
    if (lane == 0) {
      __threadfence();  // the warp's adds, then its arrival
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(cnt_add) : "memory");
    }
  }
}

// x as the kernel keeps it, from the stack's bf16 input [B][D]; sequences past B are zero.  A thread per 4 values.
__global__ void k_batch_x_in(const uint16_t* __restrict__ in, float* __restrict__ x, int B, int NS, int D) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // [D / 8][NS][2]
  if (i >= D / 4 * NS) return;
  const int half = i & 1, seq = (i >> 1) % NS, tile = (i >> 1) / NS;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (seq < B) {
    const uint16_t* p = in + (size_t)seq * D + tile * 8 + half * 4;  // the caller's vector: any alignment
    v = make_float4(bf16_lo(p[0]), bf16_lo(p[1]), bf16_lo(p[2]), bf16_lo(p[3]));
  }
  reinterpret_cast<float4*>(x)[i] = v;
}
__global__ void k_batch_x_out(const float* __restrict__ x, float* __restrict__ out, int B, int NS, int D) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // [B][D / 4]
  if (i >= B * (D / 4)) return;
  const int seq = i / (D / 4), c = i % (D / 4);
  reinterpret_cast<float4*>(out)[i] = reinterpret_cast<const float4*>(x)[((size_t)(c >> 1) * NS + seq) * 2 + (c & 1)];
}

namespace {

struct Plan {
  int Q, R, np, ng, max_rows, run_layers;
  uint32_t slot_bytes;
  size_t smem;
};

// `rows`: most rows a layer can have (the capacity, or the rows of a dense layer)
bool make_plan(const Dims& d, int rows, bool dense, int nsg, int sm_count, Plan* p) {
  if (d.D % 16 || d.C > 65535) return false;
  const int nkt = d.D / 16;
  // At least four slices: a block's share of x, and of what it adds to x, shrinks with their number (12 layers' mean at
  // sixteen sequences: 1024 columns and 400 rows 11.1 us with one slice, 9.3 with two, 8.2 with four; 2432 and 619 14.2 with
  // two, 13.2 with four).  No more than the operands need: the exchange polls four slices at a time (4096 columns and 1101
  // rows 16.6 us with four, 23.7 with eight).
  int Q = std::min(4, nkt);
  while (Q <= kMaxQ && (nkt + Q - 1) / Q > kMaxNk) Q *= 2;
  if (Q > kMaxQ || nkt < Q || sm_count < Q) return false;
  const int nk = (nkt + Q - 1) / Q;  // the widest slice
  p->Q = Q;
  p->R = sm_count / Q;
  p->np = (nk + kWarps - 1) / kWarps;
  p->max_rows = (rows + p->R - 1) / p->R;
  const int max_chunks = (p->max_rows + kChunk - 1) / kChunk;
  p->slot_bytes = 16u * (uint32_t)(nk * 32 + kPad);
  const size_t budget = 227 * 1024 - 2560;  // static shared memory of the kernel
  const size_t fixed = (size_t)2 * 2 * nsg * kWarps * 32 * 16 + (size_t)max_chunks * (nsg == 2 ? 3 : 2) * 512 + 256;
  const size_t cache_min = dense ? 0 : 2 * (size_t)p->max_rows * 8;
  if (fixed + cache_min + 3 * (size_t)p->slot_bytes > budget) return false;
  p->ng = (int)std::min<size_t>(kMaxSlots, (budget - fixed - cache_min) / p->slot_bytes);
  if (d.ring_stages >= 2) p->ng = std::max(3, std::min(p->ng, d.ring_stages));
  const size_t left = budget - fixed - (size_t)p->ng * p->slot_bytes;
  p->run_layers = dense ? kMaxLayers : (int)std::max<size_t>(1, std::min<size_t>(kMaxLayers, left / (2 * (size_t)p->max_rows)));
  p->smem = (size_t)p->ng * p->slot_bytes + fixed + (dense ? 0 : 2 * (size_t)p->max_rows * p->run_layers);
  return true;
}

template <int NSG, int NP>
cudaError_t launch_one(const KArgs& ka, size_t sm, int grid, cudaStream_t s) {
  auto kfn = k_mlp_batch<NSG, NP>;
  static std::atomic<uint64_t> done{0};
  cudaError_t e = allow_shared(reinterpret_cast<const void*>(kfn), &done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all blocks co-resident: no wait can starve
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kfn, ka);
}

}  // namespace

bool supported(const Dims& d, int sm_count) {
  Plan p;
  const int nsg = d.Bmax > 8 ? 2 : 1;
  if (d.dense < d.L && !make_plan(d, d.C, false, nsg, sm_count, &p)) return false;
  if (d.dense > 0 && !make_plan(d, d.M, true, nsg, sm_count, &p)) return false;
  return true;
}
size_t cnt_words() { return (size_t)2 * kMaxQ * kCntStride; }
size_t xch_words(int sm_count) { return (size_t)sm_count * (2 * kExchGroups) * kAreaWords; }

cudaError_t launch_in(const Dims& d, const void* x_bf16, float* x, int B, cudaStream_t s) {
  const int NS = B > 8 ? 16 : 8, n = d.D / 4 * NS;
  k_batch_x_in<<<(n + 255) / 256, 256, 0, s>>>(static_cast<const uint16_t*>(x_bf16), x, B, NS, d.D);
  return cudaGetLastError();
}
cudaError_t launch_out(const Dims& d, const float* x, float* out, int B, cudaStream_t s) {
  const int NS = B > 8 ? 16 : 8, n = B * (d.D / 4);
  k_batch_x_out<<<(n + 255) / 256, 256, 0, s>>>(x, out, B, NS, d.D);
  return cudaGetLastError();
}

cudaError_t launch(const Dims& d, const ChainArgs& a, float* x, int B, State* st, cudaStream_t s, int sm_count, int* launches) {
  const bool dense = a.dense_rows > 0;
  const int nsg = B > 8 ? 2 : 1;
  Plan p;
  if (!make_plan(d, dense ? a.dense_rows : d.C, dense, nsg, sm_count, &p)) return cudaErrorInvalidValue;
  *launches = 0;
  for (int l0 = a.l_begin; l0 < a.l_end; l0 += p.run_layers) {
    KArgs ka;
    ka.gate = static_cast<const unsigned char*>(a.gate);
    ka.up = static_cast<const unsigned char*>(a.up);
    ka.downT = static_cast<const unsigned char*>(a.downT);
    ka.slots = a.active_slots;
    ka.counters = a.counters;
    ka.x = x;
    ka.cnt = st->cnt;
    ka.xch = st->xch;
    ka.status = a.status;
    ka.row_pitch = (size_t)d.D * (dense ? 6 : 2);
    ka.layer_bytes = dense ? (size_t)a.dense_rows * d.D * 6 : (size_t)d.C * d.D * 2;
    ka.read_base = st->read_base;
    ka.add_base = st->add_base;
    ka.seq_base = st->seq_base;
    ka.l_begin = l0;
    ka.l_end = std::min(a.l_end, l0 + p.run_layers);
    ka.B = B;
    ka.D = d.D;
    ka.C = d.C;
    ka.check = a.check;
    ka.Q = p.Q;
    ka.dense_rows = a.dense_rows;
    ka.ng = p.ng;
    ka.max_rows = p.max_rows;
    ka.slot_bytes = p.slot_bytes;
    const int grid = p.R * p.Q;
    cudaError_t e;
    if (nsg == 1) {
      if (p.np <= 2) e = launch_one<1, 2>(ka, p.smem, grid, s);
      else if (p.np <= 4) e = launch_one<1, 4>(ka, p.smem, grid, s);
      else if (p.np <= 8) e = launch_one<1, 8>(ka, p.smem, grid, s);
      else e = launch_one<1, 10>(ka, p.smem, grid, s);
    } else {
      if (p.np <= 2) e = launch_one<2, 2>(ka, p.smem, grid, s);
      else if (p.np <= 4) e = launch_one<2, 4>(ka, p.smem, grid, s);
      else if (p.np <= 8) e = launch_one<2, 8>(ka, p.smem, grid, s);
      else e = launch_one<2, 10>(ka, p.smem, grid, s);
    }
    if (e != cudaSuccess) return e;
    // Counters and stamps only ever grow; the next launch starts where this one ends.  (A launch that failed counts nothing.)
    const unsigned int nl = (unsigned int)(ka.l_end - ka.l_begin);
    st->read_base += nl * (unsigned int)p.R;
    st->add_base += nl * (unsigned int)(p.R * kWarps);
    st->seq_base += nl * (unsigned int)((p.max_rows + kChunk - 1) / kChunk) + 1u;
    *launches += 1;
  }
  return cudaSuccess;
}

}  // namespace chain_batch
}  // namespace npi
