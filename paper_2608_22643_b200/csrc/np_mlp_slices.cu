// Stage 4 over a run of consecutive layers in ONE resident kernel, partitioned in two
// directions (B = 1):
//
//   x_{l+1} = x_l + sum_{i in act_l} silu(gate_l[s_i].n_l) * (up_l[s_i].n_l) * downT_l[s_i],
//   n_l = x_l / sqrt(mean(x_l^2) + 1e-6)   (pre-MLP RMS normalisation, unit gain)
//
// (Section 3.4: the sparse MLP reads each active row through the slot map.)
//
// A layer moves ~27 MB at the 7B shape, 4 us of HBM time, and its rows do not depend on x, so they
// stream ahead of it; what a layer costs beyond that is the chain of dependent steps from x_l to
// x_{l+1}.  The partition keeps that chain short:
//
// blocks   The grid is Q column slices x R row groups.  Block (r, q) owns the rows of row group r
//          and slice q of the columns: the K range of its dot products is the column range of its
//          outputs, so of x it only ever needs slice q.  Phase 1 gives partial dot products over a
//          slice; the Q blocks of a row group exchange them once per 64 rows through 64-bit (value,
//          stamp) words (one store, polled by the readers: no fence, no counter).  Phase 2 gives a
//          partial sum of the slice's outputs, and the hand-over of x spans the R blocks of a slice.
// warps    Inside a block the columns are dealt once more: a warp owns KB K blocks of 16 columns.  It
//          polls the sums of these columns, keeps their x, makes the B operand of its K blocks from
//          them, multiplies every row of the block by it, and in phase 2 forms and adds the outputs of
//          the same columns.  Nothing but the partial dot products crosses between the warps: no
//          block-wide barrier, and x is never read from another warp's part of shared memory.  (With
//          the rows dealt to the warps instead, eight of them, x went through shared memory and a
//          barrier to all, and every warp read half of it back: 7.3 us per layer at the 7B shape, 5.1 now;
//          13B 8.1 and 6.6, 70B 15.1 and 11.4, 256 columns and 60 rows 4.7 and 2.7.)
// rows     What a phase multiplies is in registers as A fragments before its operand arrives: gate
//          and up tiles are loaded while the sums of the layer before are on their way, down tiles
//          during the exchange.  A tile's ring slot is free as soon as it is loaded, so the registers
//          (128 KB of the block's rows) extend the ring.
//
// Between two layers of a launch the R partial sums of a column meet in a 64-bit word that carries
// its own arrival count: a block adds, with one 64-bit reduction per column, 2^56 + round(y * 2^30),
// so the word's top byte counts the blocks that have added and the rest is their sum in fixed point
// (resolution 2^-30, |y| < 2^19 per block, checked).  A reader polls the words of its own columns
// until the count is R: no fence, no arrival counter and no second trip to read the sums, the adds
// commute exactly (the result does not depend on their order), and nothing is cleared while it is in
// use: the words only grow, two sets of them alternate by layer, and a reader subtracts what it saw
// at the set's previous completion (all arithmetic modulo 2^64).  What the sets held when the launch
// began is read at its start; a block's first adds wait until every block of its slice has done that
// reading (one arrival counter per slice, counted once per launch and long complete by the time the
// first layer ends).  The launch's last layer leaves its sums as fp32 in the stack's rotating
// accumulators, the form every other kernel of the chain reads -- unless the launch ends the stack:
// then the last layer's sums go through the counted words too, and the blocks of row group 0 wait
// for them and write the stack's result.
//
// Both phases run on the tensor cores (mma.sync m16n8k16, bf16 x bf16 -> fp32).  Phase 1: A = 16
// gate / up vectors over a K block, B = x as three truncated bf16 terms (exact to 2^-24) in columns
// 0-2.  Phase 2: A = 16 output columns x 16 down rows (ldmatrix.trans of the row-major pieces), B =
// the activations as three bf16 terms.  In both, columns 4-6 of B repeat columns 0-2, so that the
// upper two lanes of a quad hold a second tile's sums without a shuffle.
//
// On the way from the sums to the next layer's sums a branch around some lanes, or a loop that lanes leave one by one, parts a warp and
// costs it hundreds of cycles per layer: where those were taken out, the place says what it gave.  Two are left: the poll of the sums
// themselves (add_sums), which every lane leaves when its own columns are there, and lane 0's wait for arrivals in a launch's first layer.
//
// Shared memory is one ring of load groups in the order they are consumed: the gate|up pieces of a
// layer's rows, then its down pieces, then the next layer's.  A producer warp fills it with 1-D bulk
// copies (one mbarrier per group) and runs ahead across layers.  Pieces are 16 bytes further apart
// than they are long, so that the eight row addresses of an ldmatrix fall into different banks.  An
// exchange warp adds the warps' partial dot products, trades them and leaves the activations.
//
// Every wait (mbarrier, exchange words, counted sums) is bounded; once one has run out the block
// records kStatTimeout and skips all later waits except those for its ring (np_ring.h), so the kernel
// drains; the blocks that depend on it follow at their next wait.  The producer stays until its copies
// have landed.
#include <algorithm>

#include "np_device.cuh"
#include "np_internal.h"
#include "np_pipe.cuh"

namespace npi {
namespace chain_slices {
using namespace npd;

constexpr int kQ = 4;                  // column slices
constexpr int kWarps = 8;              // consumer warps, at most.  (Sixteen, with half the K blocks and 104 registers each: 7B shape 190 us
                                       // per 32 layers against 188, 13B 315 against 284, 256 columns 64 per 20 layers against 60.)
constexpr int kBlock = (kWarps + 4) * 32;  // plus the producer warp, two exchange warps and an idle one (a warpgroup changes
                                           // its register share as a whole)
constexpr int kConsumerRegs = 208;     // 256 x 208 + 128 x 88 = 384 x 168, what the block is launched with
constexpr int kOtherRegs = 88;
constexpr int kExchWarps = 2;              // each takes 32 rows of a round
constexpr int kSlotPieces = 16;        // pieces of a ring slot: an MMA tile.  (Slots of 8 or 4: 7B shape 210 and 288 us where 16 took 204.)
constexpr int kMaxSlots = 32;          // ring slots
constexpr int kBarStride = 32;         // one 128-byte line per counter
constexpr int kFixShift = 30;          // fixed-point position of the counted sums
constexpr float kFixLimit = 524288.f;  // |partial sum| a block may add (2^19: 63 of them stay below 2^25 = 2^(55 - kFixShift))
constexpr int kMaxR = 63;              // row groups whose counts and sums fit a word
constexpr int kPad = 16;               // bytes between pieces in shared memory
constexpr int kChunkVec = 128;         // gate and up vectors of one round of the exchange, at most (64 rows)
constexpr int kXchStride = kChunkVec + 16;  // 64-bit words a block publishes per round: its vectors' sums, the sum of squares

// Tiles of 16 vectors whose A fragments a warp holds at a time (up to 128 registers), and down tiles beside the accumulators: as
// many as fit the registers.  What is spilled costs more than a tile loaded late (the shared memory leaves the L1 no room: 7B shape
// 273 us with 90 words spilled), and with sixteen K blocks a single tile is best (70B shape 1.00 ms, 1.03 with two).
__host__ __device__ constexpr int tiles_up(int KB) { return KB <= 8 ? 4 : KB <= 10 ? 3 : KB <= 12 ? 2 : 1; }
__host__ __device__ constexpr int tiles_down(int KB) { return KB <= 4 ? 4 : KB <= 10 ? 2 : 1; }
// Tiles of those that are waited for, loaded and given back at a time.  A wait costs instructions (2048 columns: 76 us per 20
// layers with one wait for all four, 78 with two), a late return leaves the ring full (7B shape 185 us with one wait, 173 with
// two; 3000 rows of 4096 columns 177 and 160 us per 12 layers).
__host__ __device__ constexpr int tiles_wait(int KB) { return KB <= 4 ? 4 : tiles_up(KB) > 2 ? 2 : tiles_up(KB); }
// Whether the producer's wait for a free slot is lane 0's or the whole warp's.  What lies between a free slot and its copies sets the
// stream's pace, so the rows' addresses are formed before the wait (behind it, lane 0's: 7B shape 164.0 us per 32 layers where all
// lanes' took 162.3 in front, 70B 945 per 80 where lane 0's took 909).  Which wait is shorter is measured, not understood.  us per 20 layers, all
// lanes / lane 0, with a tenth of the neurons active: below eight K blocks alike (256 columns 54.2 / 54.2, 1536 68.0 / 68.1, 2560 84.7 /
// 84.8, 3072 87.8 / 87.9), eight 104.8 / 106.7, ten 163.1 / 157.9 (4464 columns 167.5 / 165.3), twelve 203.6 / 219.2 (5296 columns 192.3 /
// 189.4).  At sixteen it turns with the rows of a block: 39 rows, the 70B shape, 998 / 908 per 80 layers; 60 rows of 8192 columns 358.8 / 364.2, 52 of
// 7008 297.2 / 309.4.  There the line follows the shape that the kernel meets in the configurations.
__host__ __device__ constexpr bool lane0_waits(int KB) { return KB == 10 || KB == 16; }
// tiles of a round of the exchange: whole groups of tiles_up
__host__ __device__ constexpr int tiles_chunk(int KB) { return kChunkVec / 16 / tiles_up(KB) * tiles_up(KB); }

struct KArgs {
  const unsigned char* gate;   // layer 0 of each buffer; layer stride = C * D * 2 bytes
  const unsigned char* up;
  const unsigned char* downT;
  const int32_t* slots;        // active_slots [L][C]
  const int32_t* counters;     // [L][NP_N_COUNTERS]
  const uint16_t* x_bf16;      // not NULL: the run starts the stack (layer 0) and reads its input from here (bf16 [D])
  float* xbuf[2];              // x_l of the run's last layer is stored to xbuf[l & 1]
  float* x_out;                // may be NULL; the launch ends the stack and leaves x_L = x_{L-1} + MLP_{L-1} here
  float* zbuf[3];              // MLP_l(x_l) of the launch's last layer goes to zbuf[l % 3]: kZRep copies of [D]
  unsigned long long* zfix;    // [2][D] counted fixed-point sums of MLP_l(x_l), sets alternate by layer, never cleared
  unsigned int* bars;          // [kQ][kBarStride] arrival counters, never reset (the host tracks their value): blocks of a
                               // slice that have read the sets at the launch's start
  unsigned int bar_base;       // value of every counter when the launch starts
  unsigned long long* xch;     // [2][grid][kXchStride] (value, stamp) words
  int32_t* status;
  unsigned int seq_base;       // stamp of the launch's first exchange minus one
  int l_begin, l_end, D, C, check;
  int nw, kw;                  // consumer warps that own columns, K blocks of each (the last may have fewer)
  int ng;                      // ring slots
  int max_rows;                // most rows a block can have in a layer
  int part_bufs;               // rounds of partial dot products held (1 or 2)
  uint32_t slot_bytes;
};

// 32-bit words a consumer warp's B operand takes: [K block pair][term][lane of the quad][K block of the pair][half].  A fourth, zero
// "term" stands in the columns that have none: every lane loads its column, and no branch parts the warp between x and the
// multiplications.  (7B shape 170.1 us per 32 layers with a branch around those lanes, 166.9 without; 13B 278.9 and 272.3.)  The zeros
// take a slot of the ring at one width in twenty.  With 16 bytes of zeros per block in their place the slot is there and gives nothing,
// and the step from pair to pair costs: us per 20 layers, as it is / so, all of widths that lose a slot: 6496 columns 263.4 / 262.1, 6416
// 260.7 / 260.4, 6432 with few rows 177.5 / 181.0, 5296 191.8 / 195.8, 4464 166.4 / 166.5, 3840 109.8 / 110.2, 3008 94.4 / 93.6.
__host__ __device__ constexpr int bstage_words(int KB) { return (KB + 1) / 2 * 64; }

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_row)
               : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_row)
               : "memory");
}
// fp32 -> three bf16 terms by truncation: v = t0 + t1 + t2 up to 2^-24 |v|; the terms come back
// as fp32 bit patterns whose low 16 bits are zero
__device__ __forceinline__ void split3(float v, uint32_t (&t)[3]) {
  t[0] = __float_as_uint(v) & 0xffff0000u;
  const float r1 = v - __uint_as_float(t[0]);
  t[1] = __float_as_uint(r1) & 0xffff0000u;
  const float r2 = r1 - __uint_as_float(t[1]);
  t[2] = __float_as_uint(r2) & 0xffff0000u;
}
// two truncated terms -> one packed bf16x2 word (first element in the low half)
__device__ __forceinline__ uint32_t pack_hi16(uint32_t first, uint32_t second) { return __byte_perm(first, second, 0x7632); }
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void ld_relaxed_v2u64(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_v2u64(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_add_f32(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ unsigned long long stamped(float v, unsigned int stamp) {
  return ((unsigned long long)stamp << 32) | (unsigned long long)__float_as_uint(v);
}

// An arrival whose address is formed with a loaded register.  The order of the loads and what is written behind the arrival does
// not need it (__syncwarp and the arrival's release give that); it keeps the compiler from moving loads across the arrival:
// with a plain one the instances with sixteen K blocks spill 104 to 148 bytes (70B shape 1046 us per 80 layers against 968).
__device__ __forceinline__ void mbar_arrive_after(uint64_t* bar, uint32_t loaded) {
  asm volatile("{\n\t.reg .b32 t;\n\tand.b32 t, %1, 0;\n\tadd.u32 t, t, %0;\n\tmbarrier.arrive.shared::cta.b64 _, [t];\n\t}" ::"r"(npp::smem_addr(bar)), "r"(loaded)
               : "memory");
}

// One exchange warp's part of a round: row `row0 + lane` of it (row0 = 0 or 32, rows in all).  Adds the consumer warps' partial
// sums, publishes them, collects the other slices', leaves the activations as three bf16 terms.  `first`: the layer's first
// round, which also collects the sums of squares and leaves inv_rms.
__device__ __forceinline__ void exchange_rows(const KArgs& a, const float* part, const float* ssq_part, uint16_t* aterm, int apad,
                                              unsigned long long* mine, const unsigned long long* base, int row0, int rows, bool first,
                                              int q, int lane, unsigned int stamp, uint64_t* ss_bar, uint32_t ss_par, float& inv_rms, volatile int* ok) {
  const int row = row0 + lane;
  const bool has_row = row < rows, want_ss = first && lane == 0;
  float own_ss = 0.f;
  const float2* pp = reinterpret_cast<const float2*>(part) + row;
  float2 pv[kWarps];
#pragma unroll
  for (int w = 0; w < kWarps; ++w)  // rows past the round's: whatever is there, not looked at
    pv[w] = w < a.nw ? pp[w * (kChunkVec / 2)] : make_float2(0.f, 0.f);
#pragma unroll
  for (int o = kWarps / 2; o > 0; o >>= 1)  // in pairs: three roundings of a sum where one after the other takes seven
#pragma unroll
    for (int w = 0; w < o; ++w) {
      pv[w].x += pv[w + o].x;
      pv[w].y += pv[w + o].y;
    }
  const float own_g = pv[0].x, own_u = pv[0].y;
  if (has_row) st_relaxed_v2u64(mine + 2 * row, stamped(own_g, stamp), stamped(own_u, stamp));
  if (first) {  // the sums of squares come behind the dot products
    npp::wait_or_flag(ss_bar, ss_par, ok, a.status);
    if (lane < a.nw) own_ss = ssq_part[lane];
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) own_ss += __shfl_xor_sync(0xffffffffu, own_ss, o);
    if (row0 == 0 && lane == 0) st_relaxed_u64(mine + kChunkVec, stamped(own_ss, stamp));
  }
  // One 16-byte load per row and peer (its gate and up words), issued only by the lanes that
  // have a row; lane 0 also fetches the peers' sums of squares.  Strong loads are not merged
  // across lanes, so every load that is not needed costs a request of its own at the L2 (all
  // blocks poll at about the same moment).
  float gsum[kQ], usum[kQ], ssv[kQ];  // indexed by unrolled constants only (registers)
  bool done = __any_sync(0xffffffffu, !*ok);
#pragma unroll 1
  for (uint32_t spin = 0; spin < npp::kSpinLimit && !done; ++spin) {
    unsigned long long wg[kQ], wu[kQ], ws[kQ];  // every load of the round is issued before any is looked at
#pragma unroll
    for (int qq = 0; qq < kQ; ++qq) {
      const unsigned long long* w = base + (size_t)qq * kXchStride;
      const bool peer = qq != q;
      wg[qq] = wu[qq] = ws[qq] = (unsigned long long)stamp << 32;
      if (peer && has_row) ld_relaxed_v2u64(w + 2 * row, wg[qq], wu[qq]);
      if (peer && want_ss) ws[qq] = ld_relaxed_u64(w + kChunkVec);
    }
    unsigned int bad = 0;
#pragma unroll
    for (int qq = 0; qq < kQ; ++qq) {
      bad |= ((unsigned int)(wg[qq] >> 32) ^ stamp) | ((unsigned int)(wu[qq] >> 32) ^ stamp) | ((unsigned int)(ws[qq] >> 32) ^ stamp);
      gsum[qq] = __uint_as_float((unsigned int)wg[qq]);
      usum[qq] = __uint_as_float((unsigned int)wu[qq]);
      ssv[qq] = __uint_as_float((unsigned int)ws[qq]);
    }
    // The lanes leave together: with an exit of its own for each the warp runs on in pieces (256 columns 59.6 us per 20 layers, 56.4
    // with the vote; 7B shape 172.0 per 32 and 170.2).
    done = __all_sync(0xffffffffu, bad == 0);
  }
  if (!done && *ok) {
    *ok = 0;
    atomicOr(a.status, npp::kStatTimeout);
  }
  __syncwarp();
  if (first) {
    float ss = 0.f;
#pragma unroll
    for (int qq = 0; qq < kQ; ++qq) ss += qq == q ? own_ss : ssv[qq];  // the same order in every block
    inv_rms = __shfl_sync(0xffffffffu, rsqrtf(ss / (float)a.D + kRmsEps), 0);  // lane 0 holds the peers' sums
  }
  // All lanes form an activation, those without a row a zero: the last 16-row block is padded with some of them, the others lie
  // behind the last round's end.  (With branches around the lanes that have a row 256 columns take 55.7 us per 20 layers, 54.4
  // without; 7B shape 171.0 per 32 and 170.1.)
  float gsv = 0.f, usv = 0.f;
#pragma unroll
  for (int qq = 0; qq < kQ; ++qq) {
    gsv += qq == q ? own_g : gsum[qq];
    usv += qq == q ? own_u : usum[qq];
  }
  // the MLP's input is x_l scaled to unit RMS; the dot products are linear in it
  gsv *= inv_rms;
  usv *= inv_rms;
  const float av = has_row ? gsv / (1.f + __expf(-gsv)) * usv : 0.f;
  uint32_t tt[3];
  split3(av, tt);
  aterm[row] = (uint16_t)(tt[0] >> 16);
  aterm[apad + row] = (uint16_t)(tt[1] >> 16);
  aterm[2 * apad + row] = (uint16_t)(tt[2] >> 16);
}

// KB: K blocks (16 columns) of a warp.  FULL: every warp of every slice has exactly KB.
template <int KB, bool FULL>
__global__ void __launch_bounds__(kBlock, 1) k_mlp_slices(const __grid_constant__ KArgs a) {
  extern __shared__ __align__(128) unsigned char csm[];
  __shared__ __align__(8) uint64_t full_bar[kMaxSlots];   // the slot's copies have landed
  __shared__ __align__(8) uint64_t empty_bar[kMaxSlots];  // every consumer warp has loaded the slot
  __shared__ __align__(8) uint64_t p1_bar;                // every consumer warp has left its partial sums of a round
  __shared__ __align__(8) uint64_t ss_bar;                // ... and its sum of x_l^2
  __shared__ __align__(8) uint64_t act_bar;               // the exchange warp has left the round's activations
  __shared__ float ssq_part[kWarps];                      // per-warp sums of x_l^2
  __shared__ int s_ok[2];                                 // no wait has run out; the ring was given up
  __shared__ int lay_rb[kMaxLayers];  // first active-list index of this block's row group, per layer
  __shared__ int lay_n[kMaxLayers];   // rows of this row group

  constexpr int PT = tiles_up(KB), WT = tiles_wait(KB), PD = tiles_down(KB), CT = tiles_chunk(KB);
  constexpr int KH = KB > 12 ? KB / 2 : KB;  // column tiles whose down fragments are held at a time
  constexpr int J = (KB * 8 + 31) / 32;  // pairs of columns a lane owns
  const bool fin = a.x_out != nullptr;   // counted sums behind the launch's last layer, too
  constexpr int Q = kQ;
  const int q = blockIdx.x % Q, r = blockIdx.x / Q;
  const int G = gridDim.x, R = G / Q, D = a.D;
  const int kq0 = q * (D >> 4) / Q;                // first K block of the slice (uneven slices: one more in some of them)
  const int nk = (q + 1) * (D >> 4) / Q - kq0;     // 16-wide K blocks = 16-column tiles of the slice
  const uint32_t piece_bytes = (uint32_t)nk * 32u;
  const uint32_t pstride = piece_bytes + kPad;     // distance between pieces in shared memory
  const int ng = a.ng;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nl = a.l_end - a.l_begin;
  const int apad = ((a.max_rows + 15) & ~15) + 16;  // activations per term, padded so that a 16-row block never runs out
  // dynamic shared memory: ring | B operands | partial sums | activations | slots of two layers
  uint32_t* bstage = reinterpret_cast<uint32_t*>(csm + (size_t)ng * a.slot_bytes);         // [nw][bstage_words]
  float* part = reinterpret_cast<float*>(bstage + (size_t)a.nw * bstage_words(KB));        // [part_bufs][nw][kChunkVec]
  uint16_t* aterm = reinterpret_cast<uint16_t*>(part + (size_t)a.part_bufs * a.nw * kChunkVec);  // [3][apad] bf16 terms of a_i
  int32_t* slot_buf = reinterpret_cast<int32_t*>(aterm + 3 * apad);                        // [2][max_rows]
  volatile int* ok = s_ok;

  // ---- this row group's share of every layer of the run ----
  if (tid < nl) {
    int n = a.counters[(size_t)(a.l_begin + tid) * NP_N_COUNTERS + NP_CNT_ACTIVE];
    if (a.check && (n < 0 || n > a.C)) {
      atomicOr(a.status, kStatBadCount);
      n = 0;
    }
    const int rb = (int)(((long long)n * r) / R);
    const int re = (int)(((long long)n * (r + 1)) / R);
    lay_rb[tid] = rb;
    lay_n[tid] = min(re - rb, a.max_rows);
  }
  if (tid == kBlock - 1) {
    for (int s = 0; s < ng; ++s) {
      npp::mbar_init(&full_bar[s], 1);
      npp::mbar_init(&empty_bar[s], (uint32_t)a.nw);
    }
    npp::mbar_init(&p1_bar, (uint32_t)a.nw);
    npp::mbar_init(&ss_bar, (uint32_t)a.nw);
    npp::mbar_init(&act_bar, kExchWarps);
    npp::fence_barrier_init();
    s_ok[0] = 1, s_ok[1] = 0;
  }
  __syncthreads();
  if (wid >= kWarps) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));

  if (wid == kWarps) {
    // =========================== producer warp ===========================
    // The groups are requested in the order they are consumed.  (Lanes that wait on different barriers must not be used: the compiler
    // may reconverge the warp after a wait.)  A slot's copies are issued by as many lanes as it has pieces.  The slots of a layer's rows
    // are fetched a layer ahead.
    int slot = 0;
    uint32_t par = 0;
    // A row is read once per token: the copies mark their lines evict-first, so that the 27 MB a layer streams
    // through the L2 do not push out the few hundred KB every layer meets in (exchange words, counted sums).
    const uint64_t l2_policy = npp::policy_evict_first();
    const size_t row_bytes = (size_t)D * 2, layer_bytes = (size_t)a.C * row_bytes;
    auto fetch_slots = [&](int li) {
      const int32_t* src = a.slots + (size_t)(a.l_begin + li) * a.C + lay_rb[li];
      const uint32_t dst = npp::smem_addr(slot_buf + (size_t)(li & 1) * a.max_rows);
#pragma unroll 1
      for (int i = lane; i < lay_n[li]; i += 32) cp_async4(dst + 4u * (uint32_t)i, src + i);
    };
    fetch_slots(0);
#pragma unroll 1
    for (int li = 0; li < nl; ++li) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      if (li + 1 < nl) fetch_slots(li + 1);
      const int nrows = lay_n[li];
      const int32_t* rows = slot_buf + (size_t)(li & 1) * a.max_rows;
      const size_t lbase = (size_t)(a.l_begin + li) * layer_bytes + (size_t)kq0 * 32;
      // pass 0: gate|up pieces (8 rows a slot, two pieces each); pass 1: down pieces (16 rows)
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        const int step = pass == 0 ? kSlotPieces / 2 : kSlotPieces;
#pragma unroll 1
        for (int r0 = 0; r0 < nrows; r0 += step) {
          const int npieces = min(step, nrows - r0) << (pass == 0 ? 1 : 0);
          const unsigned char* src = nullptr;
          if (lane < npieces) {
            int sl = rows[r0 + (pass == 0 ? lane >> 1 : lane)];
            if (a.check && (sl < 0 || sl >= a.C)) {
              atomicOr(a.status, kStatBadSlot);
              sl = 0;
            }
            src = (pass == 0 ? ((lane & 1) ? a.up : a.gate) : a.downT) + lbase + (size_t)sl * row_bytes;
          }
          if (!lane0_waits(KB) || lane == 0) npp::ring_wait(&empty_bar[slot], par ^ 1u, ok, a.status);
          if (lane == 0) npp::mbar_expect_tx(&full_bar[slot], (uint32_t)npieces * piece_bytes);
          __syncwarp();  // the expect_tx precedes the copies
          if (src) npp::bulk_g2s_stream(csm + (size_t)slot * a.slot_bytes + (size_t)lane * pstride, src, piece_bytes, &full_bar[slot], l2_policy);
          __syncwarp();
          if (++slot == ng) {
            slot = 0;
            par ^= 1u;
          }
        }
      }
    }
    uint32_t patience = npp::kSpinLimit;
    if (lane == 0) npp::drain_ring(full_bar, ng, slot, par, patience);
    return;
  }

  if (wid > kWarps) {
    // =========================== exchange warps ===========================
    const int e = wid - kWarps - 1;
    if (e >= kExchWarps) return;
    unsigned int nx = 0, nss = 0;  // rounds, layers with rows so far
#pragma unroll 1
    for (int li = 0; li < nl; ++li) {
      const int nrows = lay_n[li];
      float inv_rms = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < nrows; c0 += CT * 8) {
        npp::wait_or_flag(&p1_bar, nx & 1u, ok, a.status);
        __syncwarp();
        const unsigned int stamp = a.seq_base + 1u + nx;
        unsigned long long* mine = a.xch + ((size_t)(nx & 1u) * G + blockIdx.x) * kXchStride;
        const unsigned long long* base = a.xch + ((size_t)(nx & 1u) * G + (size_t)r * Q) * kXchStride;
        const float* pt = part + (size_t)(nx & (unsigned int)(a.part_bufs - 1)) * a.nw * kChunkVec;
        const int rows = min(CT * 8, nrows - c0);
        // (a warp without rows in the first round has none in a later one, for which it would need the sum of squares)
        if (32 * e < rows) exchange_rows(a, pt, ssq_part, aterm + c0, apad, mine, base, 32 * e, rows, c0 == 0, q, lane, stamp, &ss_bar, nss & 1u, inv_rms, ok);
        __syncwarp();
        if (lane == 0) npp::mbar_arrive(&act_bar);
        ++nx;
      }
      nss += nrows > 0 ? 1u : 0u;
    }
    return;
  }

  // =========================== consumer warps ===========================
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsumerRegs));
  if (wid >= a.nw) return;
  const int l_last = a.l_end - 1;
  const int kw0 = wid * (FULL ? KB : a.kw);                                      // the warp's first K block of the slice
  const int nkb = FULL ? KB : max(0, min(a.kw, nk - kw0));         // and how many it has
  const int col0 = (kq0 + kw0) * 16;                             // its first column
  const int g8 = lane >> 2, t4 = lane & 3;                       // mma fragment coordinates of this lane
  const int m4 = lane >> 3, rr = lane & 7;                       // ldmatrix: lanes 8 m4 .. 8 m4 + 7 give the row addresses of 8x8 matrix m4
  const int term = g8 & 3;                                       // column g8 of B: term g8 & 3 (the fourth is zero)
  const uint32_t ring = npp::smem_addr(csm) + (uint32_t)kw0 * 32u;
  uint32_t* bs = bstage + (size_t)wid * bstage_words(KB);
  int slot = 0;
  uint32_t par = 0;
  unsigned int nx = 0, acts = 0;  // rounds of the exchange begun, rounds whose activations are known to be there

  // waits for the slots of the next `n` pieces (a group of tiles)
  auto group_wait = [&](int n) {
    int s = slot;
    uint32_t p = par;
#pragma unroll 1
    for (; n > 0; n -= kSlotPieces) {
      npp::ring_wait(&full_bar[s], p, ok, a.status);
      if (++s == ng) s = 0, p ^= 1u;
    }
  };
  // address of tile u of the group: a slot each
  auto tile_at = [&](int u) -> uint32_t {
    int s = slot + u;
    if (s >= ng) s -= ng;
    return ring + (uint32_t)s * a.slot_bytes;
  };
  // gives the group's slots back; `last`: a register loaded from its last tile
  auto group_release = [&](int n, uint32_t last) {
    __syncwarp();  // every lane has loaded its part
#pragma unroll 1
    for (; n > 0; n -= kSlotPieces) {
      if (lane == 0) mbar_arrive_after(&empty_bar[slot], last);
      if (++slot == ng) slot = 0, par ^= 1u;
    }
  };

  // counted sums: what the words of this lane's columns held when their set was last complete
  // (zprev: the set read next, zprev2: the other one; they trade places after every read)
  for (int i = lane; i < bstage_words(KB); i += 32) bs[i] = 0u;  // the fourth term stays zero
  __syncwarp();
  float2 xown[J];  // x_l of the columns this lane owns, for the whole run
  unsigned long long zprev[J][2], zprev2[J][2];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    xown[j] = make_float2(0.f, 0.f);
    zprev[j][0] = zprev[j][1] = zprev2[j][0] = zprev2[j][1] = 0ull;
  }
  if (nl > 1 || fin) {
    unsigned long long seen = 0ull;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int c = lane + 32 * j;
      if (c < nkb * 8) {
        const ulonglong2 p0 = __ldcg(reinterpret_cast<const ulonglong2*>(a.zfix + col0) + c);
        const ulonglong2 p1 = __ldcg(reinterpret_cast<const ulonglong2*>(a.zfix + (size_t)D + col0) + c);
        zprev[j][0] = p0.x, zprev[j][1] = p0.y;
        zprev2[j][0] = p1.x, zprev2[j][1] = p1.y;
        seen ^= p0.x ^ p0.y ^ p1.x ^ p1.y;
      }
    }
    // Every value has arrived (it is compared, to no effect) before the block counts itself in: only then may any block of the
    // slice add to these words.
    if (seen == 0xffffffffffffffffull) static_cast<volatile uint32_t*>(bs)[lane] = 0u;
    asm volatile("bar.sync 1, %0;" ::"r"(a.nw * 32) : "memory");
    if (tid == 0) atomicAdd(a.bars + q * kBarStride, 1u);
  }

  // x += the sums in the set at `zw`, once every row group has added its part.  Two pairs of columns are polled together.
  auto add_sums = [&](const unsigned long long* zw) {
#pragma unroll
    for (int j0 = 0; j0 < J; j0 += 2) {
      unsigned long long w[2][2];
      bool done = !*ok;
#pragma unroll
      for (int v = 0; v < 2; ++v) w[v][0] = w[v][1] = 0ull;
      uint32_t spin = 0;
#pragma unroll 1
      while (!done) {  // every load of the round is issued before any is looked at
#pragma unroll
        for (int v = 0; v < 2 && j0 + v < J; ++v)
          if (lane + 32 * (j0 + v) < nkb * 8) ld_relaxed_v2u64(zw + 2 * (lane + 32 * (j0 + v)), w[v][0], w[v][1]);
        done = true;
#pragma unroll
        for (int v = 0; v < 2 && j0 + v < J; ++v)
          if (lane + 32 * (j0 + v) < nkb * 8)
#pragma unroll
            for (int e = 0; e < 2; ++e)
              done = done && (((long long)(w[v][e] - zprev[j0 + v][e]) + (1ll << 55)) >> 56) == (long long)R;
        if (!done && ++spin == npp::kSpinLimit) {
          *ok = 0;
          atomicOr(a.status, npp::kStatTimeout);
          break;
        }
      }
#pragma unroll
      for (int v = 0; v < 2 && j0 + v < J; ++v) {
        const int j = j0 + v;
        float z[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          z[e] = __ll2float_rn((long long)(w[v][e] - zprev[j][e]) - ((long long)R << 56)) * (1.f / (float)(1u << kFixShift));
          zprev[j][e] = zprev2[j][e];  // the other set is read next; this one, as it stands now, after that
          zprev2[j][e] = w[v][e];
        }
        if (done && lane + 32 * j < nkb * 8) xown[j].x += z[0], xown[j].y += z[1];
      }
    }
  };

#pragma unroll 1
  for (int li = 0; li < nl; ++li) {
    const int l = a.l_begin + li;
    const int nrows = lay_n[li], nvec = 2 * nrows;
    const int nt = (nvec + 15) >> 4;
    uint32_t xb[(KB + 1) / 2][4];
    float ssq = 0.f;
    int t0 = 0;
#pragma unroll 1
    do {
      // ---- the next gate|up tiles; the layer's first ones before x arrives.  Vectors past the last one read the last one:
      //      their results are not looked at ----
      uint32_t af[PT][KB][4];
#pragma unroll
      for (int v = 0; v < PT; v += WT) {
        const int n = min(16 * (WT < PT - v ? WT : PT - v), nvec - 16 * (t0 + v));
        uint32_t last = 0u;
        group_wait(n);
#pragma unroll
        for (int u = 0; u < WT && v + u < PT; ++u) {
          if (16 * u < n) {
            const uint32_t p = tile_at(u) + (uint32_t)min(rr + 8 * (m4 & 1), n - 1 - 16 * u) * pstride + (uint32_t)(m4 >> 1) * 16u;
#pragma unroll
            for (int i = 0; i < KB; ++i) {
              if (FULL || i < nkb) ldmatrix_x4(af[v + u][i], p + (uint32_t)i * 32u);
              else af[v + u][i][0] = af[v + u][i][1] = af[v + u][i][2] = af[v + u][i][3] = 0u;
            }
            last = af[v + u][KB - 1][3] | af[v + u][0][0];
          } else {  // not used; set, so that what the registers held before does not live on
#pragma unroll
            for (int i = 0; i < KB; ++i) af[v + u][i][0] = af[v + u][i][1] = af[v + u][i][2] = af[v + u][i][3] = 0u;
          }
        }
        group_release(n, last);
      }
      if (t0 == 0) {
        // ---- x_l of this lane's columns: first layer of the run from global, afterwards x_l = x_{l-1} + MLP_{l-1} once every
        //      row group has added its part ----
        if (li == 0) {
          const float* xa = a.xbuf[(l + 1) & 1] + col0;
          const float* zb = l > 0 ? a.zbuf[(l - 1) % 3] + col0 : nullptr;
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const int c = lane + 32 * j;
            if (c < nkb * 8) {
              if (a.x_bf16) {  // the stack's input: bf16 values widened here (no kernel in front for that)
                const uint32_t h = __ldg(reinterpret_cast<const uint32_t*>(a.x_bf16 + col0) + c);
                xown[j] = make_float2(bf16_lo(h), bf16_hi(h));
              } else {
                xown[j] = __ldcg(reinterpret_cast<const float2*>(xa) + c);
              }
              if (zb) {
#pragma unroll
                for (int rep = 0; rep < kZRep; ++rep) {
                  const float2 w = __ldcg(reinterpret_cast<const float2*>(zb + (size_t)rep * D) + c);
                  xown[j].x += w.x, xown[j].y += w.y;
                }
              }
            }
          }
        } else {
          add_sums(a.zfix + (size_t)((li - 1) & 1) * D + col0);
          __syncwarp();
          // the launch's last layer adds into an accumulator that other blocks cleared one layer earlier (and fenced before they
          // added the sums read above): the fence that completes that order on this side
          if (li == nl - 1 && !fin) __threadfence();
        }
        // ---- three bf16 terms of x, into the layout of the B operand ----
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const int c = lane + 32 * j;
          if (c < nkb * 8) {
            ssq += xown[j].x * xown[j].x + xown[j].y * xown[j].y;
            uint32_t p0[3], p1[3];
            split3(xown[j].x, p0);
            split3(xown[j].y, p1);
            // columns 2 c, 2 c + 1: K block c >> 3, half (c >> 2) & 1 of it, lane c & 3 of the quad
            uint32_t* w = bs + (c >> 4) * 64 + (c & 3) * 4 + ((c >> 3) & 1) * 2 + ((c >> 2) & 1);
#pragma unroll
            for (int e = 0; e < 3; ++e) w[e * 16] = pack_hi16(p0[e], p1[e]);
            if (r == 0 && l == l_last) *reinterpret_cast<float2*>(a.xbuf[l & 1] + col0 + 2 * c) = xown[j];  // x for the next launch
          }
        }
        // The launch's last layer adds fp32 sums into the stack's rotating accumulators: its own is cleared one layer ahead (by
        // the layer before it; a launch of one layer finds it cleared by the kernel in front), and it clears the one the next
        // kernel's first layer adds into.  Every row group takes a share.
        if (!fin && li >= nl - 2) {
          float* znext = a.zbuf[(l + 1) % 3] + col0;
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const int c = lane + 32 * j;
#pragma unroll
            for (int rep = 0; rep < kZRep; ++rep)
              if (c < nkb * 8 && (c * kZRep + rep) % R == r) *reinterpret_cast<float2*>(znext + (size_t)rep * D + 2 * c) = make_float2(0.f, 0.f);
          }
          if (li == nl - 2) __threadfence();  // ahead of this warp's counted sums of this layer, which every adder has read
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < (KB + 1) / 2; ++i) {
          const uint4 v = *reinterpret_cast<const uint4*>(bs + i * 64 + term * 16 + t4 * 4);
          xb[i][0] = v.x, xb[i][1] = v.y, xb[i][2] = v.z, xb[i][3] = v.w;
        }
      }
      // ---- phase 1: [16 vectors of a tile] x [x as 3 terms] over this warp's K blocks, all rows of the block ----
      // the round's buffer is free once the exchange has read the round that used it before
      const int tc = t0 % CT;
      if (tc == 0) {
#pragma unroll 1
        for (; acts + (unsigned int)a.part_bufs <= nx; ++acts) npp::wait_or_flag(&act_bar, acts & 1u, ok, a.status);
      }
      // Two tiles at a time (registers).  C: [0], [1] = (vector g8, terms 2 t4, 2 t4 + 1); [2], [3] = (vector g8 + 8, same terms).
      // Lanes t4 = 0, 1 of a quad hold terms 0 + 1 and 2 of a tile, lanes 2, 3 the same again: they take the second tile.
      float* pw = part + ((size_t)(nx & (unsigned int)(a.part_bufs - 1)) * a.nw + wid) * kChunkVec + tc * 16 + g8 + 8 * (t4 & 1);
#pragma unroll
      for (int u = 0; u < PT; u += 2) {
        float c[2][2][4];  // a tile's odd K blocks add up beside its even ones: half the roundings of one chain
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int e = 0; e < 4; ++e) c[v][0][e] = c[v][1][e] = 0.f;
#pragma unroll
        for (int i = 0; i < KB; ++i)
#pragma unroll
          for (int v = 0; v < 2 && u + v < PT; ++v)
            if (FULL || i < nkb) mma_bf16_16816(c[v][i & 1], af[u + v][i], xb[i >> 1][(i & 1) * 2], xb[i >> 1][(i & 1) * 2 + 1]);
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int e = 0; e < 4; ++e) c[v][0][e] += c[v][1][e];
        const float lo = t4 < 2 ? c[0][0][0] + c[0][0][1] : c[1][0][0] + c[1][0][1];
        const float hi = t4 < 2 ? c[0][0][2] + c[0][0][3] : c[1][0][2] + c[1][0][3];
        const float other = __shfl_xor_sync(0xffffffffu, (t4 & 1) ? lo : hi, 1);
        const int tile = u + (t4 >> 1);
        if (tile < PT && t0 + tile < nt) pw[tile * 16] = ((t4 & 1) ? hi : lo) + other;
        if (t0 + u + 2 >= nt) break;
      }
      if (nt > 0 && (tc + PT == CT || t0 + PT >= nt)) {
        // one round at a time: the parity of act_bar tells only the current phase from the one before
#pragma unroll 1
        for (; acts != nx; ++acts) npp::wait_or_flag(&act_bar, acts & 1u, ok, a.status);
        __syncwarp();
        if (lane == 0) npp::mbar_arrive(&p1_bar);
        ++nx;
      }
      if (t0 == 0 && nt > 0) {  // behind the dot products: the exchange needs it last
        ssq = warp_sum(ssq);
        if (lane == 0) {
          ssq_part[wid] = ssq;
          npp::mbar_arrive(&ss_bar);
        }
      }
      t0 += PT;
    } while (t0 < nt);
    // ---- phase 2: y[cols] += a_i * downT[s_i][cols]: [16 columns x 16 rows] x [a as 3 terms], this warp's columns ----
    float acc[KB][4];
#pragma unroll
    for (int j = 0; j < KB; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll 1
    for (int r0 = 0; r0 < nrows; r0 += 16 * PD) {
      const int n = min(16 * PD, nrows - r0);
      group_wait(n);
#pragma unroll
      for (int j0 = 0; j0 < KB; j0 += KH) {
        uint32_t df[PD][KH][4], last = 0u;
#pragma unroll
        for (int u = 0; u < PD; ++u) {
          if (16 * u < n) {
            const uint32_t p = tile_at(u) + (uint32_t)min(rr + 8 * (m4 >> 1), n - 1 - 16 * u) * pstride + (uint32_t)(m4 & 1) * 16u;
#pragma unroll
            for (int j = 0; j < KH; ++j) {
              if (FULL || j0 + j < nkb) ldmatrix_x4_trans(df[u][j], p + (uint32_t)(j0 + j) * 32u);
              else df[u][j][0] = df[u][j][1] = df[u][j][2] = df[u][j][3] = 0u;
            }
            last = df[u][KH - 1][3] | df[u][0][0];
          } else {
#pragma unroll
            for (int j = 0; j < KH; ++j) df[u][j][0] = df[u][j][1] = df[u][j][2] = df[u][j][3] = 0u;
          }
        }
        if (j0 + KH >= KB) group_release(n, last);
        if (j0 == 0) {
#pragma unroll 1
          for (; acts != nx; ++acts) npp::wait_or_flag(&act_bar, acts & 1u, ok, a.status);
        }
#pragma unroll
        for (int u = 0; u < PD; ++u) {
          if (16 * u < n) {
            // (loaded by all lanes here, too: 7B shape 166.9 and 164.1, 70B 958 and 940; with a fourth term in shared memory instead
            // of the selection 167.5 and 939)
            const uint16_t* ap = aterm + (size_t)(term < 3 ? term : 0) * apad + r0 + 16 * u + 2 * t4;
            uint32_t b0 = *reinterpret_cast<const uint32_t*>(ap), b1 = *reinterpret_cast<const uint32_t*>(ap + 8);
            if (term == 3) b0 = b1 = 0u;
#pragma unroll
            for (int j = 0; j < KH; ++j)
              if (FULL || j0 + j < nkb) mma_bf16_16816(acc[j0 + j], df[u][j], b0, b1);
          }
        }
      }
    }
    // ---- this block's partial MLP_l(x_l) over the warp's columns ----
    const bool counted = li + 1 < nl || fin;
    if (li == 0 && counted) {  // the launch's first adds: every block of the slice has read what the sets held before
      if (lane == 0 && *ok) {
        const unsigned int target = a.bar_base + (unsigned int)R;
        bool arrived = false;
#pragma unroll 1
        for (uint32_t spin = 0; spin < npp::kSpinLimit && !arrived; ++spin) {
          unsigned int v;
          asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bars + q * kBarStride) : "memory");
          arrived = (int)(v - target) >= 0;
        }
        if (!arrived) {
          *ok = 0;
          atomicOr(a.status, npp::kStatTimeout);
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < KB; j += 2) {
      const int j1 = j + 1 < KB ? j + 1 : j;
      const float lo = t4 < 2 ? acc[j][0] + acc[j][1] : acc[j1][0] + acc[j1][1];
      const float hi = t4 < 2 ? acc[j][2] + acc[j][3] : acc[j1][2] + acc[j1][3];
      const float other = __shfl_xor_sync(0xffffffffu, (t4 & 1) ? lo : hi, 1);
      const float y = ((t4 & 1) ? hi : lo) + other;
      const int tile = j + (t4 >> 1);
      if (tile < (FULL ? KB : nkb)) {
        const int col = col0 + tile * 16 + g8 + 8 * (t4 & 1);
        if (counted) {
          // One 64-bit reduction per column carries the value and this block's arrival (a row group without rows still counts).
          long long fx = 0;
          if (fabsf(y) < kFixLimit) fx = __float2ll_rn(y * (float)(1u << kFixShift));
          else atomicOr(a.status, kStatRange);  // also a NaN: the sum would not mean anything
          red_add_u64(a.zfix + (size_t)(li & 1) * D + col, (unsigned long long)fx + (1ull << 56));
        } else if (nrows > 0) {
          red_add_f32(a.zbuf[l % 3] + (size_t)(r % kZRep) * D + col, y);
        }
      }
    }
  }
  // ---- the launch ends the stack: the blocks of row group 0 wait for the last layer's sums like a next layer
  //      would and leave x_L (no kernel behind this one has to add the accumulator copies up) ----
  if (fin && r == 0) {
    add_sums(a.zfix + (size_t)((nl - 1) & 1) * D + col0);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int c = lane + 32 * j;
      if (c < nkb * 8) *reinterpret_cast<float2*>(a.x_out + col0 + 2 * c) = xown[j];
    }
  }
}

namespace {
struct Plan {
  int R, kb, kw, nw, ng, max_rows, part_bufs;
  bool full;  // every warp of every slice has kb K blocks
  size_t slot_bytes, smem;
};

bool plan(const Dims& d, int sm_count, Plan* p) {
  const int nkt = d.D / 16;
  if (d.D % 16 || nkt < kQ || d.D > kMaxD || sm_count < kQ) return false;
  constexpr int Q = kQ;
  const int nk = (nkt + Q - 1) / Q;  // K blocks of the widest slice
  const int need = (nk + kWarps - 1) / kWarps;
  int KB = need;
  if (KB > 6) KB = KB <= 8 ? 8 : KB <= 10 ? 10 : KB <= 12 ? 12 : 16;
  p->R = std::min(kMaxR, sm_count / Q);
  p->kb = KB;
  p->kw = need;
  p->nw = (nk + need - 1) / need;
  p->full = nkt % Q == 0 && nk % KB == 0 && KB == need;
  p->max_rows = (d.C + p->R - 1) / p->R;  // whatever the active count turns out to be
  const int expect = (int)((std::min<long long>(d.C, std::max(1, d.k)) + p->R - 1) / p->R);
  p->part_bufs = expect > tiles_chunk(KB) * 8 ? 2 : 1;  // rounds follow each other where a share has more rows than one
  const int apad = ((p->max_rows + 15) & ~15) + 16;
  const size_t fixed = (size_t)p->nw * bstage_words(KB) * 4 + (size_t)p->part_bufs * p->nw * kChunkVec * 4 +
                       (size_t)(3 * apad) * 2 + (size_t)2 * p->max_rows * 4 + 128;
  const size_t budget = 227 * 1024 - 2560;  // static shared memory of the kernel
  const size_t pstride = (size_t)nk * 32 + kPad;
  // the tiles a warp loads at a time and one more (every width to 8192 and capacity to 40960 has room for that on 100 SMs and more)
  const int ng_min = std::max(tiles_up(KB), tiles_down(KB)) + 1;
  p->slot_bytes = pstride * kSlotPieces;
  if (fixed + ng_min * p->slot_bytes > budget) return false;
  p->ng = (int)std::min<size_t>(kMaxSlots, (budget - fixed) / p->slot_bytes);
  if (d.ring_stages >= 2) p->ng = std::max(ng_min, std::min(p->ng, d.ring_stages));
  p->smem = (size_t)p->ng * p->slot_bytes + fixed;
  return true;
}
}  // namespace

bool supported(const Dims& d, int sm_count) {
  Plan p;
  return plan(d, sm_count, &p);
}
// room for a launch on all SMs and for one beside the pull kernel
size_t xch_words(const Dims& d, int sm_count) {
  size_t most = 16;
  for (const int n : {sm_count, sm_count - kPullReserve}) {
    Plan p;
    if (plan(d, n, &p)) most = std::max(most, (size_t)2 * (p.R * kQ) * kXchStride);
  }
  return most;
}
size_t zfix_words(const Dims& d) { return (size_t)2 * d.D; }
size_t bar_words() { return (size_t)kQ * kBarStride; }

template <int KB, bool FULL>
static cudaError_t launch_one(const KArgs& ka, size_t sm, int grid_x, cudaStream_t s) {
  auto kfn = k_mlp_slices<KB, FULL>;
  static std::atomic<uint64_t> done{0};
  cudaError_t e = allow_shared(reinterpret_cast<const void*>(kfn), &done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid_x);
  cfg.blockDim = dim3(kBlock);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all blocks co-resident: no wait can starve
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kfn, ka);
}

cudaError_t launch(const Dims& d, const ChainArgs& a, State* st, cudaStream_t s, int sm_count) {
  Plan p;
  if (!plan(d, sm_count, &p) || !st || !st->zfix || !st->bars || !st->xch) return cudaErrorInvalidValue;
  for (int l0 = a.l_begin; l0 < a.l_end; l0 += kMaxLayers) {
    KArgs ka;
    ka.gate = static_cast<const unsigned char*>(a.gate);
    ka.up = static_cast<const unsigned char*>(a.up);
    ka.downT = static_cast<const unsigned char*>(a.downT);
    ka.slots = a.active_slots;
    ka.counters = a.counters;
    ka.x_bf16 = l0 == 0 ? static_cast<const uint16_t*>(a.x_bf16) : nullptr;
    for (int i = 0; i < 2; ++i) ka.xbuf[i] = a.xbuf[i];
    // the launch that ends the stack leaves the result itself
    ka.x_out = std::min(a.l_end, l0 + kMaxLayers) == a.l_end ? a.x_out : nullptr;
    for (int i = 0; i < 3; ++i) ka.zbuf[i] = a.zbuf[i];
    ka.zfix = st->zfix;
    ka.bars = st->bars;
    ka.bar_base = st->bar_base;
    ka.xch = st->xch;
    ka.status = a.status;
    ka.seq_base = st->seq_base;
    ka.l_begin = l0;
    ka.l_end = std::min(a.l_end, l0 + kMaxLayers);
    ka.D = d.D;
    ka.C = d.C;
    ka.check = a.check;
    ka.nw = p.nw;
    ka.kw = p.kw;
    ka.ng = p.ng;
    ka.max_rows = p.max_rows;
    ka.part_bufs = p.part_bufs;
    ka.slot_bytes = (uint32_t)p.slot_bytes;
    const int grid = p.R * kQ;
    cudaError_t e;
#define NP_SLICES(kb) \
  case kb: e = p.full ? launch_one<kb, true>(ka, p.smem, grid, s) : launch_one<kb, false>(ka, p.smem, grid, s); break
    switch (p.kb) {
      NP_SLICES(1);
      NP_SLICES(2);
      NP_SLICES(3);
      NP_SLICES(4);
      NP_SLICES(5);
      NP_SLICES(6);
      NP_SLICES(8);
      NP_SLICES(10);
      NP_SLICES(12);
      NP_SLICES(16);
      default: e = cudaErrorInvalidValue;
    }
#undef NP_SLICES
    if (e != cudaSuccess) return e;
    // The counters and stamps only ever grow; the next launch starts where this one ends.  (A launch that failed counts nothing.)
    const unsigned int nl = (unsigned int)(ka.l_end - ka.l_begin);
    const int chunk_rows = tiles_chunk(p.kb) * 8;
    st->bar_base += (nl > 1 || ka.x_out) ? (unsigned int)p.R : 0u;
    st->seq_base += nl * (unsigned int)((p.max_rows + chunk_rows - 1) / chunk_rows) + 1u;
    st->wrote_out = ka.x_out != nullptr;
  }
  return cudaSuccess;
}

}  // namespace chain_slices
}  // namespace npi
