// Stage 2: per-layer top-k of the predictor's logits -> active-neuron bitmap.
// (The paper turns predictor outputs into one active set per layer, Section 3.4;
// here the set is the k highest-scoring neurons, the K_max budget of Section 4.1.)
//
// One block of 1024 (or 512) threads per (layer, sequence).  A layer is only 44 KB of logits: the
// kernel is a chain of block-wide steps on one SM, and what it costs is the instructions of
// those steps.  Every thread keeps its logits in registers, index tid + threads * j, so that the 32
// lanes of a warp hold the 32 neurons of one bitmap word and a ballot is a word.
//
// Fast path (finite logits that are not all equal): ONE histogram pass over 2048 bins that
// are linear in the logit's value, bin = floor((z - min) * 2047 / (max - min)).  Every step of
// that formula is monotone in z, so the bins are ordered like the keys and every key above
// the bin of the k-th largest belongs to the set; values spread over the bins like their
// density, so the adds to shared memory rarely meet (a radix digit of the float's bits puts
// most of a layer into a handful of bins: sign and exponent are shared).  The few keys inside
// that one bin are listed and ranked against each other exactly, by (key, then lower index).
//
// General path (an infinity or NaN among the logits, a degenerate range, or more than 1024
// keys in the deciding bin, i.e. heavy ties): a radix select on the order-preserving uint32
// image of the fp32 bits, 8 + 12 + 12 bits; the first digit counts into one histogram per warp.
// Both paths select the same set: the k largest keys, ties broken towards the lower index.
#include "np_device.cuh"
#include "np_internal.h"
#include "np_pipe.cuh"

namespace npi {
using namespace npd;

constexpr int kTopkHist = 8192;   // ints: 32 warps x 256 bins in the first radix pass, 4096 bins after; 2048 linear bins + candidate list
constexpr int kLinBins = 2048;
constexpr int kMaxCand = 1024;    // keys of the deciding bin that are ranked directly

#ifdef NP_TRACE  // development builds only: clock stamps of one block
__device__ long long np_tk_clk[32];
extern "C" int np_debug_tk(void* out) { return (int)cudaMemcpyFromSymbol(out, np_tk_clk, sizeof(np_tk_clk)); }
#define TK(ev) do { if (blockIdx.x == 5 && blockIdx.y == 0 && threadIdx.x == 0) np_tk_clk[ev] = clock64(); } while (0)
#else
#define TK(ev) do { } while (0)
#endif

// bit pattern of an fp32 value -> order-preserving uint32 (larger float, larger key; +0 above -0)
__device__ __forceinline__ uint32_t order_key(uint32_t b) { return (b & 0x80000000u) ? ~b : (b | 0x80000000u); }

// Inclusive scan of one int per thread in thread order over a block of T threads; wsum: 33 ints.  Two block-wide barriers; a
// caller that scans again puts one between the calls.
template <int T>
__device__ __forceinline__ int block_inclusive_scan(int v, int* wsum, int lane, int wid) {
  if (T == 1024) return block_inclusive_scan_1024(v, wsum, lane, wid);
  constexpr int NW = T / 32;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const int ws = lane < NW ? wsum[lane] : 0;
    int winc = ws;
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += t;
    }
    if (lane < NW) wsum[lane] = winc - ws;
  }
  __syncthreads();
  return wsum[wid] + inc;
}

// T: threads (512 or 1024).  KPT: keys per thread, ceil(M / T)
template <int T, int KPT>
__global__ void __launch_bounds__(T, 1024 / T) k_topk(const float* __restrict__ logits,  // [B][L][M]
                                                       uint32_t* __restrict__ bitmap,     // [L][W]
                                                       uint32_t* __restrict__ bitmap2,    // a second copy, or NULL
                                                       int L, int M, int k, int use_atomic) {
  constexpr int NW = T / 32;
  extern __shared__ __align__(16) int wsm[];  // [W] per word: selected keys of the deciding bin / count of threshold-equal keys
  __shared__ __align__(16) int hist[kTopkHist];
  __shared__ int wsum[33];
  __shared__ float wlo[32], whi[32];
  __shared__ uint32_t s_prefix;
  __shared__ int s_remaining, s_bin_count, s_bin, s_ncand;

  const int W = M >> 5;
  const int layer = blockIdx.x, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const float* z = logits + ((size_t)b * L + layer) * M;
  uint32_t* out = bitmap + (size_t)layer * W;
  uint32_t* out2 = bitmap2 ? bitmap2 + (size_t)layer * W : nullptr;
  // a word of the result: stored (one sequence), or ORed into what the other sequences left (a batch)
  auto put = [&](int w, uint32_t word) {
    if (use_atomic) {
      if (word) {
        atomicOr(out + w, word);
        if (out2) atomicOr(out2 + w, word);
      }
    } else {
      out[w] = word;
      if (out2) out2[w] = word;
    }
  };

  TK(0);
  npp::pdl_launch_dependents();
  npp::pdl_wait_prior();  // the logits are the previous kernel's
  TK(1);

  if (k <= 0) {  // nothing selected
    for (int w = tid; w < W; w += T) put(w, 0u);
    return;
  }
  if (k >= M) {
    for (int w = tid; w < W; w += T) put(w, 0xffffffffu);
    return;
  }

  // The logits are kept as bit patterns: the keys must be exact, and floating-point moves under flush-to-zero
  // arithmetic need not preserve a denormal.  Only the fast path's bin arithmetic looks at them as numbers.
  uint32_t zb[KPT];
  float lo = __int_as_float(0x7f800000), hi = __int_as_float(0xff800000);
  int bad = 0;
  const uint32_t* zbits = reinterpret_cast<const uint32_t*>(z);
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int i = tid + T * j;
    zb[j] = i < M ? zbits[i] : 0u;  // entries past the layer's end are never counted (every use tests the index)
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    if (tid + T * j < M) {
      bad |= (zb[j] & 0x7f800000u) == 0x7f800000u;  // infinity or NaN
      lo = fminf(lo, __uint_as_float(zb[j]));
      hi = fmaxf(hi, __uint_as_float(zb[j]));
    }
  }
#pragma unroll
  for (int i = 0; i < kLinBins / T; ++i) hist[tid + T * i] = 0;
  for (int w = tid; w < W; w += T) wsm[w] = 0;
  if (tid == 0) s_ncand = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    wlo[wid] = lo;
    whi[wid] = hi;
  }
  TK(2);
  const int any_bad = __syncthreads_or(bad);
  lo = wlo[lane & (NW - 1)];
  hi = whi[lane & (NW - 1)];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const float range = hi - lo;
  const float scale = (float)(kLinBins - 1) / range;
  // block-uniform: every thread holds the same lo, hi and flags
  const bool linear = !any_bad && range > 0.f && (__float_as_uint(range) & 0x7f800000u) != 0x7f800000u &&
                      (__float_as_uint(scale) & 0x7f800000u) != 0x7f800000u;
  TK(3);
  if (linear) {
    auto bin_of = [&](float v) { return min(kLinBins - 1, (int)((v - lo) * scale)); };
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (tid + T * j < M) atomicAdd(&hist[bin_of(__uint_as_float(zb[j]))], 1);
    __syncthreads();
    TK(4);
    // the bin of the k-th largest key: thread t takes the highest bins not taken by the threads below it
    constexpr int BPT = kLinBins / T;
    const int top = kLinBins - 1 - BPT * tid;
    int c[BPT], mine = 0;
#pragma unroll
    for (int i = 0; i < BPT; ++i) mine += c[i] = hist[top - i];
    const int above = block_inclusive_scan<T>(mine, wsum, lane, wid) - mine;  // keys in higher bins
    if (above < k && k <= above + mine) {  // exactly one thread
      int acc = above, i = 0;
#pragma unroll
      for (int q = 0; q < BPT - 1; ++q) {
        if (i == q && k > acc + c[q]) {
          acc += c[q];
          i = q + 1;
        }
      }
      int cnt = c[0];
#pragma unroll
      for (int q = 1; q < BPT; ++q) cnt = i == q ? c[q] : cnt;
      s_bin = top - i;
      s_remaining = k - acc;
      s_bin_count = cnt;
    }
    __syncthreads();
    TK(5);
    const int bstar = s_bin, need = s_remaining, ncand = s_bin_count;
    if (ncand <= kMaxCand) {  // block-uniform
      uint32_t* ckey = reinterpret_cast<uint32_t*>(hist + kLinBins);
      int* cidx = hist + kLinBins + kMaxCand;
      // one pass: the words of the keys above the bin are formed, a lane keeps a round's, the keys inside the bin are
      // listed.  (Lane 0 stored the word of every round behind a branch: np_predict for sixteen sequences of the 7B shape 103.5 us, 100.7
      // with one store of each lane's; three such contexts in turn 80.0 and 78.5 a pass.)
      uint32_t word[(KPT + 31) / 32] = {};
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const int i = tid + T * j;
        const int bn = i < M ? bin_of(__uint_as_float(zb[j])) : -1;
        const uint32_t gt = __ballot_sync(0xffffffffu, bn > bstar);
        if (lane == (j & 31)) word[j >> 5] = gt;
        if (bn == bstar) {
          const int q = atomicAdd(&s_ncand, 1);
          ckey[q] = order_key(zb[j]);
          cidx[q] = i;
        }
      }
#pragma unroll
      for (int v = 0; v < (KPT + 31) / 32; ++v) {
        const int j = lane + 32 * v, w = wid + NW * j;  // the word of neurons 32 w .. 32 w + 31: this warp's logits of round j
        if (j < KPT && w < W) put(w, word[v]);
      }
      __syncthreads();  // the list is complete; the words stored above are ordered before the bits added below
      TK(6);
      for (int t = tid; t < ncand; t += T) {  // rank among the keys of the bin: larger key first, then lower index
        const uint32_t mk = ckey[t];
        const int mi = cidx[t];
        int rank = 0;
        for (int q = 0; q < ncand; ++q) {
          const uint32_t qk = ckey[q];
          rank += (qk > mk || (qk == mk && cidx[q] < mi)) ? 1 : 0;
        }
        if (rank < need) {
          atomicOr(out + (mi >> 5), 1u << (mi & 31));
          if (out2) atomicOr(out2 + (mi >> 5), 1u << (mi & 31));
        }
      }
      TK(16);
      return;
    }
    __syncthreads();  // heavy ties: the general path reuses the histogram and the per-word array
    for (int w = tid; w < W; w += T) wsm[w] = 0;
  }

  // ---- general path: radix select on the keys --------------------------------------------
  if (tid == 0) {
    s_prefix = 0u;
    s_remaining = k;
  }
  uint32_t mask = 0u;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 24 : (pass == 1 ? 12 : 0);
    const uint32_t dmask = pass == 0 ? 0xffu : 0xfffu;
    // pass 0: one histogram of 256 bins per warp (8192 ints); passes 1 and 2: one of 4096 bins
    int4* h4 = reinterpret_cast<int4*>(hist);
    __syncthreads();
    const int nz = (pass == 0 ? NW * 256 : 4096) / 4;
    for (int i = tid; i < nz; i += T) h4[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    const uint32_t prefix = s_prefix;
    const int remaining = s_remaining;
    int* my_hist = pass == 0 ? hist + wid * 256 : hist;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const uint32_t key = order_key(zb[j]);
      const bool in = tid + T * j < M && (key & mask) == prefix;
      // lanes with the same digit add once
      const uint32_t d = in ? (key >> shift) & dmask : 0xffffffffu;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      if (in && lane == __ffs(peers) - 1) atomicAdd(&my_hist[d], __popc(peers));
    }
    __syncthreads();
    // the bin of the remaining-th largest key: thread t takes the highest bins not taken by the threads below it
    constexpr int BPP = 4096 / T;
    int c[BPP];
#pragma unroll
    for (int i = 0; i < BPP; ++i) c[i] = 0;
    int top;
    if (pass == 0) {
      top = 255 - tid;
      if (tid < 256) {
#pragma unroll 8
        for (int w = 0; w < NW; ++w) c[0] += hist[w * 256 + top];
      }
    } else {
      top = 4095 - BPP * tid;
#pragma unroll
      for (int i = 0; i < BPP; ++i) c[i] = hist[top - i];
    }
    int mine = 0;
#pragma unroll
    for (int i = 0; i < BPP; ++i) mine += c[i];
    const int above = block_inclusive_scan<T>(mine, wsum, lane, wid) - mine;  // keys with a higher digit
    if (above < remaining && remaining <= above + mine) {  // exactly one thread
      int acc = above, bin = top, cnt = c[0];
#pragma unroll
      for (int i = 0; i < BPP - 1; ++i) {
        if (remaining > acc + c[i] && bin == top - i) {
          acc += c[i];
          bin = top - i - 1;
          cnt = c[i + 1];
        }
      }
      s_prefix = prefix | ((uint32_t)bin << shift);
      s_remaining = remaining - acc;
      s_bin_count = cnt;
    }
    mask |= dmask << shift;
    __syncthreads();
  }

  const uint32_t thr = s_prefix;   // key of the k-th largest element
  const int admit = s_remaining;   // how many keys equal to thr are taken, lowest index first
  const bool surplus = s_bin_count > admit;  // more keys equal to thr than fit: rank them by index

  if (surplus) {  // block-uniform: ranks of the equal keys in index order
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const int w = wid + NW * j;
      const uint32_t eq = __ballot_sync(0xffffffffu, tid + T * j < M && order_key(zb[j]) == thr);
      if (lane == 0 && w < W) wsm[w] = __popc(eq);
    }
    block_exclusive_scan(wsm, W, hist);
  }
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int w = wid + NW * j;
    const bool valid = tid + T * j < M;
    const uint32_t key = order_key(zb[j]);
    const uint32_t gt = __ballot_sync(0xffffffffu, valid && key > thr);
    const uint32_t eq = __ballot_sync(0xffffffffu, valid && key == thr);
    if (lane == 0 && w < W) {
      put(w, gt | (surplus ? lowest_bits(eq, admit - wsm[w]) : eq));
    }
  }
}

template <int T, int KPT>
static cudaError_t topk_launch(const Dims& d, const float* logits, int B, uint32_t* bitmap, uint32_t* bitmap2, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.L, B);
  cfg.blockDim = dim3(T);
  cfg.dynamicSmemBytes = (size_t)d.W * 4;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // its prologue overlaps the predictor's tail
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_topk<T, KPT>, logits, bitmap, bitmap2, d.L, d.M, d.k, B > 1 ? 1 : 0);
}

cudaError_t launch_topk(const Dims& d, const float* logits, int B, uint32_t* bitmap, uint32_t* bitmap2, bool cleared,
                        cudaStream_t s, int sm_count) {
  if (B > 1 && !cleared) {
    const size_t bytes = (size_t)d.L * d.W * 4;
    cudaError_t e = cudaMemsetAsync(bitmap, 0, bytes, s);
    if (e == cudaSuccess && bitmap2) e = cudaMemsetAsync(bitmap2, 0, bytes, s);
    if (e != cudaSuccess) return e;
  }
  // More jobs than SMs: blocks of 512 threads, of which two share an SM's registers where one of 1024 fills them; a job is a
  // chain of block-wide steps, and two chains side by side take little longer than one (np_predict for sixteen sequences of
  // the 7B shape, 512 jobs: 82 us against 86).  With a job per SM at most the wider block is the shorter chain (one
  // sequence on its own: 79 us against 83).
  if (d.L * B > sm_count) {
    const int kpt = (d.M + 511) / 512;
    if (kpt <= 12) return topk_launch<512, 12>(d, logits, B, bitmap, bitmap2, s);
    if (kpt <= 22) return topk_launch<512, 22>(d, logits, B, bitmap, bitmap2, s);
    if (kpt <= 28) return topk_launch<512, 28>(d, logits, B, bitmap, bitmap2, s);
  }
  const int kpt = (d.M + 1023) / 1024;
  if (kpt <= 12) return topk_launch<1024, 12>(d, logits, B, bitmap, bitmap2, s);
  if (kpt <= 16) return topk_launch<1024, 16>(d, logits, B, bitmap, bitmap2, s);
  if (kpt <= 28) return topk_launch<1024, 28>(d, logits, B, bitmap, bitmap2, s);
  if (kpt <= 40) return topk_launch<1024, 40>(d, logits, B, bitmap, bitmap2, s);
  return cudaErrorInvalidValue;  // d_ffn > 40960 is rejected by np_init
}

}  // namespace npi
