"""A small library over the internal launch functions of libnp.so, compiled against the internal header, for tests that hand a
resident kernel its device words themselves."""
import ctypes as C
import os
import subprocess
import tempfile

from paper_2608_22643_b200 import build as nbuild

_SOURCE = r"""
#include "np_internal.h"
using namespace npi;
static Dims dims(int D, int C, int k, int L) {
  Dims d = {};
  d.L = d.Lp = L; d.D = D; d.M = C; d.H = 64; d.k = k; d.C = C; d.W = C / 32; d.Bmax = 16;
  return d;
}
// ptr: gate, up, downT, slots, counters, x (bf16), xbuf[2], zbuf[3], x_out, status, zfix, bars, xch
extern "C" int t_slices(int D, int C, int k, int L, int sms, void* const* ptr, unsigned int* base, void* stream) {
  const Dims d = dims(D, C, k, L);
  ChainArgs a = {};
  a.gate = ptr[0]; a.up = ptr[1]; a.downT = ptr[2];
  a.active_slots = static_cast<const int32_t*>(ptr[3]);
  a.counters = static_cast<const int32_t*>(ptr[4]);
  a.x_bf16 = ptr[5];
  for (int i = 0; i < 2; ++i) a.xbuf[i] = static_cast<float*>(ptr[6 + i]);
  for (int i = 0; i < 3; ++i) a.zbuf[i] = static_cast<float*>(ptr[8 + i]);
  a.x_out = static_cast<float*>(ptr[11]);
  a.status = static_cast<int32_t*>(ptr[12]);
  a.l_end = L;
  a.check = 1;
  chain_slices::State st = {};
  st.zfix = static_cast<unsigned long long*>(ptr[13]);
  st.bars = static_cast<unsigned int*>(ptr[14]);
  st.xch = static_cast<unsigned long long*>(ptr[15]);
  st.bar_base = base[0]; st.seq_base = base[1];
  const int e = (int)chain_slices::launch(d, a, &st, static_cast<cudaStream_t>(stream), sms);
  base[0] = st.bar_base; base[1] = st.seq_base; base[2] = (unsigned int)st.wrote_out;
  return e;
}
extern "C" int t_slices_supported(int D, int C, int k, int sms) { return chain_slices::supported(dims(D, C, k, 1), sms); }
extern "C" void t_slices_words(int D, int C, int k, int sms, unsigned long long* n) {
  const Dims d = dims(D, C, k, 1);
  n[0] = chain_slices::zfix_words(d); n[1] = chain_slices::bar_words(); n[2] = chain_slices::xch_words(d, sms);
}
// ptr: gate, up, downT, slots, counters, x (bf16 [B][D]), x as the kernel keeps it, result, status, cnt, xch
extern "C" int t_batch(int D, int C, int k, int L, int B, int sms, void* const* ptr, unsigned int* base, void* stream) {
  const Dims d = dims(D, C, k, L);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ChainArgs a = {};
  a.gate = ptr[0]; a.up = ptr[1]; a.downT = ptr[2];
  a.active_slots = static_cast<const int32_t*>(ptr[3]);
  a.counters = static_cast<const int32_t*>(ptr[4]);
  a.status = static_cast<int32_t*>(ptr[8]);
  a.l_end = L;
  a.check = 1;
  chain_batch::State st = {};
  st.cnt = static_cast<unsigned int*>(ptr[9]);
  st.xch = static_cast<unsigned long long*>(ptr[10]);
  st.read_base = base[0]; st.add_base = base[1]; st.seq_base = base[2];
  float* x = static_cast<float*>(ptr[6]);
  int n = 0;
  int e = (int)chain_batch::launch_in(d, ptr[5], x, B, s);
  if (!e) e = (int)chain_batch::launch(d, a, x, B, &st, s, sms, &n);
  if (!e) e = (int)chain_batch::launch_out(d, x, static_cast<float*>(ptr[7]), B, s);
  base[0] = st.read_base; base[1] = st.add_base; base[2] = st.seq_base;
  return e;
}
extern "C" int t_batch_record(unsigned int* base) {  // a launch that the caller knows to fail
  chain_batch::State st = {};
  st.read_base = base[0]; st.add_base = base[1]; st.seq_base = base[2];
  ChainArgs a = {};
  a.l_end = 3;
  int n = 0;
  const int e = (int)chain_batch::launch(dims(256, 512, 60, 3), a, nullptr, 4, &st, nullptr, 148, &n);
  base[0] = st.read_base; base[1] = st.add_base; base[2] = st.seq_base;
  return e;
}
// ptr: as for t_slices up to the status, then accumulators, counters; the result is in xbuf[(L - 1) & 1]
extern "C" int t_rows(int D, int C, int k, int L, int sms, void* const* ptr, unsigned int* base, void* stream) {
  const Dims d = dims(D, C, k, L);
  ChainArgs a = {};
  a.gate = ptr[0]; a.up = ptr[1]; a.downT = ptr[2];
  a.active_slots = static_cast<const int32_t*>(ptr[3]);
  a.counters = static_cast<const int32_t*>(ptr[4]);
  a.x_bf16 = ptr[5];
  for (int i = 0; i < 2; ++i) a.xbuf[i] = static_cast<float*>(ptr[6 + i]);
  for (int i = 0; i < 3; ++i) a.zbuf[i] = static_cast<float*>(ptr[8 + i]);
  a.status = static_cast<int32_t*>(ptr[12]);
  a.l_end = L;
  a.check = 1;
  chain_rows::State st = {};
  st.z4 = static_cast<float*>(ptr[13]);
  st.cnt = static_cast<unsigned int*>(ptr[14]);
  st.cnt_base = base[0]; st.seq = base[1];
  if (!chain_rows::prepare(d, sms, &st) || chain_rows::run_layers(d, st) < L) return -1;
  const int e = (int)chain_rows::launch(d, a, &st, static_cast<cudaStream_t>(stream));
  base[0] = st.cnt_base; base[1] = st.seq;
  return e;
}
extern "C" unsigned long long t_rows_words(int D) { return chain_rows::z_floats(dims(D, 1024, 1, 1)); }
extern "C" void t_batch_words(int sms, unsigned long long* n) {
  n[0] = chain_batch::cnt_words(); n[1] = chain_batch::xch_words(sms);
}
"""


def load():
    lib = nbuild.build()
    out = tempfile.mkdtemp(prefix="np_internals_")
    src, so = os.path.join(out, "t.cpp"), os.path.join(out, "t.so")
    with open(src, "w") as f:
        f.write(_SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(nbuild._nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", nbuild.CSRC, "-I", nbuild.INCLUDE, "-I", cuda, src,
                    lib, "-Wl,-rpath," + os.path.dirname(lib), "-o", so], check=True)
    return C.CDLL(so)


def uints(*v):
    return (C.c_uint * len(v))(*v)


def pointers(*v):
    return (C.c_void_p * len(v))(*v)
