"""A ring of slots that bulk copies fill, replayed on the host: the wait of csrc/np_ring.h over a model of its barriers, one warp that
fills it, readers that are held up elsewhere until the block's flag falls, copies that land in any order."""
import ctypes as C
import subprocess

import pytest

from paper_2608_22643_b200 import build as nbuild

_SOURCE = r"""
#include <random>
#include <utility>
#include <vector>
#include "np_ring.h"

namespace {
// An mbarrier: a phase completes when its arrivals are in and no bytes are on their way.  A wait names a parity and is over when
// the current phase has the other one.
struct Barrier {
  int count, pending, bytes = 0;
  uint32_t phase = 0;
  bool overrun = false;  // an arrival more than a phase has
  explicit Barrier(int n) : count(n), pending(n) {}
  void look() {
    if (pending == 0 && bytes == 0) pending = count, ++phase;
  }
  void arrive() {
    if (pending == 0) overrun = true;
    else --pending;
    look();
  }
  bool complete(uint32_t parity) const { return (phase & 1u) != parity; }
};

struct Reader {
  int use = 0;
  bool through = false;  // is behind its wait for the slot
  uint32_t polls = 0;
};

struct Block {
  std::mt19937 rng;
  int n, uses, held;
  bool up = true, lost = false;
  std::vector<Barrier> full, empty;
  std::vector<Reader> readers;
  std::vector<int> holds;                      // the use whose bytes are in a slot
  std::vector<std::pair<int, int>> under_way;  // (slot, use) of the copies
  int armed_over_copies = 0, read_wrong = 0;

  Block(unsigned seed, int n_, int readers_, int uses_, int held_)
      : rng(seed), n(n_), uses(uses_), held(held_), full(n_, Barrier(1)), empty(n_, Barrier(readers_)), readers(readers_), holds(n_, -1) {}

  // what the wait asks of a block
  bool stands() { return up; }
  void lower() { up = false; }
  void pause() {}
  bool given_up() { return lost; }
  void give_up() { lost = true; }
  bool wait_over(const Barrier& b, uint32_t parity, uint32_t& polls) {
    return b.complete(parity) || npp::ring_wait_step<4096>(polls, *this);
  }

  void reader(Reader& r) {
    if (r.use == uses) return;
    const int s = r.use % n;
    if (!r.through) {
      r.through = wait_over(full[s], (uint32_t)(r.use / n) & 1u, r.polls);
      if (r.through && holds[s] != r.use) ++read_wrong;
    } else if (r.use != held || !up) {  // held: something that does not come, until the flag falls
      empty[s].arrive();
      r = Reader{r.use + 1};
    }
  }
  void land() {
    if (under_way.empty()) return;
    std::swap(under_way[rng() % under_way.size()], under_way.back());
    const std::pair<int, int> c = under_way.back();
    under_way.pop_back();
    holds[c.first] = c.second;
    full[c.first].bytes -= 1;
    full[c.first].look();
  }
  // everybody but the warp that fills the ring, in any order and at any pace
  void others() {
    const unsigned slow = rng() % 3 == 0 ? 3 : 0;  // the copies, now and then
    for (unsigned k = rng() % 6; k > 0; --k) {
      const unsigned who = rng() % (readers.size() + 1 + slow);
      if (who < readers.size()) reader(readers[who]);
      else if (who == readers.size()) land();
    }
  }
  // a wait of another warp may run out at any time once a reader is held
  void run(int fall) {
    uint32_t par = 0;
    int slot = 0, step = 0;
    for (int u = 0; u < uses; ++u) {
      uint32_t polls = 0;
      do {
        others();
        if (++step == fall) up = false;
      } while (!wait_over(empty[slot], par ^ 1u, polls));
      others();
      for (const std::pair<int, int>& c : under_way) armed_over_copies += c.first == slot;
      full[slot].bytes += 3;
      full[slot].arrive();
      for (int k = 0; k < 3; ++k) under_way.push_back({slot, u});
      if (++slot == n) slot = 0, par ^= 1u;
    }
    // the end of the ring: the slots before `slot` in the use with parity `par`, the others in the one before
    for (int s = 0; s < n; ++s)
      for (int k = 0; k < 1000000 && !full[s].complete(s < slot ? par : par ^ 1u); ++k) others();
  }
};
}  // namespace

// out: slots armed over copies or barriers out of step, blocks left with copies under way, slots read before they were there, uses
// not read, rings given up
extern "C" void t_replay(int seeds, int n, int readers, int uses, int held, int fall, int* out) {
  for (int i = 0; i < 5; ++i) out[i] = 0;
  for (int seed = 0; seed < seeds; ++seed) {
    Block b((unsigned)seed, n, readers, uses, held);
    b.run(fall > 0 ? 1 + (int)((unsigned)seed * 2654435761u % (unsigned)fall) : -1);
    out[1] += !b.under_way.empty();
    for (int k = 0; k < 100000; ++k) b.others();
    out[0] += b.armed_over_copies;
    for (const Barrier& f : b.full) out[0] += f.overrun;
    for (const Barrier& e : b.empty) out[0] += e.overrun;
    out[2] += b.read_wrong;
    for (const Reader& r : b.readers) out[3] += uses - r.use;
    out[4] += b.lost;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = tmp_path_factory.mktemp("ring")
    src, so = str(out / "t.cpp"), str(out / "t.so")
    with open(src, "w") as f:
        f.write(_SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", nbuild.CSRC, src, "-o", so], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("slots,readers", [(2, 1), (3, 2), (4, 8), (11, 8), (32, 8)])
@pytest.mark.parametrize("held,fall", [(-1, 0), (-1, 60), (1, 0), (1, 200), (40, 2000)])
def test_ring_keeps_step(lib, slots, readers, held, fall):
    """No time-out; one at any moment; readers held up in a use until the wait for a free slot itself, or another one, runs out."""
    out = (C.c_int * 5)()
    lib.t_replay(50, slots, readers, 5 * slots + 1, held, fall, out)
    assert list(out) == [0] * 5
