"""The slots through which the resident step kernel's blocks exchange their sums: no block may find
its attempt's sums overwritten, however far the others run ahead.

A model of the exchange around the kernel's own index (res_slot), without any coupling between the
blocks but the sums: a block posts attempt k, then reads every block's slot until it carries k's tag,
then goes on to k + 1.  The schedules hold single blocks back as long as the others can move, and
draw the next block at random."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "internal.h"
using namespace pdlp;

static size_t one_set(unsigned tag, int reps, int replica, int G, int b) {
  return res_slot(0 * tag, reps, replica, G, b);
}

struct Block {
  int att = 0, read = -1;  // read: the next slot to read of this attempt, -1: not posted yet
};

// steps of one block until it waits or has finished; false: it found a newer attempt's sums
template <typename Slot>
static bool step(std::vector<Block>& B, std::vector<unsigned>& mem, int b, int G, int reps,
                 unsigned first, int attempts, bool* moved, Slot slot) {
  Block& q = B[b];
  *moved = false;
  if (q.att == attempts) return true;
  const unsigned tag = 2u * (first + (unsigned)q.att + 1u);
  if (q.read < 0) {
    for (int r = 0; r < reps; ++r) mem[slot(tag, reps, r, G, b)] = tag;
    q.read = 0;
    *moved = true;
    return true;
  }
  const unsigned seen = mem[slot(tag, reps, b & (reps - 1), G, 0) + q.read];
  if ((int)(seen - tag) > 0) return false;
  if (seen != tag) return true;
  *moved = true;
  if (++q.read == G) {
    ++q.att;
    q.read = -1;
  }
  return true;
}

template <typename Slot>
static int run(int G, int reps, unsigned first, int attempts, unsigned seed, Slot slot) {
  std::vector<Block> B(G);
  std::vector<unsigned> mem((size_t)kResSlotSets * reps * G, 2u * first);
  srand(seed);
  bool moved;
  // each block held back in turn for as long as any other can move
  for (int held = 0;; held = (held + 1) % G) {
    bool any = true;
    while (any) {
      any = false;
      for (int k = 0; k < G; ++k) {
        const int b = rand() % G;
        if (b == held) continue;
        if (!step(B, mem, b, G, reps, first, attempts, &moved, slot)) return 1;
        any |= moved;
      }
      for (int b = 0; b < G && !any; ++b) {
        if (b == held) continue;
        if (!step(B, mem, b, G, reps, first, attempts, &moved, slot)) return 1;
        any |= moved;
      }
    }
    for (int k = rand() % (2 * G); k >= 0; --k)
      if (!step(B, mem, held, G, reps, first, attempts, &moved, slot)) return 1;
    bool done = true;
    for (const Block& q : B) done &= q.att == attempts;
    if (done) return 0;
  }
}

int main() {
  int lost = 0, caught = 0, runs = 0;
  for (int G : {2, 3, 7, 33, 152})
    for (int reps : {4, 8, 16})
      for (unsigned first : {0u, 5u, 0x7ffffff0u}) {
        ++runs;
        // the slots stay within what is allotted, and no two (set, replica, block) share one
        std::vector<int> hits((size_t)kResSlotSets * reps * G, 0);
        for (unsigned a = 0; a < (unsigned)kResSlotSets; ++a)
          for (int r = 0; r < reps; ++r)
            for (int b = 0; b < G; ++b) {
              const size_t i = res_slot(2u * (first + a + 1u), reps, r, G, b);
              if (i >= hits.size() || hits[i]++) return printf("bad index\n"), 1;
            }
        lost += run(G, reps, first, 12, 1u + first + G, res_slot);
        caught += run(G, reps, first, 12, 1u + first + G, one_set);
      }
  printf("%d runs: %d lost, %d with a single set\n", runs, lost, caught);
  return 0;
}
"""


def test_no_sums_are_overwritten_before_they_are_read(tmp_path):
    from paper_2503_10344_gb300 import build as B
    src, exe = tmp_path / "slots.cu", tmp_path / "slots"
    src.write_text(PROGRAM)
    r = subprocess.run([B._nvcc(), "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                        "-I" + B.CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    runs, lost, single = (int(out.stdout.split()[i]) for i in (0, 2, 4))
    assert lost == 0, out.stdout
    assert single == runs, out.stdout  # (the model does find the fault of a single set)
