"""The ring of the star solves on the CPU: a host program takes the kernel's steps (copies asked
for, waits, slots reused) and gives up at every record in turn; the copies then waited for must
be those in flight, each by the phase its slot is in.  A wait for a copy that was never asked for
would run until its limit, a copy left out would land in memory of the next block."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_07488_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "star_ring.cuh"
using namespace spnet;
int main() {
  for (int nrec = 1; nrec <= 3 * SLOTS + 1; ++nrec)
    for (int stop = 0; stop < nrec; ++stop) {
      std::set<int> flight;
      int done[SLOTS] = {}, asked[SLOTS] = {};  // phases of each slot
      auto fetch = [&](int i) { flight.insert(i); ++asked[i % SLOTS]; };
      for (int i = 0; i < SLOTS && i < nrec; ++i) fetch(i);
      for (int rec = 0; rec < stop; ++rec) {  // the wait for rec ends, then the next copy is asked for
        flight.erase(rec);
        ++done[rec % SLOTS];
        if (rec > 0 && rec - 1 + SLOTS < nrec) fetch(rec - 1 + SLOTS);
      }
      for (int i = stop; i < ring_issued(stop, nrec); ++i) {
        if (!flight.count(i)) return printf("%d records, stop at %d: waits for %d\n", nrec, stop, i), 1;
        if (asked[i % SLOTS] != done[i % SLOTS] + 1 || ring_parity(i) != (unsigned)(done[i % SLOTS] & 1)) return printf("parity of %d\n", i), 1;
        flight.erase(i);
      }
      if (!flight.empty()) return printf("%d records, stop at %d: %d left in flight\n", nrec, stop, *flight.begin()), 1;
    }
  return 0;
}
"""


def test_a_block_that_gives_up_waits_for_the_copies_in_flight(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
