"""A CTA may not exit while an arrival is on its way to one of its barriers.  The protocol of the GEMM's rings on the CPU: an
arrival counts as landed only once somebody has waited for the phase it completes.  After the owner's loop the last round
has no waiter; after drain_ring, the one the kernel calls, everything has landed, whatever the number of uses."""
import os
import re
import subprocess

from paper_2104_08378_b200 import build

HARNESS = r"""
#include <cstdio>
#include "sp24_gemm.cuh"
using namespace sp24;
struct Barrier {
  int sent = 0, landed = 0;                              // phases whose arrivals were sent, were waited for
  // as mbarrier.try_wait.parity: true for the phase before the current one; sees every arrival sent before it
  bool wait(uint32_t parity) {
    if (((uint32_t)(sent & 1) ^ 1u) != parity) return false;   // not complete: would block
    landed = sent;
    return true;
  }
};
int main() {
  for (int slots = 1; slots <= 12; ++slots)
    for (int uses = 0; uses <= 40; ++uses) {
      Barrier bars[12];
      int slot = 0, on_the_way = 0, left = 0, blocked = 0;
      uint32_t phase = 0;
      for (int u = 0; u < uses; ++u) {                   // the owner: wait for a free slot, use it; the user hands it back
        if (!bars[slot].wait(phase ^ 1u)) ++blocked;
        ++bars[slot].sent;
        if (++slot == slots) { slot = 0; phase ^= 1u; }
      }
      for (int s = 0; s < slots; ++s) on_the_way += bars[s].sent != bars[s].landed;
      if (!drain_ring(slots, slot, phase, [&](int s, uint32_t parity) { return bars[s].wait(parity); })) ++blocked;
      for (int s = 0; s < slots; ++s) left += bars[s].sent != bars[s].landed;
      if (blocked || left || on_the_way != (uses < slots ? uses : slots)) {
        printf("slots %d uses %d: %d on the way, %d left, %d blocked\n", slots, uses, on_the_way, left, blocked);
        return 1;
      }
    }
  printf("ok");
}
"""


def test_nothing_is_on_its_way_after_drain_ring(tmp_path):
    src, exe = tmp_path / "harness.cu", tmp_path / "harness"
    src.write_text(HARNESS)
    subprocess.check_call([build._nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I",
                           f"{build._ROOT}/include", "-I", f"{build._HERE}/csrc", "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok"


def test_the_owners_of_a_pairs_rings_drain_them():
    """The producer (ring of stages) and the issuer (accumulators), the two whose barriers the other CTA arrives at."""
    text = open(os.path.join(build._HERE, "csrc", "sp24_gemm_kernel.cuh")).read()
    assert re.findall(r"if \(CTAS == 2 && !sh->abort\)\s+drain_ring\(([^,]+),", text) == ["p.stages", "C::kAccStages"]
