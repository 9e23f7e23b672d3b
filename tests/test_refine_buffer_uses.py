"""The refinement's counts of buffer uses (rf_uses in hfq_delayed.cuh, compiled
for the host): however many uses a sweep call makes, every use but a buffer's
first waits for the use before it, at the parity that the mbarrier has then.
The counts are 32 bits, so the walk goes past 2^32 uses.  No GPU is used."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0801_1222_gb300", "csrc")
OUT = os.path.join(HERE, "_build", "uses_probe")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "hfq_delayed.cuh"
using namespace hfq;
// Walks 2000 refinements of per uses from an exact count of n uses; the first
// wrong use, or -1.  plain: the count left to run, a mistake the walk must find
static long long first_wrong(unsigned long long n, uint32_t bufs, uint32_t per, bool plain) {
  uint32_t c = plain ? (uint32_t)n : rf_uses((uint32_t)n, bufs);
  for (int r = 0; r < 2000; ++r) {
    for (uint32_t k = 0; k < per; ++k) {
      const unsigned long long e = n + k;
      const uint32_t u = c + k;
      if (u % bufs != e % bufs || (u >= bufs) != (e >= bufs) || ((u / bufs) & 1u) != ((e / bufs) & 1u)) return (long long)e;
    }
    n += per;
    c = plain ? c + per : rf_uses(c + per, bufs);
  }
  return -1;
}
int main(int argc, char** argv) {
  const uint32_t bufs = atoi(argv[1]), per = atoi(argv[2]);
  const unsigned long long late = (1ull << 32) - 1000ull * per - 1;
  printf("%lld %lld %lld\n", first_wrong(0, bufs, per, false), first_wrong(late, bufs, per, false),
         first_wrong(late, bufs, per, true));
  return 0;
}
"""


@pytest.fixture(scope="module")
def probe():
    nvcc = os.environ.get("NVCC", "nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("nvcc not found")
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    with open(OUT + ".cu", "w") as f:
        f.write(SRC)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, "-o", OUT, OUT + ".cu"], check=True, capture_output=True)

    def run(bufs, per):
        r = subprocess.run([OUT, str(bufs), str(per)], check=True, capture_output=True, text=True)
        return [int(v) for v in r.stdout.split()]
    return run


# uses per refinement: K steps of 16 through four buffers at Lambda 16, 37, 240
# and 512; chunks of 32 through two stages at Lambda 16, 240 and 500
@pytest.mark.parametrize("bufs,per", [(4, 1), (4, 3), (4, 120), (4, 1024), (2, 1), (2, 8), (2, 64)])
def test_every_use_waits_for_the_one_before(probe, bufs, per):
    fresh, late, plain = probe(bufs, per)
    assert fresh == -1 and late == -1
    assert 1 << 32 <= plain < (1 << 32) + bufs
