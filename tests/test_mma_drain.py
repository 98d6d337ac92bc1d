"""The tensor-core M2L's MMA thread leaves with no MMA in flight, whichever of its waits runs out: tensor memory is freed
and shared memory given up right behind it.  Its branch of the kernel is compiled for the CPU with a model of the barriers,
since a wait that runs out cannot be brought about on a GPU without stopping it."""
import os
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_01334_gb300", "csrc", "m2l_tc.cuh")

MODEL = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
constexpr int TC_WAIT = 1, TC_ROWS = 128, TC_NST = 6, TC_WORKERS = 256;
struct Bar { int commits = 0; long covers = 0; };
std::map<uint64_t *, Bar> bars;  // by address: commits so far, MMAs that the last one covers
long issued = 0, waited = 0, fail_at, drained = 0;
namespace tc {
uint32_t smem_u32(const void *) { return 0; }
uint64_t sdesc(uint32_t) { return 0; }
uint32_t idesc_f16(int, int) { return 0; }
void fence_after() {}
void mma_f16(uint32_t, uint64_t, uint64_t, uint32_t, uint32_t) { ++issued; }
void commit(uint64_t *b) { Bar &x = bars[b]; ++x.commits; x.covers = issued; }
// the fail_at-th wait runs out; one for a barrier's last commit returns with all that it covers complete
bool mbar_wait(uint64_t *b, uint32_t parity, int) {
  if (waited++ == fail_at) return false;
  auto f = bars.find(b);
  if (f != bars.end() && parity == (uint32_t)((f->second.commits - 1) & 1)) drained = f->second.covers;
  return true;
}
}
int tc_stage_bytes(int) { return 0; }
int main(int argc, char **argv) {
  const int NC = atoi(argv[1]), ns = atoi(argv[2]), N = 32 * NC, NST = TC_NST, S = ns * NC;
  fail_at = atol(argv[3]);
  const uint32_t SA = 0, tmem = 0;
  uint64_t full[TC_NST], empty[TC_NST], accbar[2], foldbar[2], wfull[TC_NST], done;
  unsigned char smem[1], *sbase = smem;
  bool fail = false;
  const int tid = TC_WORKERS;
  (void)S; (void)SA; (void)done;
  if (tid < 0) {
  BRANCH
  }
  printf("%ld %ld %ld %d\n", issued, drained, waited, (int)fail);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    s = open(SRC).read()
    a = s.index("} else if (tid == TC_WORKERS) {")
    branch = s[a:s.index("} else if (tid == TC_WORKERS + 32) {", a)].replace("constexpr uint32_t IDESC", "const uint32_t IDESC")
    d = tmp_path_factory.mktemp("mma")
    (d / "m.cpp").write_text(MODEL.replace("BRANCH", branch))
    subprocess.run(["g++", "-std=c++17", "-w", "-o", str(d / "m"), str(d / "m.cpp")], check=True)
    return lambda *a: [int(v) for v in subprocess.run([str(d / "m")] + [str(v) for v in a], check=True,
                                                      capture_output=True, text=True).stdout.split()]


@pytest.mark.parametrize("nc", [1, 2, 3, 4])
def test_nothing_in_flight_after_any_timeout(program, nc):
    ns = 5
    issued, drained, waits, fail = program(nc, ns, -1)
    assert issued == 6 * nc * ns and drained == issued and not fail
    for k in range(waits - 1):  # the last wait is the one for the MMAs
        issued, drained, _, fail = program(nc, ns, k)
        assert fail and drained == issued, (k, issued, drained)
