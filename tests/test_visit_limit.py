"""The time limit of a visit in the kernel of explicit options, on the host: the end
of the look-ahead window, and none where the window reaches the last bucket.  That
bucket holds every later time, so with a limit a tile whose candidates lie beyond it
would be deferred to the same bucket and taken again without end."""
import re

import pytest

from . import device_fragments as frag

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#define __device__
#define __forceinline__ inline
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
static unsigned long long bits_of(double x) { unsigned long long u; std::memcpy(&u, &x, 8); return u; }
FUNCTIONS
// A visit at `lo` of a tile whose earliest candidate is at time t: accepted, or deferred
// to the bucket that the next visit has as its lowest.  Returns the visits it takes.
static long visits(unsigned lo, unsigned window, double delta, double t, long most) {
  for (long k = 1; k <= most; ++k) {
    if (bits_of(t) < visit_limit(lo, window, delta)) return k;
    const double q = t / delta;
    unsigned b = q < kMaxBucket ? (unsigned)q : kMaxBucket;
    if (b < lo + window + 1u) b = lo + window + 1u;
    if (b - lo >= 128u) b = lo + 127u;
    lo = b > kMaxBucket ? kMaxBucket : b;
  }
  return -1;
}
int main(int, char **v) {
  const unsigned lo = (unsigned)std::strtoul(v[1], nullptr, 10), window = (unsigned)std::strtoul(v[2], nullptr, 10);
  std::printf("%ld\n", visits(lo, window, 0.25, std::atof(v[3]), 1000));
}
"""
LAST = (1 << 30) - 1


@pytest.mark.parametrize("lo,window,t,want", [
    (0, 16, 4.0, 1), (0, 16, 4.25, 2), (0, 31, 7.99, 1), (0, 31, 8.0, 2),
    (LAST, 16, 1e15, 1), (LAST - 17, 16, 1e15, 2), (LAST - 16, 16, 1e15, 1), (LAST - 5, 1 << 30, 1e300, 1),
    (LAST, 1, 0.25 * LAST * 8, 1), (LAST - 1000, 31, 1e12, 9), (0, (1 << 31) - 1, 1e300, 1)])
def test_a_candidate_is_accepted_in_the_end(tmp_path, lo, window, t, want):
    text = frag.source("eik_solver.cu")
    last = re.search(r"constexpr uint32_t kMaxBucket = [^;]*;", frag.source("eik_internal.h")).group(0)
    body = last.replace("uint32_t", "unsigned") + "\n" + frag.block(
        text, "__device__ __forceinline__ unsigned long long visit_limit(")
    out = frag.run(tmp_path, PROGRAM.replace("FUNCTIONS", body), lo, window, t)
    assert out.stdout.strip() == str(want), out


def test_the_kernel_has_no_other_limit():
    text = frag.source("eik_solver.cu")
    assert len(re.findall(r"= visit_limit\(", text)) == 2
    assert not re.search(r"window \+ 1u\) \* s_delta", text)
