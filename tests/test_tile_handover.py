"""A tile is handed on with a release: the fence of the thread that gives it up
comes before the atomic that names it free, or the next visitor may load older
values of the tile's cells than the last one stored and store over them.  The
order of the accesses, without a GPU: the hand-over itself runs on the host with a
recording fence and atomic; the kernels are read."""
import re

import pytest

from . import device_fragments as frag

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#define __device__
#define __forceinline__ inline
struct Ctl { int x; };
struct SolveParams { unsigned long long *state; Ctl *ctl; };
enum { kStIdle = 0, kStQueued = 1, kStRunning = 2, kStDirty = 3 };
enum { kEtimeout = 1 };
static std::string ops;
static unsigned long long late = 0;     // written by another thread before the first CAS
static void fence_ar() { ops += "F"; }
static void raise_status(Ctl *, unsigned, unsigned long long) { ops += "!"; }
static unsigned long long atomicCAS(unsigned long long *p, unsigned long long old, unsigned long long v) {
  if (late) { *p = late; late = 0; }
  const unsigned long long was = *p;
  if (was == old) { *p = v; ops += "C"; }
  return was;
}
FUNCTIONS
int main(int, char **argv) {
  unsigned long long state[2] = {make_state(kStRunning, 0, 0), make_state(kStRunning, 0, 0)};
  SolveParams p{state, nullptr};
  if (argv[1][0] == 'd') late = make_state(kStDirty, 7, 0x15);
  const int r = end_visit(p, 0);
  std::printf("%s %x %d\n", ops.c_str(), r, (int)state_of(state[0]));
}
"""


@pytest.mark.parametrize("case,want", [("idle", "FC 0 0"), ("dirty", "FCF 115 2")])
def test_end_visit_releases(tmp_path, case, want):
    text = frag.source("eik_sched.cuh")
    heads = ["__device__ __forceinline__ unsigned long long make_state(",
             "__device__ __forceinline__ unsigned long long state_of(",
             "__device__ __forceinline__ unsigned faces_of(",
             "__device__ __forceinline__ int end_visit("]
    out = frag.run(tmp_path, PROGRAM.replace("FUNCTIONS", "\n".join(frag.block(text, h) for h in heads)), case)
    assert out.stdout.strip() == want, out


@pytest.mark.parametrize("name", ["eik_front.cu", "eik_guided.cu"])
def test_kernels_end_visits_that_way(name):
    text = frag.source(name)
    assert "end_visit(" in text
    assert not re.search(r"atomicCAS\(&\w+\.state", text)


@pytest.mark.parametrize("name,call", [("eik_front.cu", "activate(p,"), ("eik_guided.cu", "activate(p,"),
                                       ("eik_adjoint.cu", "        activate(sp,"),
                                       ("eik_adjoint.cu", "finish_tile(sp,")])
def test_fence_after_the_last_barrier(name, call):
    """Another lane's stores are covered only by a fence of the thread itself after
    the barrier between them."""
    text = frag.source(name)
    before = text[:text.index(call)]
    assert before.rfind("fence_ar();") > before.rfind("__syncwarp();")


def test_adjoint_mask_bytes_are_stored_as_they_are_read():
    """Visits of neighbouring tiles read the bytes while this one sets them: both
    sides relaxed, neither plain."""
    kernel = frag.block(frag.source("eik_adjoint.cu"), "adj_tiles_kernel(")
    assert "ld_rlx_u8(mask" in kernel and "st_rlx_u8(mask" in kernel
    assert not re.search(r"\bmask\[[^\]]*\]\s*[|&^]?=[^=]", kernel)
