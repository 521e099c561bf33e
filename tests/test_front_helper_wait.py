"""The front kernel's third warp waits for mail and for the end of the rounds with
votes of the whole warp.  Its 32 lanes run on the host as threads whose votes
meet at barriers and whose clocks differ, as they do on the device: mail is
delivered, the end is seen, a visit longer than timeout_ms is no fault, and the
limit, when it is reached, takes all lanes out together."""
import pytest

from . import device_fragments as frag

PROGRAM = r"""
#include <atomic>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
struct Ctl { int x; };
struct SolveParams { Ctl *ctl; long long timeout_ns; };
constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kEmpty = ~0ull;
constexpr unsigned kEtimeout = 3;
struct Lane { int x; };
thread_local Lane threadIdx;

// A collective: all 32 lanes must come to the same one; a lane that has left, or
// that waits at another, is a divergent exit.
std::mutex mu;
std::condition_variable cv;
int arrived = 0, gone = 0, kind = 0, set_any = 0, set_all = 1, from0 = 0;
int out_any, out_all, out0;
unsigned long generation = 0;
[[noreturn]] void divergent() { std::printf("divergent\n"); std::fflush(stdout); std::_Exit(0); }
int meet(int k, int v, int want) {
  std::unique_lock<std::mutex> lk(mu);
  if (gone) divergent();
  if (arrived == 0) { kind = k; set_any = 0; set_all = 1; }
  if (kind != k) divergent();
  set_any |= v != 0;
  set_all &= v != 0;
  if (threadIdx.x == 0) from0 = v;
  if (++arrived == 32) {
    arrived = 0; out_any = set_any; out_all = set_all; out0 = from0;
    ++generation;
    cv.notify_all();
  } else {
    const unsigned long g = generation;
    cv.wait(lk, [&] { return generation != g; });
  }
  const int r = want == 0 ? out_any : want == 1 ? out_all : out0;
  return r;
}
int __any_sync(unsigned, bool v) { return meet(1, v, 0); }
int __all_sync(unsigned, bool v) { return meet(2, v, 1); }
int __shfl_sync(unsigned, int v, int) { return meet(3, v, 2); }
void __threadfence_block() { std::atomic_thread_fence(std::memory_order_seq_cst); }
void __nanosleep(unsigned) {}
unsigned long long atomicExch(unsigned long long *p, unsigned long long v) {
  return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST);
}
unsigned raised = 0;
void raise_status(Ctl *, unsigned code, unsigned long long) { raised = code; }
// a clock of its own for each lane: a second per look and more
thread_local long long looks = 0;
volatile int fin = 0;
int looks_to_end = 0;
long long now_ns() {
  ++looks;
  if (threadIdx.x == 0 && looks == looks_to_end) fin = 1;
  return looks * (1000000000ll + threadIdx.x * 10000000ll);
}
FUNCTIONS
int main(int, char **argv) {
  looks_to_end = std::atoi(argv[1]);           // the rounds end after that many looks at the clock
  static unsigned long long mail[4] = {kEmpty, 5, kEmpty, 9};
  Ctl ctl;
  SolveParams p{&ctl, std::atoll(argv[2]) * 1000000ll};
  std::atomic<int> got{0};
  auto deliver = [&](unsigned set, unsigned long long m) { if (set) got += (int)m; };
  std::vector<std::thread> lanes;
  for (int k = 0; k < 32; ++k)
    lanes.emplace_back([&, k] {
      threadIdx.x = k;
      serve_mail(mail, &fin, p, deliver);
      std::lock_guard<std::mutex> lk(mu);
      ++gone;
      if (arrived) divergent();
    });
  for (auto &t : lanes) t.join();
  std::printf("mail %d status %u end %d\n", got.load(), raised, (int)fin);
}
"""


@pytest.mark.parametrize("looks,timeout_ms,want", [(2, 12000, "mail 14 status 0 end 1"),
                                                   (6, 1, "mail 14 status 0 end 1"),
                                                   (1000, 1, "mail 14 status 3 end 0"),
                                                   (1000, 12000, "mail 14 status 3 end 0")])
def test_helper_wait(tmp_path, looks, timeout_ms, want):
    text = frag.source("eik_front.cu")
    body = "constexpr long long kVisitNs" + text.split("constexpr long long kVisitNs", 1)[1].split(";", 1)[0] + ";\n"
    body += "template <class Deliver>\n" + frag.block(text, "__device__ __forceinline__ void serve_mail(")
    out = frag.run(tmp_path, PROGRAM.replace("FUNCTIONS", body), looks, timeout_ms)
    assert out.stdout.strip() == want, out
