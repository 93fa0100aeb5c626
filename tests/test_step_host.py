"""Rules the step kernels must keep that no GPU run shows when they are broken
(the hardware may still do the expected thing), checked on the CPU: functions of
the kernels' source, compiled for the host with stand-ins for the device."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1802_01272_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _function(text, name):
    """The definition of the function `name`, from its template line (if any) to its last brace."""
    m = re.search(r"^(?:template <[^\n]*>\n)?[^\n/]*\b%s\(" % re.escape(name), text, re.M)
    assert m, name
    depth = 0
    for i in range(text.index("{", m.start()), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[m.start():i + 1]
    raise AssertionError(name)


def _run(tmp_path, code):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(code)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


@pytest.mark.parametrize("regu", ["false", "true"])
def test_register_exchange_is_one_instruction_per_warpgroup(tmp_path, regu):
    """setmaxnreg.aligned: the four warps of a warpgroup execute the same instruction, so
    every one of them comes to the same place of stream_roles; and each role gets its own."""
    code = r"""
#include <cstdio>
#define __device__
#define __forceinline__ inline
struct { int x; } threadIdx;
int __shfl_sync(unsigned, int v, int) { return v; }
struct Feed {};
template <typename ST> struct StreamSmem {};
template <bool REGU> struct StreamRegs { enum { LAUNCH = 1, ADVECT = 2, COLLIDE = 3 }; };
int place, amount, role;
template <int FROM, int TO> void role_registers(int line = __builtin_LINE()) { place = line; amount = TO; }
template <typename ST, bool V, bool D, bool R, typename F>
void collide_role(F, const StreamSmem<ST>&, int w, double&) { role = 40 + w; }
template <int SX, int O, int L, typename ST, bool V, typename F>
void advect_role(F, const StreamSmem<ST>&, int w) { role = 10 * (SX > 0) + w; }
""" + _function(_source("step_stream.cuh"), "stream_roles") + r"""
int main() {
  StreamSmem<float> S;
  double m = 0;
  for (int t = 0; t < 256; t += 32) {
    threadIdx.x = t;
    stream_roles<2, 0, float, true, false, REGU>(Feed(), S, m);
    printf("%d %d %d\n", place, amount, role);
  }
}
""".replace("REGU", regu)
    warps = [tuple(map(int, s.split())) for s in _run(tmp_path, code).splitlines()]
    assert len(warps) == 8
    assert len({w[0] for w in warps[:4]}) == 1 and len({w[0] for w in warps[4:]}) == 1, warps
    assert [w[1] for w in warps] == [2] * 4 + [3] * 4
    # quadrants (+,+), (-,+), (-,-), (+,-): the sign of xi_x of each advect warp
    assert [w[2] for w in warps] == [10, 1, 2, 13, 40, 41, 42, 43]


def test_wait_gives_a_warp_one_answer(tmp_path):
    """stream_wait on 32 threads as the lanes of a warp, each with its own clock and its own view
    of the barrier: whatever mix of completions and timeouts the lanes see, all return the same;
    a timeout is reported, and a warp that saw the phase complete in every lane goes on."""
    code = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include <pthread.h>
#define __device__
#define __forceinline__ inline
constexpr unsigned WAIT_NS = 1000000000u;
int scenario;
thread_local int lane, polls;
thread_local unsigned long long clock_ns;
std::atomic<int> seen;
std::atomic<unsigned> errors;
pthread_barrier_t gate;
// 0: complete at once; 1: complete later; 2: never; 3: lane 7's clock runs out, the others then
// see the phase complete; 4: lane 0 sees it at the first poll, the others never
bool bar_try_wait(unsigned, unsigned) {
  ++polls;
  switch (scenario) {
    case 0: return true;
    case 1: return polls > 5;
    case 2: return false;
    case 3:
      if (lane != 7) while (!errors.load()) std::this_thread::yield();
      return lane != 7;
    default: return lane == 0;
  }
}
unsigned long long global_ns() { return clock_ns += (scenario == 3 && lane == 7 ? 600000000ull : 100000000ull); }
void atomicOr(unsigned*, unsigned v) { errors |= v; }
bool __all_sync(unsigned, bool v) {
  if (v) ++seen;
  pthread_barrier_wait(&gate);
  return seen.load() == 32;
}
""" + _function(_source("step_stream.cuh"), "stream_wait") + r"""
int main() {
  for (scenario = 0; scenario < 5; ++scenario) {
    int abort = 0;
    unsigned err = 0;
    bool got[32];
    seen = 0;
    errors = 0;
    pthread_barrier_init(&gate, nullptr, 32);
    std::vector<std::thread> warp;
    for (int l = 0; l < 32; ++l)
      warp.emplace_back([&, l] { lane = l; got[l] = stream_wait(0, 0, &abort, &err); });
    for (auto& t : warp) t.join();
    int n = 0;
    for (bool g : got) n += g;
    printf("%d %d %u\n", n, abort, errors.load());
  }
}
"""
    got = [tuple(map(int, s.split())) for s in _run(tmp_path, code).splitlines()]
    assert got == [(32, 0, 0), (32, 0, 0), (0, 1, 2), (0, 1, 2), (0, 1, 2)], got


@pytest.mark.parametrize("name", ["lbm_kernels.cuh", "pair_node.cuh", "step_stream.cuh",
                                  "step_split64.cuh"])
def test_dependently_launched_kernels_read_coherently(name):
    """A step's kernel is on the device while the one before it still writes the buffers it will
    read.  A non-coherent load is only defined on data that nothing writes during the kernel, and
    may be moved before the wait for the previous kernel: none in these sources."""
    code = re.sub(r"//[^\n]*", "", _source(name))
    assert re.findall(r"__ldg\b|ld\.global\.(?:\w+\.)*nc\b|__restrict__", code) == []
