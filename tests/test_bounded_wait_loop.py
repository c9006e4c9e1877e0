"""A wait of the attention kernels that runs out: it gives up after about two seconds, and every wait of the CTA after it
within a few probes, so that the kernel still ends.  No wait is made to run out on a GPU: the loop (csrc/bounded_wait.cuh) is compiled for
the host and driven by a clock and a probe of the test's own."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include "bounded_wait.cuh"
int main() {
  volatile int abort_word = 0;
  uint64_t now = 5;
  long probes = 0;
  const uint64_t kProbeNs = 20000;                       // a probe may park its thread this long
  auto clock = [&] { return now; };
  auto never = [&] { ++probes; now += kProbeNs; return false; };
  bool r = lynx::bounded_wait(never, clock, &abort_word);                       // runs out by itself
  std::printf("%d %d %ld %llu\n", r, (int)abort_word, probes, (unsigned long long)now);
  probes = 0; now = 5;
  r = lynx::bounded_wait(never, clock, &abort_word);                            // another wait of the CTA gave up before
  std::printf("%d %d %ld %llu\n", r, (int)abort_word, probes, (unsigned long long)now);
  probes = 0; now = 5; abort_word = 0;
  auto other = [&] { if (++probes == 100) abort_word = 1; now += kProbeNs; return false; };
  r = lynx::bounded_wait(other, clock, &abort_word);                            // one gives up during this wait
  std::printf("%d %d %ld %llu\n", r, (int)abort_word, probes, (unsigned long long)now);
  probes = 0; now = 5; abort_word = 0;
  auto late = [&] { now += kProbeNs; return ++probes == 1000; };
  r = lynx::bounded_wait(late, clock, &abort_word);                             // it comes after all
  std::printf("%d %d %ld %llu\n", r, (int)abort_word, probes, (unsigned long long)now);
  auto tick = [&] { return now += 100; };
  now = 0; abort_word = 0;
  lynx::land_after_abort(tick, &abort_word);                                    // nothing has given up: not a moment
  std::printf("%llu ", (unsigned long long)now);
  abort_word = 1;
  lynx::land_after_abort(tick, &abort_word);                                    // time for what is in flight
  std::printf("%llu\n", (unsigned long long)now);
}
"""


def test_waiting_loop(tmp_path):
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    alone, after, during, late = ([int(x) for x in line.split()] for line in out[:4])
    assert alone[:2] == [0, 1] and 2.0e9 <= alone[3] <= 2.1e9      # gives up after two seconds and says so
    assert after[:2] == [0, 1] and after[2] <= 16                  # within a few probes
    assert during[:2] == [0, 1] and during[2] <= 100 + 16          # within a few probes of the other's giving up
    assert late[:3] == [1, 0, 1000]
    untouched, landed = (int(x) for x in out[4].split())
    assert untouched == 0 and 1.0e6 <= landed <= 1.1e6


def test_memory_is_given_back_behind_what_is_in_flight():
    """The warps that issue copies and products arrive at a barrier behind their last one; tensor memory is released, and with it
    the CTA can end, behind that barrier and the pause."""
    for name, bar in (("attention_i8.cuh", r"named_bar\(9, C::kThreads\)"), ("attention_f16.cuh", r"named_bar\(5, C::kDoneThreads\)"),
                      ("attention_pipe.cuh", r"named_bar\(9, C::kDoneThreads\)")):
        code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        done, land, free = (re.search(x, code).start() for x in (bar, r"land_after_abort\(", r"tcgen05\.dealloc"))
        assert done < land < free
        assert re.search(bar.replace("named_bar", "bar_arrive"), code), "the producers arrive there"


def test_every_wait_of_the_kernels_goes_through_it():
    text = "".join(open(os.path.join(CSRC, n)).read() for n in ("attention.cu", "attention_i8.cuh", "attention_f16.cuh", "attention_pipe.cuh"))
    loops = re.findall(r"mbar_try_wait\(bar, parity\)", text)
    assert len(loops) == 3                                          # mbar_wait's own, and one in each bounded wait
    assert len(re.findall(r"\bbounded_wait\(", text)) == 2
