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


def test_every_wait_of_the_kernels_goes_through_it():
    text = "".join(open(os.path.join(CSRC, n)).read() for n in ("attention.cu", "attention_i8.cuh", "attention_f16.cuh"))
    loops = re.findall(r"mbar_try_wait\(bar, parity\)", text)
    assert len(loops) == 3                                          # mbar_wait's own, and one in each bounded wait
    assert len(re.findall(r"\bbounded_wait\(", text)) == 2
