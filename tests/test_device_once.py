"""Kernel attributes belong to a device: they are set once on each, not once in a process (host code, no GPU needed)."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_01399_b200", "csrc")

PROGRAM = r'''
#include <stdio.h>
#include "device_once.h"
int main() {
  static quasar::DeviceOnce once;
  int runs = 0, fails = 0;
  auto work = [&] { ++runs; return 0; };
  const int devices[] = {0, 0, 1, 1, 0, 63, 63, 64, 64};   // (beyond 63 nothing is remembered: it runs each time)
  for (int d : devices)
    if (once.run(d, work) != 0) return 1;
  if (once.run(2, [&] { ++fails; return -5; }) != -5 || once.run(2, [&] { ++fails; return 0; }) != 0) return 2;
  if (once.run(2, [&] { ++fails; return 0; }) != 0) return 3;
  printf("%d %d", runs, fails);
  return 0;
}
'''


def test_work_runs_once_on_each_device_and_again_after_a_failure(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)], text=True) == "5 2"


ANSWERS = r'''
#include <stdio.h>
#include "device_once.h"
int main() {
  static quasar::DeviceAnswers<5> kept;
  int asked = 0, next = 0;
  auto ask = [&] { ++asked; return next; };
  if (kept.get(0, 2, ask) != 0 || asked != 1) return 1;                       // could not be had: not kept
  next = 33;
  if (kept.get(0, 2, ask) != 33 || kept.get(0, 2, ask) != 33 || asked != 2) return 2;
  next = 15;
  if (kept.get(0, 4, ask) != 15 || kept.get(0, 2, ask) != 33 || asked != 3) return 3;      // another question
  if (kept.get(1, 2, ask) != 15 || kept.get(0, 2, ask) != 33 || kept.get(1, 2, ask) != 15 || asked != 4) return 4;   // another device
  if (kept.get(63, 0, ask) != 15 || kept.get(63, 0, ask) != 15 || asked != 5) return 5;
  if (kept.get(64, 0, ask) != 15 || kept.get(64, 0, ask) != 15 || kept.get(-1, 0, ask) != 15 || asked != 8) return 6;   // beyond what is kept: each time
  printf("ok");
  return 0;
}
'''


def test_answers_are_kept_for_their_device_and_only_when_there_is_one(tmp_path):
    src, exe = tmp_path / "answers.cpp", tmp_path / "answers"
    src.write_text(ANSWERS)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)], text=True) == "ok"


def test_what_a_device_holds_at_once_is_asked_in_one_place():
    """clusters_at_once, which keeps answers only: a function of its own beside it once kept a failed question for the process."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            found += [name] * text.count("cudaOccupancyMaxActiveClusters")
    assert found == ["common.cuh"]


def test_no_kernel_sets_its_attributes_any_other_way():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            found += [name] * text.count("cudaFuncSetAttribute")
    assert found == ["common.cuh", "common.cuh"]      # allow_shared_memory: the size and the carveout
