"""csrc/launch.h without a GPU: compiled against a stand-in for the CUDA runtime
whose current device and launch limit the test sets."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = """
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1,
                   cudaErrorCooperativeLaunchTooLarge = 82 };
inline int fake_device = 0;
inline int fake_cleared = 0;
inline cudaError_t cudaGetDevice(int* d) { *d = fake_device; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { ++fake_cleared; return cudaSuccess; }
"""


def _run(tmp_path, body):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    src = tmp_path / "t.cpp"
    src.write_text('#include "launch.h"\nint main() {\n' + body + "\nreturn 0;\n}\n")
    exe = tmp_path / "t"
    subprocess.check_call([gxx, "-std=c++17", "-Wall", "-Werror", "-I", str(tmp_path), "-I",
                           os.path.join(ROOT, "paper_2609_07204_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    return subprocess.run([str(exe)], timeout=60).returncode


def test_set_up_runs_once_on_each_device(tmp_path):
    assert _run(tmp_path, """
  static mc::OncePerDevice once;
  int runs = 0;
  auto good = [&] { ++runs; return true; };
  auto bad = [&] { ++runs; return false; };
  if (!once(good) || !once(good) || runs != 1) return 1;
  fake_device = 1;  // the second device of a process needs its own
  if (once(bad) || runs != 2) return 2;
  if (!once(good) || !once(good) || runs != 3) return 3;
  fake_device = 127;
  if (!once(good) || !once(good) || runs != 4) return 4;
  fake_device = 128;  // beyond what is remembered: every time
  if (!once(good) || !once(good) || runs != 6) return 5;
  fake_device = 0;
  if (!once(good) || runs != 6) return 6;
""") == 0


def test_refused_cooperative_launches_shrink(tmp_path):
    assert _run(tmp_path, """
  int tried = 0, last = 0, room = 0;
  auto launch = [&](int blocks) {
    ++tried;
    last = blocks;
    return blocks <= room ? cudaSuccess : cudaErrorCooperativeLaunchTooLarge;
  };
  for (room = 1; room <= 400; ++room) {
    tried = fake_cleared = 0;
    if (mc::launch_fitting(304, launch) != cudaSuccess || last > room || last < 1) return 1;
    if (last != 304 && 2 * last + 1 <= room) return 2;  // (halved no further than needed)
    if (fake_cleared != tried - 1) return 3;            // (each refusal is cleared)
  }
  room = 0;  // not even one block
  if (mc::launch_fitting(304, launch) != cudaErrorCooperativeLaunchTooLarge || last != 1) return 4;
  tried = 0;  // other errors are the caller's
  auto broken = [&](int) { ++tried; return cudaErrorInvalidValue; };
  if (mc::launch_fitting(304, broken) != cudaErrorInvalidValue || tried != 1) return 5;
""") == 0
