"""Facts kept per CUDA context (csrc/context.cuh), compiled for the host with a context id of the test's
own: made once in every context, again after a failure, and once by many threads."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_01039_gb300", "csrc")
PROGRAM = r"""
#include "context.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
static thread_local uint64_t cur = 1;
uint64_t fpeps::context_id() { return cur; }
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  static fpeps::PerContext<int> per;
  int made = 0, v = 0;
  auto make = [&] { return 10 * (int)cur + made++; };
  CHECK(!per.peek(v));
  CHECK(per.get(make) == 10 && per.get(make) == 10 && made == 1);
  cur = 2;                                   // another device, or this one after a reset
  CHECK(!per.peek(v));
  CHECK(per.get(make) == 21 && per.get(make) == 21 && made == 2);
  cur = 1;
  CHECK(per.get(make) == 10 && made == 2 && per.peek(v) && v == 10);
  cur = 3;
  bool threw = false;
  try { per.get([]() -> int { throw 5; }); } catch (int) { threw = true; }
  CHECK(threw && !per.peek(v) && per.get(make) == 32);
  fpeps::PerContext<int> many;
  std::atomic<int> calls{0}, wrong{0};
  std::vector<std::thread> th;
  for (int t = 0; t < 8; ++t)
    th.emplace_back([&, t] {
      cur = 100 + t % 2;
      for (int i = 0; i < 1000; ++i) wrong += many.get([&] { ++calls; return (int)cur; }) != (int)cur;
    });
  for (auto& t : th) t.join();
  CHECK(calls == 2 && wrong == 0);
  return 0;
}
"""


def test_made_once_per_context(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe), "-pthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
