"""The library's host bookkeeping (csrc/workspace.h) on devices that are counters: a workspace that
cannot grow keeps what it had; a kernel's shared-memory limit is raised once on every device."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2003_13245_gb300", "csrc")

HEAD = r'''
#include "workspace.h"
#include <cassert>
#include <cstdio>
#include <cstdlib>
#include <map>
enum Err { OK = 0, OOM = 2, BROKEN = 9 };
struct Device {
  std::size_t room, used = 0, most = 0;
  bool broken = false;
  std::map<void*, std::size_t> live;
  Err get(void** q, std::size_t n) {
    if (broken) return BROKEN;
    if (used + n > room) return OOM;
    *q = std::malloc(1);
    live[*q] = n;
    used += n;
    return OK;
  }
  void put(void* q) {
    assert(live.count(q));
    used -= live[q];
    live.erase(q);
    std::free(q);
  }
};
struct Block { void* p = nullptr; std::size_t bytes = 0; };
Err grow(Device& d, Block& b, std::size_t want) {
  return tdmrg::grow_block<Err>(b.p, b.bytes, want, [&](void** q, std::size_t n) { return d.get(q, n); },
                                [&](void* q) { d.put(q); }, [](Err e) { return e == OOM; });
}
'''

GROW = HEAD + r'''
int main() {
  {  // room for both: grows
    Device d{100};
    Block b;
    assert(grow(d, b, 30) == OK && b.bytes == 30);
    assert(grow(d, b, 60) == OK && b.bytes == 60 && d.used == 60 && d.live.size() == 1);
  }
  {  // no room for both, room for the larger one alone
    Device d{100};
    Block b;
    assert(grow(d, b, 50) == OK && grow(d, b, 90) == OK && b.bytes == 90 && d.used == 90);
  }
  {  // no room for the larger one: the old size stays
    Device d{100};
    Block b;
    assert(grow(d, b, 50) == OK && grow(d, b, 120) == OOM && b.p && b.bytes == 50 && d.used == 50);
  }
  {  // nothing at all
    Device d{10};
    Block b;
    assert(grow(d, b, 20) == OOM && !b.p && b.bytes == 0 && d.live.empty());
  }
  {  // another error: reported, the block untouched
    Device d{100};
    Block b;
    assert(grow(d, b, 50) == OK);
    d.broken = true;
    assert(grow(d, b, 60) == BROKEN && b.p && b.bytes == 50);
  }
  std::puts("ok");
  return 0;
}
'''


ONCE = r'''
#include "workspace.h"
#include <atomic>
#include <chrono>
#include <cassert>
#include <cstdio>
#include <thread>
#include <vector>
enum Err { OK = 0, BROKEN = 9, BAD = 7 };
int main() {
  tdmrg::OncePerDevice once;
  std::atomic<int> calls[3] = {{0}, {0}, {0}};
  assert(once.run(0, BAD, [&] { ++calls[0]; return OK; }) == OK);
  assert(once.run(0, BAD, [&] { ++calls[0]; return OK; }) == OK);
  assert(calls[0] == 1);
  // another device has its own, a failed one is tried again
  assert(once.run(1, BAD, [&] { ++calls[1]; return BROKEN; }) == BROKEN);
  assert(once.run(1, BAD, [&] { ++calls[1]; return OK; }) == OK);
  assert(once.run(1, BAD, [&] { ++calls[1]; return BROKEN; }) == OK);
  assert(calls[1] == 2);
  assert(once.run(-1, BAD, [] { return OK; }) == BAD && once.run(64, BAD, [] { return OK; }) == BAD);
  // several threads: nobody goes on before the one call is through
  std::vector<std::thread> t;
  std::atomic<bool> through{false};
  std::atomic<int> early{0};
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&] {
      once.run(2, BAD, [&] {
        ++calls[2];
        std::this_thread::sleep_for(std::chrono::milliseconds(20));
        through = true;
        return OK;
      });
      if (!through) ++early;
    });
  for (auto& x : t) x.join();
  assert(calls[2] == 1 && early == 0);
  std::puts("ok");
  return 0;
}
'''


def compile_and_run(tmp_path, text, extra=()):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text(text)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I" + CSRC, str(src), "-o",
                    str(tmp_path / "t"), *extra], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stderr


def test_a_workspace_that_cannot_grow_keeps_what_it_had(tmp_path):
    compile_and_run(tmp_path, GROW)


def test_once_per_device(tmp_path):
    compile_and_run(tmp_path, ONCE, ["-pthread"])


def test_shared_memory_limits_are_raised_per_device():
    """A limit raised with one flag for the process leaves the other devices without it."""
    for f in ("zgemm_digits.cu", "qr_tensor.cu"):
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        assert "static bool attr" not in text, f
        assert "static OncePerDevice" in text, f


def test_the_engine_goes_on_without_the_workspace():
    """Running out of memory for a digit workspace is no error of the engine: only `reserve` grows one,
    and it lets that error pass."""
    with open(os.path.join(CSRC, "engine.cu")) as fh:
        text = fh.read()
    assert "CK(zg_reserve" not in text
    assert text.count("zg_reserve(") == 1
    i = text.index("void Engine::reserve(")
    body = text[i:text.index("\n}", i)]
    assert "if (e != cudaErrorMemoryAllocation) CK(e);" in body


def test_the_workspaces_make_room_for_everything_else():
    """Every other allocation of an engine goes through `dev_alloc`, which gives the workspaces back
    before it fails."""
    for f in ("engine.cu", "step_adjoint.cu"):
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        if f == "engine.cu":            # the constructor and the MPO tables come before any workspace
            text = text[text.index("void Engine::ensure_workspace("):]
            i = text.index("void Engine::dev_alloc_bytes(")
            j = text.index("\n}", i)
            assert text[i:j].count("cudaMalloc(") == 2 and text[i:j].count("zg_free(") == 2
            text = text[:i] + text[j:]
        assert "cudaMalloc(" not in text, f
