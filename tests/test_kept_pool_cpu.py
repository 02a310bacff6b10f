"""The workspaces that rtcc_nms keeps between calls (kept_pool.h), with a stand-in
workspace on the host: up to four per context, whatever other contexts hold or
held; workspaces of a context that is gone are dropped without being touched;
threads never share one."""
import os
import shutil
import subprocess

import pytest

from paper_2608_08330_gb300 import build as B

SOURCE = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <set>
#include <thread>
#include "kept_pool.h"

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

static std::atomic<int> made{0}, destroyed{0}, touched_dead{0};
static std::atomic<unsigned long long> dead{0};       // contexts with an id up to this are gone
static bool refuse = false;

struct Space {
  unsigned long long ctx = 0;
  std::atomic<int> users{0};
  bool create(unsigned long long id) { ctx = id; if (refuse) return false; ++made; return true; }
  void destroy() { if (gone()) ++touched_dead; ++destroyed; }
  bool gone() const { return ctx <= dead; }
};
using Pool = rtcc::KeptPool<Space, 4>;

// n calls at once in a context, all given back
static void calls(Pool& p, unsigned long long ctx, int n) {
  std::unique_ptr<Space> s[16];
  std::set<Space*> all;
  for (int i = 0; i < n; ++i) { s[i] = p.take(ctx); CHECK(s[i] && s[i]->ctx == ctx); all.insert(s[i].get()); }
  CHECK((int)all.size() == n);
  for (int i = 0; i < n; ++i) p.give(std::move(s[i]));
}

int main() {
  {
    Pool p;
    calls(p, 1, 6);                                   // six at once: four stay
    CHECK(made == 6 && destroyed == 2);
    calls(p, 1, 4);
    CHECK(made == 6 && destroyed == 2);
    // another context, the first one's four idle and alive: it keeps four of its own
    calls(p, 2, 4);
    CHECK(made == 10 && destroyed == 2);
    calls(p, 2, 4);
    calls(p, 1, 4);
    CHECK(made == 10 && destroyed == 2);
    // both are gone: their eight are dropped untouched, a new context keeps its own
    dead = 2;
    for (int i = 0; i < 10; ++i) calls(p, 3, 1);
    CHECK(made == 11 && destroyed == 2 && touched_dead == 0);
    // and so on over many resets
    for (unsigned long long c = 4; c < 200; ++c) {
      dead = c - 1;
      for (int i = 0; i < 5; ++i) calls(p, c, 4);
    }
    CHECK(made == 11 + 196 * 4 && destroyed == 2 && touched_dead == 0);
    refuse = true;
    CHECK(!p.take(1000));
    refuse = false;
  }
  {
    Pool p;
    std::thread t[8];
    for (int k = 0; k < 8; ++k)
      t[k] = std::thread([&p, k] {
        for (int i = 0; i < 20000; ++i) {
          auto s = p.take(1000 + k % 2);
          CHECK(s && s->users.fetch_add(1) == 0);
          s->users.fetch_sub(1);
          p.give(std::move(s));
        }
      });
    for (auto& x : t) x.join();
  }
  std::puts("ok");
  return 0;
}
"""


def test_kept_workspaces(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + os.path.abspath(B.CSRC), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
