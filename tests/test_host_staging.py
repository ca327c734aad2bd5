"""The context's staging memory (csrc/thor_staging.h) where page-locked memory cannot be had: runs and
grid creation go on through ordinary memory instead of being refused, page-locked memory is used
again once there is some, none is locked for a context of few calls, every block is freed once, no
block in use is freed before its copies are waited for, and a call that fails half way waits for
its own."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cassert>
#include <cstdio>
#include <cstring>
#include "thor_staging.h"
static int live = 0, allow = 0, drains = 0;
static bool lock(void** p, std::size_t n) { if (!allow) return false; ++live; *p = std::malloc(n); return true; }
static void unlock(void* p) { --live; std::free(p); }
int main() {
  auto drain = []() { ++drains; };
  {
    thor::HostStaging s(lock, unlock, 1 << 20);
    for (int i = 0; i < thor::HostStaging::kPlain; ++i) assert(!s.locked(100, drain));
    assert(!s.locked(100, drain));                   // none to be had
    char* a = (char*)s.any(100, drain);
    assert(a); std::memset(a, 1, 100);
    assert(s.any(50, drain) == a);                   // kept
    char* b = (char*)s.any(100000, drain);
    assert(b && drains >= 1); std::memset(b, 2, 100000);
    char* big = (char*)s.any((1 << 20) + 8, drain);  // beyond the page-locked limit
    assert(big); std::memset(big, 3, (1 << 20) + 8);
    allow = 1;
    char* c = (char*)s.any(100, drain);
    assert(c && live == 1 && c == s.locked(16384, drain));
    std::memset(c, 4, 16384);
    drains = 0;
    assert(s.locked(20000, drain) && drains == 1 && live == 1 && s.locked(32768, drain) && drains == 1);
    allow = 0;
    assert(!s.locked(40000, drain) && live == 0 && s.any(40000, drain));
    allow = 1;
    assert(s.any(40000, drain) && live == 1 && !s.locked((1 << 20) + 1, drain) && s.locked(1 << 20, drain));
  }
  assert(live == 0);
  {  // nothing is locked for a context of few calls
    thor::HostStaging s(lock, unlock, 1 << 20);
    for (int i = 0; i < thor::HostStaging::kPlain; ++i) assert(s.any(100, drain) && live == 0);
    assert(s.any(100, drain) && live == 1);
  }
  assert(live == 0);
  drains = 0;
  auto call = [&](int fails_at) {  // a call that fails at step 0, 1 or 2, or not at all
    if (fails_at == 0) return 1;   // nothing in flight yet
    thor::DrainGuard g(drain);
    if (fails_at == 1) return 2;
    if (fails_at == 2) return 3;
    g.done();
    return 0;
  };
  assert(call(0) == 1 && drains == 0);
  assert(call(1) == 2 && drains == 1 && call(2) == 3 && drains == 2);
  assert(call(3) == 0 && drains == 2);
  std::puts("ok");
}
"""


def test_ordinary_memory_where_none_can_be_locked(tmp_path):
    cc = shutil.which("g++") or shutil.which("c++")
    if cc is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([cc, "-std=c++17", "-Wall", "-Werror", "-fsanitize=address,undefined", "-I",
                    os.path.join(ROOT, "paper_2507_11603_gb300", "csrc"), str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "ok\n"


def test_runs_and_grids_use_the_fallback():
    """Only callers with a fallback of their own ask for page-locked memory alone."""
    with open(os.path.join(ROOT, "paper_2507_11603_gb300", "csrc", "thor_capi.cu")) as f:
        calls = [line.strip() for line in f if "ctx->pinned(" in line]
    assert calls == ["double* h_out = (double*)ctx->pinned(ob);"]


def test_no_copy_outlives_a_failed_call():
    """Calls that upload from the staging block drain the stream on every early return: the guard
    stands before the first copy, and is released only after the call's last synchronisation."""
    with open(os.path.join(ROOT, "paper_2507_11603_gb300", "csrc", "thor_capi.cu")) as f:
        text = f.read()
    for name in ("thor_run", "thor_reweight"):
        body = text[text.index(f'extern "C" int {name}(thor_ctx_t'):]
        body = body[:body.index("\n}\n")]
        guard, done = body.index("DrainGuard drain("), body.index("drain.done();")
        assert guard < body.index("cudaMemcpyAsync(") and done > body.rindex("cudaStreamSynchronize(s),")
        assert body.count("drain.done();") == 1
