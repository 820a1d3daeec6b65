"""The datastore's 5-gram index where memory runs out while it is built: the host code is compiled with an allocator that fails at
the n-th request, for every n that building the index makes.  Whatever was refused, the index must be as it was, and the next
attempt must give all postings once and in order."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_13519_b200", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "drafter.h"
static long g_left = -1;   // requests until one fails, -1: none does
void *operator new(size_t n) {
  if (g_left == 0) { g_left = -1; throw std::bad_alloc(); }
  if (g_left > 0) --g_left;
  void *p = malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void *operator new(size_t n, const std::nothrow_t &) noexcept { return malloc(n ? n : 1); }
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }

static void add(ts_datastore &d, int len, unsigned &seed, int alphabet) {
  for (int i = 0; i < len; ++i) { seed = seed * 1664525u + 1013904223u; d.tokens.push_back((int)((seed >> 16) % alphabet)); }
  d.offset.push_back((int64_t)d.tokens.size());
  d.tool_of.push_back(0);
}
static const char *fault(const ts_datastore &d, size_t want) {
  if (d.index.size() != want) return "number of postings";
  for (size_t i = 1; i < want; ++i) {
    const auto &a = d.index[i - 1], &b = d.index[i];
    if (a.key > b.key || (a.key == b.key && (a.entry > b.entry || (a.entry == b.entry && a.m >= b.m)))) return "order";
  }
  return nullptr;
}
int main(int argc, char **argv) {
  const int entries[2] = {atoi(argv[1]), atoi(argv[2])};   // before and in the attempt that fails
  const int alphabet = atoi(argv[3]);
  int failed = 0;
  for (long n = 0;; ++n) {
    ts_datastore d;
    unsigned seed = 7;
    size_t want = 0;
    auto fill = [&](int count) {
      for (int e = 0; e < count; ++e) { const int len = 3 + e % 60; add(d, len, seed, alphabet); want += len > 5 ? len - 5 : 0; }
    };
    fill(entries[0]);
    d.ensure_index();
    const size_t before = want;
    fill(entries[1]);
    g_left = n;
    bool threw = false;
    try { d.ensure_index(); } catch (const std::bad_alloc &) { threw = true; }
    g_left = -1;
    if (threw) {
      ++failed;
      const char *f = fault(d, before);
      if (f) { printf("after request %ld failed: %s\n", n, f); return 1; }
      d.ensure_index();
    }
    const char *f = fault(d, want);
    if (f) { printf("request %ld, next attempt: %s\n", n, f); return 1; }
    if (!threw) break;
  }
  printf("requests %d\n", failed);
  return failed > 0 ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("index")
    (d / "main.cpp").write_text(HARNESS)
    exe = str(d / "index")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "main.cpp"),
                           os.path.join(CSRC, "drafter.cpp"), "-o", exe])
    return exe


# few postings and many (dealt out by their keys), into an empty index and a full one; 3 ids: the same 5-grams over and over
@pytest.mark.parametrize("before,then,alphabet", [(0, 20, 1000), (300, 20, 1000), (0, 300, 1000), (300, 400, 1000), (0, 300, 3), (50, 300, 3)])
def test_a_refused_allocation_leaves_the_index_as_it_was(harness, before, then, alphabet):
    r = subprocess.run([harness, str(before), str(then), str(alphabet)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
