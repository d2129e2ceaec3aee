"""The streams beside a caller's (fan.h) against a stand-in for the runtime (no
GPU): work that cannot be ordered behind the caller's stream stays on it, a
stream in somebody else's capture or of another priority is not used, and the
caller's streams do not share side streams while there are enough."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <string>
#include <vector>
#include "fan.h"
struct Fake {
  using Stream = int;
  using Event = long;  // another type than Stream, for create() and destroy()
  struct Capture { bool active; unsigned long long id; };
  static inline int next = 100, dev = 0, live = 0, fail_wait = -1, fail_record = -1, synced = 0;
  static inline std::map<int, int> prio, cap;  // stream -> priority, capture id
  static inline std::vector<std::string> log;
  static void say(const char *what, int a, long b) { log.push_back(std::string(what) + " " + std::to_string(a) + " " + std::to_string(b)); }
  static bool device(int *d) { *d = dev; return true; }
  static bool priority(Stream s, int *p) { *p = prio[s]; return true; }
  static bool capture(Stream s, Capture *c) { c->active = cap[s] != 0; c->id = cap[s]; return true; }
  static bool create(Event *e) { *e = ++next; ++live; return true; }
  static bool create(Stream *s, int p) { *s = ++next; prio[*s] = p; ++live; return true; }
  static void destroy(Event) { --live; }
  static void destroy(Stream) { --live; }
  static bool record(Event e, Stream s) { if (s == fail_record) return false; say("record", s, e); return true; }
  static bool wait(Stream s, Event e) { if (s == fail_wait) return false; say("wait", s, e); return true; }
  static void synchronize(Stream) { ++synced; }
};
using namespace hs;
using Set = SideSet<Fake>;
using Fan = FanOf<Fake>;
static int bad = 0;
#define CHECK(x) do { if (!(x)) { ++bad; printf("line %d: %s\n", __LINE__, #x); } } while (0)
int main() {
  constexpr int M = 1, N = 2;
  Set a;
  CHECK(a.make(M));
  {  // forked behind the caller's stream, joined to it
    Fan f(M, 0xf, &a);
    CHECK(f.stream(0) == M && f.stream(1) == a.s[0] && f.stream(3) == a.s[2] && f.stream(1) == a.s[0]);
    CHECK(f.join());
    const std::vector<std::string> want = {
        "record 1 " + std::to_string(a.fork),
        "wait " + std::to_string(a.s[0]) + " " + std::to_string(a.fork),
        "wait " + std::to_string(a.s[2]) + " " + std::to_string(a.fork),
        "record " + std::to_string(a.s[0]) + " " + std::to_string(a.join[0]), "wait 1 " + std::to_string(a.join[0]),
        "record " + std::to_string(a.s[2]) + " " + std::to_string(a.join[2]), "wait 1 " + std::to_string(a.join[2])};
    CHECK(Fake::log == want);
  }
  Fake::log.clear();
  {  // a wait that fails: that group stays on the caller's stream
    Fake::fail_wait = a.s[1];
    Fan f(M, 0xf, &a);
    CHECK(f.stream(2) == M && f.stream(1) == a.s[0] && f.stream(2) == M);
    CHECK(f.join());
    for (const auto &x : Fake::log) CHECK(x.rfind("record " + std::to_string(a.s[1]), 0) != 0);
    Fake::fail_wait = -1;
  }
  {  // the fork itself fails, one group only, no set
    Fake::fail_record = M;
    Fan f(M, 0xf, &a);
    CHECK(f.stream(1) == M && f.join());
    Fake::fail_record = -1;
    Fan g(M, 4, &a), h(M, 0xf, nullptr);
    CHECK(g.stream(2) == M && h.stream(2) == M && g.join() && h.join());
  }
  {  // a join that fails is reported, and waited for on the host
    Fan f(M, 0xf, &a);
    f.stream(1);
    Fake::fail_wait = M;
    CHECK(!f.join() && Fake::synced == 1);
    Fake::fail_wait = -1;
  }
  {  // captures: one that the caller's stream takes part in is fine, another is not
    Fake::cap[M] = 7;
    Fan f(M, 0xf, &a);
    CHECK(f.stream(1) == a.s[0]);
    Fake::cap[a.s[0]] = 7;
    CHECK(f.join());
    Fan again(M, 0xf, &a);
    CHECK(again.stream(1) == a.s[0] && again.join());
    Fan eager(N, 0xf, &a);
    CHECK(eager.stream(1) == N && eager.stream(3) == N && eager.join());
    Fake::cap[N] = 8;
    Fan other(N, 0xf, &a);
    CHECK(other.stream(1) == N && other.join());
    Fake::cap.clear();
    Fan after(N, 0xf, &a);
    CHECK(after.stream(1) == a.s[0] && after.join());
  }
  {  // a caller's priority, another device
    Fake::prio[N] = -5;
    Fan f(N, 0xf, &a);
    CHECK(f.stream(1) == N);
    Set high;
    CHECK(high.make(N) && Fake::prio[high.s[0]] == -5 && Fake::prio[high.s[2]] == -5);
    Fan g(N, 0xf, &high);
    CHECK(g.stream(1) == high.s[0] && g.join());
    Fake::dev = 1;
    Fan h(M, 0xf, &a);
    CHECK(h.stream(1) == M);
    Fake::dev = 0;
  }
  {  // a thread's sets: one per stream, a bounded number, the oldest taken over, none of another priority
    const int before = Fake::live;
    {
      SidePool<Fake> pool;
      std::vector<Set *> of;
      for (int s = 10; s < 10 + SidePool<Fake>::MOST; ++s) of.push_back(pool.of(s));
      for (size_t i = 0; i < of.size(); ++i)
        for (size_t j = 0; j < i; ++j) CHECK(of[i] && of[i] != of[j]);
      CHECK(pool.of(10) == of[0] && pool.of(13) == of[3]);
      const int full = Fake::live;
      CHECK(pool.of(50) == of[1] && pool.of(11) == of[2] && Fake::live == full);
      CHECK(pool.of(N) == nullptr);  // all sets are of another priority
    }
    CHECK(Fake::live == before);
    SidePool<Fake> pool;
    Set *low = pool.of(10), *high = pool.of(N);
    CHECK(low && high && low != high && high->priority == -5 && pool.of(N) == high && pool.of(10) == low);
  }
  printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_side_streams_keep_the_callers_order(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "fan.cpp", tmp_path / "fan"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_1109_3739_gb300", "csrc")
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-I", csrc, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout
