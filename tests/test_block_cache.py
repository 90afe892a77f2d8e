"""The cache of freed device blocks (csrc/blocks.h) over a driver that is a
host program: what it hands out under stream capture, what it gives back when an
allocation fails, its bounds and sizes, several threads."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_07811_gb300", "csrc")

SOURCE = r"""
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <atomic>
#include <set>
#include <string>
#include <thread>
#include "blocks.h"

#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); exit(1); } } while (0)

struct Memory {  // one device
  std::mutex mu;
  size_t size, used = 0;
  std::map<char*, size_t> live;
  char* next = (char*)4096;
};

struct Fake final : BlockDevice {
  Memory* m;
  int no;
  bool cap = false;
  int settled = 0;
  std::vector<size_t> asked;
  Fake(Memory* mem, int id) : m(mem), no(id) {}
  int id() override { return no; }
  bool alloc(void** p, size_t n) override {
    std::lock_guard<std::mutex> lk(m->mu);
    asked.push_back(n);
    if (m->used + n > m->size) return false;
    m->used += n;
    m->live[m->next] = n;
    *p = m->next;
    m->next += n;
    return true;
  }
  void release(void* p) override {
    std::lock_guard<std::mutex> lk(m->mu);
    auto it = m->live.find((char*)p);
    CHECK(it != m->live.end());
    m->used -= it->second;
    m->live.erase(it);
  }
  bool capturing() override { return cap; }
  void settle() override { ++settled; }
};

const size_t MB = 1 << 20;

static void capture() {
  Memory m{{}, 1000 * MB};
  Fake d(&m, 0);
  BlockCache c(&d);
  void *before, *inside, *p;
  CHECK(c.alloc(&before, 1000));
  d.cap = true;
  CHECK(c.alloc(&inside, 1000));
  CHECK(d.asked.back() == 1000);  // a node of the graph, of the size asked for
  c.free(before);                 // a replay may still use it
  c.free(inside);                 // a node of the graph too
  CHECK(m.live.count((char*)before) && !m.live.count((char*)inside));
  d.cap = false;
  for (int i = 0; i < 4; ++i) {
    CHECK(c.alloc(&p, 1000));
    CHECK(p != before);
  }
  c.release();
  CHECK(m.live.count((char*)before));
  c.finish();
  CHECK(!m.live.count((char*)before));
  void* cached;
  CHECK(c.alloc(&cached, 2000));
  c.free(cached);
  d.cap = true;  // nothing cached goes into a graph
  CHECK(c.alloc(&p, 2000));
  CHECK(p != cached);
}

static void failure() {
  Memory m{{}, 100 * MB};
  Memory other{{}, 100 * MB};
  Fake a(&m, 0), b(&m, 0), g(&m, 0), o(&other, 1);
  BlockCache ca(&a), cb(&b), cg(&g), co(&o);
  void *p, *q;
  for (auto* c : {&ca, &cb, &cg, &co}) {
    CHECK(c->alloc(&p, 20 * MB));
    c->free(p);
  }
  g.cap = true;
  CHECK(m.used == 60 * MB && other.used == 20 * MB);
  CHECK(ca.alloc(&p, 79 * MB));  // asks for the blocks of a and b, not of the captured one or the other device
  CHECK(m.used == 99 * MB && other.used == 20 * MB);
  CHECK(b.settled == 1 && a.settled == 0 && g.settled == 0 && o.settled == 0);
  CHECK(!cb.alloc(&q, 2 * MB));
  ca.free(p);
  CHECK(m.used == 20 * MB);
  // the size itself where its class does not fit
  CHECK(cb.alloc(&p, 50 * MB));
  const size_t rest = 30 * MB - 1000;
  m.size = m.used + rest;
  CHECK(BlockCache::size_class(rest) > rest);
  CHECK(ca.alloc(&q, rest));
  CHECK(m.used == m.size);
  ca.free(q);  // not of a class's size: back to the driver
  CHECK(m.used == m.size - rest);
  // a context that has ended is not asked any more
  CHECK(ca.alloc(&q, 5 * MB));
  ca.free(q);
  ca.finish();
  const int n = a.settled;
  CHECK(!cb.alloc(&q, 60 * MB));
  CHECK(a.settled == n);
}

static void bounds() {
  Memory m{{}, (size_t)1 << 40};
  std::vector<Fake*> d;
  std::vector<BlockCache*> c;
  std::vector<std::pair<BlockCache*, void*>> v;
  void* p;
  for (int i = 0; i < 7; ++i) {
    d.push_back(new Fake(&m, 0));
    c.push_back(new BlockCache(d.back()));
    for (int k = 0; k < 20; ++k) {
      CHECK(c[i]->alloc(&p, 30 * MB));
      v.push_back({c[i], p});
    }
  }
  for (auto& x : v) x.first->free(x.second);
  CHECK(m.used <= BlockCache::kMaxTotal && m.used > BlockCache::kMaxTotal - 40 * MB);
  for (auto* x : c) x->finish();
  CHECK(m.used == 0);
  CHECK(c[0]->alloc(&p, 200 * MB + 1));  // above the largest cached block: as asked, and straight back
  CHECK(m.used == 200 * MB + 1);
  c[0]->free(p);
  CHECK(m.used == 0);
  for (size_t n = 1; n < ((size_t)1 << 34); n += 1 + n / 7) {
    const size_t k = BlockCache::size_class(n);
    CHECK(k >= n && BlockCache::size_class(k) == k);
    if (n > BlockCache::kMaxBlock) CHECK(k == n);
    else if (n > MB) CHECK(k - n <= n / 32);
    else if (n > 512) CHECK(k - n <= n / 8);
  }
}

static void threads() {
  Memory m{{}, 300 * MB};
  Fake d(&m, 0), e(&m, 0);
  BlockCache c(&d), f(&e);
  std::mutex mu;
  std::set<void*> held;
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&, i] {
      unsigned s = 77 + i;
      for (int k = 0; k < 3000; ++k) {
        s = s * 1664525u + 1013904223u;
        BlockCache& b = i & 1 ? c : f;
        void* p;
        if (!b.alloc(&p, 1 + (s >> 8) % (40 * MB))) continue;
        {
          std::lock_guard<std::mutex> lk(mu);
          CHECK(held.insert(p).second);  // nobody else has it
        }
        {
          std::lock_guard<std::mutex> lk(mu);
          held.erase(p);
        }
        b.free(p);
      }
    });
  for (auto& x : t) x.join();
  c.finish();
  f.finish();
  CHECK(m.used == 0);
}

int main(int, char** a) {
  const std::string w = a[1];
  if (w == "capture") capture();
  if (w == "failure") failure();
  if (w == "bounds") bounds();
  if (w == "threads") threads();
  puts("ok");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("blocks")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-pthread", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("what", ["capture", "failure", "bounds", "threads"])
def test_block_cache(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
