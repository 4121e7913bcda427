"""The device memory pool of a context (csrc/device_pool.h) on a host stand-in for the device: after every
call the device holds no more than the live requests and the limit, requests that fit are served again without
the device, a failing allocation gives back the free blocks and is tried again, and nothing is lost."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>
#include "device_pool.h"
struct Device {
  std::map<void*, size_t> blocks;
  size_t used = 0, capacity = 0;
  long allocs = 0, failed = 0;
};
static size_t up(size_t n);
struct Fake {
  using Error = int;
  static constexpr int ok = 0, out_of_memory = 2;
  Device* d;
  int alloc(void** p, size_t n) {
    if (d->used + up(n) > d->capacity) { ++d->failed; return out_of_memory; }
    *p = std::malloc(1);
    d->blocks[*p] = n;
    d->used += up(n);
    ++d->allocs;
    return 0;
  }
  void release(void* p) {
    if (!d->blocks.count(p)) { std::puts("released twice or unknown"); std::exit(1); }
    d->used -= up(d->blocks[p]);
    d->blocks.erase(p);
    std::free(p);
  }
};
static size_t up(size_t n) { return DevicePool<Fake>::device_bytes(n); }  // whole pages
#define REQUIRE(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
int main() {
  for (unsigned seed = 0; seed < 200; ++seed) {
    std::mt19937 rng(seed);
    Device dev;
    dev.capacity = seed % 2 ? 40000000 : (size_t)-1 / 4;
    {
      const size_t limit = seed % 3 == 0 ? 0 : 1000000u << (seed % 5);
      DevicePool<Fake> pool(Fake{&dev}, limit);
      std::map<void*, size_t> live;
      size_t total = 0;
      bool hold = false;
      for (int k = 0; k < 600; ++k) {
        if (seed % 4 == 1 && k % 50 == 0) pool.hold(hold = !hold);
        if (live.empty() || rng() % 5 < (k % 200 < 120 ? 3u : 1u)) {
          const size_t n = (size_t)1 << (rng() % 23), bytes = n + rng() % n;
          void* p = &dev;
          const int e = pool.take(&p, bytes);
          if (e) {
            REQUIRE(!p && pool.held() == pool.slack() && dev.used + up(bytes) > dev.capacity);  // no free block left
            continue;
          }
          REQUIRE(p && !live.count(p) && dev.blocks.at(p) >= bytes);
          live[p] = up(bytes);
          total += up(bytes);
        } else {
          auto it = live.begin();
          std::advance(it, rng() % live.size());
          total -= it->second;
          pool.give(it->first);
          live.erase(it);
        }
        REQUIRE(dev.used == total + pool.held());  // nothing lost
        REQUIRE((hold ? pool.slack() : pool.held()) <= limit);  // the bound, at any time
      }
    }
    REQUIRE(dev.used == 0 && dev.blocks.empty());  // live blocks too
  }
  {  // the same requests again: no new device allocation while they fit the limit
    Device dev;
    dev.capacity = 1u << 30;
    DevicePool<Fake> pool(Fake{&dev}, 100000);
    void* p[3];
    for (int round = 0; round < 2; ++round) {
      REQUIRE(!pool.take(&p[0], 10000) && !pool.take(&p[1], 30000) && !pool.take(&p[2], 1));
      for (void* q : p) pool.give(q);
    }
    REQUIRE(dev.allocs == 3);
  }
  {  // held over: all blocks serve again, whatever the limit
    Device dev;
    dev.capacity = 1u << 30;
    DevicePool<Fake> pool(Fake{&dev}, 0);
    void *a, *b;
    REQUIRE(!pool.take(&a, 100 << 20) && !pool.take(&b, 10));
    pool.hold(true);
    pool.give(a), pool.give(b);
    REQUIRE(!pool.take(&b, 10) && !pool.take(&a, 99 << 20 | 1) && dev.allocs == 2);
    pool.give(b);
    pool.hold(false);
    REQUIRE(pool.held() == 0 && dev.used == up(100 << 20));
    pool.give(a);
    REQUIRE(dev.used == 0);
  }
  {  // a block serves half its size, not less; a request that fails gives the free blocks back first
    Device dev;
    dev.capacity = 102400;
    DevicePool<Fake> pool(Fake{&dev}, 102400);
    void *a, *b;
    REQUIRE(!pool.take(&a, 51200));
    pool.give(a);
    REQUIRE(!pool.take(&b, 25600) && b == a && pool.held() == 25600);
    pool.give(b);
    REQUIRE(!pool.take(&b, 25088) && dev.allocs == 2 && pool.held() == 51200);
    REQUIRE(!pool.take(&a, 76800) && dev.failed == 1 && pool.held() == 0);
    REQUIRE(pool.take(&a, 1024) == 2 && !a && pool.take(&a, (size_t)-1) == 2 && !a);
  }
  std::puts("ok");
}
"""


def test_pool_on_a_host_device(tmp_path):
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I" + os.path.join(ROOT, "paper_2402_02075_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
