// Device memory of one context: blocks that are given back stay with the context, within a bound, and serve
// its later requests.  Host code without CUDA calls of its own: Api has `Error`, `ok`, `out_of_memory`, and
// the functions alloc(void**, size_t) -> Error and release(void*), so that it runs on a host stand-in too.
//
// Every use of a block is on the context's stream, so a block is taken over in stream order.
//
// What the pool holds beyond the live requests (free blocks, and the slack of blocks larger than their
// request) never exceeds `limit`: what a give would bring above it is released at once, a free block is not
// taken for a request that would leave more slack than that, and a failing allocation first gives back
// every free block.  Other users of the device (torch, further contexts) find the rest free.  Only
// between hold(true) and hold(false) do free blocks stay whatever their sum: for an upload that is about to
// ask for the same blocks again.
#pragma once
#include <cstddef>
#include <new>
#include <vector>

template <class Api>
class DevicePool {
 public:
  using Error = typename Api::Error;

  DevicePool(Api api, size_t limit) : api_(api), limit_(limit) {}
  ~DevicePool() {
    for (const Block& b : blocks_) api_.release(b.p);
  }
  DevicePool(const DevicePool&) = delete;
  DevicePool& operator=(const DevicePool&) = delete;

  // what an allocation takes of the device, which the bound counts: from 1 MiB on, whole pages of 2 MiB
  static size_t device_bytes(size_t bytes) {
    const size_t n = round_up(bytes, 512);
    return n < ((size_t)1 << 20) ? n : round_up(n, (size_t)2 << 20);
  }

  // a block of at least `bytes`; the smallest free one that fits without wasting more than half of it
  Error take(void** p, size_t bytes) noexcept {
    *p = nullptr;
    const size_t want = round_up(bytes, 512), cost = device_bytes(bytes);
    if (cost < bytes) return Api::out_of_memory;
    Block* best = nullptr;
    for (Block& b : blocks_)
      if (!b.live && b.bytes >= want && b.bytes / 2 <= want && slack_ + (b.cost - cost) <= limit_ &&
          (!best || b.bytes < best->bytes))
        best = &b;
    if (!best) {
      try {
        if (blocks_.size() == blocks_.capacity()) blocks_.reserve(2 * blocks_.size() + 64);
      } catch (const std::bad_alloc&) {
        return Api::out_of_memory;
      }
      void* q = nullptr;
      Error e = api_.alloc(&q, want);
      if (e != Api::ok && drop(0)) e = api_.alloc(&q, want);
      if (e != Api::ok) return e;
      blocks_.push_back({q, want, cost, 0, false});  // within the capacity
      best = &blocks_.back();
      free_ += cost;
    }
    best->live = true;
    best->used = cost;
    free_ -= best->cost;
    slack_ += best->cost - cost;
    *p = best->p;
    return Api::ok;
  }

  // the block back; p came from take
  void give(void* p) noexcept {
    for (Block& b : blocks_)
      if (b.p == p && b.live) {
        b.live = false;
        free_ += b.cost;
        slack_ -= b.cost - b.used;
        break;
      }
    if (!hold_) drop(limit_);
  }

  void hold(bool on) noexcept {
    hold_ = on;
    if (!on) drop(limit_);
  }

  size_t held() const { return free_ + slack_; }
  size_t slack() const { return slack_; }

 private:
  static size_t round_up(size_t bytes, size_t grain) { return (bytes + grain - 1) / grain * grain; }

  struct Block {
    void* p;
    size_t bytes, cost, used;  // of the block, on the device, of that the live request's
    bool live;
  };

  // releases free blocks, the largest first, while more than `keep` is held; whether any was
  bool drop(size_t keep) noexcept {
    bool any = false;
    while (held() > keep) {
      size_t big = blocks_.size();
      for (size_t k = 0; k < blocks_.size(); ++k)
        if (!blocks_[k].live && (big == blocks_.size() || blocks_[k].bytes > blocks_[big].bytes)) big = k;
      if (big == blocks_.size()) break;
      api_.release(blocks_[big].p);
      free_ -= blocks_[big].cost;
      blocks_[big] = blocks_.back();
      blocks_.pop_back();
      any = true;
    }
    return any;
  }

  Api api_;
  size_t limit_, free_ = 0, slack_ = 0;  // bytes of free blocks, of live blocks beyond their requests
  bool hold_ = false;
  std::vector<Block> blocks_;
};
