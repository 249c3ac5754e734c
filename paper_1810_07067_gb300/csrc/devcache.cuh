// Process-wide cache of freed device blocks, per device.  A build, a solve or a
// field evaluation takes tens of buffers, and a cudaMalloc, a cudaFree or the
// mapping of several GB costs tens of microseconds to milliseconds each (the
// N = 64 sphere: 1.5 of 7.5 ms); released blocks are handed out again for
// requests of the same rounded size on the same device.  Blocks of at least 64 MiB
// are rounded up to 2 MiB and kept up to a cap (32 GiB by default,
// mueller_cache_limit); smaller ones are rounded up to a quarter of their power of
// two and kept up to 256 MiB (none when the cap is 0); beyond its cap a kind gives
// up what was released longest ago.  A block belongs to the device that was current
// when it was allocated, whichever is current when it comes back (a context may be
// destroyed anywhere).  Releasing synchronizes each block's device first, once per
// group of buffers, as cudaFree does for each, so no kernel of any stream still uses
// a block when it is reused.  When an allocation fails the cache is emptied and the
// allocation retried; mueller_cache_trim empties it too.
//
// Api: the runtime calls (device, use, alloc, free, sync, clear_error), and Guard,
// held while blocks are freed or a device is synchronized.
#pragma once
#include <cstddef>
#include <iterator>
#include <list>
#include <mutex>
#include <vector>

struct DevBlock {
  void* p;
  size_t bytes;  // as requested by its user, rounded up in the cache
  int dev;
};

template <class Api>
class DeviceCache {
 public:
  static constexpr size_t kMinBlock = (size_t)64 << 20, kRound = (size_t)2 << 20, kSmallCap = (size_t)256 << 20;

  static size_t rounded(size_t b) {
    if (b >= kMinBlock) return (b + kRound - 1) / kRound * kRound;
    if (b <= 512) return 512;
    size_t q = 128;  // a quarter of the largest power of two up to b
    while (q * 8 <= b) q *= 2;
    return (b + q - 1) / q * q;
  }

  void trim() { shrink(0, 0); }

  // Sets the cap of the large blocks and returns the previous one.
  size_t limit(size_t bytes) {
    size_t old;
    {
      std::lock_guard<std::mutex> lk(mu_);
      old = cap_;
      cap_ = bytes;
    }
    shrink(bytes, bytes > 0 ? kSmallCap : 0);
    return old;
  }

  size_t bytes_held() {
    std::lock_guard<std::mutex> lk(mu_);
    return held_[0] + held_[1];
  }

  // A block of at least `bytes` on the current device.
  typename Api::Error alloc(DevBlock* b, size_t bytes) {
    const size_t req = rounded(bytes);
    const int kind = req >= kMinBlock ? 0 : 1;
    *b = DevBlock{nullptr, bytes, Api::device()};
    {
      std::lock_guard<std::mutex> lk(mu_);
      for (auto it = blocks_[kind].rbegin(); it != blocks_[kind].rend(); ++it)
        if (it->bytes == req && it->dev == b->dev) {
          b->p = it->p;
          held_[kind] -= req;
          blocks_[kind].erase(std::next(it).base());
          return Api::ok;
        }
    }
    auto e = Api::alloc(&b->p, req);
    if (e != Api::ok && bytes_held() > 0) {
      Api::clear_error();
      trim();
      e = Api::alloc(&b->p, req);
    }
    return e;
  }

  // Gives blocks back; those beyond the caps leave, the least recently released first.
  void release(const DevBlock* b, size_t count) {
    if (count == 0) return;
    typename Api::Guard guard;
    sync_devices(b, count);
    std::vector<DevBlock> out;
    {
      std::lock_guard<std::mutex> lk(mu_);
      for (size_t k = 0; k < count; ++k) {
        const size_t req = rounded(b[k].bytes);
        const int kind = req >= kMinBlock ? 0 : 1;
        blocks_[kind].push_back(DevBlock{b[k].p, req, b[k].dev});
        held_[kind] += req;
      }
      take_over(0, cap_, out);
      take_over(1, cap_ > 0 ? kSmallCap : 0, out);
    }
    free_blocks(out);
  }

 private:
  // large (0) and small (1) blocks, least recently released first
  std::mutex mu_;
  std::list<DevBlock> blocks_[2];
  size_t held_[2] = {0, 0}, cap_ = (size_t)32 << 30;

  // Waits for every device that one of the blocks belongs to.
  static void sync_devices(const DevBlock* b, size_t count) {
    const int cur = Api::device();
    for (size_t k = 0; k < count; ++k) {
      bool seen = false;
      for (size_t q = 0; q < k && !seen; ++q) seen = b[q].dev == b[k].dev;
      if (seen) continue;
      if (b[k].dev != cur) Api::use(b[k].dev);
      Api::sync();
      if (b[k].dev != cur) Api::use(cur);
    }
  }

  // Takes blocks off the front until at most `most` bytes of the kind are held (mu_ held).
  void take_over(int kind, size_t most, std::vector<DevBlock>& out) {
    while (held_[kind] > most) {
      out.push_back(blocks_[kind].front());
      held_[kind] -= out.back().bytes;
      blocks_[kind].pop_front();
    }
  }

  static void free_blocks(const std::vector<DevBlock>& v) {
    const int cur = Api::device();
    for (const DevBlock& b : v) {
      if (b.dev != cur) Api::use(b.dev);
      Api::free(b.p);
      if (b.dev != cur) Api::use(cur);
    }
  }

  void shrink(size_t most_large, size_t most_small) {
    typename Api::Guard guard;
    std::vector<DevBlock> out;
    {
      std::lock_guard<std::mutex> lk(mu_);
      take_over(0, most_large, out);
      take_over(1, most_small, out);
    }
    free_blocks(out);
  }
};
