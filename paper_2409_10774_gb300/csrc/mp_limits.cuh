// Shared-memory limits and occupancy of kernels, kept per device (host side).
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>

namespace mp {

// Api supplies the runtime calls: Error, ok, invalid, device(int&),
// static_smem(fn, size_t&), raise(fn, dynamic bytes), occupancy(fn, threads,
// smem, int&).
//
// A kernel's dynamic shared-memory limit is an attribute of the device's copy
// of it, so what has been raised is known by (device, kernel).  Answers lie in
// a fixed table, an entry displacing another of the same place: asking the
// runtime costs microseconds and the component calls ask each time, but a
// displaced answer is only asked for again.  Nothing is allocated (the
// allocation-free component call passes here), and one mutex makes the table
// safe for contexts used from several threads.
template <class Api>
class KernelLimits {
 public:
  using Error = typename Api::Error;

  // optin: shared memory a block may have; reserve: what a tiled kernel's
  // static shared memory may take of it (its largest tiles need the rest).
  KernelLimits(size_t optin, size_t reserve) : optin_(optin), reserve_(reserve) {}

  // Lets `fn` use the shared memory its static part leaves of the opt-in
  // maximum on the current device.
  Error raise(const void* fn, bool tiled) {
    int blocks = 0;
    return lookup(fn, tiled, 0, 0, blocks);
  }

  // Blocks of `fn` an SM of the current device holds, its limit raised first
  // (0 on an error).
  int resident(const void* fn, bool tiled, int threads, size_t smem) {
    int blocks = 0;
    return lookup(fn, tiled, threads, smem, blocks) == Api::ok ? blocks : 0;
  }

 private:
  struct Entry {
    const void* fn;
    size_t smem;
    int dev, threads, blocks;  // threads == 0: the limit alone
  };
  static constexpr int kEntries = 2048;

  Error lookup(const void* fn, bool tiled, int threads, size_t smem, int& blocks) {
    int dev = 0;
    Error e = Api::device(dev);
    if (e != Api::ok) return e;
    uint64_t h = reinterpret_cast<uintptr_t>(fn) ^ ((uint64_t)smem << 20) ^ ((uint64_t)threads << 44) ^ ((uint64_t)dev << 56);
    h *= 0x9e3779b97f4a7c15ull;
    Entry& slot = table_[h >> 53];
    std::lock_guard<std::mutex> lock(mu_);
    if (slot.fn == fn && slot.smem == smem && slot.dev == dev && slot.threads == threads) {
      blocks = slot.blocks;
      return Api::ok;
    }
    size_t stat = 0;
    if ((e = Api::static_smem(fn, stat)) != Api::ok) return e;
    if (stat > optin_ || (tiled && stat > reserve_)) return Api::invalid;
    if ((e = Api::raise(fn, optin_ - stat)) != Api::ok) return e;
    if (threads > 0 && (e = Api::occupancy(fn, threads, smem, blocks)) != Api::ok) return e;
    slot = Entry{fn, smem, dev, threads, blocks};
    return Api::ok;
  }

  const size_t optin_, reserve_;
  std::mutex mu_;
  Entry table_[kEntries] = {};
};

}  // namespace mp
