// KernelLimits (mp_limits.cuh) against a runtime of two devices that counts
// what it is asked: limits hold per device, answers are kept, nothing is
// allocated after construction, and threads may share the table.
#include <cstdio>
#include <cstdlib>
#include <new>
#include <thread>
#include <vector>

#include "mp_limits.cuh"

static long allocations = 0;
void* operator new(std::size_t n) {
  ++allocations;
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

constexpr int kKernels = 400;
static thread_local int current = 0;
static size_t limit[2][kKernels];
static long queries = 0;
static char kernels[kKernels];

struct Fake {
  using Error = int;
  static constexpr Error ok = 0, invalid = 1;
  static Error device(int& d) { d = current; return ok; }
  static Error static_smem(const void* fn, size_t& b) {
    ++queries;
    b = (static_cast<const char*>(fn) - kernels) == 7 ? 3000 : 100;
    return ok;
  }
  static Error raise(const void* fn, size_t bytes) { limit[current][static_cast<const char*>(fn) - kernels] = bytes; return ok; }
  static Error occupancy(const void*, int threads, size_t smem, int& blocks) {
    blocks = (int)(2048 / threads < (int)(200000 / (smem + 1)) ? 2048 / threads : 200000 / (smem + 1));
    return ok;
  }
};

#define CHECK(x) \
  if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }

int main() {
  static mp::KernelLimits<Fake> limits(232448, 2048);
  const long before = allocations;
  for (int dev = 0; dev < 2; ++dev) {
    current = dev;
    for (int round = 0; round < 2; ++round)
      for (int k = 0; k < kKernels; ++k) {
        if (k == 7) continue;
        CHECK(limits.raise(kernels + k, true) == 0);
        CHECK(limits.resident(kernels + k, true, 256, 50000) == 3);
        CHECK(limits.resident(kernels + k, true, 128, 1000) == 16);
        CHECK(limit[dev][k] == 232448 - 100);
      }
    // static memory beyond the reserve: refused where the tiles need the rest
    CHECK(limits.raise(kernels + 7, true) == 1 && limits.resident(kernels + 7, true, 256, 1000) == 0);
    CHECK(limit[dev][7] == 0);
    CHECK(limits.raise(kernels + 7, false) == 0 && limit[dev][7] == 232448 - 3000);
  }
  current = 0;
  queries = 0;
  for (int i = 0; i < 1000; ++i) CHECK(limits.resident(kernels + 3, true, 256, 50000) == 3);
  CHECK(queries <= 1);
  CHECK(allocations == before);
  std::vector<std::thread> ts;
  bool good[8] = {};
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      current = t & 1;
      bool ok = true;
      for (int i = 0; i < 20000; ++i) ok &= limits.resident(kernels + 8 + (i * 7 + t) % 300, true, 256, 50000) == 3;
      good[t] = ok;
    });
  for (auto& t : ts) t.join();
  for (bool g : good) CHECK(g);
  std::puts("ok");
  return 0;
}
