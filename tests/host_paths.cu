// The host side of the library's copies and pools against a CUDA runtime that is a fake (host_paths_fake.cpp).  Built and run by
// test_host_paths.py, one scenario per process.
#include "../paper_2105_09837_b200/csrc/host_io.cuh"

#include "host_paths_fake.h"

#include <sys/mman.h>

#include <atomic>
#include <chrono>
#include <stdexcept>

using namespace pd;
static int check(bool ok, const char *what) { printf("%s: %s\n", what, ok ? "yes" : "NO"); return ok ? 0 : 1; }

int main(int argc, char **argv) {
  main_thread = true;
  const std::string what = argc > 1 ? argv[1] : "";
  constexpr size_t rows = 20000, width = 400, pitch = 512;           // 8 MB: four threads
  std::vector<char> host(rows * width), dev(rows * pitch);
  if (what == "copies") {
    return check(copy_rows(0, nullptr, host.data(), dev.data(), pitch, width, rows, true) == PDADMM_OK && launches > 1, "a copy in pieces succeeds");
  }
  if (what == "launch fails in workers") {
    launches_fail_in_workers = true;
    return check(copy_rows(0, nullptr, host.data(), dev.data(), pitch, width, rows, true) == PDADMM_ECUDA, "the failed launch is reported");
  }
  if (what == "launch fails") {
    launches_fail = true;
    return check(copy_rows(0, nullptr, host.data(), dev.data(), pitch, width, 100, true) == PDADMM_ECUDA, "one piece: reported") +
           check(launch_pack(nullptr, dev.data(), pitch, width, 100, host.data()) != cudaSuccess, "the launch says so itself");
  }
  if (what == "device pointer") {                                    // neither readable nor writable for the host
    on_device = mmap(nullptr, rows * width, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    int bad = 0;
    for (const bool out : {true, false})
      for (const size_t n : {size_t(1), size_t(100), rows})
        bad += check(copy_rows(0, nullptr, on_device, dev.data(), pitch, width, n, out) == PDADMM_OK, "copied");
    return bad + check(direct_copies >= 6 && launches == 0, "by the driver");
  }
  if (what == "no host memory") {
    int bad = 0;
    for (int n = 0; n < 40; ++n) {                                   // the n-th allocation and all that follow fail
      allocations_left = n;
      const int rc = guarded([&]() -> int { return copy_rows(0, nullptr, host.data(), dev.data(), pitch, width, rows, n % 2 == 0); });
      allocations_left = -1;
      bad += rc != PDADMM_OK && rc != PDADMM_ENOMEM;
      DevicePool pool;
      std::vector<DeviceBlock> blocks;
      DeviceBlock b;
      for (int i = 0; i < 3; ++i) if (pool.take(100, &b) == cudaSuccess) blocks.push_back(b);
      allocations_left = n % 5;
      pool.give(blocks);
      allocations_left = -1;
      pool.trim();
    }
    stage_pool().trim();
    return check(bad == 0, "an answer or PDADMM_ENOMEM") + check(live_stages == 0, "nothing is lost") +
           check(guarded([]() -> int { throw std::length_error("x"); }) == PDADMM_ECUDA, "another exception is an error too");
  }
  if (what == "asking for free memory") {
    static DevicePool pool;
    static std::atomic<bool> took{false}, asked{false};
    DeviceBlock b;
    if (pool.take(1000, &b) != cudaSuccess) return 1;
    while_asking = [] {                                              // waits (two seconds at most) for the other thread's take
      asked = true;
      for (int i = 0; i < 2000 && !took; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    };
    std::thread other([] {
      while (!asked) std::this_thread::yield();
      DeviceBlock d;
      if (pool.take(5000, &d) == cudaSuccess) took = true;
    });
    const auto t0 = std::chrono::steady_clock::now();
    pool.give({b});
    const bool waited = std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(1500);
    other.join();
    return check(!waited, "another thread's take does not wait for the question");
  }
  return 2;
}
