// What the scenarios of host_paths.cu ask of the fake CUDA runtime.
#pragma once

#include <atomic>

extern thread_local bool main_thread;
extern std::atomic<int> launches, direct_copies, live_stages;
extern std::atomic<int> allocations_left;      // operator new fails once this many more have succeeded; -1: never
extern bool launches_fail_in_workers, launches_fail;
extern void *on_device;              // pointers from here on are device memory
extern void (*while_asking)();       // runs inside the question for free memory
