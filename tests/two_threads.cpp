// Two native threads calling sim_step_batch in tight loops, each on a handle, buffers and a
// stream of its own; returns how many of the calls failed.
#include <atomic>
#include <thread>

using Step = int (*)(void*, const void*, const void*, const void*, void*, void*, void*);
extern "C" int two_threads(Step step, void** a, void** b, int calls) {
  std::atomic<int> failed{0}, ready{0};
  auto loop = [&](void** x) {
    ++ready;
    while (ready < 2) std::this_thread::yield();
    for (int i = 0; i < calls; ++i)
      if (step(x[0], x[1], x[2], x[3], x[4], x[5], x[6]) != 0) ++failed;
  };
  std::thread t(loop, a);
  loop(b);
  t.join();
  return failed;
}
