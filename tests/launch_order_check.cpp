// The order of launches on a fake runtime: prints one line per call that reaches it.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <thread>

#include "../paper_2403_03507_b200/csrc/launch_order.h"

struct Fake {
  using Status = int;
  using Stream = int;
  using Event = int;
  static inline int captured_stream = -1, next_event = 0;
  static int capturing(int st, bool* on) { *on = st == captured_stream; return 0; }
  static int wait(int st, int e) { std::printf("wait stream %d event %d\n", st, e); return 0; }
  static int create(int* e) { *e = ++next_event; return 0; }
  static inline bool quiet = false;
  static int record(int e, int st) {
    if (!quiet) std::printf("record event %d stream %d\n", e, st);
    return 0;
  }
};

// two launches on two devices, each of which ends once the other has begun; which: whose thread starts first
static void both(int which) {
  Fake::quiet = true;
  galore::LaunchOrder<Fake> order;
  std::atomic<int> begun{0};
  bool met[2] = {};
  auto on = [&](int dev) {
    order.run(dev, dev, [&]() {
      ++begun;
      for (int i = 0; i < 1000 && begun < 2; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(10));
      met[dev] = begun == 2;
      return 0;
    });
  };
  std::thread first(on, which), second(on, 1 - which);
  first.join();
  second.join();
  std::printf("%s\n", met[0] && met[1] ? "both launches at once" : "one after the other");
}

// arguments: "call STREAM", "fail STREAM" (the launch returns an error), "device N", "capture STREAM", "end", "both N"
int main(int argc, char** argv) {
  galore::LaunchOrder<Fake> order;
  int dev = 0;
  for (int i = 1; i < argc; ++i) {
    const std::string what = argv[i];
    if (what == "end") { Fake::captured_stream = -1; continue; }
    const int n = std::atoi(argv[++i]);
    if (what == "device") dev = n;
    else if (what == "both") both(n);
    else if (what == "capture") Fake::captured_stream = n;
    else {
      const int s = order.run(dev, n, [&]() { std::printf("launch stream %d\n", n); return what == "fail" ? -5 : 0; });
      std::printf("status %d\n", s);
    }
  }
  return 0;
}
