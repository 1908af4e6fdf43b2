// The order of launches on a fake runtime: prints one line per call that reaches it.
#include <cstdio>
#include <cstdlib>
#include <string>

#include "../paper_2403_03507_b200/csrc/launch_order.h"

struct Fake {
  using Status = int;
  using Stream = int;
  using Event = int;
  static inline int captured_stream = -1, next_event = 0;
  static int capturing(int st, bool* on) { *on = st == captured_stream; return 0; }
  static int wait(int st, int e) { std::printf("wait stream %d event %d\n", st, e); return 0; }
  static int create(int* e) { *e = ++next_event; return 0; }
  static int record(int e, int st) { std::printf("record event %d stream %d\n", e, st); return 0; }
};

// arguments: "call STREAM", "fail STREAM" (the launch returns an error), "device N", "capture STREAM", "end"
int main(int argc, char** argv) {
  galore::LaunchOrder<Fake> order;
  int dev = 0;
  for (int i = 1; i < argc; ++i) {
    const std::string what = argv[i];
    if (what == "end") { Fake::captured_stream = -1; continue; }
    const int n = std::atoi(argv[++i]);
    if (what == "device") dev = n;
    else if (what == "capture") Fake::captured_stream = n;
    else {
      const int s = order.run(dev, n, [&]() { std::printf("launch stream %d\n", n); return what == "fail" ? -5 : 0; });
      std::printf("status %d\n", s);
    }
  }
  return 0;
}
