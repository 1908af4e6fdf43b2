// Order of launches that allocate tensor memory, per device.
//
// Launches given on different streams are chained with an event, in the order of the calls.  One CTA takes a whole SM's
// tensor memory and nearly all of its shared memory, so two of them never share an SM and little is lost; runs that kept
// several streams of them in flight did not finish on the test machines, and no cause was found in the code.
//
// A call on a stream that is being captured is left alone: an event from outside the capture must not be waited for in it, and
// one recorded in it is of no use outside.  What a graph runs beside is up to the program that replays it.
//
// No CUDA header: the runtime's calls come through Api, so that the order can be tested without a GPU.  Api has the types
// Status (negative: error), Stream and Event (value-initialised: none), and
//   static Status capturing(Stream, bool*);  static Status wait(Stream, Event);
//   static Status create(Event*);  static Status record(Event, Stream);
#pragma once

#include <mutex>

namespace galore {

template <class Api>
class LaunchOrder {
 public:
  using Status = typename Api::Status;
  using Stream = typename Api::Stream;
  using Event = typename Api::Event;
  static constexpr int kDevices = 64;

  // runs `launch`, which queues kernels on st, a stream of device dev (0 .. kDevices - 1)
  template <class F>
  Status run(int dev, Stream st, F&& launch) {
    bool captured = false;
    const Status s = Api::capturing(st, &captured);
    if (s < 0) return s;
    if (captured) return launch();
    Device& d = devices_[dev];
    std::lock_guard<std::mutex> lock(d.mutex);      // for the whole call: its kernels follow one another on the stream
    if (d.used && d.last != st) {
      const Status w = Api::wait(st, d.done);
      if (w < 0) return w;
    }
    const Status l = launch();
    const Status r = after(d, st);      // also behind a call that failed half-way: what it had queued runs
    return l < 0 ? l : r;
  }

 private:
  struct Device {
    std::mutex mutex;
    bool used = false;
    Stream last = {};
    Event done = {};
  };
  Status after(Device& d, Stream st) {
    if (!d.done) {
      const Status c = Api::create(&d.done);
      if (c < 0) return c;
    }
    const Status r = Api::record(d.done, st);
    if (r < 0) return r;
    d.last = st;
    d.used = true;
    return r;
  }
  Device devices_[kDevices];
};

}  // namespace galore
