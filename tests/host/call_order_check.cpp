// Host check of nlv::CallOrder over a fake runtime: which stream a call runs on and which wait it queues.
#include <cstdio>
#include <string>

#include "call_order.h"

struct Fake {
  using Stream = int;            // 0: the default stream; 9: the per-thread stream, which has no id
  using Event = int;
  using Error = int;
  static constexpr Error kSuccess = 0;
  static inline int device = 0, device_error = 0, capturing = -1, capture_error = 0;
  static inline std::string log;
  static Error current_device(int* d) { *d = device; return device_error; }
  static Error is_capturing(Stream s, bool* yes) { *yes = s == capturing; return capture_error; }
  static inline int reborn = -1;         // a handle whose stream was destroyed and created anew
  static bool stream_id(Stream s, unsigned long long* id) {
    if (s == capturing) log += "id-of-captured ";
    if (s == 9) return false;
    *id = 1000ull + (unsigned long long)s + (s == reborn ? 100000ull : 0ull);
    return true;
  }
  static Error create(Event* e) { *e = 7; return 0; }
  static Error record(Event, Stream s) { log += "record" + std::to_string(s) + " "; return 0; }
  static Error wait(Stream s, Event) { log += "wait" + std::to_string(s) + " "; return 0; }
  static Error sync(Event) { log += "sync "; return 0; }
  static Error destroy(Event) { return 0; }
  static void clear_error() { log += "clear "; }
};

static int bad = 0;
static void check(bool ok, const char* what) {
  if (!ok) { ++bad; std::printf("FAIL %s (log: %s)\n", what, Fake::log.c_str()); }
}
// One call on the stream that the caller asks for; what it queues, with where it ran.
static std::string call(nlv::CallOrder<Fake>& o, int s) {
  Fake::log.clear();
  o.choose(s);
  o.enter(o.take());
  const int ran = o.run;
  o.leave();
  return Fake::log + "ran" + std::to_string(ran);
}

int main() {
  const int own = 50;
  {
    nlv::CallOrder<Fake> o;
    o.init(own, 0);
    check(call(o, own) == "ran50", "own stream: nothing to order");
    check(call(o, 1) == "record50 wait1 record1 ran1", "first caller's stream follows the own stream");
    check(call(o, 1) == "record1 ran1", "the same stream again needs no wait");
    check(call(o, 0) == "wait0 record0 ran0", "the default stream follows stream 1");
    check(call(o, own) == "wait50 record50 ran50", "the own stream follows the default stream");
    Fake::log.clear();
    o.finish();
    check(Fake::log == "sync ", "the end waits for the last call");
  }
  {                                                 // another device is current: the handle is that device's
    nlv::CallOrder<Fake> o;
    o.init(own, 0);
    call(o, 0);
    Fake::device = 1;
    check(!o.choose(0), "default stream of another device is not taken");
    check(!o.choose(1), "no stream is taken under another device");
    check(call(o, 0) == "wait50 record50 ran50", "the call keeps to the object's own stream");
    Fake::device = 0;
    check(call(o, 0) == "wait0 record0 ran0", "taken again under the right device");
    Fake::device_error = 3;
    Fake::log.clear();
    check(!o.choose(0) && Fake::log == "clear ", "unknown device: not taken, the error is not left behind");
    Fake::device_error = 0;
  }
  {                                                 // one handle, another stream
    nlv::CallOrder<Fake> o;
    o.init(own, 0);
    call(o, 1);
    Fake::reborn = 1;
    check(call(o, 1) == "wait1 record1 ran1", "a new stream at an old handle follows the call on the old one");
    check(call(o, 1) == "record1 ran1", "and needs no wait after itself");
    Fake::reborn = -1;
    check(call(o, 9) == "wait9 record9 ran9", "the per-thread stream follows");
    check(call(o, 9) == "wait9 record9 ran9", "the per-thread stream, perhaps another thread's, follows again");
    check(call(o, 1) == "wait1 record1 ran1", "a stream follows the per-thread one");
  }
  {                                                 // captured streams
    nlv::CallOrder<Fake> o;
    o.init(own, 0);
    Fake::capturing = 2;
    check(!o.choose(2), "a captured stream is not taken");
    Fake::capturing = own;
    check(!o.choose(1), "no event is recorded into a capture");
    Fake::capturing = -1;
    call(o, 1);
    Fake::capturing = own;
    check(call(o, own) == "ran50", "a captured call on the own stream: no wait on, no mark of, work outside the capture");
    Fake::capturing = -1;
    Fake::capture_error = 4;
    Fake::log.clear();
    check(!o.choose(0) && Fake::log == "clear ", "unknown capture: not taken, the error is not left behind");
    Fake::capture_error = 0;
    check(o.choose(1) && o.take() == 1 && o.take() == own, "a choice is for one call");
    o.choose(1);
    o.enter_own();
    check(o.run == own && o.take() == own, "a call on the own stream uses the choice up");
  }
  std::printf("%d failures\n", bad);
  return bad != 0;
}
