// The order of an object's calls over the streams that they run on.
//
// Calls go to the object's own stream, or, one call at a time, to a stream that the caller chose for it (choose).  They
// share the object's device memory, so each follows the one before it: `done` marks the end of the last call, and a call
// on another stream waits for it.  The event is there only once a caller's stream has been used.
//
// Whether two calls share a stream is told by the stream's id, which the runtime never gives out twice.  The handle does
// not tell: that of a destroyed stream, whose work may still be running, can come back for a new one, and
// cudaStreamPerThread is one handle for a stream per host thread (it has no id here: a call on it always waits).
//
// Api supplies the runtime calls, so that the decisions can be tested without a GPU (tests/test_call_order_host.py).
#pragma once

namespace nlv {

template <class Api> struct CallOrder {
  using Stream = typename Api::Stream;
  using Event = typename Api::Event;
  using Error = typename Api::Error;

  Stream own = {};           // the object's own stream
  Stream run = {};           // where launches go: `own` outside a call on a caller's stream
  int device = 0;            // the object's device
  Event done = {};

  void init(Stream own_stream, int dev) {
    own = run = own_stream;
    device = dev;
  }
  // Whether the next call is to run on s.  Not on the object's own stream, for which nothing is to be chosen; not on one
  // that is being captured, which takes no dependency on work outside its capture; and not while another device is
  // current: a handle such as that of the default stream then names a stream of that device.
  bool choose(Stream s) {
    next_set = false;
    int current = -1;
    if (Api::current_device(&current) != Api::kSuccess) {
      Api::clear_error();
      return false;
    }
    if (current != device || s == own || capturing(s)) return false;
    if (!done) {             // from here on the end of every call is marked
      if (capturing(own)) return false;
      if (Api::create(&done) != Api::kSuccess || Api::record(done, own) != Api::kSuccess) {
        Api::clear_error();
        if (done) Api::destroy(done);
        done = {};
        return false;
      }
      last_known = Api::stream_id(own, &last);
    }
    next = s;
    next_set = true;
    return true;
  }
  // The stream of the call that begins now; the choice is used up.
  Stream take() {
    const Stream s = next_set ? next : own;
    next_set = false;
    return s;
  }
  // Orders the call's work, on stream s, after the call before it and sends launches there.
  Error enter(Stream s) {
    run = s;
    run_known = false;
    // (a chosen stream is not captured; the runtime takes asking a captured one for its id as an error of the capture)
    if (!done || (s == own && capturing(s))) return Api::kSuccess;
    run_known = Api::stream_id(s, &run_id);
    return run_known && last_known && run_id == last ? Api::kSuccess : Api::wait(s, done);
  }
  Error enter_own() {
    next_set = false;
    return enter(own);
  }
  // The end of the call's work on `run`; launches go to the own stream again.
  Error leave() {
    Error e = Api::kSuccess;
    if (done && !(run == own && capturing(run))) {
      e = Api::record(done, run);
      last_known = run_known;
      last = run_id;
    }
    run = own;
    return e;
  }
  // Waits for the last call on a caller's stream.
  void finish() {
    if (!done) return;
    Api::sync(done);
    Api::destroy(done);
    done = {};
  }

 private:
  static bool capturing(Stream s) {
    bool yes = false;
    if (Api::is_capturing(s, &yes) == Api::kSuccess) return yes;
    Api::clear_error();      // (the default stream while a stream that it blocks is captured; not this call's error)
    return true;
  }
  Stream next = {};          // the stream of the next call, if next_set
  bool next_set = false;
  // the ids of `run` and of the stream where `done` was recorded, if they have one
  unsigned long long run_id = 0, last = 0;
  bool run_known = false, last_known = false;
};

#if defined(__CUDACC__)
struct CudaOrderApi {
  using Stream = cudaStream_t;
  using Event = cudaEvent_t;
  using Error = cudaError_t;
  static constexpr Error kSuccess = cudaSuccess;
  static Error current_device(int* d) { return cudaGetDevice(d); }
  static Error is_capturing(Stream s, bool* yes) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const Error e = cudaStreamIsCapturing(s, &st);
    *yes = st != cudaStreamCaptureStatusNone;
    return e;
  }
  static bool stream_id(Stream s, unsigned long long* id) {
    if (s == cudaStreamPerThread) return false;
    if (s == nullptr || s == cudaStreamLegacy) {      // one stream that lasts: no need to ask (0.2 us)
      *id = ~0ull;
      return true;
    }
    if (cudaStreamGetId(s, id) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  static Error create(Event* e) { return cudaEventCreateWithFlags(e, cudaEventDisableTiming); }
  static Error record(Event e, Stream s) { return cudaEventRecord(e, s); }
  static Error wait(Stream s, Event e) { return cudaStreamWaitEvent(s, e, 0); }
  static Error sync(Event e) { return cudaEventSynchronize(e); }
  static Error destroy(Event e) { return cudaEventDestroy(e); }
  static void clear_error() { cudaGetLastError(); }
};
using StreamOrder = CallOrder<CudaOrderApi>;
#endif

}  // namespace nlv
