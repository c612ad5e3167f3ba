// The order of copies, launches and waits of the host entry point, apart from the CUDA calls themselves: `Api` makes
// them (pyramidsd.cu) or counts and fails them (the CPU test).
//   bool record(event, stream)   bool wait(stream, event)       events 0: the stream's earlier work, 1: stage 1's inputs
//   bool copy_in(i, stream)      0 draft, 1 qualifier, 2 target logits, 3 tokens             are there, 2: all inputs
//   int  run()                   enqueues both stages; with `overlap` stage 2 waits for event 2 (an error is returned)
//   bool copy_out()              bool sync(stream)
// The call is synchronous, so the caller may free its buffers once it has returned, with whatever status: every way out
// behind the first copy waits for both streams.
#pragma once

namespace psd {

enum HostStream { kHostMain = 0, kHostCopy = 1 };

template <class Api>
struct HostDrain {
  Api& api;
  const bool overlap;
  bool armed = true;
  ~HostDrain() {
    if (!armed) return;
    if (overlap) api.sync(kHostCopy);
    api.sync(kHostMain);
  }
};

// Large inputs (`overlap`): the copies go through a stream of their own, so that stage 1 runs while the target's logits are
// on their way. Returns `ok`, what run() returned, or `cuda_error`.
template <class Api>
int host_pipeline(Api& api, bool overlap, int ok, int cuda_error) {
  const HostStream cs = overlap ? kHostCopy : kHostMain;
  if (overlap && (!api.record(0, kHostMain) || !api.wait(kHostCopy, 0))) return cuda_error;
  HostDrain<Api> drain{api, overlap};
  if (!api.copy_in(3, cs) || !api.copy_in(0, cs) || !api.copy_in(1, cs)) return cuda_error;
  if (overlap && (!api.record(1, kHostCopy) || !api.wait(kHostMain, 1))) return cuda_error;
  if (!api.copy_in(2, cs)) return cuda_error;
  if (overlap && !api.record(2, kHostCopy)) return cuda_error;
  const int rc = api.run();
  if (rc != ok) return rc;
  if (!api.copy_out()) return cuda_error;
  if (!api.sync(kHostMain)) return cuda_error;   // both stages are behind every copy
  drain.armed = false;
  return ok;
}

}  // namespace psd
