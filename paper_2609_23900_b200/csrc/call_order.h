// What is known, on the host, of the call in front of the present one in its stream.  No CUDA in here.
#pragma once
#include <atomic>
#include <cstdint>

namespace lumo {

// A commit and a scan without convolution can read some of their inputs (accepted path, recorded operands, state) ahead of
// their dependency wait, while the kernel in front of them still runs.  That is sound only if this kernel is known not to write
// them, and a context sees its own calls alone: the kernel in front may have come from another context on the same stream.
// Hence one count of library calls per device, shared by all contexts.  A context knows what is in front of a call when the
// last library call on the device was its own, on the same stream, and succeeded; otherwise the answer is kNone and nothing
// is read ahead.  (One atomic addition per call.  Contexts that take turns on one device lose the early reads, about a
// microsecond of a small commit, never an order.)
class CallOrder {
 public:
  enum Kind { kNone = 0, kVerify, kCommit, kCommitVerify, kOther };
  // Starts a call: returns the kind of the call in front of it, kNone if that is not known.
  Kind begin(int device, const void* stream) {
    const uint64_t now = calls_[device & (kDevices - 1)].fetch_add(1) + 1;
    const Kind before = now == at_ + 1 && stream == stream_ ? kind_ : kNone;
    at_ = now;
    stream_ = stream;
    kind_ = kNone;
    return before;
  }
  // The call begun last has enqueued all its kernels.
  void done(Kind kind) { kind_ = kind; }

 private:
  static constexpr int kDevices = 64;
  static inline std::atomic<uint64_t> calls_[kDevices] = {};
  uint64_t at_ = 0;
  const void* stream_ = nullptr;
  Kind kind_ = kNone;
};

}  // namespace lumo
