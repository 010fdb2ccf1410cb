// capture_guard.h -- a stream capture that ends on every way out.
#pragma once

namespace dca {

// start() and finish() call begin() and end() and return their error code (0:
// done).  A capture that start() opened and finish() has not ended is ended when
// the guard leaves its scope: the stream can be captured again, and the error
// that the caller reports is the one that stopped it.
template <typename Begin, typename End>
class CaptureGuard {
 public:
  CaptureGuard(Begin begin, End end) : begin_(begin), end_(end) {}
  CaptureGuard(const CaptureGuard&) = delete;
  CaptureGuard& operator=(const CaptureGuard&) = delete;
  ~CaptureGuard() {
    if (open_) end_();
  }
  auto start() {
    const auto e = begin_();
    open_ = static_cast<int>(e) == 0;
    return e;
  }
  auto finish() {
    open_ = false;
    return end_();
  }

 private:
  Begin begin_;
  End end_;
  bool open_ = false;
};

}  // namespace dca
