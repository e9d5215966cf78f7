// Host-side gather of several requests' prefix caches ([planes][len][row] each, ordinary memory) into one packed buffer
// ([planes][total][row], page-locked), on a few threads of the handle's own: one thread copies at about a fifth of what the
// copy engine takes, and the engine starts on the first planes while the others are still being gathered.
#pragma once

#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

#if defined(__SSE2__)
#include <emmintrin.h>
#endif

namespace phyai {

// Copy past the caches: the destination is read next by the copy engine, not by this core (a third less memory traffic than
// stores that first fetch the line).
inline void copy_streaming(uint8_t* d, const uint8_t* s, size_t n) {
#if defined(__SSE2__)
  if (n >= 4096) {
    const size_t head = (16 - (reinterpret_cast<uintptr_t>(d) & 15)) & 15;
    memcpy(d, s, head);
    d += head, s += head, n -= head;
    for (; n >= 64; n -= 64, d += 64, s += 64) {
      const __m128i a = _mm_loadu_si128(reinterpret_cast<const __m128i*>(s)), b = _mm_loadu_si128(reinterpret_cast<const __m128i*>(s + 16));
      const __m128i c = _mm_loadu_si128(reinterpret_cast<const __m128i*>(s + 32)), e = _mm_loadu_si128(reinterpret_cast<const __m128i*>(s + 48));
      _mm_stream_si128(reinterpret_cast<__m128i*>(d), a), _mm_stream_si128(reinterpret_cast<__m128i*>(d + 16), b);
      _mm_stream_si128(reinterpret_cast<__m128i*>(d + 32), c), _mm_stream_si128(reinterpret_cast<__m128i*>(d + 48), e);
    }
    _mm_sfence();
  }
#endif
  memcpy(d, s, n);
}

class HostPacker {
 public:
  ~HostPacker() {
    {
      std::lock_guard<std::mutex> lock(mu_);
      stop_ = true;
    }
    cv_.notify_all();
    for (auto& t : threads_) t.join();
  }
  // Starts the gather of `planes` planes: request b contributes lens[b] rows from src[b].  The arrays must stay valid until
  // wait(planes) has returned.  False: out of memory, nothing was started.  (A process that may start no more threads has
  // fewer, or none: wait() then gathers by itself.)
  bool start(uint8_t* dst, const void* const* src, const uint32_t* lens, int batch, int planes, size_t row) noexcept {
    if (threads_.empty()) {
      const unsigned hw = std::thread::hardware_concurrency();
      const unsigned n = hw > 10 ? 8 : (hw > 3 ? hw - 2 : 1);
      try {
        threads_.reserve(n);
        for (unsigned i = 0; i < n; ++i) threads_.emplace_back([this] { work(); });
      } catch (const std::exception&) {
      }
    }
    try {
      std::lock_guard<std::mutex> lock(mu_);
      done_.assign(planes, 0);
      dst_ = dst, src_ = src, lens_ = lens, batch_ = batch, planes_ = planes, row_ = row;
      next_ = 0, ready_ = 0;
      ++job_;
    } catch (const std::exception&) {
      return false;
    }
    cv_.notify_all();
    return true;
  }
  // Blocks until the first `n` planes are complete.
  void wait(int n) {
    std::unique_lock<std::mutex> lock(mu_);
    while (threads_.empty() && ready_ < n) gather_next(lock);
    cv_done_.wait(lock, [&] { return ready_ >= n; });
  }

 private:
  void gather_next(std::unique_lock<std::mutex>& lock) {
    const int p = next_++;
    lock.unlock();
    size_t total = 0;
    for (int b = 0; b < batch_; ++b) total += lens_[b];
    uint8_t* d = dst_ + (size_t)p * total * row_;
    for (int b = 0; b < batch_; ++b) {
      const size_t n = (size_t)lens_[b] * row_;
      if (n) copy_streaming(d, static_cast<const uint8_t*>(src_[b]) + (size_t)p * n, n);
      d += n;
    }
    lock.lock();
    done_[p] = 1;
    bool moved = false;
    while (ready_ < planes_ && done_[ready_]) ++ready_, moved = true;
    if (moved) cv_done_.notify_one();
  }
  void work() {
    uint64_t seen = 0;
    for (;;) {
      std::unique_lock<std::mutex> lock(mu_);
      cv_.wait(lock, [&] { return stop_ || (job_ != seen && next_ < planes_); });
      if (stop_) return;
      while (next_ < planes_) gather_next(lock);
      seen = job_;
    }
  }

  std::mutex mu_;
  std::condition_variable cv_, cv_done_;
  std::vector<std::thread> threads_;
  bool stop_ = false;
  uint64_t job_ = 0;
  uint8_t* dst_ = nullptr;
  const void* const* src_ = nullptr;
  const uint32_t* lens_ = nullptr;
  int batch_ = 0, planes_ = 0, next_ = 0, ready_ = 0;
  size_t row_ = 0;
  std::vector<char> done_;
};

}  // namespace phyai
