// The error words of the layer entry points (unet.cu), one for each call in
// progress: who holds which, and when one may be handed out again.  Host code alone.
#pragma once

#include <atomic>
#include <cstdint>
#include <thread>

namespace picgb {

// Which of 64 words are free.
class ErrWords {
 public:
  // a free word, after a wait while 64 calls are in progress; -1 when all are lost
  int take() {
    uint64_t t = taken_.load(std::memory_order_relaxed);
    for (;;) {
      if (t == ~uint64_t(0)) {
        if (lost_.load(std::memory_order_relaxed) == t) return -1;
        std::this_thread::yield();
        t = taken_.load(std::memory_order_relaxed);
        continue;
      }
      const int k = __builtin_ctzll(~t);
      if (taken_.compare_exchange_weak(t, t | (uint64_t(1) << k), std::memory_order_acquire)) return k;
    }
  }
  void give(int k) { taken_.fetch_and(~(uint64_t(1) << k), std::memory_order_release); }
  void lose(int k) { lost_.fetch_or(uint64_t(1) << k, std::memory_order_relaxed); }

 private:
  std::atomic<uint64_t> taken_{0}, lost_{0};
};

// What a wait for a call's launches says: they have ended, or the call failed and
// none of them will run, or neither is known.
enum class Drain { kEnded, kNotRun, kUnknown };

// A call's word, from before its first launch to its end.  It is zero when the call
// gets it, whatever an earlier call left there, and goes back only when nothing of
// this call can write it any more: after drain(), on every way out of the call.
template <class F>   // Drain()
class ErrLease {
 public:
  ErrLease(ErrWords &pool, volatile int *words, F drain) : pool_(pool), words_(words), drain_(drain), k_(pool.take()) {
    if (k_ >= 0 && words_[k_] != 0) words_[k_] = 0;
  }
  ~ErrLease() { end(); }
  ErrLease(const ErrLease &) = delete;
  ErrLease &operator=(const ErrLease &) = delete;
  int index() const { return k_; }
  // waits for the call's launches; what the word holds then, or -1 if they did not all run
  int end() {
    if (k_ < 0) return -1;
    const Drain d = drain_();
    const int e = d == Drain::kEnded ? words_[k_] : -1;
    if (d == Drain::kUnknown) pool_.lose(k_);
    else pool_.give(k_);
    k_ = -1;
    return e;
  }

 private:
  ErrWords &pool_;
  volatile int *words_;
  F drain_;
  int k_;
};

}  // namespace picgb
