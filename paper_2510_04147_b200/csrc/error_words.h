// Which of a fixed set of error words belongs to which call: a call borrows a word, and nobody else gets it until it is
// given back.  (Handed out in turn, a call that waits behind long work while others make as many calls as there are words would
// share its word with one of them: an error could be cleared before it is read, or read by the wrong call.)
#pragma once
#include <atomic>
#include <thread>

namespace ssd {

template <int N>
class ErrorWords {
 public:
  // the index of a word that no other call holds; with all N lent out, as soon as one comes back
  int borrow() {
    for (unsigned i = next_.fetch_add(1, std::memory_order_relaxed), tried = 1;; ++i, ++tried) {
      if (!lent_[i % N].exchange(true, std::memory_order_acquire)) return (int)(i % N);
      if (tried % N == 0) std::this_thread::yield();
    }
  }
  void give_back(int word) { lent_[word].store(false, std::memory_order_release); }

 private:
  std::atomic<bool> lent_[N] = {};
  std::atomic<unsigned> next_{0};
};

}  // namespace ssd
