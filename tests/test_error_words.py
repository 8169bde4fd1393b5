"""The loans of error words to overlapping projection calls: no word is with two calls at a time, however many calls come and go
while one of them waits."""
import os
import subprocess

import pytest

from paper_2510_04147_b200 import build

SOURCE = r"""
#include "error_words.h"
#include <cstdio>
#include <vector>
constexpr int kWords = 8;
ssd::ErrorWords<kWords> loans;
std::atomic<int> holders[kWords];
std::atomic<int> clashes{0};
int take() {
  const int w = loans.borrow();
  if (w < 0 || w >= kWords || holders[w].fetch_add(1) != 0) clashes++;
  return w;
}
void leave(int w) {
  holders[w].fetch_sub(1);
  loans.give_back(w);
}
int main() {
  const int held = take();                                   // a call that waits all along
  for (int i = 0; i < 20 * kWords; ++i) leave(take());
  std::vector<std::thread> threads;                          // more callers than words
  for (int t = 0; t < 2 * kWords; ++t)
    threads.emplace_back([] { for (int i = 0; i < 20000; ++i) leave(take()); });
  for (std::thread& t : threads) t.join();
  if (holders[held] != 1) clashes++;
  leave(held);
  int all[kWords];
  for (int& w : all) w = take();                             // every word came back
  for (int w : all) leave(w);
  std::printf("%d\n", clashes.load());
}
"""


def test_no_word_is_lent_twice(tmp_path):
    (tmp_path / "loans.cpp").write_text(SOURCE)
    exe = str(tmp_path / "loans")
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", build.CSRC, "-o", exe, str(tmp_path / "loans.cpp")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([exe], capture_output=True, text=True, timeout=60).stdout.strip() == "0"
