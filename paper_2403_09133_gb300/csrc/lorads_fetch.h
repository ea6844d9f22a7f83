// Results of a device call into the caller's host buffers, behind the call's error word: the word is
// read first, and a call that failed leaves every buffer as it was.
#pragma once
#include <stddef.h>

namespace lorads {

struct FetchItem {
  void* dst;          // host; NULL: not wanted
  const void* src;    // device
  size_t bytes;
};

// copy(dst, src, bytes) enqueues a download, wait() waits for those enqueued; both return 0 or a
// status, which ends the fetch.  A set error word returns `failed`.
template <class Copy, class Wait>
int fetch_outputs(const int* error_word, const FetchItem* items, int count, int failed, Copy copy,
                  Wait wait) {
  int word = 0;
  int st = copy(&word, error_word, sizeof(word));
  if (st == 0) st = wait();
  if (st != 0) return st;
  if (word != 0) return failed;
  for (int i = 0; i < count; ++i) {
    if (items[i].dst == nullptr || items[i].bytes == 0) continue;
    st = copy(items[i].dst, items[i].src, items[i].bytes);
    if (st != 0) return st;
  }
  return wait();
}

}  // namespace lorads
