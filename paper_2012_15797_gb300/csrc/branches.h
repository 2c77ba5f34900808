// Work of one call on several streams: branches forked from the caller's stream
// and joined back into it.  Plain C++ (tests/test_branches_cpu.py runs it
// without a device).
#pragma once

namespace mog {

// For branch 0 .. n - 1 in turn: fork(i) (the branch's stream waits for the
// caller's), then launch(i); after the last, join(i) for every branch that was
// forked.  Each returns a status, `ok` if it did its part.  The first failure
// ends the launches and is returned, but what has been forked by then is joined
// all the same: the caller's stream, and with it the caller's buffers and the
// workspace that the next call plans into, must not run ahead of kernels that
// were launched.
template <class Status, class Fork, class Launch, class Join>
Status run_branches(int n, Status ok, Fork&& fork, Launch&& launch, Join&& join) {
  Status first = ok;
  int forked = 0;
  for (int i = 0; i < n && first == ok; ++i) {
    first = fork(i);
    if (first != ok) break;
    forked = i + 1;
    first = launch(i);
  }
  for (int i = 0; i < forked; ++i) {
    const Status st = join(i);
    if (first == ok) first = st;
  }
  return first;
}

}  // namespace mog
