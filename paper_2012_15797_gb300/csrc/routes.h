// Which of two kernels renders a bucket.  Plain C++ (tests/test_routes_cpu.py
// runs it without a device).
#pragma once

#include <stdint.h>

#include "branches.h"

namespace mog {

// 256 x 256 galaxies have two kernels, one for few (a cluster of CTAs per galaxy)
// and one for many (a CTA per galaxy), with the same results; `line` is the most
// galaxies of the first.  How many there are is known on the device only: a
// batch may have any share of them, whatever its count and the sides it names.
// So where the batch's count (max_galaxies) does not settle it, both are
// launched, each with the range of bucket counts that are its own, and the one on
// whose side the bucket's count is not returns at once.  They are launched side
// by side, few(q, true) between fork() and join(): behind one another the second
// would first wait for SMs that the other sides' kernels hold (gradients of 1000
// galaxies of mixed sides with the Lanczos shift 0.17 against 0.22 ms, renders
// with it of 1250 of 128 x 128 and 1250 of 256 x 256 0.40 to 0.45 against 0.48).
// Above `far` galaxies in the batch the kernel of many alone: there the others
// take about as long as it needs for a few.
// Params: max_galaxies, bucket_min, bucket_max.
template <class Status, class Params, class Fork, class Few, class Many, class Join>
Status launch_by_count(const Params& p, int line, int far, Status ok, Fork&& fork, Few&& few, Many&& many, Join&& join) {
  Params q = p;
  q.bucket_min = 0;
  q.bucket_max = INT32_MAX;
  if (p.max_galaxies <= line) return few(q, false);
  if (p.max_galaxies > far) return many(q);
  return run_branches<Status>(
      2, ok, [&](int i) { return i == 0 ? fork() : ok; },
      [&](int i) {
        q.bucket_min = i == 0 ? 0 : line + 1;
        q.bucket_max = i == 0 ? line : INT32_MAX;
        return i == 0 ? few(q, true) : many(q);
      },
      [&](int i) { return i == 0 ? join() : ok; });
}

}  // namespace mog
