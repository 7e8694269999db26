// Rules by which the host chooses between kernels and launch shapes.  Plain C++, so that they can be checked without a GPU.
#pragma once

#include <algorithm>

namespace gproj {

// The count that `query` writes, or none where it fails: a launch shape that the device cannot vouch for is not used, and the
// calls that do not need it run all the same.
template <typename Query>
int count_or_none(Query query) {
  int n = 0;
  return query(&n) ? std::max(n, 0) : 0;
}

}  // namespace gproj
