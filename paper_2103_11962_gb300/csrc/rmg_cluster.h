// Choice of a thread-block cluster's width (host code without CUDA types, so that it can be tested
// without a device).
#pragma once

#include <initializer_list>

namespace rmg {

// The wider of 16 and 8 blocks of which a cluster fits, or 0. allow_wide() opts in to 16, active(n,
// &count) says how many clusters of n blocks fit; both return whether the call succeeded. After one
// that failed clear() takes its error back: the next launch's check would find it.
template <class Allow, class Active, class Clear>
int widest_cluster(Allow allow_wide, Active active, Clear clear) {
  for (int cluster : {16, 8}) {
    int count = 0;
    if ((cluster == 16 && !allow_wide()) || !active(cluster, &count)) clear();
    else if (count > 0) return cluster;
  }
  return 0;
}

}  // namespace rmg
