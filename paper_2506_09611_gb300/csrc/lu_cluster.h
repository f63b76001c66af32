// lu_cluster.h -- whether a kernel may run in clusters of 16 CTAs (host only, no CUDA).
#pragma once
#include <stddef.h>

#include <map>
#include <mutex>
#include <utility>

namespace afq {

// How many 16-CTA clusters fit on a device depends on the shared memory of a CTA, so an answer is kept per
// (device, bytes).  query() returns the number of resident clusters, negative when it could not tell: then
// the answer is no, and it is asked again next time.  Safe with several threads.
class BigClusterCache {
public:
    template <typename Query>
    bool fits(int dev, size_t bytes, Query query) {
        std::lock_guard<std::mutex> lk(mu);
        const auto key = std::make_pair(dev, bytes);
        auto it = known.find(key);
        if (it != known.end()) return it->second;
        const int n = query();
        if (n < 0) return false;
        return known[key] = n >= 2;
    }

private:
    std::mutex mu;
    std::map<std::pair<int, size_t>, bool> known;
};

}  // namespace afq
