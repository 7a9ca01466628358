// A setting that only grows, raised by several host threads (a kernel's dynamic shared memory: rosar_api.cu).
#pragma once

#include <mutex>

namespace rosar {

// Calls set(want) unless *limit says that at least `want` is set; *limit is what was set last.  One thread at a time sets
// and records: a smaller value set late would otherwise stand under a larger one recorded.  Returns set's status, 0: done.
template <typename F>
int raise_limit(int *limit, int want, F set) {
    if (__atomic_load_n(limit, __ATOMIC_ACQUIRE) >= want) return 0;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (__atomic_load_n(limit, __ATOMIC_ACQUIRE) >= want) return 0;
    const int status = set(want);
    if (status == 0) __atomic_store_n(limit, want, __ATOMIC_RELEASE);
    return status;
}

}  // namespace rosar
