// nls_attr.h -- function attributes that a kernel needs before its launch.
#pragma once

#include <climits>
#include <set>

namespace nls {

// More than 48 KB of dynamic shared memory needs an opt-in.  A function
// attribute belongs to one device, so every handle (which belongs to one device,
// current when it launches) keeps the kernels that it has opted in.
struct SmemOptIns {
    std::set<const void *> done;

    // set(func, bytes) makes the opt-in and returns 0 or an error code, which is
    // passed on and not remembered.  bytes: the most that any launch of func asks for.
    template <class Set>
    int ensure(const void *func, int bytes, Set &&set)
    {
        if (bytes <= 48 * 1024 || done.count(func)) return 0;
        const int rc = set(func, bytes);
        if (!rc) done.insert(func);
        return rc;
    }
    // Likewise for another attribute, set(func), of the kernels that want it.
    template <class Set>
    int ensure_if(bool wanted, const void *func, Set &&set)
    {
        return ensure(func, wanted ? INT_MAX : 0, [&](const void *f, int) { return set(f); });
    }
};

} // namespace nls
