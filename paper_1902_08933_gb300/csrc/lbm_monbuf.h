// lbm_monbuf.h -- device buffers of a persistent launch that records every step
// (mon_step_store): all of them or none.
#pragma once

#include <cstddef>

#include "lbm_internal.h"

namespace lbm {

struct MultiMonitor {
    double* slots = nullptr;   // [steps][items][kMonQ]
    double* sub = nullptr;     // [steps][instances][kMonSub][kMonQ]
    int* count = nullptr;      // [steps][instances][kMonSub + 1]
    // One allocation (alloc(void**, bytes): whether it was had); slots is its address.
    template <typename Alloc>
    bool allocate(size_t steps, size_t items, size_t instances, Alloc&& alloc) {
        const size_t a = steps * items * kMonQ, b = steps * instances * kMonSub * kMonQ;
        void* p = nullptr;
        *this = MultiMonitor();
        if (!alloc(&p, (a + b) * sizeof(double) + steps * instances * (kMonSub + 1) * sizeof(int)) || !p) return false;
        slots = static_cast<double*>(p);
        sub = slots + a;
        count = reinterpret_cast<int*>(sub + b);
        return true;
    }
};

}  // namespace lbm
