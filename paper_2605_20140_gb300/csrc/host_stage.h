// A context's host buffer for values that are summed on the host in array order.
// Pinned, one half is copied while the other is summed; pinning itself takes longer
// than a call with few values gains, and may be refused, so a buffer can begin as
// ordinary memory and stay it.
#pragma once

#include <stddef.h>
#include <stdlib.h>

namespace sipf {

struct HostStage {
    double* p = nullptr;
    bool pinned = false;
    bool tried = false;      // pinning, once

    // Makes room for n values (the same n on every call); false if no memory is to be had.
    // The buffer is pinned on the first call (at_once), on the second (later) or never,
    // where pin(&q, bytes) says that it could.
    template <class Pin>
    bool get(size_t n, bool at_once, bool later, Pin pin) {
        void* q = nullptr;
        if (!tried && (at_once || (later && p))) {
            tried = true;
            if (pin(&q, n * sizeof(double))) {
                free(p);
                p = static_cast<double*>(q);
                pinned = true;
            }
        }
        if (!p) p = static_cast<double*>(malloc(n * sizeof(double)));
        return p != nullptr;
    }

    template <class Unpin>
    void release(Unpin unpin) {
        if (pinned) unpin(p);
        else free(p);
        *this = HostStage{};
    }
};

}  // namespace sipf
