// The word that a kernel sets when one of its bounded waits ran out, and who is told.
// Plain C++, so that the rules can be run on the host too.
#pragma once

#include "ups.h"

namespace ups {

// One word of pinned host memory that the device writes to (a kernel writes it only when
// a wait is lost), so that the host reads it without a copy: after an event or a host
// function on the stream, it holds what all launches before that point left.
struct LostWait {
    int *word = nullptr;
    // whether a wait was lost since the last call
    bool take() const {
        return word && __atomic_exchange_n(word, 0, __ATOMIC_ACQ_REL) != 0;
    }
};

// Status of a request when its batch has ended on the GPU; lost: a wait of the batch ran
// out, so that its results are not to be used.
inline int settled_status(int status, bool lost) {
    if (status != UPS_PENDING) return status;
    return lost ? UPS_ERR_TIMEOUT : UPS_OK;
}

}  // namespace ups
