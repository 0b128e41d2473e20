// Copying several arrays of a result to the caller with one wait.
#pragma once

#include <stddef.h>

#include <initializer_list>

namespace mgb {

struct CopyOut {
    void* dst;                   // null: not asked for
    const void* src;
    size_t bytes;
};

// Queues the copies in order and waits once for all that were queued, also when
// one of them fails: the caller's arrays are not written to after the call has
// returned. queue(item) and wait() return a status (0: ok); the result is the
// first that is not.
template <class Queue, class Wait>
int copy_all(std::initializer_list<CopyOut> items, Queue queue, Wait wait)
{
    int status = 0;
    bool queued = false;
    for (const CopyOut& c : items) {
        if (!c.dst || c.bytes == 0) continue;
        queued = true;
        if ((status = queue(c))) break;
    }
    if (queued) {
        const int w = wait();
        if (!status) status = w;
    }
    return status;
}

}  // namespace mgb
