// Page-locked host memory that grows on demand.
#pragma once

#include <cstddef>

namespace lmk {

// Makes *p hold at least `want` doubles (*n: how many it holds).  The new block
// is allocated before the old one is given back, so that after a failure *p
// and *n are as they were: the memory is written to without a check by every
// call that reads a flag or scalars back.  alloc(void**, bytes) and
// release(void*) return an error code, zero for success.
template <typename Error, typename Alloc, typename Release>
Error grow_host_doubles(double** p, size_t* n, size_t want, Alloc alloc, Release release) {
    if (*p != nullptr && *n >= want) return Error{};
    void* q = nullptr;
    const Error e = alloc(&q, want * sizeof(double));
    if (e != Error{}) return e;
    if (*p != nullptr) release(*p);
    *p = static_cast<double*>(q);
    *n = want;
    return Error{};
}

}  // namespace lmk
