// Growth of a scratch buffer whose contents need not be kept.
#pragma once
#include <cstddef>

namespace oct {

// Gives *p room for n elements by alloc(&new, n) and release(old), which return
// an error code (0: success).  The old buffer goes only once the new one is
// there: after a failed allocation *p and *cap are what they were, so that a
// launch whose size was checked earlier still finds its scratch.
template <class T, class Alloc, class Release>
auto grow_buffer(T **p, size_t *cap, size_t n, Alloc alloc, Release release) -> decltype(release(*p)) {
    T *q = nullptr;
    decltype(release(*p)) e = alloc(&q, n);
    if (e != decltype(e)()) return e;
    T *const old = *p;
    *p = q;
    *cap = n;
    return old ? release(old) : e;
}

}  // namespace oct
