// Places of the arrays of a batch launch in its work buffer, in elements.  Host code
// without CUDA, so that the layout can be checked on any machine.
#pragma once

#include <cstddef>

namespace mpax {

// m, n: rows and columns of all instances; za: stored elements of each of the two value
// arrays (nonzeros and padding).  Every array starts at a multiple of 16 elements, and
// `total` counts what that rounding adds: up to 15 elements for each of the fifteen arrays,
// more than the arrays themselves for a batch of a few rows.
struct BatchWork {
  size_t total = 0;
  size_t val, valt, c, l, u, lc, uc, w, xa, xhat, gbuf, ya, yhat, gys, gxs;
  BatchWork(size_t m, size_t n, size_t za) {
    val = take(za), valt = take(za);
    c = take(n), l = take(n), u = take(n), lc = take(m), uc = take(m);
    w = take(n), xa = take(n), xhat = take(n), gbuf = take(n);
    ya = take(m), yhat = take(m), gys = take(m), gxs = take(n);
  }

 private:
  size_t take(size_t k) {
    const size_t r = total;
    total += (k + 15) / 16 * 16;
    return r;
  }
};

}  // namespace mpax
