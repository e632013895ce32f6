// How many samples a batched call works on at once when device memory is short.
#pragma once

namespace wd {

// The largest of want, want / 2, want / 4, ... 1 (rounded up) for which alloc(chunk) succeeds, 0 if none does. After a
// failure drop() gives back what alloc had got, so that a smaller chunk finds that memory.
template <class Alloc, class Drop> int largest_chunk(int want, Alloc alloc, Drop drop) {
    for (int chunk = want;; chunk = (chunk + 1) / 2) {
        if (alloc(chunk)) return chunk;
        drop();
        if (chunk <= 1) return 0;
    }
}

}  // namespace wd
