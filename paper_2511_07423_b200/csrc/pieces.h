// A range of positions as launches of a bounded number of pages each.  Host code, no CUDA.
#pragma once
#include <algorithm>
#include <cstdint>

namespace syn {

// launch(position, positions, positions before it) for pieces of at most `max_pages` pages, cut at page boundaries, until one
// fails; then wait().  The wait also follows a failed launch: the pieces before it still use the caller's buffers.  Returns the
// first error (0: none).
template <typename Launch, typename Wait>
int for_pieces(int pos0, int n_pos, int page_size, int max_pages, Launch&& launch, Wait&& wait) {
    int r = 0;
    for (int64_t done = 0; done < n_pos && r == 0;) {
        const int at = (int)(pos0 + done);
        const int n = (int)std::min<int64_t>(n_pos - done, (int64_t)max_pages * page_size - at % page_size);
        r = launch(at, n, done);
        done += n;
    }
    const int w = wait();
    return r ? r : w;
}

}  // namespace syn
