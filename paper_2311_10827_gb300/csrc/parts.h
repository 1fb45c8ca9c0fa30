// Several buffers that are made and freed together.  Internal header.
#pragma once

#include <stddef.h>

namespace wblbm {

struct Part {
    void **p;
    size_t bytes;
};

// Allocates parts[0 .. n) (256-byte aligned; alloc's blocks are) and lists the blocks to
// free in blocks[0 .. n), unused entries null.  One block holds all of them where
// alloc gives one that large, because every block costs a synchronisation when it is
// freed; else each part gets its own, so that what fits in pieces still does.
// alloc(void **, size_t) and release(void *) return and take one block; false:
// not even the single parts could be had, and nothing is held.
template <class Alloc, class Release>
bool alloc_parts(const Part *parts, int n, void **blocks, Alloc alloc, Release release)
{
    auto padded = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t total = 0;
    for (int k = 0; k < n; ++k) {
        blocks[k] = nullptr;
        total += padded(parts[k].bytes);
    }
    if (alloc(&blocks[0], total)) {
        char *q = static_cast<char *>(blocks[0]);
        for (int k = 0; k < n; ++k) {
            *parts[k].p = q;
            q += padded(parts[k].bytes);
        }
        return true;
    }
    blocks[0] = nullptr;
    for (int k = 0; k < n; ++k) {
        if (!alloc(&blocks[k], parts[k].bytes)) {
            blocks[k] = nullptr;
            for (int j = 0; j < k; ++j) {
                release(blocks[j]);
                blocks[j] = nullptr;
            }
            return false;
        }
        *parts[k].p = blocks[k];
    }
    return true;
}

}  // namespace wblbm
