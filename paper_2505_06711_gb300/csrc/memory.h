// Host-side rules for a list's device memory, free of CUDA calls so that they can be tested anywhere.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <initializer_list>

namespace reann {

// Rows of edge records that a list keeps: all of them, or the largest half, quarter, ... (at
// least kMinEdgeRows) that together with what the list's later calls take leaves a quarter of the
// free device memory to everything else.  An evaluation recomputes the records of one run of rows
// at a time when it has not all of them: slower, with the same results.
constexpr int64_t kMinEdgeRows = 1024;
inline int64_t fewer_edge_rows(int64_t rows) { return std::max(kMinEdgeRows, (rows + 1) / 2); }
inline int64_t edge_rows_within(int64_t rows, uint64_t row_bytes, uint64_t later, uint64_t free_bytes) {
    while (rows > kMinEdgeRows && (uint64_t)rows * row_bytes + later > free_bytes / 4 * 3) rows = fewer_edge_rows(rows);
    return rows;
}

// When the free memory is asked for: before records that, with those taken since the last answer, come to a
// 64th of it (what others take meanwhile is seen at the next answer)
struct FreeMemory {
    uint64_t bytes = 0, since = 0;
    bool ask(uint64_t want) {
        since += want;
        return since >= bytes / 64;
    }
    void told(uint64_t free_bytes) { bytes = free_bytes, since = 0; }
};

// Bytes per atom that a list may still take after its build: virials (36 + 9 / 32), host staging
// (36), MD (12 + 1 / 16), rounded up
constexpr uint64_t kLaterBytesPerAtom = 96;

// a block wanted: the address of the pointer (of any type) that receives it, and its size
struct Block {
    void* place;
    size_t bytes;
    void set(void* p) const { std::memcpy(place, &p, sizeof(p)); }
    void* get() const {
        void* p;
        std::memcpy(&p, place, sizeof(p));
        return p;
    }
};

// All of the blocks or none: where one cannot be had, the ones before it are given back and every
// place is left null; make_room() may then free memory, and after a true all are tried again.
template <class Take, class Give, class MakeRoom>
bool take_all(std::initializer_list<Block> want, Take take, Give give, MakeRoom make_room) {
    do {
        bool ok = true;
        for (const Block& b : want) b.set(nullptr);
        for (const Block& b : want) {
            b.set(take(b.bytes));
            ok = ok && b.get();
            if (!ok) break;
        }
        if (ok) return true;
        for (const Block& b : want)
            if (b.get()) {
                give(b.get());
                b.set(nullptr);
            }
    } while (make_room());
    return false;
}

}  // namespace reann
