// Pieces that a batch with pinned host arrays is copied and run in.  Host
// arithmetic alone, compiled without CUDA too.
#pragma once

#include <cstdint>

namespace cht {

constexpr uint64_t kPipeChunk = 1ull << 24;  // operations of a piece at most
constexpr uint64_t kPipeMin = 1ull << 20;    // operations of a batch at least
constexpr int kPipePieces = 8;               // pieces of a batch of at most kPipeChunk operations, at most

// Operations of a piece of an n-operation batch: an eighth, rounded up (to
// whole blocks of 2^16), so that kPipePieces of them always cover the batch.
constexpr uint64_t pipe_piece(uint64_t n) {
    const uint64_t unit = (1ull << 16) * kPipePieces;
    const uint64_t p = (n / unit + (n % unit != 0)) * (1ull << 16);
    return p < kPipeChunk ? p : kPipeChunk;
}

// Whether two arrays (nbytes long, null: none) share memory.  Inputs are read
// before results are written in a batch staged whole; in pieces, the results of
// one would land in the inputs of another still to be copied.
inline bool share_memory(const void* a, uint64_t abytes, const void* b, uint64_t bbytes) {
    const uint64_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return a && b && (x < y ? y - x < abytes : x - y < bbytes);
}

}  // namespace cht
