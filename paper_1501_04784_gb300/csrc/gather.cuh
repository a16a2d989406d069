// gather.cuh -- plan and launch interfaces of the gather assembly (gather.cu,
// gather_plan.cu): a patch's element matrices are kept in shared memory and every
// owned CSR entry is summed by one thread, from a list of their positions.
#pragma once

#include "common.cuh"

namespace fem {

// One patch as the gather kernels read it.  `list` is the offset (32-bit words, a
// multiple of 4) of the patch's list block:
//   chunk table   (n_chunks + n_diag) x {word offset of the chunk's words, words,
//                 first row, row marks (of a diagonal chunk: the lanes whose row's
//                 diagonal is summed FP64-accurately in mixed precision)}
//   row starts    n_rows x int64: CSR position of the row's first entry minus its
//                 off-diagonal number (so entry i of the patch goes to it + i)
//   diagonals     n_own x int64: CSR position of the row's diagonal
//   words         [words][32] per chunk: two 16-bit positions each
// Off-diagonal entries are numbered row by row in patch order; rows without any are
// left out of the row starts.  A chunk is 32 consecutive numbers, one per lane; bit j
// of its row marks is set where lane j starts a row, and bit 0 always (lane 0 is in
// the first row).  The last n_diag chunks are the diagonals, 32 consecutive owned rows
// each.  A chunk's words hold each lane's contributions in the closure's order, filled
// up with the position of a zero.  A position is closure element x packed entries +
// packed entry.
struct alignas(16) GatherPatch {
    int64_t eb, cb, nb, list;
    int32_t n_elems, n_cnodes, n_own, n_off;
    int32_t n_rows, n_words, reserved, pad;
    __host__ __device__ int n_chunks() const { return (n_off + 31) / 32; }
    __host__ __device__ int n_diag() const { return (n_own + 31) / 32; }
};

// The list blocks of a closure's patches.
struct GatherLists {
    DevBuf<GatherPatch> patch;
    DevBuf<uint32_t> words;
    int zero = 0;  // position of the zero (past the largest closure's element matrices)
    bool ready = false;
    void free() {
        patch.free();
        words.free();
        zero = 0;
        ready = false;
    }
    size_t bytes() const { return patch.bytes() + words.bytes(); }
};

}  // namespace fem
