// Where the 16-byte pieces of a row lie in shared memory while a permutation gathers from it (fp32 rows: harp_f32.cu, the rows of a
// gradient: harp_grad.cu).  Pieces are exchanged within groups of eight, 128 bytes, by higher bits of the index: under a digit
// reversal the coordinates that a warp gathers are powers of two apart (4-way conflicts instead of 16-way; finer exchanges would split the
// pieces).  A group that the end of a row cuts short is exchanged over all of its eight places, so that rows are whole groups
// apart.  Plain C++ beside the annotation, so that a host program can replay it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define HARP_PERMUTE_FN __host__ __device__ __forceinline__
#else
#define HARP_PERMUTE_FN inline
#endif

// V: elements of a piece, eight or four
template <int V>
HARP_PERMUTE_FN int permute_piece(int c) { return c ^ ((c >> (V == 8 ? 3 : 4)) & 7); }
// place of element i of a row
template <int V>
HARP_PERMUTE_FN int permute_place(int i) { return V * permute_piece<V>(i / V) + i % V; }
// elements from one row to the next; d a multiple of V
template <int V>
HARP_PERMUTE_FN int permute_pitch(int64_t d) { return (int)((d / V + 7) / 8 * 8 * V); }
