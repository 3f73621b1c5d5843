// Weight scales with groups of 128: two bytes {pos, neg} per row and step of 128, copied as the aligned 4-byte words around a run of
// steps.  Which words those are, and how many bytes of each belong to the tensor.  (Host and device: the ranges are checked on
// the CPU over all starts and lengths.)
#pragma once
#include <stdint.h>

namespace amx {

// Words around the pairs first .. first + n - 1, counted from the tensor's (4-byte aligned) start: from word first / 2 on.
__host__ __device__ constexpr int pair_words(int64_t first, int n) { return ((int)(first & 1) + n + 1) >> 1; }
// Whether all of word `word` belongs to a tensor of `pairs` pairs: an odd number ends in the middle of a word.
__host__ __device__ constexpr bool pair_word_whole(int64_t word, int64_t pairs) { return 2 * word + 2 <= pairs; }

}  // namespace amx
