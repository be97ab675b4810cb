// TMA descriptors of the attention kernels' operands: host-side interface.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace spec {

// 3-D view of a K or V pool [num_pages][G][page_size][hd]: dim0 = 64 elements (128 bytes), dim1 = every key row of
// the pool (pitch hd * 2 bytes), dim2 = the hd / 64 column halves (128 bytes apart).  One box = one page of one head.
// depth: 64-column halves per box (hd / 64: one box = one page of one head; 1: one half of it).  Cached; nullptr if refused.
const CUtensorMap *kv_map(const void *pool, int num_pages, int G, int ps, int hd, int depth = 0);
// q [rows][H][128] as {128 elements, H heads, rows}: one box = 64 elements of `box_rows` rows of one head, 128-byte
// swizzle.  Not cached (the pointer may be a caller's); false if refused.
bool q_map(CUtensorMap *out, const void *q, int rows, int H, int box_rows);
// kd / vd [J][T][G][128] as {128 elements, G heads, T positions, J steps}: one box = 64 elements of `box_rows` positions of
// one head and step, 128-byte swizzle.  Not cached; false if refused.
bool diag_map(CUtensorMap *out, const void *kd, int J, int T, int G, int box_rows);

}  // namespace spec
