// staging.cuh -- chunk staging of the library's section and fused kernels: a table, one per CTA, of
// the 16-byte pieces of a chunk buffer and where each lives in global memory.
//
// A piece costs one 16-byte table load, a multiply-add for its address and the copy.  The search
// over the slices that it replaces (compare with the slice's end, load its pointer, divide out its
// stride) cost about 20 instructions per piece, and the section kernels are bound by instruction
// issue (65-78% issue active at 0.4 of the copy bandwidth).
#pragma once

#include <cstdint>

#include "internal.h"
#include "ptx.cuh"

namespace adha {

struct StagePiece {
  const uint8_t* base;   // the piece in chunk 0
  int32_t step;          // bytes from one chunk's piece to the next
  int32_t at;            // offset in the chunk buffer; sign bit: the piece is written back
};
static_assert(sizeof(StagePiece) == 16, "one 16-byte load per piece");

// Pieces of a chunk of R records of the slices load[0..n_slices).
template <class Args>
__host__ __device__ __forceinline__ int stage_pieces(const Args& a, int R) {
  const int n_slices = a.n_load + (a.perm_slot >= 0 ? 1 : 0);
  int rec = 0;
  for (int k = 0; k < n_slices; ++k) rec += a.load[k].stride;
  return R * rec / 16;
}

// Builds the table (all threads of the CTA; the caller synchronizes).
template <class Args>
__device__ __forceinline__ void fill_pieces(const Args& a, int R, int n_pieces, StagePiece* tab, int tid) {
  for (int q = tid; q < n_pieces; q += kThreads) {
    int p = q * 16, k = 0;
    while (p >= R * a.load[k].stride) p -= R * a.load[k++].stride;
    const int at = a.load[k].start + p + (a.pad[k] ? p / a.load[k].stride * 16 : 0);
    tab[q] = StagePiece{a.load[k].ptr + p, R * a.load[k].stride, at | (a.writeback[k] ? (int)0x80000000 : 0)};
  }
}

// Where a piece of chunk ch lives: one wide multiply-add (ch is below 2^32, see plan_section).
__device__ __forceinline__ const uint8_t* piece_address(const StagePiece& pc, int64_t ch) {
  return pc.base + (uint64_t)(uint32_t)ch * (uint32_t)pc.step;
}

// Chunk ch into `buf` (asynchronous copies; the caller commits the group).
__device__ __forceinline__ void stage_chunk(const StagePiece* tab, int n_pieces, int64_t ch, uint8_t* buf, int lane) {
  const uint32_t sbuf = smem_addr(buf);
#pragma unroll 2
  for (int q = lane; q < n_pieces; q += 32) {
    const StagePiece pc = tab[q];
    cp_async16_at(sbuf + (pc.at & 0x7FFFFFFF), piece_address(pc, ch));
  }
}

// The written-back pieces of chunk ch from `buf`.
__device__ __forceinline__ void unstage_chunk(const StagePiece* tab, int n_pieces, int64_t ch, const uint8_t* buf, int lane) {
#pragma unroll 2
  for (int q = lane; q < n_pieces; q += 32) {
    const StagePiece pc = tab[q];
    if (pc.at < 0)
      *reinterpret_cast<uint4*>(const_cast<uint8_t*>(piece_address(pc, ch))) =
          *reinterpret_cast<const uint4*>(buf + (pc.at & 0x7FFFFFFF));
  }
}

// REDUCE by the walk: the record of zeros after every slice of a chunk buffer.
template <class Args>
__device__ __forceinline__ void zero_records(const Args& a, int R, uint8_t* buf, int lane) {
  for (int k = 0; k < a.n_load; ++k)
    for (int p = lane * 4; p < a.load[k].stride; p += 128)
      *reinterpret_cast<uint32_t*>(buf + a.load[k].start + R * (a.load[k].stride + 16 * a.pad[k]) + p) = 0u;
}

}  // namespace adha
