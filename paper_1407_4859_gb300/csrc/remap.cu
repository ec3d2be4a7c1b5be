// remap.cu -- the layout remap kernel (paper Section 2: the remap between two sections' layouts;
// Table 4: CPU-ODS(1-3) remap GPU-ODS(4-7)).
//
// Two kernels: column_kernel, lane = record, the default (described below), and remap_kernel, by an
// element schedule, for tuned or forced shapes, records too wide for the other and the pairs of layouts
// that it moves faster (schedule_faster in capi.cu).  In both every warp works alone on chunks of R
// consecutive records, so that the main loop has no block-wide barrier.
// remap_kernel (R a multiple of 8):
//   1. the warp copies the chunk's slice of every source group into its own shared buffer with
//      16-byte cp.async (coalesced: lane l moves bytes 16l, 16l+512, ...): one chunk ahead of
//      the one it works on (two buffers), or, with one buffer, as soon as the moves have read
//      the current chunk (half the input buffers' shared memory, so more warps per SM);
//   2. it moves every field of every destination record, one move per lane per step: a move is
//      one field (8, 4 or 2 bytes, whole) or an aligned piece of zero padding (read from 16 zero
//      bytes after the chunk buffer), taken from a schedule table built once per CTA.  Moves into one-field destination groups are stored
//      straight to global memory (consecutive lanes on consecutive records, so the stores are
//      coalesced); moves into wider groups are assembled in a second buffer.  This is the tile
//      transpose between the source and destination record strides; the host picks, per move
//      class, the schedule order with the fewest shared-memory bank conflicts;
//   3. it writes the assembled wider destination slices back with 16-byte stores.
// Where each 16-byte piece of the two buffers lives in global memory is the same for every chunk
// up to the chunk's offset; when a buffer's slices are narrower than a warp step (many groups
// per step), a per-CTA table of the pieces replaces the search over the groups.
// Global traffic is one contiguous read stream per source group and one write stream per
// destination group.  The ragged tail (fewer than R records) goes move by move through the warp
// that would own the next chunk.
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "remap_common.cuh"
#include "staging.cuh"

namespace adha {

__device__ __forceinline__ int align16(int x) { return (x + 15) & ~15; }

template <bool DIRECT>
__global__ void __launch_bounds__(kThreads) remap_kernel(const __grid_constant__ RemapArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int in_pieces = (a.pieces & 1) ? a.in_bytes / 16 : 0, out_pieces = (a.pieces & 2) ? a.out_bytes / 16 : 0;
  Piece* pin = reinterpret_cast<Piece*>(smem);
  Piece* pout = pin + in_pieces;
  GroupRef* tin = reinterpret_cast<GroupRef*>(pout + out_pieces);
  GroupRef* tout = tin + a.n_src;
  const int n_entries = a.R * a.n_moves;
  uint32_t* sched = reinterpret_cast<uint32_t*>(tout + a.n_dst);
  uint8_t* wbase = reinterpret_cast<uint8_t*>(sched) + align16(n_entries * 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb = a.buffers;
  uint8_t* buf0 = wbase + (size_t)warp * (nb * (a.in_bytes + kZeroTail) + a.out_bytes);
  uint8_t* buf1 = buf0 + (nb - 1) * (a.in_bytes + kZeroTail);
  uint8_t* outb = buf0 + nb * (a.in_bytes + kZeroTail);
  if (lane < nb) *reinterpret_cast<uint4*>((lane ? buf1 : buf0) + a.in_bytes) = make_uint4(0, 0, 0, 0);

  for (int q = tid; q < in_pieces; q += kThreads) pin[q] = piece_of(q, a.src, a.R);
  for (int q = tid; q < out_pieces; q += kThreads) pout[q] = piece_of(q, a.dst, a.R);
  for (int k = tid; k < a.n_src; k += kThreads) tin[k] = a.src[k];
  for (int k = tid; k < a.n_dst; k += kThreads) tout[k] = a.dst[k];
  for (int t = tid; t < n_entries; t += kThreads)
    sched[t] = schedule_entry(t, a.R, a.cls_count, a.cls_order, a.move, a.src, a.dst, a.in_bytes);
  __syncthreads();

  const int64_t W = (int64_t)gridDim.x * kWarps;
  const int64_t R = a.R;
  // lane l moves pieces l, l + 32, ... (16 bytes each: coalesced within every slice), finding
  // each piece's group by a search that resumes where the last piece's ended, or in the table
  auto stage = [&](int64_t ch, uint8_t* buf) {
    if (a.pieces & 1) {
#pragma unroll 1
      for (int q = lane; q < in_pieces; q += 32) {
        const Piece pc = pin[q];
        cp_async16(buf + q * 16, pc.base + ch * pc.step);
      }
    } else {
      int g = 0;
      for (int p = lane * 16; p < a.in_bytes; p += 512) {
        while (p >= tin[g].start + a.R * tin[g].stride) ++g;
        cp_async16(buf + p, tin[g].ptr + ch * R * tin[g].stride + (p - tin[g].start));
      }
    }
  };

  int64_t c = (int64_t)blockIdx.x * kWarps + warp;
  if (c < a.n_chunks) stage(c, buf0);
  cp_async_commit();
  for (int i = 0; c < a.n_chunks; c += W, ++i) {
    uint8_t* cur = (i & 1) ? buf1 : buf0;
    if (nb == 2) {
      if (c + W < a.n_chunks) stage(c + W, (i & 1) ? buf0 : buf1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    move_chunk<DIRECT>(sched, a.R, a.cls_count, cur, outb, tout, c * R, lane);
    __syncwarp();
    if (nb == 1 && c + W < a.n_chunks) {   // one buffer: the next chunk once the moves have read this one
      stage(c + W, buf0);
      cp_async_commit();
    }
    if (a.pieces & 2) {
#pragma unroll 1
      for (int q = lane; q < out_pieces; q += 32) {
        const Piece pc = pout[q];
        *reinterpret_cast<uint4*>(const_cast<uint8_t*>(pc.base) + c * pc.step) =
            *reinterpret_cast<const uint4*>(outb + q * 16);
      }
    } else {
      write_back<DIRECT>(tout, a.R, a.out_bytes, outb, c, lane);
    }
    __syncwarp();
  }
  cp_async_wait<0>();

  // ragged tail: the warp whose next chunk would be n_chunks
  const int64_t t0 = a.n_chunks * R;
  if (c == a.n_chunks && t0 < a.n) tail_moves(t0, a.n, a.n_moves, a.cls_count, a.move, tin, tout, lane);
}

size_t remap_smem_bytes(const RemapArgs& a) {
  auto al = [](size_t x) { return (x + 15) / 16 * 16; };
  const size_t pieces = ((a.pieces & 1) ? a.in_bytes / 16 : 0) + ((a.pieces & 2) ? a.out_bytes / 16 : 0);
  return pieces * sizeof(Piece) + (size_t)(a.n_src + a.n_dst) * sizeof(GroupRef) + al((size_t)a.R * a.n_moves * 4) +
         (size_t)kWarps * ((size_t)a.buffers * ((size_t)a.in_bytes + kZeroTail) + a.out_bytes);
}

// ---------------------------------------------------------------------------------------------
// Remap by columns: the default for a pair of layouts that has not been tuned.
//
// The kernel above moves a chunk element by element through a schedule (three shared-memory
// accesses and the unpacking per element, a table of R x fields entries built by every CTA).  Here a
// lane is a record and a step is one field of 32 records, so that a field's place is one table entry
// for the whole chunk and the consecutive records of a one-field destination group are one coalesced
// store: such groups need no output buffer and no 16-byte copy loop.
//   into a one-field group:  shared load, global store
//   into a struct:           shared load, shared store; the structs go out in 16-byte pieces
// Sources come in in 16-byte pieces, slice by slice, or through the piece table of staging.cuh where
// there are several slices.  Structs of an even number of pieces are staged with 16 bytes of room, or
// 32 records' fields would lie on a few banks.  (One-field sources read straight into the structs, by
// 4-byte cp.async or through registers: 190 and 157-184 us per 1 GB where the staged form takes
// 157-183.)
template <int M>
struct Columns {
  const ColumnArgs& a;
  const ColMove* col;
  const ColSlice *in, *out;
  const StagePiece* tab;   // the input pieces of a chunk, NULL: slice by slice
  int n_pieces;
  int R, lane;
  uint8_t *ibuf, *obuf;   // the warp's buffers

  __device__ __forceinline__ bool on(int m, int cnt) const { return lane + 32 * m < cnt; }

  // Places of the 16-byte pieces of `bytes` bytes of a slice: f(piece offset in memory, in the buffer).
  template <class F>
  __device__ __forceinline__ void pieces(const ColSlice& s, int bytes, F f) const {
    if (s.stride & kColRoom) {
      for (int p = lane * 16; p < bytes; p += 512) f(p, p + 16 * (int)__umulhi((unsigned)p, s.magic));
    } else {
      for (int p = lane * 16; p < bytes; p += 512) f(p, p);
    }
  }

  // The chunk's source slices into the input buffer.
  template <bool WHOLE>
  __device__ __forceinline__ void stage(int64_t ch, int cnt) const {
    if (WHOLE && tab) return stage_chunk(tab, n_pieces, ch, ibuf, lane);
    const uint32_t si = smem_addr(ibuf);
    for (int k = 0; k < a.n_in; ++k) {
      const ColSlice s = in[k];
      const int stride = s.stride & kColStride, bytes = cnt * stride;
      const uint8_t* src = s.ptr + (uint64_t)(uint32_t)ch * (uint32_t)(R * stride);
      const uint32_t dst = si + s.at;
      pieces(s, bytes, [&](int p, int at) {
        if (WHOLE) cp_async16_at(dst + at, src + p);
        else cp_async16_part(dst + at, src + p, min(16, bytes - p));
      });
    }
  }

  template <class V, bool WHOLE>
  __device__ __forceinline__ void column_out(int k, int end, const uint8_t* src0, int64_t i0, int cnt) const {
    const int64_t at = (i0 + lane) * (int64_t)sizeof(V);
#pragma unroll 4
    for (; k < end; ++k) {
      const ColMove t = col[k];
      const uint8_t* src = src0 + t.off + lane * t.stride;
      V* dst = reinterpret_cast<V*>(const_cast<uint8_t*>(t.g) + at);
      V v[M];
#pragma unroll
      for (int m = 0; m < M; ++m)
        if ((WHOLE && M > 1) || on(m, cnt)) v[m] = *reinterpret_cast<const V*>(src + m * 32 * t.stride);
#pragma unroll
      for (int m = 0; m < M; ++m)
        if ((WHOLE && M > 1) || on(m, cnt)) dst[m * 32] = v[m];
    }
  }

  template <class V, bool WHOLE>
  __device__ __forceinline__ void column_across(int k, int end, const uint8_t* __restrict__ src0, uint8_t* __restrict__ dst0,
                                                int cnt) const {
#pragma unroll 4
    for (; k < end; ++k) {
      const ColMove t = col[k];
      const uint8_t* src = src0 + t.off + lane * t.stride;
      uint8_t* dst = dst0 + t.off2 + lane * t.stride2;
      V v[M];
#pragma unroll
      for (int m = 0; m < M; ++m)
        if ((WHOLE && M > 1) || on(m, cnt)) v[m] = *reinterpret_cast<const V*>(src + m * 32 * t.stride);
#pragma unroll
      for (int m = 0; m < M; ++m)
        if ((WHOLE && M > 1) || on(m, cnt)) *reinterpret_cast<V*>(dst + m * 32 * t.stride2) = v[m];
    }
  }

  template <bool WHOLE>
  __device__ __forceinline__ void moves(int64_t ch, int cnt) const {
    const int64_t i0 = ch * R;
    const uint8_t* src = ibuf;
    int k = 0, e = a.cnt[0];
    column_out<unsigned long long, WHOLE>(k, e, src, i0, cnt);
    k = e, e += a.cnt[1];
    column_out<uint32_t, WHOLE>(k, e, src, i0, cnt);
    k = e, e += a.cnt[2];
    column_out<uint16_t, WHOLE>(k, e, src, i0, cnt);
    k = e, e += a.cnt[3];
    column_across<unsigned long long, WHOLE>(k, e, src, obuf, cnt);
    k = e, e += a.cnt[4];
    column_across<uint32_t, WHOLE>(k, e, src, obuf, cnt);
    k = e, e += a.cnt[5];
    column_across<uint16_t, WHOLE>(k, e, src, obuf, cnt);
  }

  // The built (or carried) structs of the chunk to memory.
  template <bool WHOLE>
  __device__ __forceinline__ void write_out(int64_t ch, int cnt) const {
    for (int k = 0; k < a.n_out; ++k) {
      const ColSlice s = out[k];
      const int stride = s.stride & kColStride, bytes = cnt * stride;
      uint8_t* dst = const_cast<uint8_t*>(s.ptr) + (uint64_t)(uint32_t)ch * (uint32_t)(R * stride);
      const uint8_t* src = (s.stride & kColFromIn ? ibuf : obuf) + s.at;
      pieces(s, bytes, [&](int p, int at) {
        if (WHOLE || p + 16 <= bytes) {
          *reinterpret_cast<uint4*>(dst + p) = *reinterpret_cast<const uint4*>(src + at);
        } else {
          for (int q = 0; q < bytes - p; q += 2)
            *reinterpret_cast<uint16_t*>(dst + p + q) = *reinterpret_cast<const uint16_t*>(src + at + q);
        }
      });
    }
  }
};

template <int M>
__global__ void __launch_bounds__(kThreads, 4) column_kernel(const __grid_constant__ ColumnArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int n_col = 0;
  for (int k = 0; k < kColClasses; ++k) n_col += a.cnt[k];
  ColMove* col = reinterpret_cast<ColMove*>(smem);
  ColSlice* in = reinterpret_cast<ColSlice*>(col + n_col);
  ColSlice* out = in + a.n_in;
  for (int k = tid; k < n_col; k += kThreads) col[k] = a.col[k];
  for (int k = tid; k < a.n_in; k += kThreads) in[k] = a.in[k];
  for (int k = tid; k < a.n_out; k += kThreads) out[k] = a.out[k];
  const int R = M == 1 ? a.R : 32 * M;
  StagePiece* tab = reinterpret_cast<StagePiece*>(out + a.n_out);
  for (int q = tid; q < a.n_pieces; q += kThreads) {
    int p = q * 16, k = 0;
    while (p >= R * (a.in[k].stride & kColStride)) p -= R * (a.in[k++].stride & kColStride);
    const int stride = a.in[k].stride & kColStride;
    const int room = a.in[k].stride & kColRoom ? 16 * (int)__umulhi((unsigned)p, a.in[k].magic) : 0;
    tab[q] = StagePiece{a.in[k].ptr + p, R * stride, a.in[k].at + p + room};
  }
  uint8_t* mine = reinterpret_cast<uint8_t*>(tab + a.n_pieces) + (size_t)warp * (a.in_bytes + a.out_bytes);
  if (a.fill)
    for (int p = lane * 16; p < a.out_bytes; p += 512)
      *reinterpret_cast<uint4*>(mine + a.in_bytes + p) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  const Columns<M> w{a, col, in, out, a.n_pieces ? tab : nullptr, a.n_pieces, R, lane, mine, mine + a.in_bytes};
  const int64_t W = (int64_t)gridDim.x * kWarps;
  // the next chunk may come in once the moves have read this one, unless groups are written from it
  bool early = true;
  for (int k = 0; k < a.n_out; ++k) early = early && !(out[k].stride & kColFromIn);

  int64_t c = (int64_t)blockIdx.x * kWarps + warp;
  if (c < a.n_chunks) w.template stage<true>(c, R);
  cp_async_commit();
  for (; c < a.n_chunks; c += W) {
    const bool more = c + W < a.n_chunks;
    cp_async_wait<0>();
    __syncwarp();
    w.template moves<true>(c, R);
    __syncwarp();
    if (early && more) {
      w.template stage<true>(c + W, R);
      cp_async_commit();
    }
    w.template write_out<true>(c, R);
    __syncwarp();
    if (!early && more) {
      w.template stage<true>(c + W, R);
      cp_async_commit();
    }
  }
  // fewer than R records at the end: the warp whose next chunk would be n_chunks
  const int rest = (int)(a.n - a.n_chunks * R);
  if (c == a.n_chunks && rest > 0) {
    cp_async_wait<0>();
    __syncwarp();
    w.template stage<false>(c, rest);
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    w.template moves<false>(c, rest);
    __syncwarp();
    w.template write_out<false>(c, rest);
  }
  cp_async_wait<0>();
}

size_t columns_smem_bytes(const ColumnArgs& a) {
  int n_col = 0;
  for (int k = 0; k < kColClasses; ++k) n_col += a.cnt[k];
  return (size_t)(n_col + a.n_in + a.n_out + a.n_pieces) * 16 + (size_t)kWarps * ((size_t)a.in_bytes + a.out_bytes);
}

template <int M>
static int launch_c(const ColumnArgs& a, int grid, size_t smem, void* stream) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(column_kernel<M>), smem, "cudaFuncSetAttribute(columns)")) return rc;
  column_kernel<M><<<grid, kThreads, smem, (cudaStream_t)stream>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "column remap launch");
  return 0;
}

int launch_columns(const ColumnArgs& a, int grid, size_t smem, void* stream) {
  return a.R == 128  ? launch_c<4>(a, grid, smem, stream)
         : a.R == 64 ? launch_c<2>(a, grid, smem, stream)
                     : launch_c<1>(a, grid, smem, stream);
}

template <int M>
static int occ_c(size_t smem, int* blocks) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(column_kernel<M>), smem, "cudaFuncSetAttribute(columns)")) return rc;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, column_kernel<M>, kThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor(columns)");
  return 0;
}

int columns_occupancy(int R, size_t smem, int* blocks) {
  return R == 128 ? occ_c<4>(smem, blocks) : R == 64 ? occ_c<2>(smem, blocks) : occ_c<1>(smem, blocks);
}

template <bool DIRECT>
static int launch_d(const RemapArgs& a, int grid, size_t smem, void* stream) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(remap_kernel<DIRECT>), smem, "cudaFuncSetAttribute(remap)")) return rc;
  remap_kernel<DIRECT><<<grid, kThreads, smem, (cudaStream_t)stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "remap kernel launch");
  return 0;
}

int launch_remap(const RemapArgs& a, int grid, size_t smem, void* stream) {
  const bool direct = a.cls_count[0] + a.cls_count[1] + a.cls_count[2] > 0;
  return direct ? launch_d<true>(a, grid, smem, stream) : launch_d<false>(a, grid, smem, stream);
}

template <bool DIRECT>
static int occ_d(size_t smem, int* blocks) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(remap_kernel<DIRECT>), smem, "cudaFuncSetAttribute(remap)")) return rc;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, remap_kernel<DIRECT>, kThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor(remap)");
  return 0;
}

int remap_occupancy(int direct, size_t smem, int* blocks) {
  return direct ? occ_d<true>(smem, blocks) : occ_d<false>(smem, blocks);
}

}  // namespace adha
