// chain.cu -- a run of fp32 chain sections (axpb, mul, tanh) and its gradient in one pass each
// (paper Section 2: the combine edge joins consecutive sections that share a layout).
//
// Section by section, a forward + backward step moves about 16 + 32 bytes per record and section,
// all of it through HBM: 51 GB for 64 sections over 2^24 records, 9.0 ms of a 10.0 ms step.  Here
// a warp holds a chunk of R = 32*M records in shared memory, one row of R floats per field, and
// walks the whole run there, so HBM sees each field once:
//   forward:  read the fields, write the written ones, and keep their values from before the run
//             (`saved`, one row per written field);
//   backward: read `saved` (and the fields the run does not write), write them back into the
//             state, run the sections again in shared memory, then walk them in reverse on the
//             adjoints: read once, written once.
// At 24 fields that is 288 + 384 bytes per record against 64 x 48.  Running the sections again costs
// arithmetic (the tanh polynomials), not memory: a lane's records are carried as pairs in the packed
// fp32 instructions (each half an IEEE operation on its own, as in the per-record rule).
//
// What the reverse walk needs of the values in between is found on the host (chain.cu's planner): a
// version of a field is needed if a mul reads it or a tanh made it (the tanh adjoint takes
// t = tanh(x) from the section's own result).  Only needed versions go to the tape when they are
// overwritten, and only sections that lead to one are run again.
//
// M: two records per lane (one packed pair), one where the rows and the tape of two leave fewer than 12
// warps per SM (forward) or 8 (backward) in shared memory.  The walk's per-section work (operands,
// branch, loop) is shared by a lane's records, but with four the warps that are left show the walk's
// latency.  The forward pass gets 16 waves of CTAs, which evens out the SMs' distances from memory;
// the backward pass is not bound by it.  Measured, 64 sections (23 of 24 fields written, 39 run
// again, 14 tape values) over 2^24 records, one array per field:
//   M         4                2                1
//   forward   0.94 - 0.97 ms   0.91 (one wave: 1.00)   2.1     (64 section launches with saves: 2.8 ms)
//   backward  3.07 ms          2.06 ms          2.58    (64 adjoint launches and a copy of the gradients: 6.1 ms)
// What bounds it now: forward HBM at 0.78 of the copy bandwidth; backward the walk's chains of dependent
// shared-memory loads and packed arithmetic at 12 warps per SM.  Operands from the parameter space
// instead of shared memory one section ahead: 1.07 and 2.47 ms; two IEEE divisions per tanh pair
// instead of tanh_pair's quotient: backward 2.24 ms.
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "section_ops.cuh"

namespace adha {

constexpr int kChainWarps = kChainThreads / 32;

// Bytes of the tables before the warps' rows.
__host__ __device__ __forceinline__ int chain_tables(const ChainArgs& a, bool backward) {
  return a.n_rows * (int)sizeof(ChainRow) + (a.n_sec + (backward ? a.n_live : 0)) * (int)sizeof(ChainSec);
}

// M floats of a lane as packed pairs (M = 1: the upper half is zero).
template <int M>
struct LaneVec {
  static constexpr int H = (M + 1) / 2;
  unsigned long long p[H];
  __device__ __forceinline__ void load(const uint8_t* q) {
    if constexpr (M == 2) {
      p[0] = *reinterpret_cast<const unsigned long long*>(q);
    } else {
      p[0] = f2_pack(*reinterpret_cast<const float*>(q), 0.0f);
    }
  }
  __device__ __forceinline__ void store(uint8_t* q) const {
    if constexpr (M == 2) {
      *reinterpret_cast<unsigned long long*>(q) = p[0];
    } else {
      float lo, hi;
      f2_unpack(p[0], &lo, &hi);
      *reinterpret_cast<float*>(q) = lo;
    }
  }
};

// One section on the lane's records (`s`: the lane's first record of row 0); TAPE: z's value from
// before it goes to its tape slot, if it has one.
template <int M, bool TAPE>
__device__ __forceinline__ void chain_section(const ChainSec& c, uint8_t* s, uint8_t* tape, const unsigned long long* P,
                                              const unsigned long long* Q, unsigned long long nz) {
  constexpr int H = LaneVec<M>::H;
  LaneVec<M> x, v;
  x.load(s + c.x);
  if (TAPE && c.tape >= 0) {
    v.load(s + c.z);
    v.store(tape + c.tape);
  }
  if (c.op == ADHA_OP_AXPB) {
#pragma unroll
    for (int h = 0; h < H; ++h) v.p[h] = f2_add_rn(f2_mul_alone(f2_pack(c.a, c.a), x.p[h], nz), f2_pack(c.b, c.b));
  } else if (c.op == ADHA_OP_MUL) {
    LaneVec<M> y;
    y.load(s + c.y);
#pragma unroll
    for (int h = 0; h < H; ++h) v.p[h] = f2_mul_alone(x.p[h], y.p[h], nz);
  } else {
#pragma unroll
    for (int h = 0; h < H; ++h) v.p[h] = tanh_pair(x.p[h], P, Q, nz);
  }
  v.store(s + c.z);
}

// The adjoint of one section (adha_section_backward's rule, in its order): z restored from the tape,
// gz = g[z], g[z] = 0, then g[x] (and g[y]) added to.  Every step goes through shared memory in
// program order, so x, y and z may be the same field in any combination.
template <int M>
__device__ __forceinline__ void chain_adjoint(const ChainSec& c, uint8_t* s, uint8_t* g, const uint8_t* tape,
                                              unsigned long long nz) {
  constexpr int H = LaneVec<M>::H;
  LaneVec<M> gz, gx, t, zero, old;
#pragma unroll
  for (int h = 0; h < H; ++h) zero.p[h] = 0ull;
  gz.load(g + c.z);
  zero.store(g + c.z);
  gx.load(g + c.x);
  if (c.op == ADHA_OP_AXPB) {
#pragma unroll
    for (int h = 0; h < H; ++h) gx.p[h] = f2_add_rn(gx.p[h], f2_mul_alone(f2_pack(c.a, c.a), gz.p[h], nz));
    gx.store(g + c.x);
    if (c.tape >= 0) {
      old.load(tape + c.tape);
      old.store(s + c.z);
    }
  } else if (c.op == ADHA_OP_TANH) {
    t.load(s + c.z);   // the section's result: tanh(x)
    const unsigned long long one = f2_pack(1.0f, 1.0f);
#pragma unroll
    for (int h = 0; h < H; ++h)
      gx.p[h] = f2_add_rn(gx.p[h], f2_mul_alone(gz.p[h], f2_sub_rn(one, f2_mul_alone(t.p[h], t.p[h], nz)), nz));
    gx.store(g + c.x);
    if (c.tape >= 0) {
      old.load(tape + c.tape);
      old.store(s + c.z);
    }
  } else {
    LaneVec<M> x, y, gy;
    if (c.tape >= 0) {   // before x and y are read: either may be z
      old.load(tape + c.tape);
      old.store(s + c.z);
    }
    x.load(s + c.x);
    y.load(s + c.y);
#pragma unroll
    for (int h = 0; h < H; ++h) gx.p[h] = f2_add_rn(gx.p[h], f2_mul_alone(gz.p[h], y.p[h], nz));
    gx.store(g + c.x);
    gy.load(g + c.y);
#pragma unroll
    for (int h = 0; h < H; ++h) gy.p[h] = f2_add_rn(gy.p[h], f2_mul_alone(gz.p[h], x.p[h], nz));
    gy.store(g + c.y);
  }
}

// Which of a row's addresses a load or store uses.
enum ChainSide { kState, kGradIn, kGradOut };

template <ChainSide SIDE>
__device__ __forceinline__ uint8_t* row_base(const ChainRow& r) {
  return SIDE == kState ? r.state : SIDE == kGradIn ? const_cast<uint8_t*>(r.gin) : r.gout;
}

// Rows that are one contiguous array (one-field groups): 16-byte pieces, all rows in one walk.
// FROM_SAVED: rows of written fields come from `saved` (contiguous whatever the layout), and rows
// of wide groups that are not written are left to load_wide.
template <int M, ChainSide SIDE, bool FROM_SAVED>
__device__ __forceinline__ void load_rows(const ChainArgs& a, const ChainRow* rows, uint8_t* buf, int64_t i0, int lane) {
  constexpr int PP = 8 * M;   // pieces per row
  for (int p = lane; p < a.n_rows * PP; p += 32) {
    const ChainRow& r = rows[p / PP];
    const int q = (p % PP) * 16;
    if (FROM_SAVED && r.saved >= 0) cp_async16(buf + p * 16, reinterpret_cast<const uint8_t*>(a.saved + r.saved * a.pitch + i0) + q);
    else if (r.stride == 4) cp_async16(buf + p * 16, row_base<SIDE>(r) + i0 * 4 + q);
  }
}

// Rows of groups wider than one field: lane = record, 16 bytes at a time where the struct allows,
// else field by field.  SKIP_SAVED: only rows whose field the run does not write.
template <int M, ChainSide SIDE, bool SKIP_SAVED>
__device__ __forceinline__ void load_wide(const ChainArgs& a, const ChainRow* rows, uint8_t* buf, int64_t i0, int lane) {
  constexpr int R = 32 * M;
  for (int k = 0; k < a.n_wide; ++k) {
    const int row0 = a.wide_row[k], nf = a.wide_len[k], stride = rows[row0].stride;
    const uint8_t* base = row_base<SIDE>(rows[row0]) + (i0 + lane) * stride;
    float* dst = reinterpret_cast<float*>(buf) + row0 * R + lane;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint8_t* q = base + (int64_t)(32 * m) * stride;
      if (!SKIP_SAVED && stride % 16 == 0) {
#pragma unroll 4
        for (int j = 0; j < nf; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(q + 4 * j);
          float* d = dst + j * R + 32 * m;
          d[0] = v.x;
          d[R] = v.y;
          d[2 * R] = v.z;
          d[3 * R] = v.w;
        }
      } else {
#pragma unroll 4
        for (int j = 0; j < nf; ++j)
          if (!SKIP_SAVED || rows[row0 + j].saved < 0) dst[j * R + 32 * m] = *reinterpret_cast<const float*>(q + 4 * j);
      }
    }
  }
}

// Rows back to memory: contiguous rows in 16-byte pieces, wide groups lane = record.  WRITTEN: only
// what the run writes (a wide group with a written field goes back whole where 16 bytes fit).
template <int M, ChainSide SIDE, bool WRITTEN>
__device__ __forceinline__ void store_rows(const ChainArgs& a, const ChainRow* rows, const uint8_t* buf, int64_t i0,
                                           int lane) {
  constexpr int R = 32 * M, PP = 8 * M;
  for (int p = lane; p < a.n_rows * PP; p += 32) {
    const ChainRow& r = rows[p / PP];
    if (r.stride == 4 && (!WRITTEN || r.saved >= 0))
      *reinterpret_cast<uint4*>(row_base<SIDE>(r) + i0 * 4 + (p % PP) * 16) = *reinterpret_cast<const uint4*>(buf + p * 16);
  }
  for (int k = 0; k < a.n_wide; ++k) {
    if (WRITTEN && !a.wide_written[k]) continue;
    const int row0 = a.wide_row[k], nf = a.wide_len[k], stride = rows[row0].stride;
    uint8_t* base = row_base<SIDE>(rows[row0]) + (i0 + lane) * stride;
    const float* src = reinterpret_cast<const float*>(buf) + row0 * R + lane;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      uint8_t* q = base + (int64_t)(32 * m) * stride;
      if (stride % 16 == 0) {
#pragma unroll 4
        for (int j = 0; j < nf; j += 4) {
          const float* d = src + j * R + 32 * m;
          *reinterpret_cast<float4*>(q + 4 * j) = make_float4(d[0], d[R], d[2 * R], d[3 * R]);
        }
      } else {
        for (int j = 0; j < nf; ++j)
          if (!WRITTEN || rows[row0 + j].saved >= 0) *reinterpret_cast<float*>(q + 4 * j) = src[j * R + 32 * m];
      }
    }
  }
}

// The last chunk, fewer than R records: field by field, records beyond n as zeros.
template <int M, ChainSide SIDE, bool FROM_SAVED>
__device__ __forceinline__ void load_tail(const ChainArgs& a, const ChainRow* rows, uint8_t* buf, int64_t i0, int lane) {
  for (int k = 0; k < a.n_rows; ++k) {
    const ChainRow& r = rows[k];
    for (int m = 0; m < M; ++m) {
      const int64_t i = i0 + lane + 32 * m;
      float v = 0.0f;
      if (i < a.n) {
        if (FROM_SAVED && r.saved >= 0) v = a.saved[r.saved * a.pitch + i];
        else v = *reinterpret_cast<const float*>(row_base<SIDE>(r) + i * r.stride);
      }
      reinterpret_cast<float*>(buf)[k * 32 * M + lane + 32 * m] = v;
    }
  }
}

template <int M, ChainSide SIDE, bool WRITTEN>
__device__ __forceinline__ void store_tail(const ChainArgs& a, const ChainRow* rows, const uint8_t* buf, int64_t i0,
                                           int lane) {
  for (int k = 0; k < a.n_rows; ++k) {
    const ChainRow& r = rows[k];
    if (WRITTEN && r.saved < 0) continue;
    for (int m = 0; m < M; ++m) {
      const int64_t i = i0 + lane + 32 * m;
      if (i < a.n) *reinterpret_cast<float*>(row_base<SIDE>(r) + i * r.stride) = reinterpret_cast<const float*>(buf)[k * 32 * M + lane + 32 * m];
    }
  }
}

// The row table and the sections' operands in shared memory, one copy per CTA: the walks read an
// operand block with two broadcast loads, one section ahead of its use.
template <class T>
__device__ __forceinline__ T* copy_table(const T* from, int n, uint8_t* to) {
  static_assert(sizeof(T) % 16 == 0, "copied in 16-byte words");
  for (int k = threadIdx.x; k < n * (int)(sizeof(T) / 16); k += kChainThreads)
    reinterpret_cast<uint4*>(to)[k] = reinterpret_cast<const uint4*>(from)[k];
  return reinterpret_cast<T*>(to);
}

template <int M>
__global__ void __launch_bounds__(kChainThreads) chain_forward_kernel(const __grid_constant__ ChainArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int R = 32 * M, R4 = R * 4, PP = 8 * M;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const ChainRow* rows = copy_table(a.row, a.n_rows, smem);
  const ChainSec* sec = copy_table(a.sec, a.n_sec, smem + a.n_rows * sizeof(ChainRow));
  __syncthreads();
  uint8_t* S = smem + chain_tables(a, false) + (size_t)warp * a.n_rows * R4;
  uint8_t* mine = S + lane * M * 4;
  for (int64_t c = (int64_t)blockIdx.x * kChainWarps + warp; c < a.n_chunks; c += (int64_t)gridDim.x * kChainWarps) {
    const int64_t i0 = c * R;
    const bool whole = i0 + R <= a.n;
    if (whole) {
      load_rows<M, kState, false>(a, rows, S, i0, lane);
      cp_async_commit();
      load_wide<M, kState, false>(a, rows, S, i0, lane);
      cp_async_wait<0>();
    } else {
      load_tail<M, kState, false>(a, rows, S, i0, lane);
    }
    __syncwarp();
    // the written fields' values from before the run (rows of `saved` are padded to whole chunks)
    for (int p = lane; p < a.n_rows * PP; p += 32) {
      const int sv = rows[p / PP].saved;
      if (sv >= 0)
        *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(a.saved + sv * a.pitch + i0) + (p % PP) * 16) =
            *reinterpret_cast<const uint4*>(S + p * 16);
    }
    __syncwarp();
    ChainSec next = sec[0];
#pragma unroll 1
    for (int s = 0; s < a.n_sec; ++s) {
      const ChainSec c = next;
      next = sec[min(s + 1, a.n_sec - 1)];
      chain_section<M, false>(c, mine, nullptr, a.tanh_p, a.tanh_qn, a.neg_zero);
    }
    __syncwarp();
    if (whole) store_rows<M, kState, true>(a, rows, S, i0, lane);
    else store_tail<M, kState, true>(a, rows, S, i0, lane);
    __syncwarp();
  }
}

template <int M>
__global__ void __launch_bounds__(kChainThreads) chain_backward_kernel(const __grid_constant__ ChainArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int R = 32 * M, R4 = R * 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const ChainRow* rows = copy_table(a.row, a.n_rows, smem);
  const ChainSec* sec = copy_table(a.sec, a.n_sec, smem + a.n_rows * sizeof(ChainRow));
  const ChainSec* live = copy_table(a.live, a.n_live, smem + a.n_rows * sizeof(ChainRow) + a.n_sec * sizeof(ChainSec));
  __syncthreads();
  uint8_t* S = smem + chain_tables(a, true) + (size_t)warp * (2 * a.n_rows + a.n_tape) * R4;
  uint8_t* G = S + a.n_rows * R4;
  uint8_t* T = G + a.n_rows * R4;
  const int at = lane * M * 4;
  for (int64_t c = (int64_t)blockIdx.x * kChainWarps + warp; c < a.n_chunks; c += (int64_t)gridDim.x * kChainWarps) {
    const int64_t i0 = c * R;
    const bool whole = i0 + R <= a.n;
    if (whole) {
      load_rows<M, kState, true>(a, rows, S, i0, lane);
      cp_async_commit();
      load_rows<M, kGradIn, false>(a, rows, G, i0, lane);   // arrives while the sections run again
      cp_async_commit();
      load_wide<M, kState, true>(a, rows, S, i0, lane);
      load_wide<M, kGradIn, false>(a, rows, G, i0, lane);
      cp_async_wait<1>();
    } else {
      load_tail<M, kState, true>(a, rows, S, i0, lane);
      load_tail<M, kGradIn, false>(a, rows, G, i0, lane);
    }
    __syncwarp();
    // the state as it was before the run
    if (whole) store_rows<M, kState, true>(a, rows, S, i0, lane);
    else store_tail<M, kState, true>(a, rows, S, i0, lane);
    __syncwarp();
    ChainSec next = live[0];
#pragma unroll 1
    for (int s = 0; s < a.n_live; ++s) {
      const ChainSec c = next;
      next = live[min(s + 1, a.n_live - 1)];
      chain_section<M, true>(c, S + at, T + at, a.tanh_p, a.tanh_qn, a.neg_zero);
    }
    next = sec[a.n_sec - 1];
    cp_async_wait<0>();
    __syncwarp();
#pragma unroll 1
    for (int s = a.n_sec - 1; s >= 0; --s) {
      const ChainSec c = next;
      next = sec[max(s - 1, 0)];
      chain_adjoint<M>(c, S + at, G + at, T + at, a.neg_zero);
    }
    __syncwarp();
    if (whole) store_rows<M, kGradOut, false>(a, rows, G, i0, lane);
    else store_tail<M, kGradOut, false>(a, rows, G, i0, lane);
    // gradients of groups the run does not touch, when they go to buffers of their own
    for (int k = 0; k < a.n_copy; ++k) {
      const ChainCopy& cp = a.copy[k];
      const int64_t b0 = i0 * cp.stride;
      const int bytes = (int)((whole ? (int64_t)R : a.n - i0) * cp.stride);
      for (int p = lane * 4; p < bytes; p += 128)
        *reinterpret_cast<float*>(cp.dst + b0 + p) = *reinterpret_cast<const float*>(cp.src + b0 + p);
    }
    __syncwarp();
  }
}

size_t chain_smem_bytes(const ChainArgs& a, int M, bool backward) {
  return chain_tables(a, backward) + (size_t)kChainWarps * (backward ? 2 * a.n_rows + a.n_tape : a.n_rows) * 128 * M;
}

template <class K>
static int launch_k(K kernel, const ChainArgs& a, int grid, size_t smem, void* stream) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(kernel), smem, "cudaFuncSetAttribute(chain)")) return rc;
  kernel<<<grid, kChainThreads, smem, (cudaStream_t)stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "chain kernel launch");
  return 0;
}

template <class K>
static int occ_k(K kernel, size_t smem, int* blocks) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(kernel), smem, "cudaFuncSetAttribute(chain)")) return rc;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kernel, kChainThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor(chain)");
  return 0;
}

int launch_chain(const ChainArgs& a, int M, bool backward, int grid, size_t smem, void* stream) {
  if (backward) return M == 2 ? launch_k(chain_backward_kernel<2>, a, grid, smem, stream)
                              : launch_k(chain_backward_kernel<1>, a, grid, smem, stream);
  return M == 2 ? launch_k(chain_forward_kernel<2>, a, grid, smem, stream)
                : launch_k(chain_forward_kernel<1>, a, grid, smem, stream);
}

int chain_occupancy(int M, bool backward, size_t smem, int* blocks) {
  if (backward) return M == 2 ? occ_k(chain_backward_kernel<2>, smem, blocks) : occ_k(chain_backward_kernel<1>, smem, blocks);
  return M == 2 ? occ_k(chain_forward_kernel<2>, smem, blocks) : occ_k(chain_forward_kernel<1>, smem, blocks);
}

}  // namespace adha
