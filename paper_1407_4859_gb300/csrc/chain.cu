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
// What the reverse walk needs of the values in between is found on the host (chain_slots in capi.cu): a
// version of a field is needed if a mul reads it or a tanh made it (the tanh adjoint takes
// t = tanh(x) from the section's own result).  Only sections that lead to a needed version are run
// again, and each version gets a slot of its own, so that nothing is copied or restored: the slot of a
// version that is no longer needed, or a new one.  Gradients that are zero because they have just been
// passed on are known there too: they are read from one row of zeros, and not stored.
//
// A CTA is one warp, so that the walks' loops are uniform to the compiler: the operand records come
// from the parameter space into uniform registers one section ahead, 32 bytes of ready offsets, and an
// address is one register plus one uniform register.  (Records in shared memory took 2 of 3 of the walk's
// shared-memory instructions; records packed into 16 bytes took a third more instructions.)
//
// M: two records per lane (one packed pair), one where the rows and slots of two leave fewer than 12
// warps per SM (forward) or 8 (backward) in shared memory.  The walk's per-section work (operands,
// branch, loop) is shared by a lane's records, but with four the warps that are left show the walk's
// latency.  16 waves of CTAs even out the SMs' distances from memory and the ends of their chunks
// (backward with 1 wave 1.715 ms, 4 1.681, 8 1.655, 16 1.63).
//
// Measured, 64 sections (23 of 24 fields written, 39 run again, 9 slots beyond the fields') over 2^24
// records, one array per field:
//   forward   0.726 ms (64 section launches with saves: 2.8 ms); records in shared memory 0.910
//   backward  1.63 ms (64 adjoint launches and a copy of the gradients: 6.1 ms); with a tape that old
//             values were copied to and restored from, stored zeros and records in shared memory 2.060
// What bounds it now: forward HBM, at 0.95 of the copy bandwidth; backward the walk's chains of dependent
// shared-memory loads and packed arithmetic at 13 warps per SM (shared memory; issue active 0.55).
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "section_ops.cuh"

namespace adha {

// Bytes of the span lists before the warp's rows.
__host__ __device__ __forceinline__ int chain_tables(const ChainArgs& a) {
  int n = 0;
  for (int k = 0; k < 4; ++k) n += a.n_span[k];
  return n * (int)sizeof(ChainSpan);
}

// A lane's M floats, 1 or 2, as a packed pair (M = 1: the upper half is zero).
template <int M>
__device__ __forceinline__ unsigned long long lane_load(const uint8_t* q) {
  if constexpr (M == 2) return *reinterpret_cast<const unsigned long long*>(q);
  return f2_pack(*reinterpret_cast<const float*>(q), 0.0f);
}
template <int M>
__device__ __forceinline__ void lane_store(uint8_t* q, unsigned long long v) {
  if constexpr (M == 2) {
    *reinterpret_cast<unsigned long long*>(q) = v;
  } else {
    float lo, hi;
    f2_unpack(v, &lo, &hi);
    *reinterpret_cast<float*>(q) = lo;
  }
}

// One section on the lane's records (`s`: the lane's first record of row 0).
template <int M>
__device__ __forceinline__ void chain_section(const ChainSec& c, uint8_t* s, const unsigned long long* P,
                                              const unsigned long long* Q, unsigned long long nz) {
  const unsigned long long x = lane_load<M>(s + c.x);
  unsigned long long v;
  if (c.op == ADHA_OP_AXPB) {
    v = f2_add_rn(f2_mul_alone(f2_pack(c.a, c.a), x, nz), f2_pack(c.b, c.b));
  } else if (c.op == ADHA_OP_MUL) {
    v = f2_mul_alone(x, lane_load<M>(s + c.y), nz);
  } else {
    v = tanh_pair(x, P, Q, nz);
  }
  lane_store<M>(s + c.z, v);
}

// The adjoint of one section (adha_section_backward's rule, in its order): gz = g[z], g[z] = 0, then
// g[x] (and g[y]) added to.  A zero is not stored: the planner knows which gradients are zero when and
// has them read from the row of zeros; zero_rows says which are left so.
template <int M>
__device__ __forceinline__ void chain_adjoint(const ChainAdj& c, const uint8_t* s, uint8_t* g, unsigned long long nz) {
  const unsigned long long gz = lane_load<M>(g + c.gz);
  unsigned long long gx = lane_load<M>(g + c.gx_in);
  if (c.op == ADHA_OP_AXPB) {
    gx = f2_add_rn(gx, f2_mul_alone(f2_pack(c.a, c.a), gz, nz));
  } else if (c.op == ADHA_OP_TANH) {
    const unsigned long long t = lane_load<M>(s + c.vx), one = f2_pack(1.0f, 1.0f);
    gx = f2_add_rn(gx, f2_mul_alone(gz, f2_sub_rn(one, f2_mul_alone(t, t, nz)), nz));
  } else {
    const unsigned long long x = lane_load<M>(s + c.vx), y = lane_load<M>(s + c.vy);
    lane_store<M>(g + c.gx, f2_add_rn(gx, f2_mul_alone(gz, y, nz)));
    // after the store: x and y may be the same field
    lane_store<M>(g + c.gy, f2_add_rn(lane_load<M>(g + c.gy_in), f2_mul_alone(gz, x, nz)));
    return;
  }
  lane_store<M>(g + c.gx, gx);
}

// Which of a row's addresses a load or store uses.
enum ChainSide { kState, kGradIn, kGradOut };

template <ChainSide SIDE>
__device__ __forceinline__ uint8_t* row_base(const ChainRow& r) {
  return SIDE == kState ? r.state : SIDE == kGradIn ? const_cast<uint8_t*>(r.gin) : r.gout;
}

// Contiguous arrays to rows or back, 16-byte pieces; a piece's place within its row depends on the lane
// alone, so a piece costs one table load, one address addition and the copy.
template <int M>
__device__ __forceinline__ void load_spans(const ChainSpan* t, int n, uint8_t* buf, int64_t i0, int lane) {
  constexpr int PP = 8 * M;   // pieces per row
  const int64_t from = i0 * 4 + lane % PP * 16;
  uint8_t* to = buf + lane % PP * 16;
#pragma unroll 2
  for (int k = lane / PP; k < n; k += 32 / PP) {
    const ChainSpan s = t[k];
    cp_async16(to + s.at, s.base + from);
  }
}
template <int M>
__device__ __forceinline__ void store_spans(const ChainSpan* t, int n, const uint8_t* buf, int64_t i0, int lane) {
  constexpr int PP = 8 * M;
  const int64_t to = i0 * 4 + lane % PP * 16;
  const uint8_t* from = buf + lane % PP * 16;
#pragma unroll 2
  for (int k = lane / PP; k < n; k += 32 / PP) {
    const ChainSpan s = t[k];
    *reinterpret_cast<uint4*>(s.base + to) = *reinterpret_cast<const uint4*>(from + s.at);
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

// Rows of wide groups back to memory, lane = record.  WRITTEN: only what the run writes (a group with
// a written field goes back whole where 16 bytes fit).
template <int M, ChainSide SIDE, bool WRITTEN>
__device__ __forceinline__ void store_wide(const ChainArgs& a, const ChainRow* rows, const uint8_t* buf, int64_t i0,
                                           int lane) {
  constexpr int R = 32 * M;
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

// Spans list l of the launch, copied to shared memory after the lists before it.
__device__ __forceinline__ const ChainSpan* spans(const ChainArgs& a, int l, uint8_t* smem) {
  int first = 0;
  for (int k = 0; k < l; ++k) first += a.n_span[k];
  ChainSpan* t = reinterpret_cast<ChainSpan*>(smem) + first;
  for (int k = threadIdx.x; k < a.n_span[l]; k += kChainThreads) t[k] = a.span[l][k];
  return t;
}

template <int M>
__global__ void __launch_bounds__(kChainThreads) chain_forward_kernel(const __grid_constant__ ChainArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int R = 32 * M;
  const int lane = threadIdx.x;
  const ChainRow* rows = a.row;
  const ChainSec* sec = a.sec;
  const ChainSpan *in = spans(a, 0, smem), *save = spans(a, 1, smem), *out = spans(a, 2, smem);
  __syncthreads();
  uint8_t* S = smem + chain_tables(a);
  uint8_t* mine = S + lane * M * 4;
  for (int64_t c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
    const int64_t i0 = c * R;
    const bool whole = i0 + R <= a.n;
    if (whole) {
      load_spans<M>(in, a.n_span[0], S, i0, lane);
      cp_async_commit();
      load_wide<M, kState, false>(a, rows, S, i0, lane);
      cp_async_wait<0>();
    } else {
      load_tail<M, kState, false>(a, rows, S, i0, lane);
    }
    __syncwarp();
    // the written fields' values from before the run (rows of `saved` are padded to whole chunks)
    store_spans<M>(save, a.n_span[1], S, i0, lane);
    __syncwarp();
    ChainSec next = sec[0];
#pragma unroll 1
    for (int s = 0; s < a.n_sec; ++s) {
      const ChainSec c = next;
      next = sec[s + 1];   // one beyond the last is never run
      chain_section<M>(c, mine, a.tanh_p, a.tanh_qn, a.neg_zero);
    }
    __syncwarp();
    if (whole) {
      store_spans<M>(out, a.n_span[2], S, i0, lane);
      store_wide<M, kState, true>(a, rows, S, i0, lane);
    } else {
      store_tail<M, kState, true>(a, rows, S, i0, lane);
    }
    __syncwarp();
  }
}

template <int M>
__global__ void __launch_bounds__(kChainThreads) chain_backward_kernel(const __grid_constant__ ChainArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int R = 32 * M, R4 = R * 4;
  const int lane = threadIdx.x;
  const ChainRow* rows = a.row;
  const ChainSec* live = a.sec;
  const ChainAdj* adj = a.adj;
  const ChainSpan *in = spans(a, 0, smem), *out = spans(a, 1, smem), *gin = spans(a, 2, smem), *gout = spans(a, 3, smem);
  __syncthreads();
  uint8_t* S = smem + chain_tables(a);
  uint8_t* G = S + (a.n_rows + a.n_extra) * R4;
  const int at = lane * M * 4;
  lane_store<M>(G + a.n_rows * R4 + at, 0ull);   // the row of zeros
  for (int64_t c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
    const int64_t i0 = c * R;
    const bool whole = i0 + R <= a.n;
    if (whole) {
      load_spans<M>(in, a.n_span[0], S, i0, lane);
      cp_async_commit();
      load_spans<M>(gin, a.n_span[2], G, i0, lane);   // arrives while the sections run again
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
    if (whole) {
      store_spans<M>(out, a.n_span[1], S, i0, lane);
      store_wide<M, kState, true>(a, rows, S, i0, lane);
    } else {
      store_tail<M, kState, true>(a, rows, S, i0, lane);
    }
    __syncwarp();
    ChainSec next = live[0];
#pragma unroll 1
    for (int s = 0; s < a.n_live; ++s) {
      const ChainSec c = next;
      next = live[s + 1];
      chain_section<M>(c, S + at, a.tanh_p, a.tanh_qn, a.neg_zero);
    }
    ChainAdj nadj = adj[0];
    cp_async_wait<0>();
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < a.n_sec; ++s) {
      const ChainAdj c = nadj;
      nadj = adj[s + 1];
      chain_adjoint<M>(c, S + at, G + at, a.neg_zero);
    }
    for (uint64_t left = a.zero_rows; left; left &= left - 1) lane_store<M>(G + (__ffsll((long long)left) - 1) * R4 + at, 0ull);
    __syncwarp();
    if (whole) {
      store_spans<M>(gout, a.n_span[3], G, i0, lane);
      store_wide<M, kGradOut, false>(a, rows, G, i0, lane);
    } else {
      store_tail<M, kGradOut, false>(a, rows, G, i0, lane);
    }
    // gradients of groups the run does not touch, when they go to buffers of their own
    for (int k = 0; k < a.n_copy; ++k) {
      const ChainCopy& cp = a.copy[k];
      const int64_t b0 = i0 * cp.stride;
      const int bytes = (int)((whole ? (int64_t)R : a.n - i0) * cp.stride), whole16 = bytes / 16 * 16;
      // (R * 4 bytes is a multiple of 16: every chunk starts on one)
#pragma unroll 4
      for (int p = lane * 16; p < whole16; p += 512)
        *reinterpret_cast<uint4*>(cp.dst + b0 + p) = *reinterpret_cast<const uint4*>(cp.src + b0 + p);
      for (int p = whole16 + lane * 4; p < bytes; p += 128)
        *reinterpret_cast<float*>(cp.dst + b0 + p) = *reinterpret_cast<const float*>(cp.src + b0 + p);
    }
    __syncwarp();
  }
}

size_t chain_smem_bytes(const ChainArgs& a, int M, bool backward) {
  return chain_tables(a) + (size_t)(backward ? 2 * a.n_rows + a.n_extra + 1 : a.n_rows) * 128 * M;
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
