// sections.cu -- layout-templated section kernels (paper Section 2: a section is one
// data-parallel loop; its layout decides which bytes it drags through memory) and the reverse
// (adjoint) kernel of the fp32 chain sections.
//
// The forward kernel works per warp on chunks of R = 32*M records, like remap.cu: it copies the
// chunk's slice of every group that holds a field the section reads into its own shared buffer
// (16-byte cp.async through the piece table of staging.cuh, one chunk ahead), computes the M records of each lane from the staged
// bytes, and stores the written fields straight to global memory (a partial-record store
// touches only the sectors of the written field).  The op is a template parameter; the layout is
// the FieldRef table (where each field sits in the stage and in global memory).  Every floating
// operation is an explicitly rounded-to-nearest intrinsic, so no contraction can change a bit.
#include <cuda_runtime.h>

#include <type_traits>

#include "internal.h"
#include "ptx.cuh"
#include "section_ops.cuh"
#include "staging.cuh"

namespace adha {

template <int OP, int M, bool VEC>
__global__ void __launch_bounds__(kThreads) section_kernel(const __grid_constant__ SectionArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int R = 32 * M;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_pieces = stage_pieces(a, R);
  StagePiece* tab = reinterpret_cast<StagePiece*>(smem);
  fill_pieces(a, R, n_pieces, tab, tid);
  const int nb = a.buffers;   // 2: the next chunk is staged while one is computed; 1: one buffer
  uint8_t* bufs = smem + n_pieces * sizeof(StagePiece);
  uint8_t* buf0 = bufs + (size_t)warp * nb * a.in_bytes;
  uint8_t* buf1 = buf0 + (nb - 1) * a.in_bytes;
  uint8_t* extra = bufs + (size_t)kWarps * nb * a.in_bytes;
  // REDUCE: counts and (walk) sums in registers; after the chunk buffers the warp's two sum
  // tables (not walk) or its record list (walk), see reduce_smem_bytes
  long long* acc = nullptr;
  int* idx = nullptr;
  unsigned long long cnt = 0;   // REDUCE: lane k counts cluster k
  long long sum[kMaxClusters];
  ReduceLane rq{};
  if constexpr (OP == ADHA_OP_REDUCE) {
    rq = reduce_lane(a.s, a.f, lane, a.reduce_walk != 0);
    if (!rq.walk) {
      acc = reinterpret_cast<long long*>(extra) + (size_t)warp * 2 * (kMaxClusters + 1) * 32;
      for (int k = lane; k < 2 * (kMaxClusters + 1) * 32; k += 32) acc[k] = 0;
      extra += kReduceTableBytes;
    } else {
      zero_records(a, R, buf0, lane);
      if (nb == 2) zero_records(a, R, buf1, lane);
    }
    idx = reinterpret_cast<int*>(extra) + warp * kReduceList;
#pragma unroll
    for (int k = 0; k < kMaxClusters; ++k) sum[k] = 0;
  }
  // ASSIGN: the centroid table after the chunk buffers
  float* cT = nullptr;
  if constexpr (OP == ADHA_OP_ASSIGN) {
    cT = reinterpret_cast<float*>(extra);
    fill_centroids(a.s, a.f, cT, tid, kThreads);
  }
  constexpr bool kHoisted = OP != ADHA_OP_MIX && OP != ADHA_OP_ASSIGN && OP != ADHA_OP_REDUCE && !VEC;
  constexpr int kOps = kHoisted ? kOperands<OP> : 1;
  OpRef ref[kOps];
  LocalOp lo;
  if constexpr (kHoisted) {
#pragma unroll
    for (int k = 0; k < kOps; ++k) {
      const FieldRef& F = a.f[a.s.arg[k]];
      ref[k] = OpRef{F.s0 + lane * F.ss, 32 * F.ss, F.g, F.gs, F.wsm};
      lo.arg[k] = k;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      lo.par[k] = a.s.par[k];
      lo.gidx[k] = a.s.gidx[k];
    }
    lo.gvec = a.s.gvec;
  }
  __syncthreads();

  const int64_t W = (int64_t)gridDim.x * kWarps;
  int64_t c = (int64_t)blockIdx.x * kWarps + warp;
  if (c < a.n_chunks) stage_chunk(tab, n_pieces, c, buf0, lane);
  cp_async_commit();
  for (int i = 0; c < a.n_chunks; c += W, ++i) {
    uint8_t* cur = (i & 1) ? buf1 : buf0;
    if (nb == 2) {
      if (c + W < a.n_chunks) stage_chunk(tab, n_pieces, c + W, (i & 1) ? buf0 : buf1, lane);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const int64_t i0 = c * R;
    if constexpr (OP == ADHA_OP_REDUCE) {
      reduce_chunk_any<M>(rq, cur, lane, acc, acc + (kMaxClusters + 1) * 32, idx, sum, &cnt);
    } else if constexpr (OP == ADHA_OP_ASSIGN) {
      assign_chunk<M>(a.s, a.f, cur, i0, lane, cT);
    } else if constexpr (OP == ADHA_OP_MIX && VEC) {
      mix_chunk_vec<M>(a.s, a.f, cur, i0, lane);
    } else if constexpr (VEC) {
      chain_chunk_vec<OP, M>(a.s, a.f, a.tanh_p, a.tanh_q, a.save, cur, i0, lane);
    } else if constexpr (OP == ADHA_OP_MIX) {
      mix_chunk<M>(a.s, a.f, cur, i0, lane);
    } else {
      const int32_t* ps = a.perm_slot >= 0 ? reinterpret_cast<const int32_t*>(cur + a.load[a.perm_slot].start) : nullptr;
      if ((OP == ADHA_OP_DRIFT || OP == ADHA_OP_GATHER || OP == ADHA_OP_KICK) && a.alias) {
#pragma unroll 1
        for (int m = 0; m < M; ++m) {
          const int r = lane + 32 * m;
          run_record<OP>(a.s, a.f, a.tanh_p, a.tanh_q, a.save, StagedRec{a.f, cur, r, i0 + r}, i0 + r, ps ? ps[r] : 0);
        }
      } else {
        unsigned long long out[M][kOps];
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const int r = lane + 32 * m;
          run_record<OP>(lo, ref, a.tanh_p, a.tanh_q, a.save, HoistedRec{ref, cur, m, out[m]}, i0 + r, ps ? ps[r] : 0);
        }
#pragma unroll
        for (int k = 0; k < kOps; ++k) {
          if (!(kWrites<OP> >> k & 1)) continue;
          using V = std::conditional_t<kWriteSize<OP> == 8, unsigned long long, uint32_t>;
          if (ref[k].wsm) {
#pragma unroll
            for (int m = 0; m < M; ++m) *reinterpret_cast<V*>(cur + ref[k].s + m * ref[k].step) = (V)out[m][k];
          } else {
            uint8_t* q = ref[k].g + (i0 + lane) * ref[k].gs;
#pragma unroll
            for (int m = 0; m < M; ++m) *reinterpret_cast<V*>(q + (int64_t)(32 * m) * ref[k].gs) = (V)out[m][k];
          }
        }
      }
    }
    if (a.n_writeback) {   // wide written groups go back whole, 16 bytes per lane per step
      __syncwarp();
      unstage_chunk(tab, n_pieces, c, cur, lane);
    }
    __syncwarp();
    if (nb == 1 && c + W < a.n_chunks) {   // one buffer: the next chunk once this one is done with it
      stage_chunk(tab, n_pieces, c + W, buf0, lane);
      cp_async_commit();
    }
  }
  cp_async_wait<0>();

  // ragged tail: the warp whose next chunk would be n_chunks
  const int64_t t0 = a.n_chunks * R;
  if constexpr (OP == ADHA_OP_REDUCE) {
    if (c == a.n_chunks && t0 < a.n) reduce_tail(rq, a.s, a.f, t0, a.n, lane, acc, sum, &cnt);
    // the CTA adds its sums and counts into the result (zeroed before the launch)
    reduce_flush(rq, a.s, warp, lane, reinterpret_cast<long long*>(idx - warp * kReduceList), acc, sum, &cnt);
  } else {
    if (c == a.n_chunks && t0 < a.n) {
      for (int64_t i = t0 + lane; i < a.n; i += 32)
        run_record<OP>(a.s, a.f, a.tanh_p, a.tanh_q, a.save, GlobalRec{a.f, i}, i, a.perm_slot >= 0 ? a.perm[i] : 0);
    }
  }
}

// Reverse of one fp32 chain section (AXPB, MUL, TANH).  Every value a record needs is loaded
// first (4 records per thread, independent loads), the oracle's sequential update
//   restore z; gz = g[z]; g[z] = 0; then g[x] (and g[y]) += ...
// is carried out in registers with the aliasing of x, y, z resolved explicitly (they are
// launch-uniform), and the results are stored last.
template <int OP>
__device__ __forceinline__ void backward_record(const BackwardArgs& a, int64_t i, float sv, float xs, float ys,
                                                float gz, float gx, float gy) {
  const bool xz = a.x == a.z, yz = a.y == a.z, xy = a.x == a.y;
  const float xo = xz ? sv : xs;                   // x before the section
  const float yo = yz ? sv : ys;
  float gxn = xz ? 0.0f : gx;                      // after g[z] = 0
  if (OP == ADHA_OP_AXPB) {
    gxn = __fadd_rn(gxn, __fmul_rn(a.a, gz));
  } else if (OP == ADHA_OP_TANH) {
    const float t = tanh_cf(xo, a.tanh_p, a.tanh_q);
    gxn = __fadd_rn(gxn, __fmul_rn(gz, __fsub_rn(1.0f, __fmul_rn(t, t))));
  } else {
    gxn = __fadd_rn(gxn, __fmul_rn(gz, yo));
    float gyn = xy ? gxn : (yz ? 0.0f : gy);
    gyn = __fadd_rn(gyn, __fmul_rn(gz, xo));
    *reinterpret_cast<float*>(a.g[1] + i * a.gs[1]) = gyn;
    if (!xy) *reinterpret_cast<float*>(a.g[0] + i * a.gs[0]) = gxn;
    if (!xz && !yz) *reinterpret_cast<float*>(a.g[2] + i * a.gs[2]) = 0.0f;
    *reinterpret_cast<float*>(a.s[2] + i * a.ss[2]) = sv;
    return;
  }
  *reinterpret_cast<float*>(a.g[0] + i * a.gs[0]) = gxn;
  if (!xz) *reinterpret_cast<float*>(a.g[2] + i * a.gs[2]) = 0.0f;
  *reinterpret_cast<float*>(a.s[2] + i * a.ss[2]) = sv;
}

template <int OP>
__global__ void __launch_bounds__(kThreads) backward_kernel(const __grid_constant__ BackwardArgs a) {
  constexpr int K = 4;
  const int64_t T = (int64_t)gridDim.x * blockDim.x;
  const bool need_y = OP == ADHA_OP_MUL;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; base < a.n; base += K * T) {
    float sv[K], xs[K], ys[K], gz[K], gx[K], gy[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int64_t i = base + k * T;
      if (i < a.n) {
        sv[k] = a.save[i];
        xs[k] = *reinterpret_cast<const float*>(a.s[0] + i * a.ss[0]);
        ys[k] = need_y ? *reinterpret_cast<const float*>(a.s[1] + i * a.ss[1]) : 0.0f;
        gz[k] = *reinterpret_cast<const float*>(a.g[2] + i * a.gs[2]);
        gx[k] = *reinterpret_cast<const float*>(a.g[0] + i * a.gs[0]);
        gy[k] = need_y ? *reinterpret_cast<const float*>(a.g[1] + i * a.gs[1]) : 0.0f;
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int64_t i = base + k * T;
      if (i < a.n) backward_record<OP>(a, i, sv[k], xs[k], ys[k], gz[k], gx[k], gy[k]);
    }
  }
}

size_t section_smem_bytes(const SectionArgs& a) {
  const size_t acc = a.s.op == ADHA_OP_REDUCE ? reduce_smem_bytes(a.reduce_walk != 0) : 0;
  const size_t cent = a.s.op == ADHA_OP_ASSIGN ? (size_t)kCentroidBytes : 0;
  return (size_t)stage_pieces(a, a.R) * sizeof(StagePiece) + (size_t)kWarps * a.buffers * a.in_bytes + acc + cent;
}

template <int OP, int M, bool VEC>
static int launch_om(const SectionArgs& a, int grid, size_t smem, void* stream) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(section_kernel<OP, M, VEC>), smem, "cudaFuncSetAttribute(section)")) return rc;
  cudaError_t e = cudaSuccess;
  if (OP == ADHA_OP_REDUCE && !a.accumulate) {   // the sums are added into a zeroed result
    const int K = a.s.arg[1], d = a.s.rd_off[ADHA_F32 + 1] - a.s.rd_off[ADHA_F32];
    e = cudaMemsetAsync(const_cast<void*>(a.s.aux), 0, (size_t)K * (d + 1) * 8, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(reduce result)");
  }
  section_kernel<OP, M, VEC><<<grid, kThreads, smem, (cudaStream_t)stream>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "section kernel launch");
  return 0;
}

template <int OP>
static int launch_op(const SectionArgs& a, int grid, size_t smem, void* stream) {
  if constexpr (kVectorOp<OP>) {
    if (a.vec && a.R == 64) return launch_om<OP, 2, true>(a, grid, smem, stream);
    if (a.vec && a.R == 128) return launch_om<OP, 4, true>(a, grid, smem, stream);
  }
  switch (a.R) {
    case 32: return launch_om<OP, 1, false>(a, grid, smem, stream);
    case 64: return launch_om<OP, 2, false>(a, grid, smem, stream);
    default: return launch_om<OP, 4, false>(a, grid, smem, stream);
  }
}

template <int OP, int M, bool VEC>
static int occ_om(size_t smem, int* blocks) {
  if (int rc = allow_smem(reinterpret_cast<const void*>(section_kernel<OP, M, VEC>), smem, "cudaFuncSetAttribute(section)")) return rc;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, section_kernel<OP, M, VEC>, kThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor(section)");
  return 0;
}

// The kernel that launch_op picks for R records per chunk.
template <int OP>
static int occ_op(int R, bool vec, size_t smem, int* blocks) {
  if constexpr (kVectorOp<OP>) {
    if (vec && R == 64) return occ_om<OP, 2, true>(smem, blocks);
    if (vec && R == 128) return occ_om<OP, 4, true>(smem, blocks);
  }
  switch (R) {
    case 32: return occ_om<OP, 1, false>(smem, blocks);
    case 64: return occ_om<OP, 2, false>(smem, blocks);
    default: return occ_om<OP, 4, false>(smem, blocks);
  }
}

#define ADHA_FOR_EACH_OP(X)                                                                              \
  X(ADHA_OP_MADD3) X(ADHA_OP_XORSHIFT) X(ADHA_OP_ADD) X(ADHA_OP_MIX) X(ADHA_OP_DRIFT) X(ADHA_OP_BIN)     \
  X(ADHA_OP_KE) X(ADHA_OP_FLAGS) X(ADHA_OP_GATHER) X(ADHA_OP_KICK) X(ADHA_OP_AXPB) X(ADHA_OP_MUL)        \
  X(ADHA_OP_TANH) X(ADHA_OP_ASSIGN) X(ADHA_OP_REDUCE)

int launch_section(const SectionArgs& a, int grid, size_t smem, void* stream) {
  switch (a.s.op) {
#define X(op) case op: return launch_op<op>(a, grid, smem, stream);
    ADHA_FOR_EACH_OP(X)
#undef X
    default: return fail(ADHA_EINVAL, "unknown section op %d", a.s.op);
  }
}

int section_occupancy(int op, int R, bool vec, size_t smem, int* blocks) {
  switch (op) {
#define X(o) case o: return occ_op<o>(R, vec, smem, blocks);
    ADHA_FOR_EACH_OP(X)
#undef X
    default: return fail(ADHA_EINVAL, "unknown section op %d", op);
  }
}

int launch_backward(const BackwardArgs& a, void* stream) {
  int sms = 0;
  if (int rc = sm_count(&sms)) return rc;
  int64_t blocks = (a.n + 4 * kThreads - 1) / (4 * kThreads);
  if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
  if (blocks < 1) blocks = 1;
  if (a.op == ADHA_OP_AXPB) backward_kernel<ADHA_OP_AXPB><<<(int)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
  else if (a.op == ADHA_OP_MUL) backward_kernel<ADHA_OP_MUL><<<(int)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
  else backward_kernel<ADHA_OP_TANH><<<(int)blocks, kThreads, 0, (cudaStream_t)stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "backward kernel launch");
  return 0;
}

}  // namespace adha
