// section_ops.cuh -- per-record and per-chunk arithmetic of the section kinds, shared by the
// single-section kernel (sections.cu) and the fused kernel (fused.cu).  A record's fields are
// reached through a FieldRef table: in the warp's chunk buffer when staged, else in global memory.
// Every floating operation is an explicitly rounded-to-nearest intrinsic, so no contraction can
// change a bit.
#pragma once

#ifndef __CUDACC_RTC__
#include <cstdint>
#include <cstring>
#endif

#include "device_types.h"
#include "ptx.cuh"

// Loops over a section's listed fields: unrolled in windows specialised at run time (constant
// bounds), left to the compiler's own choice in the library's kernels (bounds known at run time).
#ifdef __CUDACC_RTC__
#define ADHA_FIELD_LOOP _Pragma("unroll")
#else
#define ADHA_FIELD_LOOP
#endif

namespace adha {

// Exact IEEE operations done with integer instructions, so that the fp64 pipe (a small fraction
// of the fp32 rate on this GPU) only does the additions.  Every case is a select between integer
// results: a branch to the fp64 instruction for the rare inputs would be turned into a select by
// the compiler too, and then the fp64 instruction would run for every value.

// The common cases of the two below, taken for a whole warp when every lane's values qualify
// (one vote per field): a normal double whose half is normal, and a normal float.
__device__ __forceinline__ bool half_is_plain(double x) {
  return ((unsigned)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FFu) - 2u <= 2044u;
}
__device__ __forceinline__ double half_plain(double x) {
  return __longlong_as_double(__double_as_longlong(x) - (1ll << 52));
}
// (a zero is plain too: a section that reads no fp32 field has t = 0 for one record in 256)
__device__ __forceinline__ bool widen_is_plain(float t) {
  const unsigned u = __float_as_uint(t);
  return ((u >> 23) & 0xFFu) - 1u <= 253u || (u & 0x7FFFFFFFu) == 0u;
}
__device__ __forceinline__ double widen_plain(float t) {
  const unsigned u = __float_as_uint(t);
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned long long normal = sign | ((unsigned long long)(((u >> 23) & 0xFFu) + 896u) << 52) |
                                    ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)((u & 0x7FFFFFFFu) ? normal : sign));
}

// x * 0.5 rounded to nearest.  A normal x whose half is normal (biased exponent 2..2046): the
// exponent lowered by one.  Exponent 0 or 1 (zeros, subnormals, the smallest normals): the half is
// subnormal, its significand the full significand q of x (with the implicit bit for exponent 1)
// halved with ties to even (q odd is exactly a tie); a carry into the exponent field gives the
// smallest normal, as it should.  Infinities and NaNs are returned unchanged.
__device__ __forceinline__ double half_rn_int(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned e = (unsigned)(b >> 52) & 0x7FFu;
  const unsigned long long q = (b & 0xFFFFFFFFFFFFFull) | (e ? (1ull << 52) : 0ull);
  const unsigned long long h = (q >> 1) + (q & (q >> 1) & 1ull);
  const unsigned long long small = (b & (1ull << 63)) | h;
  const unsigned long long big = e == 0x7FFu ? b : b - (1ull << 52);
  return __longlong_as_double((long long)(e <= 1u ? small : big));
}

// float -> double, exact.  Normal: sign and significand kept (the significand shifted into the
// wider field), exponent rebiased from 127 to 1023.  Zero: the sign alone.  Subnormal m * 2^-149
// (m < 2^23): normal in double, its leading bit p = 31 - clz(m) becomes the implicit one, exponent
// p - 149.  Infinity: exponent all ones; NaN: its payload shifted likewise, made quiet.
__device__ __forceinline__ double widen_int(float t) {
  const unsigned u = __float_as_uint(t);
  const unsigned e = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned long long mm = (unsigned long long)m << 29;
  const unsigned long long normal = sign | ((unsigned long long)(e + 896u) << 52) | mm;
  const unsigned long long special = sign | (0x7FFull << 52) | mm | (m ? (1ull << 51) : 0ull);
  const int p = 31 - __clz((int)(m | 1u));
  const unsigned long long sub = sign | ((unsigned long long)(p + 874) << 52) |
                                 (((unsigned long long)m << (52 - p)) & 0xFFFFFFFFFFFFFull);
  const unsigned long long zero_or_sub = m ? sub : sign;
  return __longlong_as_double((long long)(e == 0u ? zero_or_sub : (e == 0xFFu ? special : normal)));
}

// The same two with the IEEE instruction for the rare inputs: the compiler turns the choice into
// a select, so the fp64 multiply (or the conversion) runs for every value next to the integer
// result.  That costs fp64-pipe time but few registers and instructions, the better trade in
// the memory-bound single-section kernels; fused runs, which compute long per chunk, take the
// integer forms above behind a warp vote.
__device__ __forceinline__ double half_rn(double x) {
  return half_is_plain(x) ? half_plain(x) : __dmul_rn(x, 0.5);
}
__device__ __forceinline__ double widen(float t) { return widen_is_plain(t) ? widen_plain(t) : (double)t; }

// The integer forms behind one warp vote per value, for code whose 32 lanes run it together.
__device__ __forceinline__ double half_vote(double x) {
  return __all_sync(0xFFFFFFFFu, half_is_plain(x)) ? half_plain(x) : half_rn_int(x);
}
__device__ __forceinline__ double widen_vote(float t) {
  return __all_sync(0xFFFFFFFFu, widen_is_plain(t)) ? widen_plain(t) : widen_int(t);
}

struct StagedRec {      // record r of a staged chunk (global record i)
  const FieldRef* f;
  uint8_t* stage;
  int r;
  int64_t i;
  template <class V>
  __device__ __forceinline__ V ld(int k) const {
    const FieldRef& F = f[k];
    if (F.s0 >= 0) return *reinterpret_cast<const V*>(stage + F.s0 + r * F.ss);
    return *reinterpret_cast<const V*>(F.g + i * F.gs);
  }
  template <class V>
  __device__ __forceinline__ void st(int k, V v) const {
    const FieldRef& F = f[k];
    if (F.wsm) *reinterpret_cast<V*>(stage + F.s0 + r * F.ss) = v;
    else *reinterpret_cast<V*>(F.g + i * F.gs) = v;
  }
};

struct GlobalRec {      // record i in global memory (ragged tail)
  const FieldRef* f;
  int64_t i;
  template <class V>
  __device__ __forceinline__ V ld(int k) const {
    return *reinterpret_cast<const V*>(f[k].g + i * f[k].gs);
  }
  template <class V>
  __device__ __forceinline__ void st(int k, V v) const {
    *reinterpret_cast<V*>(f[k].g + i * f[k].gs) = v;
  }
};

// A section's operands as the single-section kernel holds them, in registers for the whole launch:
// operand k stands for itself (arg[k] = k) in run_record, so every address below is a constant
// index into these, and the per-record lookups of field ids, offsets and strides in the parameter
// space disappear (they were most of a light section's 100-140 instructions per 32 records).  With
// the piece table of staging.cuh, 2^23 particles in [pos+charge] [vel] groups: drift 87 -> 69 us,
// bin 35 -> 33, KE 43 -> 36, gather 168 -> 126 (also 32 records per chunk), kick 70 -> 56.
struct OpRef {
  int s;         // chunk-buffer offset of the operand in the lane's first record, if staged
  int step;      // chunk-buffer bytes per 32 records
  uint8_t* g;    // global address of the operand in record 0
  int gs;        // global stride
  int wsm;       // writes go into the chunk buffer
};
struct LocalOp {
  int arg[8];
  float par[4];
  int8_t gvec;
  int8_t gidx[4];
};

// Operands of an op, which of them it writes (bit k), and the size of what it writes.
template <int OP>
constexpr int kOperands = OP == ADHA_OP_DRIFT ? 6 : OP == ADHA_OP_GATHER ? 7 : OP == ADHA_OP_KE ? 5
                          : OP == ADHA_OP_BIN || OP == ADHA_OP_KICK ? 4
                          : OP == ADHA_OP_MADD3 || OP == ADHA_OP_ADD || OP == ADHA_OP_MUL ? 3 : 2;
template <int OP>
constexpr int kWrites = OP == ADHA_OP_DRIFT || OP == ADHA_OP_GATHER || OP == ADHA_OP_KICK ? 7 : OP == ADHA_OP_KE ? 16
                        : OP == ADHA_OP_BIN ? 8 : OP == ADHA_OP_MADD3 || OP == ADHA_OP_ADD || OP == ADHA_OP_MUL ? 4
                        : OP == ADHA_OP_FLAGS ? 1 : 2;
template <int OP>
constexpr int kWriteSize = OP == ADHA_OP_KE ? 8 : 4;

// Record m of the lane's M records: reads from the chunk buffer (every field an op reads at its own
// record is staged), writes kept in registers until all M records are computed, so that no store
// stands between one record's loads and the next one's.
struct HoistedRec {
  const OpRef* ref;
  const uint8_t* buf;
  int m;
  unsigned long long* out;   // by operand
  template <class V>
  __device__ __forceinline__ V ld(int k) const {
    return *reinterpret_cast<const V*>(buf + ref[k].s + m * ref[k].step);
  }
  template <class V>
  __device__ __forceinline__ void st(int k, V v) const {
    unsigned long long b = 0;
    memcpy(&b, &v, sizeof v);
    out[k] = b;
  }
};

template <class V, class FR>
__device__ __forceinline__ V gld(const FR* f, int k, int64_t i) {
  return __ldg(reinterpret_cast<const V*>(f[k].g + i * f[k].gs));
}

// Lambert's continued fraction for tanh cut after the partial denominator 25, as x*Q(a)/P(a) with
// a = x*x: Horner's rule over the 7 coefficients of each polynomial, then one IEEE division.
__device__ __forceinline__ float tanh_cf(float x, const float* P, const float* Q) {
  if (fabsf(x) >= 9.0f) return copysignf(1.0f, x);
  const float a = __fmul_rn(x, x);
  float q = Q[6], p = P[6];
#pragma unroll
  for (int j = 5; j >= 0; --j) {
    q = __fadd_rn(__fmul_rn(q, a), Q[j]);
    p = __fadd_rn(__fmul_rn(p, a), P[j]);
  }
  return __fdiv_rn(__fmul_rn(x, q), p);
}

// tanh_cf of two values in the packed fp32 instructions, bit for bit: the polynomials as there (P, QN: the
// coefficients of P and of -Q as pairs, so that nn = -x*Q(a) exactly, every rounding being symmetric),
// and the quotient by Markstein's method (IBM J. Res. Dev. 34, 1990) instead of two IEEE divisions: a
// reciprocal approximation refined once, y; q = n*y; the exact remainder r = n - d*q; q + r*y is the
// correctly rounded quotient.  The signs are arranged so that a zero keeps its sign.  |x| >= 9 is
// evaluated at +-10, where the quotient is exactly +-1.  About 40 instructions a pair, 75 with the
// divisions; equal to tanh_cf for every float (tested).
__device__ __forceinline__ unsigned long long tanh_pair(unsigned long long x, const unsigned long long* P,
                                                        const unsigned long long* QN, unsigned long long nz) {
  float lo, hi;
  f2_unpack(x, &lo, &hi);
  const unsigned long long xe = f2_pack(fabsf(lo) >= 9.0f ? copysignf(10.0f, lo) : lo, fabsf(hi) >= 9.0f ? copysignf(10.0f, hi) : hi);
  const unsigned long long a = f2_mul_alone(xe, xe, nz);
  unsigned long long q = QN[6], d = P[6];
#pragma unroll
  for (int j = 5; j >= 0; --j) {
    q = f2_add_rn(f2_mul_alone(q, a, nz), QN[j]);
    d = f2_add_rn(f2_mul_alone(d, a, nz), P[j]);
  }
  const unsigned long long nn = f2_mul_alone(xe, q, nz);
  float dl, dh;
  f2_unpack(d, &dl, &dh);
  const unsigned long long m = f2_pack(rcp_approx(-dl), rcp_approx(-dh));           // about -1/d
  const unsigned long long ym = f2_fma_rn(f2_fma_rn(d, m, f2_pack(1.0f, 1.0f)), m, m);   // -1/d, rounded
  const unsigned long long t = f2_mul_alone(nn, ym, nz);
  return f2_fma_rn(f2_fma_rn(d, t, nn), ym, t);
}

// MIX over the M records r = lane + 32m of a staged chunk, field-major: every field's shared
// and global addresses are computed once for the M records.
template <int M>
__device__ __forceinline__ void mix_chunk(const SecOp& so, const FieldRef* fr, uint8_t* stage, int64_t i0, int lane) {
  float s[M];
  uint32_t h[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    s[m] = 0.0f;
    h[m] = 0u;
  }
  // V value of field F for the lane's record m: from the chunk buffer if staged, else global
#define ADHA_MIX_READ(V, LIST, BODY)                                                        \
  for (int j = so.rd_off[LIST]; j < so.rd_off[LIST + 1]; ++j) {                            \
    const FieldRef& F = fr[so.rd[j]];                                                       \
    if (F.s0 >= 0) {                                                                        \
      const uint8_t* p = stage + F.s0 + lane * F.ss;                                        \
      _Pragma("unroll") for (int m = 0; m < M; ++m) {                                       \
        const V v = *reinterpret_cast<const V*>(p + m * 32 * F.ss);                         \
        BODY;                                                                               \
      }                                                                                     \
    } else {                                                                                \
      const uint8_t* p = F.g + (i0 + lane) * F.gs;                                          \
      _Pragma("unroll") for (int m = 0; m < M; ++m) {                                       \
        const V v = *reinterpret_cast<const V*>(p + (int64_t)m * 32 * F.gs);                \
        BODY;                                                                               \
      }                                                                                     \
    }                                                                                       \
  }
  ADHA_MIX_READ(float, ADHA_F32, s[m] = __fadd_rn(s[m], v))
  ADHA_MIX_READ(unsigned long long, ADHA_F64, h[m] ^= (uint32_t)v ^ (uint32_t)(v >> 32))
  ADHA_MIX_READ(uint32_t, ADHA_I32, h[m] ^= v)
  ADHA_MIX_READ(uint16_t, ADHA_BF16, h[m] ^= (uint32_t)v)
#undef ADHA_MIX_READ
  float t[M];
  uint32_t k[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    t[m] = __fadd_rn(s[m], __fmul_rn(__uint2float_rn(h[m] & 255u), 0.00390625f));
    k[m] = (h[m] ^ __float_as_uint(t[m])) >> 3;
  }
  // written fields: old value from the chunk buffer if staged, else global; new value to global
#define ADHA_MIX_WRITE(V, LIST, EXPR)                                                       \
  for (int j = so.wr_off[LIST]; j < so.wr_off[LIST + 1]; ++j) {                            \
    const FieldRef& F = fr[so.wr[j]];                                                       \
    uint8_t* p = stage + F.s0 + lane * F.ss;                                                \
    if (F.wsm) {                                                                            \
      _Pragma("unroll") for (int m = 0; m < M; ++m) {                                       \
        V* x = reinterpret_cast<V*>(p + m * 32 * F.ss);                                     \
        const V old = *x;                                                                   \
        *x = EXPR;                                                                          \
      }                                                                                     \
    } else {                                                                                \
      uint8_t* q = F.g + (i0 + lane) * F.gs;                                                \
      _Pragma("unroll") for (int m = 0; m < M; ++m) {                                       \
        const V old = *reinterpret_cast<const V*>(p + m * 32 * F.ss);                       \
        *reinterpret_cast<V*>(q + (int64_t)m * 32 * F.gs) = EXPR;                           \
      }                                                                                     \
    }                                                                                       \
  }
  ADHA_MIX_WRITE(float, ADHA_F32, __fadd_rn(__fmul_rn(old, 0.5f), t[m]))
  if (so.wr_off[ADHA_F64 + 1] > so.wr_off[ADHA_F64]) {
    double td[M];
#pragma unroll
    for (int m = 0; m < M; ++m) td[m] = widen(t[m]);
    ADHA_MIX_WRITE(double, ADHA_F64, __dadd_rn(half_rn(old), td[m]))
  }
  ADHA_MIX_WRITE(uint32_t, ADHA_I32, old ^ k[m])
  ADHA_MIX_WRITE(uint16_t, ADHA_BF16, (uint16_t)(old ^ (uint16_t)(k[m] & 0xFFFFu)))
#undef ADHA_MIX_WRITE
}

// M consecutive values of one field for records lane*M .. lane*M+M-1 of a one-field slice
// (contiguous, M*sizeof(V)-byte aligned): moved with 8- or 16-byte accesses.
template <class V, int M>
__device__ __forceinline__ void ld_vec(const uint8_t* p, V (&v)[M]) {
  constexpr int B = M * (int)sizeof(V);
  if constexpr (B % 16 == 0) {
#pragma unroll
    for (int k = 0; k < B / 16; ++k) {
      const uint4 x = reinterpret_cast<const uint4*>(p)[k];
      memcpy(reinterpret_cast<uint8_t*>(v) + 16 * k, &x, 16);
    }
  } else if constexpr (B == 8) {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    memcpy(v, &x, 8);
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = reinterpret_cast<const V*>(p)[m];
  }
}

template <class V, int M>
__device__ __forceinline__ void st_vec(uint8_t* p, const V (&v)[M]) {
  constexpr int B = M * (int)sizeof(V);
  if constexpr (B % 16 == 0) {
#pragma unroll
    for (int k = 0; k < B / 16; ++k) {
      uint4 x;
      memcpy(&x, reinterpret_cast<const uint8_t*>(v) + 16 * k, 16);
      reinterpret_cast<uint4*>(p)[k] = x;
    }
  } else if constexpr (B == 8) {
    uint2 x;
    memcpy(&x, v, 8);
    *reinterpret_cast<uint2*>(p) = x;
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) reinterpret_cast<V*>(p)[m] = v[m];
  }
}

// MIX when every accessed group holds one field (SoA-like): lane takes records lane*M + m, so
// each field is one vector load from the chunk buffer and one vector store, to global memory or
// (TO_STAGE, inside a fused run) back into the chunk buffer.  The field loops are unrolled so that
// several fields' loads are in flight before their (ordered) sums consume them.
template <int M, bool TO_STAGE = false>
__device__ __forceinline__ void mix_chunk_vec(const SecOp& so, const FieldRef* fr, uint8_t* stage, int64_t i0,
                                              int lane) {
  float s[M];
  uint32_t h[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    s[m] = 0.0f;
    h[m] = 0u;
  }
  // the lane's M records of a field of size b start at stage + s0 + lane*M*b
#define RD_S0(j) (TO_STAGE ? (int)so.rd_s0[j] : fr[so.rd[j]].s0)
#define WR_S0(j) (TO_STAGE ? (int)so.wr_s0[j] : fr[so.wr[j]].s0)
#define b2 (stage + lane * M * 2)
#define b4 (stage + lane * M * 4)
#define b8 (stage + lane * M * 8)
#pragma unroll 4
  for (int j = so.rd_off[ADHA_F32]; j < so.rd_off[ADHA_F32 + 1]; ++j) {
    float v[M];
    ld_vec<float, M>(b4 + RD_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) s[m] = __fadd_rn(s[m], v[m]);
  }
#pragma unroll 4
  for (int j = so.rd_off[ADHA_F64]; j < so.rd_off[ADHA_F64 + 1]; ++j) {
    unsigned long long v[M];
    ld_vec<unsigned long long, M>(b8 + RD_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) h[m] ^= (uint32_t)v[m] ^ (uint32_t)(v[m] >> 32);
  }
#pragma unroll 4
  for (int j = so.rd_off[ADHA_I32]; j < so.rd_off[ADHA_I32 + 1]; ++j) {
    uint32_t v[M];
    ld_vec<uint32_t, M>(b4 + RD_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) h[m] ^= v[m];
  }
#pragma unroll 4
  for (int j = so.rd_off[ADHA_BF16]; j < so.rd_off[ADHA_BF16 + 1]; ++j) {
    uint16_t v[M];
    ld_vec<uint16_t, M>(b2 + RD_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) h[m] ^= (uint32_t)v[m];
  }
  float t[M];
  uint32_t k[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    t[m] = __fadd_rn(s[m], __fmul_rn(__uint2float_rn(h[m] & 255u), 0.00390625f));
    k[m] = (h[m] ^ __float_as_uint(t[m])) >> 3;
  }
  const int64_t r0 = i0 + (int64_t)lane * M;
#pragma unroll 4
  for (int j = so.wr_off[ADHA_F32]; j < so.wr_off[ADHA_F32 + 1]; ++j) {
    float v[M];
    ld_vec<float, M>(b4 + WR_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = __fadd_rn(__fmul_rn(v[m], 0.5f), t[m]);
    st_vec<float, M>(TO_STAGE ? b4 + WR_S0(j) : fr[so.wr[j]].g + r0 * 4, v);
  }
  if (so.wr_off[ADHA_F64 + 1] > so.wr_off[ADHA_F64]) {
    double td[M];
    if constexpr (TO_STAGE) {   // fused run: no fp64 instruction but the additions (see half_rn_int)
      bool plain = true;
#pragma unroll
      for (int m = 0; m < M; ++m) plain = plain && widen_is_plain(t[m]);
      if (__all_sync(0xFFFFFFFFu, plain)) {
#pragma unroll
        for (int m = 0; m < M; ++m) td[m] = widen_plain(t[m]);
      } else {
#pragma unroll
        for (int m = 0; m < M; ++m) td[m] = widen_int(t[m]);
      }
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m) td[m] = widen(t[m]);
    }
#pragma unroll 4
    for (int j = so.wr_off[ADHA_F64]; j < so.wr_off[ADHA_F64 + 1]; ++j) {
      double v[M];
      ld_vec<double, M>(b8 + WR_S0(j), v);
      if constexpr (TO_STAGE) {
        bool ok = true;
#pragma unroll
        for (int m = 0; m < M; ++m) ok = ok && half_is_plain(v[m]);
        if (__all_sync(0xFFFFFFFFu, ok)) {
#pragma unroll
          for (int m = 0; m < M; ++m) v[m] = __dadd_rn(half_plain(v[m]), td[m]);
        } else {
#pragma unroll
          for (int m = 0; m < M; ++m) v[m] = __dadd_rn(half_rn_int(v[m]), td[m]);
        }
      } else {
#pragma unroll
        for (int m = 0; m < M; ++m) v[m] = __dadd_rn(half_rn(v[m]), td[m]);
      }
      st_vec<double, M>(TO_STAGE ? b8 + WR_S0(j) : fr[so.wr[j]].g + r0 * 8, v);
    }
  }
#pragma unroll 4
  for (int j = so.wr_off[ADHA_I32]; j < so.wr_off[ADHA_I32 + 1]; ++j) {
    uint32_t v[M];
    ld_vec<uint32_t, M>(b4 + WR_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] ^= k[m];
    st_vec<uint32_t, M>(TO_STAGE ? b4 + WR_S0(j) : fr[so.wr[j]].g + r0 * 4, v);
  }
#pragma unroll 4
  for (int j = so.wr_off[ADHA_BF16]; j < so.wr_off[ADHA_BF16 + 1]; ++j) {
    uint16_t v[M];
    ld_vec<uint16_t, M>(b2 + WR_S0(j), v);
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = (uint16_t)(v[m] ^ (uint16_t)(k[m] & 0xFFFFu));
    st_vec<uint16_t, M>(TO_STAGE ? b2 + WR_S0(j) : fr[so.wr[j]].g + r0 * 2, v);
  }
#undef b2
#undef b4
#undef b8
#undef RD_S0
#undef WR_S0
}

// AXPB, MUL, TANH under the vector mapping (x, y, z each a one-field group): lane takes records
// lane*M + m; x, y and the old z come from the chunk buffer (the values before the section, so
// any aliasing of x, y, z reads what the per-record rule reads), z and `save` get vector stores
// (z into the chunk buffer when TO_STAGE).
template <int OP, int M, bool TO_STAGE = false>
__device__ __forceinline__ void chain_chunk_vec(const SecOp& so, const FieldRef* fr, const float* tp, const float* tq,
                                                uint8_t* save, uint8_t* stage, int64_t i0, int lane) {
  const int* g = so.arg;
  const int z = OP == ADHA_OP_MUL ? g[2] : g[1];
  const int64_t r0 = i0 + (int64_t)lane * M;
  float x[M], v[M];
  ld_vec<float, M>(stage + fr[g[0]].s0 + lane * M * 4, x);
  if (save) {
    float old[M];
    ld_vec<float, M>(stage + fr[z].s0 + lane * M * 4, old);
    st_vec<float, M>(save + r0 * 4, old);
  }
  if (OP == ADHA_OP_MUL) {
    float y[M];
    ld_vec<float, M>(stage + fr[g[1]].s0 + lane * M * 4, y);
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = __fmul_rn(x[m], y[m]);
  } else if (OP == ADHA_OP_AXPB) {
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = __fadd_rn(__fmul_rn(so.par[0], x[m]), so.par[1]);
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = tanh_cf(x[m], tp, tq);
  }
  st_vec<float, M>(TO_STAGE ? stage + fr[z].s0 + lane * M * 4 : fr[z].g + r0 * 4, v);
}

template <int OP>
constexpr bool kVectorOp = OP == ADHA_OP_MIX || OP == ADHA_OP_AXPB || OP == ADHA_OP_MUL || OP == ADHA_OP_TANH;

// One record of one section: its fields through `rec` (staged chunk, global memory, or registers
// in a specialised window), fields read through the permutation from global memory (record pj),
// the old z to `save` when asked.  VOTE: the fp64 halving and widening take the integer forms
// behind a warp vote (every lane of the warp must run the call).  The field loops are unrolled
// where their bounds are compile-time constants (specialised windows), so that every field index
// folds to a constant there.
template <int OP, bool VOTE = false, class SO, class FR, class Rec>
__device__ __forceinline__ void run_record(const SO& so, const FR* fr, const float* tp, const float* tq,
                                           uint8_t* save, const Rec& rec, int64_t i, int32_t pj) {
  const int* g = so.arg;
  if constexpr (OP == ADHA_OP_MADD3) {
    const float m = __fmul_rn(rec.template ld<float>(g[0]), rec.template ld<float>(g[1]));
    rec.template st<float>(g[2], __fadd_rn(m, rec.template ld<float>(g[2])));
  } else if constexpr (OP == ADHA_OP_XORSHIFT) {
    const uint32_t u = rec.template ld<uint32_t>(g[0]);
    rec.template st<uint32_t>(g[1], u ^ (u >> 3));
  } else if constexpr (OP == ADHA_OP_ADD) {
    rec.template st<float>(g[2], __fadd_rn(rec.template ld<float>(g[0]), rec.template ld<float>(g[1])));
  } else if constexpr (OP == ADHA_OP_MIX) {
    float s = 0.0f;
    uint32_t h = 0u;
ADHA_FIELD_LOOP
    for (int j = so.rd_off[ADHA_F32]; j < so.rd_off[ADHA_F32 + 1]; ++j) s = __fadd_rn(s, rec.template ld<float>(so.rd[j]));
ADHA_FIELD_LOOP
    for (int j = so.rd_off[ADHA_F64]; j < so.rd_off[ADHA_F64 + 1]; ++j) {
      const unsigned long long b = rec.template ld<unsigned long long>(so.rd[j]);
      h ^= (uint32_t)b ^ (uint32_t)(b >> 32);
    }
ADHA_FIELD_LOOP
    for (int j = so.rd_off[ADHA_I32]; j < so.rd_off[ADHA_I32 + 1]; ++j) h ^= rec.template ld<uint32_t>(so.rd[j]);
ADHA_FIELD_LOOP
    for (int j = so.rd_off[ADHA_BF16]; j < so.rd_off[ADHA_BF16 + 1]; ++j) h ^= (uint32_t)rec.template ld<uint16_t>(so.rd[j]);
    const float t = __fadd_rn(s, __fmul_rn(__uint2float_rn(h & 255u), 0.00390625f));
    const uint32_t k = (h ^ __float_as_uint(t)) >> 3;
ADHA_FIELD_LOOP
    for (int j = so.wr_off[ADHA_F32]; j < so.wr_off[ADHA_F32 + 1]; ++j) {
      const int f = so.wr[j];
      rec.template st<float>(f, __fadd_rn(__fmul_rn(rec.template ld<float>(f), 0.5f), t));
    }
    if (so.wr_off[ADHA_F64 + 1] > so.wr_off[ADHA_F64]) {
      const double td = VOTE ? widen_vote(t) : widen(t);
ADHA_FIELD_LOOP
      for (int j = so.wr_off[ADHA_F64]; j < so.wr_off[ADHA_F64 + 1]; ++j) {
        const int f = so.wr[j];
        const double x = rec.template ld<double>(f);
        rec.template st<double>(f, __dadd_rn(VOTE ? half_vote(x) : half_rn(x), td));
      }
    }
ADHA_FIELD_LOOP
    for (int j = so.wr_off[ADHA_I32]; j < so.wr_off[ADHA_I32 + 1]; ++j) {
      const int f = so.wr[j];
      rec.template st<uint32_t>(f, rec.template ld<uint32_t>(f) ^ k);
    }
ADHA_FIELD_LOOP
    for (int j = so.wr_off[ADHA_BF16]; j < so.wr_off[ADHA_BF16 + 1]; ++j) {
      const int f = so.wr[j];
      rec.template st<uint16_t>(f, (uint16_t)(rec.template ld<uint16_t>(f) ^ (uint16_t)(k & 0xFFFFu)));
    }
  } else if constexpr (OP == ADHA_OP_DRIFT) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const float d = __fmul_rn(so.par[0], rec.template ld<float>(g[3 + ax]));
      float q = __fadd_rn(rec.template ld<float>(g[ax]), d);
      if (q >= 1.0f) q = __fsub_rn(q, 1.0f);
      else if (q < 0.0f) q = __fadd_rn(q, 1.0f);
      rec.template st<float>(g[ax], q);
    }
  } else if constexpr (OP == ADHA_OP_BIN) {
    const int G = (int)so.par[0];
    int c[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      int k = __float2int_rz(__fmul_rn(rec.template ld<float>(g[ax]), so.par[0]));
      k = k < 0 ? 0 : (k > G - 1 ? G - 1 : k);
      c[ax] = k;
    }
    rec.template st<int32_t>(g[3], c[0] + G * (c[1] + G * c[2]));
  } else if constexpr (OP == ADHA_OP_KE) {
    const float vx = rec.template ld<float>(g[0]), vy = rec.template ld<float>(g[1]),
                vz = rec.template ld<float>(g[2]);
    float s = __fadd_rn(__fmul_rn(vx, vx), __fmul_rn(vy, vy));
    s = __fadd_rn(s, __fmul_rn(vz, vz));
    const float e = __fmul_rn(__fmul_rn(0.5f, rec.template ld<float>(g[3])), s);
    rec.template st<double>(g[4], VOTE ? widen_vote(e) : widen(e));
  } else if constexpr (OP == ADHA_OP_FLAGS) {
    const uint32_t fl = rec.template ld<uint32_t>(g[0]);
    const uint32_t bit = rec.template ld<double>(g[1]) > (double)so.par[0] ? 1u : 0u;
    rec.template st<uint32_t>(g[0], ((fl << 1) | bit) & 255u);
  } else if constexpr (OP == ADHA_OP_GATHER) {
    const int64_t j = pj;
    float pv[4];   // px, py, pz, q of record j
    if (so.gvec) {   // all four in one 16-byte struct: one load
      const uint8_t* base = fr[g[3]].g - 4 * so.gidx[0];
      const uint4 w = __ldg(reinterpret_cast<const uint4*>(base + j * 16));
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int q = so.gidx[a];
        pv[a] = __uint_as_float(q == 0 ? w.x : q == 1 ? w.y : q == 2 ? w.z : w.w);
      }
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a) pv[a] = gld<float>(fr, g[3 + a], j);
    }
    const float c = __fmul_rn(so.par[0], pv[3]);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const float d = __fsub_rn(pv[ax], 0.5f);
      rec.template st<float>(g[ax], __fadd_rn(rec.template ld<float>(g[ax]), __fmul_rn(c, d)));
    }
  } else if constexpr (OP == ADHA_OP_KICK) {
    const float c = __fmul_rn(so.par[0], rec.template ld<float>(g[3]));
#pragma unroll
    for (int ax = 0; ax < 3; ++ax)
      rec.template st<float>(g[ax], __fadd_rn(rec.template ld<float>(g[ax]), __fmul_rn(c, so.par[1 + ax])));
  } else if constexpr (OP == ADHA_OP_ASSIGN) {
    // D_k summed over the features in ascending order, all K distances side by side, by the rule of
    // assign_chunk_k: the square and the sum in one fma (a record's membership must not depend on whether
    // it lies in a chunk or in the ragged tail)
    const int K = so.arg[1], j0 = so.rd_off[ADHA_F32], d = so.rd_off[ADHA_F32 + 1] - j0;
    const float* cent = static_cast<const float*>(so.aux);
    float D[kMaxClusters];
#pragma unroll
    for (int k = 0; k < kMaxClusters; ++k) D[k] = 0.0f;
    for (int j = 0; j < d; j += 4) {   // four features' loads in flight together
      float x[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) x[b] = rec.template ld<float>(so.rd[j0 + min(j + b, d - 1)]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (j + b >= d) break;
#pragma unroll
        for (int k = 0; k < kMaxClusters; ++k)
          if (k < K) {
            const float df = __fsub_rn(x[b], __ldg(cent + k * d + j + b));
            D[k] = __fmaf_rn(df, df, D[k]);
          }
      }
    }
    int best = 0;
    float bd = D[0];
#pragma unroll
    for (int k = 1; k < kMaxClusters; ++k)
      if (k < K && D[k] < bd) {
        bd = D[k];
        best = k;
      }
    rec.template st<int32_t>(g[0], best);
  } else {   // AXPB, MUL, TANH: z = op(x[, y]); the old z goes to `save` when asked
    const int z = OP == ADHA_OP_MUL ? g[2] : g[1];
    if (save) reinterpret_cast<float*>(save)[i] = rec.template ld<float>(z);
    const float x = rec.template ld<float>(g[0]);
    float v;
    if (OP == ADHA_OP_AXPB) v = __fadd_rn(__fmul_rn(so.par[0], x), so.par[1]);
    else if (OP == ADHA_OP_MUL) v = __fmul_rn(x, rec.template ld<float>(g[1]));
    else v = tanh_cf(x, tp, tq);
    rec.template st<float>(z, v);
  }
}

// Fixed-point value of a REDUCE feature: x * 2^23 (exact) rounded to the nearest integer, ties to
// even; 2^31 - 1 or -2^31 beyond the int32 range; 0 for NaN.  That is the float-to-int32
// conversion PTX defines (cvt.rni.s32.f32: the result clamped to the range, NaN to 0), so one
// conversion instruction does it.
__device__ __forceinline__ int fix32(float x) { return __float2int_rn(__fmul_rn(x, 8388608.0f)); }
__device__ __forceinline__ long long fixq(float x) { return (long long)fix32(x); }

// s + v, one wide multiply-add instead of a sign extension and a 64-bit addition.
__device__ __forceinline__ long long add_wide(long long s, int v) {
  asm("mad.wide.s32 %0, %1, 1, %0;" : "+l"(s) : "r"(v));
  return s;
}

// ASSIGN's tables in shared memory, one per CTA: the centroids, c[k][j] at cT[j*8 + k], and after
// them each feature's place in the chunk buffer (offset, stride from bit 16), so that the per-chunk
// loop reads both with broadcast shared loads.  kFour on every fourth feature: it and the next three
// are one aligned 16-byte piece of each record.
constexpr uint32_t kFour = 1u << 31;
constexpr int kCentroidBytes = kMaxFields * kMaxClusters * 4 + kMaxFields * 4;

__device__ __forceinline__ void fill_centroids(const SecOp& so, const FieldRef* fr, float* cT, int tid, int nthreads) {
  const int j0 = so.rd_off[ADHA_F32], K = so.arg[1], d = so.rd_off[ADHA_F32 + 1] - j0;
  const float* cent = static_cast<const float*>(so.aux);
  for (int t = tid; t < d * kMaxClusters; t += nthreads) {
    const int j = t / kMaxClusters, k = t - j * kMaxClusters;
    cT[t] = k < K ? __ldg(cent + k * d + j) : 0.0f;
  }
  uint32_t* off = reinterpret_cast<uint32_t*>(cT + kMaxFields * kMaxClusters);
  for (int j = tid; j < d; j += nthreads) {
    const FieldRef& F = fr[so.rd[j0 + j]];
    bool four = j % 4 == 0 && j + 4 <= d && F.s0 % 16 == 0 && F.ss % 16 == 0;
    for (int b = 1; b < 4 && four; ++b) four = fr[so.rd[j0 + j + b]].s0 == F.s0 + 4 * b;
    // (a warp's chunk buffer is below 64 KB, a stride below 8 KB)
    off[j] = (uint32_t)F.s0 | ((uint32_t)F.ss << 16) | (four ? kFour : 0u);
  }
}

// ASSIGN over the M records of each lane of a staged chunk (r = lane + 32m), for K clusters, the
// distances carried in registers: D_k = ((+0 + sq_0) + sq_1) + ..., sq_j = (x_j - c_kj)^2, features
// in ascending order, square and sum in one fma.  Two clusters share a packed instruction (their
// centroid coordinates are neighbours in the table); an odd last cluster pairs two records instead.
// A broadcast load still writes every lane's register (128 bytes per cycle and SM): a table of (c, c)
// pairs, two records per packed instruction, took 12 such cycles per feature and 64 records for 5
// clusters, this one 5.  8388608 x 32 features, one array per field: 300 -> 204 us.  In 132-byte
// structs 317 -> 291 us, and 200 us with the membership stores left out: the 4-byte stores, one dirty
// 32-byte sector per record, are what bounds it there (writing the whole sector instead: 310 us,
// the whole record: 354 us).
template <int M, int K>
__device__ __forceinline__ void assign_chunk_k(const SecOp& so, const FieldRef* fr, uint8_t* stage, int64_t i0,
                                               int lane, const float* cT) {
  const int d = so.rd_off[ADHA_F32 + 1] - so.rd_off[ADHA_F32];
  constexpr int P = K / 2, H = (M + 1) / 2;
  unsigned long long D[P + 1][M], Do[H];   // clusters 2p, 2p + 1 of record m; the odd cluster of records 2h, 2h + 1
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int m = 0; m < M; ++m) D[p][m] = 0ull;   // +0.0f in both halves
#pragma unroll
  for (int h = 0; h < H; ++h) Do[h] = 0ull;
  const uint32_t* off = reinterpret_cast<const uint32_t*>(cT + kMaxFields * kMaxClusters);
  auto load = [&](uint32_t o, float (&x)[M]) {
    const int ss = (int)(o >> 16 & 0x7FFFu);
    const uint8_t* p = stage + (o & 0xFFFFu) + lane * ss;
#pragma unroll
    for (int m = 0; m < M; ++m) x[m] = *reinterpret_cast<const float*>(p + m * 32 * ss);
  };
  auto add = [&](int j, const float (&x)[M]) {
    const float* c = cT + j * kMaxClusters;
    unsigned long long c2[4];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (K >= 4 * q + 4) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(c + 4 * q);
        c2[2 * q] = v.x;
        c2[2 * q + 1] = v.y;
      } else if (K >= 4 * q + 2) {
        c2[2 * q] = *reinterpret_cast<const unsigned long long*>(c + 4 * q);
      }
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const unsigned long long xx = f2_pack(x[m], x[m]);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const unsigned long long df = f2_sub_rn(xx, c2[p]);
        D[p][m] = f2_fma_rn(df, df, D[p][m]);
      }
    }
    if constexpr (K % 2 != 0) {
      const unsigned long long co = f2_pack(c[K - 1], c[K - 1]);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const unsigned long long df = f2_sub_rn(f2_pack(x[2 * h], 2 * h + 1 < M ? x[2 * h + 1] : 0.0f), co);
        Do[h] = f2_fma_rn(df, df, Do[h]);
      }
    }
  };
  // four features at a time: their places, then their values, then the arithmetic, so that a block's
  // shared-memory loads are in flight together (the loop's bound is a run-time value)
  int j = 0;
  for (; j + 4 <= d; j += 4) {
    const uint4 o = *reinterpret_cast<const uint4*>(off + j);
    float x[4][M];
    if (o.x & kFour) {
      const int ss = (int)(o.x >> 16 & 0x7FFFu);
      const uint8_t* p = stage + (o.x & 0xFFFFu) + lane * ss;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const float4 v = *reinterpret_cast<const float4*>(p + m * 32 * ss);
        x[0][m] = v.x;
        x[1][m] = v.y;
        x[2][m] = v.z;
        x[3][m] = v.w;
      }
    } else {
      load(o.x, x[0]);
      load(o.y, x[1]);
      load(o.z, x[2]);
      load(o.w, x[3]);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) add(j + b, x[b]);
  }
  for (; j < d; ++j) {
    float x[M];
    load(off[j], x);
    add(j, x);
  }
#pragma unroll
  for (int m = 0; m < M; ++m) {
    float Dm[kMaxClusters + 1];
#pragma unroll
    for (int p = 0; p < P; ++p) f2_unpack(D[p][m], &Dm[2 * p], &Dm[2 * p + 1]);
    if constexpr (K % 2 != 0) {
      float lo, hi;
      f2_unpack(Do[m / 2], &lo, &hi);
      Dm[K - 1] = m % 2 ? hi : lo;
    }
    int best = 0;
    float bd = Dm[0];
#pragma unroll
    for (int k = 1; k < K; ++k)
      if (Dm[k] < bd) {
        bd = Dm[k];
        best = k;
      }
    const int r = lane + 32 * m;
    StagedRec{fr, stage, r, i0 + r}.template st<int32_t>(so.arg[0], best);
  }
}

template <int M>
__device__ __forceinline__ void assign_chunk(const SecOp& so, const FieldRef* fr, uint8_t* stage, int64_t i0, int lane,
                                             const float* cT) {
  switch (so.arg[1]) {   // K, uniform over the launch
    case 1: assign_chunk_k<M, 1>(so, fr, stage, i0, lane, cT); break;
    case 2: assign_chunk_k<M, 2>(so, fr, stage, i0, lane, cT); break;
    case 3: assign_chunk_k<M, 3>(so, fr, stage, i0, lane, cT); break;
    case 4: assign_chunk_k<M, 4>(so, fr, stage, i0, lane, cT); break;
    case 5: assign_chunk_k<M, 5>(so, fr, stage, i0, lane, cT); break;
    case 6: assign_chunk_k<M, 6>(so, fr, stage, i0, lane, cT); break;
    case 7: assign_chunk_k<M, 7>(so, fr, stage, i0, lane, cT); break;
    default: assign_chunk_k<M, 8>(so, fr, stage, i0, lane, cT); break;
  }
}

// Where a REDUCE lane finds its feature (lane j = feature j, if j < d) and the membership in a
// staged chunk; looked up once per kernel, since the lanes index the field table differently.
struct ReduceLane {
  int d, K;
  int sx, ssx, sm, ssm;   // chunk-buffer offset and stride of the lane's feature and of the membership
  int skew;               // one-field feature slice: the lane starts at its own record (spread banks)
  bool walk;              // sum cluster by cluster into registers (see reduce_chunk_any)
};

// Shared memory of a REDUCE per CTA: every warp's record list (walk), or the two sum tables of every warp;
// and the table of reduce_flush, in the lists' place or after the tables.  (Lists that are not used left an
// SM with one CTA instead of two: 4000037 records of 32 features in 13 groups, one-field ones among them,
// 237 us, 170 without.)
constexpr size_t kReduceTableBytes = (size_t)kWarps * 2 * (kMaxClusters + 1) * 32 * 8;
constexpr int kReduceList = 128 + 4 * kMaxClusters + 8;   // 128 records, clusters in whole fours, 8 to read ahead
constexpr size_t kReduceListBytes = (size_t)kWarps * kReduceList * 4;
constexpr size_t kReduceFlushBytes = (size_t)kMaxClusters * (kMaxReduceFeatures + 1) * 8;
static_assert(kReduceListBytes >= kReduceFlushBytes, "the flush table fits the record lists");
__host__ __device__ constexpr size_t reduce_smem_bytes(bool walk) {
  return walk ? kReduceListBytes : kReduceTableBytes + kReduceFlushBytes;
}

// walk: every feature lies in a slice wider than one field (decided on the host, which sizes the
// shared tables only for the other way).
__device__ __forceinline__ ReduceLane reduce_lane(const SecOp& so, const FieldRef* fr, int lane, bool walk) {
  ReduceLane q;
  const int j0 = so.rd_off[ADHA_F32];
  q.d = so.rd_off[ADHA_F32 + 1] - j0;
  q.K = so.arg[1];
  const FieldRef& Fm = fr[so.arg[0]];
  q.sm = Fm.s0;
  q.ssm = Fm.ss;
  q.sx = q.ssx = 0;
  if (lane < q.d) {
    const FieldRef& Fx = fr[so.rd[j0 + lane]];
    q.sx = Fx.s0;
    q.ssx = Fx.ss;
  }
  q.skew = q.ssx == 4 ? lane : 0;
  q.walk = walk;
  return q;
}

template <int M>
__device__ __forceinline__ void reduce_sums(const ReduceLane& q, const uint8_t* stage, int lane,
                                            long long* __restrict__ acc, long long* __restrict__ acc2);

// REDUCE over the R = 32*M records of a staged chunk.  Counts: lane = record, one ballot per
// cluster and 32 records, lane k keeping cluster k's count (one register).
// Sums, lane j = feature j, integer sums (any order gives the same result):
// * walk (every feature in a slice wider than one field, e.g. AoS): the warp lists the chunk's
//   records cluster by cluster (a counting sort by ballots into its list `idx`), each cluster's
//   part rounded up to whole fours with the index R, a record of zeros that follows every slice
//   of such a chunk (q(0) = 0).  Cluster by cluster, all lanes then read the listed records
//   (consecutive words of a struct) four at a time, one 16-byte load for the four indices, and
//   add into the register sums sum[k]: no remainder loop, no shared-memory accumulator, no chain
//   through memory.  8388608 records of 132 bytes, 5 clusters: 314 us and 1043 instructions per 32
//   records with a list per 32 records read index by index and a remainder loop per cluster, 248 us
//   with this list, 223 us with the loads ahead of the sums (576 instructions; 0.73 of the copy
//   bandwidth, what is left is the latency of a chunk's phases at 16 warps per SM);
// * else (one-field slices, where the lanes reading one record would all hit one bank): each
//   lane starts at its own record and adds every record into its row of two (K+1) x 32 tables in
//   shared memory, even records into the first and odd into the second, so that two
//   read-add-write chains are in flight (row K takes memberships outside [0, K)).
template <int M>
__device__ __forceinline__ void reduce_chunk_any(const ReduceLane& q, const uint8_t* stage, int lane,
                                                 long long* __restrict__ acc, long long* __restrict__ acc2,
                                                 int* __restrict__ idx, long long (&sum)[kMaxClusters],
                                                 unsigned long long* cnt) {
  if (q.walk) {
    const unsigned lt = (1u << lane) - 1u;
    int mm[M], end[kMaxClusters];
#pragma unroll
    for (int m = 0; m < M; ++m) mm[m] = *reinterpret_cast<const int32_t*>(stage + q.sm + (lane + 32 * m) * q.ssm);
    int at = 0;
#pragma unroll
    for (int k = 0; k < kMaxClusters; ++k) {
      end[k] = at;
      if (k < q.K) {
        const int first = at;
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const unsigned b = __ballot_sync(0xFFFFFFFFu, mm[m] == k);
          if (mm[m] == k) idx[at + __popc(b & lt)] = lane + 32 * m;
          at += __popc(b);
        }
        if (lane == k) *cnt += (unsigned long long)(at - first);
        const int up = (at + 3) & ~3;
        if (lane < up - at) idx[at + lane] = 32 * M;
        at = up;
        end[k] = at;
      }
    }
    if (lane < 8) idx[at + lane] = 32 * M;   // what the loads ahead of the last fours read
    __syncwarp();
    if (lane < q.d) {
      // the indices two fours ahead and the values one four ahead of the sums, across clusters
      const uint8_t* px = stage + q.sx;
      auto four = [&](const int4& r) {
        return make_float4(*reinterpret_cast<const float*>(px + r.x * q.ssx), *reinterpret_cast<const float*>(px + r.y * q.ssx),
                           *reinterpret_cast<const float*>(px + r.z * q.ssx), *reinterpret_cast<const float*>(px + r.w * q.ssx));
      };
      float4 x = four(*reinterpret_cast<const int4*>(idx));
      int4 r = *reinterpret_cast<const int4*>(idx + 4);
      int t = 0;
#pragma unroll
      for (int k = 0; k < kMaxClusters; ++k) {
#pragma unroll 1
        for (; t < end[k]; t += 4) {
          const float4 v = x;
          x = four(r);
          r = *reinterpret_cast<const int4*>(idx + t + 8);
          sum[k] = add_wide(sum[k], fix32(v.x));
          sum[k] = add_wide(sum[k], fix32(v.y));
          sum[k] = add_wide(sum[k], fix32(v.z));
          sum[k] = add_wide(sum[k], fix32(v.w));
        }
      }
    }
    __syncwarp();   // the list is rewritten for the next chunk
    return;
  }
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int mm = *reinterpret_cast<const int32_t*>(stage + q.sm + (lane + 32 * m) * q.ssm);
#pragma unroll
    for (int k = 0; k < kMaxClusters; ++k)
      if (k < q.K) {
        const unsigned b = __ballot_sync(0xFFFFFFFFu, mm == k);
        if (lane == k) *cnt += (unsigned long long)__popc(b);
      }
  }
  reduce_sums<M>(q, stage, lane, acc, acc2);
}


template <int M>
__device__ __forceinline__ void reduce_sums(const ReduceLane& q, const uint8_t* stage, int lane,
                                            long long* __restrict__ acc, long long* __restrict__ acc2) {
  constexpr int R = 32 * M;
  if (lane < q.d) {
    long long* __restrict__ col = acc + lane;
    long long* __restrict__ col2 = acc2 + lane;
    const uint8_t* pm = stage + q.sm;
    const uint8_t* px = stage + q.sx;
#pragma unroll 2
    for (int i = 0; i < R; i += 2) {
      const int r0 = (i + q.skew) & (R - 1), r1 = (i + 1 + q.skew) & (R - 1);
      const int m0 = *reinterpret_cast<const int32_t*>(pm + r0 * q.ssm);
      const int m1 = *reinterpret_cast<const int32_t*>(pm + r1 * q.ssm);
      const long long v0 = fixq(*reinterpret_cast<const float*>(px + r0 * q.ssx));
      const long long v1 = fixq(*reinterpret_cast<const float*>(px + r1 * q.ssx));
      // a membership outside [0, K) goes to the scratch row kMaxClusters, never read back
      const int row0 = (unsigned)m0 < (unsigned)q.K ? m0 : kMaxClusters;
      const int row1 = (unsigned)m1 < (unsigned)q.K ? m1 : kMaxClusters;
      col[row0 * 32] += v0;
      col2[row1 * 32] += v1;
    }
  }
}

// REDUCE over records [t0, n) read from global memory (the ragged tail): lane j = feature j, lane k
// counts cluster k; sums into the register sums (walk) or row mm of the first shared table.  Up to 127
// records by one warp: 32 memberships and then eight records' features are read at a time, or their
// latencies are most of a short launch.
__device__ __forceinline__ void reduce_tail(const ReduceLane& q, const SecOp& so, const FieldRef* fr, int64_t t0,
                                            int64_t n, int lane, long long* acc, long long (&sum)[kMaxClusters],
                                            unsigned long long* cnt) {
  const FieldRef& Fm = fr[so.arg[0]];
  const FieldRef& Fx = fr[so.rd[so.rd_off[ADHA_F32] + (lane < q.d ? lane : 0)]];
  const uint8_t* x0 = Fx.g;
  const int xs = Fx.gs;
  for (int64_t b = t0; b < n; b += 32) {
    const int m = (int)(n - b < 32 ? n - b : 32);
    const int member = lane < m ? *reinterpret_cast<const int32_t*>(Fm.g + (b + lane) * Fm.gs) : -1;
#pragma unroll 1
    for (int r = 0; r < m; r += 8) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = r + u < m ? *reinterpret_cast<const float*>(x0 + (b + r + u) * xs) : 0.0f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int mm = __shfl_sync(0xFFFFFFFFu, member, r + u);   // -1 beyond the last record
        if ((unsigned)mm >= (unsigned)q.K) continue;
        if (lane == mm) *cnt += 1ull;
        if (lane < q.d) {
          const long long v = fixq(x[u]);
          if (q.walk) {
#pragma unroll
            for (int k = 0; k < kMaxClusters; ++k) sum[k] += k == mm ? v : 0ll;
          } else {
            acc[mm * 32 + lane] += v;
          }
        }
      }
    }
  }
}

// The warps' sums and counts added into the result (K rows of [count, d sums], zeroed before the launch
// unless the caller accumulates), by all threads of the CTA.  They are added up in shared memory first
// (`table`: see reduce_smem_bytes; the record lists are done with by now): warp by warp, over a million additions to a few
// hundred addresses took most of a short launch (2^16 records of 32 features in 5 clusters 21 -> 14.8 us,
// 2^20 57.9 -> 41.5, 2^23 222 -> 213.5).  Whole numbers: the order does not matter.
__device__ __forceinline__ void reduce_flush(const ReduceLane& q, const SecOp& so, int warp, int lane, long long* table,
                                             const long long* acc, const long long (&sum)[kMaxClusters],
                                             const unsigned long long* cnt) {
  const int d = q.d, row = d + 1;
  for (int w = 0; w < kWarps; ++w) {
    __syncthreads();
    if (warp != w) continue;
#pragma unroll
    for (int k = 0; k < kMaxClusters; ++k)
      if (k < q.K && lane < d) {
        const long long v = q.walk ? sum[k] : acc[k * 32 + lane] + acc[(kMaxClusters + 1 + k) * 32 + lane];
        table[k * row + 1 + lane] = w ? table[k * row + 1 + lane] + v : v;
      }
    if (lane < q.K) table[lane * row] = (w ? table[lane * row] : 0) + (long long)*cnt;
  }
  __syncthreads();
  unsigned long long* out = static_cast<unsigned long long*>(const_cast<void*>(so.aux));
  for (int e = warp * 32 + lane; e < q.K * row; e += kThreads) atomicAdd(out + e, (unsigned long long)table[e]);
}

}  // namespace adha
