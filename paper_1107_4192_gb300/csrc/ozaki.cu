// Exact-slice (Ozaki-scheme) products on the 5th-generation tensor cores.
//
// Slicing (oz_slice_kernel): one CTA per row finds the row's largest
// magnitude, takes its binary exponent e (max < 2^e), rounds each element to
// the integer X_int = RNE(x 2^(7 + 8(S-1) - e)) and writes its signed base-256
// digits (|q_p| <= 128) as bf16 planes, in integer arithmetic on the bits of
// x (the float64 units of this GPU would make float64 slicing the slow part).
//
// Product (oz_gemm_kernel): one 128 x 64 output tile per CTA, 19 warps.
//   warp 0  one lane issues the TMA loads (64-byte swizzle) of all slices of a
//           32-wide k-slice (two MMA k-steps) of A and B into a shared-memory
//           stage;
//   warp 1  allocates TMEM (LV + 1 buffers of 128 x 64 float32, rotating among
//           the levels so a level's drain overlaps the MMAs); the whole warp
//           runs the issue loop (warp-uniform arithmetic) and one elected lane
//           issues, per stage, the MMAs of every slice pair: per A slice, its
//           partner levels in runs of up to four whose buffers are adjacent,
//           one MMA of N = 64 x run each; after the last k-slice of a level's
//           chunk it commits the level's buffer to its "ready"
//           barrier, and a level's next chunk starts (overwriting) in a buffer
//           the epilogue has drained;
//   warp 2  the gate: waits for each step's operands and drained buffer and releases it to warp 1;
//   warps 3-18 per chunk and level, read the accumulator (an exact integer
//           below 2^24), convert it to an integer and add it into 64-bit
//           fixed-point accumulators in registers (levels 0-2 and levels 3..
//           in two of them); at the end scale by the row and column exponents
//           and apply the float64 epilogue.
// Every pipeline wait is bounded (kernel argument, as in the split-bf16 kernel).
#include <type_traits>

#include "ozaki.cuh"
#include "tc_ptx.cuh"

namespace kfm {

namespace {

constexpr int OZ_BM = 128;      // output rows per CTA (TMEM lanes)
constexpr int OZ_BN = 64;       // output columns per CTA (TMEM columns per level)
constexpr int OZ_SPLIT_K = 128; // K splits begin at multiples of this
constexpr int OZ_EPI_WARPS = 16;  // 4 TMEM lane quadrants x 4 column quarters of 16
constexpr int OZ_GATE_WARP = 2;   // waits for each step's operands and buffer
constexpr int OZ_EPI0 = 3;        // first epilogue warp
constexpr int OZ_THREADS = 32 * (OZ_EPI0 + OZ_EPI_WARPS);
constexpr int OZ_GROUP = 8;     // row tiles per rasterisation group (operand reuse in L2)
constexpr int OZ_ROW_PAD = 128;
constexpr int kOzBK = 32;       // k per pipeline stage of the launched kernels (two MMA k-steps)
constexpr int kOzBadRow = 0x7fffffff;  // exponent marking a row that holds an infinity or NaN
constexpr int kOzScaleMax = 80;        // of a balancing exponent: float32 diagonals stay within it

// LV slice levels, LA <= LV slices of A and LV of B; BK values of k per pipeline stage, one swizzled row
// of bf16 (16: 32-byte swizzle, one MMA k-step; 32: 64-byte swizzle, two k-steps, half the stages and wider
// TMA rows).
template <int LV, int LA, int BK>
struct OzCfg {
  static_assert(LA >= 1 && LA <= LV, "slices of A");
  static_assert(BK == 16 || BK == 32, "one 32- or 64-byte swizzled row of bf16 per stage");
  static constexpr int SWZ = BK * 2;                         // swizzle width in bytes
  static constexpr uint32_t LAYOUT = BK == 16 ? kLayoutSw32 : kLayoutSw64;  // descriptor swizzle mode
  static constexpr uint32_t SBO = 8 * SWZ;                   // bytes between 8-row groups
  // values of k per exact chunk: a level has at most LA slice pairs, whose products are at most 2^14 in
  // magnitude, so a chunk sums to an integer of at most 2^24, exact in float32.  As long as that allows: draining
  // a level costs the epilogue about 1100 cycles whatever the chunk's length, and with 128 for all the
  // drains, not the MMAs, set the pace of the products with few slices of A (<7, 3> 21.1 ms and <5, 2>
  // 14.4 ms at N = 8196; with these chunks 19.7 and 12.5 ms).
  static constexpr int KC = LA <= 2 ? 512 : LA <= 4 ? 256 : LA == 5 ? 192 : 128;
  // SK MMA k-steps (of 16) make one step, the unit in which levels start chunks and the roles synchronise: a
  // whole stage where a chunk still has more stages than there are levels, since a step costs about 390
  // cycles (gate, commits, an empty MMA queue) beside its MMAs (N = 8196: <7, 3> 19.7 -> 15.8 ms, 0.74 of the
  // sustained bf16 rate; <5, 2> 12.5 -> 9.4 ms).
  static constexpr int SK = KC / BK > LV ? BK / 16 : 1;
  static constexpr int KS = BK / 16 / SK;                    // steps per stage
  static constexpr int CKS = KC / (16 * SK);                 // steps per exact chunk
  static constexpr int A_BYTES = OZ_BM * BK * 2;
  static constexpr int B_BYTES = OZ_BN * BK * 2;
  static constexpr int STAGE_BYTES = LA * A_BYTES + LV * B_BYTES;
  static constexpr int FIT = (210 * 1024) / STAGE_BYTES;
  static constexpr int STAGES = FIT > 8 ? 8 : FIT;
  static_assert(STAGES >= 2, "double-buffered pipeline");
  // NB = LV + 1 accumulators rotate among the levels (chunk k of level l in buffer (l + k) mod NB),
  // so the buffer a level leaves is drained while the MMAs continue in the spare one
  static constexpr int NB = LV + 1;
  static_assert(NB * OZ_BN <= 512, "one TMEM accumulator per level plus a spare");
  static_assert(LV < CKS, "one level changes chunk per step");
  static_assert(LA * KC * 16384 <= (1 << 24), "exact chunk");
  static_assert(2 * STAGES + 2 * NB + 1 <= 28, "barriers fit their 256 bytes");
  static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024 + 256;
  // instruction descriptor: D = f32, A = B = bf16, both K-major, M >> 4; N >> 3 at bit 17 per MMA
  static constexpr uint32_t IDESC_M = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(OZ_BM >> 4) << 24);
};

struct OzMaps {
  CUtensorMap a, b;  // all slice planes of A (box 32 x 128) and of B (box 32 x 64)
};

// Full epilogue of element (gi, gj), gi >= gj when sym, from its product value c.
__device__ __forceinline__ double oz_qv(int kind, const double* q, int64_t ldq, int i, int j) {
  if (kind == 0) return i == j ? q[0] : 0.0;
  if (kind == 1) return i == j ? q[i] : 0.0;
  if (kind == 2) return q[(int64_t)i * ldq + j];
  return 0.0;
}

// The epilogue keeps off the float64 unit, which runs one warp instruction per 19 cycles and SM: a tile of
// 128 x 64 elements with the six or so float64 operations per element of the plain formulas (two
// scalings, their sum, alpha, beta, a zero from Q, the float32 conversion) cost 16 us, as much as the
// products of a short K.  Scaling and conversions are integer operations on the bits with the same
// rounding (to nearest, ties to even); what is left is at most one float64 addition per element, and
// a tile's sweep takes 3 us (M x N x K = 1664 x 128 x 128: the launch 28 us before, 15 us now).

__device__ __noinline__ double scaled_general(unsigned long long m, int e) { return scalbn((double)m, e); }

// (H 2^32 + L) 2^e rounded to float64, for a magnitude whose leading bit is bit 62 (so that rounding up
// cannot overflow; any bits lost before are or-ed into bit 0); sign is the result's sign bit.
__device__ __forceinline__ double round53(uint32_t H, uint32_t L, int e, uint32_t sign) {
  const uint32_t add = 0x1ffu + ((L >> 10) & 1u);  // ties to even
  const uint32_t l = L + add;
  const uint32_t h = H + (l < add ? 1u : 0u);
  const uint32_t mh = h >> 10, ml = __funnelshift_r(l, h, 10);
  const int E = 1023 + 62 + e;  // biased exponent of the leading bit
  if ((unsigned)(E - 1) > 2043u) {
    const double v = scaled_general(((unsigned long long)mh << 32) | ml, e + 10);
    return __hiloint2double(__double2hiint(v) | (int)sign, __double2loint(v));
  }
  return __hiloint2double((int)((mh + ((uint32_t)(E - 1) << 20)) | sign), (int)ml);  // mh holds the leading bit
}

// t 2^e rounded to float64, |t| < 2^63.
__device__ __forceinline__ double fixed_to_double(long long t, int e) {
  const uint32_t sgn = (uint32_t)(t >> 63);
  const unsigned long long u = ((unsigned long long)t ^ (((unsigned long long)sgn << 32) | sgn)) + (sgn & 1u);
  uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  if (hi == 0) {
    if (lo == 0) return 0.0;
    hi = lo >> 1;  // keeps the leading bit below bit 63
    lo = lo << 31;
    e -= 31;
    if (hi == 0) {  // u == 1
      hi = 1u << 30;
      lo = 0;
      e -= 31;
    }
  }
  const int sh = __clz((int)hi) - 1;
  return round53(__funnelshift_l(lo, hi, sh), lo << sh, e - sh, sgn & 0x80000000u);
}

// (hi 2^s + lo) 2^e rounded to float64, for s <= 32, |hi| < 2^61, |lo| < 2^(30 + s) (K <= 2^20 keeps within).
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int s, int e) {
  // in units 2^(s - 32): hi 2^32 + lo 2^(32 - s), as a 96-bit integer (w2, w1, w0)
  const long long l = (long long)((unsigned long long)lo << (32 - s));
  const long long top = hi + (l >> 32);
  const uint32_t sgn = (uint32_t)(top >> 63);
  uint32_t w0 = (uint32_t)l ^ sgn;
  unsigned long long w = (unsigned long long)top ^ (((unsigned long long)sgn << 32) | sgn);
  if (sgn && ++w0 == 0) ++w;
  e -= 32 - s;
  const uint32_t w2 = (uint32_t)(w >> 32), w1 = (uint32_t)w;
  if (w2 == 0) {  // below 2^64
    if (w1 == 0) {
      const double v = fixed_to_double((long long)w0, e);
      return __hiloint2double(__double2hiint(v) | (int)(w0 ? sgn & 0x80000000u : 0u), __double2loint(v));
    }
    const int n = __clz((int)w1);
    if (n == 0) return round53(w1 >> 1, (w1 << 31) | (w0 >> 1) | (w0 & 1u), e + 1, sgn & 0x80000000u);
    return round53(__funnelshift_l(w0, w1, n - 1), w0 << (n - 1), e - (n - 1), sgn & 0x80000000u);
  }
  const int sh = __clz((int)w2) - 1;  // |top| < 2^62
  const uint32_t lost = w0 << sh;
  return round53(__funnelshift_l(w1, w2, sh), __funnelshift_l(w0, w1, sh) | (lost ? 1u : 0u), e + 32 - sh,
                 sgn & 0x80000000u);
}

// float64 to float32, to nearest, ties to even.
__device__ __noinline__ float narrow_general(double v) { return (float)v; }
__device__ __forceinline__ float narrow(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned E = (unsigned)(b >> 52) & 0x7ffu;
  if (E - 897u > 1149u - 897u) return narrow_general(v);  // outside float32's normal range (zero, infinity, NaN too)
  const unsigned long long mag = (b & 0x7fffffffffffffffull) - (896ull << 52);
  unsigned f = (unsigned)(mag >> 29);
  const unsigned rem = (unsigned)mag & 0x1fffffffu;
  f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1))) ? 1u : 0u;
  return __uint_as_float(f | ((unsigned)(b >> 32) & 0x80000000u));
}

// alpha c + beta cin.  alpha_unit and beta_unit are set on the host (a float64 comparison costs as much as
// an addition), and the general form is a call: inlined, its float64 instructions would be predicated, and
// predicated-off ones still take their turn.
__device__ __noinline__ double oz_axpby_general(double alpha, double c, double beta, double cin) {
  return fma(beta, cin, alpha * c);
}
template <bool CIN>
__device__ __forceinline__ double oz_axpby(const OzEpilogue& e, double c, double cin) {
  if (e.alpha_unit == 0 || (CIN && !e.beta_unit)) return oz_axpby_general(e.alpha, c, CIN ? e.beta : 0.0, CIN ? cin : 0.0);
  const double ac = __longlong_as_double(__double_as_longlong(c) ^ (e.alpha_unit < 0 ? 1ll << 63 : 0ll));
  if constexpr (CIN) return cin + ac;
  return ac;
}

// v + Q[i][j]
__device__ __forceinline__ double oz_addq(double v, int kind, const double* q, int64_t ldq, int i, int j) {
  return (kind == 2 || (kind >= 0 && i == j)) ? v + oz_qv(kind, q, ldq, i, j) : v;
}

__device__ __forceinline__ void oz_apply(const OzEpilogue& e, int gi, int gj, double c) {
  double v = e.alpha * c;
  if (e.cin) v += e.beta * e.cin[(int64_t)gi * e.ldcin + gj];
  if (gi == gj) v += e.delta;
  if (e.radd_kind >= 0) v += oz_qv(e.radd_kind, e.radd, e.ldradd, gi, gj);
  const bool mirror = e.sym && gi != gj;
  if (e.out) {
    e.out[(int64_t)gi * e.ldo + gj] = v;
    if (mirror) e.out[(int64_t)gj * e.ldo + gi] = v;
  }
  if (e.outf) {
    e.outf[(int64_t)gi * e.ldof + gj] = (float)v;
    if (mirror) e.outf[(int64_t)gj * e.ldof + gi] = (float)v;
  }
  if (e.outT) e.outT[(int64_t)gj * e.ldoT + gi] = v;
  if (e.out2) {
    e.out2[(int64_t)gi * e.ldo2 + gj] = v + oz_qv(e.q_kind, e.q, e.ldq, gi, gj);
    if (mirror) e.out2[(int64_t)gj * e.ldo2 + gi] = v + oz_qv(e.q_kind, e.q, e.ldq, gj, gi);
  }
  if (gi == gj) {
    if (e.diag_out) e.diag_out[gi] = v;
    if (e.check_diag && !(v > 0.0 && isfinite(v))) status_set(e.status, KF_ERR_NUMERIC, e.step, gi);
  }
}

struct OzArgs {
  int M, N, nk;                  // nk = k-slices of BK (all of K)
  int kt_per_split;              // k-slices per split (blockIdx.y)
  double* partials;              // splits > 1: raw sums, split s at partials + s M N (ld N)
  long long* sums;               // exact splits: integer sums, split s at sums + s M ld_sums
  int64_t ld_sums;
  int a_rows_pad, b_rows_pad;    // plane p starts at row p * rows_pad of its map
  const int* ea;
  const int* eb;
  OzEpilogue e;
  uint64_t wait_ns;
};

// Sign, integer mantissa and binary exponent of x (x = sign mant 2^exp2), read from its bits;
// false for an infinity or NaN.
__device__ __forceinline__ bool decompose(double x, long long& mant, int& exp2, bool& neg) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  neg = (b >> 63) != 0;
  mant = (long long)(b & 0xFFFFFFFFFFFFFull) | (E ? (1ll << 52) : 0ll);
  exp2 = (E ? E : 1) - 1075;
  return E != 0x7FF;
}
__device__ __forceinline__ bool decompose(float x, long long& mant, int& exp2, bool& neg) {
  const unsigned b = __float_as_uint(x);
  const int E = (int)((b >> 23) & 0xFF);
  neg = (b >> 31) != 0;
  mant = (long long)(b & 0x7FFFFFu) | (E ? (1ll << 23) : 0ll);
  exp2 = (E ? E : 1) - 150;
  return E != 0xFF;
}

// Magnitude bits of x as an unsigned integer: ordered like |x| for finite values, and above
// every finite value for infinities and NaNs.
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long mag_bits(float x) {
  return ((unsigned long long)(__float_as_uint(x) & 0x7FFFFFFFu)) << 29;  // same order as a double's bits
}
// Magnitude bits from which on a value is an infinity or NaN.
template <typename T>
__device__ __forceinline__ unsigned long long mag_inf() {
  return sizeof(T) == 8 ? 0x7FF0000000000000ull : 0x7F800000ull << 29;
}
// The binary exponent e of magnitude bits: 2^(e-1) <= value < 2^e (0 for zero), as frexp gives it.
template <typename T>
__device__ __forceinline__ int mag_exponent(unsigned long long mag) {
  const int E = (int)(mag >> 52);
  if (E > 0) return E - (sizeof(T) == 8 ? 1022 : 126);
  if (mag == 0) return 0;
  const int top = 63 - __clzll((long long)mag);  // subnormal: leading bit of the mantissa
  return sizeof(T) == 8 ? top - 1073 : top - 29 - 148;
}

// x 2^shift rounded to the nearest integer, ties to even (exact integer arithmetic).
__device__ __forceinline__ long long fixed_rne(long long mant, int exp2, bool neg, int shift) {
  const int total = exp2 + shift;
  long long r;
  if (total >= 0) {
    // |x| 2^shift < 2^(7 + 8(S-1)) <= 2^55 for every element of the row, so the shift cannot overflow
    r = total >= 63 ? 0 : mant << total;
  } else {
    const int sh = -total;
    r = sh >= 63 ? 0 : (mant + ((1ll << (sh - 1)) - 1) + ((mant >> sh) & 1)) >> sh;
  }
  return neg ? -r : r;
}

// Eight consecutive values of a row, from k0 on (zero at and beyond cols).
template <typename T>
__device__ __forceinline__ void load8(const T* row, int64_t k0, int64_t cols, bool vec, T (&v)[8]) {
  if (vec && k0 + 8 <= cols) {
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        const double2 d = *reinterpret_cast<const double2*>(row + k0 + i);
        v[i] = d.x;
        v[i + 1] = d.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; i += 4) {
        const float4 f = *reinterpret_cast<const float4*>(row + k0 + i);
        v[i] = f.x;
        v[i + 1] = f.y;
        v[i + 2] = f.z;
        v[i + 3] = f.w;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = k0 + i < cols ? row[k0 + i] : T(0);
  }
}

// Eight consecutive values of a 16-byte aligned row from k0 on, up to cols.
__device__ __forceinline__ void store8(float* row, int64_t k0, int64_t cols, const float (&v)[8]) {
  if (k0 + 8 <= cols) {
    reinterpret_cast<float4*>(row + k0)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(row + k0)[1] = make_float4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (k0 + i < cols) row[k0 + i] = v[i];
  }
}

// The exponent e of x 2^w, 2^(e-1) <= |x| 2^w < 2^e; kOzZero for zero, kOzBadRow for an infinity or NaN.
constexpr int kOzZero = -0x7fffffff;
__device__ __forceinline__ int exponent_of(double x, int w) {
  const unsigned long long m = mag_bits(x);
  const int E = (int)(m >> 52);
  if (E == 0x7ff) return kOzBadRow;
  return E > 0 ? E - 1022 + w : m == 0 ? kOzZero : 63 - __clzll((long long)m) - 1073 + w;
}
__device__ __forceinline__ int exponent_of(float x, int w) {
  const unsigned m = __float_as_uint(x) & 0x7fffffffu;
  const int E = (int)(m >> 23);
  if (E == 0xff) return kOzBadRow;
  return E > 0 ? E - 126 + w : m == 0 ? kOzZero : 31 - __clz((int)m) - 148 + w;
}

// Eight weights sign scale[0..7], 16-byte aligned.
__device__ __forceinline__ void weights8(const int* scale, int sign, int (&w)[8]) {
  const int4 a = reinterpret_cast<const int4*>(scale)[0], b = reinterpret_cast<const int4*>(scale)[1];
  const int v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) w[i] = sign * v[i];
}

// q 2^k for an integer |q| <= 2^24, rounded like ldexpf.
__device__ __forceinline__ float scaled(int q, int k) {
  return (unsigned)(k + 126) <= 252u ? (float)q * __int_as_float((k + 127) << 23) : ldexpf((float)q, k);
}

// Signed base-256 digits of eight integers |x| <= 2^(8S - 1), written as bf16 to S planes (16-byte stores).
// Digit p is q_p = Q_p - 256 Q_{p-1} with Q_p = x / 2^(8(S-1-p)) rounded to nearest, ties to even: the
// successive rounding of the remainders, since a remainder differs from x by multiples of 256 2^(8(S-1-p)).
// The low 32 bits of each Q_p are enough.
__device__ __forceinline__ void write_digits8(const long long (&x)[8], int S, __nv_bfloat16* dst, int64_t pstride) {
  uint32_t prev[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) prev[i] = 0;
  for (int p = 0; p < S; ++p, dst += pstride) {
    const int sp = 8 * (S - 1 - p);
    uint32_t w[4];
    float f[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t q;
      if (sp > 0)
        q = (uint32_t)((x[i] + ((1ll << (sp - 1)) - 1) + ((x[i] >> sp) & 1)) >> sp);
      else
        q = (uint32_t)x[i];
      const uint32_t d = q - (prev[i] << 8);
      prev[i] = q;
      f[i] = __uint_as_float(0x4B400000u + d) - 12582912.0f;  // (float)(int)d for |d| < 2^22
    }
#pragma unroll
    for (int i = 0; i < 8; i += 2)  // |d| <= 128: exact in bf16, the upper half of the float32
      w[i / 2] = __byte_perm(__float_as_uint(f[i]), __float_as_uint(f[i + 1]), 0x7632);
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// w: a power of two for each value.
template <typename T>
__device__ __forceinline__ void slice8(const T (&v)[8], const int (&w)[8], int shift, bool bad, int S, __nv_bfloat16* dst,
                                       int64_t pstride) {
  long long x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    long long mant;
    int exp2;
    bool neg;
    decompose(v[i], mant, exp2, neg);
    x[i] = bad ? 0 : fixed_rne(mant, exp2 + w[i], neg, shift);
  }
  write_digits8(x, S, dst, pstride);
}

// Maximum over the warp (kGroup 32) or the 256-thread block, to all its threads.
template <int kGroup, typename V>
__device__ __forceinline__ V group_max(V mx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const V v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if constexpr (kGroup == 256) {
    __shared__ V red[8];
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = red[w] > mx ? red[w] : mx;
  }
  return mx;
}

// Slices of the rows: X[r][k] = 2^(e - 7 - 8(S-1)) X_int with X_int = RNE(X[r][k] 2^(7 + 8(S-1) - e)), in
// signed base-256 digits (|q_p| <= 128), all in integer arithmetic.  A group (a warp for short rows, else a
// 256-thread block) holds its row in registers, 8 NCH values per thread, so a row is read once: HBM-bound from
// a few thousand columns on (5124 x 5124 float64, 5 slices: 246 us with the digits in 64-bit arithmetic and two
// reads, 85 us now; 1664 x 128: 14.5 us and 5 us).  NCH = 0: two passes, for rows too long for that.
//
// WEIGH: the slices of X[r][k] 2^(sign scale[k]) (below; scale is readable up to ldk).
template <typename T, int kGroup, int NCH, bool WEIGH>
__global__ void __launch_bounds__(256) oz_slice_kernel(const T* X, int64_t ld, int64_t rows, int64_t cols, int S,
                                                       __nv_bfloat16* planes, int64_t rows_pad, int64_t ldk,
                                                       int* exps, const int* scale, int sign) {
  constexpr int kRows = 256 / kGroup;
  const int64_t r = (int64_t)blockIdx.x * kRows + threadIdx.x / kGroup;  // rows_pad is a multiple of kRows
  const int t = threadIdx.x % kGroup;
  const T* row = X + (r < rows ? r : 0) * ld;
  const int64_t n = r < rows ? cols : 0;  // rows beyond the matrix are zero
  const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && (ld * sizeof(T)) % 16 == 0;
  T v[NCH > 0 ? NCH : 1][8];
  int w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  bool bad;  // an infinity or NaN: zero slices, marked exponent
  int e;     // max |X[r]| < 2^e
  if constexpr (NCH > 0) {
#pragma unroll
    for (int c = 0; c < NCH; ++c) load8(row, (int64_t)(c * kGroup + t) * 8, n, vec, v[c]);
  }
  if constexpr (WEIGH) {
    int mx = kOzZero;
    auto take = [&](int64_t k0, const T (&x)[8]) {
      if (k0 >= ldk) return;
      weights8(scale + k0, sign, w);
#pragma unroll
      for (int i = 0; i < 8; ++i) mx = max(mx, exponent_of(x[i], w[i]));
    };
    if constexpr (NCH > 0) {
#pragma unroll
      for (int c = 0; c < NCH; ++c) take((int64_t)(c * kGroup + t) * 8, v[c]);
    } else {
      for (int64_t k0 = (int64_t)t * 8; k0 < ldk; k0 += kGroup * 8) {
        load8(row, k0, n, vec, v[0]);
        take(k0, v[0]);
      }
    }
    mx = group_max<kGroup>(mx);
    bad = mx == kOzBadRow;
    e = bad || mx == kOzZero ? 0 : mx;
  } else {
    unsigned long long mx = 0;
    if constexpr (NCH > 0) {
#pragma unroll
      for (int c = 0; c < NCH; ++c)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const unsigned long long m = mag_bits(v[c][i]);
          mx = m > mx ? m : mx;
        }
    } else {
      for (int64_t k = t; k < n; k += kGroup) {
        const unsigned long long m = mag_bits(row[k]);
        mx = m > mx ? m : mx;
      }
    }
    mx = group_max<kGroup>(mx);
    bad = mx >= mag_inf<T>();
    e = bad ? 0 : mag_exponent<T>(mx);
  }
  if (t == 0) exps[r] = bad ? kOzBadRow : e;
  const int shift = 7 + 8 * (S - 1) - e;
  const int64_t pstride = rows_pad * ldk;
  __nv_bfloat16* dst = planes + r * ldk;
  if constexpr (NCH > 0) {
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int64_t k0 = (int64_t)(c * kGroup + t) * 8;
      if (k0 >= ldk) continue;
      if constexpr (WEIGH) weights8(scale + k0, sign, w);
      slice8(v[c], w, shift, bad, S, dst + k0, pstride);
    }
  } else {
    for (int64_t k0 = (int64_t)t * 8; k0 < ldk; k0 += kGroup * 8) {
      load8(row, k0, n, vec, v[0]);
      if constexpr (WEIGH) weights8(scale + k0, sign, w);
      slice8(v[0], w, shift, bad, S, dst + k0, pstride);
    }
  }
}

// ---- slices of a refined inverse's operands, balanced
//
// The refinement rounds iterates to few digits below their row maxima, which is harmless only when P has rows of one
// scale.  So it works on D P D with D_i = 2^(s_i), s_i = -round(log2(P_ii) / 2), whose diagonal lies in [1/2, 2), and
// on D^{-1} X D^{-1}.  All of that stays in the slices: a row's own factor belongs to its exponent, and the slices of
// row i of X hold X[i][k] 2^(-s_k), those of row j of P hold P[j][k] 2^(s_k), so the product is X P as it stands.

// s_i from the diagonal (0 for one that is not positive and finite, which the factorisation reports), zero up to ldk.
__global__ void oz_balance_kernel(const void* P, int f64, int64_t ld, int64_t n, int64_t ldk, int* scale) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ldk; i += (int64_t)gridDim.x * blockDim.x) {
    int e = 0;
    if (i < n)
      e = f64 ? exponent_of(static_cast<const double*>(P)[i * ld + i], 0)
              : exponent_of(static_cast<const float*>(P)[i * ld + i], 0);
    scale[i] = e == kOzZero || e == kOzBadRow ? 0 : max(-kOzScaleMax, min(kOzScaleMax, -(e >> 1)));
  }
}

// Exponents alone of the rows of a float32 X[r][k] 2^(-scale[k]).
__global__ void __launch_bounds__(256) oz_exps_kernel(const float* X, int64_t ld, int64_t n, int64_t ldk, const int* scale,
                                                      int* exps) {
  const int64_t r = blockIdx.x;
  const int64_t cols = r < n ? n : 0;
  const float* row = X + (r < n ? r : 0) * ld;
  int mx = kOzZero, w[8];
  for (int64_t k0 = threadIdx.x * 8; k0 < ldk; k0 += 256 * 8) {
    float v[8];
    load8(row, k0, cols, true, v);  // ld is a multiple of 4 and rows are 16-byte aligned
    weights8(scale + k0, -1, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) mx = max(mx, exponent_of(v[i], w[i]));
  }
  mx = group_max<256>(mx);
  if (threadIdx.x == 0) exps[r] = mx == kOzZero ? 0 : mx;
}

// A symmetric float32 matrix rounded so that three slices of its weighed rows hold it exactly and it stays symmetric:
// with b_i = exps[i] - scale[i] the exponents of the balanced rows, element (i, j) of the balanced matrix to the
// nearest multiple of 2^(max(b_i, b_j) - 23), written back, with its three slices by rows.
__global__ void __launch_bounds__(256) oz_slice_symmetric_kernel(float* X, int64_t ld, int64_t n, const int* scale,
                                                                 __nv_bfloat16* planes, int64_t rows_pad, int64_t ldk,
                                                                 const int* exps) {
  const int64_t r = blockIdx.x;
  const bool live = r < n && exps[r] != kOzBadRow;
  const int sr = r < n ? scale[r] : 0, br = live ? exps[r] - sr : 0;
  float* row = X + (r < n ? r : 0) * ld;
  for (int64_t k0 = threadIdx.x * 8; k0 < ldk; k0 += 256 * 8) {
    long long x[8];
    float v[8];
    int sk[8], ek[8];
    load8(row, k0, live ? n : 0, true, v);
    weights8(scale + k0, 1, sk);
    weights8(exps + k0, 1, ek);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int g = k0 + i >= n || ek[i] == kOzBadRow ? br : max(br, ek[i] - sk[i]);
      long long mant;
      int exp2;
      bool neg;
      decompose(v[i], mant, exp2, neg);
      const long long q = fixed_rne(mant, exp2 - sr - sk[i], neg, 23 - g);
      x[i] = q << min(g - br, 40);  // |x| <= 2^23: the grid only gets coarser as g - br grows
      v[i] = scaled((int)q, g - 23 + sr + sk[i]);
    }
    write_digits8(x, 3, planes + r * ldk + k0, rows_pad * ldk);
    if (live) store8(row, k0, n, v);
  }
}

// Two slices of the weighed rows of a float32 correction C (rounded to nearest), and X = Y + Cs in float64 for a
// float32 Y and the correction Cs that the slices hold.
__global__ void __launch_bounds__(256) oz_slice_correction_kernel(const float* C, const float* Y, int64_t ld, int64_t n,
                                                                  const int* scale, __nv_bfloat16* planes, int64_t rows_pad,
                                                                  int64_t ldk, int* exps, double* X, int64_t ldx) {
  const int64_t r = blockIdx.x;
  const int64_t cols = r < n ? n : 0;
  const float *row = C + (r < n ? r : 0) * ld, *yrow = Y + (r < n ? r : 0) * ld;
  int mx = kOzZero, w[8];
  for (int64_t k0 = threadIdx.x * 8; k0 < ldk; k0 += 256 * 8) {
    float v[8];
    load8(row, k0, cols, true, v);
    weights8(scale + k0, -1, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) mx = max(mx, exponent_of(v[i], w[i]));
  }
  mx = group_max<256>(mx);
  const bool bad = mx == kOzBadRow;
  const int e = bad || mx == kOzZero ? 0 : mx;
  if (threadIdx.x == 0) exps[r] = bad ? kOzBadRow : e;
  for (int64_t k0 = threadIdx.x * 8; k0 < ldk; k0 += 256 * 8) {
    long long x[8];
    float v[8], y[8];
    load8(row, k0, cols, true, v);
    load8(yrow, k0, cols, true, y);
    weights8(scale + k0, -1, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      long long mant;
      int exp2;
      bool neg;
      decompose(v[i], mant, exp2, neg);
      x[i] = bad ? 0 : fixed_rne(mant, exp2 + w[i], neg, 15 - e);
      v[i] = scaled((int)x[i], e - 15 - w[i]);
    }
    write_digits8(x, 2, planes + r * ldk + k0, rows_pad * ldk);
    if (r < n) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (k0 + i < n) X[r * ldx + k0 + i] = (double)y[i] + (double)v[i];
    }
  }
}

// One level's drain by an epilogue warp: read its 16 accumulator columns (exact integers below
// 2^24), hand the buffer back to the MMA issuer, and add the values into the 64-bit fixed-point
// sums: all levels in units of level LV-1 (lo), or where that needs more than 64 bits (WIDE) levels 0-2
// in units of level 2 (hi) and the others in lo.
template <int L, int LV, bool WIDE>
__device__ __forceinline__ void oz_drain(uint32_t taddr, uint32_t dbar, int lane, long long (&hi)[WIDE ? 16 : 1],
                                         long long (&lo)[16]) {
  if constexpr (L < LV) {
    uint32_t r[16];
    tmem_ld16(taddr, r);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(dbar) : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const long long v = (long long)__float2int_rn(__uint_as_float(r[j]));
      if constexpr (WIDE && L < 3)
        hi[j] += v << (8 * (2 - L));
      else
        lo[j] += v << (8 * (LV - 1 - L));
    }
  }
}

// The MMAs of one step t with r = t mod CKS.  Level l's exact chunks are staggered by l steps
// and chunk k of level l accumulates in TMEM buffer (l + k) mod NB, so at this step level l sits
// in buffer (l + [l >= CKS - r] + cm) mod NB, cm = (t / CKS) mod NB.  PAT is what that depends on: the level
// CKS - r that starts a chunk here (all above it have moved on), 0 for r = 0, LV where none does.  Per A
// slice pa, its partner levels pa .. LV-1 go in runs of up to four levels, split at the level that has
// moved on (so the runs and all shared-memory offsets are compile-time): one MMA with
// N = 64 x run takes the adjacent B slices pb .. pb+run-1 into the run's adjacent accumulators; a
// run whose buffers pass the last one (known from cm at run time) is issued as two MMAs.  The level
// that starts a chunk at this step gets its own MMA at pa = 0, the chunk's first, which
// overwrites the accumulator instead of adding to it (at the first step every level starts, and
// all of pa = 0's MMAs overwrite).  `pre` runs after the MMAs of the first A slices, about half
// of the step's work.
template <int LV, int LA, int BK, int PAT, typename Pre>
__device__ __forceinline__ void oz_issue_step(bool leader, uint32_t tmem, uint64_t adesc0, uint64_t bdesc0, int cm,
                                               bool first_step, Pre&& pre) {
  using C = OzCfg<LV, LA, BK>;
  constexpr int MOVED = PAT == 0 ? LV : PAT;      // levels from here on have moved on
#pragma unroll
  for (int sub = 0; sub < C::SK; ++sub) {
    // the next 32 bytes of every swizzled row (start address in 16-byte units)
    const uint64_t as = adesc0 + (uint64_t)(2 * sub), bs = bdesc0 + (uint64_t)(2 * sub);
    const int LS = sub == 0 ? PAT : LV;           // the level that starts a chunk (LV: none)
#pragma unroll
    for (int pa = 0; pa < LA; ++pa) {
      if (C::SK == 1 ? pa == (LA >= 5 ? 2 : 1) : (sub == C::SK - 1 && pa == 0)) pre();
      int l0 = pa;
#pragma unroll
      for (int l = pa + 1; l <= LV; ++l) {
        if (l == LV || l - l0 == 4 || l == MOVED || (pa == 0 && LS < LV && l == LS + 1)) {
          const int run = l - l0;
          const uint32_t acc = (pa == 0 && sub == 0 && (first_step || l0 == LS)) ? 0u : 1u;
          int b = l0 + (l0 >= MOVED ? 1 : 0) + cm;
          if (b >= C::NB) b -= C::NB;
          const int first = min(run, C::NB - b);
          // the start-address field (bits 0-13, 16-byte units) absorbs the in-stage offsets
          const uint64_t ad = as + (uint64_t)((pa * C::A_BYTES) >> 4);
          const uint64_t bd = bs + (uint64_t)(((l0 - pa) * C::B_BYTES) >> 4);
          if (leader) {
            mma_bf16(tmem + (uint32_t)(b * OZ_BN), ad, bd, C::IDESC_M | ((uint32_t)(first * OZ_BN) >> 3 << 17), acc);
            if (first < run)
              mma_bf16(tmem, ad, bd + (uint64_t)((first * C::B_BYTES) >> 4),
                       C::IDESC_M | ((uint32_t)((run - first) * OZ_BN) >> 3 << 17), acc);
          }
          l0 = l;
        }
      }
    }
  }
}

// The gate counter: the number of steps whose operands have landed and whose starting level's
// buffer has been drained (written by the gate warp with release, read by the MMA warp with acquire).
__device__ __forceinline__ uint32_t oz_gate_load(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void oz_gate_store(uint32_t addr, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Bounded wait until the gate passes step t; false on timeout or abort.
__device__ __forceinline__ bool oz_gate_wait(uint32_t addr, uint32_t t, volatile int* abort_flag, uint64_t limit_ns,
                                             uint32_t& gate) {
  gate = oz_gate_load(addr);
  if (gate > t) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    gate = oz_gate_load(addr);
    if (gate > t) return true;
    if (*abort_flag || globaltimer() - t0 > limit_ns) return false;
  }
}

template <int LV, int LA, bool WIDE, int BK>
__global__ void __launch_bounds__(OZ_THREADS, 1) oz_gemm_kernel(const __grid_constant__ OzMaps maps, const OzArgs a) {
  using C = OzCfg<LV, LA, BK>;
  extern __shared__ uint8_t smem_raw[];
  // grouped rasterisation: OZ_GROUP row tiles sweep the column tiles together
  const int tiles_m = (a.M + OZ_BM - 1) / OZ_BM, tiles_n = (a.N + OZ_BN - 1) / OZ_BN;
  const int per_group = OZ_GROUP * tiles_n;
  const int t = blockIdx.x, grp = t / per_group, first_m = grp * OZ_GROUP;
  const int gsize = min(tiles_m - first_m, OZ_GROUP);
  const int local = t - grp * per_group;
  const int m0 = (first_m + local % gsize) * OZ_BM, n0 = (local / gsize) * OZ_BN;
  if (a.e.sym && m0 + OZ_BM - 1 < n0) return;  // tile entirely above the diagonal
  // this CTA's k-slices: [kt0, kt0 + nk)
  const int kt0 = blockIdx.y * a.kt_per_split;
  const int nk = min(a.nk - kt0, a.kt_per_split);

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + C::STAGES * C::STAGE_BYTES;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (C::STAGES + s); };
  auto ready_bar = [&](int b) { return bars + 8u * (2 * C::STAGES + b); };          // buffer b holds a chunk
  auto drained_bar = [&](int b) { return bars + 8u * (2 * C::STAGES + C::NB + b); };  // buffer b is free
  const uint32_t done_bar = bars + 8u * (2 * C::STAGES + 2 * C::NB);
  uint32_t* tmem_slot =
      reinterpret_cast<uint32_t*>(gbase + C::STAGES * C::STAGE_BYTES + 8 * (2 * C::STAGES + 2 * C::NB + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* skip_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);
  const uint32_t gate_addr = smem_u32(tmem_slot + 3);  // steps released to the MMA warp
  volatile int never = 0;  // abort flag of the clean-up waits, which must not stop early

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < C::NB; ++b) {
      mbar_init(ready_bar(b), 1);
      mbar_init(drained_bar(b), OZ_EPI_WARPS);
    }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    *skip_flag = status_failed(a.e.status) ? 1 : 0;
    tmem_slot[3] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const bool skip = *skip_flag != 0 || nk <= 0;
  bool mma_issued = false;
  bool leader = false;  // the MMA warp's issuing lane: it issues every MMA and every commit

  if (skip) {
    // an earlier kernel failed: do nothing but release TMEM below
  } else if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    int last_round[8] = {-1, -1, -1, -1, -1, -1, -1, -1};
    for (int it = 0; it < nk; ++it) {
      const int s = it % C::STAGES;
      const uint32_t ph = (uint32_t)(it / C::STAGES) & 1u;
      if (!mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, a.wait_ns)) {
        *abort_flag = 1;
        status_set(a.e.status, KF_ERR_TIMEOUT, a.e.step, 11);
        break;
      }
      const uint32_t st = base + s * C::STAGE_BYTES;
      mbar_expect_tx(full_bar(s), C::STAGE_BYTES);
      const int x = (kt0 + it) * BK;
#pragma unroll
      for (int p = 0; p < LA; ++p) tma_load_2d(st + p * C::A_BYTES, &maps.a, x, p * a.a_rows_pad + m0, full_bar(s));
#pragma unroll
      for (int p = 0; p < LV; ++p)
        tma_load_2d(st + LA * C::A_BYTES + p * C::B_BYTES, &maps.b, x, p * a.b_rows_pad + n0, full_bar(s));
      last_round[s] = it / C::STAGES;
    }
    if (*abort_flag) {  // let issued copies land before the CTA's shared memory goes away
      for (int s = 0; s < C::STAGES; ++s)
        if (last_round[s] >= 0) mbar_wait(full_bar(s), (uint32_t)last_round[s] & 1u, &never);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the whole warp runs the loop, so the stage, buffer and descriptor
    // arithmetic is warp-uniform; one elected lane issues.  TMEM buffer b = columns [64 b, 64 b + 64).
    // The gate warp tells it which steps may start (operands landed, new buffer drained); the
    // MMA queue is shallow, so the issuer does no barrier test of its own between steps: it reads
    // the gate counter half-way through each step's MMAs, and that load's latency overlaps them.
    leader = elect_one();
    bool ok = true;
    uint32_t gate = 0;  // steps released so far (last value read)
    const int nks = nk * C::KS;
    int s = 0, t = 0, r = 0, cm = 0;  // stage, step, step in the chunk, chunk mod NB
    for (int it = 0; it < nk && ok; ++it) {
      const uint32_t st = base + s * C::STAGE_BYTES;
      const uint64_t adesc_s = smem_desc_sw(st, C::SBO, C::LAYOUT);
      const uint64_t bdesc_s = smem_desc_sw(st + LA * C::A_BYTES, C::SBO, C::LAYOUT);
#pragma unroll
      for (int j = 0; j < C::KS; ++j) {
        if (gate <= (uint32_t)t) {
          ok = __all_sync(0xffffffffu, oz_gate_wait(gate_addr, (uint32_t)t, abort_flag, a.wait_ns, gate));
          gate = __shfl_sync(0xffffffffu, gate, 0);
          if (!ok) {
            if (lane == 0 && !*abort_flag) {
              *abort_flag = 1;
              status_set(a.e.status, KF_ERR_TIMEOUT, a.e.step, 12);
            }
            break;
          }
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        auto buf = [&](int l) {  // buffer of level l at this step
          const int b = l + cm + (l >= C::CKS - r ? 1 : 0);
          return b >= C::NB ? b - C::NB : b;
        };
        uint32_t gate_ahead = gate;
        auto pre = [&]() { gate_ahead = oz_gate_load(gate_addr); };
        const uint64_t adesc0 = adesc_s + (uint64_t)(2 * j * C::SK), bdesc0 = bdesc_s + (uint64_t)(2 * j * C::SK);
        switch (r == 0 ? 0 : min(C::CKS - r, LV)) {
          case 0: oz_issue_step<LV, LA, BK, 0>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre); break;
          case 1: oz_issue_step<LV, LA, BK, 1>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre); break;
          case 2: oz_issue_step<LV, LA, BK, 2>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre); break;
          case 3: oz_issue_step<LV, LA, BK, 3>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre); break;
          case 4:
            if constexpr (LV > 4) oz_issue_step<LV, LA, BK, 4>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            else oz_issue_step<LV, LA, BK, LV>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            break;
          case 5:
            if constexpr (LV > 5) oz_issue_step<LV, LA, BK, 5>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            else oz_issue_step<LV, LA, BK, LV>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            break;
          case 6:
            if constexpr (LV > 6) oz_issue_step<LV, LA, BK, 6>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            else oz_issue_step<LV, LA, BK, LV>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre);
            break;
          default: oz_issue_step<LV, LA, BK, LV>(leader, tmem, adesc0, bdesc0, cm, t == 0, pre); break;
        }
        __syncwarp();
        mma_issued = true;
        if (leader) {  // the level whose chunk ends here (every level at the last step) is ready
          if (t == nks - 1) {
#pragma unroll
            for (int l = 0; l < LV; ++l) mma_commit(ready_bar(buf(l)));
          } else if (C::CKS - 1 - r < LV) {
            mma_commit(ready_bar(buf(C::CKS - 1 - r)));
          }
        }
        gate = __shfl_sync(0xffffffffu, max(gate, gate_ahead), 0);
        ++t;
        if (++r == C::CKS) {
          r = 0;
          if (++cm == C::NB) cm = 0;
        }
      }
      if (!ok) break;
      if (leader) mma_commit(empty_bar(s));
      __syncwarp();
      if (++s == C::STAGES) s = 0;
    }
  } else if (warp == OZ_GATE_WARP) {
    // ---------------- gate: per step, wait (bounded) for its stage's operands (at the stage's
    // first step) and, when a level starts a chunk there in a buffer used before, for that
    // buffer's drain; then release the step to the MMA warp.  Level l's exact chunks are
    // staggered by l steps (chunk k covers steps [k CKS - l, (k + 1) CKS - l)), so at most one
    // level starts a chunk per step, and chunk k of level l accumulates in buffer (l + k) mod NB.
    // That buffer last held chunk k - 1 of level l + 1, which ended two steps earlier: its drain
    // has a full step of MMAs to finish.
    uint32_t used = 0, par = 0;  // per buffer: used before; parity of its uses so far
    const int nks = nk * C::KS;
    for (int t = 0; t < nks; ++t) {
      const int it = t / C::KS;
      if (t == it * C::KS) {
        const int s = it % C::STAGES;
        const uint32_t ph = (uint32_t)(it / C::STAGES) & 1u;
        if (!__all_sync(0xffffffffu, mbar_wait(full_bar(s), ph, abort_flag, a.wait_ns))) {
          if (lane == 0 && !*abort_flag) {
            *abort_flag = 1;
            status_set(a.e.status, KF_ERR_TIMEOUT, a.e.step, 15);
          }
          break;
        }
      }
      const int ck = t / C::CKS, r = t - ck * C::CKS, cm = ck % C::NB;
      if (t == 0) {
        used = par = (1u << LV) - 1u;
      } else {
        const int ls = r == 0 ? 0 : C::CKS - r;
        if (ls < LV) {
          int b = ls + cm + 1;  // the starting level has moved on: (ls + (t + ls) / CKS) mod NB
          if (r == 0) b = cm;
          if (b >= C::NB) b -= C::NB;
          if ((used >> b) & 1u) {
            if (!__all_sync(0xffffffffu, mbar_wait(drained_bar(b), ((par >> b) & 1u) ^ 1u, abort_flag, a.wait_ns))) {
              if (lane == 0 && !*abort_flag) {
                *abort_flag = 1;
                status_set(a.e.status, KF_ERR_TIMEOUT, a.e.step, 13);
              }
              break;
            }
          }
          used |= 1u << b;
          par ^= 1u << b;
        }
      }
      __syncwarp();
      if (lane == 0) oz_gate_store(gate_addr, (uint32_t)(t + 1));
    }
  } else if (warp >= OZ_EPI0) {
    // ---------------- epilogue: exact level sums into 64-bit fixed point, then scale and store
    const int q = warp % 4, h = (warp - OZ_EPI0) / 4;  // TMEM lane quadrant (fixed by the warp index), column quarter
    const int gi = m0 + 32 * q + lane;
    long long hi[WIDE ? 16 : 1], lo[16];  // the element's fixed-point sums (oz_drain)
#pragma unroll
    for (int j = 0; j < 16; ++j) lo[j] = 0;
#pragma unroll
    for (int j = 0; j < (WIDE ? 16 : 1); ++j) hi[j] = 0;
    bool ok = true;
    // drain events in the MMA issuer's order: at step t, the level whose staggered chunk ends
    // there; at the last step, every level
    uint32_t rpar = 0;  // per buffer: parity of its drains so far
    const int nks = nk * C::KS;
    for (int t = 0; t < nks && ok; ++t) {
      const bool final_step = t == nks - 1;
      const int lone = (C::CKS - 1 - t % C::CKS);  // the level whose chunk ends at step t
      for (int l = final_step ? 0 : lone; l < (final_step ? LV : min(lone + 1, LV)); ++l) {
        const int b = (l + (t + l) / C::CKS) % C::NB;
        const uint32_t ph = (rpar >> b) & 1u;
        rpar ^= 1u << b;
        if (!mbar_wait(ready_bar(b), ph, abort_flag, a.wait_ns)) {
          if (!*abort_flag) {
            *abort_flag = 1;
            status_set(a.e.status, KF_ERR_TIMEOUT, a.e.step, 14);
          }
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * OZ_BN + h * 16);
        const uint32_t dbar = drained_bar(b);
        // compile-time level, so the shifts are constants and the conversions 32-bit
        switch (l) {
          case 0: oz_drain<0, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 1: oz_drain<1, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 2: oz_drain<2, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 3: oz_drain<3, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 4: oz_drain<4, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 5: oz_drain<5, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          case 6: oz_drain<6, LV, WIDE>(taddr, dbar, lane, hi, lo); break;
          default: break;
        }
      }
    }
    // Stage the tile's integer sums in shared memory (the operand stages are idle once the last chunk has
    // been drained), then sweep it by rows for the direct outputs (lane -> column, so every warp access is
    // contiguous) and by columns for the mirrored and transposed outputs.  The scaling to float64 is done in
    // the row sweep's loop: a CTA runs this once, so unrolled code would mostly wait for its instructions
    // (per-thread unrolled scaling and batched rows took 30 k cycles per tile, this loop about a third).
    // A slot of the first plane holds the sum, and after the row sweep the value.
    constexpr int PITCH = OZ_BN + 1;  // odd pitch: row and column sweeps are both conflict-free
    constexpr int SH = 8 * (LV - 3);  // unit of hi over the unit of lo
    static_assert((size_t)OZ_BM * PITCH * (WIDE ? 2 : 1) * sizeof(double) <= (size_t)C::STAGES * C::STAGE_BYTES, "tile fits");
    long long* tile1 = reinterpret_cast<long long*>(gbase);
    constexpr int PLANE = OZ_BM * PITCH;  // wide sums: lo in the first plane, hi in the second
    if (a.sums) {
      if (ok && gi < a.M) {  // columns padded to 64
        longlong2* dst = reinterpret_cast<longlong2*>(a.sums + ((int64_t)blockIdx.y * a.M + gi) * a.ld_sums + n0 + h * 16);
#pragma unroll
        for (int j = 0; j < 16; j += 2)
          dst[j / 2] = make_longlong2(lo[j], lo[j + 1]);
      }
    } else if (ok) {
      const int slot = (32 * q + lane) * PITCH + h * 16;
#pragma unroll
      for (int j = 0; j < 16; ++j) tile1[slot + j] = lo[j];
      if constexpr (WIDE) {
#pragma unroll
        for (int j = 0; j < 16; ++j) tile1[PLANE + slot + j] = hi[j];
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * OZ_EPI_WARPS) : "memory");
    const bool go = !*abort_flag && !a.sums;
    const int ew = warp - OZ_EPI0;  // epilogue warp 0..15
    const OzEpilogue& e = a.e;
    double* part = a.partials ? a.partials + (int64_t)blockIdx.y * a.M * a.N : nullptr;
    auto value_slot = [&](int r, int c) { return reinterpret_cast<double*>(tile1) + r * PITCH + c; };
    // One row per warp and turn, two columns per lane.  A sweep is bound by its instructions, and one loop
    // for every kind of output takes twice the time of a loop for the kind at hand, so the usual kinds have
    // their own loop for the tiles that hold no diagonal element; the others take the general one.
    const bool crosses = n0 < m0 + OZ_BM && n0 + OZ_BN > m0;
    const bool fast = e.simple == 2 || (e.simple == 1 && !crosses);
    constexpr int NR = OZ_BM / OZ_EPI_WARPS;  // rows per warp
    constexpr int SC = -14 - 8 * (LV - 1);
    const int gj0 = n0 + lane, gj1 = gj0 + 32;
    const bool in0 = gj0 < a.N, in1 = gj1 < a.N;
    const int ej0 = go && in0 ? a.eb[gj0] : 0, ej1 = go && in1 ? a.eb[gj1] : 0;
    const int my_row = m0 + ew + OZ_EPI_WARPS * lane;
    const int ei_all = go && lane < NR && my_row < a.M ? a.ea[my_row] : 0;
    const bool any_bad = __any_sync(0xffffffffu, ej0 == kOzBadRow || ej1 == kOzBadRow || ei_all == kOzBadRow);
    const bool columns = !part && (e.sym || e.outT);  // the column sweep wants the values
    auto product = [&](int r, int ei, double& v0, double& v1) {
      if constexpr (WIDE) {
        const long long* t = tile1 + r * PITCH + lane;
        v0 = fixed_to_double(t[PLANE], t[0], SH, ei + SC + ej0);
        v1 = fixed_to_double(t[PLANE + 32], t[32], SH, ei + SC + ej1);
      } else {
        v0 = fixed_to_double(tile1[r * PITCH + lane], ei + SC + ej0);
        v1 = fixed_to_double(tile1[r * PITCH + lane + 32], ei + SC + ej1);
      }
      if (any_bad) {  // a non-finite operand row
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        if (ei == kOzBadRow || ej0 == kOzBadRow) v0 = nan;
        if (ei == kOzBadRow || ej1 == kOzBadRow) v1 = nan;
      }
    };
    auto fast_sweep = [&](auto with_cin, auto with_f32) {
      constexpr bool CIN = decltype(with_cin)::value, F32 = decltype(with_f32)::value;
      const int64_t first = m0 + ew;
      // every row's cin before the first store (cin may be the output array)
      double cb[CIN ? NR : 1][2];
      if constexpr (CIN) {
        const double* pc = e.cin + first * e.ldcin + gj0;
        const int64_t step = OZ_EPI_WARPS * e.ldcin;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          const bool row = m0 + ew + OZ_EPI_WARPS * k < a.M;
          cb[k][0] = row && in0 ? pc[0] : 0.0;
          cb[k][1] = row && in1 ? pc[32] : 0.0;
          pc += step;
        }
      }
      const int64_t ld = part ? (int64_t)a.N : e.out ? e.ldo : e.ldo2;
      double* po = (part ? part : e.out ? e.out : e.out2) + first * ld + gj0;
      const int64_t so = OZ_EPI_WARPS * ld, sf = OZ_EPI_WARPS * e.ldof;
      float* pf = F32 ? e.outf + first * e.ldof + gj0 : nullptr;
      const unsigned long long flip = !part && e.alpha_unit < 0 ? 1ull << 63 : 0ull;
#pragma unroll 1
      for (int k = 0; k < NR; ++k) {
        const int r = ew + OZ_EPI_WARPS * k;
        if (m0 + r >= a.M) break;
        double v0, v1;
        product(r, __shfl_sync(0xffffffffu, ei_all, k), v0, v1);
        v0 = __longlong_as_double(__double_as_longlong(v0) ^ flip);
        v1 = __longlong_as_double(__double_as_longlong(v1) ^ flip);
        if constexpr (CIN) {
          v0 = cb[0][0] + v0;
          v1 = cb[0][1] + v1;
#pragma unroll
          for (int j = 0; j + 1 < NR; ++j) {
            cb[j][0] = cb[j + 1][0];
            cb[j][1] = cb[j + 1][1];
          }
        }
        if (in0) po[0] = v0;
        if (in1) po[32] = v1;
        po += so;
        if constexpr (F32) {
          if (in0) pf[0] = narrow(v0);
          if (in1) pf[32] = narrow(v1);
          pf += sf;
        }
        if (columns) {
          *value_slot(r, lane) = v0;
          *value_slot(r, lane + 32) = v1;
        }
      }
    };
    auto general_sweep = [&]() {
#pragma unroll 1
      for (int k = 0; k < NR; ++k) {
        const int r = ew + OZ_EPI_WARPS * k, gi2 = m0 + r;
        if (gi2 >= a.M) break;
        double v0, v1;
        product(r, __shfl_sync(0xffffffffu, ei_all, k), v0, v1);
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
          const int gj = u ? gj1 : gj0;
          double v = u ? v1 : v0;
          if (gj >= a.N || (e.sym && gj > gi2)) continue;
          if (part) {
            part[(int64_t)gi2 * a.N + gj] = v;
            continue;
          }
          v = e.cin ? oz_axpby<true>(e, v, e.cin[(int64_t)gi2 * e.ldcin + gj]) : oz_axpby<false>(e, v, 0.0);
          if (gi2 == gj) v += e.delta;
          v = oz_addq(v, e.radd_kind, e.radd, e.ldradd, gi2, gj);
          if (e.out) e.out[(int64_t)gi2 * e.ldo + gj] = v;
          if (e.outf) e.outf[(int64_t)gi2 * e.ldof + gj] = narrow(v);
          if (e.out2) e.out2[(int64_t)gi2 * e.ldo2 + gj] = oz_addq(v, e.q_kind, e.q, e.ldq, gi2, gj);
          if (gi2 == gj) {
            if (e.diag_out) e.diag_out[gi2] = v;
            if (e.check_diag && !(v > 0.0 && isfinite(v))) status_set(e.status, KF_ERR_NUMERIC, e.step, gi2);
          }
          *value_slot(r, lane + 32 * u) = v;
        }
      }
    };
    if (go) {
      if (part || (fast && !e.cin)) {
        fast_sweep(std::false_type{}, std::false_type{});
      } else if (!WIDE && fast) {  // the wide sums leave no registers for a batch of cin
        if constexpr (!WIDE) {
          if (e.outf)
            fast_sweep(std::true_type{}, std::true_type{});
          else
            fast_sweep(std::true_type{}, std::false_type{});
        }
      } else {
        general_sweep();
      }
    }
    if (columns && !a.sums) {
      asm volatile("bar.sync 1, %0;" ::"n"(32 * OZ_EPI_WARPS) : "memory");
      const int rows = min(OZ_BM, a.M - m0);
      // columns (gj, gi) of the mirrored and transposed outputs: consecutive lanes write consecutive places
      auto fast_columns = [&](double* dst, int64_t ld, float* dstf) {
        dst += (int64_t)(n0 + ew) * ld + m0 + lane;
        const int64_t sd = OZ_EPI_WARPS * ld, sf = OZ_EPI_WARPS * e.ldof;
        if (dstf) dstf += (int64_t)(n0 + ew) * e.ldof + m0 + lane;
#pragma unroll 1
        for (int c = ew; c < OZ_BN && n0 + c < a.N; c += OZ_EPI_WARPS) {
          double v[OZ_BM / 32];
#pragma unroll
          for (int k = 0; k < OZ_BM / 32; ++k) v[k] = *value_slot(lane + 32 * k, c);
#pragma unroll
          for (int k = 0; k < OZ_BM / 32; ++k)
            if (lane + 32 * k < rows) dst[32 * k] = v[k];
          dst += sd;
          if (dstf) {
#pragma unroll
            for (int k = 0; k < OZ_BM / 32; ++k)
              if (lane + 32 * k < rows) dstf[32 * k] = narrow(v[k]);
            dstf += sf;
          }
        }
      };
      if (go && fast && e.outT) {
        fast_columns(e.outT, e.ldoT, nullptr);
      } else if (go && fast) {
        fast_columns(e.out ? e.out : e.out2, e.out ? e.ldo : e.ldo2, e.outf);
      } else if (go) {
#pragma unroll 1
        for (int c = ew; c < OZ_BN; c += OZ_EPI_WARPS) {
          const int gj = n0 + c;
          if (gj >= a.N) break;
#pragma unroll 1
          for (int r = lane; r < rows; r += 32) {
            const int gi2 = m0 + r;
            if (e.sym && gj > gi2) continue;
            const double v = *value_slot(r, c);
            if (e.outT) e.outT[(int64_t)gj * e.ldoT + gi2] = v;
            if (e.sym && gi2 != gj) {  // mirror (gj, gi2)
              if (e.out) e.out[(int64_t)gj * e.ldo + gi2] = v;
              if (e.outf) e.outf[(int64_t)gj * e.ldof + gi2] = narrow(v);
              if (e.out2) e.out2[(int64_t)gj * e.ldo2 + gi2] = oz_addq(v, e.q_kind, e.q, e.ldq, gj, gi2);
            }
          }
        }
      }
    }
  }
  // every issued MMA must have finished before TMEM is freed
  if (!skip && warp == 1 && leader && mma_issued) {
    mma_commit(done_bar);
    mbar_wait(done_bar, 0, &never);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// Sum of the split-K partials in split order, then the epilogue (one thread per element).
__global__ void oz_reduce_kernel(int M, int N, int splits, const double* partials, OzEpilogue e) {
  if (status_failed(e.status)) return;
  const int64_t total = (int64_t)M * N;
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < total; u += (int64_t)gridDim.x * blockDim.x) {
    const int gi = (int)(u / N), gj = (int)(u % N);
    if (e.sym && gj > gi) continue;
    double c = 0.0;
    for (int sp = 0; sp < splits; ++sp) c += partials[(int64_t)sp * total + u];
    oz_apply(e, gi, gj, c);
  }
}

// Exact splits: integer sums of one 32 x 32 tile over the splits, scaled once, so the result is the one an
// unsplit product gives; out along rows, outT along columns through shared memory.
__global__ void __launch_bounds__(256) oz_sums_reduce_kernel(int M, int N, int splits, const long long* sums, int64_t ld,
                                                             const int* ea, const int* eb, int scale, OzEpilogue e) {
  __shared__ double tile[32][33];
  __shared__ int skip;
  if (threadIdx.x == 0) skip = status_failed(e.status) ? 1 : 0;
  __syncthreads();
  if (skip) return;
  const int m0 = blockIdx.y * 32, n0 = blockIdx.x * 32, lane = threadIdx.x % 32, w = threadIdx.x / 32;
  long long t[4] = {0, 0, 0, 0};
  for (int sp = 0; sp < splits; ++sp) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int gi = m0 + w + 8 * k;
      if (gi < M) t[k] += sums[((int64_t)sp * M + gi) * ld + n0 + lane];
    }
  }
  const int gj = n0 + lane;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int gi = m0 + w + 8 * k;
    if (gi >= M || gj >= N) continue;
    const int ei = ea[gi], ej = eb[gj];
    const double c = (ei == kOzBadRow || ej == kOzBadRow) ? __longlong_as_double(0x7ff8000000000000ll)
                                                          : fixed_to_double(t[k], ei + ej + scale);
    const double v = e.cin ? oz_axpby<true>(e, c, e.cin[(int64_t)gi * e.ldcin + gj]) : oz_axpby<false>(e, c, 0.0);
    if (e.out) e.out[(int64_t)gi * e.ldo + gj] = v;
    tile[w + 8 * k][lane] = v;
  }
  if (!e.outT) return;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int gjt = n0 + w + 8 * k, gi = m0 + lane;
    if (gjt < N && gi < M) e.outT[(int64_t)gjt * e.ldoT + gi] = tile[lane][w + 8 * k];
  }
}

template <int LV, int LA, bool WIDE, int BK>
kf_status launch_oz(cudaStream_t s, const OzSlices& A, const OzSlices& B, int M, int N, int K, const OzEpilogue& e,
                    int splits, double* partials, long long* sums) {
  using C = OzCfg<LV, LA, BK>;
  OzMaps maps;
  KF_TRY(tma_map_bf16(&maps.a, A.planes, (int64_t)A.S * A.rows_pad, A.ldk, A.ldk, BK, OZ_BM, C::SWZ));
  KF_TRY(tma_map_bf16(&maps.b, B.planes, (int64_t)B.S * B.rows_pad, B.ldk, B.ldk, BK, OZ_BN, C::SWZ));
  OzArgs a;
  a.M = M;
  a.N = N;
  a.nk = (int)ceil_div(K, BK);
  a.kt_per_split = (int)(ceil_div(ceil_div(K, OZ_SPLIT_K), splits) * (OZ_SPLIT_K / BK));
  a.partials = splits > 1 && !sums ? partials : nullptr;
  a.sums = sums;
  a.ld_sums = round_up(N, OZ_BN);
  a.a_rows_pad = (int)A.rows_pad;
  a.b_rows_pad = (int)B.rows_pad;
  a.ea = A.exps;
  a.eb = B.exps;
  a.e = e;
  a.e.alpha_unit = e.alpha == 1.0 ? 1 : e.alpha == -1.0 ? -1 : 0;
  a.e.beta_unit = e.beta == 1.0;
  // one float64 output (plus a float32 copy with cin, or its transpose), unit alpha and beta, diagonal R and Q
  const bool plain = a.e.alpha_unit != 0 && (!e.cin || a.e.beta_unit) && e.radd_kind != 2 && e.q_kind != 2 &&
                     (e.out != nullptr) != (e.out2 != nullptr) && (!e.outf || e.cin) && !(e.sym && e.outT);
  const bool no_diagonal = !e.sym && e.delta == 0.0 && e.radd_kind < 0 && e.q_kind < 0 && !e.diag_out;
  a.e.simple = !plain ? 0 : no_diagonal ? 2 : 1;
  a.wait_ns = g_tc_wait_ns.load();
  KF_CUDA_TRY(smem_limit_per_device((const void*)oz_gemm_kernel<LV, LA, WIDE, BK>, (int)C::SMEM));
  const int64_t tiles = ceil_div(M, OZ_BM) * ceil_div(N, OZ_BN);
  if (g_oz_timer) g_oz_timer->before(s);
  oz_gemm_kernel<LV, LA, WIDE, BK><<<dim3((unsigned)tiles, (unsigned)splits), OZ_THREADS, C::SMEM, s>>>(maps, a);
  if (g_oz_timer) g_oz_timer->after(s);
  note_launch();
  KF_TRY(launch_check("oz_gemm"));
  if (sums) {
    oz_sums_reduce_kernel<<<dim3((unsigned)ceil_div(N, 32), (unsigned)ceil_div(M, 32)), 256, 0, s>>>(
        M, N, splits, sums, a.ld_sums, A.exps, B.exps, -14 - 8 * (LV - 1), a.e);
    note_launch();
    return launch_check("oz_sums_reduce");
  }
  if (splits > 1) {
    const int64_t total = (int64_t)M * N;
    oz_reduce_kernel<<<(unsigned)std::min<int64_t>(ceil_div(total, 256), 4096), 256, 0, s>>>(M, N, splits, partials, e);
    note_launch();
    KF_TRY(launch_check("oz_reduce"));
  }
  return KF_OK;
}

// One warp per row up to 512 columns (a block's threads would mostly idle), a block per row with the row in
// registers up to 10240, two passes beyond.
template <typename T, bool WEIGH>
void slice_rows(cudaStream_t s, const T* X, int64_t ld, int64_t rows, int64_t cols, int S, const OzSlices& out,
                const int* scale = nullptr, int sign = 0) {
  const unsigned blocks = (unsigned)out.rows_pad;
#define OZ_SLICE(G, NCH)                                                                                              \
  oz_slice_kernel<T, G, NCH, WEIGH><<<blocks / (256 / G), 256, 0, s>>>(X, ld, rows, cols, S, out.planes, out.rows_pad, \
                                                                       out.ldk, out.exps, scale, sign)
  if (out.ldk <= 256)
    OZ_SLICE(32, 1);
  else if (out.ldk <= 512)
    OZ_SLICE(32, 2);
  else if (out.ldk <= 2048)
    OZ_SLICE(256, 1);
  else if (out.ldk <= 4096)
    OZ_SLICE(256, 2);
  else if (out.ldk <= 6144)
    OZ_SLICE(256, 3);
  else if (out.ldk <= 10240)
    OZ_SLICE(256, 5);
  else
    OZ_SLICE(256, 0);
#undef OZ_SLICE
}

}  // namespace

thread_local TcLaunchTimer* g_oz_timer = nullptr;

// Splits of K that give every SM a CTA when the output has too few tiles (U^T = P H^T at N = 1664, m = 128:
// 26 tiles; 74 us as one pass over K, 25 us in five splits and 7 us for their sum).  At least two chunks per
// split: its fixed part (pipeline fill, drain, epilogue, the sum) is worth about three.
int64_t oz_sums_splits(int64_t M, int64_t N, int64_t K) {
  const int64_t tiles = ceil_div(M, OZ_BM) * ceil_div(N, OZ_BN), chunks = ceil_div(K, OZ_SPLIT_K);
  if (tiles >= 152 || chunks < 4) return 1;
  const int64_t s = std::min<int64_t>(std::min<int64_t>(152 / tiles, chunks / 2), 16);
  if (s < 2) return 1;
  return ceil_div(chunks, ceil_div(chunks, s));
}

uint64_t oz_slice_bytes(int64_t rows, int64_t cols, int S) {
  const uint64_t rp = round_up(std::max<int64_t>(rows, 1), OZ_ROW_PAD), ldk = round_up(std::max<int64_t>(cols, 1), 64);
  return round_up((int64_t)(S * rp * ldk * 2), 256) + rp * 4;
}

void oz_slice_layout(OzSlices& out, void* mem, int64_t rows, int64_t cols, int S) {
  out.rows = rows;
  out.rows_pad = round_up(std::max<int64_t>(rows, 1), OZ_ROW_PAD);
  out.ldk = round_up(std::max<int64_t>(cols, 1), 64);
  out.S = S;
  out.planes = static_cast<__nv_bfloat16*>(mem);
  out.exps = reinterpret_cast<int*>(static_cast<char*>(mem) + round_up((int64_t)(S * out.rows_pad * out.ldk * 2), 256));
}

kf_status oz_slice(cudaStream_t s, const void* X, int64_t ld, int f64, int64_t rows, int64_t cols, int S,
                   OzSlices& out) {
  if (rows < 1 || cols < 1 || S < 1 || S > out.S || rows > out.rows_pad || cols > out.ldk || ld < cols || !X)
    return KF_ERR_ARG;
  out.rows = rows;
  out.filled = S;
  if (f64)
    slice_rows<double, false>(s, static_cast<const double*>(X), ld, rows, cols, S, out);
  else
    slice_rows<float, false>(s, static_cast<const float*>(X), ld, rows, cols, S, out);
  note_launch();
  return launch_check("oz_slice");
}

kf_status oz_balance(cudaStream_t s, const void* P, int64_t ld, int f64, int64_t n, int64_t ldk, int* scale) {
  if (n < 1 || ld < n || ldk < n || !P || !scale) return KF_ERR_ARG;
  oz_balance_kernel<<<(unsigned)std::min<int64_t>(ceil_div(ldk, 64), 1024), 64, 0, s>>>(P, f64, ld, n, ldk, scale);
  note_launch();
  return launch_check("oz_balance");
}

kf_status oz_slice_weighed(cudaStream_t s, const void* X, int64_t ld, int f64, int64_t n, const int* scale, int sign, int S,
                           OzSlices& out) {
  if (n < 1 || S < 1 || S > out.S || n > out.rows_pad || n > out.ldk || ld < n || !X || !scale ||
      (reinterpret_cast<uintptr_t>(scale) & 15))
    return KF_ERR_ARG;
  out.rows = n;
  out.filled = S;
  if (f64)
    slice_rows<double, true>(s, static_cast<const double*>(X), ld, n, n, S, out, scale, sign);
  else
    slice_rows<float, true>(s, static_cast<const float*>(X), ld, n, n, S, out, scale, sign);
  note_launch();
  return launch_check("oz_slice_weighed");
}

kf_status oz_slice_symmetric(cudaStream_t s, float* X, int64_t ld, int64_t n, const int* scale, OzSlices& out) {
  if (n < 1 || out.S < 3 || n > out.rows_pad || n > out.ldk || ld < n || ld % 4 || (reinterpret_cast<uintptr_t>(X) & 15) ||
      !scale)
    return KF_ERR_ARG;
  out.rows = n;
  out.filled = 3;
  oz_exps_kernel<<<(unsigned)out.rows_pad, 256, 0, s>>>(X, ld, n, out.ldk, scale, out.exps);
  note_launch();
  KF_TRY(launch_check("oz_exps"));
  oz_slice_symmetric_kernel<<<(unsigned)out.rows_pad, 256, 0, s>>>(X, ld, n, scale, out.planes, out.rows_pad, out.ldk,
                                                                   out.exps);
  note_launch();
  return launch_check("oz_slice_symmetric");
}

kf_status oz_slice_correction(cudaStream_t s, const float* C, const float* Y, int64_t ld, int64_t n, const int* scale,
                              double* X, int64_t ldx, OzSlices& out) {
  if (n < 1 || out.S < 2 || n > out.rows_pad || n > out.ldk || ld < n || ldx < n || ld % 4 ||
      (reinterpret_cast<uintptr_t>(C) & 15) || (reinterpret_cast<uintptr_t>(Y) & 15) || !scale)
    return KF_ERR_ARG;
  out.rows = n;
  out.filled = 2;
  oz_slice_correction_kernel<<<(unsigned)out.rows_pad, 256, 0, s>>>(C, Y, ld, n, scale, out.planes, out.rows_pad, out.ldk,
                                                                    out.exps, X, ldx);
  note_launch();
  return launch_check("oz_slice_correction");
}

kf_status oz_gemm(cudaStream_t s, const OzSlices& A, const OzSlices& B, int M, int N, int K, int levels,
                  const OzEpilogue& e, int splits, double* partials, const OzSums& work, int a_slices) {
  const int la = a_slices > 0 ? a_slices : levels;
  if (M <= 0 || N <= 0) return KF_OK;
  if (K < 1 || K > (1 << 20)) return KF_ERR_ARG;
  if (!e.out && !e.outf && !e.outT && !e.out2 && !e.diag_out) return KF_ERR_ARG;
  if (M > A.rows || N > B.rows || K > A.ldk || K > B.ldk) return KF_ERR_ARG;
  if (A.filled < la || B.filled < levels || (e.sym && M != N)) return KF_ERR_ARG;
  if (splits < 1 || splits > 64 || (splits > 1 && !partials)) return KF_ERR_ARG;
  long long* sums = nullptr;
  if (splits == 1 && levels == 5 && work.p && K <= kOzSumsMaxK && !e.sym && !e.outf && !e.out2 && !e.diag_out &&
      e.radd_kind < 0 && e.delta == 0.0) {
    const int64_t want = oz_sums_splits(M, N, K);
    if (want > 1 && want * M * round_up(N, OZ_BN) <= work.count) {
      splits = (int)want;
      sums = work.p;
    }
  }
  // whole multiples of OZ_SPLIT_K per split, every split non-empty
  const int64_t chunks = ceil_div(K, OZ_SPLIT_K);
  splits = (int)std::min<int64_t>(splits, chunks);
  splits = (int)ceil_div(chunks, ceil_div(chunks, splits));
  // the sums of all levels fit 64 bits up to K 2^(8 LV + 6.1) < 2^62
  const bool narrow_sums = levels < 5 || (levels == 5 && K <= kOzSumsMaxK);
  switch (levels * 16 + la) {
    case 4 * 16 + 4: return launch_oz<4, 4, false, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
    case 5 * 16 + 5:
      return narrow_sums ? launch_oz<5, 5, false, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums)
                         : launch_oz<5, 5, true, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
    case 6 * 16 + 6: return launch_oz<6, 6, true, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
    case 7 * 16 + 7: return launch_oz<7, 7, true, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
    case 7 * 16 + 3: return launch_oz<7, 3, true, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
    case 5 * 16 + 2:
      return narrow_sums ? launch_oz<5, 2, false, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums)
                         : launch_oz<5, 2, true, kOzBK>(s, A, B, M, N, K, e, splits, partials, sums);
  }
  return KF_ERR_ARG;
}

}  // namespace kfm
