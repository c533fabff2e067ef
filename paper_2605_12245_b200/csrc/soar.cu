// SOAR NVFP4 weight quantizer for NVIDIA B200 (sm_100a): kernels and the C ABI of soar.h.
//
// What runs on the device, in order (Algorithm 1 of the SOAR paper), as passes over W:
//   amax       tensor-wide max |W|, sum W^2 and a non-finite check               (Eq. 1)
//   init       max-based scales, first codes, first tensor sums                  (Eq. 1-2, Alg. 1 "Initialization")
//   iterate    T times: global scale (Eq. 5) from the previous pass's sums, block scale (Eq. 6), candidate search
//              (Eq. 8, App. B.3), winners stored, next sums accumulated
//   report     early-stop bookkeeping (Sec. 4.1), alpha and the report; a 128x4-tiled copy of the scales if asked for
//
// Launches.  A pass cannot begin before the sums of the one before are known to every CTA, so the passes of a call run in
// one persistent cooperative kernel whose CTAs meet between them: solo_kernel for one matrix, quantize_kernel for up to
// 16 matrices at once, whose tiles form one sequence walked by the whole grid, so that a model's many small matrices
// share passes; matrices that have stopped early drop out of later ones.  Small matrices run in one cluster, calls
// without iterations on large ones in two chained kernels (see solo_kernel.cuh).  A staged or traced call, and one whose grid
// the context has no room for (grid_refused), enqueues each stage as a launch of its own (the names in a trace are the
// stages').
//
// Data movement.  Every warp feeds itself with tiles of 32 blocks (1 KB of bf16), in registers or through its own slots
// of shared memory (see quantize_kernel.cuh).
//
// State between iterations is 8 bytes per block in the workspace or in shared memory: the winner's
// A = sum |W| m (binary32, exact), 4B = sum (2m)^2, its E4M3 scale code and the block maximum's exponent (pack_state).
// That is all Eq. 6 and the choice of the path need; the transient quantization scale of Sec. 3.3 is never stored.
//
// Arithmetic.  Whatever feeds a rounding decision is a fixed chain of IEEE binary32
// round-to-nearest operations (explicit __f*_rn intrinsics, never contracted); the E2M1
// rounding itself is the sm_100a conversion cvt.rn.satfinite.e2m1x2.f32 (nearest, ties to
// even, saturating, sign kept on zero).  Block sums A and B are integer dot products over
// 16-bit fixed-point magnitudes and the codes' byte values (dp2a / dp4a), exact whenever
// the block maximum times the reciprocal scale is at most 32; otherwise a binary64 path is
// taken.  Tensor sums and candidate comparisons are binary64.
//
// Column-weighted objective (Sec. 5 in diagonal form; soar_quantize_weighted): the same stages with passes of their own,
// whose block sums are binary64 (see weighted_kernel.cuh).
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <memory>
#include <mutex>
#include <new>
#include <numeric>
#include <random>
#include <vector>

#include "soar.h"

namespace {

constexpr size_t kWsFixedBytes = 2048;
constexpr unsigned int kGridWaitLimit = 1u << 21;  // polls of the grid's arrival counter before a CTA gives up (each most of a microsecond)
constexpr unsigned int kClusterWaitLimit = 1u << 24;  // polls of an mbarrier of its own shared memory (each some tens of nanoseconds)
// What soar_debug_fail_waits makes the CTAs of a launch withhold: their arrivals, what a cluster's CTAs send each other, either
// from the second meeting of a call on one matrix on; or it has one CTA say that its share of the error does not fit.
enum WaitHook : int { kNobodyArrives = 1, kNobodySends = 2, kNobodyMeetsAgain = 3, kShareBeyond = 4 };
constexpr int kBracketMinBeta = 2;             // the bracket needs two multipliers; a single one is modes 1-3

struct Ws {
  unsigned int amax_bits;            // max over the tensor of the bf16 magnitude bit pattern
  unsigned int error;                // kErr* bits; non-zero stops the remaining passes
  unsigned long long zero_blocks;
  unsigned long long wide;
  double sumsq;                      // sum W^2
  double num[SOAR_MAX_ITERS + 1];    // stage s: sum A_i * dd_i        (numerator of Eq. 5)
  double den[SOAR_MAX_ITERS + 1];    // stage s: sum B_i * dd_i^2      (denominator of Eq. 5)
  double gsum[SOAR_MAX_ITERS + 1];   // stage s: sum of block errors minus sum W^2 (Eq. 4)
};
static_assert(sizeof(Ws) <= kWsFixedBytes, "workspace header too large");
// the same layout is published as soar_workspace_header
static_assert(kWsFixedBytes == SOAR_WORKSPACE_HEADER_BYTES && sizeof(Ws) == sizeof(soar_workspace_header) &&
                  offsetof(Ws, amax_bits) == offsetof(soar_workspace_header, amax_bits) &&
                  offsetof(Ws, error) == offsetof(soar_workspace_header, error) &&
                  offsetof(Ws, zero_blocks) == offsetof(soar_workspace_header, zero_blocks) &&
                  offsetof(Ws, wide) == offsetof(soar_workspace_header, wide) &&
                  offsetof(Ws, sumsq) == offsetof(soar_workspace_header, sumsq) &&
                  offsetof(Ws, num) == offsetof(soar_workspace_header, num) &&
                  offsetof(Ws, den) == offsetof(soar_workspace_header, den) &&
                  offsetof(Ws, gsum) == offsetof(soar_workspace_header, gsum),
              "Ws and soar_workspace_header differ");
constexpr unsigned int kErrWait = 1u;     // a bounded wait gave up
constexpr unsigned int kErrWeight = 2u;   // a column weight outside the accepted set

// Deterministic reduce mode (SOAR_FLAG_DETERMINISTIC) of quantize_kernel: instead of adding its sums to the tensor's
// accumulators with atomics (in arrival order), every CTA of a pass stores them in a slot of its
// own, and the head of the next stage adds the slots in index order.  Two stage buffers alternate
// so that a pass can fill one while late CTAs of it still read the other.  (solo_kernel and the max-based kernels add in
// a fixed order anyway and use none of this; a call on one matrix reserves it for when it goes stage by stage.)
constexpr int kMaxGrid = 1024;   // stage_grid's limit (two CTAs per SM are 296)
struct DetParts {
  double sumsq[kMaxGrid];          // amax pass
  double stage[2][3][kMaxGrid];    // num, den, gsum of stage s in buffer s & 1
};

struct Params {
  DetParts* det;       // per-CTA partial sums; null unless SOAR_FLAG_DETERMINISTIC
  const uint16_t* W;
  uint8_t* packed;
  uint8_t* scales;     // row-major scale bytes, either the caller's buffer or workspace
  uint2* state;        // per block 8 bytes (pack_state; weighted_state); null when T == 0
  Ws* ws;
  long long ld;
  unsigned int nblk;   // rows * cols/16
  unsigned int nbc;    // cols/16
  unsigned int ntiles;
  unsigned int nbc_magic, nbc_shift;   // b / nbc == __umulhi(2 b, nbc_magic) >> nbc_shift for every b < 2^31
  int contiguous;      // ld == cols: a tile is one contiguous run of bytes
  int max_iters;
  float early_stop_rel;
  int n_dq;
  int n_beta;
  int beta_step_pct;
  int flags;           // SOAR_FLAG_* bits
};

// One launch works on up to kMaxBatch tensors: their tiles form one sequence (tensor 0's tiles,
// then tensor 1's, ...), which the CTAs of the persistent grid walk together.
constexpr int kMaxBatch = 16;
struct Batch {
  int n;
  int idle;                   // test hook: no CTA arrives anywhere, so every wait runs out
  Params t[kMaxBatch];
};
// The same for one tensor (a smaller parameter block makes a cheaper launch).
struct Single {
  static constexpr int n = 1;
  Params t[1];
};
static_assert(sizeof(Batch) <= 3072, "kernel parameter block too large");

// ------------------------------------------------------------------ number formats

__device__ __forceinline__ float bits_to_mag(unsigned int bf16_bits) {
  return __uint_as_float((bf16_bits & 0x7FFFu) << 16);
}

// Value of a non-negative E4M3 code (bias 7, 3 mantissa bits, subnormals below 2^-6).
// code<<20 read as binary32 is (1+f/8)*2^(e-127) for e>0 and f*2^-129 for e==0; times 2^120
// gives (1+f/8)*2^(e-7) and f*2^-9.
__device__ __forceinline__ float e4m3_value(int code) {
  return __fmul_rn(__uint_as_float(static_cast<unsigned int>(code) << 20), 0x1p120f);
}

// Nearest E4M3 code of v >= 0 (ties to even, saturating at 448) via the sm_100a conversion.
__device__ __forceinline__ int e4m3_encode(float v) {
  unsigned short r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.0f), "f"(v));
  return r & 0xFF;
}

// Eq. 2 for eight signed values at once: nearest point of {0,.5,1,1.5,2,3,4,6} with the
// input's sign, ties to the even code, saturating at 6.  Returns eight 4-bit codes
// (sign << 3 | magnitude code), element 0 in the low nibble.
__device__ __forceinline__ unsigned int e2m1x8(float x0, float x1, float x2, float x3, float x4, float x5,
                                               float x6, float x7) {
  unsigned int out;
  asm("{\n"
      ".reg .b8 b0, b1, b2, b3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n"
      "mov.b32 %0, {b0, b1, b2, b3};\n"
      "}"
      : "=r"(out)
      : "f"(x0), "f"(x1), "f"(x2), "f"(x3), "f"(x4), "f"(x5), "f"(x6), "f"(x7));
  return out;
}

// Four magnitude codes (the low four nibbles of `codes`, sign bits already cleared) to four
// bytes holding 2m: a byte permute over the table 0,1,2,3,4,6,8,12.
__device__ __forceinline__ unsigned int twice_magnitude_x4(unsigned int codes) {
  unsigned int out;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(out) : "r"(0x03020100u), "r"(0x0C080604u), "r"(codes));
  return out;
}

// 2*magnitude of a 3-bit E2M1 code: 0,1,2,3,4,6,8,12.
__device__ __forceinline__ float e2m1_code_value(unsigned int code3) {
  const unsigned long long lut = 0x0C08060403020100ull;
  return 0.5f * static_cast<float>(static_cast<unsigned int>(lut >> (8 * code3)) & 0xFFu);
}

// Unsigned integer to binary64 (exact).  The conversion instruction issues on the pipe of the
// special-function unit, busy for a quarter of the search's cycles; building the value from bit
// patterns instead costs two register moves and a binary64 add on pipes that are busier.
__device__ __forceinline__ double uint_to_double(unsigned int v) { return __uint2double_rn(v); }

__device__ __forceinline__ unsigned int smem_u32(const void* p) {
  return static_cast<unsigned int>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void record_failure(const Batch& bt) {
  for (int i = 0; i < bt.n; ++i)
    if (bt.t[i].ws != nullptr) atomicOr(&bt.t[i].ws->error, kErrWait);
}

// ------------------------------------------------------------------ block helpers

struct Block {
  float w[16];   // the block's elements, signed
  float bmax;    // max |w_j|
};

__device__ __forceinline__ void unpack_block(const uint4& v0, const uint4& v1, Block& blk) {
  const unsigned int u[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
  float mx = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    blk.w[2 * i] = __uint_as_float(u[i] << 16);
    blk.w[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    mx = fmaxf(mx, fmaxf(fabsf(blk.w[2 * i]), fabsf(blk.w[2 * i + 1])));
  }
  blk.bmax = mx;
}

// Two binary32 products with one instruction (sm_100a packed multiply; each half rounds to
// nearest even exactly like a scalar multiply).
__device__ __forceinline__ void mul2(float a0, float a1, float r, float& x0, float& x1) {
  asm("{\n.reg .b64 pa, pb, pd;\n"
      "mov.b64 pa, {%2, %3};\n"
      "mov.b64 pb, {%4, %4};\n"
      "mul.rn.f32x2 pd, pa, pb;\n"
      "mov.b64 {%0, %1}, pd;\n}"
      : "=f"(x0), "=f"(x1)
      : "f"(a0), "f"(a1), "f"(r));
}

// Codes of the block under reciprocal scale r (Eq. 2): x_j = fl(w_j * r), rounded to E2M1.
__device__ __forceinline__ void round_block(const Block& blk, float r, unsigned int& c0, unsigned int& c1) {
  float x[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) mul2(blk.w[2 * i], blk.w[2 * i + 1], r, x[2 * i], x[2 * i + 1]);
  c0 = e2m1x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
  c1 = e2m1x8(x[8], x[9], x[10], x[11], x[12], x[13], x[14], x[15]);
}

// 16-bit fixed-point magnitudes of a block: a_j = fix_j * 2^(e - 15) with 2^e <= bmax < 2^(e+1),
// exact for every element within 2^8 of the block maximum (smaller ones are rounded, and
// only ever multiplied by a zero code when bmax * r <= 32).  Two values per word.
struct Fixed {
  unsigned int pair[8];
  double unit;   // 2^(e - 16): A = unit * sum fix_j * (2 m_j)
  bool ok;       // false for block maxima below 2^-110, which take the binary64 path
};

__device__ __forceinline__ void make_fixed(const Block& blk, Fixed& fx) {
  const unsigned int eb = __float_as_uint(blk.bmax) >> 23;   // biased exponent of bmax
  fx.ok = eb >= 17u;
  const unsigned int ebc = max(eb, 17u);
  const float S = __uint_as_float((269u - ebc) << 23);       // 2^(15 - e)
  fx.unit = __hiloint2double(static_cast<int>((ebc + 880u) << 20), 0);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned int lo = __float_as_uint(__fmaf_rn(fabsf(blk.w[2 * i]), S, 8388608.0f));
    const unsigned int hi = __float_as_uint(__fmaf_rn(fabsf(blk.w[2 * i + 1]), S, 8388608.0f));
    fx.pair[i] = __byte_perm(lo, hi, 0x5410);   // low halves of lo and hi side by side
  }
}

// Integer sums of a code vector: afix = sum fix_j * (2 m_j), b4 = sum (2 m_j)^2.
__device__ __forceinline__ void code_sums(const Fixed& fx, unsigned int c0, unsigned int c1, unsigned int& afix,
                                          unsigned int& b4) {
  const unsigned int m0 = c0 & 0x77777777u, m1 = c1 & 0x77777777u;
  const unsigned int t0 = twice_magnitude_x4(m0), t1 = twice_magnitude_x4(m0 >> 16);
  const unsigned int t2 = twice_magnitude_x4(m1), t3 = twice_magnitude_x4(m1 >> 16);
  unsigned int b = __dp4a(t0, t0, 0u);
  b = __dp4a(t1, t1, b);
  b = __dp4a(t2, t2, b);
  b4 = __dp4a(t3, t3, b);
  unsigned int a = __dp2a_lo(fx.pair[0], t0, 0u);
  a = __dp2a_hi(fx.pair[1], t0, a);
  a = __dp2a_lo(fx.pair[2], t1, a);
  a = __dp2a_hi(fx.pair[3], t1, a);
  a = __dp2a_lo(fx.pair[4], t2, a);
  a = __dp2a_hi(fx.pair[5], t2, a);
  a = __dp2a_lo(fx.pair[6], t3, a);
  afix = __dp2a_hi(fx.pair[7], t3, a);
}

// The same sums for a code vector whose scale lies far below the block maximum: binary64
// accumulation in element order.
__device__ __forceinline__ void code_sums_wide(const float (&w)[16], unsigned int c0, unsigned int c1, double& A,
                                               double& B) {
  double sa = 0.0;
  float sb = 0.0f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const unsigned int code = ((j < 8 ? c0 : c1) >> (4 * (j & 7))) & 7u;
    const float m = e2m1_code_value(code);
    sa = fma(static_cast<double>(fabsf(w[j])), static_cast<double>(m), sa);
    sb = __fmaf_rn(m, m, sb);
  }
  A = sa;
  B = static_cast<double>(sb);
}

// A = sum |w_j| m_j and B = sum m_j^2 of a code vector made with reciprocal scale r.
__device__ __forceinline__ void block_sums(const Block& blk, const Fixed& fx, float r, unsigned int c0,
                                           unsigned int c1, double& A, double& B, unsigned int& wide) {
  if (fx.ok && __fmul_rn(blk.bmax, r) <= 32.0f) {
    unsigned int afix, b4;
    code_sums(fx, c0, c1, afix, b4);
    A = uint_to_double(afix) * fx.unit;
    B = uint_to_double(b4) * 0.25;
  } else {
    code_sums_wide(blk.w, c0, c1, A, B);
    ++wide;
  }
}


// 1/s rounded to nearest for s in [2^-125, 2^126): the hardware's approximate reciprocal
// followed by one step of Newton's iteration for 1/s, y + y * (1 - s y), both as fused multiply-adds.  On sm_100a this
// equals rcp.rn for every binary32 input of that range (soar_selftest_reciprocal compares all
// of them); it is a third of the instructions.  Callers check the range (recip_fast_ok).  The
// flush-to-zero form of the approximation is used: on that range neither s nor 1/s is
// subnormal, and the plain form carries extra instructions that rescale subnormal inputs.
__device__ __forceinline__ float recip_fast(float s) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
  return __fmaf_rn(y, __fmaf_rn(-s, y, 1.0f), y);
}
__device__ __forceinline__ bool recip_fast_ok(float s) {
  return ((__float_as_uint(s) >> 23) - 2u) <= 250u;   // positive, biased exponent 2 .. 252
}

// fl(1 / fl(alpha * dq)): the reciprocal scale of Eq. 2.
__device__ __forceinline__ float recip_scale(float alpha, float dq) {
  const float s = __fmul_rn(alpha, dq);
  return recip_fast_ok(s) ? recip_fast(s) : __frcp_rn(s);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Deterministic mode, whole warp: the sum of the n per-CTA values at `parts` in a fixed order (lane l
// adds entries l, l + 32, ... in turn, then a fixed exchange tree); every lane gets the same bits.
__device__ __forceinline__ double ordered_sum(const double* parts, int n) {
  double acc = 0.0;
  for (int j = threadIdx.x & 31; j < n; j += 32) acc += __ldcg(parts + j);
  return warp_sum(acc);
}

// Data-dependent status from the tensor maximum (bf16 magnitude bits).
__device__ __forceinline__ int status_from_amax(unsigned int amax_bits) {
  if (amax_bits >= 0x7F80u) return SOAR_STATUS_NONFINITE;
  if (amax_bits == 0) return SOAR_STATUS_ZERO_TENSOR;
  const float amax = bits_to_mag(amax_bits);
  if (!(amax >= 0x1p-100f && amax <= 0x1p100f)) return SOAR_STATUS_RANGE;
  return 0;
}

// Sec. 4.1 early stop: after an iteration, stop when the relative error gain is below eps.
__device__ __forceinline__ bool stops_after(double prev, double cur, float eps) {
  if (!(eps > 0.0f)) return false;
  if (prev == 0.0) return true;
  return (prev - cur) / prev < static_cast<double>(eps);
}

// ------------------------------------------------------------------ kernels

// The two bf16 values of a word in binary64 (exact).  The conversion instruction takes the halves as they are, and issues
// beside the integer pipe that carries the rest of a pass.
__device__ __forceinline__ double widen_low(unsigned int u) {
  double d;
  asm("{\n.reg .b16 l, h;\nmov.b32 {l, h}, %1;\ncvt.f64.bf16 %0, l;\n}" : "=d"(d) : "r"(u));
  return d;
}
__device__ __forceinline__ double widen_high(unsigned int u) {
  double d;
  asm("{\n.reg .b16 l, h;\nmov.b32 {l, h}, %1;\ncvt.f64.bf16 %0, h;\n}" : "=d"(d) : "r"(u));
  return d;
}

// Sum of squares of a block's sixteen bf16 values in binary64 (every square is exact).
__device__ __forceinline__ void sumsq_block(const unsigned int (&u)[8], double& s0, double& s1) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double dl = widen_low(u[i]), dh = widen_high(u[i]);
    s0 = fma(dl, dl, s0);
    s1 = fma(dh, dh, s1);
  }
}

// Error of stage s (Eq. 4) from the tensor sums.
__device__ __forceinline__ double stage_sse(const Ws* ws, int s) {
  return fmax(ws->sumsq + ws->gsum[s], 0.0);
}

// Head of an iteration (one thread): has the loop already stopped (Sec. 4.1), and the global
// scale of Eq. 5 from the sums of the stages so far.
// `latest` (deterministic mode): num, den, gsum of stage t, which the workspace does not hold yet.
__device__ __forceinline__ void iteration_head(const Params& p, int t, float& alpha_out, int& run_out,
                                               const double* latest = nullptr) {
  const Ws* ws = p.ws;
  int run = 1;
  const unsigned int amax_bits = ws->amax_bits;
  if (status_from_amax(amax_bits) != 0 || ws->error != 0) run = 0;
  float alpha = __fdiv_rn(bits_to_mag(amax_bits), 2688.0f);
  if (run) {
    double prev = stage_sse(ws, 0);
    if (latest != nullptr && t == 0) prev = fmax(ws->sumsq + latest[2], 0.0);
    for (int i = 0; i < t; ++i) {           // did an earlier iteration trigger the stop?
      const double cur = (latest != nullptr && i + 1 == t) ? fmax(ws->sumsq + latest[2], 0.0) : stage_sse(ws, i + 1);
      if (stops_after(prev, cur, p.early_stop_rel)) { run = 0; break; }
      prev = cur;
    }
    if (!(p.flags & SOAR_FLAG_KEEP_ALPHA))
      for (int i = 0; i <= t; ++i) {        // Eq. 5: alpha^(i+1) from stage-i sums
        const double num = (latest != nullptr && i == t) ? latest[0] : ws->num[i];
        const double den = (latest != nullptr && i == t) ? latest[1] : ws->den[i];
        if (den > 0.0) alpha = static_cast<float>(num / den);
      }
  }
  alpha_out = alpha;
  run_out = run;
}

// App. B.3's E4M3 codes around a block's analytic scale: d_lo .. d_hi before clipping (the
// nearest code alone for n_dq == 1, else n_dq codes bracketing the scale).
__device__ __forceinline__ void candidate_window(float center, int n_dq, int& d_lo, int& d_hi) {
  const int cn = e4m3_encode(center);
  if (n_dq <= 1) {
    d_lo = d_hi = cn;
  } else {
    const int cf = (e4m3_value(cn) > center) ? cn - 1 : cn;   // largest code with value <= center
    d_lo = cf - (n_dq / 2 - 1);
    d_hi = cf + n_dq / 2;
  }
}

__device__ __forceinline__ int clip_code(int d) { return max(1, min(0x7E, d)); }

// fl(alpha * fl(center * beta)): the divisor of Eq. 2 for one multiplier of the App. B.3 grid.
__device__ __forceinline__ float grid_divisor(float alpha, float center, float beta) {
  return __fmul_rn(alpha, __fmul_rn(center, beta));
}

// Which multipliers of the App. B.3 grid can win Eq. 8 for one E4M3 code, without visiting the grid.
//
// For a fixed dequantization scale sd = alpha * value(code) the error of element j,
// (a_j - m sd)^2, is convex in its code value m with its minimum at a_j / sd.  The codes
// m_j(k) = E2M1(fl(a_j * fl(1 / s_k))), s_k = grid_divisor(beta_k), never rise with k, because every
// step of that binary32 chain is monotone.  While s_k <= sd (1 - 2^-21) every fl(a_j * fl(1 / s_k)) lies
// above a_j / sd (by at least 2^-22 of it: the chain's two roundings cost 2^-24 each), so every code
// is at or above the nearest one to a_j / sd and each element's error can only fall as k grows; once
// s_k >= sd (1 + 2^-21) every scaled value lies below a_j / sd, every code is at or below the nearest
// one and the error can only rise.  The block error of Eq. 8 is therefore smallest at the last
// multiplier of the first kind, at the first of the second kind, or at one in between (the band is
// 2^-20 wide against a grid step of a hundredth: almost always empty): two multipliers in the typical
// case, where the grid has 101.
//
// Equal errors.  Two multipliers with the same codes are one outcome (the quantization scale is
// never stored).  Different codes of an element cost the same only when a_j / sd is exactly a
// rounding midpoint; because the band keeps the scaled value of such an element strictly above the
// midpoint before it and strictly below after it, the element holds its upper code for every
// multiplier before the band and its lower code for every one after, whatever the tie rule of
// the rounding: all of its free code changes happen among the multipliers of [ka, kb].  Those are
// scored in grid order with Algorithm 1's strict comparison, and outside [ka, kb] the error changes
// strictly with every code change, so the first minimum of the whole grid has the codes of the
// first minimum found here.

// Binary32 bounds of the band around sd = alpha * dv (the exact product): lo <= sd (1 - 2^-21) and
// hi >= sd (1 + 2^-21), by directed roundings.
__device__ __forceinline__ void divisor_band(float alpha, float dv, float& lo, float& hi) {
  lo = __fmul_rd(__fmul_rd(alpha, dv), 1.0f - 0x1p-21f);
  hi = __fmul_ru(__fmul_ru(alpha, dv), 1.0f + 0x1p-21f);
}

// The range [ka, kb] of multipliers that can win for a code whose band is [lo, hi], for any start
// index k: walks to the last multiplier with s_k <= lo, then on to the first with s_k >= hi.
// s_beta: pairs of neighbouring multipliers.
__device__ __forceinline__ void winning_range(const float2* s_beta, int n_beta, float alpha, float center, float lo, float hi,
                                           int k, int& ka, int& kb) {
  k = max(0, min(n_beta - 1, k));
  while (k >= 0 && grid_divisor(alpha, center, s_beta[k].x) > lo) --k;
  while (k + 1 < n_beta && grid_divisor(alpha, center, s_beta[k + 1].x) <= lo) ++k;
  ka = max(k, 0);
  kb = k + 1;
  while (kb < n_beta && grid_divisor(alpha, center, s_beta[kb].x) < hi) ++kb;
  kb = min(kb, n_beta - 1);
}

// Offset of scale (row, col) in the 128x4-tiled layout: tiles of 128 rows x 4 scale columns
// (512 bytes), tile rows outermost; inside a tile row r and column c sit at
// (r % 32) * 16 + (r / 32) * 4 + c.
__device__ __forceinline__ size_t swizzled_offset(unsigned int row, unsigned int col, unsigned int col_tiles) {
  const size_t tile = static_cast<size_t>(row >> 7) * col_tiles + (col >> 2);
  const unsigned int r = row & 127u;
  return tile * 512 + (r & 31u) * 16 + (r >> 5) * 4 + (col & 3u);
}

#include "quantize_kernel.cuh"
#include "solo_kernel.cuh"
#include "weighted_kernel.cuh"
#include "mx_kernel.cuh"
#include "error_kernel.cuh"

// Counts the binary32 inputs with biased exponent lo_exp..hi_exp (all 2^23 significands each)
// on which recip_fast differs from rcp.rn.
__global__ void selftest_reciprocal_kernel(unsigned int lo_exp, unsigned int hi_exp, unsigned long long* mismatches) {
  const unsigned long long total = static_cast<unsigned long long>(hi_exp - lo_exp + 1) << 23;
  unsigned long long bad = 0;
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<unsigned long long>(gridDim.x) * blockDim.x) {
    const float s = __uint_as_float((lo_exp << 23) + static_cast<unsigned int>(i));
    if (__float_as_uint(recip_fast(s)) != __float_as_uint(__frcp_rn(s))) ++bad;
  }
  if (bad) atomicAdd(mismatches, bad);
}

// ------------------------------------------------------------------ host side

// Optional launch tracing for benchmarks: while enabled, every kernel this library launches
// is bracketed by two CUDA events on the launching stream.
enum KernelId {
  K_AMAX = 0, K_INIT, K_ITERATE, K_FINALIZE, K_SWIZZLE, K_DEQUANT_ERROR,
  K_WEIGHTED_AMAX, K_WEIGHTED_INIT, K_WEIGHTED_ITERATE, K_MX, K_COUNT
};
const char* const kKernelNames[K_COUNT] = {"amax_kernel",          "init_kernel",          "iterate_kernel",
                                           "finalize_kernel",      "swizzle_kernel",       "dequant_error_kernel",
                                           "weighted_amax_kernel", "weighted_init_kernel", "weighted_iterate_kernel",
                                           "mx_kernel"};
struct TraceRec {
  int id;
  cudaEvent_t e0, e1;
};
struct Tracer {
  std::mutex mu;
  bool on = false;
  std::vector<TraceRec> recs;
};
Tracer g_trace;

struct ScopedLaunch {
  bool active = false;
  TraceRec rec;
  cudaStream_t st;
  ScopedLaunch(int id, cudaStream_t stream) : st(stream) {
    if (!g_trace.on) return;
    rec.id = id;
    if (cudaEventCreate(&rec.e0) != cudaSuccess) return;
    if (cudaEventCreate(&rec.e1) != cudaSuccess) { cudaEventDestroy(rec.e0); return; }
    cudaEventRecord(rec.e0, st);
    active = true;
  }
  ~ScopedLaunch() {
    if (!active) return;
    cudaEventRecord(rec.e1, st);
    std::lock_guard<std::mutex> lk(g_trace.mu);
    g_trace.recs.push_back(rec);
  }
};

int g_sm_count[64];

// Test hook (soar_debug_fail_waits): what the launches put into Batch::idle and its like, read only where CTAs meet.
int g_idle = 0;

int sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (g_sm_count[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    g_sm_count[dev] = n;
  }
  return g_sm_count[dev];
}

size_t round256(size_t n) { return (n + 255) / 256 * 256; }

bool cfg_ok(const soar_cfg* cfg) {
  return cfg != nullptr && cfg->struct_size == sizeof(soar_cfg);
}

int check_shape(const void* W, int64_t rows, int64_t cols, int64_t ld) {
  if (W == nullptr || rows <= 0 || cols <= 0) return SOAR_ERR_INVALID_ARG;
  if (cols % 16 != 0 || ld < cols || ld % 8 != 0) return SOAR_ERR_UNSUPPORTED;
  if (reinterpret_cast<uintptr_t>(W) % 16 != 0) return SOAR_ERR_UNSUPPORTED;
  if (rows * (cols / 16) >= (1ll << 31)) return SOAR_ERR_UNSUPPORTED;
  return SOAR_OK;
}

int check_cfg(const soar_cfg* cfg) {
  if (!cfg_ok(cfg)) return SOAR_ERR_INVALID_ARG;
  if (cfg->block != 16) return SOAR_ERR_UNSUPPORTED;
  if (cfg->max_iters < 0 || cfg->max_iters > SOAR_MAX_ITERS) return SOAR_ERR_INVALID_ARG;
  if (cfg->n_dq < 1 || cfg->n_dq > SOAR_MAX_DQ) return SOAR_ERR_INVALID_ARG;
  if (cfg->n_beta < 1 || cfg->n_beta > SOAR_MAX_BETA) return SOAR_ERR_INVALID_ARG;
  if (cfg->beta_step_pct < 0) return SOAR_ERR_INVALID_ARG;
  // every multiplier must stay positive
  if (100 - (cfg->n_beta / 2) * cfg->beta_step_pct <= 0) return SOAR_ERR_INVALID_ARG;
  if ((cfg->scale_layout & ~(SOAR_SCALES_LINEAR | SOAR_SCALES_SWIZZLED)) != 0 || cfg->scale_layout == 0)
    return SOAR_ERR_INVALID_ARG;
  if ((cfg->flags & ~(SOAR_FLAG_COUPLED_SCALE | SOAR_FLAG_KEEP_ALPHA | SOAR_FLAG_KEEP_BLOCK_SCALE |
                      SOAR_FLAG_DETERMINISTIC)) != 0)
    return SOAR_ERR_INVALID_ARG;
  return SOAR_OK;
}

}  // namespace

extern "C" {

int soar_default_cfg(soar_cfg* cfg, int preset) {
  if (cfg == nullptr) return SOAR_ERR_INVALID_ARG;
  memset(cfg, 0, sizeof(*cfg));
  cfg->struct_size = sizeof(soar_cfg);
  cfg->block = 16;
  cfg->scale_layout = SOAR_SCALES_LINEAR;
  cfg->beta_step_pct = 1;
  switch (preset) {
    case SOAR_PRESET_PAPER:
      cfg->max_iters = 15; cfg->early_stop_rel = 1e-3f; cfg->n_dq = 2; cfg->n_beta = 101;
      return SOAR_OK;
    case SOAR_PRESET_SINGLE_PASS:
      cfg->max_iters = 1; cfg->early_stop_rel = 0.0f; cfg->n_dq = 2; cfg->n_beta = 1;
      return SOAR_OK;
    case SOAR_PRESET_RTN:
      cfg->max_iters = 0; cfg->early_stop_rel = 0.0f; cfg->n_dq = 1; cfg->n_beta = 1;
      return SOAR_OK;
    case SOAR_PRESET_CJSO_ONLY:
      cfg->max_iters = 15; cfg->early_stop_rel = 1e-3f; cfg->n_dq = 1; cfg->n_beta = 1;
      cfg->flags = SOAR_FLAG_COUPLED_SCALE;
      return SOAR_OK;
    case SOAR_PRESET_COUPLED_PAIR:
      cfg->max_iters = 15; cfg->early_stop_rel = 1e-3f; cfg->n_dq = 2; cfg->n_beta = 1;
      cfg->flags = SOAR_FLAG_COUPLED_SCALE;
      return SOAR_OK;
    case SOAR_PRESET_DSS_ONLY:
      cfg->max_iters = 1; cfg->early_stop_rel = 0.0f; cfg->n_dq = 2; cfg->n_beta = 101;
      cfg->flags = SOAR_FLAG_KEEP_ALPHA | SOAR_FLAG_KEEP_BLOCK_SCALE;
      return SOAR_OK;
    default:
      return SOAR_ERR_INVALID_ARG;
  }
}

size_t soar_workspace_bytes(int64_t rows, int64_t cols, const soar_cfg* cfg) {
  if (check_cfg(cfg) != SOAR_OK || rows <= 0 || cols <= 0 || cols % 16 != 0) return 0;
  const size_t nblk = static_cast<size_t>(rows) * static_cast<size_t>(cols / 16);
  size_t n = kWsFixedBytes;
  if (cfg->max_iters > 0) n += round256(nblk * sizeof(uint2));
  if (!(cfg->scale_layout & SOAR_SCALES_LINEAR)) n += round256(nblk);
  if (cfg->flags & SOAR_FLAG_DETERMINISTIC) n += round256(sizeof(DetParts));
  return n + exchange_bytes(static_cast<unsigned int>((nblk + 31) / 32));
}

size_t soar_swizzled_scale_bytes(int64_t rows, int64_t cols) {
  if (rows <= 0 || cols <= 0 || cols % 16 != 0) return 0;
  const size_t rt = (static_cast<size_t>(rows) + 127) / 128;
  const size_t ct = (static_cast<size_t>(cols / 16) + 3) / 4;
  return rt * ct * 512;
}

int soar_quantize_launches(const soar_cfg* cfg) {
  if (check_cfg(cfg) != SOAR_OK) return 0;
  return 3 + cfg->max_iters + ((cfg->scale_layout & SOAR_SCALES_SWIZZLED) ? 1 : 0);
}

size_t soar_batch_workspace_bytes(const soar_tensor_desc* tensors, int n, const soar_cfg* cfg) {
  if (tensors == nullptr || n <= 0) return 0;
  size_t total = 0;
  for (int i = 0; i < n; ++i) {
    const size_t b = soar_workspace_bytes(tensors[i].rows, tensors[i].cols, cfg);
    if (b == 0) return 0;
    total += b;
  }
  return total;
}

}  // extern "C"

namespace {

// nbc's multiply-and-shift division, exact for every dividend below 2^31.
void set_division(Params& p) {
  unsigned int l = 0;
  while ((1ull << l) < p.nbc) ++l;
  p.nbc_shift = l;
  p.nbc_magic = static_cast<unsigned int>(((1ull << (31 + l)) + p.nbc - 1) / p.nbc);
}

// The driver's questions about the SMs of a context, found at run time (the library links the runtime alone).
struct SmQueries {
  CUresult (*current)(CUcontext*) = nullptr;
  CUresult (*stream_contexts)(CUstream, CUcontext*, CUgreenCtx*) = nullptr;
  CUresult (*context_resource)(CUcontext, CUdevResource*, CUdevResourceType) = nullptr;
  CUresult (*green_resource)(CUgreenCtx, CUdevResource*, CUdevResourceType) = nullptr;
  bool found = false;   // false: a driver that has no green contexts
  template <typename F>
  static bool find(const char* name, F& f) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult how;
    if (cudaGetDriverEntryPointByVersion(name, &p, 12050, cudaEnableDefault, &how) != cudaSuccess ||
        how != cudaDriverEntryPointSuccess)
      return false;
    f = reinterpret_cast<F>(p);
    return p != nullptr;
  }
  SmQueries() {
    found = find("cuCtxGetCurrent", current) && find("cuStreamGetCtx", stream_contexts) &&
            find("cuCtxGetDevResource", context_resource) && find("cuGreenCtxGetDevResource", green_resource);
    if (!found) (void)cudaGetLastError();
  }
};

// SMs that a launch on `st` is sure to get: those of the current context or of the stream's, whichever are fewer (a launch
// runs on the stream's, a captured one's node on those of the context it was captured in).  0 when that cannot be told.
unsigned int sms_for(cudaStream_t st) {
  static const SmQueries ask;
  if (!ask.found) return static_cast<unsigned int>(sm_count());
  CUcontext now = nullptr;
  if (ask.current(&now) == CUDA_SUCCESS && now == nullptr) {   // the thread's first call: the runtime has yet to bind the device
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) (void)cudaSetDevice(dev);
    (void)ask.current(&now);
  }
  CUdevResource sms;
  memset(&sms, 0, sizeof(sms));
  if (now == nullptr || ask.context_resource(now, &sms, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return 0;
  const unsigned int here = sms.sm.smCount;
  CUcontext of_stream = nullptr;
  CUgreenCtx green = nullptr;
  if (ask.stream_contexts(st, &of_stream, &green) != CUDA_SUCCESS) return 0;
  if (green == nullptr) return here;
  if (ask.green_resource(green, &sms, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return 0;
  return std::min(here, sms.sm.smCount);
}

// Whether `st` is being captured (the default stream cannot be, and must not be asked while another one is).
bool captured(cudaStream_t st) {
  if (st == nullptr || st == cudaStreamLegacy) return false;
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) == cudaSuccess) return status != cudaStreamCaptureStatusNone;
  (void)cudaGetLastError();
  return true;
}

// A cooperative launch of a grid that has room, `per_sm` CTAs on an SM.  The runtime refuses one that has none, but not
// while it is captured: replayed, such a grid would wait for its room for ever.
cudaError_t launch_cooperative(const void* kernel, unsigned int grid, unsigned int per_sm, unsigned int threads, void** args,
                               size_t dynamic, cudaStream_t st) {
  if (grid > per_sm * sms_for(st)) return cudaErrorCooperativeLaunchTooLarge;
  return cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(threads), args, dynamic, st);
}

// Grid of a stage machine's launch: every SM filled to the kernel's occupancy (`per_sm`, asked of the runtime once per
// device), never more CTAs than eight tiles each give work.
template <typename K>
unsigned int stage_grid(K kernel, std::atomic<int> (&known)[64], unsigned int tiles, unsigned int* per_sm = nullptr) {
  int dev = 0, n = 1;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
    n = known[dev].load(std::memory_order_relaxed);
    if (n == 0) {
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kQThreads, 0) != cudaSuccess || n <= 0) n = 1;
      known[dev].store(n, std::memory_order_relaxed);
    }
  }
  if (per_sm != nullptr) *per_sm = static_cast<unsigned int>(n);
  unsigned int grid = static_cast<unsigned int>(sm_count() * n);
  if (grid > static_cast<unsigned int>(kMaxGrid)) grid = kMaxGrid;   // the deterministic mode keeps one slot per CTA
  const unsigned int want = (tiles + kQWarps - 1) / kQWarps;
  return want < grid ? (want > 0 ? want : 1u) : grid;
}

// Whether a cooperative launch was refused because its grid, one for the whole device, does not fit the SMs at hand: the
// stream's context or the current one may own a part of them (a green context).  The caller then goes stage by stage,
// whose launches wait for nobody.
bool grid_refused(cudaError_t err) {
  if (err != cudaErrorCooperativeLaunchTooLarge) return false;
  (void)cudaGetLastError();
  return true;
}

// Launches stages [lo, hi) of the quantizer for one group of matrices; more than one stage makes the launch
// cooperative, so that its CTAs, which meet between stages, run at the same time.
template <int kMode, bool kDet>
cudaError_t launch_stages(const Batch& bt, const Reports& rp, unsigned int tiles, int lo, int hi, cudaStream_t st) {
  static std::atomic<int> known[64];
  unsigned int per_sm = 1;
  const unsigned int grid = stage_grid(quantize_kernel<kMode, kDet>, known, tiles, &per_sm);
  if (hi - lo == 1) {
    quantize_kernel<kMode, kDet><<<grid, kQThreads, 0, st>>>(bt, rp, lo, hi);
    return cudaGetLastError();
  }
  void* args[] = {const_cast<Batch*>(&bt), const_cast<Reports*>(&rp), &lo, &hi};
  return launch_cooperative(reinterpret_cast<const void*>(&quantize_kernel<kMode, kDet>), grid, per_sm, kQThreads, args, 0, st);
}

cudaError_t launch_stages(int mode, bool det, const Batch& bt, const Reports& rp, unsigned int tiles, int lo, int hi,
                          cudaStream_t st) {
#define SOAR_STAGES(M) (det ? launch_stages<M, true>(bt, rp, tiles, lo, hi, st) : launch_stages<M, false>(bt, rp, tiles, lo, hi, st))
  switch (mode) {
    case 0: return SOAR_STAGES(0);
    case 1: return SOAR_STAGES(1);
    case 2: return SOAR_STAGES(2);
    case 3: return SOAR_STAGES(3);
    case 4: return SOAR_STAGES(4);
    default: return SOAR_STAGES(5);
  }
#undef SOAR_STAGES
}

// The same for the weighted kernel.
template <bool kFast, bool kColumns>
cudaError_t launch_weighted(const Batch& bt, const Weighted& wt, const Reports& rp, unsigned int tiles, int lo, int hi,
                            cudaStream_t st) {
  static std::atomic<int> known[64];
  unsigned int per_sm = 1;
  const unsigned int grid = stage_grid(weighted_kernel<kFast, kColumns>, known, tiles, &per_sm);
  if constexpr (kColumns)
    if (!has_steady_columns(bt, grid * kQWarps)) return launch_weighted<kFast, false>(bt, wt, rp, tiles, lo, hi, st);
  if (hi - lo == 1) {
    weighted_kernel<kFast, kColumns><<<grid, kQThreads, 0, st>>>(bt, wt, rp, lo, hi);
    return cudaGetLastError();
  }
  void* args[] = {const_cast<Batch*>(&bt), const_cast<Weighted*>(&wt), const_cast<Reports*>(&rp), &lo, &hi};
  return launch_cooperative(reinterpret_cast<const void*>(&weighted_kernel<kFast, kColumns>), grid, per_sm, kQThreads, args, 0, st);
}
cudaError_t launch_weighted(bool fast, const Batch& bt, const Weighted& wt, const Reports& rp, unsigned int tiles, int lo, int hi,
                            cudaStream_t st) {
  return fast ? launch_weighted<true, true>(bt, wt, rp, tiles, lo, hi, st) : launch_weighted<false, true>(bt, wt, rp, tiles, lo, hi, st);
}

// kMode of quantize_kernel for a call's settings (see iterate_pass).
int search_mode(const soar_cfg* cfg) {
  const bool coupled = (cfg->flags & SOAR_FLAG_COUPLED_SCALE) != 0;
  // one quantization scale per block: the codes are made once (any number of E4M3 codes scored on them; the coupled
  // arm, where every code rounds the block anew, only with at most two)
  if (cfg->n_beta == 1 && (cfg->n_dq <= 2 || !coupled)) return coupled ? 2 : 1;
  // a grid of several multipliers with one quantization scale per multiplier: only those that can win are visited;
  // the coupled arm with a grid, and multipliers that all coincide, visit them all
  if (coupled || cfg->n_beta < kBracketMinBeta || cfg->beta_step_pct < 1) return 0;
  // the brackets of two E4M3 codes around the Eq. 6 solution lie at multipliers 0.89 .. 1.13 (E4M3 values are at most
  // an eighth apart): a grid from 0.85 to 1.15 or wider holds them whole, a shorter one (and another number of codes)
  // needs the path that knows the grid's ends
  const int half = cfg->n_beta / 2;
  const bool spans = 100 - half * cfg->beta_step_pct <= 85 && 100 + (cfg->n_beta - 1 - half) * cfg->beta_step_pct >= 115;
  if (!spans || cfg->n_dq != 2) return 5;
  return (cfg->flags & SOAR_FLAG_KEEP_BLOCK_SCALE) ? 3 : 4;
}

// Launches a kernel that may begin while the one before it in the stream ends (programmatic stream serialization): the
// kernel waits at its head (after_previous) for everything before it, and the gap between two launches shrinks from 1 to 2
// us, a multiple of about a microsecond from start to start, to half a microsecond.  Cooperative launches cannot.  cluster: CTAs of
// a cluster, or 0.
template <typename... Want, typename... Have>
cudaError_t launch_chained(void (*kernel)(Want...), unsigned int grid, unsigned int threads, size_t dynamic, unsigned int cluster,
                           cudaStream_t st, const Have&... args) {
  cudaLaunchAttribute how[2];
  memset(how, 0, sizeof(how));
  how[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  how[0].val.programmaticStreamSerializationAllowed = 1;
  how[1].id = cudaLaunchAttributeClusterDimension;
  how[1].val.clusterDim.x = cluster;
  how[1].val.clusterDim.y = how[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = dynamic;
  lc.stream = st;
  lc.attrs = how;
  lc.numAttrs = cluster > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, kernel, args...);
}

// A number no earlier call of this process used, and that memory left by another is not likely to hold: a counter
// from a random start through a 64-bit mixing function (the finalizer of SplitMix64; Steele, Lea and Flood, "Fast
// splittable pseudorandom number generators", OOPSLA 2014).
unsigned long long call_nonce() {
  static const unsigned long long seed = [] {
    const unsigned long long now =
        static_cast<unsigned long long>(std::chrono::system_clock::now().time_since_epoch().count());
    try {
      std::random_device rd;
      return now ^ (static_cast<unsigned long long>(rd()) << 32) ^ rd();
    } catch (...) {   // no source of random numbers, and no exception may leave a C entry: the clock and an address remain
      return now ^ (static_cast<unsigned long long>(reinterpret_cast<uintptr_t>(&now)) << 20);
    }
  }();
  static std::atomic<unsigned long long> calls;
  unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (calls.fetch_add(1, std::memory_order_relaxed) + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Launches with attributes set on the kernels beforehand: `set()` sets them, once per device (`raised` says for which),
// and once more where a launch fails that has them from an earlier call, since cudaDeviceReset takes them away.
template <typename Set, typename Launch>
cudaError_t launch_with(std::atomic<bool> (&raised)[64], Set set, Launch launch) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  cudaError_t err;
  if (raised[dev].load(std::memory_order_acquire)) {
    err = launch();
    if (err == cudaSuccess || err == cudaErrorCooperativeLaunchTooLarge) return err;
    (void)cudaGetLastError();
  }
  err = set();
  if (err != cudaSuccess) return err;
  raised[dev].store(true, std::memory_order_release);
  return launch();
}

// One matrix in one launch (see solo_grid, cluster_size); the tiles stay in shared memory when every warp's fit its slots.
template <int kMode, int kPlace>
cudaError_t launch_solo(const SoloArgs& a, unsigned int grid, unsigned int warps, cudaStream_t st) {
  const unsigned int slots = warps * (kPlace != kStreamed ? a.per_warp : static_cast<unsigned int>(kQStages));
  const size_t dynamic = static_cast<size_t>(slots) * (kQTileBytes + kQStateBytes);
  const auto kernel = solo_kernel<kMode, kPlace>;
  static std::atomic<bool> raised[64];
  return launch_with(
      raised,
      [&]() {
        const unsigned int most = kPlace != kStreamed ? kResidentTiles : kSoloWarps * kQStages;
        const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     static_cast<int>(most * (kQTileBytes + kQStateBytes)));
        return err == cudaSuccess && kPlace == kKeptInCluster
                   ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
                   : err;
      },
      [&]() {
        if (grid == 1 || kPlace == kKeptInCluster)
          return launch_chained(kernel, grid, warps * 32, dynamic, grid == 1 ? 0 : grid, st, a);
        void* args[] = {const_cast<SoloArgs*>(&a)};
        return launch_cooperative(reinterpret_cast<const void*>(kernel), grid, 1, warps * 32, args, dynamic, st);
      });
}

// A call without iterations on a matrix of more than kClusterTiles tiles.
cudaError_t launch_max_based(const SoloArgs& a, cudaStream_t st) {
  constexpr size_t dynamic = static_cast<size_t>(kMaxBasedThreads / 32) * kQStages * (kQTileBytes + kQStateBytes);
  static std::atomic<bool> raised[64];
  // as many slots as exchange_bytes gave room for; a CTA for every sixteen tiles until every SM has one
  const unsigned int sms = static_cast<unsigned int>(sm_count());
  const unsigned int grid = solo_grid(a.m.t[0].ntiles, sms < kSoloMaxGrid ? sms : kSoloMaxGrid);
  const unsigned int threads = a.m.t[0].ntiles > sms * kSoloWarps ? kMaxBasedThreads : kSoloWarps * 32;
  return launch_with(
      raised,
      []() {
        const cudaError_t err =
            cudaFuncSetAttribute(max_based_amax_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(dynamic));
        return err == cudaSuccess ? cudaFuncSetAttribute(max_based_codes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         static_cast<int>(dynamic))
                                  : err;
      },
      [&]() {
        const cudaError_t err = launch_chained(max_based_amax_kernel, grid, threads, dynamic, 0, st, a);
        return err == cudaSuccess ? launch_chained(max_based_codes_kernel, grid, threads, dynamic, 0, st, a) : err;
      });
}

// Whether this device has a cluster of the largest size for us (asked once per device).
bool clusters_fit() {
  static std::atomic<int> known[64];   // 0: not asked, 1: yes, 2: no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  int k = known[dev].load(std::memory_order_relaxed);
  if (k == 0) {
    const auto kernel = solo_kernel<4, kKeptInCluster>;
    cudaLaunchAttribute how;
    memset(&how, 0, sizeof(how));
    how.id = cudaLaunchAttributeClusterDimension;
    how.val.clusterDim.x = kClusterMost;
    how.val.clusterDim.y = how.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    lc.gridDim = dim3(kClusterMost);
    lc.blockDim = dim3(kSoloWarps * 32);
    lc.dynamicSmemBytes = 0;
    lc.attrs = &how;
    lc.numAttrs = 1;
    int n = 0;
    const bool yes = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                     cudaOccupancyMaxActiveClusters(&n, kernel, &lc) == cudaSuccess && n > 0;
    if (!yes) (void)cudaGetLastError();
    k = yes ? 1 : 2;
    known[dev].store(k, std::memory_order_relaxed);
  }
  return k == 1;
}

cudaError_t run_solo(const soar_tensor_desc& d, const soar_cfg* cfg, uint8_t* workspace, int mode, cudaStream_t st) {
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  SoloArgs a;
  memset(&a, 0, sizeof(a));
  Params& p = a.m.t[0];
  uint8_t* next = workspace + kWsFixedBytes;
  p.W = static_cast<const uint16_t*>(d.W_bf16);
  p.packed = static_cast<uint8_t*>(d.out_fp4_packed);
  p.ws = reinterpret_cast<Ws*>(workspace);
  p.ld = d.ld;
  p.nbc = static_cast<unsigned int>(d.cols / 16);
  p.nblk = static_cast<unsigned int>(d.rows * (d.cols / 16));
  p.ntiles = (p.nblk + 31) / 32;
  set_division(p);
  p.contiguous = (d.ld == d.cols) ? 1 : 0;
  if (cfg->max_iters > 0) {
    p.state = reinterpret_cast<uint2*>(next);
    next += round256(static_cast<size_t>(p.nblk) * sizeof(uint2));
  }
  if (want_lin) {
    p.scales = static_cast<uint8_t*>(d.out_e4m3_scales);
  } else {
    p.scales = next;
    next += round256(p.nblk);
  }
  p.max_iters = cfg->max_iters;
  p.early_stop_rel = cfg->early_stop_rel;
  p.n_dq = cfg->n_dq;
  p.n_beta = cfg->n_beta;
  p.beta_step_pct = cfg->beta_step_pct;
  p.flags = cfg->flags;
  a.alpha = d.out_global_fp32;
  a.result = d.out_result;
  a.tiled = want_sw ? static_cast<uint8_t*>(d.out_e4m3_scales_sw) : nullptr;
  a.exchange = next;
  a.nonce = call_nonce();
  a.rows = static_cast<unsigned int>(d.rows);
  a.tiled_only = want_lin ? 0 : 1;
  a.idle = g_idle;
  const unsigned int sms = static_cast<unsigned int>(sm_count());
  if (cfg->max_iters == 0) mode = kNoIterations;
  auto run = [&](bool cluster) {
    const unsigned int warps = cluster ? cluster_warps(p.ntiles) : p.ntiles <= kOneCtaTiles ? kOneCtaTiles : kSoloWarps;
    const unsigned int grid = cluster ? cluster_size(p.ntiles) : solo_grid(p.ntiles, sms < kSoloMaxGrid ? sms : kSoloMaxGrid);
    a.per_warp = (p.ntiles + grid * warps - 1) / (grid * warps);
    const bool kept = a.per_warp * warps <= kResidentTiles;
#define SOAR_SOLO(M)                                            \
  (cluster ? launch_solo<M, kKeptInCluster>(a, grid, warps, st) \
   : kept  ? launch_solo<M, kKept>(a, grid, warps, st)          \
           : launch_solo<M, kStreamed>(a, grid, warps, st))
    switch (mode) {
      case kNoIterations:
        return cluster     ? launch_solo<kNoIterations, kKeptInCluster>(a, grid, warps, st)
               : grid == 1 ? launch_solo<kNoIterations, kKept>(a, grid, warps, st)
                           : launch_max_based(a, st);
      case 0: return SOAR_SOLO(0);
      case 1: return SOAR_SOLO(1);
      case 2: return SOAR_SOLO(2);
      case 3: return SOAR_SOLO(3);
      case 4: return SOAR_SOLO(4);
      default: return SOAR_SOLO(5);
    }
#undef SOAR_SOLO
  };
  // (a cluster that finds no room is refused where it is launched, but where it is captured only as the graph is made)
  const bool cluster = p.ntiles > kOneCtaTiles && p.ntiles <= kClusterTiles && clusters_fit() && (!captured(st) || sms_for(st) >= sms);
  cudaError_t err = run(cluster);
  if (err != cudaSuccess && cluster) {   // a context that owns a few SMs may have no room for a cluster where the device has
    (void)cudaGetLastError();
    err = run(false);
  }
  return err;
}

// The MXFP4 pass.  Up to a tile a warp the call is bound by the host's launches (7.1 us in one, 8.7 in two) and the pass
// clears its result itself; cooperative, because its CTAs then wait for CTA 0.  From there on two chained launches are
// shorter on the device.
template <int kSearch, bool kPlain>
cudaError_t launch_mx(MxArgs& a, cudaStream_t st) {
  static std::atomic<int> known[64];
  unsigned int per_sm = 1;
  const unsigned int tiles = (a.m.t[0].nblk / 2 + 31) / 32;   // a block of 32 a lane
  const unsigned int grid = stage_grid(mx_kernel<kSearch, kPlain>, known, tiles, &per_sm);
  auto chained = [&]() {
    a.chained = 1;
    const cudaError_t err = launch_chained(clear_mx_kernel, 1, 32, 0, 0, st, a.res);
    return err != cudaSuccess ? err : launch_chained(mx_kernel<kSearch, kPlain>, grid, kQThreads, 0, 0, st, a);
  };
  if (tiles > grid * kQWarps) return chained();
  a.tag = call_nonce();
  if (grid == 1) {
    mx_kernel<kSearch, kPlain><<<1, kQThreads, 0, st>>>(a);
    return cudaGetLastError();
  }
  void* args[] = {&a};
  const cudaError_t err =
      launch_cooperative(reinterpret_cast<const void*>(&mx_kernel<kSearch, kPlain>), grid, per_sm, kQThreads, args, 0, st);
  return grid_refused(err) ? chained() : err;
}

// Which part of a call is wanted: all of it (soar_quantize_batch), or one stage (soar_quantize_stage; iterations
// t_lo <= t < t_hi for kStageIterate).
enum : int { kStageAmax = 1, kStageInit = 2, kStageIterate = 4, kStageFinalize = 8, kStageAll = 15 };

int run_batch(const soar_tensor_desc* tensors, int n, const soar_cfg* cfg, void* workspace, size_t workspace_bytes,
              void* stream, int stages, int t_lo, int t_hi) {
  int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  if (tensors == nullptr || n <= 0) return SOAR_ERR_INVALID_ARG;
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  const bool det = (cfg->flags & SOAR_FLAG_DETERMINISTIC) != 0;
  // a stage run alone leaves its sums in the per-CTA slots, which the caller of the stages cannot combine
  if (det && stages != kStageAll) return SOAR_ERR_UNSUPPORTED;
  for (int i = 0; i < n; ++i) {   // every argument is checked before anything is enqueued
    const soar_tensor_desc& d = tensors[i];
    rc = check_shape(d.W_bf16, d.rows, d.cols, d.ld);
    if (rc != SOAR_OK) return rc;
    if (d.out_fp4_packed == nullptr || d.out_global_fp32 == nullptr) return SOAR_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d.out_fp4_packed) % 16 != 0) return SOAR_ERR_UNSUPPORTED;
    if (want_lin && d.out_e4m3_scales == nullptr) return SOAR_ERR_INVALID_ARG;
    if (want_sw && d.out_e4m3_scales_sw == nullptr) return SOAR_ERR_INVALID_ARG;
  }
  const size_t need = soar_batch_workspace_bytes(tensors, n, cfg);
  if (workspace == nullptr || need == 0 || workspace_bytes < need) return SOAR_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return SOAR_ERR_UNSUPPORTED;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // workspace: the n headers first (one memset clears them all), then each tensor's arrays
  uint8_t* const headers = static_cast<uint8_t*>(workspace);
  uint8_t* next = headers + static_cast<size_t>(n) * kWsFixedBytes;
  const int mode = search_mode(cfg);
  bool by_stage = stages != kStageAll || g_trace.on;
  if (n == 1 && !by_stage) {
    const cudaError_t err = run_solo(tensors[0], cfg, headers, mode, st);
    by_stage = grid_refused(err);
    if (!by_stage) return err == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
  }
  if ((stages & kStageAmax) &&
      cudaMemsetAsync(headers, 0, static_cast<size_t>(n) * kWsFixedBytes, st) != cudaSuccess)
    return SOAR_ERR_CUDA;

  for (int first = 0; first < n; first += kMaxBatch) {
    Batch bt;
    Reports rp;
    memset(&bt, 0, sizeof(bt));
    memset(&rp, 0, sizeof(rp));
    bt.n = (n - first < kMaxBatch) ? n - first : kMaxBatch;
    bt.idle = g_idle == kNobodyArrives;
    unsigned int tiles = 0;
    for (int j = 0; j < bt.n; ++j) {
      const soar_tensor_desc& d = tensors[first + j];
      Params& p = bt.t[j];
      p.W = static_cast<const uint16_t*>(d.W_bf16);
      p.packed = static_cast<uint8_t*>(d.out_fp4_packed);
      p.ws = reinterpret_cast<Ws*>(headers + static_cast<size_t>(first + j) * kWsFixedBytes);
      p.ld = d.ld;
      p.nbc = static_cast<unsigned int>(d.cols / 16);
      p.nblk = static_cast<unsigned int>(d.rows * (d.cols / 16));
      p.ntiles = (p.nblk + 31) / 32;
      set_division(p);
      p.contiguous = (d.ld == d.cols) ? 1 : 0;
      p.state = nullptr;
      if (cfg->max_iters > 0) {
        p.state = reinterpret_cast<uint2*>(next);
        next += round256(static_cast<size_t>(p.nblk) * sizeof(uint2));
      }
      if (want_lin) {
        p.scales = static_cast<uint8_t*>(d.out_e4m3_scales);
      } else {
        p.scales = next;
        next += round256(p.nblk);
      }
      p.det = nullptr;
      if (det) {
        p.det = reinterpret_cast<DetParts*>(next);
        next += round256(sizeof(DetParts));
      }
      next += exchange_bytes(p.ntiles);   // used by calls on one matrix
      p.max_iters = cfg->max_iters;
      p.early_stop_rel = cfg->early_stop_rel;
      p.n_dq = cfg->n_dq;
      p.n_beta = cfg->n_beta;
      p.beta_step_pct = cfg->beta_step_pct;
      p.flags = cfg->flags;
      tiles += p.ntiles;
      rp.alpha[j] = d.out_global_fp32;
      rp.result[j] = d.out_result;
      rp.scales_sw[j] = want_sw ? static_cast<uint8_t*>(d.out_e4m3_scales_sw) : nullptr;
      rp.rows[j] = static_cast<unsigned int>(d.rows);
    }

    const int report = kQStageIterate + cfg->max_iters, end = report + 1 + (want_sw ? 1 : 0);
    cudaError_t err = cudaSuccess;
    if (!by_stage) {
      // the whole call in one launch
      err = launch_stages(mode, det, bt, rp, tiles, 0, end, st);
      by_stage = grid_refused(err);
    }
    if (by_stage) {
      // stage by stage: a caller that combines the headers between stages, a trace that times each of them, or a context
      // that has no room for the grid
      err = cudaSuccess;
      auto one = [&](int id, int s) {
        if (err != cudaSuccess) return;
        ScopedLaunch sl(id, st);
        err = launch_stages(mode, det, bt, rp, tiles, s, s + 1, st);
      };
      if (stages & kStageAmax) one(K_AMAX, kQStageAmax);
      if (stages & kStageInit) one(K_INIT, kQStageInit);
      if (stages & kStageIterate)
        for (int t = t_lo; t < t_hi; ++t) one(K_ITERATE, kQStageIterate + t);
      if (stages & kStageFinalize) {
        one(K_FINALIZE, report);
        if (want_sw) one(K_SWIZZLE, report + 1);
      }
    }
    if (err != cudaSuccess) return SOAR_ERR_CUDA;
  }
  return cudaGetLastError() == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
}

}  // namespace

extern "C" {

int soar_quantize_batch(const soar_tensor_desc* tensors, int n, const soar_cfg* cfg, void* workspace,
                        size_t workspace_bytes, void* stream) {
  const int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  return run_batch(tensors, n, cfg, workspace, workspace_bytes, stream, kStageAll, 0, cfg->max_iters);
}

int soar_quantize_stage(const soar_tensor_desc* tensors, int n, const soar_cfg* cfg, void* workspace,
                        size_t workspace_bytes, int stage, void* stream) {
  const int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  if (stage == SOAR_STAGE_AMAX) return run_batch(tensors, n, cfg, workspace, workspace_bytes, stream, kStageAmax, 0, 0);
  if (stage == SOAR_STAGE_INIT) return run_batch(tensors, n, cfg, workspace, workspace_bytes, stream, kStageInit, 0, 0);
  if (stage == SOAR_STAGE_FINALIZE)
    return run_batch(tensors, n, cfg, workspace, workspace_bytes, stream, kStageFinalize, 0, 0);
  if (stage < 0 || stage >= cfg->max_iters) return SOAR_ERR_INVALID_ARG;
  return run_batch(tensors, n, cfg, workspace, workspace_bytes, stream, kStageIterate, stage, stage + 1);
}

int soar_quantize(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, const soar_cfg* cfg,
                  void* out_fp4_packed, void* out_e4m3_scales, void* out_e4m3_scales_sw,
                  float* out_global_fp32, void* workspace, size_t workspace_bytes,
                  soar_result* out_result, void* stream) {
  soar_tensor_desc d;
  d.W_bf16 = W_bf16;
  d.rows = rows;
  d.cols = cols;
  d.ld = ld;
  d.out_fp4_packed = out_fp4_packed;
  d.out_e4m3_scales = out_e4m3_scales;
  d.out_e4m3_scales_sw = out_e4m3_scales_sw;
  d.out_global_fp32 = out_global_fp32;
  d.out_result = out_result;
  return soar_quantize_batch(&d, 1, cfg, workspace, workspace_bytes, stream);
}

// Built-in scratch of soar_quantize_static.  In host code the symbol below is only a handle:
// the device address comes from cudaGetSymbolAddress, looked up once per device.
static __device__ __align__(256) unsigned char g_static_scratch[SOAR_STATIC_SCRATCH_BYTES];
// the largest accepted matrix needs exactly this much: the header, 8 bytes of state and one scale byte per block, and the
// packets its CTAs exchange
static_assert(kWsFixedBytes + (SOAR_STATIC_MAX_ELEMENTS / 16) * (sizeof(uint2) + 1) + exchange_bytes(SOAR_STATIC_MAX_ELEMENTS / 512) ==
                  SOAR_STATIC_SCRATCH_BYTES,
              "SOAR_STATIC_SCRATCH_BYTES does not match the workspace of SOAR_STATIC_MAX_ELEMENTS");

namespace {
std::mutex g_static_mu;
void* g_static_ptr[64];

// Device address of g_static_scratch on the current device (nullptr on failure).
void* static_scratch_ptr() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (g_static_ptr[dev] == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess) return nullptr;
    g_static_ptr[dev] = ptr;
  }
  return g_static_ptr[dev];
}
}  // namespace

int soar_quantize_static(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, const soar_cfg* cfg,
                         void* out_fp4_packed, void* out_e4m3_scales, void* out_e4m3_scales_sw,
                         float* out_global_fp32, soar_result* out_result, void* stream) {
  int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  rc = check_shape(W_bf16, rows, cols, ld);
  if (rc != SOAR_OK) return rc;
  if (rows * cols > SOAR_STATIC_MAX_ELEMENTS) return SOAR_ERR_TOO_LARGE;
  if (soar_workspace_bytes(rows, cols, cfg) > static_cast<size_t>(SOAR_STATIC_SCRATCH_BYTES))
    return SOAR_ERR_TOO_LARGE;
  void* scratch = static_scratch_ptr();
  if (scratch == nullptr) return SOAR_ERR_CUDA;
  return soar_quantize(W_bf16, rows, cols, ld, cfg, out_fp4_packed, out_e4m3_scales, out_e4m3_scales_sw,
                       out_global_fp32, scratch, SOAR_STATIC_SCRATCH_BYTES, out_result, stream);
}

namespace {
int dequant_error_impl(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, const float* h,
                       const void* fp4_packed, const void* e4m3_scales, int scale_layout,
                       const float* global_fp32, double* out_sse, double* out_sumsq, void* stream) {
  const int rc = check_shape(W_bf16, rows, cols, ld);
  if (rc != SOAR_OK) return rc;
  if (fp4_packed == nullptr || e4m3_scales == nullptr || global_fp32 == nullptr || out_sse == nullptr ||
      out_sumsq == nullptr)
    return SOAR_ERR_INVALID_ARG;
  if (scale_layout != SOAR_SCALES_LINEAR && scale_layout != SOAR_SCALES_SWIZZLED) return SOAR_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(fp4_packed) % 8 != 0) return SOAR_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ErrorArgs a;
  memset(&a, 0, sizeof(a));
  Params& p = a.m.t[0];
  p.W = static_cast<const uint16_t*>(W_bf16);
  p.packed = const_cast<uint8_t*>(static_cast<const uint8_t*>(fp4_packed));
  p.ld = ld;
  p.nbc = static_cast<unsigned int>(cols / 16);
  p.nblk = static_cast<unsigned int>(rows * (cols / 16));
  p.ntiles = (p.nblk + 31) / 32;
  set_division(p);
  p.contiguous = (ld == cols) ? 1 : 0;
  a.scales = static_cast<const uint8_t*>(e4m3_scales);
  a.alpha = global_fp32;
  a.h = h;
  a.sse = out_sse;
  a.sumsq = out_sumsq;
  a.tiled = scale_layout == SOAR_SCALES_SWIZZLED ? 1 : 0;
  // the two sums start at zero (a kernel of ours rather than a memset, so that the next one can be chained to it)
  ScopedLaunch sl(K_DEQUANT_ERROR, st);
  cudaError_t err = launch_chained(clear_sums_kernel, 1, 32, 0, 0, st, out_sse, out_sumsq);
  if (err != cudaSuccess) return SOAR_ERR_CUDA;
  if (h == nullptr) {
    static std::atomic<int> known[64];
    err = launch_chained(dequant_error_kernel<false>, stage_grid(dequant_error_kernel<false>, known, p.ntiles), kQThreads, 0, 0, st, a);
  } else {
    static std::atomic<int> known[64];
    err = launch_chained(dequant_error_kernel<true>, stage_grid(dequant_error_kernel<true>, known, p.ntiles), kQThreads, 0, 0, st, a);
  }
  return err == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
}
}  // namespace

int soar_dequant_error(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, const void* fp4_packed,
                       const void* e4m3_scales, int scale_layout, const float* global_fp32,
                       double* out_sse, double* out_sumsq, void* stream) {
  return dequant_error_impl(W_bf16, rows, cols, ld, nullptr, fp4_packed, e4m3_scales, scale_layout, global_fp32,
                            out_sse, out_sumsq, stream);
}

int soar_dequant_error_weighted(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld,
                                const float* col_weight, const void* fp4_packed, const void* e4m3_scales,
                                int scale_layout, const float* global_fp32, double* out_sse,
                                double* out_sumsq, void* stream) {
  if (col_weight == nullptr) return SOAR_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(col_weight) % 16 != 0) return SOAR_ERR_UNSUPPORTED;
  return dequant_error_impl(W_bf16, rows, cols, ld, col_weight, fp4_packed, e4m3_scales, scale_layout,
                            global_fp32, out_sse, out_sumsq, stream);
}

size_t soar_weighted_workspace_bytes(int64_t rows, int64_t cols, const soar_cfg* cfg) {
  if (check_cfg(cfg) != SOAR_OK || rows <= 0 || cols <= 0 || cols % 16 != 0) return 0;
  const size_t nblk = static_cast<size_t>(rows) * static_cast<size_t>(cols / 16);
  size_t n = kWsFixedBytes;
  // 17 bytes a block, as published; the state takes 8 of them (weighted_state)
  if (cfg->max_iters > 0) n += round256(nblk * sizeof(double2)) + round256(nblk);
  if (!(cfg->scale_layout & SOAR_SCALES_LINEAR)) n += round256(nblk);
  return n;
}

size_t soar_weighted_batch_workspace_bytes(const soar_tensor_desc* tensors, int n, const soar_cfg* cfg) {
  if (tensors == nullptr || n <= 0) return 0;
  size_t total = 0;
  for (int i = 0; i < n; ++i) {
    const size_t b = soar_weighted_workspace_bytes(tensors[i].rows, tensors[i].cols, cfg);
    if (b == 0) return 0;
    total += b;
  }
  return total;
}

int soar_quantize_weighted_batch(const soar_tensor_desc* tensors, const float* const* col_weights, int n,
                                 const soar_cfg* cfg, void* workspace, size_t workspace_bytes, void* stream) {
  int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  if (cfg->flags & SOAR_FLAG_DETERMINISTIC) return SOAR_ERR_UNSUPPORTED;   // the weighted passes add with atomics only
  if (tensors == nullptr || col_weights == nullptr || n <= 0) return SOAR_ERR_INVALID_ARG;
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  for (int i = 0; i < n; ++i) {   // every argument is checked before anything is enqueued
    const soar_tensor_desc& d = tensors[i];
    rc = check_shape(d.W_bf16, d.rows, d.cols, d.ld);
    if (rc != SOAR_OK) return rc;
    if (col_weights[i] == nullptr || d.out_fp4_packed == nullptr || d.out_global_fp32 == nullptr)
      return SOAR_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(col_weights[i]) % 16 != 0 || reinterpret_cast<uintptr_t>(d.out_fp4_packed) % 16 != 0)
      return SOAR_ERR_UNSUPPORTED;
    if (want_lin && d.out_e4m3_scales == nullptr) return SOAR_ERR_INVALID_ARG;
    if (want_sw && d.out_e4m3_scales_sw == nullptr) return SOAR_ERR_INVALID_ARG;
  }
  const size_t need = soar_weighted_batch_workspace_bytes(tensors, n, cfg);
  if (workspace == nullptr || need == 0 || workspace_bytes < need) return SOAR_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return SOAR_ERR_UNSUPPORTED;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // workspace: the n headers first (one memset clears them all), then each tensor's arrays
  uint8_t* const headers = static_cast<uint8_t*>(workspace);
  uint8_t* next = headers + static_cast<size_t>(n) * kWsFixedBytes;
  if (cudaMemsetAsync(headers, 0, static_cast<size_t>(n) * kWsFixedBytes, st) != cudaSuccess) return SOAR_ERR_CUDA;
  const bool fast = search_mode(cfg) == 4;
  bool by_stage = g_trace.on;
  for (int first = 0; first < n; first += kMaxBatch) {
    Batch bt;
    Weighted wt;
    Reports rp;
    memset(&bt, 0, sizeof(bt));
    memset(&wt, 0, sizeof(wt));
    memset(&rp, 0, sizeof(rp));
    bt.n = (n - first < kMaxBatch) ? n - first : kMaxBatch;
    bt.idle = g_idle == kNobodyArrives;
    unsigned int tiles = 0;
    for (int j = 0; j < bt.n; ++j) {
      const soar_tensor_desc& d = tensors[first + j];
      Params& p = bt.t[j];
      p.W = static_cast<const uint16_t*>(d.W_bf16);
      p.packed = static_cast<uint8_t*>(d.out_fp4_packed);
      p.ws = reinterpret_cast<Ws*>(headers + static_cast<size_t>(first + j) * kWsFixedBytes);
      p.ld = d.ld;
      p.nbc = static_cast<unsigned int>(d.cols / 16);
      p.nblk = static_cast<unsigned int>(d.rows * (d.cols / 16));
      p.ntiles = (p.nblk + 31) / 32;
      set_division(p);
      p.contiguous = (d.ld == d.cols) ? 1 : 0;
      wt.h[j] = col_weights[first + j];
      if (cfg->max_iters > 0) {
        p.state = reinterpret_cast<uint2*>(next);
        next += round256(static_cast<size_t>(p.nblk) * sizeof(double2)) + round256(p.nblk);
      }
      if (want_lin) {
        p.scales = static_cast<uint8_t*>(d.out_e4m3_scales);
      } else {
        p.scales = next;
        next += round256(p.nblk);
      }
      p.max_iters = cfg->max_iters;
      p.early_stop_rel = cfg->early_stop_rel;
      p.n_dq = cfg->n_dq;
      p.n_beta = cfg->n_beta;
      p.beta_step_pct = cfg->beta_step_pct;
      p.flags = cfg->flags;
      tiles += p.ntiles;
      rp.alpha[j] = d.out_global_fp32;
      rp.result[j] = d.out_result;
      rp.scales_sw[j] = want_sw ? static_cast<uint8_t*>(d.out_e4m3_scales_sw) : nullptr;
      rp.rows[j] = static_cast<unsigned int>(d.rows);
    }
    const int report = kQStageIterate + cfg->max_iters, end = report + 1 + (want_sw ? 1 : 0);
    cudaError_t err = cudaSuccess;
    if (!by_stage) {
      err = launch_weighted(fast, bt, wt, rp, tiles, 0, end, st);
      by_stage = grid_refused(err);
    }
    if (by_stage) {   // each stage timed, or no room for the grid
      err = cudaSuccess;
      for (int s = 0; s < end && err == cudaSuccess; ++s) {
        ScopedLaunch sl(s == kQStageAmax ? K_WEIGHTED_AMAX : s == kQStageInit ? K_WEIGHTED_INIT
                        : s < report ? K_WEIGHTED_ITERATE : s == report ? K_FINALIZE : K_SWIZZLE, st);
        err = launch_weighted(fast, bt, wt, rp, tiles, s, s + 1, st);
      }
    }
    if (err != cudaSuccess) return SOAR_ERR_CUDA;
  }
  return SOAR_OK;
}

int soar_quantize_weighted(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, const float* col_weight,
                           const soar_cfg* cfg, void* out_fp4_packed, void* out_e4m3_scales,
                           void* out_e4m3_scales_sw, float* out_global_fp32, void* workspace,
                           size_t workspace_bytes, soar_result* out_result, void* stream) {
  soar_tensor_desc d;
  d.W_bf16 = W_bf16;
  d.rows = rows;
  d.cols = cols;
  d.ld = ld;
  d.out_fp4_packed = out_fp4_packed;
  d.out_e4m3_scales = out_e4m3_scales;
  d.out_e4m3_scales_sw = out_e4m3_scales_sw;
  d.out_global_fp32 = out_global_fp32;
  d.out_result = out_result;
  return soar_quantize_weighted_batch(&d, &col_weight, 1, cfg, workspace, workspace_bytes, stream);
}

int soar_quantize_host(const void* W_host, int64_t rows, int64_t cols, int64_t ld, const soar_cfg* cfg,
                       void* out_fp4_packed_host, void* out_e4m3_scales_host, void* out_e4m3_scales_sw_host,
                       float* out_global_host, soar_result* out_result_host, const soar_staging* dev,
                       void* stream) {
  if (dev == nullptr || W_host == nullptr || dev->W == nullptr) return SOAR_ERR_INVALID_ARG;
  int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  if (rows <= 0 || cols <= 0 || ld < cols) return SOAR_ERR_INVALID_ARG;
  if (out_fp4_packed_host == nullptr || out_global_host == nullptr) return SOAR_ERR_INVALID_ARG;
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  if (want_lin && (out_e4m3_scales_host == nullptr || dev->scales == nullptr)) return SOAR_ERR_INVALID_ARG;
  if (want_sw && (out_e4m3_scales_sw_host == nullptr || dev->scales_sw == nullptr)) return SOAR_ERR_INVALID_ARG;
  if (dev->packed == nullptr || dev->alpha == nullptr) return SOAR_ERR_INVALID_ARG;
  if (out_result_host != nullptr && dev->result == nullptr) return SOAR_ERR_INVALID_ARG;
  // every check soar_quantize would make on the staging buffers, before anything is enqueued
  rc = check_shape(dev->W, rows, cols, ld);
  if (rc != SOAR_OK) return rc;
  if (reinterpret_cast<uintptr_t>(dev->packed) % 16 != 0) return SOAR_ERR_UNSUPPORTED;
  const size_t need = soar_workspace_bytes(rows, cols, cfg);
  if (dev->workspace == nullptr || need == 0 || dev->workspace_bytes < need) return SOAR_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(dev->workspace) % 256 != 0) return SOAR_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t in_bytes = static_cast<size_t>(rows) * static_cast<size_t>(ld) * 2;
  if (cudaMemcpyAsync(dev->W, W_host, in_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return SOAR_ERR_CUDA;
  rc = soar_quantize(dev->W, rows, cols, ld, cfg, dev->packed, dev->scales, dev->scales_sw, dev->alpha,
                     dev->workspace, dev->workspace_bytes, out_result_host ? dev->result : nullptr, stream);
  if (rc != SOAR_OK) return rc;
  const size_t n = static_cast<size_t>(rows) * static_cast<size_t>(cols);
  bool ok = cudaMemcpyAsync(out_fp4_packed_host, dev->packed, n / 2, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (want_lin)
    ok = ok && cudaMemcpyAsync(out_e4m3_scales_host, dev->scales, n / 16, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (want_sw)
    ok = ok && cudaMemcpyAsync(out_e4m3_scales_sw_host, dev->scales_sw, soar_swizzled_scale_bytes(rows, cols),
                               cudaMemcpyDeviceToHost, st) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(out_global_host, dev->alpha, sizeof(float), cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (out_result_host != nullptr)
    ok = ok && cudaMemcpyAsync(out_result_host, dev->result, sizeof(soar_result), cudaMemcpyDeviceToHost, st) ==
                   cudaSuccess;
  return ok ? SOAR_OK : SOAR_ERR_CUDA;
}

}  // extern "C"

// Host bookkeeping of a pipeline: the slots, three events per slot, the streams and whose turn it is.
struct soar_pipeline {
  std::vector<soar_slot> slots;
  std::vector<cudaEvent_t> loaded, computed, stored;   // per slot: input landed, quantized, results left
  cudaStream_t h2d, compute, d2h;
  size_t next;
};

namespace {
void release_events(soar_pipeline* p) {
  for (cudaEvent_t e : p->loaded) cudaEventDestroy(e);
  for (cudaEvent_t e : p->computed) cudaEventDestroy(e);
  for (cudaEvent_t e : p->stored) cudaEventDestroy(e);
}

// Every rule a matrix must meet to go through slot `sl` (nothing is enqueued before all matrices pass).
int check_host_matrix(const soar_host_matrix& m, const soar_slot& sl, const soar_cfg* cfg, bool weighted) {
  if (m.W_host == nullptr || m.out_fp4_packed_host == nullptr || m.out_global_host == nullptr)
    return SOAR_ERR_INVALID_ARG;
  int rc = check_shape(sl.dev.W, m.rows, m.cols, m.ld);
  if (rc != SOAR_OK) return rc;
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  if (want_lin && (m.out_e4m3_scales_host == nullptr || sl.dev.scales == nullptr)) return SOAR_ERR_INVALID_ARG;
  if (want_sw && (m.out_e4m3_scales_sw_host == nullptr || sl.dev.scales_sw == nullptr)) return SOAR_ERR_INVALID_ARG;
  if (m.out_result_host != nullptr && sl.dev.result == nullptr) return SOAR_ERR_INVALID_ARG;
  const size_t n = static_cast<size_t>(m.rows) * static_cast<size_t>(m.cols);
  if (static_cast<size_t>(m.rows) * static_cast<size_t>(m.ld) * 2 > sl.W_bytes || n / 2 > sl.packed_bytes)
    return SOAR_ERR_TOO_LARGE;
  if (want_lin && n / 16 > sl.scales_bytes) return SOAR_ERR_TOO_LARGE;
  if (want_sw && soar_swizzled_scale_bytes(m.rows, m.cols) > sl.scales_sw_bytes) return SOAR_ERR_TOO_LARGE;
  const size_t need = weighted ? soar_weighted_workspace_bytes(m.rows, m.cols, cfg)
                               : soar_workspace_bytes(m.rows, m.cols, cfg);
  if (need == 0 || sl.dev.workspace_bytes < need) return SOAR_ERR_WORKSPACE;
  return SOAR_OK;
}
}  // namespace

extern "C" {

int soar_pipeline_create(soar_pipeline** out, const soar_slot* slots, int n_slots, void* stream_h2d,
                         void* stream_compute, void* stream_d2h) {
  if (out == nullptr || slots == nullptr || n_slots < 1) return SOAR_ERR_INVALID_ARG;
  if (stream_h2d == stream_compute || stream_compute == stream_d2h || stream_h2d == stream_d2h)
    return SOAR_ERR_INVALID_ARG;
  for (int i = 0; i < n_slots; ++i) {
    const soar_staging& d = slots[i].dev;
    if (d.W == nullptr || d.packed == nullptr || d.alpha == nullptr || d.workspace == nullptr)
      return SOAR_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d.W) % 16 != 0 || reinterpret_cast<uintptr_t>(d.packed) % 16 != 0 ||
        reinterpret_cast<uintptr_t>(d.workspace) % 256 != 0)
      return SOAR_ERR_UNSUPPORTED;
  }
  soar_pipeline* p = new (std::nothrow) soar_pipeline();
  if (p == nullptr) return SOAR_ERR_INVALID_ARG;
  p->slots.assign(slots, slots + n_slots);
  p->h2d = static_cast<cudaStream_t>(stream_h2d);
  p->compute = static_cast<cudaStream_t>(stream_compute);
  p->d2h = static_cast<cudaStream_t>(stream_d2h);
  p->next = 0;
  bool ok = true;
  for (int i = 0; i < 3 * n_slots && ok; ++i) {
    cudaEvent_t e;
    ok = cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (ok) (i % 3 == 0 ? p->loaded : i % 3 == 1 ? p->computed : p->stored).push_back(e);
  }
  // a slot is free from the start: its "results left" event is recorded once on the third stream
  for (size_t i = 0; i < p->stored.size() && ok; ++i) ok = cudaEventRecord(p->stored[i], p->d2h) == cudaSuccess;
  if (!ok || p->stored.size() != static_cast<size_t>(n_slots)) {
    release_events(p);
    delete p;
    return SOAR_ERR_CUDA;
  }
  *out = p;
  return SOAR_OK;
}

int soar_pipeline_run(soar_pipeline* pipe, const soar_host_matrix* mats, int n, const soar_cfg* cfg,
                      const float* const* col_weights) {
  if (pipe == nullptr || mats == nullptr || n < 0) return SOAR_ERR_INVALID_ARG;
  int rc = check_cfg(cfg);
  if (rc != SOAR_OK) return rc;
  const size_t ns = pipe->slots.size();
  // Everything is checked before anything is enqueued.  The order: what follows the last copy in is that matrix's own
  // quantizing and copying out, so the list ends with its smallest matrix (the four attention matrices of an 8B layer:
  // 1.89 -> 1.73 ms), where every slot takes the matrix it then gets; otherwise it keeps the caller's order.
  auto check = [&](const int* order) {   // null: the caller's order
    for (int k = 0; k < n; ++k) {
      const int i = order != nullptr ? order[k] : k;
      const float* h = col_weights != nullptr ? col_weights[i] : nullptr;
      if (h != nullptr && reinterpret_cast<uintptr_t>(h) % 16 != 0) return static_cast<int>(SOAR_ERR_UNSUPPORTED);
      const int bad = check_host_matrix(mats[i], pipe->slots[(pipe->next + static_cast<size_t>(k)) % ns], cfg, h != nullptr);
      if (bad != SOAR_OK) return bad;
    }
    return static_cast<int>(SOAR_OK);
  };
  rc = check(nullptr);
  if (rc != SOAR_OK) return rc;
  std::unique_ptr<int[]> order(new (std::nothrow) int[static_cast<size_t>(n)]);   // without memory for it: the caller's order
  if (order != nullptr) {
    std::iota(order.get(), order.get() + n, 0);
    std::stable_sort(order.get(), order.get() + n, [&](int a, int b) { return mats[a].rows * mats[a].ld > mats[b].rows * mats[b].ld; });
    if (check(order.get()) != SOAR_OK) order.reset();
  }
  const bool want_lin = (cfg->scale_layout & SOAR_SCALES_LINEAR) != 0;
  const bool want_sw = (cfg->scale_layout & SOAR_SCALES_SWIZZLED) != 0;
  for (int k = 0; k < n; ++k) {
    const int i = order != nullptr ? order[k] : k;
    const soar_host_matrix& m = mats[i];
    const size_t si = pipe->next % ns;
    ++pipe->next;
    const soar_staging& d = pipe->slots[si].dev;
    const float* h = col_weights != nullptr ? col_weights[i] : nullptr;
    // copy in, once the slot's previous results have left
    bool ok = cudaStreamWaitEvent(pipe->h2d, pipe->stored[si], 0) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(d.W, m.W_host, static_cast<size_t>(m.rows) * static_cast<size_t>(m.ld) * 2,
                               cudaMemcpyHostToDevice, pipe->h2d) == cudaSuccess;
    ok = ok && cudaEventRecord(pipe->loaded[si], pipe->h2d) == cudaSuccess;
    ok = ok && cudaStreamWaitEvent(pipe->compute, pipe->loaded[si], 0) == cudaSuccess;
    if (!ok) return SOAR_ERR_CUDA;
    soar_result* res = m.out_result_host != nullptr ? d.result : nullptr;
    rc = h == nullptr ? soar_quantize(d.W, m.rows, m.cols, m.ld, cfg, d.packed, d.scales, d.scales_sw, d.alpha,
                                      d.workspace, d.workspace_bytes, res, pipe->compute)
                      : soar_quantize_weighted(d.W, m.rows, m.cols, m.ld, h, cfg, d.packed, d.scales, d.scales_sw,
                                               d.alpha, d.workspace, d.workspace_bytes, res, pipe->compute);
    if (rc != SOAR_OK) return rc;
    ok = cudaEventRecord(pipe->computed[si], pipe->compute) == cudaSuccess;
    ok = ok && cudaStreamWaitEvent(pipe->d2h, pipe->computed[si], 0) == cudaSuccess;
    const size_t ne = static_cast<size_t>(m.rows) * static_cast<size_t>(m.cols);
    ok = ok && cudaMemcpyAsync(m.out_fp4_packed_host, d.packed, ne / 2, cudaMemcpyDeviceToHost, pipe->d2h) ==
                   cudaSuccess;
    if (want_lin)
      ok = ok && cudaMemcpyAsync(m.out_e4m3_scales_host, d.scales, ne / 16, cudaMemcpyDeviceToHost, pipe->d2h) ==
                     cudaSuccess;
    if (want_sw)
      ok = ok && cudaMemcpyAsync(m.out_e4m3_scales_sw_host, d.scales_sw, soar_swizzled_scale_bytes(m.rows, m.cols),
                                 cudaMemcpyDeviceToHost, pipe->d2h) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(m.out_global_host, d.alpha, sizeof(float), cudaMemcpyDeviceToHost, pipe->d2h) ==
                   cudaSuccess;
    if (res != nullptr)
      ok = ok && cudaMemcpyAsync(m.out_result_host, d.result, sizeof(soar_result), cudaMemcpyDeviceToHost,
                                 pipe->d2h) == cudaSuccess;
    ok = ok && cudaEventRecord(pipe->stored[si], pipe->d2h) == cudaSuccess;
    if (!ok) return SOAR_ERR_CUDA;
  }
  return SOAR_OK;
}

int soar_pipeline_synchronize(soar_pipeline* pipe) {
  if (pipe == nullptr) return SOAR_ERR_INVALID_ARG;
  return cudaStreamSynchronize(pipe->d2h) == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
}

void soar_pipeline_destroy(soar_pipeline* pipe) {
  if (pipe == nullptr) return;
  cudaStreamSynchronize(pipe->h2d);
  cudaStreamSynchronize(pipe->compute);
  cudaStreamSynchronize(pipe->d2h);
  release_events(pipe);
  delete pipe;
}

int soar_selftest_reciprocal(int lo_exp, int hi_exp, unsigned long long* out_mismatches, void* stream) {
  if (out_mismatches == nullptr || lo_exp < 2 || hi_exp > 252 || lo_exp > hi_exp) return SOAR_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(out_mismatches, 0, sizeof(unsigned long long), st) != cudaSuccess) return SOAR_ERR_CUDA;
  selftest_reciprocal_kernel<<<sm_count() * 8, 256, 0, st>>>(static_cast<unsigned int>(lo_exp),
                                                             static_cast<unsigned int>(hi_exp), out_mismatches);
  return cudaGetLastError() == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
}

int soar_mx_quantize(const void* W_bf16, int64_t rows, int64_t cols, int64_t ld, int n_dq, int n_beta,
                     int beta_step_pct, void* out_fp4_packed, void* out_e8m0_scales, soar_mx_result* out_result,
                     void* stream) {
  const int rc = check_shape(W_bf16, rows, cols, ld);
  if (rc != SOAR_OK) return rc;
  if (cols % 32 != 0) return SOAR_ERR_UNSUPPORTED;
  if (out_fp4_packed == nullptr || out_e8m0_scales == nullptr || out_result == nullptr) return SOAR_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(out_fp4_packed) % 16 != 0 || reinterpret_cast<uintptr_t>(out_result) % 8 != 0)
    return SOAR_ERR_UNSUPPORTED;
  if (n_beta < 0 || n_beta > SOAR_MAX_BETA || n_dq < 1 || n_dq > SOAR_MAX_DQ || beta_step_pct < 0)
    return SOAR_ERR_INVALID_ARG;
  if (n_beta > 0 && 100 - (n_beta / 2) * beta_step_pct <= 0) return SOAR_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  MxArgs a;
  memset(&a, 0, sizeof(a));
  Params& p = a.m.t[0];
  p.W = static_cast<const uint16_t*>(W_bf16);
  p.packed = static_cast<uint8_t*>(out_fp4_packed);
  p.ld = ld;
  p.nbc = static_cast<unsigned int>(cols / 16);
  p.nblk = static_cast<unsigned int>(rows * (cols / 16));
  p.ntiles = (p.nblk + 31) / 32;
  set_division(p);
  p.contiguous = (ld == cols) ? 1 : 0;
  a.scales = static_cast<uint8_t*>(out_e8m0_scales);
  a.res = out_result;
  a.n_dq = n_dq;
  a.n_beta = n_beta;
  a.step_pct = beta_step_pct;
  a.idle = g_idle == kNobodyArrives;
  ScopedLaunch sl(K_MX, st);
  cudaError_t err;
  // every block of 32 is 64 bytes at a multiple of 32: two 256-bit loads
  const bool plain = p.contiguous && reinterpret_cast<uintptr_t>(W_bf16) % 32 == 0;
  if (n_beta == 0) err = plain ? launch_mx<0, true>(a, st) : launch_mx<0, false>(a, st);
  else if (n_dq == 2 && n_beta >= kBracketMinBeta && beta_step_pct >= 1 && beta_step_pct <= 25 &&
           100 - (n_beta / 2) * beta_step_pct <= 50 && (n_beta - 1 - n_beta / 2) >= 1)
    err = plain ? launch_mx<2, true>(a, st) : launch_mx<2, false>(a, st);
  else err = launch_mx<1, false>(a, st);
  return err == cudaSuccess ? SOAR_OK : SOAR_ERR_CUDA;
}

int soar_debug_fail_waits(int on) {
  g_idle = on >= 0 && on <= kShareBeyond ? on : kNobodyArrives;
  return SOAR_OK;
}

int soar_trace_begin(void) {
  std::lock_guard<std::mutex> lk(g_trace.mu);
  for (TraceRec& r : g_trace.recs) { cudaEventDestroy(r.e0); cudaEventDestroy(r.e1); }
  g_trace.recs.clear();
  g_trace.on = true;
  return SOAR_OK;
}

int soar_trace_end(soar_trace_entry* out, int capacity, int* count) {
  std::lock_guard<std::mutex> lk(g_trace.mu);
  g_trace.on = false;
  double total[K_COUNT] = {0};
  int64_t launches[K_COUNT] = {0};
  bool ok = true;
  for (TraceRec& r : g_trace.recs) {
    float ms = 0.0f;
    if (cudaEventSynchronize(r.e1) != cudaSuccess || cudaEventElapsedTime(&ms, r.e0, r.e1) != cudaSuccess) ok = false;
    total[r.id] += ms;
    launches[r.id] += 1;
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  g_trace.recs.clear();
  int n = 0;
  for (int k = 0; k < K_COUNT; ++k) {
    if (launches[k] == 0) continue;
    if (out != nullptr && n < capacity) {
      memset(&out[n], 0, sizeof(out[n]));
      strncpy(out[n].kernel, kKernelNames[k], sizeof(out[n].kernel) - 1);
      out[n].launches = launches[k];
      out[n].total_ms = total[k];
    }
    ++n;
  }
  if (count != nullptr) *count = n;
  return ok ? SOAR_OK : SOAR_ERR_CUDA;
}

const char* soar_status_string(int status) {
  switch (status) {
    case SOAR_OK: return "ok";
    case SOAR_ERR_INVALID_ARG: return "invalid argument";
    case SOAR_ERR_UNSUPPORTED: return "unsupported shape, alignment or block size";
    case SOAR_ERR_WORKSPACE: return "workspace missing or too small";
    case SOAR_ERR_CUDA: return "CUDA runtime or launch error";
    case SOAR_ERR_TOO_LARGE: return "matrix exceeds the built-in scratch of soar_quantize_static or a pipeline slot";
    default: return "unknown status";
  }
}

}  // extern "C"
