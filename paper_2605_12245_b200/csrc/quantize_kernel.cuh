// The NVFP4 quantizer as one persistent kernel: every pass of Algorithm 1 over a batch of matrices, with the
// tensor-wide sums of one pass combined before the next begins.  Included by soar.cu.
//
// Shape of the kernel.  Work is dealt in warp tiles of 32 blocks (1 KB of bf16, one 16-element block per lane):
// warp w of the grid takes tiles w, w + warps, ... of the concatenated tiles of the tensors a pass works on.  A warp
// feeds itself; there is no producer to poll, no block-wide barrier in the tile loop and no wait that could run out.
//   Light passes (the maximum, the start, one candidate per block) are bound by HBM: the lanes start 16-byte
//   asynchronous copies of the tile kQStages - 1 turns ahead into the warp's own slots of shared memory (registers four to
//   six tiles deep instead were no faster).
//   The search is bound by instruction issue: a lane loads its next block, 32 bytes with one 256-bit load, into
//   registers one tile ahead, which costs 20 instructions a block less.
// 28672 x 8192, one pass as a launch of its own: maximum 82 -> 77 us (2.01 bytes an element, 6.1 TB/s), start 127 -> 111 us
// (2.43 bytes, 180 instructions a block), iteration of the search 307 -> 210 us (3.45 bytes, 352 instructions a block issued
// in 71 % of the cycles).
// Two CTAs of 256 threads per SM leave 128 registers a thread, which holds a block, the next one, the four candidates
// of the search and their sums without spills (the deterministic forms spill up to 34 bytes, one of a single matrix that
// streams 8).
//
// Bytes 16 apart in a slot are exchanged between its two 128-byte halves (tile_chunk) so that the 32-byte reads
// of neighbouring lanes meet no bank conflict.

#pragma once

constexpr int kQThreads = 256;
constexpr int kQWarps = kQThreads / 32;
constexpr int kQStages = 4;                        // slots of a warp's ring
constexpr unsigned int kQTileBytes = 1024;         // 32 blocks of 16 bf16
constexpr unsigned int kQStateBytes = 256;         // 32 block states of 8 bytes

// Stages of a call, in order: amax, init, the iterations, the report.
constexpr int kQStageAmax = 0, kQStageInit = 1, kQStageIterate = 2;

struct Reports {   // where each tensor of a batch wants its alpha and its report (report may be null)
  float* alpha[kMaxBatch];
  soar_result* result[kMaxBatch];
  uint8_t* scales_sw[kMaxBatch];   // tiled copy of the scales; null when the layout is not requested
  unsigned int rows[kMaxBatch];
};

// A block's carried state: {A as binary32, eb << 23 | d << 12 | 4B} with eb the biased exponent of the block's
// largest magnitude, d its E4M3 scale code and 4B = sum (2m)^2 <= 2304; all zero for an all-zero block.
__device__ __forceinline__ unsigned int pack_state(unsigned int eb_field, int d, unsigned int b4) {
  return eb_field | (static_cast<unsigned int>(d) << 12) | b4;
}

// Head of a kernel launched by launch_chained: waits until everything before it in the stream is done and visible.
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// From here on the next such kernel may take its place on the SMs.
__device__ __forceinline__ void let_next_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Position of 16-byte chunk j in a tile slot.
__device__ __forceinline__ unsigned int tile_chunk(unsigned int j) { return j ^ ((j >> 3) & 1u); }

__device__ __forceinline__ void copy16(unsigned int dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint4 lds128(unsigned int a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
// A block's 32 bytes, 32-byte aligned, read once per pass (not kept in L1).
__device__ __forceinline__ void load_block32(const void* src, uint4& v0, uint4& v1) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v0.x), "=r"(v0.y), "=r"(v0.z), "=r"(v0.w), "=r"(v1.x), "=r"(v1.y), "=r"(v1.z), "=r"(v1.w)
               : "l"(src));
}
// A block state: written by other SMs in the pass before, so from L2.
__device__ __forceinline__ uint2 load_state(const void* src) {
  uint2 v;
  asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(src));
  return v;
}
// Block b of a matrix wherever it lies: rows may be apart, 16-byte alignment is all that is given.
__device__ __forceinline__ void load_block(const Params& p, unsigned int b, uint4& v0, uint4& v1) {
  const unsigned int row = __umulhi(2u * b, p.nbc_magic) >> p.nbc_shift;
  const uint4* src = reinterpret_cast<const uint4*>(p.W + static_cast<long long>(row) * p.ld +
                                                    static_cast<long long>(b - row * p.nbc) * 16);
  v0 = __ldg(src);
  v1 = __ldg(src + 1);
}
__device__ __forceinline__ uint2 lds64(unsigned int a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}

// High words of the binary64 forms of 4m for the four codes in the low half of `codes` (the low words are zero), negative
// where kSigned and the code is.  Scaled by four the eight values 0, 2, 4, 6, 8, 12, 16, 24 have high words 0, 4000,
// 4010, 4018, 4020, 4028, 4030, 4038 over sixteen zero bits: two lookups per four codes give the two bytes, and one
// permute per element places them; its two zero bytes are the second byte's sign bit, which is always clear, replicated.
template <bool kSigned>
__device__ __forceinline__ void code_words(unsigned int codes, unsigned int (&hi)[4]) {
  const unsigned int m = codes & 0x77777777u;
  unsigned int b3 = __byte_perm(0x40404000u, 0x40404040u, m);
  const unsigned int b2 = __byte_perm(0x18100000u, 0x38302820u, m);
  if (kSigned) {
    // a set sign bit in a selector replicates the top bit of the byte: 0xFF where negative, 0xC0 where not (the instruction
    // itself: the intrinsic drops that bit)
    unsigned int neg;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(neg) : "r"(0xC0C0C0C0u), "r"(codes));
    b3 |= (neg << 2) & 0x80808080u;
  }
  asm("prmt.b32 %0, %1, %2, 0x4088;" : "=r"(hi[0]) : "r"(b2), "r"(b3));
  asm("prmt.b32 %0, %1, %2, 0x5199;" : "=r"(hi[1]) : "r"(b2), "r"(b3));
  asm("prmt.b32 %0, %1, %2, 0x62AA;" : "=r"(hi[2]) : "r"(b2), "r"(b3));
  asm("prmt.b32 %0, %1, %2, 0x73BB;" : "=r"(hi[3]) : "r"(b2), "r"(b3));
}

// Two binary32 values in one register pair, and the packed operations on them (each half rounds to nearest like
// the scalar operation).
typedef unsigned long long pair_t;
__device__ __forceinline__ pair_t pair_of(float lo, float hi) {
  pair_t p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
  return p;
}
__device__ __forceinline__ void halves(pair_t p, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ pair_t pair_mul(pair_t a, pair_t b) {
  pair_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ pair_t pair_fma(pair_t a, pair_t b, pair_t c) {
  pair_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// recip_fast of two divisors, given negated.
__device__ __forceinline__ void pair_recip(pair_t neg, float& r_lo, float& r_hi) {
  float lo, hi, y_lo, y_hi;
  halves(neg, lo, hi);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y_lo) : "f"(-lo));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y_hi) : "f"(-hi));
  const pair_t y = pair_of(y_lo, y_hi);
  halves(pair_fma(y, pair_fma(neg, y, pair_of(1.0f, 1.0f)), y), r_lo, r_hi);
}

// fl(n / d) from y = fl(1 / d) (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34, 1990: with y correctly rounded and n * y within an ulp of n / d, one exact
// remainder and one fused step give the correctly rounded quotient).  Callers keep n, d and n / d far enough from
// the ends of the exponent range for the remainder to be exact.
__device__ __forceinline__ float quotient(float n, float d, float y) {
  const float q = __fmul_rn(n, y);
  return __fmaf_rn(__fmaf_rn(-q, d, n), y, q);
}

// Tensors whose alpha lies in [2^-60, 2^60] (every real weight matrix) keep all divisors of the search inside
// the ranges of recip_fast and quotient; any other alpha takes the general path block by block.
__device__ __forceinline__ bool tame_alpha(float alpha) { return alpha >= 0x1p-60f && alpha <= 0x1p60f; }

// The block as eight register pairs of signed binary32 values.
struct PairBlock {
  pair_t w[8];
};
__device__ __forceinline__ void unpack_pairs(const uint4& v0, const uint4& v1, PairBlock& b) {
  const unsigned int u[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) b.w[i] = pair_of(__uint_as_float(u[i] << 16), __uint_as_float(u[i] & 0xFFFF0000u));
}

// Codes of the block under reciprocal scale r (Eq. 2), as round_block.
__device__ __forceinline__ void round_pairs(const PairBlock& b, float r, unsigned int& c0, unsigned int& c1) {
  const pair_t rr = pair_of(r, r);
  float x[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) halves(pair_mul(b.w[i], rr), x[2 * i], x[2 * i + 1]);
  c0 = e2m1x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
  c1 = e2m1x8(x[8], x[9], x[10], x[11], x[12], x[13], x[14], x[15]);
}

// 16-bit fixed-point magnitudes fix_j = |w_j| * S, S = 2^(10 - e) for the smallest scale s of the search,
// 2^e <= s < 2^(e+1).  Exact for every element that some candidate gives a non-zero code (it is at least 2^(e-2), so
// its last bit is at least 2^(e-9)); smaller ones are rounded and only ever multiplied by zero.  Fits 16 bits while
// the largest magnitude is below 2^(e+5), which the callers check; sum fix_j * 2 m_j then stays below 2^23.
// Scaling by the search's own scale instead of by the block maximum saves finding that maximum in every pass.
struct FixedPairs {
  unsigned int pair[8];
};
__device__ __forceinline__ float fixed_scale(float s) {
  return __uint_as_float((264u << 23) - (__float_as_uint(s) & 0x7F800000u));
}
__device__ __forceinline__ void make_fixed_pairs(const PairBlock& b, float S, FixedPairs& fx) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float lo, hi;
    halves(b.w[i], lo, hi);
    fx.pair[i] = __byte_perm(__float_as_uint(__fmaf_rn(fabsf(lo), S, 8388608.0f)),
                             __float_as_uint(__fmaf_rn(fabsf(hi), S, 8388608.0f)), 0x5410);
  }
}

// The integer sums of a code vector, as code_sums: afix = sum fix_j * (2 m_j), b4 = sum (2 m_j)^2.
__device__ __forceinline__ void pair_code_sums(const FixedPairs& fx, unsigned int c0, unsigned int c1,
                                               unsigned int& afix, unsigned int& b4) {
  const unsigned int m0 = c0 & 0x77777777u, m1 = c1 & 0x77777777u;
  const unsigned int t[4] = {twice_magnitude_x4(m0), twice_magnitude_x4(m0 >> 16), twice_magnitude_x4(m1),
                             twice_magnitude_x4(m1 >> 16)};
  unsigned int a = 0, b = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    b = __dp4a(t[q], t[q], b);
    a = __dp2a_lo(fx.pair[2 * q], t[q], a);
    a = __dp2a_hi(fx.pair[2 * q + 1], t[q], a);
  }
  afix = a;
  b4 = b;
}

// One candidate scored: codes (signs included), integer sums, and e = rho * 4B - afix in binary64, which orders the
// candidates of one E4M3 code like their errors (error minus sum W^2 = alpha dv e / S with rho = alpha dv S / 4).
struct Candidate {
  unsigned int c0, c1, afix, b4;
  double e;
};
__device__ __forceinline__ void score_pairs(const PairBlock& b, const FixedPairs& fx, float r, double rho, Candidate& o) {
  round_pairs(b, r, o.c0, o.c1);
  pair_code_sums(fx, o.c0, o.c1, o.afix, o.b4);
  o.e = fma(rho, uint_to_double(o.b4), -uint_to_double(o.afix));
}

// A positive normal binary32 value times a power of two as binary64, from its bit pattern (exact): dv * 2^k for
// an E4M3 value dv, whose trailing significand bits are zero.
__device__ __forceinline__ double scaled_value(unsigned int dv_bits, int k_field) {
  return __hiloint2double(static_cast<int>((dv_bits >> 3) + 0x38000000u) + k_field, 0);
}

// What a pass has found for a block: codes, 4B, A, scale code, error minus sum W^2.
struct Found {
  unsigned int c0, c1, b4;
  float A;
  int d;
  double g;
};

// The winner of Eq. 8 for one block by the general rules: any number of E4M3 codes, clipped windows, scales of any
// size, sums in binary64 where the integer ones do not hold, the coupled arm.  Out of line: the common blocks
// never come here, and nothing of it weighs on their registers.  kMode as iterate_pass.
template <int kMode>
__device__ __noinline__ Found search_general(const Params& p, unsigned int b, float alpha, float center, const float2* s_beta,
                                             int n_beta, int n_dq, float k_scale, float k_off, unsigned int* wide_out) {
  uint4 v0, v1;
  load_block(p, b, v0, v1);
  Block blk;
  unpack_block(v0, v1, blk);
  Fixed fx;
  make_fixed(blk, fx);
  const double alpha_d = static_cast<double>(alpha);
  unsigned int wide = 0;
  int d_lo, d_hi;
  candidate_window(center, n_dq, d_lo, d_hi);
  double best = __longlong_as_double(0x7FF0000000000000ll), bestA = 0.0, bestB = 0.0;
  unsigned int best0 = 0, best1 = 0;
  int best_d = clip_code(d_lo);
  if (kMode == 1) {
    // one quantization scale (beta = 1): the codes are fixed, only the E4M3 code is chosen
    const float r = recip_scale(alpha, center);
    round_block(blk, r, best0, best1);
    block_sums(blk, fx, r, best0, best1, bestA, bestB, wide);
    for (int d = d_lo; d <= d_hi; ++d) {
      const int dc = clip_code(d);
      const double sd = alpha_d * static_cast<double>(e4m3_value(dc));
      const double g = sd * fma(sd, bestB, -2.0 * bestA);
      if (g < best) { best = g; best_d = dc; }
    }
  } else if (kMode == 2) {
    // beta = 1 and the coupled scale of Sec. 3.2: each E4M3 candidate rounds the block with its own value
    for (int d = d_lo; d <= d_hi; ++d) {
      const int dc = clip_code(d);
      const float r = recip_scale(alpha, e4m3_value(dc));
      unsigned int c0, c1;
      double A, B;
      round_block(blk, r, c0, c1);
      block_sums(blk, fx, r, c0, c1, A, B, wide);
      const double sd = alpha_d * static_cast<double>(e4m3_value(dc));
      const double g = sd * fma(sd, B, -2.0 * A);
      if (g < best) { best = g; best_d = dc; bestA = A; bestB = B; best0 = c0; best1 = c1; }
    }
  } else {
    // the grid of App. B.3, only the multipliers that can win (winning_range)
    const float per_center = __fdividef(k_scale, center);
    int best_k = 0, prev = -1;
    for (int d = d_lo; d <= d_hi; ++d) {
      const int dc = clip_code(d);
      if (dc == prev) continue;   // clipping at the ends of the E4M3 range repeats a code
      prev = dc;
      const float dv = e4m3_value(dc);
      const double sd = alpha_d * static_cast<double>(dv);
      float lo, hi;
      divisor_band(alpha, dv, lo, hi);
      int ka, kb;
      winning_range(s_beta, n_beta, alpha, center, lo, hi, __float2int_rd(__fmaf_rn(dv, per_center, k_off)), ka, kb);
      for (int k = ka; k <= kb; ++k) {
        const float sk = grid_divisor(alpha, center, s_beta[k].x);
        const float r = recip_fast_ok(sk) ? recip_fast(sk) : __frcp_rn(sk);
        unsigned int c0, c1;
        double A, B;
        round_block(blk, r, c0, c1);
        block_sums(blk, fx, r, c0, c1, A, B, wide);
        const double g = sd * fma(sd, B, -2.0 * A);
        // equal errors: the earlier multiplier, then the smaller code, as in grid order
        if (g < best || (g == best && k < best_k)) {
          best = g; bestA = A; bestB = B; best0 = c0; best1 = c1; best_d = dc; best_k = k;
        }
      }
    }
  }
  *wide_out += wide;
  Found f;
  f.c0 = best0;
  f.c1 = best1;
  f.b4 = static_cast<unsigned int>(bestB * 4.0);
  f.A = static_cast<float>(bestA);
  f.d = best_d;
  f.g = best;
  return f;
}

// Every multiplier in turn, for the coupled arm with a grid and for grids whose multipliers all coincide: first
// minimum in (beta, code) order.
__device__ __noinline__ Found search_every(const Params& p, unsigned int b, float alpha, float center, const float2* s_beta, int n_beta,
                                           int n_dq, bool coupled, unsigned int* wide_out) {
  uint4 v0, v1;
  load_block(p, b, v0, v1);
  Block blk;
  unpack_block(v0, v1, blk);
  Fixed fx;
  make_fixed(blk, fx);
  const double alpha_d = static_cast<double>(alpha);
  unsigned int wide = 0;
  int d_lo, d_hi;
  candidate_window(center, n_dq, d_lo, d_hi);
  const int nd = d_hi - d_lo + 1;
  double best = __longlong_as_double(0x7FF0000000000000ll);
  int best_k = 0, best_d = 0;
  for (int k = 0; k < n_beta; ++k) {
    float r = recip_scale(alpha, __fmul_rn(center, s_beta[k].x));
    unsigned int c0, c1;
    double A = 0.0, B = 0.0;
    if (!coupled) {
      round_block(blk, r, c0, c1);
      block_sums(blk, fx, r, c0, c1, A, B, wide);
    }
    for (int d = 0; d < nd; ++d) {
      const float dv = e4m3_value(clip_code(d_lo + d));
      if (coupled) {
        r = recip_scale(alpha, __fmul_rn(dv, s_beta[k].x));
        round_block(blk, r, c0, c1);
        block_sums(blk, fx, r, c0, c1, A, B, wide);
      }
      const double sd = alpha_d * static_cast<double>(dv);
      const double g = sd * fma(sd, B, -2.0 * A);
      if (g < best) { best = g; best_k = k; best_d = d; }
    }
  }
  *wide_out += wide;
  // the winner, made again from its index
  Found f;
  f.d = clip_code(d_lo + best_d);
  const float r = recip_scale(alpha, __fmul_rn(coupled ? e4m3_value(f.d) : center, s_beta[best_k].x));
  round_block(blk, r, f.c0, f.c1);
  double A, B;
  unsigned int unused = 0;
  block_sums(blk, fx, r, f.c0, f.c1, A, B, unused);
  f.b4 = static_cast<unsigned int>(B * 4.0);
  f.A = static_cast<float>(A);
  f.g = best;
  return f;
}

// The max-based start of one block (Eq. 1-2) by the general rules, for an alpha outside tame_alpha.
__device__ __noinline__ Found start_general(const Params& p, unsigned int b, float alpha, unsigned int* wide_out) {
  uint4 v0, v1;
  load_block(p, b, v0, v1);
  Block blk;
  unpack_block(v0, v1, blk);
  Fixed fx;
  make_fixed(blk, fx);
  Found f;
  f.d = max(e4m3_encode(__fdiv_rn(blk.bmax, __fmul_rn(alpha, 6.0f))), 1);
  const float v = e4m3_value(f.d);
  const float r = recip_scale(alpha, v);
  round_block(blk, r, f.c0, f.c1);
  double A, B;
  unsigned int wide = 0;
  block_sums(blk, fx, r, f.c0, f.c1, A, B, wide);
  *wide_out += wide;
  f.b4 = static_cast<unsigned int>(B * 4.0);
  f.A = static_cast<float>(A);
  const double sd = static_cast<double>(alpha) * static_cast<double>(v);
  f.g = sd * fma(sd, B, -2.0 * A);
  return f;
}

// ------------------------------------------------------------------ one CTA's shared state

// Where a tensor's outputs go, kept in shared memory: two 16-byte reads per tile.  Left to itself the compiler re-reads
// the parameter block at a computed address for every pointer and tile (18 instructions of 374), and held in registers
// they would spill.
struct __align__(16) View {
  uint8_t* packed;
  uint8_t* scales;
  uint2* state;
  uint8_t* tiled;   // tiled scales written by the start pass itself; null for none
};
__device__ __forceinline__ void load_view(unsigned int at, uint8_t*& packed, uint8_t*& scales, uint2*& state) {
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(packed), "=l"(scales) : "r"(at));
  asm volatile("ld.shared.u64 %0, [%1];" : "=l"(state) : "r"(at + 16));
  __builtin_assume(__isGlobal(packed) && __isGlobal(scales) && __isGlobal(state));
}

// A count in shared memory that can pass 32 bits, in two words: shared memory adds 32 bits at a time.
__device__ __forceinline__ void add_count(unsigned int& low, unsigned int& high, unsigned long long n) {
  const unsigned int l = static_cast<unsigned int>(n);
  const unsigned int h = static_cast<unsigned int>(n >> 32) + (atomicAdd(&low, l) > ~l ? 1u : 0u);
  if (h) atomicAdd(&high, h);
}
__device__ __forceinline__ unsigned long long count_of(unsigned int low, unsigned int high) {
  return low | (static_cast<unsigned long long>(high) << 32);
}

template <bool kDet>
struct __align__(128) QShared {
  static constexpr bool kOrdered = kDet, kSolo = false, kResident = false;
  // whether the start pass is known to be the last one; otherwise a kernel for one matrix (kSolo) has iterations
  static constexpr bool kFinal = false;
  unsigned char ring[kQWarps][kQStages * (kQTileBytes + kQStateBytes)];   // also write_report's scratch
  View view[kMaxBatch];
  float2 beta[SOAR_MAX_BETA];              // {multiplier k, multiplier k + 1}
  // sums of the stage in hand, per tensor: {sum W^2, -} in the amax pass, {4 den, gsum} later
  double acc[kMaxBatch][2];
  double part[kDet ? kMaxBatch : 1][kDet ? kQWarps : 1][2];   // deterministic mode: per warp, added in warp order
  double sse[kMaxBatch];                   // error after the last stage the early stop has looked at
  float alpha[kMaxBatch];
  unsigned int amax[kMaxBatch], zeros[kMaxBatch], wide[kMaxBatch], wide_high[kMaxBatch];
  unsigned int start[kMaxBatch], count[kMaxBatch];   // positions of each tensor's tiles in the pass's sequence
  unsigned int total;                      // tiles of the pass
  unsigned int run;                        // bit per tensor the next pass works on
  unsigned int visited;                    // bit per tensor this CTA has sums for
  int failed;
};

// The grid's arrival counter, in the part of the first tensor's header that the public layout leaves free.
__device__ __forceinline__ unsigned int* arrivals(const Batch& bt) {
  return reinterpret_cast<unsigned int*>(reinterpret_cast<unsigned char*>(bt.t[0].ws) + kWsFixedBytes - 64);
}
static_assert(sizeof(Ws) <= kWsFixedBytes - 64, "no room for the arrival counter");

// All CTAs of the (cooperative) launch: everything written before is visible after.  The wait is bounded: when
// it runs out, every tensor's error word is set and the CTA leaves the kernel.
template <typename S>
__device__ __forceinline__ bool grid_sync(S& sh, const Batch& bt, unsigned int target) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int* const bar = arrivals(bt);
    __threadfence();
    if (!bt.idle) atomicAdd(bar, 1u);   // test hook: nobody arrives, every wait runs out
    unsigned int seen = 0, polls = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
    } while (seen < target && ++polls < kGridWaitLimit);
    if (seen < target) {
      sh.failed = 1;
      record_failure(bt);
    }
  }
  __syncthreads();
  return sh.failed == 0;
}

// Which tiles the coming pass works on: those of the tensors in `run`, in order.
template <typename S>
__device__ __forceinline__ void lay_out_pass(S& sh, const Batch& bt) {
  if (threadIdx.x == 0) {
    unsigned int at = 0;
    for (int i = 0; i < bt.n; ++i) {
      sh.start[i] = at;
      sh.count[i] = ((sh.run >> i) & 1u) ? bt.t[i].ntiles : 0u;
      at += sh.count[i];
    }
    sh.total = at;
  }
  __syncthreads();
}

// One warp's run of tiles within one tensor: local tile numbers tile, tile + step, ... (`left` of them), those whose
// positions in the pass's sequence are the warp's own number modulo the number of warps.  For `reverse` the same
// tiles from the last to the first: consecutive passes alternate so that a pass starts on what the previous one
// left in L2.
struct Run {
  int ti;
  unsigned int left;
  int tile, step;
};

// Warps that share tensor ti's tiles.
template <typename S>
__device__ __forceinline__ unsigned int span_of(const S&, int, unsigned int warps) { return warps; }

// The run after `r` (r.ti = -1: the first one); left == 0 when the warp's share of the pass is over.
template <typename S>
__device__ __forceinline__ void next_run(const S& sh, int n, bool reverse, unsigned int warp, unsigned int warps, Run& r) {
  r.left = 0;
  int at = reverse ? n - 1 - r.ti : r.ti;
  if (r.ti < 0) at = -1;
  while (++at < n) {
    const int ti = reverse ? n - 1 - at : at;
    const unsigned int count = sh.count[ti], span = span_of(sh, ti, warps);
    unsigned int first = warp;
    if constexpr (!S::kSolo) {
      const unsigned int past = sh.start[ti] % warps;
      first = warp >= past ? warp - past : warp + warps - past;
    }
    if (first < count && first < span) {
      r.ti = ti;
      r.left = (count - 1 - first) / span + 1;
      r.tile = static_cast<int>(reverse ? first + (r.left - 1) * span : first);
      r.step = reverse ? -static_cast<int>(span) : static_cast<int>(span);
      return;
    }
  }
}

// Warps of a CTA, and the shared address of a warp's tile slots.
template <typename S>
__device__ __forceinline__ unsigned int cta_warps() {
  if constexpr (S::kSolo) return blockDim.x >> 5;
  else return kQWarps;
}
template <typename S>
__device__ __forceinline__ unsigned int slots_of(S& sh, unsigned int warp) {
  if constexpr (S::kSolo) return sh.slots + warp * sh.per_warp * (kQTileBytes + kQStateBytes);
  else return smem_u32(sh.ring[warp]);
}

// A warp's number in the grid.  Neighbouring numbers lie in different CTAs, so that the last, partial turn over the tiles
// gives every SM its part instead of some SMs a whole turn and the others none (2048 x 2048: 8192 tiles over 2368 warps are
// 55 or 56 an SM instead of 48 or 64).
__device__ __forceinline__ unsigned int warp_number(unsigned int warp) { return warp * gridDim.x + blockIdx.x; }
// The first block of a lane's first tile of a forward pass over one tensor.
__device__ __forceinline__ unsigned int first_block() {
  return warp_number(threadIdx.x >> 5) * 32 + (threadIdx.x & 31u);
}

// Waits until at most n of the lane's copy groups are in flight.
__device__ __forceinline__ void copies_wait_upto(unsigned int n) {
  switch (n) {
    case 0: copies_wait<0>(); break;
    case 1: copies_wait<1>(); break;
    case 2: copies_wait<2>(); break;
    case 3: copies_wait<3>(); break;
    default: copies_wait<4>(); break;
  }
}

// The walk over tiles that stay in shared memory for the whole call: the warp's own slots, filled once by load_resident
// (one copy group per tile), the block states beside them.
template <bool kState, typename S, typename B, typename Enter, typename Leave, typename Body>
__device__ __forceinline__ void walk_resident(S& sh, const B& bt, Enter enter, Leave leave, Body body) {
  const unsigned int lane = threadIdx.x & 31u, warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
  const unsigned int warps = gridDim.x * cta_warps<S>(), me = warp_number(warp), tiles = bt.t[0].ntiles;
  if (me >= tiles) return;
  const unsigned int n = (tiles - 1 - me) / warps + 1;
  unsigned int at = slots_of(sh, warp);
  unsigned int b = me * 32 + lane;
  const unsigned int get = tile_chunk(2 * lane) * 16;
  enter(0);
  for (unsigned int k = 0; k < n; ++k) {
    if (!kState) {   // (the passes that read states come later)
      copies_wait_upto(n - 1 - k);
      __syncwarp();
    }
    const uint4 v0 = lds128(at + get), v1 = lds128((at + get) ^ 16u);
    const unsigned int state_at = at + kQTileBytes + lane * 8;
    uint2 st = make_uint2(0u, 0u);
    if (kState) st = lds64(state_at);
    body(b, v0, v1, st, []() {}, state_at);
    at += kQTileBytes + kQStateBytes;
    b += warps * 32;
  }
  leave(0);
}

// Starts the copies of every tile of the warp into its slots, per_warp of them at `slots` for each warp.
template <typename B>
__device__ __forceinline__ void load_resident(const B& bt, unsigned int slots, unsigned int per_warp) {
  const Params& p = bt.t[0];
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = gridDim.x * (blockDim.x >> 5);
  unsigned int at = slots + warp * per_warp * (kQTileBytes + kQStateBytes) + tile_chunk(lane) * 16;
  const unsigned char* const w = reinterpret_cast<const unsigned char*>(p.W);
  for (unsigned int tile = warp_number(warp); tile < p.ntiles; tile += warps) {
#pragma unroll
    for (unsigned int h = 0; h < 2; ++h) {
      const unsigned int b = tile * 32 + h * 16 + (lane >> 1);
      const unsigned int row = p.contiguous ? 0u : __umulhi(2u * b, p.nbc_magic) >> p.nbc_shift;
      const unsigned char* src = w + (static_cast<long long>(row) * (p.ld - static_cast<long long>(p.nbc) * 16) +
                                      static_cast<long long>(b) * 16) * 2 + (lane & 1u) * 16;
      if (b < p.nblk) copy16(at + 512 * h, src);
    }
    copies_commit();
    at += kQTileBytes + kQStateBytes;
  }
}

// One warp's walk over its share of the pass's tiles.  `enter(ti)` and `leave(ti)` bracket the tiles of one tensor;
// `body(b, v0, v1, st, next, state_at)` gets the lane's block number (past the tensor's end in the last tile: the body
// looks), its 32 bytes and, with kState, its block state, and calls next() once it is done with these registers;
// state_at is where a resident block keeps its state in shared memory.  kRing: tiles
// come through the warp's slots in shared memory, three ahead; else through registers, one ahead.  The warp
// number is broadcast so that the compiler sees the bookkeeping as uniform.  `fed()` is called once by every warp when
// the copies of its first tiles are on their way; the walk ends there if it returns false.
struct Go {
  __device__ __forceinline__ bool operator()() const { return true; }
};
template <bool kRing, bool kState, typename S, typename B, typename Enter, typename Leave, typename Body, typename Fed = Go>
__device__ __forceinline__ void walk_tiles(S& sh, const B& bt, bool reverse, Enter enter, Leave leave, Body body, Fed fed = Fed()) {
  if constexpr (S::kResident) {
    walk_resident<kState>(sh, bt, enter, leave, body);
    return;
  } else {
  const unsigned int lane = threadIdx.x & 31u, warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
  const unsigned int warps = gridDim.x * cta_warps<S>(), me = warp_number(warp);
  const unsigned int ring = slots_of(sh, warp);
  const unsigned int put = ring + tile_chunk(lane) * 16, get = ring + tile_chunk(2 * lane) * 16;
  const unsigned int put_state = ring + kQStages * kQTileBytes + lane * 16, get_state = ring + kQStages * kQTileBytes + lane * 8;

  Run f;          // the feeding side
  f.ti = -1;
  f.left = 0;
  const unsigned char *f_w = nullptr, *f_state = nullptr;
  unsigned int f_b = 0, f_step = 0;      // the lane's block (registers)
  long long f_w_step = 0, f_state_step = 0;
  bool f_plain = true;   // contiguous, every tile of the run whole, and 32-byte aligned where that matters
  auto enter_feed = [&]() {
    next_run(sh, bt.n, reverse, me, warps, f);
    if (f.left == 0) return;
    const Params& p = bt.t[f.ti];
    // the ragged last tile of a tensor is the last of a forward run, the first of a backward one
    const int top = reverse ? f.tile : f.tile + static_cast<int>(f.left - 1) * f.step;
    f_w = reinterpret_cast<const unsigned char*>(p.W);
    f_state = reinterpret_cast<const unsigned char*>(p.state);
    f_plain = p.contiguous && static_cast<unsigned int>(top) * 32 + 32 <= p.nblk &&
              (kRing || (reinterpret_cast<uintptr_t>(f_w) & 31u) == 0);
    f_b = static_cast<unsigned int>(f.tile) * 32 + lane;
    f_step = static_cast<unsigned int>(f.step) * 32;
    if (kRing) {
      if (f_plain) f_w += static_cast<size_t>(f.tile) * kQTileBytes + lane * 16;
      f_w_step = static_cast<long long>(f.step) * kQTileBytes;
      f_state += static_cast<size_t>(f.tile) * kQStateBytes + lane * 16;
      f_state_step = static_cast<long long>(f.step) * kQStateBytes;
    }
  };
  auto feed_ring = [&](unsigned int k) {
    if (f.left == 0) return;
    const unsigned int dst = put + k * kQTileBytes;
    if (f_plain) {
      copy16(dst, f_w);
      copy16(dst + 512, f_w + 512);
      f_w += f_w_step;
    } else {
      const Params& p = bt.t[f.ti];
      const unsigned int b0 = f_b - lane;
#pragma unroll
      for (unsigned int h = 0; h < 2; ++h) {
        const unsigned int b = b0 + h * 16 + (lane >> 1);
        const unsigned int row = __umulhi(2u * b, p.nbc_magic) >> p.nbc_shift;
        // (in 64 bits throughout: a row of 2^32 weights or more is accepted)
        const unsigned char* src = f_w + (static_cast<long long>(row) * (p.ld - static_cast<long long>(p.nbc) * 16) +
                                          static_cast<long long>(b) * 16) * 2 + (lane & 1u) * 16;
        if (b < p.nblk) copy16(dst + 512 * h, src);
      }
      f_b += f_step;
    }
    if (kState) {
      // the state array is padded to 256 bytes, so whole tiles stay inside it
      if (lane < 16) copy16(put_state + k * kQStateBytes, f_state);
      f_state += f_state_step;
    }
    if (--f.left == 0) enter_feed();
  };
  // (registers) Plain tiles left of the feeding run: one check a tile, everything else is out of the loop's way.
  unsigned int f_quick = 0;
  auto feed_registers = [&](uint4& v0, uint4& v1, uint2& st) {
    if (f_quick == 0) {
      if (f.left == 0) enter_feed();
      if (f.left == 0) return;
      if (!f_plain) {
        const Params& p = bt.t[f.ti];
        if (f_b < p.nblk) {
          load_block(p, f_b, v0, v1);
          if (kState) st = load_state(f_state + static_cast<size_t>(f_b) * 8);
        }
        f_b += f_step;
        --f.left;
        return;
      }
      f_quick = f.left;
      f.left = 0;
    }
    load_block32(f_w + static_cast<size_t>(f_b) * 32, v0, v1);
    if (kState) st = load_state(f_state + static_cast<size_t>(f_b) * 8);
    f_b += f_step;
    --f_quick;
  };

  uint4 v0 = make_uint4(0u, 0u, 0u, 0u), v1 = v0;
  uint2 st = make_uint2(0u, 0u);
  unsigned int slot = 0;
  enter_feed();
  if (kRing) {
#pragma unroll
    for (unsigned int k = 0; k < kQStages - 1; ++k) {
      feed_ring(k);
      copies_commit();
    }
  } else {
    feed_registers(v0, v1, st);
  }
  if (!fed()) {
    copies_wait<0>();
    return;
  }
  Run r;
  r.ti = -1;
  for (next_run(sh, bt.n, reverse, me, warps, r); r.left != 0; next_run(sh, bt.n, reverse, me, warps, r)) {
    enter(r.ti);
    unsigned int b = static_cast<unsigned int>(r.tile) * 32 + lane;
    const unsigned int b_step = static_cast<unsigned int>(r.step) * 32;
    for (unsigned int left = r.left; left != 0; --left) {
      if (kRing) {
        copies_wait<kQStages - 2>();
        __syncwarp();   // every lane's copies have landed, and every lane has read the slot that is filled next
        feed_ring((slot + kQStages - 1) % kQStages);
        copies_commit();
        const unsigned int at = get + slot * kQTileBytes;
        v0 = lds128(at);
        v1 = lds128(at ^ 16u);
        if (kState) st = lds64(get_state + slot * kQStateBytes);
        slot = (slot + 1) % kQStages;
        body(b, v0, v1, st, []() {}, 0u);
      } else {
        body(b, v0, v1, st, [&]() { feed_registers(v0, v1, st); }, 0u);
      }
      b += b_step;
    }
    leave(r.ti);
  }
  }
}

// A warp hands its sums for tensor ti to the CTA's.
template <typename S>
__device__ __forceinline__ void hand_over(S& sh, int ti, double (&v)[2]) {
  v[0] = warp_sum(v[0]);
  v[1] = warp_sum(v[1]);
  if ((threadIdx.x & 31) == 0) {
    if constexpr (S::kSolo) {
      sh.part[threadIdx.x >> 5][0] = v[0];
      sh.part[threadIdx.x >> 5][1] = v[1];
    } else if constexpr (S::kOrdered) {
      sh.part[ti][threadIdx.x >> 5][0] += v[0];
      sh.part[ti][threadIdx.x >> 5][1] += v[1];
      atomicOr(&sh.visited, 1u << ti);
    } else {
      atomicAdd(&sh.acc[ti][0], v[0]);
      atomicAdd(&sh.acc[ti][1], v[1]);
      atomicOr(&sh.visited, 1u << ti);
    }
  }
  v[0] = v[1] = 0.0;
}

// Sum of a warp's counts of candidates.  A lane's fits 32 bits (28,340 blocks of 8,192 candidates), the warp's need not.
__device__ __forceinline__ unsigned long long warp_count(unsigned int n) {
  return __reduce_add_sync(0xFFFFFFFFu, n & 0xFFFFu) +
         (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, n >> 16)) << 16);
}

template <typename S>
__device__ __forceinline__ void hand_over_counters(S& sh, int ti, unsigned int& zeros, unsigned int& wide) {
  zeros = __reduce_add_sync(0xFFFFFFFFu, zeros);
  const unsigned long long all_wide = warp_count(wide);
  if ((threadIdx.x & 31) == 0) {
    if (zeros) atomicAdd(&sh.zeros[ti], zeros);
    if (all_wide) add_count(sh.wide[ti], sh.wide_high[ti], all_wide);
  }
  zeros = wide = 0;
}

// End of a pass: the CTA's sums go to the tensors' headers (or, in the deterministic mode, to the CTA's own slots), and
// the CTA's accumulators are cleared for the next pass.  s < 0: the amax pass; else the stage of num, den, gsum.
template <bool kDet>
__device__ __forceinline__ void file_sums(QShared<kDet>& sh, const Batch& bt, int s) {
  __syncthreads();
  const int ti = threadIdx.x;
  if (ti < bt.n) {
    Ws* ws = bt.t[ti].ws;
    double a = sh.acc[ti][0], g = sh.acc[ti][1];
    if (kDet) {
      a = g = 0.0;
      for (int w = 0; w < kQWarps; ++w) {
        a += sh.part[ti][w][0];
        g += sh.part[ti][w][1];
        sh.part[ti][w][0] = sh.part[ti][w][1] = 0.0;
      }
    }
    const bool visited = (sh.visited >> ti) & 1u;
    if (s < 0) {
      if (kDet) bt.t[ti].det->sumsq[blockIdx.x] = a;
      else if (visited) atomicAdd(&ws->sumsq, a);
      if (sh.amax[ti]) atomicMax(&ws->amax_bits, sh.amax[ti]);
    } else {
      // gsum = alpha^2 den - 2 alpha num, block by block and so for the sums: two sums are carried, the third follows
      // (both terms of alpha^2 den - gsum are positive: nothing cancels)
      const double alpha = static_cast<double>(sh.alpha[ti]);
      const double den = 0.25 * a;
      const double num = (alpha * alpha * den - g) / (2.0 * alpha);
      if (kDet) {
        DetParts* dp = bt.t[ti].det;
        dp->stage[s & 1][0][blockIdx.x] = visited ? num : 0.0;
        dp->stage[s & 1][1][blockIdx.x] = den;
        dp->stage[s & 1][2][blockIdx.x] = g;
      } else if (visited) {
        atomicAdd(&ws->num[s], num);
        atomicAdd(&ws->den[s], den);
        atomicAdd(&ws->gsum[s], g);
      }
      if (sh.zeros[ti]) atomicAdd(&ws->zero_blocks, static_cast<unsigned long long>(sh.zeros[ti]));
      const unsigned long long wide = count_of(sh.wide[ti], sh.wide_high[ti]);
      if (wide) atomicAdd(&ws->wide, wide);
    }
    sh.acc[ti][0] = sh.acc[ti][1] = 0.0;
    sh.amax[ti] = sh.zeros[ti] = sh.wide[ti] = sh.wide_high[ti] = 0u;
  }
  __syncthreads();
  if (threadIdx.x == 0) sh.visited = 0u;
}

// ------------------------------------------------------------------ passes

// A block's carried state goes to the workspace, or stays in shared memory with a resident block.
template <typename S>
__device__ __forceinline__ void put_state(uint2* state, unsigned int b, unsigned int state_at, uint2 v) {
  if constexpr (S::kResident) asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(state_at), "r"(v.x), "r"(v.y) : "memory");
  else state[b] = v;
}

// A scale byte of the start pass when it is the last one: row-major, tiled, or both.
template <typename S>
__device__ __forceinline__ void put_scale(const S& sh, const Params& p, uint8_t* scales, unsigned int b, int d) {
  if constexpr (S::kFinal) {
    uint8_t* const tiled = sh.view[0].tiled;
    if (tiled != nullptr) {
      const unsigned int row = __umulhi(2u * b, p.nbc_magic) >> p.nbc_shift;
      tiled[swizzled_offset(row, b - row * p.nbc, (p.nbc + 3) / 4)] = static_cast<uint8_t>(d);
      if (sh.tiled_only) return;
    }
  }
  scales[b] = static_cast<uint8_t>(d);
}

// Eq. 1's tensor maximum, plus sum W^2 (binary64) for the error report.
template <typename S, typename B>
__device__ __forceinline__ void amax_pass(S& sh, const B& bt) {
  const unsigned int lane = threadIdx.x & 31u;
  unsigned int mx = 0;
  double sq[2] = {0.0, 0.0};
  unsigned int nblk = 0;
  walk_tiles<true, false>(
      sh, bt, false, [&](int ti) { nblk = bt.t[ti].nblk; },
      [&](int ti) {
        mx = max(mx & 0xFFFFu, mx >> 16);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (lane == 0 && mx) atomicMax(&sh.amax[ti], mx);
        double v[2] = {sq[0] + sq[1], 0.0};
        hand_over(sh, ti, v);
        mx = 0;
        sq[0] = sq[1] = 0.0;
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2&, auto next, unsigned int) {
        const bool here = b < nblk;
        const unsigned int u[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        // largest magnitude of the block with packed bf16 max (a NaN input comes out of the maximum
        // as NaN, whose bits are above the infinity pattern)
        unsigned int bmx = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          unsigned int m;
          asm("abs.bf16x2 %0, %1;" : "=r"(m) : "r"(u[i]));
          asm("max.NaN.bf16x2 %0, %0, %1;" : "+r"(bmx) : "r"(m));
        }
        if (here) {
          mx = __vmaxu2(mx, bmx & 0x7FFF7FFFu);
          sumsq_block(u, sq[0], sq[1]);
        }
        next();
      });
}

// Algorithm 1 "Initialization" (Eq. 1): dd0 = E4M3(bmax/(6 alpha0)), dq0 = dd0; first codes (Eq. 2); stage-0 sums for
// Eq. 5 and the starting error.  Codes and scales are written here only when no iteration follows, the block states only when
// one does.
template <typename S, typename B, typename Fed = Go>
__device__ __forceinline__ void init_pass(S& sh, const B& bt, Fed fed = Fed()) {
  float alpha = 1.0f, six_alpha = 6.0f, six_inv = 0.0f;
  double alpha_d = 1.0;
  bool tame = false;
  double acc[2] = {0.0, 0.0};   // 4 den, gsum
  unsigned int zeros = 0, wide = 0;
  int tensor = 0;
  unsigned int nblk = 0, view = 0;
  unsigned int keep = !S::kFinal && (S::kSolo || bt.t[0].max_iters > 0);
  if (!S::kFinal && !S::kSolo) asm volatile("" : "+r"(keep));
  walk_tiles<true, false>(
      sh, bt, true,
      [&](int ti) {
        alpha = sh.alpha[ti];
        six_alpha = __fmul_rn(alpha, 6.0f);
        tame = tame_alpha(alpha);
        six_inv = __frcp_rn(six_alpha);
        alpha_d = static_cast<double>(alpha);
        nblk = bt.t[ti].nblk;
        view = smem_u32(&sh.view[ti]);
        tensor = ti;
      },
      [&](int ti) {
        hand_over(sh, ti, acc);
        hand_over_counters(sh, ti, zeros, wide);
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2&, auto next, unsigned int state_at) {
        PairBlock blk;
        unpack_pairs(v0, v1, blk);
        next();
        if (b >= nblk) return;
        uint8_t *packed, *scales;
        uint2* state;
        load_view(view, packed, scales, state);
        float bmax = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float lo, hi;
          halves(blk.w[i], lo, hi);
          bmax = fmaxf(bmax, fmaxf(fabsf(lo), fabsf(hi)));
        }
        if (bmax == 0.0f) {
          // all-zero block: codes carry the sign bits only, scale byte 0, left out of all sums
          unsigned int c0, c1;
          round_pairs(blk, 1.0f, c0, c1);
          reinterpret_cast<uint2*>(packed)[b] = make_uint2(c0, c1);
          put_scale(sh, bt.t[tensor], scales, b, 0);
          if (keep) put_state<S>(state, b, state_at, make_uint2(0u, 0u));
          ++zeros;
          return;
        }
        Found f;
        float v;
        if (tame) {
          const int d = max(e4m3_encode(quotient(bmax, six_alpha, six_inv)), 1);
          v = e4m3_value(d);
          const float s = __fmul_rn(alpha, v);
          FixedPairs fx;
          make_fixed_pairs(blk, fixed_scale(s), fx);   // bmax / s is below 9: v is bmax / (6 alpha) rounded, or its 2^-9
          unsigned int afix;
          round_pairs(blk, recip_fast(s), f.c0, f.c1);
          pair_code_sums(fx, f.c0, f.c1, afix, f.b4);
          f.d = d;
          // A = afix / (2 S)
          f.A = __fmul_rn(__uint2float_rn(afix), __uint_as_float((__float_as_uint(s) & 0x7F800000u) - (11u << 23)));
          // error minus sum W^2 = alpha (h e) 4 / S^2 with h = v S / 4, e = alpha h 4B - afix (v may be subnormal in E4M3,
          // never in binary32)
          const unsigned int s_exp = __float_as_uint(s) & 0x7F800000u;
          const double h = scaled_value(__float_as_uint(v), static_cast<int>(135u << 20) - static_cast<int>(s_exp >> 3));
          const double e = fma(alpha_d * h, uint_to_double(f.b4), -uint_to_double(afix));
          f.g = h * e * __hiloint2double(__double2hiint(alpha_d) + static_cast<int>(s_exp >> 2) - (272 << 20),
                                         __double2loint(alpha_d));
        } else {
          f = start_general(bt.t[tensor], b, alpha, &wide);
          v = e4m3_value(f.d);
        }
        if (!keep) {
          reinterpret_cast<uint2*>(packed)[b] = make_uint2(f.c0, f.c1);
          put_scale(sh, bt.t[tensor], scales, b, f.d);
        } else {
          put_state<S>(state, b, state_at,
                       make_uint2(__float_as_uint(f.A), pack_state(__float_as_uint(bmax) & 0x7F800000u, f.d, f.b4)));
        }
        // v^2 4B is exact in binary32: 8 + 12 significant bits (no Eq. 5 follows the last pass)
        if (!S::kFinal) acc[0] += static_cast<double>(__fmul_rn(__fmul_rn(v, v), __uint2float_rn(f.b4)));
        acc[1] += f.g;
      },
      fed);
}

// One iteration of Algorithm 1 for every block: Eq. 6 with the new alpha, App. B.3 candidate sets, Eq. 8 search,
// winner stored, sums of the next stage.  Codes and scale bytes are written when `emit` is set (the state after
// this iteration may be the one returned); the block states are kept when `keep` is set (another iteration may
// follow).
//   kMode 0  every multiplier in turn (the coupled arm with a grid)
//   kMode 1  one quantization scale per block (beta = 1): the codes are made once, only the E4M3 code is chosen
//   kMode 2  beta = 1 with the coupled scale: each E4M3 code rounds the block with its own value
//   kMode 3  the grid of App. B.3 around the stored scale (Sec. 3.3 alone), only the multipliers that can win
//   kMode 4  the grid of App. B.3 around the Eq. 6 solution with two E4M3 codes, only the multipliers that can win
//   kMode 5  the same for any number of codes, and for grids so short that a block's bracket often reaches past their
//            first or last multiplier
template <int kMode, typename S, typename B>
__device__ __forceinline__ void iterate_pass(S& sh, const B& bt, bool reverse, unsigned int emit, unsigned int keep) {
  asm volatile("" : "+r"(emit), "+r"(keep));   // in registers, not worked out again per tile
  const int n_dq = bt.t[0].n_dq, n_beta = bt.t[0].n_beta, flags = bt.t[0].flags;
  const bool keep_scale = kMode == 3 || (kMode != 4 && (flags & SOAR_FLAG_KEEP_BLOCK_SCALE) != 0);
  // multiplier index of a scale ratio: k = (ratio - 1) * 100 / step + n_beta / 2
  const float k_scale = 100.0f / static_cast<float>(max(bt.t[0].beta_step_pct, 1));
  const float k_off = static_cast<float>(n_beta / 2) - k_scale;
  const unsigned int pairs = smem_u32(sh.beta);
  float alpha = 1.0f, alpha_q = 0.0f;   // alpha_q: alpha / 4 where the fast path may run, else NaN (its guards fail)
  double alpha_d = 1.0;
  double acc[2] = {0.0, 0.0};           // 4 den, gsum
  unsigned int wide = 0, zeros = 0;
  int tensor = 0;
  unsigned int nblk = 0, view = 0;
  walk_tiles<kMode == 1, true>(
      sh, bt, reverse,
      [&](int ti) {
        alpha = sh.alpha[ti];
        alpha_q = (kMode != 0 && (n_dq <= 2 || kMode == 1) && tame_alpha(alpha)) ? 0.25f * alpha : __uint_as_float(0x7FC00000u);
        alpha_d = static_cast<double>(alpha);
        nblk = bt.t[ti].nblk;
        view = smem_u32(&sh.view[ti]);
        tensor = ti;
      },
      [&](int ti) {
        hand_over(sh, ti, acc);
        hand_over_counters(sh, ti, zeros, wide);
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2& state, auto next, unsigned int state_at) {
        PairBlock blk;
        unpack_pairs(v0, v1, blk);
        const uint2 st = state;
        next();
        const bool active = b < nblk && st.y != 0u;   // past the end, or an all-zero block: nothing to optimise
        // Eq. 6, A / (alpha B): with 4B and alpha / 4 the powers of two cancel exactly
        const float b4_prev = __fsub_rn(__uint_as_float((st.y & 0xFFFu) | 0x4B000000u), 8388608.0f);
        const float stored = e4m3_value(static_cast<int>((st.y >> 12) & 0x7Fu));
        const float D = __fmul_rn(alpha_q, b4_prev);
        float center = quotient(__uint_as_float(st.x), D, recip_fast(D));
        if (keep_scale) center = alpha_q > 0.0f ? stored : alpha_q;
        // Regular block: the center inside the normal E4M3 range (which also rejects B = 0 and a NaN alpha_q), so the
        // codes below and above it are its leading bits and the next.  The candidates are made and scored for every
        // lane; what an irregular block gets from that is overwritten by the general search below.
        bool direct = __float_as_uint(center) - 0x3C800000u < 0x43E00000u - 0x3C800000u;
        unsigned int dv0 = __float_as_uint(center) & 0xFFF00000u, dv1 = dv0 + 0x00100000u;
        if (kMode != 3 && kMode != 4 && n_dq == 1) {   // the nearest code alone
          dv0 = __float_as_uint(e4m3_value(e4m3_encode(center)));
          dv1 = dv0;
        }
        const float v0f = __uint_as_float(dv0), v1f = __uint_as_float(dv1);
        Candidate w;
        unsigned int dv_bits = dv0, s_exp;
        double g_scaled;
        if (kMode >= 3) {
          float y;
          asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(center));
          const float per_center = y * k_scale;
          // floor by a round-down addition: the index sits in the low bits of the sum.  Mode 3, where the center is an
          // E4M3 value and a multiplier often falls on a code exactly, takes the multiplier before the nearest one, and
          // three candidates.
          const float k_low = kMode == 3 ? k_off - 0.5f : k_off;
          const float t0 = __fadd_rd(__fmaf_rn(v0f, per_center, k_low), 12582912.0f);
          const float t1 = __fadd_rd(__fmaf_rn(v1f, per_center, k_low), 12582912.0f);
          int k0 = static_cast<int>(__float_as_uint(t0) & (SOAR_MAX_BETA - 1)), k1 = static_cast<int>(__float_as_uint(t1) & (SOAR_MAX_BETA - 1));
          if (kMode == 5) {
            k0 = max(0, min(n_beta - 2, __float_as_int(t0) - 0x4B400000));
            k1 = max(0, min(n_beta - 2, __float_as_int(t1) - 0x4B400000));
          }
          const uint2 q0 = lds64(pairs + 8u * static_cast<unsigned int>(k0));
          const uint2 q1 = lds64(pairs + 8u * static_cast<unsigned int>(k1));
          const pair_t cc = pair_of(center, center), aa = pair_of(-alpha, -alpha);
          const pair_t m0 = pair_mul(cc, pair_of(__uint_as_float(q0.x), __uint_as_float(q0.y)));
          const pair_t m1 = pair_mul(cc, pair_of(__uint_as_float(q1.x), __uint_as_float(q1.y)));
          float a0, b0f, a1, b1;
          halves(m0, a0, b0f);
          halves(m1, a1, b1);
          pair_t m2 = m0;
          if (kMode == 3) {   // {second multiplier above code 0's pair, the same for code 1}
            m2 = pair_mul(cc, pair_of(__uint_as_float(lds64(pairs + 8u * static_cast<unsigned int>(k0 + 1)).y),
                                      __uint_as_float(lds64(pairs + 8u * static_cast<unsigned int>(k1 + 1)).y)));
            halves(m2, b0f, b1);
          }
          // The pair of multipliers must enclose the code's value with a margin that covers the three roundings
          // from here to the scaled value (2^-24 each; see winning_range): 6 * 2^-24 does.  Where one of the two lies
          // inside the band, in one block of seven thousand, its neighbour on the other side can win too.
          constexpr float kUnder = 1.0f - 0x1.8p-22f, kOver = 1.0f + 0x1.8p-22f;
          // a (1 + margin) - v and b (1 - margin) - v of either code: enclosed when the first is negative and the second is
          // not (a first one of zero counts as not enclosed: the third multiplier is then looked at without need)
          const pair_t margins = pair_of(kOver, kUnder);
          float lo0, hi0, lo1, hi1;
          halves(pair_fma(pair_of(a0, b0f), margins, pair_of(-v0f, -v0f)), lo0, hi0);
          halves(pair_fma(pair_of(a1, b1), margins, pair_of(-v1f, -v1f)), lo1, hi1);
          const bool below0 = __float_as_int(lo0) < 0, above0 = __float_as_int(hi0) >= 0;
          const bool below1 = __float_as_int(lo1) < 0, above1 = __float_as_int(hi1) >= 0;
          const bool enclosed =
              (__float_as_int(lo0) & __float_as_int(lo1) & ~(__float_as_int(hi0) | __float_as_int(hi1))) < 0;
          // Mode 5, where the grid ends before the band does: one multiplier is all that can win, the first one when
          // even its divisor lies beyond the band, the last one when even its divisor lies before it.  The pair then
          // holds that multiplier twice.
          bool low0 = false, low1 = false, high0 = false, high1 = false;
          if (kMode == 5) {
            low0 = k0 == 0 && a0 >= v0f * kOver;
            high0 = k0 == n_beta - 2 && b0f <= v0f * kUnder;
            low1 = k1 == 0 && a1 >= v1f * kOver;
            high1 = k1 == n_beta - 2 && b1 <= v1f * kUnder;
          }
          // divisors, negated as pair_recip wants them
          pair_t n0 = pair_mul(aa, m0), n1 = pair_mul(aa, m1);
          if (kMode == 5) {
            float lo, hi;
            halves(n0, lo, hi);
            n0 = pair_of(high0 ? hi : lo, low0 ? lo : hi);
            halves(n1, lo, hi);
            n1 = pair_of(high1 ? hi : lo, low1 ? lo : hi);
          }
          float s00, s01;
          halves(n0, s00, s01);
          s_exp = __float_as_uint(s00) & 0x7F800000u;
          // the largest magnitude of the block below 32 times the smallest scale, from the exponents
          direct = direct && st.y < s_exp + (5u << 23);
          if (kMode == 5) direct = direct && ((below0 && above0) || low0 || high0) && ((below1 && above1) || low1 || high1);
          if (kMode == 3) direct = direct && enclosed;
          FixedPairs fx;
          make_fixed_pairs(blk, __uint_as_float((264u << 23) - s_exp), fx);
          // h = dv S / 4; the exponent of S / 4 is 135 less s's biased one
          const int k_field = static_cast<int>(135u << 20) - static_cast<int>(s_exp >> 3);
          const double h0 = scaled_value(dv0, k_field), h1 = scaled_value(dv1, k_field);
          const double rho0 = alpha_d * h0, rho1 = alpha_d * h1;
          Candidate x, w2, y2;   // (four scored before any is dropped: independent work for the scheduler)
          float r00, r01, r10, r11;
          pair_recip(n0, r00, r01);
          pair_recip(n1, r10, r11);
          score_pairs(blk, fx, r00, rho0, w);
          score_pairs(blk, fx, r01, rho0, w2);
          score_pairs(blk, fx, r10, rho1, x);
          score_pairs(blk, fx, r11, rho1, y2);
          if (w2.e < w.e) w = w2;
          if (y2.e < x.e) x = y2;
          if (kMode == 3) {
            float r02, r12;
            pair_recip(pair_mul(aa, m2), r02, r12);
            score_pairs(blk, fx, r02, rho0, y2);
            if (y2.e < w.e) w = y2;
            score_pairs(blk, fx, r12, rho1, y2);
            if (y2.e < x.e) x = y2;
          }
          if (kMode == 4 && !enclosed) {
            // the third multiplier: before the pair when the first of it is not below the band, after it when the second
            // is not above; equal errors go to the earlier one
            if (!below0 || !above0) {
              const uint2 q = lds64(pairs + 8u * static_cast<unsigned int>(below0 ? k0 + 1 : max(k0 - 1, 0)));
              const float m = __uint_as_float(below0 ? q.y : q.x);
              score_pairs(blk, fx, recip_fast(grid_divisor(alpha, center, m)), rho0, y2);
              if (y2.e < w.e || (!below0 && y2.e == w.e)) w = y2;
            }
            if (!below1 || !above1) {
              const uint2 q = lds64(pairs + 8u * static_cast<unsigned int>(below1 ? k1 + 1 : max(k1 - 1, 0)));
              const float m = __uint_as_float(below1 ? q.y : q.x);
              score_pairs(blk, fx, recip_fast(grid_divisor(alpha, center, m)), rho1, y2);
              if (y2.e < x.e || (!below1 && y2.e == x.e)) x = y2;
            }
          }
          // equal errors: the earlier multiplier, as in grid order (the second code's are never earlier)
          const double g0 = h0 * w.e, g1 = h1 * x.e;
          g_scaled = g0;
          if (g1 < g0) { w = x; g_scaled = g1; dv_bits = dv1; }
        } else if (kMode == 1 || kMode == 2) {
          const float s0 = __fmul_rn(alpha, kMode == 1 ? center : v0f), s1 = __fmul_rn(alpha, v1f);
          s_exp = __float_as_uint(s0) & 0x7F800000u;
          direct = direct && st.y < s_exp + (5u << 23);
          FixedPairs fx;
          make_fixed_pairs(blk, fixed_scale(s0), fx);
          const int k_field = static_cast<int>(135u << 20) - static_cast<int>(s_exp >> 3);
          const double h0 = scaled_value(dv0, k_field), h1 = scaled_value(dv1, k_field);
          const double rho0 = alpha_d * h0, rho1 = alpha_d * h1;
          score_pairs(blk, fx, recip_fast(s0), rho0, w);
          g_scaled = h0 * w.e;
          if (kMode == 1 && n_dq > 2) {
            // wider code windows: n_dq / 2 codes at or below the center, n_dq / 2 above, clipped
            const int d_lo = static_cast<int>(dv0 >> 20) - 960 - (n_dq / 2 - 1);
            g_scaled = __longlong_as_double(0x7FF0000000000000ll);
            for (int i = 0; i < n_dq / 2 * 2; ++i) {
              const float dv = e4m3_value(clip_code(d_lo + i));
              const double h = static_cast<double>(dv) * __hiloint2double(k_field + (1023 << 20), 0);
              const double g = h * fma(alpha_d * h, uint_to_double(w.b4), -uint_to_double(w.afix));
              if (g < g_scaled) { g_scaled = g; dv_bits = __float_as_uint(dv); }
            }
          } else if (kMode == 1) {
            const double g1 = h1 * fma(rho1, uint_to_double(w.b4), -uint_to_double(w.afix));
            if (g1 < g_scaled) { g_scaled = g1; dv_bits = dv1; }
          } else if (n_dq == 2) {
            Candidate x;
            score_pairs(blk, fx, recip_fast(s1), rho1, x);
            const double g1 = h1 * x.e;
            if (g1 < g_scaled) { w = x; g_scaled = g1; dv_bits = dv1; }
          }
        } else {
          s_exp = 0u;
          g_scaled = 0.0;
          w.c0 = w.c1 = w.afix = w.b4 = 0u;
          direct = false;
        }
        // A = afix / (2 S); error minus sum W^2 = alpha (h e) 4 / S^2
        const float v = __uint_as_float(dv_bits), A = __fmul_rn(__uint2float_rn(w.afix), __uint_as_float(s_exp - (11u << 23)));
        const int d = (kMode == 1 && n_dq > 2) ? e4m3_encode(v) : static_cast<int>(dv_bits >> 20) - 960;
        const double g_scale = __hiloint2double(__double2hiint(alpha_d) + static_cast<int>(s_exp >> 2) - (272 << 20),
                                          __double2loint(alpha_d));
        if (active && !direct) {
          const float B0 = 0.25f * b4_prev;   // all codes zero keeps the stored scale
          center = (B0 > 0.0f && !keep_scale) ? __fdiv_rn(__uint_as_float(st.x), __fmul_rn(alpha, B0)) : stored;
          const Found f = kMode == 0 ? search_every(bt.t[tensor], b, alpha, center, sh.beta, n_beta, n_dq,
                                                    (flags & SOAR_FLAG_COUPLED_SCALE) != 0, &wide)
                                     : search_general<kMode>(bt.t[tensor], b, alpha, center, sh.beta, n_beta, n_dq, k_scale,
                                                             k_off, &wide);
          // (stored here: merging it into the common path costs that path a move per value)
          uint8_t *packed, *scales;
          uint2* states;
          load_view(view, packed, scales, states);
          if (emit) {
            reinterpret_cast<uint2*>(packed)[b] = make_uint2(f.c0, f.c1);
            scales[b] = static_cast<uint8_t>(f.d);
          }
          if (keep)
            put_state<S>(states, b, state_at, make_uint2(__float_as_uint(f.A), pack_state(st.y & 0x7F800000u, f.d, f.b4)));
          const float fv = e4m3_value(f.d);
          acc[0] += static_cast<double>(__fmul_rn(__fmul_rn(fv, fv), __uint2float_rn(f.b4)));
          acc[1] += f.g;
        } else if (active) {
          uint8_t *packed, *scales;
          uint2* states;
          load_view(view, packed, scales, states);
          if (emit) {
            reinterpret_cast<uint2*>(packed)[b] = make_uint2(w.c0, w.c1);
            scales[b] = static_cast<uint8_t>(d);
          }
          if (keep)
            put_state<S>(states, b, state_at, make_uint2(__float_as_uint(A), pack_state(st.y & 0x7F800000u, d, w.b4)));
          // v^2 4B is exact in binary32: 8 + 12 significant bits
          acc[0] += static_cast<double>(__fmul_rn(__fmul_rn(v, v), __uint2float_rn(w.b4)));
          acc[1] = fma(g_scaled, g_scale, acc[1]);
        }
      });
}

// ------------------------------------------------------------------ report

// Replays the early-stop rule over the stage sums of one tensor, writes alpha and the report.  `scratch`: 4 * 65 doubles of
// shared memory.  `latest`, if not null, holds num, den, gsum of stage `latest_stage`, which the header may not show yet.
__device__ __forceinline__ void write_report(const Params& p, float* out_alpha, soar_result* res, double* scratch,
                                             const double* latest, int latest_stage) {
  constexpr int kN = SOAR_MAX_ITERS + 1;
  double *s_num = scratch, *s_den = scratch + kN, *s_sse = scratch + 2 * kN, *s_ta = scratch + 3 * kN;
  __shared__ int s_iters;
  const Ws* ws = p.ws;
  const unsigned int amax_bits = __ldcg(&ws->amax_bits), error = __ldcg(&ws->error);
  const double sumsq = __ldcg(&ws->sumsq);
  const int st = status_from_amax(amax_bits);
  for (int i = threadIdx.x; i < kN; i += blockDim.x) {
    const bool used = i <= p.max_iters;
    const bool here = latest != nullptr && i == latest_stage;
    s_num[i] = here ? latest[0] : used ? __ldcg(&ws->num[i]) : 0.0;
    s_den[i] = here ? latest[1] : used ? __ldcg(&ws->den[i]) : 0.0;
    const double gsum = here ? latest[2] : used ? __ldcg(&ws->gsum[i]) : 0.0;
    s_sse[i] = (used && st == 0) ? fmax(sumsq + gsum, 0.0) : 0.0;
    s_ta[i] = 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float alpha = (st & SOAR_STATUS_ZERO_TENSOR) ? 1.0f : __fdiv_rn(bits_to_mag(amax_bits), 2688.0f);
    int iters = 0;
    s_ta[0] = static_cast<double>(alpha);
    if (st == 0 && error == 0) {
      double prev = s_sse[0];
      for (int i = 0; i < p.max_iters; ++i) {
        if (s_den[i] > 0.0 && !(p.flags & SOAR_FLAG_KEEP_ALPHA)) alpha = static_cast<float>(s_num[i] / s_den[i]);
        const double cur = s_sse[i + 1];
        iters = i + 1;
        s_ta[iters] = static_cast<double>(alpha);
        if (stops_after(prev, cur, p.early_stop_rel)) break;
        prev = cur;
      }
    }
    s_iters = iters;
    *out_alpha = alpha;
    if (res != nullptr) {
      res->status = st | ((error & kErrWait) ? SOAR_STATUS_INTERNAL : 0) | ((error & kErrWeight) ? SOAR_STATUS_BAD_WEIGHT : 0);
      res->iters_run = iters;
      res->alpha = alpha;
      res->amax = bits_to_mag(amax_bits);
      res->sse = s_sse[iters];
      res->sse_init = s_sse[0];
      res->sumsq = (st & SOAR_STATUS_ZERO_TENSOR) ? 0.0 : sumsq;
      res->zero_blocks = static_cast<int64_t>(__ldcg(&ws->zero_blocks));
      res->wide_candidates = static_cast<int64_t>(__ldcg(&ws->wide));
    }
  }
  __syncthreads();
  if (res != nullptr) {
    const int iters = s_iters;
    for (int i = threadIdx.x; i < kN; i += blockDim.x) {
      res->trace_alpha[i] = (i <= iters) ? s_ta[i] : 0.0;
      res->trace_sse[i] = (i <= iters) ? s_sse[i] : 0.0;
    }
  }
  __syncthreads();
}

// The 128x4-tiled copy of a tensor's scales.  A thread makes 16 consecutive bytes of a tile: rows r, r + 32, r + 64, r + 96
// of four scale columns, so a warp stores a whole 512-byte tile; rows and columns past the end are zero.
__device__ __forceinline__ void tile_scales(const Params& p, unsigned int rows, uint8_t* sw) {
  const unsigned int nbc = p.nbc, col_tiles = (nbc + 3) / 4;
  const unsigned int tiles = (rows + 127) / 128 * col_tiles;
  const bool words = nbc % 4 == 0 && reinterpret_cast<uintptr_t>(p.scales) % 4 == 0;
  const bool out16 = reinterpret_cast<uintptr_t>(sw) % 16 == 0;
  const unsigned int lane = threadIdx.x & 31u;
  const unsigned int warps = blockDim.x >> 5;
  for (unsigned int tile = blockIdx.x * warps + (threadIdx.x >> 5); tile < tiles; tile += gridDim.x * warps) {
    const unsigned int tr = tile / col_tiles, col = (tile - tr * col_tiles) * 4;
    unsigned int w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned int row = tr * 128 + lane + 32 * i;
      w[i] = 0;
      if (row < rows) {
        const uint8_t* src = p.scales + static_cast<size_t>(row) * nbc + col;
        if (words) {
          w[i] = *reinterpret_cast<const unsigned int*>(src);
        } else {
          for (unsigned int c = 0; c < 4; ++c)
            if (col + c < nbc) w[i] |= static_cast<unsigned int>(src[c]) << (8 * c);
        }
      }
    }
    uint8_t* dst = sw + static_cast<size_t>(tile) * 512 + lane * 16;
    if (out16) {
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      for (int i = 0; i < 16; ++i) dst[i] = static_cast<uint8_t>(w[i >> 2] >> (8 * (i & 3)));
    }
  }
}

// ------------------------------------------------------------------ the kernel

// Deterministic mode: the per-CTA sums of the stage just finished, added in index order (every CTA computes the same
// bits); CTA 0 files them in the header.  s is the stage about to run.
__device__ __forceinline__ void gather_sums(const Batch& bt, int s, double (*latest)[3]) {
  for (int ti = threadIdx.x >> 5; ti < bt.n; ti += kQWarps) {
    const Params& p = bt.t[ti];
    if (s == kQStageInit) {
      const double v = ordered_sum(p.det->sumsq, gridDim.x);
      if ((threadIdx.x & 31) == 0 && blockIdx.x == 0) p.ws->sumsq = v;
      continue;
    }
    const int q = s - kQStageIterate;
    double v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = ordered_sum(p.det->stage[q & 1][i], gridDim.x);
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int i = 0; i < 3; ++i) latest[ti][i] = v[i];
      if (blockIdx.x == 0) {
        p.ws->num[q] = v[0];
        p.ws->den[q] = v[1];
        p.ws->gsum[q] = v[2];
      }
    }
  }
}

// Stages [stage_lo, stage_hi) of a call: amax, init, max_iters iterations, the report, the tiled scales.  A launch
// over more than one stage is cooperative: its CTAs meet between stages.
template <bool kDet, typename S, typename Passes>
__device__ __forceinline__ void run_stages(S& sh, double (*s_latest)[3], const Batch& bt, const Reports& rp, int stage_lo,
                                           int stage_hi, const Passes& passes) {
  const int tid = threadIdx.x;
  const int T = bt.t[0].max_iters, report = kQStageIterate + T, flags = bt.t[0].flags;
  if (tid < bt.n) {
    sh.view[tid].packed = bt.t[tid].packed;
    sh.view[tid].scales = bt.t[tid].scales;
    sh.view[tid].state = bt.t[tid].state;
    sh.view[tid].tiled = nullptr;
  }
  if (tid < kMaxBatch) {
    sh.acc[tid][0] = sh.acc[tid][1] = 0.0;
    sh.amax[tid] = sh.zeros[tid] = sh.wide[tid] = sh.wide_high[tid] = 0u;
    if (kDet)
      for (int w = 0; w < kQWarps; ++w) sh.part[tid][w][0] = sh.part[tid][w][1] = 0.0;
  }
  if (tid == 0) {
    sh.visited = 0u;
    sh.failed = 0;
    sh.run = (1u << bt.n) - 1u;
  }
  if (Passes::kGrid) {
    const int n_beta = bt.t[0].n_beta, step = bt.t[0].beta_step_pct;
    for (int k = tid; k < n_beta; k += kQThreads) {
      const float lo = static_cast<float>((100.0 + static_cast<double>((k - n_beta / 2) * step)) / 100.0);
      const float hi = static_cast<float>((100.0 + static_cast<double>((k + 1 - n_beta / 2) * step)) / 100.0);
      sh.beta[k] = make_float2(lo, hi);
    }
  }
  __syncthreads();
  bool any_tiled = false;
  for (int i = 0; i < bt.n; ++i) any_tiled = any_tiled || rp.scales_sw[i] != nullptr;
  unsigned int target = 0;
  int latest_stage = -1;   // deterministic mode: the stage s_latest holds
  bool stopped = false;    // left the iterations before the last one
  int s = stage_lo;
  while (s < report && s < stage_hi) {
    // head of stage s: every tensor's alpha, and which tensors it works on
    if (kDet && s > kQStageAmax) {
      gather_sums(bt, s, s_latest);
      latest_stage = s - kQStageIterate;
      __syncthreads();
    }
    if (s == kQStageInit) {
      if (tid < 32) {
        bool go = false;
        if (tid < bt.n) {
          const unsigned int amax_bits = __ldcg(&bt.t[tid].ws->amax_bits);
          sh.alpha[tid] = amax_bits == 0 ? 1.0f : __fdiv_rn(bits_to_mag(amax_bits), 2688.0f);
          go = !(status_from_amax(amax_bits) & (SOAR_STATUS_NONFINITE | SOAR_STATUS_RANGE)) &&
               __ldcg(&bt.t[tid].ws->error) == 0u;
        }
        const unsigned int run = __ballot_sync(0xFFFFFFFFu, go);
        if (tid == 0) sh.run = run;
      }
    } else if (s >= kQStageIterate) {
      const int t = s - kQStageIterate;
      if (tid < 32) {
        bool go = false;
        if (tid < bt.n) {
          const Params& p = bt.t[tid];
          if (s == stage_lo) {   // a stage on its own: everything from the header
            int run;
            float alpha;
            iteration_head(p, t, alpha, run, kDet ? s_latest[tid] : nullptr);
            sh.alpha[tid] = alpha;
            go = run != 0;
          } else if ((sh.run >> tid) & 1u) {
            const double num = kDet ? s_latest[tid][0] : __ldcg(&p.ws->num[t]);
            const double den = kDet ? s_latest[tid][1] : __ldcg(&p.ws->den[t]);
            const double gsum = kDet ? s_latest[tid][2] : __ldcg(&p.ws->gsum[t]);
            const double cur = fmax(__ldcg(&p.ws->sumsq) + gsum, 0.0);
            go = t == 0 ? __ldcg(&p.ws->amax_bits) != 0u : !stops_after(sh.sse[tid], cur, p.early_stop_rel);
            if (go) {
              sh.sse[tid] = cur;
              if (den > 0.0 && !(flags & SOAR_FLAG_KEEP_ALPHA)) sh.alpha[tid] = static_cast<float>(num / den);   // Eq. 5
            }
          }
        }
        const unsigned int run = __ballot_sync(0xFFFFFFFFu, go);
        if (tid == 0) sh.run = run;
      }
    }
    __syncthreads();
    if (s >= kQStageIterate && sh.run == 0) {   // every tensor has stopped (Sec. 4.1): all CTAs see it alike
      s = report;
      stopped = true;
      break;
    }
    lay_out_pass(sh, bt);
    if (s == kQStageAmax) {
      passes.amax(sh, bt);
      file_sums(sh, bt, -1);
    } else if (s == kQStageInit) {
      passes.init(sh, bt);
      file_sums(sh, bt, 0);
    } else {
      const int t = s - kQStageIterate;
      const bool last = t == T - 1;
      passes.iterate(sh, bt, (t & 1) != 0, bt.t[0].early_stop_rel > 0.0f || last, !last);
      file_sums(sh, bt, t + 1);
    }
    ++s;
    if (s < stage_hi) {
      target += gridDim.x;
      if (s == report && blockIdx.x >= static_cast<unsigned int>(bt.n) && !(any_tiled && stage_hi > report + 1)) {
        // nothing left to do for this CTA: it arrives and leaves
        if (tid == 0) {
          __threadfence();
          if (!bt.idle) atomicAdd(arrivals(bt), 1u);
        }
        return;
      }
      if (!grid_sync(sh, bt, target)) {
        // the wait ran out: say so in the reports and leave
        if (tid < bt.n && rp.result[tid] != nullptr) {
          rp.result[tid]->status = SOAR_STATUS_INTERNAL;
          rp.result[tid]->iters_run = 0;
        }
        return;
      }
    }
  }
  if (s >= stage_hi) return;
  if (s == report && stage_lo <= report) {
    if (kDet && !stopped) {
      gather_sums(bt, report, s_latest);
      latest_stage = T;
      __syncthreads();
    }
    for (int ti = blockIdx.x; ti < bt.n; ti += gridDim.x)
      write_report(bt.t[ti], rp.alpha[ti], rp.result[ti], reinterpret_cast<double*>(sh.ring), kDet ? s_latest[ti] : nullptr,
                   latest_stage);
  }
  if (any_tiled && stage_hi > report + 1)
    for (int ti = 0; ti < bt.n; ++ti)
      if (rp.scales_sw[ti] != nullptr) tile_scales(bt.t[ti], rp.rows[ti], rp.scales_sw[ti]);
}

template <int kMode>
struct SearchPasses {
  static constexpr bool kGrid = kMode == 0 || kMode >= 3;
  template <typename S>
  __device__ __forceinline__ void amax(S& sh, const Batch& bt) const { amax_pass(sh, bt); }
  template <typename S>
  __device__ __forceinline__ void init(S& sh, const Batch& bt) const { init_pass(sh, bt); }
  template <typename S>
  __device__ __forceinline__ void iterate(S& sh, const Batch& bt, bool reverse, bool emit, bool keep) const {
    iterate_pass<kMode>(sh, bt, reverse, emit, keep);
  }
};

template <int kMode, bool kDet>
__global__ void __launch_bounds__(kQThreads, 2)
quantize_kernel(const __grid_constant__ Batch bt, const __grid_constant__ Reports rp, int stage_lo, int stage_hi) {
  __shared__ QShared<kDet> sh;
  __shared__ double s_latest[kDet ? kMaxBatch : 1][3];
  run_stages<kDet>(sh, s_latest, bt, rp, stage_lo, stage_hi, SearchPasses<kMode>{});
}
