// MXFP4 (Sec. 4.3, "DSS on MXFP4").  Included by soar.cu after quantize_kernel.cuh, whose tile walk it uses.
//
// The other microscaling format: E2M1 elements in blocks of 32 with one shared power-of-two scale (an E8M0 byte, value
// 2^(code - 127)) and no tensor-wide scale.  The paper reports results and no procedure; the reading built here (the
// oracle's) is Sec. 3.3 (i)-(ii) with alpha = 1:
//   plain rule  shared exponent floor(log2 bmax) - 2, elements rounded to nearest even, saturated;
//   search      high-precision scale D* = fl(bmax / 6) (Eq. 1); dequantization candidates the n_dq E8M0 values around
//               D* (App. B.3's rule on powers of two; for two candidates the plain exponent is always one of them);
//               quantization candidates D* * beta_k on App. B.3's grid; Eq. 8 over all pairs, first minimum in
//               (beta, code) order.
// One pass over W, no workspace.  A lane has a block of 32, in registers, and loads its next one (64 bytes, with two
// 256-bit loads) while it works on it.
//
// With a power-of-two scale everything Eq. 8 compares is an integer: with magnitudes in units of 2^(cf - 11), the error
// minus sum W^2 under the scale 2^cf is (4B << 9) - A' in those units, and under 2^(cf + 1) twice (4B << 10) - A'.  So a
// candidate costs no binary64 operation, and exactly equal errors compare equal.  They are common (bf16 inputs sit exactly
// on midpoints in a fifth of all blocks): inside the bracket the grid's order decides, outside it every code change changes
// the error strictly (see winning_range).
//
// Two multipliers per code are enough, the last one below the code's band and its successor, also where that successor lies
// in the band, which it does in one block in seventeen: a bf16 magnitude over a power of two has eight significant bits,
// so it is a rounding midpoint exactly or misses it by 2^-8, far more than the band's 2^-21; the successor's codes are then
// nearest ones, ties either way, its error is the least there is, and only an earlier multiplier can share the first place.
//
// The search is bound by instruction issue, 300 per sixteen elements in 71 % of the cycles: 28672 x 8192 171 us (594 MB:
// 3.5 TB/s).  The plain rule, 146 instructions in 55 % of the cycles, waits for its loads: 115 us, 5.1 TB/s.  Two lanes to
// a block, which each did the whole of the block's own work (centre, brackets, reciprocals) and exchanged their sums, took 373
// instructions and 216 us, 211 and 122 us.  The two halves of a block go through the four candidates one after the other; both
// at once spill (238 us).  Other forms on that shape, with two lanes and now: a base aligned to 16 bytes only 229 -> 183 us (plain
// rule 122.5 -> 121), a row stride 8 above the columns 230 -> 184 (151 -> 123), one code on five multipliers 426 -> 322, four codes
// on 101 1010 -> 642, where the general rules read the matrix a second time.

#pragma once

struct MxArgs {
  Single m;                 // (its block and tile counts are those of blocks of 16, as Params says)
  uint8_t* scales;
  soar_mx_result* res;
  unsigned long long tag;   // opens the result for sums (see mx_kernel)
  int chained;              // clear_mx_kernel has cleared the result
  int n_dq, n_beta, step_pct;
  int idle;                 // test hook: CTA 0 never opens the result, the waits for it run out
};

struct __align__(128) MxShared {
  float2 beta[SOAR_MAX_BETA];
  double part[kQWarps][2];
  unsigned int amax, zeros, wide, wide_high;
};

// A block of 32 as two of 16, for the general rules.
struct MxBlock {
  Block half[2];
  Fixed fix[2];
};
__device__ __forceinline__ void load_mx_block(const Params& p, unsigned int b, MxBlock& x) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint4 v0, v1;
    load_block(p, 2 * b + i, v0, v1);
    unpack_block(v0, v1, x.half[i]);
    make_fixed(x.half[i], x.fix[i]);
  }
}
__device__ __forceinline__ void mx_codes(const MxBlock& x, float r, uint4& c) {
  round_block(x.half[0], r, c.x, c.y);
  round_block(x.half[1], r, c.z, c.w);
}
// Its sums under reciprocal scale r, as block_sums.
__device__ __forceinline__ void mx_block_sums(const MxBlock& x, float r, double& A, double& B, unsigned int& wide) {
  A = B = 0.0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    unsigned int c0, c1;
    double a, b;
    round_block(x.half[i], r, c0, c1);
    block_sums(x.half[i], x.fix[i], r, c0, c1, a, b, wide);
    A += a;
    B += b;
  }
}

struct MxFound {
  double g;      // error minus sum W^2
  uint4 codes;
  int code;      // of the scale
};

// A block by the general rules, any number of codes, any grid, any magnitude.  kSearch as mx_kernel.
template <int kSearch>
__device__ __forceinline__ void mx_general(const Params& p, unsigned int b, const float2* s_beta, int n_dq, int n_beta, int step_pct,
                                           MxFound& f, unsigned int& zeros, unsigned int& wide) {
  MxBlock blk;
  load_mx_block(p, b, blk);
  const float bmax = fmaxf(blk.half[0].bmax, blk.half[1].bmax);
  f.g = 0.0;
  f.code = 0;
  float best_r = 0.0f;
  if (!(bmax >= 0x1p-120f)) {
    // zero (or vanishing) block: scale code 0, zero codes with the inputs' sign bits
    ++zeros;
  } else if (kSearch == 0) {
    const int X = static_cast<int>(__float_as_uint(bmax) >> 23) - 129;
    best_r = __uint_as_float(static_cast<unsigned int>(127 - X) << 23);   // 2^-X
    double A, B;
    mx_block_sums(blk, best_r, A, B, wide);
    const double sd = __hiloint2double((X + 127 + 896) << 20, 0);         // 2^X
    f.g = sd * fma(sd, B, -2.0 * A);
    f.code = X + 127;
  } else {
    const float center = __fdiv_rn(bmax, 6.0f);
    const int cf = static_cast<int>(__float_as_uint(center) >> 23);      // biased: value 2^(cf - 127) <= center
    int d_lo, d_hi;
    if (n_dq <= 1) {
      const float mid = __uint_as_float((static_cast<unsigned int>(cf) << 23) | 0x400000u);   // 1.5 * 2^(cf - 127)
      d_lo = d_hi = center > mid ? cf + 1 : cf;
    } else {
      d_lo = cf - (n_dq / 2 - 1);
      d_hi = cf + n_dq / 2;
    }
    f.g = __longlong_as_double(0x7FF0000000000000ll);
    const bool bracketed = n_beta >= kBracketMinBeta && step_pct >= 1;
    const float k_scale = 100.0f / static_cast<float>(max(step_pct, 1));
    const float k_off = static_cast<float>(n_beta / 2) - k_scale;
    const float per_center = __fdividef(k_scale, center);
    int best_k = 0;
    // bracketed: per code the multipliers of winning_range; otherwise every multiplier, all codes scored on it
    for (int d0 = d_lo, prev = -1; d0 <= (bracketed ? d_hi : d_lo); ++d0) {
      int ka = 0, kb = n_beta - 1;
      if (bracketed) {
        const int dc = max(0, min(254, d0));
        if (dc == prev) continue;   // clipping at the ends of the E8M0 range repeats a code
        prev = dc;
        const float sdf = static_cast<float>(__hiloint2double((dc + 896) << 20, 0));   // exact (2^-127 is a binary32 subnormal)
        winning_range(s_beta, n_beta, 1.0f, center, __fmul_rn(sdf, 1.0f - 0x1p-21f), __fmul_rn(sdf, 1.0f + 0x1p-21f),
                      __float2int_rd(__fmaf_rn(sdf, per_center, k_off)), ka, kb);
      }
      for (int k = ka; k <= kb; ++k) {
        const float r = recip_scale(1.0f, __fmul_rn(center, s_beta[k].x));
        double A, B;
        mx_block_sums(blk, r, A, B, wide);
        for (int d = d0; d <= (bracketed ? d0 : d_hi); ++d) {
          const int dc = max(0, min(254, d));
          if (!bracketed && d > d0 && dc == max(0, min(254, d - 1))) continue;
          const double sd = __hiloint2double((dc + 896) << 20, 0);
          const double g = sd * fma(sd, B, -2.0 * A);
          // equal errors: the earlier multiplier, then the smaller code, as in grid order
          if (g < f.g || (bracketed && g == f.g && k < best_k)) {
            f.g = g;
            best_r = r;
            f.code = dc;
            best_k = k;
          }
        }
      }
    }
  }
  mx_codes(blk, best_r, f.codes);
}

// Half of a candidate: codes, and (4B << shift) - A'.
__device__ __forceinline__ int mx_score(const PairBlock& b, const FixedPairs& fx, float r, int shift, unsigned int& c0, unsigned int& c1) {
  unsigned int afix, b4;
  round_pairs(b, r, c0, c1);
  pair_code_sums(fx, c0, c1, afix, b4);
  return static_cast<int>(b4 << shift) - static_cast<int>(afix);
}

__device__ __forceinline__ void clear_mx(soar_mx_result* res) {
  res->status = 0;
  res->amax_bits = 0u;
  res->amax = 0.0f;
  res->pad_ = 0;             // arrivals
  res->sse = 0.0;            // sum of the blocks' errors minus sum W^2
  res->sumsq = 0.0;
  res->zero_blocks = 0;
  res->wide_candidates = 0;
}
__global__ void clear_mx_kernel(soar_mx_result* res) {
  let_next_begin();   // (it waits for this kernel's end)
  after_previous();
  if (threadIdx.x == 0) clear_mx(res);
}

// kSearch 0: the plain rule; 1: the search by the general rules; 2: the search with two codes on a grid that starts at
// half the center or below and has steps of a quarter or less (the paper's: 0.50 .. 1.50 in hundredths): two multipliers
// per code in straight line.
//
// The result is also where the sums meet: CTA 0 clears it while the tiles are on their way and opens it by writing the
// call's tag to `reserved`, the other CTAs add when they have seen the tag, and the one that comes last turns the sums
// into the report (and `reserved` into what it documents, so that the replay of a captured call does not find the tag).
// No memset before, no kernel after.  Larger matrices (launch_mx) have it cleared by a kernel of its own that this one is
// chained to: CTAs that wait for nobody need no cooperative launch, whose gap to the launch before is longer (12288 x 4096:
// 2.4 us less with the search, 1.8 by the plain rule; 1024 x 4096: 11.7 -> 8.8).
template <int kSearch, bool kPlain>
__global__ void __launch_bounds__(kQThreads, 2) mx_kernel(const __grid_constant__ MxArgs a) {
  __shared__ MxShared sh;
  const Params& p = a.m.t[0];
  const unsigned int tid = threadIdx.x, lane = tid & 31u;
  soar_mx_result* const res = a.res;
  if (tid == 0) sh.amax = sh.zeros = sh.wide = sh.wide_high = 0u;
  if (kSearch)
    for (int k = static_cast<int>(tid); k < a.n_beta; k += kQThreads) {
      const float lo = static_cast<float>((100.0 + static_cast<double>((k - a.n_beta / 2) * a.step_pct)) / 100.0);
      const float hi = static_cast<float>((100.0 + static_cast<double>((k + 1 - a.n_beta / 2) * a.step_pct)) / 100.0);
      sh.beta[k] = make_float2(lo, hi);
    }
  if (a.chained) after_previous();
  if (!a.chained && blockIdx.x == 0 && tid == 32) {
    clear_mx(res);
    if (!a.idle) asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(&res->reserved), "l"(a.tag) : "memory");
  }
  __syncthreads();
  const float sixth = __frcp_rn(6.0f);
  const int n_beta = a.n_beta;
  const float k_scale = 100.0f / static_cast<float>(max(a.step_pct, 1));
  // (a pair is chosen so that a multiplier in the code's band is its second: see below)
  const float k_off = static_cast<float>(n_beta / 2) - k_scale - 5e-4f;
  const unsigned int pairs = smem_u32(sh.beta);
  double acc = 0.0, sq[2] = {0.0, 0.0};
  unsigned int zeros = 0, wide = 0, mx = 0;
  uint8_t* packed = p.packed;
  uint8_t* scales = a.scales;
  const unsigned char* w = reinterpret_cast<const unsigned char*>(p.W);
  const unsigned int nblk = p.nblk >> 1, step = gridDim.x * kQThreads;   // blocks of 32
  __builtin_assume(__isGlobal(packed) && __isGlobal(scales));
  uint4 v[4];
  auto fetch = [&](unsigned int b, int i) {   // half i of block b
    if (b >= nblk) return;
    if constexpr (kPlain) load_block32(w + static_cast<size_t>(b) * 64 + i * 32, v[2 * i], v[2 * i + 1]);
    else load_block(p, 2 * b + i, v[2 * i], v[2 * i + 1]);
  };
  // The lane's irregular blocks are marked with a scale byte no block has and made after the others, from the first one on
  // (the general rules called in the loop cost its common path spills: 12288 x 4096 43.9 against 41.1 us).
  unsigned int first_marked = kSearch == 1 ? first_block() : nblk;
  fetch(first_block(), 0);
  fetch(first_block(), 1);
  for (unsigned int b = first_block(); b < nblk; b += step) {
    const unsigned int u[2][8] = {{v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w},
                                  {v[2].x, v[2].y, v[2].z, v[2].w, v[3].x, v[3].y, v[3].z, v[3].w}};
    unsigned int m2 = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      unsigned int m;
      asm("abs.bf16x2 %0, %1;" : "=r"(m) : "r"(u[i >> 3][i & 7]));
      asm("max.NaN.bf16x2 %0, %0, %1;" : "+r"(m2) : "r"(m));
    }
    m2 &= 0x7FFF7FFFu;
    mx = __vmaxu2(mx, m2);
    sumsq_block(u[0], sq[0], sq[1]);
    sumsq_block(u[1], sq[0], sq[1]);
    const float largest = __uint_as_float(max(m2 << 16, m2 & 0x7FFF0000u));
    // an all-zero block goes the regular way under any scale: its codes and sums come out as zeros
    const bool zero = largest == 0.0f;
    const float bmax = fmaxf(largest, 0x1p-60f);
    if (kSearch == 1) {   // (only the maximum and the sum of squares here)
      fetch(b + step, 0);
      fetch(b + step, 1);
      continue;
    }
    const bool direct = (zero || largest >= 0x1p-60f) && largest <= 0x1p60f;
    zeros += zero ? 1u : 0u;
    unsigned int c[2][2];   // the winner's codes
    int code = 0;
    double g = 0.0;
    bool regular = direct;
    if (kSearch == 0) {
      // scale 2^X with X = floor(log2 bmax) - 2, and bmax / 2^X below 8
      const unsigned int sd_bits = (__float_as_uint(bmax) & 0x7F800000u) - (2u << 23);
      code = static_cast<int>(sd_bits >> 23);
      // S = 2^(10 - X): error minus sum W^2 = sd (sd B - 2 A) = 2^(2X - 10) ((4B << 8) - A')
      int e = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        PairBlock blk;
        FixedPairs fx;
        unpack_pairs(v[2 * i], v[2 * i + 1], blk);
        fetch(b + step, i);
        make_fixed_pairs(blk, fixed_scale(__uint_as_float(sd_bits)), fx);
        e += mx_score(blk, fx, __uint_as_float((254u << 23) - sd_bits), 8, c[i][0], c[i][1]);
      }
      g = static_cast<double>(e) * __hiloint2double((2 * (code - 127) - 10 + 1023) << 20, 0);
    } else if (kSearch == 2) {
      const float center = quotient(bmax, 6.0f, sixth);
      const unsigned int dv0 = __float_as_uint(center) & 0x7F800000u, dv1 = dv0 + 0x00800000u;
      const float v0f = __uint_as_float(dv0), v1f = __uint_as_float(dv1);
      float y;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(center));
      const float per_center = y * k_scale;
      const float t0 = __fadd_rd(__fmaf_rn(v0f, per_center, k_off), 12582912.0f);
      const float t1 = __fadd_rd(__fmaf_rn(v1f, per_center, k_off), 12582912.0f);
      const int k0 = max(0, min(n_beta - 2, __float_as_int(t0) - 0x4B400000));
      const int k1 = max(0, min(n_beta - 2, __float_as_int(t1) - 0x4B400000));
      const uint2 q0 = lds64(pairs + 8u * static_cast<unsigned int>(k0));
      const uint2 q1 = lds64(pairs + 8u * static_cast<unsigned int>(k1));
      const pair_t cc = pair_of(-center, -center);
      const pair_t n0 = pair_mul(cc, pair_of(__uint_as_float(q0.x), __uint_as_float(q0.y)));
      pair_t n1 = pair_mul(cc, pair_of(__uint_as_float(q1.x), __uint_as_float(q1.y)));
      float a0, b0f, a1, b1;
      halves(n0, a0, b0f);
      halves(n1, a1, b1);
      constexpr float kUnder = 1.0f - 0x1.8p-22f;   // as in iterate_pass
      // even the last multiplier's divisor lies before the upper code: it alone can win
      const bool high1 = k1 == n_beta - 2 && -b1 <= v1f * kUnder;
      regular = direct && -a0 <= v0f * kUnder && -b0f > v0f * kUnder && -a1 <= v1f * kUnder && (-b1 > v1f * kUnder || high1);
      if (high1) n1 = pair_of(b1, b1);
      float r00, r01, r10, r11;
      pair_recip(n0, r00, r01);
      pair_recip(n1, r10, r11);
      unsigned int d[4][2][2];
      int s0 = 0, s1 = 0, s2 = 0, s3 = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        PairBlock blk;
        FixedPairs fx;
        unpack_pairs(v[2 * i], v[2 * i + 1], blk);
        fetch(b + step, i);
        make_fixed_pairs(blk, __uint_as_float((265u << 23) - dv0), fx);   // S = 2^(11 - cf)
        s0 += mx_score(blk, fx, r00, 9, d[0][i][0], d[0][i][1]);
        s1 += mx_score(blk, fx, r01, 9, d[1][i][0], d[1][i][1]);
        s2 += mx_score(blk, fx, r10, 10, d[2][i][0], d[2][i][1]);
        s3 += mx_score(blk, fx, r11, 10, d[3][i][0], d[3][i][1]);
      }
      const bool up0 = s1 < s0, up1 = s3 < s2;
      s0 = min(s0, s1);
      s2 = min(s2, s3);
      const bool second = 2 * s2 < s0;
      s0 = min(s0, 2 * s2);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const unsigned int lower = up0 ? d[1][i][k] : d[0][i][k], upper = up1 ? d[3][i][k] : d[2][i][k];
          c[i][k] = second ? upper : lower;
        }
      code = static_cast<int>(dv0 >> 23) + (second ? 1 : 0);
      // error minus sum W^2 = 2^(2 cf - 11) s0
      g = static_cast<double>(s0) * __hiloint2double((2 * (static_cast<int>(dv0 >> 23) - 127) - 11 + 1023) << 20, 0);
    }
    reinterpret_cast<uint4*>(packed)[b] = make_uint4(c[0][0], c[0][1], c[1][0], c[1][1]);
    scales[b] = static_cast<uint8_t>(zero ? 0 : regular ? code : 255);
    if (regular) acc += g;
    else first_marked = min(first_marked, b);
  }
  for (unsigned int b = first_marked; b < nblk; b += step) {
    if (kSearch != 1 && scales[b] != 255) continue;
    MxFound f;
    mx_general<kSearch>(p, b, sh.beta, a.n_dq, n_beta, a.step_pct, f, zeros, wide);
    reinterpret_cast<uint4*>(packed)[b] = f.codes;
    scales[b] = static_cast<uint8_t>(f.code);
    acc += f.g;
  }
  {
    const double err = warp_sum(acc), ss = warp_sum(sq[0] + sq[1]);
    if (lane == 0) {
      sh.part[tid >> 5][0] = err;
      sh.part[tid >> 5][1] = ss;
    }
  }
  if (a.chained) let_next_begin();
  mx = max(mx & 0xFFFFu, mx >> 16);
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  zeros = __reduce_add_sync(0xFFFFFFFFu, zeros);
  const unsigned long long all_wide = warp_count(wide);
  if (lane == 0) {
    if (mx) atomicMax(&sh.amax, mx);
    if (zeros) atomicAdd(&sh.zeros, zeros);
    if (all_wide) add_count(sh.wide, sh.wide_high, all_wide);
  }
  __syncthreads();
  if (tid != 0) return;
  if (!a.chained) {
    unsigned long long seen = 0;
    unsigned int polls = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(&res->reserved) : "memory");
    } while (seen != a.tag && ++polls < kGridWaitLimit);
    if (seen != a.tag) {
      res->status = SOAR_STATUS_INTERNAL;
      return;
    }
  }
  double err = 0.0, ss = 0.0;
  for (int w = 0; w < kQWarps; ++w) {
    err += sh.part[w][0];
    ss += sh.part[w][1];
  }
  atomicAdd(&res->sse, err);
  atomicAdd(&res->sumsq, ss);
  if (sh.amax) atomicMax(&res->amax_bits, sh.amax);
  if (sh.zeros) atomicAdd(reinterpret_cast<unsigned long long*>(&res->zero_blocks), static_cast<unsigned long long>(sh.zeros));
  const unsigned long long cta_wide = count_of(sh.wide, sh.wide_high);
  if (cta_wide) atomicAdd(reinterpret_cast<unsigned long long*>(&res->wide_candidates), cta_wide);
  __threadfence();
  if (atomicAdd(&res->pad_, 1) != static_cast<int>(gridDim.x) - 1) return;
  // the last CTA: the report from the sums
  __threadfence();
  const unsigned int amax_bits = __ldcg(&res->amax_bits);
  const double gsum = __ldcg(&res->sse), sumsq = __ldcg(&res->sumsq);
  int st = 0;
  if (amax_bits >= 0x7F80u) st |= SOAR_STATUS_NONFINITE;
  if (amax_bits == 0) st |= SOAR_STATUS_ZERO_TENSOR;
  res->status = st;
  res->amax = bits_to_mag(amax_bits);
  res->pad_ = 0;
  res->sse = fmax(sumsq + gsum, 0.0);
  res->reserved = gsum;
}
