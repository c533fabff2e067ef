// The quantizer under a column-weighted objective.  Included by soar.cu after quantize_kernel.cuh, whose stage machine it
// runs with passes of its own.
//
// Sec. 5 proposes to minimise the output distortion ||(W - What) X||^2 in CJSO and DSS; its diagonal form is
// sum_ij h_j (W_ij - What_ij)^2 with h_j the second moment of input channel j.  Algorithm 1 is unchanged except that the
// block sums carry the weights,
//   A = sum h_j |w_j| m_j,   B = sum h_j m_j^2,
// in Eq. 5, Eq. 6 and the error of Eq. 8.  The weights are arbitrary binary32 numbers, so the integer dot products of
// the unweighted search do not apply: the sums are binary64, taken in element order, every product exact (24 + 8 + 3
// and 24 + 6 significant bits).
//
// What bounds it: instruction issue, 760 a block with the binary64 pipe, which issues one in two cycles, at 36 %.  A
// candidate costs three binary64 operations per element, p = h (4m), A += p |w|, B += p (4m); the code values become
// binary64 by byte permutes (code_words; the integer conversion instruction instead, for half or all of one candidate,
// was 0 to 4 % slower).  28672 x 8192, a launch a pass: iteration 1084 -> 508 us, the maximum 80 us, the start 181; one iteration
// within a call 980 -> 474 us.

#pragma once

struct Weighted {
  const float* h[kMaxBatch];    // cols weights of each matrix
};

// The sixteen column weights of block column cb.
__device__ __forceinline__ void weights_of(const float* h, unsigned int cb, float (&hv)[16]) {
  const float4* src = reinterpret_cast<const float4*>(h) + static_cast<size_t>(cb) * 4;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 v = __ldg(src + q);
    hv[4 * q] = v.x;
    hv[4 * q + 1] = v.y;
    hv[4 * q + 2] = v.z;
    hv[4 * q + 3] = v.w;
  }
}
// A lane whose blocks all lie in one block column reads that column's weights once and widens them once (see `steady` in the
// passes), so a tensor is walked by as many warps as make a step a whole number of rows: a multiple of
// nbc / gcd(nbc, 32) tiles.  4096 and 8192 columns divide the warps of the device's grid as it is (2368 = 64 * 37); 12288 and
// 28672 columns leave 16 of them out.  Where more than a thirtieth would be left out, or where a tensor has fewer than eight turns, all
// warps walk it and the weights are read again when the column changes.
constexpr unsigned int kColumnTurns = 8;
__host__ __device__ __forceinline__ unsigned int column_span(const Params& p, unsigned int warps) {
  const unsigned int low = p.nbc & (0u - p.nbc), unit = p.nbc / (low < 32u ? low : 32u), span = warps / unit * unit;
  return span * 30 >= warps * 29 && p.ntiles >= kColumnTurns * warps ? span : warps;
}
__host__ __device__ __forceinline__ bool whole_rows(const Params& p, unsigned int span) { return span * 32 % p.nbc == 0; }
// Whether a launch takes the kernel whose lanes stay in their columns: where a matrix of eight turns or more has lanes that do.  The
// code for it costs calls of smaller ones up to 3 % (a layer of 896, 128 and 2688 columns 163 -> 168 us, of 1600, 320 and 4800
// 355 -> 365, in the kernel without it 163 and 356; of 2048, 512 and 6144 it takes 547 -> 536, of 3072, 1024 and 8192 1050 -> 1023).
inline bool has_steady_columns(const Batch& bt, unsigned int warps) {
  for (int i = 0; i < bt.n; ++i)
    if (bt.t[i].ntiles >= kColumnTurns * warps && whole_rows(bt.t[i], column_span(bt.t[i], warps))) return true;
  return false;
}

// What a CTA shares; with columns also by how many warps each tensor is walked, and whether a lane's blocks of it then all
// lie in one block column.
template <bool kWithColumns>
struct __align__(128) WeightedShared : QShared<false> {
  static constexpr bool kColumns = kWithColumns;
  unsigned int span[kWithColumns ? kMaxBatch : 1], steady[kWithColumns ? kMaxBatch : 1];
};
__device__ __forceinline__ unsigned int span_of(const WeightedShared<true>& sh, int ti, unsigned int) { return sh.span[ti]; }

__device__ __forceinline__ bool weight_ok(float h) { return h == 0.0f || (h >= 0x1p-20f && h <= 0x1p20f); }

// Magnitudes of a block in binary64.
__device__ __forceinline__ void wide_magnitudes(const PairBlock& b, double (&wd)[16]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float lo, hi;
    halves(b.w[i], lo, hi);
    wd[2 * i] = static_cast<double>(fabsf(lo));
    wd[2 * i + 1] = static_cast<double>(fabsf(hi));
  }
}

// 4A and 16B of a code vector (sign bits ignored): sums in element order (the powers of two scale every term and every
// partial sum exactly).
struct WeightedSums {
  double a4, b16;
};
// Error minus sum h W^2, over sd / 2, of a vector under the dequantization scale sd.
__device__ __forceinline__ double weighted_rank(const WeightedSums& s, double sd) { return fma(0.125 * sd, s.b16, -s.a4); }
__device__ __forceinline__ void weighted_sums(const double (&hd)[16], const double (&wd)[16], unsigned int c0, unsigned int c1,
                                              WeightedSums& s) {
  double a = 0.0, b = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    unsigned int hi[4];
    code_words<false>((q < 2 ? c0 : c1) >> (16 * (q & 1)), hi);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double dm = __hiloint2double(static_cast<int>(hi[i]), 0);   // 4 m_j
      const double p = hd[4 * q + i] * dm;
      a = fma(p, wd[4 * q + i], a);
      b = fma(p, dm, b);
    }
  }
  s.a4 = a;
  s.b16 = b;
}

// The sums of two code vectors at once, widening each weight and magnitude where it is used, by asm that the compiler does
// not lift out: the 32 widened values kept over all candidates take 64 registers and spill (573 against 510 us an
// iteration on 28672 x 8192).
__device__ __forceinline__ void weighted_sums_of_two(const float (&hv)[16], const PairBlock& blk, const unsigned int (&ca)[2],
                                                     const unsigned int (&cb)[2], WeightedSums& sa, WeightedSums& sb) {
  double a0 = 0.0, b0 = 0.0, a1 = 0.0, b1 = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    unsigned int ha[4], hb[4];
    code_words<false>(ca[q >> 1] >> (16 * (q & 1)), ha);
    code_words<false>(cb[q >> 1] >> (16 * (q & 1)), hb);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 4 * q + i;
      float lo, hi;
      halves(blk.w[j >> 1], lo, hi);
      double w, h;
      asm volatile("cvt.f64.f32 %0, %1;" : "=d"(w) : "f"(fabsf((j & 1) ? hi : lo)));
      asm volatile("cvt.f64.f32 %0, %1;" : "=d"(h) : "f"(hv[j]));
      const double da = __hiloint2double(static_cast<int>(ha[i]), 0), db = __hiloint2double(static_cast<int>(hb[i]), 0);
      const double pa = h * da, pb = h * db;
      a0 = fma(pa, w, a0);
      b0 = fma(pa, da, b0);
      a1 = fma(pb, w, a1);
      b1 = fma(pb, db, b1);
    }
  }
  sa.a4 = a0;
  sa.b16 = b0;
  sb.a4 = a1;
  sb.b16 = b1;
}

// What a search has found for a block.
struct WeightedFound {
  unsigned int c0, c1;
  int d;
  WeightedSums s;
  double g;
};

// The search by the general rules, out of line and fed from memory: any number of codes, short grids, and, where the
// coupled arm, a grid of one multiplier or a zero weight (whose column costs nothing whatever its code, so that equal
// errors of different codes occur all along the grid) rules the bracket out, every multiplier in turn.  First minimum
// in (beta, code) order.
__device__ __noinline__ WeightedFound weighted_search_general(const Params& p, const float* h, unsigned int b, float alpha,
                                                              float center, const float2* s_beta, unsigned int* whole_grid) {
  uint4 v0, v1;
  load_block(p, b, v0, v1);
  PairBlock blk;
  unpack_pairs(v0, v1, blk);
  double hd[16], wd[16];
  bool zero_weight = false;
  {
    float hv[16];
    weights_of(h, b - (__umulhi(2u * b, p.nbc_magic) >> p.nbc_shift) * p.nbc, hv);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      hd[j] = static_cast<double>(hv[j]);
      zero_weight = zero_weight || hv[j] == 0.0f;
    }
  }
  wide_magnitudes(blk, wd);
  const int n_beta = p.n_beta, n_dq = p.n_dq;
  const bool coupled = (p.flags & SOAR_FLAG_COUPLED_SCALE) != 0;
  const double alpha_d = static_cast<double>(alpha);
  int d_lo, d_hi;
  candidate_window(center, n_dq, d_lo, d_hi);
  WeightedFound best;
  best.g = __longlong_as_double(0x7FF0000000000000ll);
  best.c0 = best.c1 = 0u;
  best.d = clip_code(d_lo);
  best.s.a4 = best.s.b16 = 0.0;
  if (!coupled && p.beta_step_pct >= 1 && n_beta >= kBracketMinBeta && !zero_weight) {
    const float k_scale = 100.0f / static_cast<float>(p.beta_step_pct);
    const float k_off = static_cast<float>(n_beta / 2) - k_scale, per_center = __fdividef(k_scale, center);
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
        unsigned int c0, c1;
        round_pairs(blk, recip_fast_ok(sk) ? recip_fast(sk) : __frcp_rn(sk), c0, c1);
        WeightedSums s;
        weighted_sums(hd, wd, c0, c1, s);
        const double g = 0.5 * sd * weighted_rank(s, sd);
        // equal errors: the earlier multiplier, then the smaller code, as in grid order
        if (g < best.g || (g == best.g && k < best_k)) {
          best.g = g; best.s = s; best.c0 = c0; best.c1 = c1; best.d = dc; best_k = k;
        }
      }
    }
    return best;
  }
  ++*whole_grid;
  for (int k = 0; k < n_beta; ++k) {
    unsigned int c0 = 0, c1 = 0;
    WeightedSums s;
    s.a4 = s.b16 = 0.0;
    if (!coupled) {
      round_pairs(blk, recip_scale(alpha, __fmul_rn(center, s_beta[k].x)), c0, c1);
      weighted_sums(hd, wd, c0, c1, s);
    }
    for (int d = d_lo; d <= d_hi; ++d) {
      const int dc = clip_code(d);
      const float dv = e4m3_value(dc);
      if (coupled) {
        round_pairs(blk, recip_scale(alpha, __fmul_rn(dv, s_beta[k].x)), c0, c1);
        weighted_sums(hd, wd, c0, c1, s);
      }
      const double sd = alpha_d * static_cast<double>(dv);
      const double g = 0.5 * sd * weighted_rank(s, sd);
      if (g < best.g) { best.g = g; best.s = s; best.c0 = c0; best.c1 = c1; best.d = dc; }
    }
  }
  return best;
}

// ------------------------------------------------------------------ passes

// Eq. 1's tensor maximum, sum h_j W^2 for the error report, and the check of the weights.
template <typename S>
__device__ __forceinline__ void weighted_amax_pass(S& sh, const Batch& bt, const Weighted& wt) {
  const unsigned int lane = threadIdx.x & 31u;
  unsigned int mx = 0, nblk = 0, nbc = 1, magic = 0, shift = 0, column = 0;
  const float* h = nullptr;
  bool bad = false, steady = false;
  double sq[2] = {0.0, 0.0}, squares[16];   // (steady) sum W^2 of each of the column's sixteen weights
#pragma unroll
  for (int j = 0; j < 16; ++j) squares[j] = 0.0;
  walk_tiles<true, false>(
      sh, bt, false,
      [&](int ti) {
        const Params& p = bt.t[ti];
        nblk = p.nblk;
        nbc = p.nbc;
        magic = p.nbc_magic;
        shift = p.nbc_shift;
        h = wt.h[ti];
        if constexpr (S::kColumns) {
          steady = sh.steady[ti] != 0u;
          column = 0;   // (a lane that meets no block of this tensor)
        }
      },
      [&](int ti) {
        if (S::kColumns && steady) {
          float hv[16];
          weights_of(h, column, hv);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            sq[j & 1] = fma(static_cast<double>(hv[j]), squares[j], sq[j & 1]);
            squares[j] = 0.0;
          }
        }
        mx = max(mx & 0xFFFFu, mx >> 16);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        const bool any_bad = __any_sync(0xFFFFFFFFu, bad);
        if (lane == 0) {
          if (mx) atomicMax(&sh.amax[ti], mx);
          if (any_bad) atomicOr(&bt.t[ti].ws->error, kErrWeight);
        }
        double v[2] = {sq[0] + sq[1], 0.0};
        hand_over(sh, ti, v);
        mx = 0;
        bad = false;
        sq[0] = sq[1] = 0.0;
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2&, auto next, unsigned int) {
        if (b >= nblk) return;
        column = b - (__umulhi(2u * b, magic) >> shift) * nbc;
        const unsigned int u[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        unsigned int bmx = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // (a NaN input comes out of the maximum as NaN, whose bits are above the infinity pattern)
          unsigned int m;
          asm("abs.bf16x2 %0, %1;" : "=r"(m) : "r"(u[i]));
          asm("max.NaN.bf16x2 %0, %0, %1;" : "+r"(bmx) : "r"(m));
        }
        mx = __vmaxu2(mx, bmx & 0x7FFF7FFFu);
        if (S::kColumns && steady) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const double wl = widen_low(u[i]), wh = widen_high(u[i]);
            squares[2 * i] = fma(wl, wl, squares[2 * i]);
            squares[2 * i + 1] = fma(wh, wh, squares[2 * i + 1]);
          }
        } else {
          float hv[16];
          weights_of(h, column, hv);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const double wl = widen_low(u[i]), wh = widen_high(u[i]);
            sq[0] = fma(static_cast<double>(hv[2 * i]) * wl, wl, sq[0]);
            sq[1] = fma(static_cast<double>(hv[2 * i + 1]) * wh, wh, sq[1]);
          }
        }
        // the blocks of the first row meet every weight once
        if (b < nbc) {
          float hv[16];
          weights_of(h, column, hv);
#pragma unroll
          for (int j = 0; j < 16; ++j) bad = bad || !weight_ok(hv[j]);
        }
        next();
      });
}

// A block's carried state: {A, B} of the current codes as binary32, which is all Eq. 6 takes from them; where it takes the
// stored scale instead (B = 0, or the arm that keeps it), {scale code, B}.  Both zero for an all-zero block.
__device__ __forceinline__ uint2 weighted_state(const WeightedSums& s, int d, bool keep_scale) {
  const float A = static_cast<float>(0.25 * s.a4), B = static_cast<float>(0.0625 * s.b16);
  return make_uint2((B > 0.0f && !keep_scale) ? __float_as_uint(A) : static_cast<unsigned int>(d), __float_as_uint(B));
}

// Algorithm 1 "Initialization" (Eq. 1; the weights play no part in it), the first codes, and the weighted stage-0
// sums of Eq. 5 and of the starting error.
template <typename S>
__device__ __forceinline__ void weighted_init_pass(S& sh, const Batch& bt, const Weighted& wt) {
  float alpha = 1.0f, six_alpha = 6.0f, six_inv = 0.0f;
  bool tame = false;
  double alpha_d = 1.0;
  double acc[2] = {0.0, 0.0};   // 4 den, gsum
  unsigned int zeros = 0, wide = 0, nblk = 0, nbc = 1, magic = 0, shift = 0, view = 0;
  const float* h = nullptr;
  const bool keep_scale = (bt.t[0].flags & SOAR_FLAG_KEEP_BLOCK_SCALE) != 0;
  unsigned int keep = bt.t[0].max_iters > 0, column = 0xFFFFFFFFu;
  double hd[16];   // the column's weights
#pragma unroll
  for (int j = 0; j < 16; ++j) hd[j] = 0.0;
  asm volatile("" : "+r"(keep));
  walk_tiles<true, false>(
      sh, bt, true,
      [&](int ti) {
        const Params& p = bt.t[ti];
        alpha = sh.alpha[ti];
        six_alpha = __fmul_rn(alpha, 6.0f);
        six_inv = __frcp_rn(six_alpha);
        tame = tame_alpha(alpha);
        alpha_d = static_cast<double>(alpha);
        nblk = p.nblk;
        nbc = p.nbc;
        magic = p.nbc_magic;
        shift = p.nbc_shift;
        view = smem_u32(&sh.view[ti]);
        h = wt.h[ti];
        column = 0xFFFFFFFFu;
      },
      [&](int ti) {
        hand_over(sh, ti, acc);
        hand_over_counters(sh, ti, zeros, wide);
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2&, auto next, unsigned int) {
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
        unsigned int c0, c1;
        if (bmax == 0.0f) {
          round_pairs(blk, 1.0f, c0, c1);
          reinterpret_cast<uint2*>(packed)[b] = make_uint2(c0, c1);
          scales[b] = 0;
          if (keep) state[b] = make_uint2(0u, 0u);
          ++zeros;
          return;
        }
        const int d = max(e4m3_encode(tame ? quotient(bmax, six_alpha, six_inv) : __fdiv_rn(bmax, six_alpha)), 1);
        const float v = e4m3_value(d);
        round_pairs(blk, recip_scale(alpha, v), c0, c1);
        const unsigned int here = b - (__umulhi(2u * b, magic) >> shift) * nbc;
        if (!S::kColumns || here != column) {
          column = here;
          float hv[16];
          weights_of(h, here, hv);
#pragma unroll
          for (int j = 0; j < 16; ++j) hd[j] = static_cast<double>(hv[j]);
        }
        double wd[16];
        wide_magnitudes(blk, wd);
        WeightedSums s;
        weighted_sums(hd, wd, c0, c1, s);
        if (keep) {
          state[b] = weighted_state(s, d, keep_scale);
        } else {
          reinterpret_cast<uint2*>(packed)[b] = make_uint2(c0, c1);
          scales[b] = static_cast<uint8_t>(d);
        }
        const double vd = static_cast<double>(v), sd = alpha_d * vd;
        acc[0] = fma(s.b16, 0.25 * vd * vd, acc[0]);
        acc[1] += 0.5 * sd * weighted_rank(s, sd);
      });
}

// One iteration of Algorithm 1 under the weighted objective: Eq. 6 per block from its stored {A, B}, App. B.3's candidates,
// Eq. 8 with the weighted error written as sum h w^2 + sd^2 B - 2 sd A, first minimum in (beta, code) order.  kFast: the
// paper's two E4M3 codes on a grid that holds their brackets; the weighted error of an element is convex in its code
// value like the unweighted one, so per code only the multipliers of winning_range can win.
template <bool kFast, typename S>
__device__ __forceinline__ void weighted_iterate_pass(S& sh, const Batch& bt, const Weighted& wt, bool reverse, unsigned int emit,
                                                      unsigned int keep) {
  asm volatile("" : "+r"(emit), "+r"(keep));
  const bool keep_scale = (bt.t[0].flags & SOAR_FLAG_KEEP_BLOCK_SCALE) != 0;
  const float k_scale = 100.0f / static_cast<float>(max(bt.t[0].beta_step_pct, 1));
  const float k_off = static_cast<float>(bt.t[0].n_beta / 2) - k_scale;
  const unsigned int pairs = smem_u32(sh.beta);
  float alpha = 1.0f, alpha_t = 0.0f;   // alpha_t: alpha where the fast path may run, else NaN (its guards fail)
  double alpha_d = 1.0;
  double acc[2] = {0.0, 0.0};           // 4 den, gsum
  unsigned int whole = 0, zeros = 0, nblk = 0, nbc = 1, magic = 0, shift = 0, view = 0;
  int tensor = 0;
  const float* h = nullptr;
  walk_tiles<true, true>(
      sh, bt, reverse,
      [&](int ti) {
        const Params& p = bt.t[ti];
        alpha = sh.alpha[ti];
        alpha_t = kFast && tame_alpha(alpha) ? alpha : __uint_as_float(0x7FC00000u);
        alpha_d = static_cast<double>(alpha);
        nblk = p.nblk;
        nbc = p.nbc;
        magic = p.nbc_magic;
        shift = p.nbc_shift;
        asm volatile("" : "+r"(nbc), "+r"(magic), "+r"(shift));
        view = smem_u32(&sh.view[ti]);
        h = wt.h[ti];
        tensor = ti;
      },
      [&](int ti) {
        hand_over(sh, ti, acc);
        hand_over_counters(sh, ti, zeros, whole);   // reported as soar_result.wide_candidates
      },
      [&](unsigned int b, const uint4& v0, const uint4& v1, const uint2& st, auto next, unsigned int) {
        const bool active = b < nblk && (st.x | st.y) != 0u;   // past the end, or an all-zero block
        WeightedFound f;
        f.c0 = f.c1 = 0u;
        f.d = 0;
        f.s.a4 = f.s.b16 = f.g = 0.0;
        bool direct = false;
        if (kFast) {
          float hv[16];
          weights_of(h, active ? b - (__umulhi(2u * b, magic) >> shift) * nbc : 0u, hv);
          PairBlock blk;
          unpack_pairs(v0, v1, blk);
          // Eq. 6 (B = 0 fails the range check)
          const float D = __fmul_rn(alpha_t, __uint_as_float(st.y));
          const float center = quotient(__uint_as_float(st.x), D, recip_fast(D));
          const unsigned int dv0 = __float_as_uint(center) & 0xFFF00000u, dv1 = dv0 + 0x00100000u;
          const float v0f = __uint_as_float(dv0), v1f = __uint_as_float(dv1);
          float y;
          asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(center));
          const float per_center = y * k_scale;
          const float t0 = __fadd_rd(__fmaf_rn(v0f, per_center, k_off), 12582912.0f);
          const float t1 = __fadd_rd(__fmaf_rn(v1f, per_center, k_off), 12582912.0f);
          const uint2 q0 = lds64(pairs + 8u * (__float_as_uint(t0) & (SOAR_MAX_BETA - 1)));
          const uint2 q1 = lds64(pairs + 8u * (__float_as_uint(t1) & (SOAR_MAX_BETA - 1)));
          const pair_t cc = pair_of(center, center), aa = pair_of(-alpha, -alpha);
          const pair_t m0 = pair_mul(cc, pair_of(__uint_as_float(q0.x), __uint_as_float(q0.y)));
          const pair_t m1 = pair_mul(cc, pair_of(__uint_as_float(q1.x), __uint_as_float(q1.y)));
          float a0, b0f, a1, b1;
          halves(m0, a0, b0f);
          halves(m1, a1, b1);
          constexpr float kUnder = 1.0f - 0x1.8p-22f, kOver = 1.0f + 0x1.8p-22f;   // as in iterate_pass
          unsigned int least = 0x7F800000u;   // smallest weight (bit patterns of non-negative floats order like them)
#pragma unroll
          for (int j = 0; j < 16; ++j) least = min(least, __float_as_uint(hv[j]));
          direct = __float_as_uint(center) - 0x3C800000u < 0x43E00000u - 0x3C800000u && a0 <= v0f * kUnder &&
                   b0f >= v0f * kOver && a1 <= v1f * kUnder && b1 >= v1f * kOver && least != 0u;
          float r00, r01, r10, r11;
          pair_recip(pair_mul(aa, m0), r00, r01);
          pair_recip(pair_mul(aa, m1), r10, r11);
          unsigned int c[4][2];
          round_pairs(blk, r00, c[0][0], c[0][1]);
          round_pairs(blk, r01, c[1][0], c[1][1]);
          const double sd0 = alpha_d * scaled_value(dv0, 0), sd1 = alpha_d * scaled_value(dv1, 0);
          WeightedSums s0, s1;
          weighted_sums_of_two(hv, blk, c[0], c[1], s0, s1);
          double e0 = weighted_rank(s0, sd0), e1 = weighted_rank(s1, sd0);
          f.c0 = c[0][0];
          f.c1 = c[0][1];
          f.s = s0;
          if (e1 < e0) { f.c0 = c[1][0]; f.c1 = c[1][1]; f.s = s1; e0 = e1; }
          f.g = 0.5 * sd0 * e0;
          f.d = static_cast<int>(dv0 >> 20) - 960;
          round_pairs(blk, r10, c[2][0], c[2][1]);
          round_pairs(blk, r11, c[3][0], c[3][1]);
          weighted_sums_of_two(hv, blk, c[2], c[3], s0, s1);
          e0 = weighted_rank(s0, sd1);
          e1 = weighted_rank(s1, sd1);
          if (e1 < e0) { c[2][0] = c[3][0]; c[2][1] = c[3][1]; s0 = s1; e0 = e1; }
          // equal errors: the earlier multiplier, as in grid order (the second code's are never earlier)
          const double g1 = 0.5 * sd1 * e0;
          if (g1 < f.g) {
            f.c0 = c[2][0];
            f.c1 = c[2][1];
            f.s = s0;
            f.g = g1;
            f.d = static_cast<int>(dv1 >> 20) - 960;
          }
        }
        next();
        if (active && !direct) {
          const float B0 = __uint_as_float(st.y);
          const float center = (B0 > 0.0f && !keep_scale) ? __fdiv_rn(__uint_as_float(st.x), __fmul_rn(alpha, B0))
                                                          : e4m3_value(static_cast<int>(st.x));
          f = weighted_search_general(bt.t[tensor], h, b, alpha, center, sh.beta, &whole);
        }
        if (active) {
          uint8_t *packed, *scales;
          uint2* state;
          load_view(view, packed, scales, state);
          if (emit) {
            reinterpret_cast<uint2*>(packed)[b] = make_uint2(f.c0, f.c1);
            scales[b] = static_cast<uint8_t>(f.d);
          }
          if (keep) state[b] = weighted_state(f.s, f.d, keep_scale);
          const double vd = static_cast<double>(e4m3_value(f.d));
          acc[0] = fma(f.s.b16, 0.25 * vd * vd, acc[0]);
          acc[1] += f.g;
        }
      });
}

template <bool kFast>
struct WeightedPasses {
  const Weighted& wt;
  static constexpr bool kGrid = true;
  template <typename S>
  __device__ __forceinline__ void amax(S& sh, const Batch& bt) const { weighted_amax_pass(sh, bt, wt); }
  template <typename S>
  __device__ __forceinline__ void init(S& sh, const Batch& bt) const { weighted_init_pass(sh, bt, wt); }
  template <typename S>
  __device__ __forceinline__ void iterate(S& sh, const Batch& bt, bool reverse, bool emit, bool keep) const {
    weighted_iterate_pass<kFast>(sh, bt, wt, reverse, emit, keep);
  }
};

template <bool kFast, bool kColumns>
__global__ void __launch_bounds__(kQThreads, 2)
weighted_kernel(const __grid_constant__ Batch bt, const __grid_constant__ Weighted wt, const __grid_constant__ Reports rp,
                int stage_lo, int stage_hi) {
  __shared__ WeightedShared<kColumns> sh;
  if constexpr (kColumns) {
    if (threadIdx.x < static_cast<unsigned int>(bt.n)) {
      const Params& p = bt.t[threadIdx.x];
      const unsigned int span = column_span(p, gridDim.x * kQWarps);
      sh.span[threadIdx.x] = span;
      sh.steady[threadIdx.x] = whole_rows(p, span);
    }
  }
  run_stages<false>(sh, static_cast<double (*)[3]>(nullptr), bt, rp, stage_lo, stage_hi, WeightedPasses<kFast>{wt});
}
