// One matrix, one launch.  The passes are quantize_kernel's; what differs is how they meet and where the weights stay.
// Included by soar.cu after quantize_kernel.cuh.
//
// Small matrices are bound by latency: what counts is the chain from the last block of one pass to the first of the
// next.  With the sums added by atomics in memory zeroed by a memset, that chain took 3.5 of the 5 microseconds of an
// iteration at any size.  Here every CTA stores its sums in a slot of its own, arrives at a counter and, when all
// have, reads everybody's slots and adds them in the same order on every run: 1.6 us when all come at the same moment;
// within a call, from the last CTA's arrival until all go on, 2.3 to 3.1 us, on 28672 x 8192 3.3 and 4.1.  (Polling tagged
// slots instead, with no counter, is 0.7 us when all CTAs come at the same moment but 3 us when some wait for others,
// as they do.)  A matrix that stays in shared memory has a shorter way after the start pass and the
// iterations (meet_by_sums).  The grid is one CTA of 16 warps per SM rather than two of 8: 296 CTAs need
// 0.7 us more.
//
// The smallest matrices (see kClusterTiles) run in one cluster of up to 16 CTAs: the sums travel through distributed shared
// memory (exchange_in_cluster), with nothing in global memory and no cooperative launch.  256 tiles: an iteration with one
// candidate 1.8 us (2.3 on a grid that meets by sums), of the search 2.3 (2.8), a max-based call 6.1 us (8.0 as two kernels).
//
// Matrices whose tiles fit the shared memory of the grid (12 million weights) are read from HBM once and stay
// there, and so do their block states (kResident); larger ones stream through the passes like a batch.
//
// Nothing has to be zero before the launch, so no memset goes ahead of it: CTA 0 clears the counter while the first
// pass runs and says so in a flag, whose value is nonce + epoch.  The nonce is new for every call the host makes; the
// epoch is a word of the workspace that CTA 0 advances at the end of a call, after every CTA has read it, so that
// the replay of a captured call does not take the flag of the replay before for its own.  Whatever the workspace
// held before a call, it would have to hold the 64-bit flag of a call not made yet to be taken for open.

#pragma once

constexpr int kSoloWarps = 16;                     // warps of a CTA: one CTA an SM
constexpr int kNoIterations = -1;                   // kMode of a call without iterations
constexpr unsigned int kSoloMaxGrid = 160;
constexpr unsigned int kResidentTiles = 160;       // slots a CTA can have: 200 KB
constexpr size_t kSlotBytes = 24;                  // three numbers of one CTA and pass

// Up to kOneCtaTiles tiles run in one CTA; up to kClusterTiles in a cluster, a warp to a tile while 256 warps suffice.  The
// cluster saves the cooperative launch and the first meetings' trips, the grid has three times the warps at 768 tiles: a search of
// one iteration 11.6 us against 16.1 there, each further one 4.8 against 3.6, so that at the usual three the cluster is
// ahead (21 against 23) and at 1024 tiles behind (24.5 against 22); with one candidate 9.7 against 14.4 and 3.1 against
// 2.7; max-based calls 9.5 against 12.0, 7.2 against 8.0 at 1024.
constexpr unsigned int kOneCtaTiles = 8, kClusterMost = 16, kClusterTiles = 768;
constexpr unsigned int cluster_warps(unsigned int tiles) {
  const unsigned int even = (tiles + kClusterMost - 1) / kClusterMost;
  return even < 4 ? 4 : even > kSoloWarps ? kSoloWarps : even;
}
constexpr unsigned int cluster_size(unsigned int tiles) {   // a power of two
  const unsigned int want = (tiles + cluster_warps(tiles) - 1) / cluster_warps(tiles);
  unsigned int n = 1;
  while (n < want && n < kClusterMost) n *= 2;
  return n;
}
constexpr unsigned int solo_grid(unsigned int tiles, unsigned int most) {
  const unsigned int want = tiles <= kOneCtaTiles ? 1 : (tiles + kSoloWarps - 1) / kSoloWarps;
  return want < most ? want : most;
}
// Workspace of the exchange: epoch, flag and counter, then the slots of even and of odd passes; none for one CTA.
constexpr size_t exchange_bytes(unsigned int tiles) {
  const size_t grid = solo_grid(tiles, kSoloMaxGrid);
  return grid > 1 ? (256 + 2 * grid * kSlotBytes + 255) / 256 * 256 : 0;
}

struct SoloArgs {
  Single m;
  float* alpha;
  soar_result* result;     // or null
  uint8_t* tiled;          // tiled scales, or null
  unsigned char* exchange;
  unsigned long long nonce;
  unsigned int rows;
  unsigned int per_warp;   // resident: slots of a warp
  int tiled_only;          // the caller wants no row-major scales
  int idle;                // test hook, see WaitHook
};

// Words that CTAs add to when they meet by sums (meet_by_sums): kSumWords that are waited for, one set on a line for the meetings
// of even and one for those of odd number, and two counts that are read at the end.  They lie in the header that only the
// stages of other calls use.  (The words of a set on lines of their own arrive up to a microsecond apart.)
constexpr unsigned int kSumWords = 5, kSetWords = 16, kWords = 3 * kSetWords;
static_assert(kWords * 8 <= kWsFixedBytes, "no room for the words of the meetings");

// Where a matrix's tiles stay and how its CTAs meet.
constexpr int kStreamed = 0, kKept = 1, kKeptInCluster = 2;

template <int kPlace, bool kNoIter>
struct __align__(128) SoloShared {
  static constexpr bool kFinal = kNoIter;
  static constexpr bool kOrdered = true, kSolo = true, kResident = kPlace != kStreamed, kCluster = kPlace == kKeptInCluster;
  View view[1];
  float2 beta[SOAR_MAX_BETA];
  double part[32][2];                // each warp's sums of the pass
  // the grid's numbers, by the warp that read them; in a cluster by the CTA that sent them
  unsigned long long red[2][kCluster ? kClusterMost : kSoloMaxGrid / 32][3];
  unsigned long long landed[2];              // (cluster) mbarriers of the meetings of even and of odd number
  unsigned long long before[2][kSumWords];   // the words of either set when its last meeting was over
  double trace_alpha[SOAR_MAX_ITERS + 1], trace_sse[SOAR_MAX_ITERS + 1];
  float alpha[1];
  unsigned int amax[1], zeros[1], wide[1], wide_high[1];
  unsigned int start[1], count[1], total;
  unsigned int slots;                // shared address of the warps' tile slots
  unsigned int per_warp;
  int tiled_only;
  int error_exp;                     // exponent under which meet_by_sums takes a share of the error
  int failed;
};

// Sums of the grid, the same bits in every thread.
struct Totals {
  double a, g;                       // sum W^2 and nothing (kMax), else 4 den and gsum
  unsigned int amax;                 // kMax: the maximum's bits
  unsigned long long counts;         // see counts_word (CTA 0 only)
};

// A CTA's counts of a pass in one word: after the start pass (`first`) zero blocks in the low half and wide candidates, at most
// one a block, in the high one; after an iteration, where no zero block is counted, the wide candidates of up to 8,192 a
// block, which pass 32 bits.  (A matrix has fewer than 2^31 blocks; sums of these words do not carry over.)
template <typename S>
__device__ __forceinline__ unsigned long long counts_word(const S& sh, bool first) {
  return count_of(first ? sh.zeros[0] : sh.wide[0], first ? sh.wide[0] : sh.wide_high[0]);
}

// Where the exchange keeps its words: epoch, then flag and counter in one sixteen-byte unit.
constexpr size_t kEpochAt = 0, kFlagAt = 16, kCounterAt = 24;

// At the start of the call (one thread of CTA 0): clears the counter and opens the flag in one store, which nothing has to
// be waited for.
__device__ __forceinline__ void open_counter(const SoloArgs& a, unsigned long long tag) {
  asm volatile("{\n.reg .b128 p;\nmov.b128 p, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], p;\n}" ::"l"(a.exchange + kFlagAt), "l"(tag),
               "l"(0ull)
               : "memory");
}
__device__ __forceinline__ unsigned long long* sum_words(const SoloArgs& a) { return reinterpret_cast<unsigned long long*>(a.m.t[0].ws); }
// Before the first arrival (one thread of every CTA).
__device__ __forceinline__ bool counter_open(const SoloArgs& a, unsigned long long tag) {
  unsigned long long seen = 0;
  unsigned int polls = 0;
  do {
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(a.exchange + kFlagAt) : "memory");
  } while (seen != tag && ++polls < kGridWaitLimit);
  return seen == tag;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Sum over lanes 0..15 of a warp whose upper lanes hold the same values again.
__device__ __forceinline__ double half_warp_sum(double v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// exchange() inside a cluster: every CTA sends its numbers into everybody's shared memory with stores that count themselves
// off at the receiver's mbarrier, so that nothing is released and nobody waits for the codes written in the pass.  From the
// last CTA's arrival until all go on 0.45 us after the maximum, 0.55 to 0.6 after the other passes (the hardware's
// cluster barrier took 0.3 to 0.4 us more a meeting).
// One try_wait, which sleeps until the numbers are there (test_wait alone: 0.1 us more a call), then polls with test_wait,
// which returns at once: how long a try_wait may stay suspended is the hardware's choice, so that a count of them bounds
// nothing.  The polls cannot run out in earnest, since a cluster's CTAs run together and a pass waits for nobody; a CTA that gives
// up all the same stays until no other can send to it (see the end of solo_kernel).
template <bool kMax, typename S>
__device__ __forceinline__ bool exchange_in_cluster(S& sh, int idle, unsigned int pass, bool first, Totals& out) {
  __syncthreads();
  const unsigned int tid = threadIdx.x, lane = tid & 31u, grid = gridDim.x, turn = pass & 1u;
  if (tid < 32) {
    double x = 0.0, g = 0.0;
    if ((lane & 15u) < blockDim.x / 32) {   // (at most sixteen warps)
      x = sh.part[lane & 15u][0];
      g = sh.part[lane & 15u][1];
    }
    x = half_warp_sum(x);
    if (!kMax) g = half_warp_sum(g);
    const unsigned long long second = kMax ? sh.amax[0] : static_cast<unsigned long long>(__double_as_longlong(g));
    const unsigned long long counts = kMax ? 0ull : counts_word(sh, first);
    __syncwarp();
    const unsigned int landed = smem_u32(&sh.landed[turn]);
    if (lane == 0) {
      sh.zeros[0] = sh.wide[0] = sh.wide_high[0] = 0u;
      asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n}" ::"r"(landed), "r"(grid * 24u) : "memory");
    }
    if (lane < grid && idle != kNobodySends && (kMax || idle != kNobodyMeetsAgain)) {
      unsigned int at, bar;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(&sh.red[turn][blockIdx.x][0])), "r"(lane));
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(landed), "r"(lane));
      const unsigned long long v[3] = {static_cast<unsigned long long>(__double_as_longlong(x)), second, counts};
#pragma unroll
      for (unsigned int i = 0; i < 3; ++i)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u64 [%0], %1, [%2];" ::"r"(at + 8 * i), "l"(v[i]), "r"(bar) : "memory");
    }
    // (the mbarrier's phase: this is its (pass - 1) / 2 th meeting)
    unsigned int done = 0, polls = 0;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done)
                 : "r"(landed), "r"(((pass - 1) >> 1) & 1u)
                 : "memory");
    while (!done && polls++ < kClusterWaitLimit)
      asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                   : "=r"(done)
                   : "r"(landed), "r"(((pass - 1) >> 1) & 1u)
                   : "memory");
    if (!done) sh.failed = 1;
  }
  __syncthreads();
  double x = 0.0, g = 0.0;
  unsigned int mx = 0;
  unsigned int counts[2] = {0, 0};   // (a cluster's 24,576 blocks have fewer than 2^32 candidates)
  if ((lane & 15u) < grid) {
    const volatile unsigned long long* const r = sh.red[turn][lane & 15u];
    x = __longlong_as_double(static_cast<long long>(r[0]));
    if (kMax) mx = static_cast<unsigned int>(r[1]);
    else g = __longlong_as_double(static_cast<long long>(r[1]));
    if (!kMax && lane < 16) {
      counts[0] = static_cast<unsigned int>(r[2]);
      counts[1] = static_cast<unsigned int>(r[2] >> 32);
    }
  }
  out.a = half_warp_sum(x);
  out.g = kMax ? 0.0 : half_warp_sum(g);
  out.amax = kMax ? __reduce_max_sync(0xFFFFFFFFu, mx) : 0u;
  out.counts = 0;
  if (!kMax && blockIdx.x == 0)
    out.counts = __reduce_add_sync(0xFFFFFFFFu, counts[0]) |
                 (static_cast<unsigned long long>(__reduce_add_sync(0xFFFFFFFFu, counts[1])) << 32);
  return sh.failed == 0;
}

// After a pass, all threads of all CTAs: exchanges the CTAs' sums.  `pass` counts from 1.  On a grid what the CTAs wrote to
// global memory before is visible to all after (in a cluster it is not), and with `last` only CTA 0 waits for the sums.  False
// when a wait ran out.
// kMax: after the pass for the maximum; first: after the start pass.
template <bool kMax, typename S>
__device__ __forceinline__ bool exchange(S& sh, const SoloArgs& a, unsigned long long tag, unsigned int pass, bool first, bool last,
                                         Totals& out) {
  if constexpr (S::kCluster) return exchange_in_cluster<kMax>(sh, a.idle, pass, first, out);
  __syncthreads();
  const unsigned int tid = threadIdx.x, lane = tid & 31u, grid = gridDim.x, turn = pass & 1u;
  unsigned long long* const slots = reinterpret_cast<unsigned long long*>(a.exchange + 256 + turn * (grid * kSlotBytes));
  if (tid < 32) {
    double x = 0.0, g = 0.0;
    if (lane < blockDim.x / 32) {
      x = sh.part[lane][0];
      g = sh.part[lane][1];
    }
    x = warp_sum(x);
    g = warp_sum(g);
    const unsigned long long second = kMax ? sh.amax[0] : static_cast<unsigned long long>(__double_as_longlong(g));
    const unsigned long long counts = kMax ? 0ull : counts_word(sh, first);
    __syncwarp();
    if (lane == 0) sh.zeros[0] = sh.wide[0] = sh.wide_high[0] = 0u;
    if (grid == 1) {
      if (lane == 0) {
        sh.red[turn][0][0] = static_cast<unsigned long long>(__double_as_longlong(x));
        sh.red[turn][0][1] = second;
        sh.red[turn][0][2] = counts;
      }
    } else {
      if (lane < 3)
        __stcg(slots + lane * grid + blockIdx.x,
               lane == 0 ? static_cast<unsigned long long>(__double_as_longlong(x)) : lane == 1 ? second : counts);
      __syncwarp();
      if (lane == 0) {
        unsigned int* const arrived = reinterpret_cast<unsigned int*>(a.exchange + kCounterAt);
        if (pass == 1 && !counter_open(a, tag)) sh.failed = 1;
        if (a.idle != kNobodyArrives && (kMax || a.idle != kNobodyMeetsAgain))
          asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
        if (!last || blockIdx.x == 0) {
          unsigned int seen = 0, polls = 0;
          do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(arrived) : "memory");
          } while (seen < pass * grid && ++polls < kGridWaitLimit);
          if (seen < pass * grid) sh.failed = 1;
        }
      }
    }
  }
  if (last && blockIdx.x != 0) return true;
  __syncthreads();
  const unsigned int warps = (grid + 31) / 32;
  if (grid > 1) {
    if (tid < warps * 32) {
      double x = 0.0, g = 0.0;
      unsigned int mx = 0;
      unsigned long long counts = 0;
      if (tid < grid) {
        x = __longlong_as_double(static_cast<long long>(__ldcg(slots + tid)));
        const unsigned long long second = __ldcg(slots + grid + tid);
        if (kMax) mx = static_cast<unsigned int>(second);
        else g = __longlong_as_double(static_cast<long long>(second));
        if (blockIdx.x == 0) counts = __ldcg(slots + 2 * grid + tid);
      }
      x = warp_sum(x);
      if (kMax) mx = __reduce_max_sync(0xFFFFFFFFu, mx);
      else g = warp_sum(g);
      if (blockIdx.x == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) counts += __shfl_xor_sync(0xFFFFFFFFu, counts, o);
      }
      if (lane == 0) {
        sh.red[turn][tid >> 5][0] = static_cast<unsigned long long>(__double_as_longlong(x));
        sh.red[turn][tid >> 5][1] = kMax ? mx : static_cast<unsigned long long>(__double_as_longlong(g));
        sh.red[turn][tid >> 5][2] = counts;
      }
    }
    __syncthreads();
  }
  out.a = out.g = 0.0;
  out.amax = 0;
  out.counts = 0;
  for (unsigned int w = 0; w < warps; ++w) {
    out.a += __longlong_as_double(static_cast<long long>(sh.red[turn][w][0]));
    if (kMax) out.amax = max(out.amax, static_cast<unsigned int>(sh.red[turn][w][1]));
    else out.g += __longlong_as_double(static_cast<long long>(sh.red[turn][w][1]));
    out.counts += sh.red[turn][w][2];
  }
  return sh.failed == 0;
}

// A sum's share as a fixed-point number of 80 bits under 2^e, in two parts of which a word holds one beside a 16-bit count of
// arrivals: sixteen bits up, so that the parts of 160 CTAs add up without reaching the count or the word's end.
__device__ __forceinline__ double power_of_two(int e) { return __hiloint2double((e + 1023) << 20, 0); }
__device__ __forceinline__ void split_fixed(double x, int e, unsigned long long& hi, unsigned long long& lo) {
  const double s = x * power_of_two(39 - e), f = floor(s);
  hi = static_cast<unsigned long long>(__double2ll_rn(f)) << 16;
  lo = static_cast<unsigned long long>(__double2ll_rn((s - f) * 0x1p40)) << 16;
}
__device__ __forceinline__ double join_fixed(unsigned long long hi, unsigned long long lo, int e) {
  return fma(static_cast<double>(lo >> 16), 0x1p-40, static_cast<double>(static_cast<long long>(hi) >> 16)) * power_of_two(e - 39);
}

// After the start pass and the iterations of a resident matrix, all threads of all CTAs of a grid: the sums of exchange() in
// one trip.  A CTA adds its parts to the words of the meeting and polls them until everybody's are in: the data is its own
// arrival, so that nothing has to be made visible before it or read after it, where exchange()'s release waits for the
// codes written in the pass and its slots are another trip.  From the last arrival until all go on 1.5 to 2.1 us on 2048 x
// 2048 and 1.3 to 1.6 on 5003 x 2352, by exchange() 2.5 to 2.9.  (A matrix that streams meets by exchange(): its passes are long, and the words cost its
// search registers, 760 -> 806 us a call of 28672 x 8192.)
// 4 den is a multiple of 2^-18 below 2^29 a block, its sum exact.  gsum, the error minus sum W^2, is rounded to multiples of at
// most 2^-77 of sum W^2, which everybody has from the first meeting: 160 CTAs are off by 2^-70 of it together, where the
// binary64 sums that the error is made of round by 2^-53, and a share above 2^-25 of it keeps every bit.  (Nearest codes
// leave hardly more error than zeros would; a share beyond twice sum W^2 is announced in the fifth word, and everybody
// sees so and goes through exchange() instead.)  Nothing that the CTAs wrote before is visible after.
template <typename S>
__device__ __forceinline__ bool meet_by_sums(S& sh, const SoloArgs& a, unsigned int pass, bool& beyond, Totals& out) {
  __syncthreads();
  const unsigned int tid = threadIdx.x, lane = tid & 31u, grid = gridDim.x, turn = pass & 1u;
  if (tid < 32) {
    double x = 0.0, g = 0.0;
    if (lane < blockDim.x / 32) {
      x = sh.part[lane][0];
      g = sh.part[lane][1];
    }
    x = warp_sum(x);
    g = warp_sum(g);
    const int blocks = 32 - __clz(a.m.t[0].nblk);   // nblk < 2^blocks
    const int e_a = 29 + blocks, e_g = sh.error_exp;
    const bool fits = fabs(g) < power_of_two(e_g) && !(a.idle == kShareBeyond && blockIdx.x == 1);
    unsigned long long word[4];
    split_fixed(x, e_a, word[0], word[1]);
    split_fixed(fits ? g : 0.0, e_g, word[2], word[3]);
    unsigned long long mine = fits ? 0ull : 1ull << 16;
#pragma unroll
    for (unsigned int i = 0; i < 4; ++i) mine = lane == i ? word[i] : mine;
    const unsigned int zeros = sh.zeros[0];
    const unsigned long long wide = count_of(sh.wide[0], sh.wide_high[0]);
    __syncwarp();
    if (lane == 0) {
      sh.zeros[0] = sh.wide[0] = sh.wide_high[0] = 0u;
      if (zeros != 0u) atomicAdd(sum_words(a) + 2 * kSetWords, static_cast<unsigned long long>(zeros));
      if (wide != 0ull) atomicAdd(sum_words(a) + 2 * kSetWords + 1, wide);
    }
    __syncwarp();
    if (zeros != 0u || wide != 0ull) __threadfence();
    unsigned long long* const at = sum_words(a) + turn * kSetWords + lane;
    unsigned long long before = 0, seen = 0;
    if (lane < kSumWords) {
      if (pass > 2) before = sh.before[turn][lane];
      if (a.idle != kNobodyMeetsAgain) atomicAdd(at, mine + 1);
    }
    // (what is done with the words is done on every poll: after a pass its code comes from L2, a microsecond better spent while
    // others are late)
    unsigned int polls = 0;
    bool all;
    do {
      if (lane < kSumWords) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(at) : "memory");
      const unsigned long long sum = seen - before - grid;
      all = __all_sync(0xFFFFFFFFu, lane >= kSumWords || (sum & 0xFFFFull) == 0ull);
#pragma unroll
      for (unsigned int i = 0; i < 4; ++i) word[i] = __shfl_sync(0xFFFFFFFFu, sum, i);
      const unsigned long long over = __shfl_sync(0xFFFFFFFFu, sum, 4);
      if (lane == 0) {
        sh.red[turn][0][0] = static_cast<unsigned long long>(__double_as_longlong(join_fixed(word[0], word[1], e_a)));
        sh.red[turn][0][1] = static_cast<unsigned long long>(__double_as_longlong(join_fixed(word[2], word[3], e_g)));
        sh.red[turn][0][2] = over;
      }
    } while (!all && ++polls < kGridWaitLimit);
    if (lane < kSumWords) sh.before[turn][lane] = seen;
    if (!all && lane == 0) sh.failed = 1;
  }
  __syncthreads();
  out.a = __longlong_as_double(static_cast<long long>(sh.red[turn][0][0]));
  out.g = __longlong_as_double(static_cast<long long>(sh.red[turn][0][1]));
  out.counts = 0;
  beyond = sh.red[turn][0][2] != 0ull;
  return sh.failed == 0;
}

// The meeting after the start pass (`first`) or an iteration: by sums where a grid goes on from it, else by exchange().
template <typename S>
__device__ __forceinline__ bool combine(S& sh, const SoloArgs& a, unsigned long long tag, unsigned int& exchanged, unsigned int& met,
                                        bool first, bool last, Totals& out) {
  if constexpr (S::kResident && !S::kCluster && !S::kFinal) {
    if (gridDim.x > 1 && !last) {
      bool beyond;
      if (!meet_by_sums(sh, a, ++met, beyond, out)) return false;
      if (!beyond) return true;
    }
  }
  return exchange<false>(sh, a, tag, ++exchanged, first, last, out);
}

// Zeroes of the tiled layout: rows up to a multiple of 128, scale columns up to a multiple of 4.  A warp clears the rows of
// one tile of the last tile row, a lane the words of rows lane, lane + 32, lane + 64 and lane + 96, which lie side by side.
// (Counted in tiles: the number of padding words can pass 2^32, at one row of 2.2e9 weights.)
__device__ __forceinline__ void clear_tile_padding(const Params& p, unsigned int rows, uint8_t* tiled) {
  const unsigned int nbc = p.nbc, ct = (nbc + 3) / 4, valid = rows & 127u, lane = threadIdx.x & 31u;
  const unsigned int me = blockIdx.x * blockDim.x + threadIdx.x, all = gridDim.x * blockDim.x;
  const bool words = reinterpret_cast<uintptr_t>(tiled) % 4 == 0;
  if (valid != 0)
    for (unsigned int tile = me >> 5; tile < ct; tile += all >> 5) {
      uint8_t* const at = tiled + (static_cast<size_t>(rows >> 7) * ct + tile) * 512 + lane * 16;
#pragma unroll
      for (unsigned int i = 0; i < 4; ++i) {
        if (lane + 32 * i < valid) continue;
        if (words) reinterpret_cast<unsigned int*>(at)[i] = 0u;
        else at[4 * i] = at[4 * i + 1] = at[4 * i + 2] = at[4 * i + 3] = 0;
      }
    }
  if (nbc % 4 != 0)
    for (unsigned int r = me; r < rows; r += all)
      for (unsigned int c = nbc; c < ct * 4; ++c) tiled[swizzled_offset(r, c, ct)] = 0;
}

// The tiled copy of a resident matrix's scales: every warp its own blocks', from their states.  (No CTA waits for another's
// scales; 5003 x 2352: the meeting before tile_scales and that pass itself took 5 us, this 1.6.)
template <typename S>
__device__ __forceinline__ void tile_resident(S& sh, const Params& p, uint8_t* tiled) {
  const unsigned int lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = gridDim.x * cta_warps<S>(), ct = (p.nbc + 3) / 4;
  unsigned int at = slots_of(sh, warp) + kQTileBytes + lane * 8;
  for (unsigned int tile = warp_number(warp); tile < p.ntiles; tile += warps) {
    const unsigned int b = tile * 32 + lane, row = __umulhi(2u * b, p.nbc_magic) >> p.nbc_shift;
    if (b < p.nblk) tiled[swizzled_offset(row, b - row * p.nbc, ct)] = static_cast<uint8_t>((lds64(at).y >> 12) & 0x7Fu);
    at += kQTileBytes + kQStateBytes;
  }
}

template <int kMode, int kPlace>
__global__ void __launch_bounds__(kSoloWarps * 32, 1) solo_kernel(const __grid_constant__ SoloArgs a) {
  extern __shared__ __align__(128) unsigned char tile_slots[];
  constexpr bool kRes = kPlace != kStreamed, kCluster = kPlace == kKeptInCluster, kNoIter = kMode == kNoIterations;
  __shared__ SoloShared<kPlace, kNoIter> sh;
  if (kCluster) {   // (waited for before anything is sent to another CTA)
    if (threadIdx.x == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sh.landed[i])) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_arrive();
  }
  after_previous();
  const int tid = threadIdx.x;
  const Params& p = a.m.t[0];
  const int T = kNoIter ? 0 : p.max_iters, flags = p.flags;   // (the other modes are launched with iterations only)
  unsigned long long epoch = 0;
  if (!kCluster && gridDim.x > 1) epoch = __ldcg(reinterpret_cast<const unsigned long long*>(a.exchange + kEpochAt));
  if (kRes) load_resident(a.m, smem_u32(tile_slots), a.per_warp);
  if (!kCluster && gridDim.x > 1 && blockIdx.x == 0) {
    if (tid == 0) open_counter(a, a.nonce + epoch);
    if (!kNoIter && tid < static_cast<int>(kWords)) __stcg(sum_words(a) + tid, 0ull);   // (seen by all after the first exchange)
  }
  if (tid == 0) {
    sh.view[0].packed = p.packed;
    sh.view[0].scales = p.scales;
    sh.view[0].state = p.state;
    sh.view[0].tiled = kNoIter ? a.tiled : nullptr;
    sh.amax[0] = sh.zeros[0] = sh.wide[0] = sh.wide_high[0] = 0u;
    sh.start[0] = 0u;
    sh.count[0] = sh.total = p.ntiles;
    sh.slots = smem_u32(tile_slots);
    sh.per_warp = kRes ? a.per_warp : kQStages;
    sh.tiled_only = a.tiled_only;
    sh.failed = 0;
  }
  if (tid < 32) sh.part[tid][0] = sh.part[tid][1] = 0.0;
  if (kMode == 0 || kMode >= 3) {
    const int n_beta = p.n_beta, step = p.beta_step_pct;
    for (int k = tid; k < n_beta; k += static_cast<int>(blockDim.x)) {
      const float lo = static_cast<float>((100.0 + static_cast<double>((k - n_beta / 2) * step)) / 100.0);
      const float hi = static_cast<float>((100.0 + static_cast<double>((k + 1 - n_beta / 2) * step)) / 100.0);
      sh.beta[k] = make_float2(lo, hi);
    }
  }
  // what of the report does not depend on the sums
  if (blockIdx.x == 0 && a.result != nullptr)
    for (int i = T + 1 + tid; i <= SOAR_MAX_ITERS; i += static_cast<int>(blockDim.x)) a.result->trace_alpha[i] = a.result->trace_sse[i] = 0.0;
  __syncthreads();
  if ((kNoIter || kRes) && a.tiled != nullptr) clear_tile_padding(p, a.rows, a.tiled);
  unsigned int exchanged = 0, met = 0;   // meetings through slots and by sums
  Totals tot;
  bool ok;
  amax_pass(sh, a.m);
  if (kCluster) {
    __syncwarp();
    cluster_wait();
  }
  ok = exchange<true>(sh, a, a.nonce + epoch, ++exchanged, false, false, tot);
  const double sumsq = tot.a;
  const unsigned int amax_bits = tot.amax;
  const int st = status_from_amax(amax_bits);
  const float alpha0 = amax_bits == 0 ? 1.0f : __fdiv_rn(bits_to_mag(amax_bits), 2688.0f);
  float alpha = alpha0;
  int iters = 0;
  unsigned long long zero_blocks = 0, wide = 0;
  double sse = 0.0;
  // every thread keeps the call's scalars itself, and writes the same alpha for the passes to read
  sh.alpha[0] = alpha;
  // 2^error_exp: more than twice sum W^2, at most four times (a matrix of zeros has no error, any will do)
  sh.error_exp = max((__double2hiint(sumsq) >> 20) - 1023, -300) + 2;
  if (ok && !(st & (SOAR_STATUS_NONFINITE | SOAR_STATUS_RANGE))) {
    const bool tile_after = !kNoIter && a.tiled != nullptr;
    init_pass(sh, a.m);
    ok = combine(sh, a, a.nonce + epoch, exchanged, met, true, kNoIter, tot);
    if (kNoIter && blockIdx.x != 0 && (ok || !kCluster)) return;   // nothing left to do but CTA 0's report
    if (st == 0) sse = fmax(sumsq + tot.g, 0.0);
    zero_blocks = tot.counts & 0xFFFFFFFFull;
    wide = tot.counts >> 32;
    if (tid == 0) {
      sh.trace_alpha[0] = static_cast<double>(alpha0);
      sh.trace_sse[0] = sse;
    }
    const bool may_stop = p.early_stop_rel > 0.0f;
    if constexpr (!kNoIter)
    for (int t = 0; st == 0 && ok && t < T; ++t) {
      // Eq. 5; the numerator follows from the two sums carried (see file_sums)
      const double ad = static_cast<double>(alpha), den = 0.25 * tot.a;
      if (den > 0.0 && !(flags & SOAR_FLAG_KEEP_ALPHA)) alpha = static_cast<float>((ad * ad * den - tot.g) / (2.0 * ad * den));
      sh.alpha[0] = alpha;
      iterate_pass<kMode>(sh, a.m, (t & 1) != 0, may_stop || t == T - 1, t != T - 1 || (kRes && tile_after));
      const bool last = t == T - 1 && !tile_after;
      ok = combine(sh, a, a.nonce + epoch, exchanged, met, false, last, tot);
      if (last && blockIdx.x != 0 && (ok || !kCluster)) return;
      const double cur = fmax(sumsq + tot.g, 0.0);
      wide += tot.counts;
      iters = t + 1;
      if (tid == 0) {
        sh.trace_alpha[iters] = static_cast<double>(alpha);
        sh.trace_sse[iters] = cur;
      }
      const bool stop = stops_after(sse, cur, p.early_stop_rel);
      sse = cur;
      if (stop) break;
    }
    if (ok && tile_after) {
      if constexpr (kRes) tile_resident(sh, p, a.tiled);
      else tile_scales(p, a.rows, a.tiled);
    }
  }
  let_next_begin();
  if (!ok) {
    // a wait ran out: say so in the report and leave, a CTA of a cluster not before everybody there has given up or ended
    if (kCluster) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
    }
    if (tid == 0) {
      if (!kCluster && gridDim.x > 1) *reinterpret_cast<volatile unsigned long long*>(a.exchange + kEpochAt) = epoch + 1;
      if (a.result != nullptr) {
        a.result->status = SOAR_STATUS_INTERNAL;
        a.result->iters_run = 0;
      }
    }
    return;
  }
  if (blockIdx.x != 0) return;
  if (tid == 0) {
    if (!kCluster && gridDim.x > 1) *reinterpret_cast<volatile unsigned long long*>(a.exchange + kEpochAt) = epoch + 1;
    if (!kCluster && !kNoIter && gridDim.x > 1 && met > 0) {   // (the last meeting's arrivals came after the counts)
      __threadfence();
      zero_blocks += __ldcg(sum_words(a) + 2 * kSetWords);
      wide += __ldcg(sum_words(a) + 2 * kSetWords + 1);
    }
    *a.alpha = alpha;
    if (a.result != nullptr) {
      soar_result* const res = a.result;
      res->status = st;
      res->iters_run = iters;
      res->alpha = alpha;
      res->amax = bits_to_mag(amax_bits);
      res->sse = sse;
      res->sse_init = st == 0 ? sh.trace_sse[0] : 0.0;
      res->sumsq = (st & SOAR_STATUS_ZERO_TENSOR) ? 0.0 : sumsq;
      res->zero_blocks = static_cast<int64_t>(zero_blocks);
      res->wide_candidates = static_cast<int64_t>(wide);
    }
  }
  if (a.result != nullptr) {
    __syncthreads();
    for (int i = tid; i <= T; i += static_cast<int>(blockDim.x)) {
      a.result->trace_alpha[i] = i == 0 ? static_cast<double>(alpha0) : i <= iters ? sh.trace_alpha[i] : 0.0;
      a.result->trace_sse[i] = (i <= iters && st == 0) ? sh.trace_sse[i] : 0.0;
    }
  }
}

// ------------------------------------------------------------------ calls without iterations on larger matrices
//
// The max-based rule alone is two light passes with one meeting between them.  As two chained kernels (launch_chained) of
// 32 warps an SM the boundary is the meeting: no cooperative launch and no arrival to wait for.  Every CTA leaves its
// numbers in a slot; the second kernel reads all of them at its head, its first tiles on their way, and the CTA that ends last
// adds up the second pass's and writes the report.  4096 x 8192: 55.7 us as launches of their own, 40.3 in the one kernel,
// 36.6 as two, 35.1 with the first tiles of the second on their way before it waits; 28672 x 8192: 79 us for the maximum,
// 105 us for the codes (5.6 TB/s, 194 instructions a block issued in 83 % of the cycles).

constexpr int kMaxBasedThreads = 1024;

struct __align__(128) MaxBasedShared {
  static constexpr bool kOrdered = true, kSolo = true, kResident = false, kFinal = true;
  View view[1];
  double part[kMaxBasedThreads / 32][2];
  double red[kMaxBasedThreads / 32][2];
  float alpha[1];
  unsigned int amax[1], zeros[1], wide[1], wide_high[1];
  unsigned int start[1], count[1], total;
  unsigned int slots, per_warp;
  int tiled_only;
  unsigned int most, zeros_all, wide_all, arrived;
};

// A CTA's numbers: sum W^2, error minus sum W^2; the maximum's bits, zero blocks, wide candidates.
struct MaxBasedSlot {
  double sumsq, gsum;
  unsigned int amax, zeros, wide, pad;
};
static_assert(sizeof(MaxBasedSlot) <= 2 * kSlotBytes, "the exchange's workspace holds a slot per CTA");

__device__ __forceinline__ MaxBasedSlot* max_based_slots(const SoloArgs& a) { return reinterpret_cast<MaxBasedSlot*>(a.exchange + 256); }

__device__ __forceinline__ void max_based_head(MaxBasedShared& sh, const SoloArgs& a) {
  extern __shared__ __align__(128) unsigned char tile_slots[];
  const Params& p = a.m.t[0];
  const unsigned int tid = threadIdx.x;
  if (tid == 0) {
    sh.view[0].packed = p.packed;
    sh.view[0].scales = p.scales;
    sh.view[0].state = nullptr;
    sh.view[0].tiled = a.tiled;
    sh.amax[0] = sh.zeros[0] = sh.wide[0] = sh.wide_high[0] = 0u;
    sh.start[0] = 0u;
    sh.count[0] = sh.total = p.ntiles;
    sh.slots = smem_u32(tile_slots);
    sh.per_warp = kQStages;
    sh.tiled_only = a.tiled_only;
    sh.most = sh.zeros_all = sh.wide_all = 0u;
  }
  if (tid < kMaxBasedThreads / 32) sh.part[tid][0] = sh.part[tid][1] = 0.0;
  __syncthreads();
}

// Sum of the CTAs' numbers `of(slot)`, the same bits in every thread: warp w adds slots 32 w .. 32 w + 31.
template <typename Of>
__device__ __forceinline__ double max_based_sum(MaxBasedShared& sh, int which, Of of) {
  const unsigned int tid = threadIdx.x, grid = gridDim.x, warps = (grid + 31) / 32;
  if (tid < warps * 32) {
    const double v = warp_sum(tid < grid ? of(tid) : 0.0);
    if ((tid & 31u) == 0) sh.red[tid >> 5][which] = v;
  }
  __syncthreads();
  double v = 0.0;
  for (unsigned int w = 0; w < warps; ++w) v += sh.red[w][which];
  return v;
}

__global__ void __launch_bounds__(kMaxBasedThreads, 1) max_based_amax_kernel(const __grid_constant__ SoloArgs a) {
  __shared__ MaxBasedShared sh;
  max_based_head(sh, a);
  after_previous();
  let_next_begin();
  amax_pass(sh, a.m);
  // (after the pass: before it, it delays the first copies: 4096 x 8192 35.4 -> 35.6 us)
  if (a.tiled != nullptr) clear_tile_padding(a.m.t[0], a.rows, a.tiled);
  __syncthreads();
  if (threadIdx.x < 32) {
    const double v = warp_sum(sh.part[threadIdx.x][0]);
    if (threadIdx.x == 0) {
      MaxBasedSlot& s = max_based_slots(a)[blockIdx.x];
      s.sumsq = v;
      s.amax = sh.amax[0];
      if (blockIdx.x == 0) *reinterpret_cast<unsigned int*>(a.exchange + kCounterAt) = 0u;
    }
  }
}

__global__ void __launch_bounds__(kMaxBasedThreads, 1) max_based_codes_kernel(const __grid_constant__ SoloArgs a) {
  __shared__ MaxBasedShared sh;
  max_based_head(sh, a);
  const unsigned int tid = threadIdx.x, grid = gridDim.x;
  MaxBasedSlot* const slots = max_based_slots(a);
  unsigned int* const counter = reinterpret_cast<unsigned int*>(a.exchange + kCounterAt);
  double sumsq = 0.0;
  unsigned int amax_bits = 0;
  int st = 0;
  float alpha = 1.0f;
  // the weights are read before the first kernel's end is waited for: it let this one begin only after its own wait, and
  // writes none
  init_pass(sh, a.m, [&]() {
    after_previous();
    if (tid < grid) atomicMax(&sh.most, __ldcg(&slots[tid].amax));
    sumsq = max_based_sum(sh, 0, [&](unsigned int j) { return __ldcg(&slots[j].sumsq); });
    amax_bits = sh.most;
    st = status_from_amax(amax_bits);
    alpha = amax_bits == 0 ? 1.0f : __fdiv_rn(bits_to_mag(amax_bits), 2688.0f);
    sh.alpha[0] = alpha;
    return !(st & (SOAR_STATUS_NONFINITE | SOAR_STATUS_RANGE));
  });
  let_next_begin();
  __syncthreads();
  if (tid < 32) {
    const double v = warp_sum(sh.part[tid][1]);
    if (tid == 0) {
      slots[blockIdx.x].gsum = v;
      slots[blockIdx.x].zeros = sh.zeros[0];
      slots[blockIdx.x].wide = sh.wide[0];   // at most one a block here
      __threadfence();
      sh.arrived = atomicAdd(counter, 1u);
    }
  }
  __syncthreads();
  if (sh.arrived != grid - 1) return;
  // the last CTA: the report
  __threadfence();
  if (tid < grid) {
    atomicAdd(&sh.zeros_all, __ldcg(&slots[tid].zeros));
    atomicAdd(&sh.wide_all, __ldcg(&slots[tid].wide));
  }
  const double gsum = max_based_sum(sh, 1, [&](unsigned int j) { return __ldcg(&slots[j].gsum); });
  soar_result* const res = a.result;
  if (tid == 0) *a.alpha = alpha;
  if (res == nullptr) return;
  const double sse = st == 0 ? fmax(sumsq + gsum, 0.0) : 0.0;
  if (tid == 0) {
    res->status = st;
    res->iters_run = 0;
    res->alpha = alpha;
    res->amax = bits_to_mag(amax_bits);
    res->sse = res->sse_init = sse;
    res->sumsq = (st & SOAR_STATUS_ZERO_TENSOR) ? 0.0 : sumsq;
    res->zero_blocks = static_cast<int64_t>(sh.zeros_all);
    res->wide_candidates = static_cast<int64_t>(sh.wide_all);
  }
  if (tid <= SOAR_MAX_ITERS) {
    res->trace_alpha[tid] = tid == 0 ? static_cast<double>(alpha) : 0.0;
    res->trace_sse[tid] = tid == 0 ? sse : 0.0;
  }
}
