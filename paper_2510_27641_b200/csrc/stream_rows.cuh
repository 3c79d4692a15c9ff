// Rows that are streamed: for calls with more rows than the GPU can keep on chip at once.  Included by
// select_topp.cu.
//
// Held in shared memory, 148 SMs take some 37 rows of 131072 entries, and the latencies of a search (barriers,
// exchanges, scans) are paid once per wave of them (256 rows: 240 us).  Here nothing of a row stays on chip but a
// histogram and bits, and a row is read twice, each time through a ring of 16-byte copies that keeps 32 to 64 KB
// per CTA under way.  A row is dealt to a cluster of one, two or four CTAs (pick_cluster_stream; at least two where it is
// longer than a CTA's words allow); the searches of different rows overlap one another's reads.
// The CTAs of a row exchange their octaves and one octave's bins after the first pass, the keys of the bin after the
// second, and their kept counts, and each decides for itself.
//
// With that, the passes are bound by instruction issue and by the wavefronts of shared-memory atomics, so each does
// as little per entry as it can:
//   pass 1  adds the top 15 mantissa bits to one word per bin (exponent and five mantissa bits) -- one atomic, not
//           two words for an exact sum -- which names the threshold's bin in all but a few of 10^4 rows.  The
//           other nine bits, times 2^e, are added up by the thread.  What bounds the pass is the atomic: 4.1
//           wavefronts of random banks, two cycles each;
//   pass 2  notes two bits per entry, above the bin / in the bin, in per-thread words (no votes) and adds up
//           the low bits of what lies above.  The keys of the bin are then fetched by their bits.
// The masses tell whether the bin was the right one; if not, the row is read again for its neighbour.  They are floating
// point sums whose rounding depends on how the row was dealt to threads, so a threshold counts only if the target
// is further from both of its masses than rounding can reach (kStreamDoubt); else -- rows whose masses meet the
// target exactly, rows of tiny values -- the row is searched once more with the low bits added up
// per octave too (a second atomic), in the same integers and with the same comparisons as the search in shared memory.
// The lists are therefore the same in every form.
// 256 rows of 131072, p = 0.9, uniform / Zipf / ties: 96 / 81 / 93 us against 117 / 102 / 142 with exact two-word bins,
// votes and 128-entry emission; the test against rounding then added 1 % (cold cache 102 / 90 / 96 -> 104 / 90 / 97).
#pragma once

constexpr int kStreamThreads = 512;
constexpr int kStreamWarps = kStreamThreads / 32;
constexpr int kStreamRound = 4 * kStreamThreads;   // entries per round of the CTA: 8 KB
constexpr int kStreamBatch = 4;                    // rounds per commit group
constexpr int kStreamGroups = 2;                   // groups in the ring
constexpr int kStreamMax = 131072;                 // entries per CTA: 64 rounds
constexpr int kStreamAlign = 32;                   // slices of a cluster start on whole 128-byte lines
constexpr int kStreamShift = 18;                   // level-1 bins: the key's bits above these
constexpr int kStreamBins = 8192;
constexpr int kStreamCand = 4096;                  // keys of the bin that are gathered
constexpr int kStreamWords = kStreamMax / 32;      // words of a bit per entry: [8 rounds][thread], 4 bits a round
constexpr int kStreamLow = kStreamBins + kOctaves;  // (exact search) sums of the low nine bits per octave, behind the bins
constexpr int kStreamStore = kStreamLow + kOctaves;
// Two ways to add up the target, or a mass it is compared with, differ by less than this share of the total.  In
// binary64 a thread adds up to 256 values and the CTA 512 such sums (2^-44 if every one rounded the same way); sixteen
// low parts in binary32 are off by at most 15 x 2^-25 of their sum, which is at most 2^-14 of the values'.
constexpr double kStreamDoubt = 0x1p-40, kStreamDoubt32 = 0x1p-34;
static_assert(2 * kStreamWords <= kStreamStore, "both bit masks take the histogram's bytes");
static_assert(static_cast<long long>(kStreamMax) << 15 <= (1ll << 32), "a bin's word cannot wrap");

struct StreamShared {
  alignas(16) unsigned int store[kStreamStore];  // histogram, then the bits "above the bin" and "in the bin"
  alignas(16) float ring[kStreamGroups * kStreamBatch * kStreamRound];
  int negative;                // a negative input was met
  int tiny;                    // (exact search) a key below 512, of which the histogram's word of bin 0 holds nothing
  int oct_min, oct_max, n_cand;
  double part;                 // this CTA's share of a sum over the row
  int kept;                    // kept entries of this CTA (these seven are read by peers, like the store and the scratch's
                               // octaves and keys)
  int row_max;                 // highest octave of the row; the last one if an input is invalid
  double row_part;             // (a level of a well filled bin) the row's sum
  Found fd;
  double sum[kStreamWarps];
  int warp_cnt[kStreamWarps];
};
// The ring is idle outside the passes and then holds the scratch of the search and the staging lines of
// the emission.
struct StreamScratch {
  unsigned long long oct[kOctaves];
  LevelHist lv;
  Picks pk;
  unsigned int keys[kStreamCand];
  unsigned int place[kStreamCand];   // entry of the slice
  unsigned int all_keys[kStreamCand];  // (clusters) the keys of the whole row's bin
};
constexpr int kStreamStage = 528;    // ints of a warp's staging line (512 entries, shifted by up to 3)
static_assert(sizeof(StreamScratch) <= sizeof(StreamShared::ring), "scratch in the ring");
static_assert(kStreamWarps * kStreamStage * sizeof(int) <= sizeof(StreamShared::ring), "staging in the ring");
static_assert(2 * (sizeof(StreamShared) + 1024) <= 227 * 1024, "two CTAs per SM");

// Word of a bin: 33 words to an octave's 32 bins, or values with one mantissa in many octaves (quantised rows) would
// share a bank.
__device__ __forceinline__ int stream_word(int bin) { return bin + (bin >> 5); }

// Adds one positive key to the histogram at shared-memory address `hist`.  The two shifts of the address are
// multiplications by values the compiler cannot see through: the multiply-add pipe has room, the integer
// pipe (half a warp instruction a clock) is what bounds the pass.
struct StreamConst {
  unsigned int by18, by23, four;
};
__device__ __forceinline__ StreamConst stream_const() {
  StreamConst c;
  asm volatile("mov.u32 %0, 16384;\n\tmov.u32 %1, 512;\n\tmov.u32 %2, 4;" : "=r"(c.by18), "=r"(c.by23), "=r"(c.four));
  return c;
}
__device__ __forceinline__ void stream_bump(uint32_t hist, const StreamConst& c, unsigned int key, unsigned int piece) {
  const unsigned int bin = __umulhi(key, c.by18), oct = __umulhi(key, c.by23);
  const uint32_t at = bin * c.four + (oct * c.four + hist);
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at), "r"(piece) : "memory");
}
// The top 15 mantissa bits of a key.  (Unless the search is exact, a denormal counts as if it were normal.)
template <bool kExact>
__device__ __forceinline__ unsigned int stream_piece(unsigned int key) {
  return ((key >> 9) & 0x3fffu) | ((!kExact || key >= 0x800000u) ? 0x4000u : 0u);
}

// Walks the row through the ring: f(round, bit patterns) for every batch of rounds, this thread's float4 of each,
// zeros beyond n, in whole batches of the CTA (all threads call f equally often).
template <class F>
__device__ __forceinline__ void stream_pass(StreamShared& sh, const float* A, int n, F f) {
  const int tid = threadIdx.x;
  const int rounds = (n + kStreamRound - 1) / kStreamRound;
  const int groups = (rounds + kStreamBatch - 1) / kStreamBatch;
  const uint32_t dst = smem_u32(sh.ring) + tid * 16;
  auto issue = [&](int gq) {
    if (gq < groups) {
#pragma unroll
      for (int j = 0; j < kStreamBatch; ++j) {
        const int at = (gq * kStreamBatch + j) * kStreamRound + 4 * tid;
        const int left = n - at;
        cp_async16_zfill(dst + ((gq % kStreamGroups) * kStreamBatch + j) * (kStreamRound * 4), A + (left > 0 ? at : 0),
                         left >= 4 ? 16u : (left > 0 ? 4u * left : 0u));
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int gq = 0; gq < kStreamGroups - 1; ++gq) issue(gq);
  for (int gq = 0; gq < groups; ++gq) {
    issue(gq + kStreamGroups - 1);  // (its slot was emptied by this thread one turn ago)
    asm volatile("cp.async.wait_group %0;" ::"n"(kStreamGroups - 1) : "memory");
    unsigned int k[4 * kStreamBatch];
#pragma unroll
    for (int j = 0; j < kStreamBatch; ++j) {
      const uint4 v = *reinterpret_cast<const uint4*>(sh.ring + ((gq % kStreamGroups) * kStreamBatch + j) * kStreamRound + 4 * tid);
      k[4 * j] = v.x;
      k[4 * j + 1] = v.y;
      k[4 * j + 2] = v.z;
      k[4 * j + 3] = v.w;
    }
    f(gq * kStreamBatch, k);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// What a key's 15 bits in the histogram leave of its value: its low nine mantissa bits.
__device__ __forceinline__ float stream_rest(unsigned int k) { return __uint_as_float(k) - __uint_as_float(k & ~0x1ffu); }

// Sum over the CTA in a fixed order; every thread gets it.  Two barriers.
__device__ __forceinline__ double stream_sum(StreamShared& sh, double s) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFull, s, d);
  if ((threadIdx.x & 31) == 0) sh.sum[threadIdx.x >> 5] = s;
  __syncthreads();
  s = sh.sum[0];
#pragma unroll
  for (int w = 1; w < kStreamWarps; ++w) s += sh.sum[w];
  __syncthreads();
  return s;
}

// kMasses: the caller wants the masses (diag), so they are added up in binary64.  Otherwise they only have to tell
// which threshold is the right one, and the low parts of a batch are added up in binary32 first, the rare row in doubt
// being searched again (256 rows of 131072, uniform / Zipf / ties: 107 / 96 / 102 us with masses, 103 / 90 / 97 without).
// kShared: a row has several CTAs (known to the compiler, since the exchanges cost one CTA a row 3 us of 104).
template <bool kMasses, bool kShared>
__global__ void __launch_bounds__(kStreamThreads, 2) stream_rows_kernel(const __grid_constant__ SelectParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamShared& sh = *reinterpret_cast<StreamShared*>(smem_raw);
  StreamScratch& sc = *reinterpret_cast<StreamScratch*>(sh.ring);
  constexpr int N = 4 * kStreamBatch;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = kShared ? static_cast<int>(cluster.num_blocks()) : 1, rank = kShared ? static_cast<int>(cluster.block_rank()) : 0;
  auto csync = [&]() {
    if (kShared) cluster.sync(); else __syncthreads();
  };
  // sum of a number of every CTA of the row, in their order (all lanes of a warp)
  auto row_sum = [&](double* at) {
    const double mine = (lane < cs) ? *cluster.map_shared_rank(at, lane < cs ? lane : 0) : 0.0;
    double s = __shfl_sync(kFull, mine, 0);
    for (int r = 1; r < cs; ++r) s += __shfl_sync(kFull, mine, r);
    return s;
  };
  const int list = kShared ? blockIdx.y : blockIdx.x;  // (used slot, sequence, group)
  const int g = list % P.G;
  const int b = (list / P.G) % P.B;
  const int slot = list / (P.G * P.B);
  const long long out_list = (static_cast<long long>(P.layer_of[slot]) * P.B + b) * P.G + g;
  unsigned int* const hist = sh.store;
  const uint32_t hist_at = smem_u32(hist);
  const StreamConst consts = stream_const();
  auto clear = [&]() {
    for (int i = tid; i < kStreamStore / 4; i += kStreamThreads) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
      sh.negative = 0;
      sh.tiny = 0;
      sh.oct_min = kOctaves;
      sh.oct_max = -1;
    }
    __syncthreads();
  };
  clear();
  pdl_wait();  // nothing is read or written before the previous kernel's end ...
  pdl_launch_dependents();  // ... and only then may the next one be scheduled
  long long Lll = P.kv_len[b];
  if (Lll < 0) Lll = 0;
  if (Lll > P.L_stride) Lll = P.L_stride;
  const int L_row = static_cast<int>(Lll);
  const int per_cta = kShared ? slice_of(L_row, cs, kStreamAlign) : L_row;
  const int lo = kShared ? min(L_row, rank * per_cta) : 0, L = kShared ? min(L_row, lo + per_cta) - lo : L_row;  // this CTA's entries
  const float* A = ((P.agg != nullptr) ? P.agg + static_cast<long long>(list) * P.L_stride
                                       : P.probs[slot] + static_cast<long long>(b) * P.H * P.gamma * P.L_stride) + lo;

  double total = 0.0, target = 0.0, m_gt = 0.0, m_ge = 0.0;
  bool invalid = false, searching = false;
  unsigned int theta = 0u;
  unsigned int* const above_bits = sh.store;
  unsigned int* const in_bits = sh.store + kStreamWords;
  bool exact = false, last_resort = false;
  auto row_word = [&](int bin) {  // a bin's word, over the row
    unsigned long long w = 0ull;
    if constexpr (!kShared) w = hist[stream_word(bin)];
    else for (int r = 0; r < cs; ++r) w += *cluster.map_shared_rank(&hist[stream_word(bin)], r);
    return w;
  };
  auto bin_mass9 = [&](int oct) {  // lane: bin of an octave
    return static_cast<double>(row_word(32 * oct + lane) << 9) * pow2_double(max(oct, 1) - 150);
  };
  int go = 0;                  // 1 / -1: the bin above / below the last one tried is wanted
  auto turn = [&](int want) {  // on to the bin above or below -- or, after a turn back, to an exact search
    if (go == -want) exact = true;
    go = (go == -want) ? 0 : want;
    csync();
    clear();
  };
  for (;;) {
    // ---- pass 1: histogram, total and validity -------------------------------------------------------
    // (unless the search is exact, bin 0 is left out, zeros apart eighteen octaves of denormals whose updates of one
    // word would be serialised; they only count in a row without larger values)
    bool negative = false, tiny = false;
    double mine[4] = {0.0, 0.0, 0.0, 0.0};  // (one sum waits for its adds)
    auto pass1 = [&](auto exactly) {
      constexpr bool kExact = decltype(exactly)::value;
      constexpr unsigned int min_key = kExact ? 1u : 1u << kStreamShift;
      stream_pass(sh, A, L, [&](int, unsigned int (&k)[N]) {
        unsigned int any = 0u;
#pragma unroll
        for (int j = 0; j < N; ++j) any |= k[j];
        if (static_cast<int>(any) < 0) {  // a sign bit: negative -- or -0.0, which is a zero
#pragma unroll
          for (int j = 0; j < N; ++j) {
            negative |= k[j] > 0x80000000u;
            k[j] = (static_cast<int>(k[j]) < 0) ? 0u : k[j];
          }
        }
        // every value of the warp in one bin (ties, constant rows): the warp reduces first
        const unsigned int bin0 = __shfl_sync(kFull, k[0] >> kStreamShift, 0);
        bool one = false;
        if (__all_sync(kFull, (k[0] >> kStreamShift) == bin0)) {
          unsigned int differ = 0u;
#pragma unroll
          for (int j = 1; j < N; ++j) differ |= k[j] ^ k[0];
          one = __all_sync(kFull, (differ >> kStreamShift) == 0u);
        }
        if (one) {
          unsigned int s = 0u, low = 0u;
#pragma unroll
          for (int j = 0; j < N; ++j) {
            s += (k[j] >= min_key) ? stream_piece<kExact>(k[j]) : 0u;
            tiny |= kExact && k[j] - 1u < 0x1ffu;
            low += k[j] & 0x1ffu;
          }
          s = __reduce_add_sync(kFull, s);
          if (lane == 0 && s != 0u) atomicAdd(&hist[stream_word(bin0 & (kStreamBins - 1))], s);
          if (kExact) {
            low = __reduce_add_sync(kFull, low);
            if (lane == 0 && low != 0u) atomicAdd(&hist[kStreamLow + ((bin0 >> 5) & (kOctaves - 1))], low);
          }
        } else {
#pragma unroll
          for (int j = 0; j < N; ++j) {
            if (k[j] >= min_key) stream_bump(hist_at, consts, k[j], stream_piece<kExact>(k[j]));
            tiny |= kExact && k[j] - 1u < 0x1ffu;
            if (kExact && (k[j] & 0x1ffu) != 0u) atomicAdd(&hist[kStreamLow + (k[j] >> 23)], k[j] & 0x1ffu);
          }
        }
        if (!kExact && kMasses) {
#pragma unroll
          for (int j = 0; j < N; ++j) mine[j & 3] += static_cast<double>(stream_rest(k[j]));
        } else if (!kExact) {
          float part = 0.f;
#pragma unroll
          for (int j = 0; j < N; ++j) part += stream_rest(k[j]);
          mine[0] += static_cast<double>(part);
        }
      });
    };
    if (exact) pass1(std::true_type()); else pass1(std::false_type());
    if (__any_sync(kFull, negative) && lane == 0) sh.negative = 1;
    if (__any_sync(kFull, tiny) && lane == 0) sh.tiny = 1;

    // ---- the bin of the threshold ---------------------------------------------------------------------
    const double rest = stream_sum(sh, (mine[0] + mine[1]) + (mine[2] + mine[3]));
    if (kShared && tid == 0) sh.part = rest;
    if (tid < kOctaves) {
      unsigned long long s = 0ull;
#pragma unroll 8
      for (int h = 0; h < 32; ++h) s += hist[33 * tid + h];
      s = (s << 9) + hist[kStreamLow + tid];  // (the low parts: zero unless the search is exact)
      sc.oct[tid] = s;
      const int first = __reduce_min_sync(kFull, (s != 0ull) ? tid : kOctaves);
      const int final = __reduce_max_sync(kFull, (s != 0ull) ? tid : -1);
      if (lane == 0 && first < kOctaves) {
        atomicMin(&sh.oct_min, first);
        atomicMax(&sh.oct_max, final);
      }
    }
    csync();
    if (warp == 0) {
      double t = 0.0, tg = 0.0, carry = 0.0, ab = 0.0, up;
      int bin = -1;
      last_resort = false;
      // of the row: octaves with an entry, and whether an input is invalid (the last octave: infinities and NaN)
      const StreamShared* const peer = (kShared && lane < cs) ? cluster.map_shared_rank(&sh, lane) : &sh;
      const int top = __reduce_max_sync(kFull, (peer->negative != 0) ? kOctaves - 1 : peer->oct_max);
      const int bottom = __reduce_min_sync(kFull, peer->oct_min);
      const bool some_tiny = __any_sync(kFull, peer->tiny != 0);
      auto mass = [&](int e) {
        unsigned long long s = 0ull;
        if constexpr (!kShared) s = sc.oct[e];
        else for (int r = 0; r < cs; ++r) s += *cluster.map_shared_rank(&sc.oct[e], r);
        return s;
      };
      const double row_rest = kShared ? row_sum(&sh.part) : rest;
      if (top >= 0 && top < kOctaves - 1) {
        const int oct = find_octave(top, bottom, P.p, mass, t, tg, carry);
        bin = 32 * oct + find_from_top<5>(bin_mass9(oct), 0.0, carry, tg, ab, up);
        if (go != 0) {  // the next one with an entry, or none
          int at = sh.fd.bin;
          bin = -1;
          for (;;) {
            at = (go > 0) ? at + 1 : at - 1;
            const int mine_at = (go > 0) ? at + lane : at - lane;
            const unsigned some = __ballot_sync(kFull, mine_at >= 0 && mine_at < kStreamBins &&
                                                           (row_word(mine_at & (kStreamBins - 1)) != 0ull || (mine_at == 0 && some_tiny)));
            if (some != 0u) {
              bin = (go > 0) ? at + __ffs(some) - 1 : at - (__ffs(some) - 1);
              break;
            }
            at = (go > 0) ? at + 31 : at - 31;
            if (at < 0 || at >= kStreamBins) break;
          }
          // (the octave of an exact search is the right one: no bin of it reaches the target only through rounding
          // between two summation orders, and the last one tried, the lowest, is kept whole)
          last_resort = exact && (bin < 0 || (bin >> 5) != oct);
          if (last_resort) bin = sh.fd.bin;
          if (bin >= 0) {
            if (!exact) {  // its mass above, octave by octave from the top
              carry = 0.0;
              for (int e = top; e > (bin >> 5); --e) carry += static_cast<double>(mass(e)) * pow2_double(max(e, 1) - 150);
            }
            ab = suffix_sum<5>((lane > (bin & 31)) ? bin_mass9(bin >> 5) : 0.0);
            ab = __shfl_sync(kFull, ab, 0);
          }
        }
      }
      const unsigned long long word = (bin >= 0) ? row_word(bin) : 0ull;
      if (lane == 0) {
        sh.row_max = top;
        sh.fd.total = t + row_rest;
        sh.fd.key = last_resort ? 1u : 0u;
        sh.fd.bin = bin;
        if (bin >= 0) {
          sh.fd.carry = exact ? carry : 0.0;
          sh.fd.above = exact ? ab : carry + ab;
          // the bin's smallest term bounds the number of its keys
          const unsigned int least = (static_cast<unsigned int>(bin & 31) << 9) | ((bin >= 32) ? 0x4000u : 0u);
          sh.fd.count = (least == 0u) ? 0x7fffffffu : static_cast<unsigned int>(word / least);  // (at most 2^32 / 2^9 a CTA)
        }
      }
    }
    __syncthreads();
    invalid = sh.row_max == kOctaves - 1;
    total = sh.fd.total;
    if (!invalid && !exact && (!(total >= 0x1p-40) || (go != 0 && sh.fd.bin < 0))) {
      // (the histogram takes a denormal for a number of at least 2^-126, which only counts in a total as small
      // as this; or there is no neighbour where the masses asked for one)
      exact = true;
      go = 0;
      csync();
      clear();
      continue;
    }
    if (invalid) total = 0.0;
    target = static_cast<double>(P.p) * total;
    m_gt = 0.0;
    m_ge = total;
    searching = !invalid && target > 0.0 && !P.keep_all;  // else p >= 1 or an all-zero row: keep all
    if (!searching) break;
    last_resort = sh.fd.key != 0u;
    unsigned int prefix = static_cast<unsigned int>(sh.fd.bin);
    const double scale = pow2_double(max(sh.fd.bin >> 5, 1) - 150);
    unsigned int M = sh.fd.count;
    int shift = kStreamShift;
    // An exact search has the mass of the octaves above apart (`carry`) and exact integer masses inside its octave.
    const double carry = sh.fd.carry, above_hist = sh.fd.above;
    const int hi_key = exact ? static_cast<int>((prefix >> 5 << 23) | 0x7fffffu) : INT_MAX;
    int want = 0;
    csync();  // the histograms and octaves have been read: the store and the ring are free
    // ---- a well filled bin: 10 (then the last 8) more bits, one pass over the row each -----------------------
    while (M > static_cast<unsigned int>(kStreamCand) && shift > 0) {
      // (the pass uses the ring, so the level histogram takes the store)
      LevelHist& lv = *reinterpret_cast<LevelHist*>(sh.store);
      const int bits = min(shift, 10), sl = shift - bits;
      const int top = static_cast<int>((prefix << shift) + ((1u << shift) - 1u));
      level_clear<kStreamThreads>(lv);
      __syncthreads();
      double s = 0.0;
      stream_pass(sh, A, L, [&](int, unsigned int (&k)[N]) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
          level_add(lv, (k[j] >> shift) == prefix && k[j] != 0u, k[j], sl, bits);
          if (static_cast<int>(k[j]) > top && static_cast<int>(k[j]) <= hi_key) s += static_cast<double>(__uint_as_float(k[j]));
        }
      });
      level_groups<kStreamThreads>(lv, prefix, sl, bits);
      s = stream_sum(sh, s);
      if (kShared && tid == 0) sh.part = s;
      csync();
      if (warp == 0) {
        double above, upto, above1, upto1;
        if (kShared) s = row_sum(&sh.part);
        unsigned long long m = lv.grp[lane];
        for (int r = 1; r < cs; ++r) m += *cluster.map_shared_rank(&lv.grp[lane], (rank + r) % cs);
        const double all = static_cast<double>(m) * scale;
        const int gi = find_from_top<5>(all, s, carry, target, above, upto);
        const int bin = gi * 32 + lane;
        unsigned int c = lv.cnt[bin];
        m = level_mass(prefix, bin, sl, c, lv.sum[bin], bits);
        for (int r = 1; r < cs; ++r) {
          const LevelHist* const peer = cluster.map_shared_rank(&lv, (rank + r) % cs);
          const unsigned int c_r = peer->cnt[bin];
          m += level_mass(prefix, bin, sl, c_r, peer->sum[bin], bits);
          c += c_r;
        }
        const int b1 = find_from_top<5>(static_cast<double>(m) * scale, above, carry, target, above1, upto1);
        const unsigned int cb = __shfl_sync(kFull, c, b1);
        if (lane == 0) {
          sh.fd.oct = gi * 32 + b1;
          sh.fd.count = cb;
          sh.fd.upto = upto1;
          sh.row_part = s;
        }
      }
      __syncthreads();
      // (only the first level can show that the bin was the wrong one)
      if (shift == kStreamShift && !last_resort) want = (carry + sh.row_part >= target) ? 1 : (carry + sh.fd.upto < target) ? -1 : 0;
      prefix = (prefix << bits) | static_cast<unsigned int>(sh.fd.oct);
      M = sh.fd.count;
      shift = sl;
      csync();
      if (exact && want == -go) want = 0;  // (never: in whole numbers the bins agree with one another)
      if (want != 0) break;
    }
    if (want != 0) {
      turn(want);
      continue;
    }
    // ---- pass 2: what lies above the bin, and in it ---------------------------------------------------
    // (a prefix of all bits is one value: it is the threshold, and counts as the bin)
    const unsigned int lo_key = (prefix != 0u) ? prefix << shift : 1u;
    const unsigned int top_key = (prefix << shift) + ((1u << shift) - 1u), span = top_key - lo_key;
    // above a whole bin the histogram has the upper part of the sum; above a part of one every value is added up
    const bool by_hist = shift == kStreamShift;
    // (masses) The low parts of a batch are added up in binary32, which is exact while their octaves lie within 2^11
    // (16 x 2^9 x 2^11 units are 2^24); batches with a key further above the bin, few of them, go the long way.
    const int far_key = exact || ((sh.fd.bin >> 5) + 12) >= kOctaves ? INT_MAX : (((sh.fd.bin >> 5) + 12) << 23) - 1;
    double inner = 0.0;
    auto pass2 = [&](auto whole) {
      double s = 0.0;
      unsigned int ab = 0u, in = 0u;
      const int last = ((L + kStreamRound - 1) / kStreamRound + kStreamBatch - 1) / kStreamBatch * kStreamBatch - kStreamBatch;
      stream_pass(sh, A, L, [&](int round, unsigned int (&k)[N]) {
        unsigned int a8 = 0u, i8 = 0u;
        float part = 0.f;
        bool apart = decltype(whole)::value;
        if (kMasses && !apart) {
          int most = 0;
#pragma unroll
          for (int j = 0; j < N; ++j) most = max(most, static_cast<int>(k[j]));
          apart = __any_sync(kFull, most > far_key);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
          const float r = stream_rest(k[j]);
          if (static_cast<int>(k[j]) > static_cast<int>(top_key)) {
            a8 |= 1u << j;
            if (static_cast<int>(k[j]) <= hi_key) part += r;
          }
          if (k[j] - lo_key <= span) i8 |= 1u << j;
        }
        if (!apart) {
          s += static_cast<double>(part);
        } else {
#pragma unroll
          for (int j = 0; j < N; ++j)
            if (static_cast<int>(k[j]) > static_cast<int>(top_key) && static_cast<int>(k[j]) <= hi_key)
              s += static_cast<double>(decltype(whole)::value ? __uint_as_float(k[j]) : stream_rest(k[j]));
        }
        const int at = 4 * (round & 7);
        ab |= a8 << at;
        in |= i8 << at;
        if ((round & 7) == 8 - kStreamBatch || round == last) {
          above_bits[(round >> 3) * kStreamThreads + tid] = ab;
          in_bits[(round >> 3) * kStreamThreads + tid] = in;
          ab = in = 0u;
        }
      });
      inner = s;
    };
    if (by_hist) pass2(std::false_type()); else pass2(std::true_type());
    if (tid == 0) sh.n_cand = 0;
    inner = stream_sum(sh, inner);
    if (kShared && tid == 0) sh.part = inner;
    if (shift > 0) level_clear<kStreamThreads>(sc.lv);
    // fetch the keys of the bin by their bits
    const int word_rows = (L + 8 * kStreamRound - 1) / (8 * kStreamRound);
    for (int r8 = 0; r8 < word_rows; ++r8) {
      unsigned int w = in_bits[r8 * kStreamThreads + tid];
      if (!__any_sync(kFull, w != 0u)) continue;
      int n = __popc(w), end = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(kFull, end, d);
        if (lane >= d) end += v;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&sh.n_cand, end);
      at = __shfl_sync(kFull, at, 31) + end - n;
      for (; w != 0u; w &= w - 1u, ++at) {
        const int bit = __ffs(w) - 1;
        const unsigned int entry = static_cast<unsigned int>((r8 * 8 + (bit >> 2)) * kStreamRound + 4 * tid + (bit & 3));
        if (at < kStreamCand) sc.place[at] = entry;
      }
    }
    __syncthreads();
    const int own = min(sh.n_cand, kStreamCand);  // (one value's entries may be more: their bits are all kept)
    if (shift > 0) {  // (all loads of a thread in flight at once: one by one, as the places are found, took 7 us)
      unsigned int key[kStreamCand / kStreamThreads];
#pragma unroll
      for (int j = 0; j < kStreamCand / kStreamThreads; ++j) {
        const int i = tid + j * kStreamThreads;
        if (i < own) key[j] = __float_as_uint(__ldg(A + sc.place[i]));
      }
#pragma unroll
      for (int j = 0; j < kStreamCand / kStreamThreads; ++j) {
        const int i = tid + j * kStreamThreads;
        if (i < own) sc.keys[i] = key[j];
      }
    }
    csync();
    if (kShared) inner = row_sum(&sh.part);
    inner += by_hist ? above_hist : 0.0;
    int n = own, n_in = sh.n_cand;  // keys of the row's bin, and its entries
    const unsigned int* keys = sc.keys;
    if (kShared) {
      const int c_r = (lane < cs) ? *cluster.map_shared_rank(&sh.n_cand, lane < cs ? lane : 0) : 0;
      n_in = __reduce_add_sync(kFull, c_r);
      n = min(n_in, kStreamCand);
      keys = sc.all_keys;
      if (shift > 0) {
        int off = 0;
        for (int r = 0; r < cs; ++r) {
          const int c = min(__shfl_sync(kFull, c_r, r), kStreamCand - off);
          const unsigned int* const src = cluster.map_shared_rank(sc.keys, r);
          for (int i = tid; i < c; i += kStreamThreads) sc.all_keys[off + i] = src[i];
          off += c;
        }
        __syncthreads();
      }
    }
    if (shift > 0 && n == 0) {
      theta = top_key + 1u;
      m_gt = m_ge = carry + inner;
    } else if (shift > 0) {
      double above, upto;
      theta = threshold_among<kStreamThreads>(keys, n, prefix, shift, inner, carry, target, scale, sc.lv, sh.fd, sc.pk, above, upto);
      m_gt = carry + above;
      m_ge = carry + upto;
    } else {
      theta = prefix;
      m_gt = carry + inner;
      m_ge = carry + (inner + static_cast<double>(n_in) * static_cast<double>(__uint_as_float(prefix)));
    }
    // the right bin?
    if (shift == kStreamShift && !last_resort) {
      want = (carry + inner >= target) ? 1 : (m_ge < target) ? -1 : 0;
      if (want != 0 && !(exact && want == -go)) {
        __syncthreads();
        if (tid == 0) sh.fd.bin = static_cast<int>(prefix);  // (threshold_among used the field)
        turn(want);
        continue;
      }
    }
    const double doubt = (kMasses ? kStreamDoubt : kStreamDoubt32) * total;
    if (!exact && !(m_gt < target - doubt && m_ge > target + doubt)) {
      exact = true;
      go = 0;
      csync();
      clear();
      continue;
    }
    // the bin's entries that make it join the bits
    if (shift > 0) {
      for (int i = tid; i < own; i += kStreamThreads) {
        if (sc.keys[i] >= theta) {
          const unsigned int e = sc.place[i];
          const unsigned int round = e / kStreamRound, t = (e % kStreamRound) >> 2;
          atomicOr(&above_bits[(round >> 3) * kStreamThreads + t], 1u << (4 * (round & 7) + (e & 3)));
        }
      }
    } else {
      for (int r8 = 0; r8 < word_rows; ++r8) above_bits[r8 * kStreamThreads + tid] |= in_bits[r8 * kStreamThreads + tid];
    }
    break;
  }
  __syncthreads();

  // ---- ordered emission ---------------------------------------------------------------------------------
  int* const out = P.idx + out_list * P.idx_stride;
  const int stride = static_cast<int>(min(P.idx_stride, static_cast<long long>(INT_MAX)));
  int count = 0;
  if (searching) {
    // A warp takes a power of two of consecutive rounds, so that they lie in one row of words.
    const int rounds = (L + kStreamRound - 1) / kStreamRound;
    const int per = (rounds <= kStreamWarps) ? 1 : (rounds <= 2 * kStreamWarps) ? 2 : 4;
    static_assert(kStreamMax / kStreamRound <= 4 * kStreamWarps, "four rounds per warp cover a row");
    const int r_lo = warp * per, r_hi = min(rounds, r_lo + per);
    const unsigned int* const words = above_bits + (r_lo >> 3) * kStreamThreads;
    int wc = 0;
    if (r_lo < r_hi) {
      const unsigned int mine = ((per == 4) ? 0xffffu : (per == 2) ? 0xffu : 0xfu) << (4 * (r_lo & 7));
#pragma unroll
      for (int c = 0; c < kStreamThreads / 32; ++c) wc += __popc(words[32 * c + lane] & mine);
    }
    wc = __reduce_add_sync(kFull, wc);
    if (lane == 0) sh.warp_cnt[warp] = wc;
    __syncthreads();
    const int v = (lane < kStreamWarps) ? sh.warp_cnt[lane] : 0;
    count = __reduce_add_sync(kFull, v);
    int pos = __reduce_add_sync(kFull, lane < warp ? v : 0);
    if (kShared) {
      if (tid == 0) sh.kept = count;
      csync();  // (every CTA is also done with its peers' keys: the ring may be written)
      const int c_r = (lane < cs) ? *cluster.map_shared_rank(&sh.kept, lane < cs ? lane : 0) : 0;
      count = __reduce_add_sync(kFull, c_r);
      pos += __reduce_add_sync(kFull, lane < rank ? c_r : 0);
      __syncwarp();
      cluster_arrive_release();  // this CTA reads no peer's shared memory from here on
    }
    // 512 entries at a time: the lanes' counts of four 128-entry chunks are scanned as four bytes of one word, the
    // kept positions go through a per-warp staging line that lies like the output modulo 16 bytes, and leave
    // in 16-byte stores.
    int* const stage = reinterpret_cast<int*>(sh.ring) + warp * kStreamStage;
    const bool wide = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    for (int r = r_lo; r < r_hi; ++r) {
      const int nib_at = 4 * (r & 7);
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        unsigned int x = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) x |= ((words[32 * (4 * q + i) + lane] >> nib_at) & 15u) << (8 * i);
        if (!__any_sync(kFull, x != 0u)) continue;
        unsigned int c = x - ((x >> 1) & 0x05050505u);
        c = (c & 0x03030303u) + ((c >> 2) & 0x03030303u);
        unsigned int incl = c;  // (at most 128 per byte)
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const unsigned int u = __shfl_up_sync(kFull, incl, d);
          if (lane >= d) incl += u;
        }
        const unsigned int t4 = __shfl_sync(kFull, incl, 31);
        incl -= c;
        const int off = pos & 3;
        int base = off;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          int at = base + static_cast<int>((incl >> (8 * i)) & 255u);
          const int first = lo + r * kStreamRound + (4 * q + i) * 128 + 4 * lane;
          const unsigned int nib = x >> (8 * i);
          if (nib & 1u) stage[at++] = first;
          if (nib & 2u) stage[at++] = first + 1;
          if (nib & 4u) stage[at++] = first + 2;
          if (nib & 8u) stage[at++] = first + 3;
          base += static_cast<int>((t4 >> (8 * i)) & 255u);
        }
        __syncwarp();
        const int from = pos - off;  // output position of stage[0]
        for (int j = 4 * lane; j < base; j += 128) {
          if (wide && j >= off && j + 4 <= base && from + j + 4 <= stride) {
            *reinterpret_cast<int4*>(out + from + j) = *reinterpret_cast<const int4*>(stage + j);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (j + e >= off && j + e < base && from + j + e < stride) out[from + j + e] = stage[j + e];
          }
        }
        __syncwarp();
        pos += base - off;
      }
    }
  } else {
    if (kShared) cluster_arrive_release();
    if (!invalid) {
      count = L_row;
      for (int i = lo + tid; i < min(lo + L, stride); i += kStreamThreads) out[i] = i;
    }
  }
  if (tid == 0 && rank == 0) {
    P.counts[out_list] = count;
    P.status[out_list] = invalid ? SPECATTN_ROW_INVALID_PROB : (count > P.idx_stride ? SPECATTN_ROW_OVERFLOW : SPECATTN_ROW_OK);
    if (P.diag != nullptr) {
      double* d = P.diag + out_list * 4;
      d[0] = total;
      d[1] = target;
      d[2] = m_gt;
      d[3] = m_ge;
    }
  }
  __syncwarp();
  if (kShared) cluster_wait();  // nobody leaves while its shared memory may still be read remotely
}
