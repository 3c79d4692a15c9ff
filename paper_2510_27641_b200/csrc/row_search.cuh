// The threshold search over one row of binary32 values: exact top-p threshold, kept counts of every
// CTA, ordered emission.  Included by select_topp.cu.
//
// A level-1 histogram of the row (exponent and a few mantissa bits) is followed by a search inside
// one of its bins.  What bounds the search is latency -- barriers, round trips to the peers' shared
// memory, chains of shuffles -- so it exchanges as little as it can:
//   1. one exact integer mass per octave (the bins of an octave share an exponent), then the bins of
//      the octave that holds the threshold; warp 0 scans both (all warps scanning the same data
//      was slower: the shuffles of 16 warps share one pipe, 1.8 us against 0.6 us);
//   2. the keys of the threshold bin, up to kCandCap of them, among which the threshold is found.
// Only a bin with more keys (heavy ties, flat rows of a narrow range) takes further histograms of
// 10 bits over the row.
//
// Exactness.  All values of an octave share one exponent, so sums of their mantissas are integers: they are
// kept as such per bin, and inside the threshold's octave every sum is an integer (below 2^53, times
// the octave's scale) held in a binary64.  The result therefore does not depend on how the row was
// dealt to CTAs, on the path that found it or on the order of any update.
#pragma once

constexpr int kSliceMax = 16384;         // entries per CTA of a cluster
constexpr int kCandCap = 4096;           // keys of the threshold bin that a cluster gathers
constexpr int kDirectMax = 128;          // up to this many gathered keys the threshold is found by comparing all pairs
constexpr int kL1Bins = 2048;            // sign(0) + 8 exponent bits + 3 mantissa bits
constexpr int kLevelBins = 1024;         // 10 mantissa bits per further level
constexpr int kOctaves = 256;
constexpr int kMaxCluster = 16;
constexpr int kMaxApart = 64;            // speculated queries of searches apart

struct SearchResult {
  unsigned int theta;   // keep every entry whose key is >= theta
  bool invalid;
  bool counted;         // the kept entries of every CTA of the cluster and of every warp of this one are
                        // known after a CTA barrier (otherwise the caller counts)
  double total, target, m_gt, m_ge;
};

__device__ __forceinline__ double pow2_double(int k) {  // 2^k, k in the normal range
  return __longlong_as_double(static_cast<long long>(k + 1023) << 52);
}

// Mantissa (hidden bit included) of a non-negative key.
__device__ __forceinline__ unsigned int mantissa_of(unsigned int key) {
  return (key & 0x7fffffu) | ((key >> 23) ? 0x800000u : 0u);
}

// Suffix sums over the first 2^STEPS lanes (zero above).
template <int STEPS>
__device__ __forceinline__ double suffix_sum(double s) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < (1 << STEPS); d <<= 1) {
    const double v = __shfl_down_sync(kFull, s, d);
    if (lane + d < (1 << STEPS)) s += v;
  }
  return s;
}

// One warp: highest lane with a mass at which the mass accumulated from the top lane down -- on top of
// `inner` and `carry` -- reaches the target; the lowest lane with a mass if none does (only reachable
// through rounding between two summation orders).  Masses of one octave and `inner` add up exactly.
// All lanes get the lane, the sum strictly above it and the sum down to it (both with `inner`).
template <int STEPS>
__device__ __forceinline__ int find_from_top(double m, double inner, double carry, double target, double& above,
                                             double& upto) {
  const double incl = inner + suffix_sum<STEPS>(m);
  const unsigned hit = __ballot_sync(kFull, m != 0.0 && carry + incl >= target);
  const unsigned some = __ballot_sync(kFull, m != 0.0);
  const int at = (hit != 0u) ? 31 - __clz(hit) : ((some != 0u) ? __ffs(some) - 1 : 0);
  upto = __shfl_sync(kFull, incl, at);
  const double next = __shfl_sync(kFull, incl, (at + 1) & 31);
  above = (at == (1 << STEPS) - 1) ? inner : next;
  return at;
}

// One warp: total mass, target and the octave that holds the threshold, from octave `top` (the
// largest key's) down, 32 octaves at a time.  mass(e): exact mass of octave e of the whole row.  Everything
// below the first window is less than 2^-30 of the largest value per entry, so its totals are
// almost always all that is needed of it.
template <class Mass>
__device__ __forceinline__ int find_octave(int top, int bottom, float p, Mass mass, double& total, double& target,
                                           double& above) {
  const int lane = threadIdx.x & 31;
  double incl0 = 0.0, m0 = 0.0;
  total = 0.0;
  for (int t = top; t >= bottom; t -= 32) {
    const int e = t - 31 + lane;
    const double m = (e >= bottom) ? static_cast<double>(mass(e)) * pow2_double(max(e, 1) - 150) : 0.0;
    const double incl = suffix_sum<5>(m);
    if (t == top) {
      incl0 = incl;
      m0 = m;
    }
    total += __shfl_sync(kFull, incl, 0);
  }
  target = static_cast<double>(p) * total;
  double carry = 0.0;
  int lowest = bottom;
  for (int t = top; t >= bottom; t -= 32) {
    const int e = t - 31 + lane;
    double m = m0, incl = incl0;
    if (t != top) {
      m = (e >= bottom) ? static_cast<double>(mass(e)) * pow2_double(max(e, 1) - 150) : 0.0;
      incl = suffix_sum<5>(m);
    }
    const unsigned hit = __ballot_sync(kFull, m != 0.0 && carry + incl >= target);
    const unsigned some = __ballot_sync(kFull, m != 0.0);
    const double next = __shfl_down_sync(kFull, incl, 1);
    const double ab = carry + ((lane == 31) ? 0.0 : next);
    if (hit != 0u) {
      const int at = 31 - __clz(hit);
      above = __shfl_sync(kFull, ab, at);
      return t - 31 + at;
    }
    if (some != 0u) {  // (kept for the case that no octave reaches the target through rounding)
      const int at = __ffs(some) - 1;
      above = __shfl_sync(kFull, ab, at);
      lowest = t - 31 + at;
    }
    carry += __shfl_sync(kFull, incl, 0);
  }
  return lowest;
}

// Histogram of 10 bits over keys that share the bits above them: number of keys and sum of the bits
// below the level per bin, then masses of 32 bins each.
struct LevelHist {
  unsigned int cnt[kLevelBins];
  unsigned int sum[kLevelBins];
  unsigned long long grp[32];
};

// Adds a key by the `bits` bits above `sh`.  All 32 lanes call this together.  When every taking lane hits one bin (ties) the warp reduces first.
__device__ __forceinline__ void level_add(LevelHist& lv, bool take, unsigned int key, int sh, int bits = 10) {
  const unsigned takers = __ballot_sync(kFull, take);
  if (takers == 0u) return;
  const unsigned int bin = (key >> sh) & ((1u << bits) - 1u), low = key & ((1u << sh) - 1u);
  const unsigned int bin0 = __shfl_sync(kFull, bin, __ffs(takers) - 1);
  if (__all_sync(kFull, !take || bin == bin0)) {
    const unsigned int s = __reduce_add_sync(kFull, take ? low : 0u);
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&lv.cnt[bin0], static_cast<unsigned int>(__popc(takers)));
      atomicAdd(&lv.sum[bin0], s);
    }
  } else if (take) {
    atomicAdd(&lv.cnt[bin], 1u);
    atomicAdd(&lv.sum[bin], low);
  }
}

// Exact mass of a level bin with c keys, s the sum of their low bits.
__device__ __forceinline__ unsigned long long level_mass(unsigned int prefix, int bin, int sh, unsigned int c, unsigned int s,
                                                        int bits = 10) {
  return static_cast<unsigned long long>(c) * mantissa_of(((prefix << bits) | static_cast<unsigned int>(bin)) << sh) + s;
}

// CTA of NT threads, between barriers: the masses of the 32 groups of bins.
template <int NT>
__device__ __forceinline__ void level_groups(LevelHist& lv, unsigned int prefix, int sh, int bits = 10) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int gi = warp; gi < 32; gi += NT / 32) {
    const int bin = gi * 32 + lane;
    unsigned long long s = level_mass(prefix, bin, sh, lv.cnt[bin], lv.sum[bin], bits);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFull, s, d);
    if (lane == 0) lv.grp[gi] = s;
  }
}

template <int NT>
__device__ __forceinline__ void level_clear(LevelHist& lv) {
  for (int i = threadIdx.x; i < kLevelBins / 4; i += NT) {
    reinterpret_cast<uint4*>(lv.cnt)[i] = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4*>(lv.sum)[i] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Results that warp 0 leaves for the CTA.
struct Found {
  int bin;
  unsigned int count, key;
  double carry;         // mass above the threshold's octave
  double above, upto;   // exact masses inside the octave: above the bin (or key), down to it
  double total, target;
  int oct;
};

struct Picks {          // the threshold among up to kDirectMax keys
  unsigned int n_few;
  unsigned int few[32];
  unsigned int key[16];
  double ge[16], gt[16];
};

// The threshold among n keys in shared memory that share the bits above `shift` (= prefix) -- by
// comparing all pairs, up to kDirectMax keys, or with one level histogram (zero on entry) and, for what is
// left in one of its bins, pairs or a second level.  inner: exact mass above those keys inside the
// octave.  Called by all threads after a barrier; all get the key and the exact masses.
template <int NT>
__device__ __forceinline__ unsigned int threshold_among(const unsigned int* keys, int n, unsigned int prefix, int shift,
                                                        double inner, double carry, double target, double scale,
                                                        LevelHist& lv, Found& fd, Picks& pk, double& above, double& upto) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  {  // One value (ties, as in a quantised row): it is the threshold.  (256 rows of 8191 such: 14.5 -> 12.0 us; a row
     // without ties leaves after one look at its few keys.)
    const unsigned int k0 = keys[0];
    bool same = true;
    for (int i = tid; i < n; i += NT) same &= keys[i] == k0;
    if (__syncthreads_and(same)) {
      above = inner;
      upto = inner + static_cast<double>(static_cast<unsigned long long>(n) * mantissa_of(k0)) * scale;
      return k0;
    }
  }
  while (n > kDirectMax && shift > 0) {
    const int bits = min(shift, 10), sh = shift - bits;
    for (int i = tid; i < ((n + 31) & ~31); i += NT) {
      const unsigned int k = (i < n) ? keys[i] : 0u;
      level_add(lv, i < n && (k >> shift) == prefix, k, sh, bits);
    }
    if (tid == 0) pk.n_few = 0u;
    __syncthreads();
    level_groups<NT>(lv, prefix, sh, bits);
    __syncthreads();
    if (warp == 0) {
      double ab, up;
      const int gi = find_from_top<5>(static_cast<double>(lv.grp[lane]) * scale, inner, carry, target, ab, up);
      const int bin = gi * 32 + lane;
      const unsigned int c = lv.cnt[bin];
      double ab1, up1;
      const int b = find_from_top<5>(static_cast<double>(level_mass(prefix, bin, sh, c, lv.sum[bin], bits)) * scale, ab,
                                     carry, target, ab1, up1);
      const unsigned int cb = __shfl_sync(kFull, c, b);
      if (lane == 0) {
        fd.bin = gi * 32 + b;
        fd.count = cb;
        fd.above = ab1;
        fd.upto = up1;
      }
    }
    __syncthreads();
    prefix = (prefix << bits) | static_cast<unsigned int>(fd.bin);
    inner = fd.above;
    shift = sh;
    if (shift == 0) {
      above = inner;
      upto = fd.upto;
      return prefix;
    }
    if (fd.count <= 32u) {  // the usual end: a handful of keys left
      for (int i = tid; i < n; i += NT) {
        const unsigned int k = keys[i];
        if ((k >> shift) == prefix) pk.few[atomicAdd(&pk.n_few, 1u)] = k;
      }
      __syncthreads();
      keys = pk.few;
      n = static_cast<int>(pk.n_few);
    } else {
      level_clear<NT>(lv);
      __syncthreads();
    }
  }
  // all pairs: for each key the exact mass of the keys >= it; the highest key that reaches the target
  if (warp * 32 < n) {
    const unsigned int ki = (tid < n) ? keys[tid] : 0xffffffffu;
    unsigned int c_ge = 0u, c_eq = 0u, s_ge = 0u;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const unsigned int kj = keys[j];
      if (kj >= ki) {
        ++c_ge;
        s_ge += kj & 0xfffffu;
      }
      c_eq += (kj == ki) ? 1u : 0u;
    }
    double ge = 0.0, gt = 0.0;
    unsigned int best = 0u, lowest = 0xffffffffu;
    if (tid < n) {
      const unsigned int base = mantissa_of(ki & 0xfff00000u);
      const unsigned long long m_ge = static_cast<unsigned long long>(c_ge) * base + s_ge;
      const unsigned long long m_gt = m_ge - static_cast<unsigned long long>(c_eq) * mantissa_of(ki);
      ge = inner + static_cast<double>(m_ge) * scale;
      gt = inner + static_cast<double>(m_gt) * scale;
      if (carry + ge >= target) best = ki;
      lowest = ki;
    }
    const unsigned int wb = __reduce_max_sync(kFull, best), wl = __reduce_min_sync(kFull, lowest);
    const unsigned int pick = (wb != 0u) ? wb : wl;
    const int src = __ffs(__ballot_sync(kFull, tid < n && ki == pick)) - 1;
    ge = __shfl_sync(kFull, ge, src);
    gt = __shfl_sync(kFull, gt, src);
    if (lane == 0) {
      pk.key[warp] = (wb != 0u) ? wb : (wl | 0x80000000u);  // (sign set: nothing reached the target)
      pk.ge[warp] = ge;
      pk.gt[warp] = gt;
    }
  }
  __syncthreads();
  // no key reaches the target only through rounding between two summation orders: keep them all
  unsigned int key = pk.key[0];
  int at = 0;
  for (int w = 1; w * 32 < n; ++w) {
    const unsigned int k = pk.key[w];
    const bool none = (key >> 31) != 0u, knone = (k >> 31) != 0u;
    if (none ? (!knone || k < key) : (!knone && k > key)) {
      key = k;
      at = w;
    }
  }
  upto = pk.ge[at];
  above = pk.gt[at];
  return key & 0x7fffffffu;
}

// ---- the row lies in the shared memory of a cluster -----------------------------------------------------
// The level-1 histogram keeps, per bin (11 bits), the sum of the low 17 mantissa bits in one word and,
// in another, the sum of the next three bits (17 bits) and the number of values (15 bits); the top three
// mantissa bits are the bin's own.  A slice of up to kSliceMax entries overflows neither.

// Shared memory of the search: the part that lives as long as the kernel ...
struct SearchFixed {
  unsigned int hist[2 * kL1Bins];  // low words, then high words; the gathered keys of the cluster later on
  unsigned int kmax;               // largest key of this CTA (above 0x7f7fffff: an invalid input); read by peers
  int oct_min;                     // lowest octave with a mass (read by peers)
  int n_cand;                      // keys of this CTA in the threshold bin (read by peers)
  int n_above;                     // keys of this CTA above it (read by peers)
  int local_kept;                  // read by peers
  unsigned int cl_kmax;            // kmax over the cluster
  Found fd;
  int warp_cnt[16];                // kept entries per warp
  int kept[kMaxCluster];           // kept entries of every CTA of the cluster
  // searches apart (one CTA per query, see select_topp_kernel); read by peers
  int bad;                         // an invalid input was met
  unsigned int theta[kMaxApart];   // thresholds of the queries this CTA searched (0xffffffff: invalid)
  double masses[4];                // of the last query
};
// ... and the part that may share its bytes with the staging ring of the aggregation.
struct SearchScratch {
  unsigned int cand[kCandCap];       // keys of this CTA in the threshold bin (read by peers)
  unsigned long long oct[kOctaves];  // exact masses of this CTA's octaves (read by peers)
  LevelHist lv;                      // (read by peers)
  Picks pk;
};

// Adds one key (not zero, sign clear) to the level-1 histogram.
__device__ __forceinline__ void hist_bump(unsigned int* hist, unsigned int key) {
  unsigned int* const p = reinterpret_cast<unsigned int*>(reinterpret_cast<char*>(hist) + ((key >> 18) & 0x1ffcu));
  atomicAdd(p, key & 0x1ffffu);
  atomicAdd(p + kL1Bins, ((key >> 17) & 7u) | 0x20000u);
}

// Adds N keys per lane (all 32 lanes call this together), except those of bin 0: zeros carry no mass, and the
// denormals below 2^-129 -- twenty octaves in one bin, on attention rows thousands of neighbours -- would serialise
// the updates of one address (a slice of them took 17 us instead of 3); hist_add_tiny enters them where
// they can matter.  When every key of the warp falls into one bin (ties, constant rows) the warp reduces first.
constexpr unsigned int kTinyKeys = 0x100000u;
template <int N>
__device__ __forceinline__ void hist_add(unsigned int* hist, const unsigned int (&k)[N]) {
  const unsigned int bin0 = __shfl_sync(kFull, k[0] >> 20, 0);
  if (__all_sync(kFull, (k[0] >> 20) == bin0)) {
    unsigned int differ = 0u;
#pragma unroll
    for (int j = 1; j < N; ++j) differ |= k[j] ^ k[0];
    if (__all_sync(kFull, (differ >> 20) == 0u)) {
      if (bin0 == 0u) return;
      unsigned int lo = 0u, hi = 0u;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        lo += k[j] & 0x1ffffu;
        hi += ((k[j] >> 17) & 7u) | 0x20000u;
      }
      lo = __reduce_add_sync(kFull, lo);
      hi = __reduce_add_sync(kFull, hi);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&hist[bin0 & (kL1Bins - 1)], lo);
        atomicAdd(&hist[kL1Bins + (bin0 & (kL1Bins - 1))], hi);
      }
      return;
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (k[j] >= kTinyKeys) hist_bump(hist, k[j]);
}

// Enters the keys of bin 0 of a slice (n4_pad float4s), if its largest key is below 2^-50: beside a larger one
// their sum, at most 2^17 times 2^-129, is less than the last place of the total.  Called by all threads between
// barriers.
template <int NT>
__device__ __forceinline__ void hist_add_tiny(unsigned int* hist, unsigned int kmax, const float* a, int n4_pad) {
  if (kmax == 0u || kmax >= 0x26800000u) return;
  unsigned int lo = 0u, hi = 0u;
  for (int i4 = threadIdx.x; i4 < n4_pad; i4 += NT) {
    const uint4 v = *reinterpret_cast<const uint4*>(a + 4 * i4);
    const unsigned int k[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (k[e] != 0u && k[e] < kTinyKeys) {
        lo += k[e] & 0x1ffffu;
        hi += ((k[e] >> 17) & 7u) | 0x20000u;
      }
    }
  }
  lo = __reduce_add_sync(kFull, lo);
  hi = __reduce_add_sync(kFull, hi);
  if ((threadIdx.x & 31) == 0 && hi != 0u) {
    atomicAdd(&hist[0], lo);
    atomicAdd(&hist[kL1Bins], hi);
  }
  __syncthreads();
}

// Exact integer mass of a level-1 bin (units of its exponent's last place).
__device__ __forceinline__ unsigned long long bin_mass(int bin, unsigned int lo, unsigned int hi) {
  const unsigned int base = (static_cast<unsigned int>(bin & 7) << 20) + ((bin >= 8) ? 0x800000u : 0u);
  return static_cast<unsigned long long>(hi >> 17) * base + (static_cast<unsigned long long>(hi & 0x1ffffu) << 17) + lo;
}

// One bit per key that a lane meets in its warp's range of the slice.
template <bool kLong> struct HitWord { using type = unsigned int; };
template <> struct HitWord<true> { using type = unsigned long long; };

// The search.  `a`: this CTA's entries (n4_pad float4s: whole rounds of NT, zero beyond the
// slice), complete and histogrammed (fx.hist, fx.kmax; fx.oct_min = kOctaves), every thread past a barrier.
// bisect: number of halvings of the literal Alg. 2 loop, 0 = exact threshold.  The caller keeps the
// cluster together (a cluster barrier) before any of the shared memory is used again or a CTA leaves.
// The row lies in the CTAs of ranks r0 ... r0 + cs - 1 (cs = 1: this one's alone).
template <int NT>
__device__ __forceinline__ SearchResult search_slice(SearchFixed& fx, SearchScratch& sc, const float* a, int n4_pad,
                                                     float p, bool keep_all, int bisect, int cs, int r0 = 0) {
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kW = NT / 32;
  auto csync = [&]() {
    if (cs > 1) cluster.sync(); else __syncthreads();
  };
  SearchResult res;
  res.theta = 0u;
  res.counted = false;
  res.m_gt = 0.0;

  // ---- level 1: octave masses --------------------------------------------------------------------
  for (int e = tid; e < kOctaves; e += NT) {
    unsigned long long s = 0ull;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 lo = *reinterpret_cast<const uint4*>(&fx.hist[8 * e + 4 * h]);
      const uint4 hi = *reinterpret_cast<const uint4*>(&fx.hist[kL1Bins + 8 * e + 4 * h]);
      if ((hi.x | hi.y | hi.z | hi.w) != 0u)
        s += bin_mass(8 * e + 4 * h, lo.x, hi.x) + bin_mass(8 * e + 4 * h + 1, lo.y, hi.y) +
             bin_mass(8 * e + 4 * h + 2, lo.z, hi.z) + bin_mass(8 * e + 4 * h + 3, lo.w, hi.w);
    }
    sc.oct[e] = s;
    const int first = __reduce_min_sync(kFull, (s != 0ull) ? e : kOctaves);
    if (lane == 0 && first < kOctaves) atomicMin(&fx.oct_min, first);
  }
  level_clear<NT>(sc.lv);
  csync();
  if (warp == 0) {
    // largest key and lowest octave over the cluster, then the octave and its eight bins
    unsigned int km = (lane < cs) ? *cluster.map_shared_rank(&fx.kmax, r0 + lane) : 0u;
    int om = (lane < cs) ? *cluster.map_shared_rank(&fx.oct_min, r0 + lane) : kOctaves;
    km = __reduce_max_sync(kFull, km);
    om = __reduce_min_sync(kFull, om);
    Found fd;
    fd.total = fd.target = fd.carry = fd.above = fd.upto = 0.0;
    fd.bin = 0;
    fd.count = 0u;
    fd.oct = 0;
    if (km <= 0x7f7fffffu && om < kOctaves) {
      fd.oct = find_octave(
          static_cast<int>(km >> 23), om, p,
          [&](int e) -> unsigned long long {
            unsigned long long s = 0ull;
            if (cs == 1) return sc.oct[e];
            for (int r = 0; r < cs; ++r) s += *cluster.map_shared_rank(&sc.oct[e], r0 + r);
            return s;
          },
          fd.total, fd.target, fd.carry);
      unsigned long long s = 0ull;
      unsigned int c = 0u;
      fd.bin = 8 * fd.oct + (lane & 7);  // lane = (bin, rank mod 4)
      for (int r = lane >> 3; r < cs; r += 4) {
        const unsigned int* h = cluster.map_shared_rank(fx.hist, r0 + r);
        const unsigned int lo = h[fd.bin], hi = h[kL1Bins + fd.bin];
        s += bin_mass(fd.bin, lo, hi);
        c += hi >> 17;
      }
#pragma unroll
      for (int d = 8; d <= 16; d <<= 1) {
        s += __shfl_xor_sync(kFull, s, d);
        c += __shfl_xor_sync(kFull, c, d);
      }
      const double m = (lane < 8) ? static_cast<double>(s) * pow2_double(max(fd.oct, 1) - 150) : 0.0;
      const int b8 = find_from_top<3>(m, 0.0, fd.carry, fd.target, fd.above, fd.upto);
      fd.bin = 8 * fd.oct + b8;
      fd.count = __shfl_sync(kFull, c, b8);
    }
    if (lane == 0) {
      fx.fd = fd;
      fx.cl_kmax = km;
      fx.n_cand = 0;
      fx.n_above = 0;
    }
  }
  __syncthreads();
  const unsigned int kmax = fx.cl_kmax;
  res.invalid = kmax > 0x7f7fffffu;
  res.total = fx.fd.total;
  res.target = fx.fd.target;
  res.m_ge = res.total;
  // p >= 1 or an all-zero row: keep all
  if (res.invalid || !(res.target > 0.0) || keep_all) return res;
  const double scale = pow2_double(max(fx.fd.oct, 1) - 150);
  const double carry = fx.fd.carry;  // mass above the octave
  unsigned int prefix = static_cast<unsigned int>(fx.fd.bin);
  unsigned int M = fx.fd.count;      // keys of the bin over the cluster
  int shift = 20;                    // candidates: keys with key >> shift == prefix
  double inner = fx.fd.above;        // exact mass above the current prefix, inside the octave
  bool deep = false;                 // a level histogram was used (its words are not zero any more)

  // ---- a well filled bin: 10 more bits over the slices --------------------------------------------
  while (M > static_cast<unsigned int>(kCandCap) && shift > 0) {
    if (deep) {
      csync();  // every peer has read the previous level's words
      level_clear<NT>(sc.lv);
      __syncthreads();
    }
    deep = true;
    const int sh = shift - 10;
    // A warp whose keys of the bin are all one value (ties) adds them up by itself; the first lane that holds two
    // values sends it to the general way, which pays two atomics for every round of 32 keys.
    unsigned int first = 0xffffffffu, last = 0u, held = 0u;
    bool ties = true;
    for (int i4 = tid; ties && i4 < n4_pad; i4 += NT) {
      const uint4 k4 = *reinterpret_cast<const uint4*>(a + 4 * i4);
      const unsigned int k[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if ((k[e] >> shift) != prefix || k[e] == 0u) continue;
        first = min(first, k[e]);
        last = max(last, k[e]);
        ++held;
      }
      ties = __all_sync(kFull, held == 0u || first == last);
    }
    first = __reduce_min_sync(kFull, first);
    last = __reduce_max_sync(kFull, last);
    held = __reduce_add_sync(kFull, held);
    if (ties && (held == 0u || first == last)) {
      if (lane == 0 && held != 0u) {
        const unsigned int bin = (first >> sh) & 1023u;
        atomicAdd(&sc.lv.cnt[bin], held);
        atomicAdd(&sc.lv.sum[bin], held * (first & ((1u << sh) - 1u)));
      }
    } else {
      for (int i4 = tid; i4 < n4_pad; i4 += NT) {
        const uint4 k4 = *reinterpret_cast<const uint4*>(a + 4 * i4);
        const unsigned int k[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) level_add(sc.lv, (k[e] >> shift) == prefix && k[e] != 0u, k[e], sh);
      }
    }
    __syncthreads();
    level_groups<NT>(sc.lv, prefix, sh);
    csync();
    if (warp == 0) {
      unsigned long long s = 0ull;
      for (int r = 0; r < cs; ++r) s += *cluster.map_shared_rank(&sc.lv.grp[lane], r0 + r);
      double above, upto;
      const int gi = find_from_top<5>(static_cast<double>(s) * scale, inner, carry, res.target, above, upto);
      const int bin = gi * 32 + lane;
      unsigned int c = 0u;
      s = 0ull;
      for (int r = 0; r < cs; ++r) {
        const LevelHist* peer = cluster.map_shared_rank(&sc.lv, r0 + r);
        c += peer->cnt[bin];
        s += peer->sum[bin];
      }
      const unsigned long long m = static_cast<unsigned long long>(c) * mantissa_of(((prefix << 10) | static_cast<unsigned int>(bin)) << sh) + s;
      double above1, upto1;
      const int b = find_from_top<5>(static_cast<double>(m) * scale, above, carry, res.target, above1, upto1);
      c = __shfl_sync(kFull, c, b);
      if (lane == 0) {
        fx.fd.bin = gi * 32 + b;
        fx.fd.count = c;
        fx.fd.above = above1;
        fx.fd.upto = upto1;
      }
    }
    __syncthreads();
    prefix = (prefix << 10) | static_cast<unsigned int>(fx.fd.bin);
    M = fx.fd.count;
    inner = fx.fd.above;
    shift = sh;
    if (shift == 0) {  // one distinct key left: the threshold
      res.theta = prefix;
      res.m_gt = carry + inner;
      res.m_ge = carry + fx.fd.upto;
    }
  }

  // ---- gather the bin's keys, find the threshold among them ----------------------------------------
  if (shift > 0) {
    // a warp walks a contiguous range of the slice (the one whose positions it will write), notes
    // its keys of the bin in one word per lane, and takes room for all of them at once
    const int w4 = n4_pad / kW;  // float4s per warp
    const unsigned int lo_key = (prefix != 0u) ? prefix << shift : 1u;  // (zeros are in no bin)
    const unsigned int top_key = (prefix << shift) + ((1u << shift) - 1u), span = top_key - lo_key;
    // (four keys per round and lane: 256 threads may hold sixteen rounds, the others hold up to eight)
    using Hits = typename HitWord<NT == 256>::type;
    Hits hits = 0;
    int n_gt = 0;
    for (int j = 0; 32 * j < w4; ++j) {
      const uint4 k4 = *reinterpret_cast<const uint4*>(a + 4 * (warp * w4 + 32 * j + lane));
      unsigned int h = 0u;
      if (k4.x - lo_key <= span) h |= 1u;
      if (k4.y - lo_key <= span) h |= 2u;
      if (k4.z - lo_key <= span) h |= 4u;
      if (k4.w - lo_key <= span) h |= 8u;
      hits |= static_cast<Hits>(h) << (4 * j);
      n_gt += (k4.x > top_key) + (k4.y > top_key) + (k4.z > top_key) + (k4.w > top_key);
    }
    n_gt = __reduce_add_sync(kFull, n_gt);
    const int mine = (sizeof(Hits) == 8) ? __popcll(hits) : __popc(static_cast<unsigned int>(hits));
    int pre_c = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(kFull, pre_c, d);
      if (lane >= d) pre_c += v;
    }
    const int wcand = __shfl_sync(kFull, pre_c, 31);
    int wbase = 0;
    if (lane == 0) {
      if (wcand != 0) wbase = atomicAdd(&fx.n_cand, wcand);
      if (n_gt != 0) atomicAdd(&fx.n_above, n_gt);
    }
    wbase = __shfl_sync(kFull, wbase, 0);
    for (int at = wbase + pre_c - mine; hits != 0; ++at) {
      const int bit = ((sizeof(Hits) == 8) ? __ffsll(static_cast<long long>(hits)) : __ffs(static_cast<int>(hits))) - 1;
      hits &= hits - 1;
      const unsigned int key = __float_as_uint(a[4 * (warp * w4 + 32 * (bit >> 2) + lane) + (bit & 3)]);
      if (at < kCandCap) sc.cand[at] = key;  // (always: the bin holds at most kCandCap keys)
    }
    csync();
    // every warp: how many keys each CTA has in the bin and above it, and where its keys begin
    const int c_r = (lane < cs) ? min(*cluster.map_shared_rank(&fx.n_cand, r0 + lane), kCandCap) : 0;
    const int above_r = (lane < cs) ? *cluster.map_shared_rank(&fx.n_above, r0 + lane) : 0;
    int end_r = c_r;
#pragma unroll
    for (int d = 1; d < kMaxCluster; d <<= 1) {
      const int v = __shfl_up_sync(kFull, end_r, d);
      if (lane >= d) end_r += v;
    }
    const int n = min(__shfl_sync(kFull, end_r, kMaxCluster - 1), kCandCap);
    const unsigned int* keys = sc.cand;
    if (cs > 1) {
      unsigned int* const all_keys = fx.hist;
      const int share = max(kW / cs, 1);  // warps per rank
      for (int r = warp / share; r < cs; r += kW / share) {
        const int c = __shfl_sync(kFull, c_r, r), off = __shfl_sync(kFull, end_r, r) - c;
        const unsigned int* src = cluster.map_shared_rank(sc.cand, r0 + r);
        for (int i = (warp % share) * 32 + lane; i < c && off + i < kCandCap; i += share * 32) all_keys[off + i] = src[i];
      }
      keys = all_keys;
      if (deep) level_clear<NT>(sc.lv);
      __syncthreads();
    } else if (deep) {
      level_clear<NT>(sc.lv);
      __syncthreads();
    }
    double above, upto;
    res.theta = threshold_among<NT>(keys, n, prefix, shift, inner, carry, res.target, scale, sc.lv, fx.fd, sc.pk, above, upto);
    res.m_gt = carry + above;
    res.m_ge = carry + upto;
    if (bisect == 0) {
      // kept entries of every CTA (its keys above the bin, and its gathered keys that made it) and
      // of every warp of this CTA
      for (int r = warp; r < cs; r += kW) {
        const int c = __shfl_sync(kFull, c_r, r), off = __shfl_sync(kFull, end_r, r) - c;
        int k = 0;
        for (int i = lane; i < c && off + i < kCandCap; i += 32) k += (keys[off + i] >= res.theta) ? 1 : 0;
        k = __reduce_add_sync(kFull, k);
        const int ab = __shfl_sync(kFull, above_r, r);
        if (lane == 0) fx.kept[r] = k + ab;
      }
      int k = 0;
      for (int i = wbase + lane; i < min(wbase + wcand, kCandCap); i += 32) k += (sc.cand[i] >= res.theta) ? 1 : 0;
      k = __reduce_add_sync(kFull, k);
      if (lane == 0) fx.warp_cnt[warp] = n_gt + k;
      res.counted = true;
    }
  }
  if (bisect > 0) {
    // Alg. 2's loop, literally: theta_high = max, theta_low = 0, n midpoints in binary32.  The mass
    // of {a >= theta} does not grow with theta, so "mass(theta_mid) < target" holds exactly when
    // theta_mid lies above the exact threshold found above: the midpoints are those of the printed
    // loop without another pass over the row.
    float th_hi = __uint_as_float(kmax), th_lo = 0.f, th_mid = 0.f;
    for (int it = 0; it < bisect; ++it) {
      th_mid = __fmul_rn(__fadd_rn(th_hi, th_lo), 0.5f);
      if (__float_as_uint(th_mid) > res.theta) th_hi = th_mid; else th_lo = th_mid;
    }
    res.theta = __float_as_uint(th_mid);
  }
  return res;
}
