// One CTA per row, for calls with more rows than the GPU can keep on chip at once.  Included by
// select_topp.cu.
//
// What bounds this regime is bandwidth as long as enough rows are in flight: held in shared memory, 148
// SMs take some 37 rows of 131072 entries, and the latencies of a search (barriers, exchanges, scans) are
// paid once per wave of them (256 rows: 240 us).  Here every row has its own CTA, two per SM, nothing of
// a row stays on chip but its histogram, and a row is read twice -- for the level-1 histogram and to mark
// what lies above the threshold bin and collect the keys inside it -- each time through a ring of
// 16-byte copies, so that the reads of the next 48 KB per CTA are under way while the last are worked on.
// The searches of different rows overlap one another's reads; there is no cluster and no exchange.
#pragma once

constexpr int kStreamThreads = 512;
constexpr int kStreamWarps = kStreamThreads / 32;
constexpr int kStreamRound = 4 * kStreamThreads;   // entries per round of the CTA: 8 KB
constexpr int kStreamBatch = 2;                    // rounds per commit group
constexpr int kStreamGroups = 4;                   // groups in the ring
constexpr int kStreamMax = 131072;                 // entries per row: 64 rounds
// Level-1 bins of the exponent and four mantissa bits: half as many keys per bin as with three.  A bin
// keeps the sum of the low 14 mantissa bits in one word and the sum of the upper ten (hidden bit included) in
// another; neither overflows in kStreamMax entries.
constexpr int kStreamBins = 4096;
// After the level-1 search the histogram's bytes hold the bit mask of the row and the keys of the bin.
constexpr int kStreamStoreWords = 2 * kStreamBins + 1024;

struct StreamShared {
  alignas(16) unsigned int store[kStreamStoreWords];
  alignas(16) float ring[kStreamGroups * kStreamBatch * kStreamRound];
  unsigned int kmax;
  int oct_min, overflow;
  unsigned int cl_kmax;
  Found fd;
  int warp_cnt[kStreamWarps];
};
// The ring is idle outside the passes and then holds the scratch of the search and the staging lines of
// the emission.
struct StreamScratch {
  unsigned long long oct[kOctaves];
  LevelHist lv;
  Picks pk;
  unsigned int keys[2 * kDirectMax];
};
static_assert(sizeof(StreamScratch) <= sizeof(float) * kStreamGroups * kStreamBatch * kStreamRound, "scratch in the ring");
static_assert(2 * (sizeof(StreamShared) + 1024) <= 227 * 1024, "two CTAs per SM");
static_assert(kStreamThreads == 512, "a key of a warp's list: 13 bits of place, 19 bits of mantissa");

__device__ __forceinline__ void stream_bump(unsigned int* hist, unsigned int key) {
  unsigned int* const p = reinterpret_cast<unsigned int*>(reinterpret_cast<char*>(hist) + ((key >> 17) & 0x3ffcu));
  atomicAdd(p, key & 0x3fffu);
  atomicAdd(p + kStreamBins, ((key >> 14) & 0x1ffu) | ((key >= 0x800000u) ? 0x200u : 0u));
}

// Walks the row through the ring: f(round, keys) for every round's float4 of this thread, zeros beyond n,
// in rounds of the whole CTA (all threads call f equally often).
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
      const float4 v = *reinterpret_cast<const float4*>(sh.ring + ((gq % kStreamGroups) * kStreamBatch + j) * kStreamRound + 4 * tid);
      k[4 * j] = __float_as_uint(v.x + 0.f);  // -0.0 reads as +0.0
      k[4 * j + 1] = __float_as_uint(v.y + 0.f);
      k[4 * j + 2] = __float_as_uint(v.z + 0.f);
      k[4 * j + 3] = __float_as_uint(v.w + 0.f);
    }
    f(gq * kStreamBatch, k);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

__global__ void __launch_bounds__(kStreamThreads, 2) stream_rows_kernel(const __grid_constant__ SelectParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamShared& sh = *reinterpret_cast<StreamShared*>(smem_raw);
  StreamScratch& sc = *reinterpret_cast<StreamScratch*>(sh.ring);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int list = blockIdx.x;  // (used slot, sequence, group)
  const int g = list % P.G;
  const int b = (list / P.G) % P.B;
  const int slot = list / (P.G * P.B);
  const long long out_list = (static_cast<long long>(P.layer_of[slot]) * P.B + b) * P.G + g;
  unsigned int* const hist = sh.store;
  for (int i = tid; i < 2 * kStreamBins / 4; i += kStreamThreads) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    sh.kmax = 0u;
    sh.oct_min = kOctaves;
    sh.overflow = 0;
  }
  __syncthreads();
  pdl_wait();  // nothing is read or written before the previous kernel's end ...
  pdl_launch_dependents();  // ... and only then may the next one be scheduled
  long long Lll = P.kv_len[b];
  if (Lll < 0) Lll = 0;
  if (Lll > P.L_stride) Lll = P.L_stride;
  const int L = static_cast<int>(Lll);
  const float* A = (P.agg != nullptr) ? P.agg + static_cast<long long>(list) * P.L_stride
                                      : P.probs[slot] + static_cast<long long>(b) * P.H * P.gamma * P.L_stride;

  // ---- first pass: level-1 histogram and validity ----------------------------------------------------
  unsigned int kmax = 0u;
  stream_pass(sh, A, L, [&](int, const unsigned int (&k)[4 * kStreamBatch]) {
    constexpr int N = 4 * kStreamBatch;
#pragma unroll
    for (int j = 0; j < N; ++j) kmax = max(kmax, k[j]);
    // every value of the warp in one bin (ties, constant rows): the warp reduces first
    const unsigned int bin0 = __shfl_sync(kFull, k[0] >> 19, 0);
    bool one = false;
    if (__all_sync(kFull, (k[0] >> 19) == bin0)) {
      unsigned int differ = 0u;
#pragma unroll
      for (int j = 1; j < N; ++j) differ |= k[j] ^ k[0];
      one = __all_sync(kFull, (differ >> 19) == 0u);
    }
    if (one) {
      unsigned int lo = 0u, hi = 0u;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        lo += k[j] & 0x3fffu;
        hi += mantissa_of(k[j]) >> 14;
      }
      lo = __reduce_add_sync(kFull, lo);
      hi = __reduce_add_sync(kFull, hi);
      if (lane == 0 && (lo | hi) != 0u) {
        atomicAdd(&hist[bin0 & (kStreamBins - 1)], lo);
        atomicAdd(&hist[kStreamBins + (bin0 & (kStreamBins - 1))], hi);
      }
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j)
        if (k[j] != 0u) stream_bump(hist, k[j]);
    }
  });
  kmax = __reduce_max_sync(kFull, kmax);
  if (lane == 0 && kmax != 0u) atomicMax(&sh.kmax, kmax);

  // ---- the octave and the bin of the threshold -------------------------------------------------------
  if (tid < kOctaves) {
    unsigned long long s = 0ull;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint4 lo = *reinterpret_cast<const uint4*>(&hist[16 * tid + 4 * h]);
      const uint4 hi = *reinterpret_cast<const uint4*>(&hist[kStreamBins + 16 * tid + 4 * h]);
      s += ((static_cast<unsigned long long>(hi.x) + hi.y + hi.z + hi.w) << 14) + lo.x + lo.y + lo.z + lo.w;
    }
    sc.oct[tid] = s;
    const int first = __reduce_min_sync(kFull, (s != 0ull) ? tid : kOctaves);
    if (lane == 0 && first < kOctaves) atomicMin(&sh.oct_min, first);
  }
  __syncthreads();
  if (warp == 0) {
    Found fd;
    fd.total = fd.target = fd.carry = fd.above = fd.upto = 0.0;
    fd.bin = fd.oct = 0;
    fd.count = 0u;
    const unsigned int km = sh.kmax;
    if (km <= 0x7f7fffffu && sh.oct_min < kOctaves) {
      fd.oct = find_octave(
          static_cast<int>(km >> 23), sh.oct_min, P.p, [&](int e) { return sc.oct[e]; }, fd.total, fd.target, fd.carry);
      const int bin = 16 * fd.oct + (lane & 15);
      const unsigned long long s = (lane < 16) ? (static_cast<unsigned long long>(hist[kStreamBins + bin]) << 14) + hist[bin] : 0ull;
      const int b16 = find_from_top<4>(static_cast<double>(s) * pow2_double(max(fd.oct, 1) - 150), 0.0, fd.carry, fd.target,
                                       fd.above, fd.upto);
      fd.bin = 16 * fd.oct + b16;
      // a bin's smallest mantissa bounds the number of its keys (not in the bin of zero)
      const unsigned long long sb = __shfl_sync(kFull, s, b16);
      const unsigned int base = mantissa_of(static_cast<unsigned int>(fd.bin) << 19);
      fd.count = (base != 0u) ? static_cast<unsigned int>(min(sb / base, 0x7fffffffull)) : 0x7fffffffu;
    }
    if (lane == 0) sh.fd = fd;
  }
  __syncthreads();
  const bool invalid = sh.kmax > 0x7f7fffffu;
  const double total = sh.fd.total, target = sh.fd.target, carry = sh.fd.carry;
  double m_gt = 0.0, m_ge = total;
  const bool searching = !invalid && target > 0.0 && !P.keep_all;  // else p >= 1 or an all-zero row: keep all
  const int groups = (L + 127) / 128;                              // groups of 128 entries: four mask words each
  unsigned int* const mask = sh.store;
  unsigned int theta = 0u;
  if (searching) {
    const double scale = pow2_double(max(sh.fd.oct, 1) - 150);
    unsigned int prefix = static_cast<unsigned int>(sh.fd.bin);
    int shift = 19;
    double inner = sh.fd.above;
    unsigned int M = sh.fd.count;
    // room for keys behind the mask, an equal part for every warp
    const int mask_words = (4 * groups + 3) & ~3;
    const int cap = (kStreamStoreWords - mask_words) / kStreamWarps;
    unsigned int* const list_w = sh.store + mask_words + warp * cap;
    int n_list = 0;
    for (;;) {
      __syncthreads();  // (the histogram's bytes, the level histogram and the flags of the last trip were read by all)
      if (tid == 0) sh.overflow = 0;
      // ---- a well filled bin: 10 (then the last 9) more bits, one pass over the row ------------------------
      while (M > static_cast<unsigned int>(kStreamWarps * cap) && shift > 0) {
        // (the pass uses the ring, whose bytes the level histogram shares: it lives in the store meanwhile)
        LevelHist& lv = *reinterpret_cast<LevelHist*>(sh.store);
        const int sh_l = max(shift - 10, 0);
        const int up = shift - sh_l;
        level_clear<kStreamThreads>(lv);
        __syncthreads();
        stream_pass(sh, A, L, [&](int, const unsigned int (&k)[4 * kStreamBatch]) {
#pragma unroll
          for (int j = 0; j < 4 * kStreamBatch; ++j)
            level_add(lv, (k[j] >> shift) == prefix && k[j] != 0u, k[j], sh_l, up);
        });
        for (int gi = warp; gi < 32; gi += kStreamWarps) {
          const int bin = gi * 32 + lane;
          unsigned long long s = 0ull;
          if (bin < (1 << up))
            s = static_cast<unsigned long long>(lv.cnt[bin]) * mantissa_of(((prefix << up) | static_cast<unsigned int>(bin)) << sh_l) + lv.sum[bin];
#pragma unroll
          for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFull, s, d);
          if (lane == 0) lv.grp[gi] = s;
        }
        __syncthreads();
        if (warp == 0) {
          double above, upto, above1, upto1;
          const int gi = find_from_top<5>(static_cast<double>(lv.grp[lane]) * scale, inner, carry, target, above, upto);
          const int bin = gi * 32 + lane;
          const unsigned int c = (bin < (1 << up)) ? lv.cnt[bin] : 0u;
          const unsigned long long m = static_cast<unsigned long long>(c) * mantissa_of(((prefix << up) | static_cast<unsigned int>(bin)) << sh_l) +
                                       (c != 0u ? lv.sum[bin] : 0u);
          const int b1 = find_from_top<5>(static_cast<double>(m) * scale, above, carry, target, above1, upto1);
          const unsigned int cb = __shfl_sync(kFull, c, b1);
          if (lane == 0) {
            sh.fd.bin = gi * 32 + b1;
            sh.fd.count = cb;
            sh.fd.above = above1;
            sh.fd.upto = upto1;
          }
        }
        __syncthreads();
        prefix = (prefix << up) | static_cast<unsigned int>(sh.fd.bin);
        M = sh.fd.count;
        inner = sh.fd.above;
        shift = sh_l;
        if (shift == 0) {  // one distinct key left: the threshold
          theta = prefix;
          m_gt = carry + inner;
          m_ge = carry + sh.fd.upto;
        }
        __syncthreads();
      }
      // ---- second pass: mark what lies above the bin (above or at a known threshold), collect its keys -----
      const unsigned int lo_key = (prefix != 0u) ? prefix << shift : 1u;
      const unsigned int top_key = (prefix << shift) + ((1u << shift) - 1u), span = top_key - lo_key;
      const unsigned int keep_key = (shift == 0) ? theta : top_key + 1u;  // kept whatever the threshold turns out to be
      n_list = 0;
      stream_pass(sh, A, L, [&](int round, const unsigned int (&k)[4 * kStreamBatch]) {
#pragma unroll
        for (int j = 0; j < kStreamBatch; ++j) {
          unsigned int mine = 0u;
          bool any = false;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const unsigned int m = __ballot_sync(kFull, k[4 * j + e] >= keep_key);
            if (lane == e) mine = m;
            any |= k[4 * j + e] - lo_key <= span;
          }
          const int grp = (round + j) * kStreamWarps + warp;
          if (lane < 4 && grp < groups) mask[4 * grp + lane] = mine;
          if (shift > 0 && __any_sync(kFull, any)) {
            // one word per key: its place among the warp's entries and its bits below the prefix
            const unsigned int place = static_cast<unsigned int>(((round + j) * 32 + lane) * 4) << 19;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const unsigned int d = k[4 * j + e] - (prefix << shift);
              const bool in = k[4 * j + e] - lo_key <= span;
              const unsigned int m = __ballot_sync(kFull, in);
              const int at = n_list + __popc(m & ((1u << lane) - 1u));
              if (in && at < cap) list_w[at] = place + (static_cast<unsigned int>(e) << 19) + d;
              n_list += __popc(m);
            }
          }
        }
      });
      if (n_list > cap && lane == 0) sh.overflow = 1;
      __syncthreads();
      if (!sh.overflow) break;
      M = 0x7fffffffu;  // one warp's part was too small: narrow the bin down first
    }
    if (shift > 0) {
      // ---- the threshold among the collected keys: 10 bits over all lists, then what is left of them -------
      unsigned int pre = prefix;
      const int sh_l = (shift == 19) ? 9 : 0;
      const int up = shift - sh_l;
      level_clear<kStreamThreads>(sc.lv);
      if (tid == 0) sh.fd.key = 0u;
      __syncthreads();
      const int n_mine = min(n_list, cap);
      const unsigned int key0 = prefix << shift;
      for (int i = lane; i < ((n_mine + 31) & ~31); i += 32) {
        const unsigned int k = (i < n_mine) ? key0 + (list_w[i] & 0x7ffffu) : 0u;
        level_add(sc.lv, i < n_mine, k, sh_l, up);
      }
      __syncthreads();
      for (int gi = warp; gi < 32; gi += kStreamWarps) {
        const int bin = gi * 32 + lane;
        unsigned long long s = 0ull;
        if (bin < (1 << up))
          s = static_cast<unsigned long long>(sc.lv.cnt[bin]) * mantissa_of(((pre << up) | static_cast<unsigned int>(bin)) << sh_l) + sc.lv.sum[bin];
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(kFull, s, d);
        if (lane == 0) sc.lv.grp[gi] = s;
      }
      __syncthreads();
      if (warp == 0) {
        double above, upto, above1, upto1;
        const int gi = find_from_top<5>(static_cast<double>(sc.lv.grp[lane]) * scale, inner, carry, target, above, upto);
        const int bin = gi * 32 + lane;
        const unsigned int c = (bin < (1 << up)) ? sc.lv.cnt[bin] : 0u;
        const unsigned long long m = static_cast<unsigned long long>(c) * mantissa_of(((pre << up) | static_cast<unsigned int>(bin)) << sh_l) +
                                     (c != 0u ? sc.lv.sum[bin] : 0u);
        const int b1 = find_from_top<5>(static_cast<double>(m) * scale, above, carry, target, above1, upto1);
        const unsigned int cb = __shfl_sync(kFull, c, b1);
        if (lane == 0) {
          sh.fd.bin = gi * 32 + b1;
          sh.fd.count = cb;
          sh.fd.above = above1;
          sh.fd.upto = upto1;
          sh.overflow = 0;  // (counts the keys of that bin below)
        }
      }
      __syncthreads();
      pre = (pre << up) | static_cast<unsigned int>(sh.fd.bin);
      inner = sh.fd.above;
      if (sh_l == 0) {
        theta = pre;
        m_gt = carry + inner;
        m_ge = carry + sh.fd.upto;
      } else {
        const int left = static_cast<int>(sh.fd.count);
        double above, upto;
        if (left <= kDirectMax) {
          for (int i = lane; i < n_mine; i += 32) {
            const unsigned int k = key0 + (list_w[i] & 0x7ffffu);
            if ((k >> sh_l) == pre) sc.keys[atomicAdd(&sh.overflow, 1)] = k;
          }
          __syncthreads();
          theta = threshold_among<kStreamThreads>(sc.keys, left, pre, sh_l, inner, carry, target, scale, sc.lv, sh.fd, sc.pk,
                                                  above, upto);
        } else {  // many equal keys: the last nine bits the same way
          level_clear<kStreamThreads>(sc.lv);
          __syncthreads();
          for (int i = lane; i < ((n_mine + 31) & ~31); i += 32) {
            const unsigned int k = (i < n_mine) ? key0 + (list_w[i] & 0x7ffffu) : 0u;
            level_add(sc.lv, i < n_mine && (k >> sh_l) == pre, k, 0, 9);
          }
          __syncthreads();
          if (warp == 0) {
            // 512 bins, 16 per lane
            unsigned long long s = 0ull;
            for (int j = 0; j < 16; ++j)
              s += static_cast<unsigned long long>(sc.lv.cnt[16 * lane + j]) * mantissa_of((pre << 9) | static_cast<unsigned int>(16 * lane + j));
            double ab, up2, ab1, up1;
            const int l = find_from_top<5>(static_cast<double>(s) * scale, inner, carry, target, ab, up2);
            const int bin = 16 * l + (lane & 15);
            const unsigned long long m = (lane < 16) ? static_cast<unsigned long long>(sc.lv.cnt[bin]) * mantissa_of((pre << 9) | static_cast<unsigned int>(bin)) : 0ull;
            const int b1 = find_from_top<4>(static_cast<double>(m) * scale, ab, carry, target, ab1, up1);
            if (lane == 0) {
              sh.fd.key = (pre << 9) | static_cast<unsigned int>(16 * l + b1);
              sh.fd.above = ab1;
              sh.fd.upto = up1;
            }
          }
          __syncthreads();
          theta = sh.fd.key;
          above = sh.fd.above;
          upto = sh.fd.upto;
        }
        m_gt = carry + above;
        m_ge = carry + upto;
      }
      // keys of the bin that made it join the mask (a warp's keys lie in its own words)
      for (int i = lane; i < n_mine; i += 32) {
        const unsigned int w = list_w[i];
        if (key0 + (w & 0x7ffffu) >= theta) {
          const int place = static_cast<int>(w >> 19);  // (round * 32 + lane) * 4 + e
          const int grp = (place >> 7) * kStreamWarps + warp;
          atomicOr(&mask[4 * grp + (place & 3)], 1u << ((place >> 2) & 31));
        }
      }
    }
    __syncthreads();
  }

  // ---- ordered emission ---------------------------------------------------------------------------------
  int* const out = P.idx + out_list * P.idx_stride;
  const int stride = static_cast<int>(min(P.idx_stride, static_cast<long long>(INT_MAX)));
  int count = 0;
  if (searching) {
    const int per_warp = (groups + kStreamWarps - 1) / kStreamWarps;
    const int g_lo = min(groups, warp * per_warp), g_hi = min(groups, g_lo + per_warp);
    int wc = 0;
    for (int w = 4 * g_lo + lane; w < 4 * g_hi; w += 32) wc += __popc(mask[w]);
    wc = __reduce_add_sync(kFull, wc);
    if (lane == 0) sh.warp_cnt[warp] = wc;
    __syncthreads();
    const int v = (lane < kStreamWarps) ? sh.warp_cnt[lane] : 0;
    count = __reduce_add_sync(kFull, v);
    int pos = __reduce_add_sync(kFull, lane < warp ? v : 0);
    // The kept positions of 128 entries go through a per-warp staging line, so that the global stores
    // are whole 128-byte runs (a lane storing its own up to four positions spreads every store
    // instruction over the whole 512-byte range: four partial writes per sector).
    int* const stage = reinterpret_cast<int*>(sh.ring) + warp * 128;
    const unsigned int lt = (1u << lane) - 1u;
    for (int gi = g_lo; gi < g_hi; ++gi) {
      const uint4 m = *reinterpret_cast<const uint4*>(mask + 4 * gi);  // (the same words in every lane)
      if ((m.x | m.y | m.z | m.w) == 0u) continue;
      const int first = 128 * gi + 4 * lane;
      int at = __popc(m.x & lt) + __popc(m.y & lt) + __popc(m.z & lt) + __popc(m.w & lt);
      const int kept = __popc(m.x) + __popc(m.y) + __popc(m.z) + __popc(m.w);
      if ((m.x >> lane) & 1u) stage[at++] = first;
      if ((m.y >> lane) & 1u) stage[at++] = first + 1;
      if ((m.z >> lane) & 1u) stage[at++] = first + 2;
      if ((m.w >> lane) & 1u) stage[at++] = first + 3;
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int t = 32 * j + lane;
        if (t < kept && pos + t < stride) out[pos + t] = stage[t];
      }
      __syncwarp();
      pos += kept;
    }
  } else if (!invalid) {
    count = L;
    for (int i = tid; i < min(L, stride); i += kStreamThreads) out[i] = i;
  }
  if (tid == 0) {
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
}
