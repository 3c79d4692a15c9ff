// specattn_select_topp: aggregation of draft attention rows, exact sorting-free top-p
// threshold search and ordered compaction, for sm_100a.
//
// Paper: Sec. 3.4 / Alg. 2 (target mass p * sum a, membership a_i >= theta) and App. A Eq. 7
// (smallest set reaching mass p).  Alg. 2 bisects theta in the probability domain with one
// full pass over the row per iteration; here the same fixed point is reached exactly by a
// histogram over the top 11 bits of the binary32 pattern and a search among the keys of one bin
// (row_search.cuh), and the row never leaves the chip between passes.
//
// Mapping to the GPU: one thread-block cluster (1 to 16 CTAs) per index list; each CTA keeps its
// slice of the searched row in shared memory.
//   - A list with one contributing row (top-p filtering, or a row that a first launch has already
//     summed) is copied there with 16-byte cp.async, all of the slice in flight at once: the row
//     is read from HBM exactly once whatever its values.
//   - Otherwise the CTA streams its slice of all contributing (head, query) rows in 8 KB row
//     pieces: every thread copies the float4 columns it will add itself into its own ring slots,
//     eight pieces ahead (64 KB in flight per CTA, no registers held, no barrier needed), adds them
//     in the fixed order that defines the aggregated row and keeps the sum in shared memory.  (A 1-D
//     bulk-copy ring fed by a producer warp was measured first: like the gather in the verify kernel
//     it stalled near 25 GB/s per SM.)
//   - The level-1 histogram is built as the values arrive; the search, the count and the ordered
//     emission of the kept positions then run on the slice.
// With a workspace the call becomes two launches: aggregate_rows_kernel sums the rows with 512
// positions per CTA (the whole GPU streams, however few the lists) and the search reads that sum.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "ptx.cuh"
#include "nvtx_range.h"
#include "specattn.h"

namespace cg = cooperative_groups;

namespace specattn {

extern std::atomic<long long> g_launch_count;
int device_sm_count();

namespace {

constexpr int kChunk = 2048;             // positions per staged row piece (8 KB)
constexpr int kDepth = 8;                // row pieces in flight per thread (ring of 8 x 8 KB)
constexpr unsigned int kFull = 0xffffffffu;

struct SelectParams {
  const float* probs[SPECATTN_MAX_DRAFT_LAYERS];  // per used slot
  int layer_of[SPECATTN_MAX_DRAFT_LAYERS];        // draft layer id of a used slot
  signed char head_group[SPECATTN_MAX_DRAFT_HEADS];
  int has_groups;
  int n_used, B, H, gamma, G;
  long long L_stride;
  const int* kv_len;
  float p;
  int keep_all;
  int* idx;
  long long idx_stride;
  int* counts;
  int* status;
  double* diag;
  int per_step;    // Alg. 2 as printed: one nucleus per speculated query, unioned
  int bisect_iters;  // > 0: the threshold is the last midpoint of that many bisection steps
  int chunk;         // > 1: selection over per-chunk sums (power of two, 4..64); kept chunks keep all positions
  int apart;         // per_step at chunk granularity: the queries are searched by one CTA each, all at once
  const float* agg;  // two-launch form: the aggregated rows, [list][L_stride], written by aggregate_rows_kernel
};

#include "row_search.cuh"

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst_smem, const void* src_gmem, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src_gmem), "r"(bytes) : "memory");
}

// Shared memory of a CTA: the fixed part of the search, the list's heads (aggregation only), the
// slice, then the scratch of the search -- over the staging ring, which is idle by then.
constexpr size_t kFixedBytes = (sizeof(SearchFixed) + 127) / 128 * 128;
constexpr size_t kHeadBytes = SPECATTN_MAX_DRAFT_HEADS * sizeof(short) + 128;
constexpr size_t kScratchBytes = (sizeof(SearchScratch) + 127) / 128 * 128;
constexpr size_t kRingBytes = static_cast<size_t>(kDepth) * kChunk * sizeof(float);
static_assert(kScratchBytes <= kRingBytes, "the ring must hold the scratch of the search");
// two CTAs of a whole slice (plus 1 KB each that the system reserves) share the 227 KB of an SM
static_assert(2 * (kFixedBytes + kSliceMax * sizeof(float) + kScratchBytes + 1024) <= 227 * 1024, "two CTAs per SM");

// Entries per CTA when n entries are dealt to cs CTAs, and the same rounded up to whole rounds of nt
// float4s (what a CTA's slice occupies).
__host__ __device__ inline int slice_of(int n, int cs, int align) { return ((n + cs - 1) / cs + align - 1) / align * align; }
__host__ __device__ inline int slice_room(int slice, int nt) { return (slice + 4 * nt - 1) / (4 * nt) * (4 * nt); }

// Writes the kept entries of a warp's range [warp * w4, (warp + 1) * w4) float4s in ascending order
// behind `pos` kept ones.  Entry i of the slice is position lo + i, or chunk lo + i of `chunk` positions
// (the last chunk of the list is cut at L).  mask: bit per entry instead of the comparison (union of
// several searches), or nullptr.
__device__ __forceinline__ void emit_kept(const float* a, const unsigned int* mask, unsigned int theta, int n_loc, int lo,
                                          int w4, int chunk, int L, int pos, int* out, int stride) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  for (int g4 = warp * w4; g4 < (warp + 1) * w4; g4 += 32) {
    if (4 * g4 >= n_loc) break;
    if (mask == nullptr) {
      // most groups of 128 entries of a peaked row hold nothing
      const uint4 k4 = *reinterpret_cast<const uint4*>(a + 4 * (g4 + lane));
      if (!__any_sync(kFull, max(max(k4.x, k4.y), max(k4.z, k4.w)) >= theta)) continue;
    }
    unsigned int m[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * g4 + 32 * e + lane;
      const bool keep = (mask != nullptr) ? ((mask[(4 * g4 >> 5) + e] >> lane) & 1u) != 0u : __float_as_uint(a[i]) >= theta;
      m[e] = __ballot_sync(kFull, keep && i < n_loc);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * g4 + 32 * e + lane;
      const bool keep = (m[e] >> lane) & 1u;
      if (chunk <= 1) {
        const int my = pos + __popc(m[e] & lt);
        if (keep && my < stride) out[my] = lo + i;
        pos += __popc(m[e]);
      } else if (m[e] != 0u) {
        // every chunk before the list's last one is whole
        const int my = pos + __popc(m[e] & lt) * chunk;
        const int p0 = (lo + i) * chunk, np = keep ? min(chunk, L - p0) : 0;
        int* const o = out + my;
        if (np == chunk && my + chunk <= stride && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
          for (int j = 0; j < chunk; j += 4)
            *reinterpret_cast<int4*>(o + j) = make_int4(p0 + j, p0 + j + 1, p0 + j + 2, p0 + j + 3);
        } else {
          for (int j = 0; j < np; ++j)
            if (my + j < stride) o[j] = p0 + j;
        }
        pos += __popc(m[e]) * chunk;
      }
    }
  }
}

// Largest of N bit patterns k[4 j + e] = at[4 NT j + e] of a copied row: above 0x7f7fffff for a
// negative, NaN or infinite input.  -0.0 is a zero and is rewritten as such.
template <int N, int NT>
__device__ __forceinline__ unsigned int checked_max(unsigned int (&k)[N], float* at) {
  unsigned int m = 0u;
#pragma unroll
  for (int i = 0; i < N; ++i) m = max(m, k[i]);
  if (m > 0x7f7fffffu) {
    m = 0u;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (k[i] == 0x80000000u) {
        k[i] = 0u;
        at[4 * NT * (i >> 2) + (i & 3)] = 0.f;
      }
      m = max(m, k[i]);
    }
  }
  return m;
}

// kAgg: the CTA sums the contributing rows itself (one-launch form over several rows); otherwise the
// list's row lies in global memory and is copied.  kVariant: the selection variants of Alg. 2 (per-step
// union, fixed-iteration bisection, chunks); the default instantiations contain none of their code.
template <bool kAgg, bool kVariant, int NT>
__global__ void __launch_bounds__(NT, NT >= 512 || kAgg ? 2 : 8) select_topp_kernel(const __grid_constant__ SelectParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr int kW = NT / 32;
  SearchFixed& fx = *reinterpret_cast<SearchFixed*>(smem_raw);
  short* const heads = reinterpret_cast<short*>(smem_raw + kFixedBytes);  // heads feeding the list, ascending
  int* const n_heads = reinterpret_cast<int*>(heads + SPECATTN_MAX_DRAFT_HEADS);
  float* const a = reinterpret_cast<float*>(smem_raw + kFixedBytes + (kAgg ? kHeadBytes : 0));

  cg::cluster_group cluster = cg::this_cluster();
  const int cs = static_cast<int>(cluster.num_blocks());
  const int rank = static_cast<int>(cluster.block_rank());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a one-CTA "cluster" needs no hardware cluster barrier
  auto csync = [&]() {
    if (cs > 1) cluster.sync(); else __syncthreads();
  };

  const int list = blockIdx.y;  // (used slot, sequence, group)
  const int g = list % P.G;
  const int b = (list / P.G) % P.B;
  const int slot = list / (P.G * P.B);
  const long long out_list = (static_cast<long long>(P.layer_of[slot]) * P.B + b) * P.G + g;

  auto clear = [&]() {
    for (int i = tid; i < 2 * kL1Bins / 4; i += NT) reinterpret_cast<uint4*>(fx.hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
      fx.kmax = 0u;
      fx.oct_min = kOctaves;
    }
  };
  clear();
  if (kAgg && tid == 0) {
    int n = 0;
    for (int h = 0; h < P.H; ++h)
      if (!P.has_groups || P.head_group[h] == g) heads[n++] = static_cast<short>(h);
    *n_heads = n;
  }
  __syncthreads();
  // Launched while the previous kernel may still run: nothing is read or written before its end.
  // Only then may the next kernel of the stream be scheduled, so that it never overtakes that one.
  pdl_wait();
  pdl_launch_dependents();

  long long Lll = P.kv_len[b];
  if (Lll < 0) Lll = 0;
  if (Lll > P.L_stride) Lll = P.L_stride;
  const int L = static_cast<int>(Lll);
  const bool chunked = kVariant && P.chunk > 1;
  const int chunk = chunked ? P.chunk : 1;
  const int per = slice_of(L, cs, chunk > 4 ? chunk : 4);  // slices start on 16 bytes and on a chunk
  const int lo = min(L, rank * per);
  const int n_loc = min(L, lo + per) - lo;
  // entries of the searched row in this slice, and the float4s they occupy with their padding
  const int n_srch = chunked ? (n_loc + chunk - 1) / chunk : n_loc;
  const int n4_pad = slice_room(n_srch, NT) / 4;
  float* const ring = a + slice_room(slice_of(static_cast<int>(P.L_stride), cs, chunk > 4 ? chunk : 4), NT);
  SearchScratch& sc = *reinterpret_cast<SearchScratch*>(ring);
  unsigned int* const mask = reinterpret_cast<unsigned int*>(reinterpret_cast<unsigned char*>(ring) + kRingBytes);

  const float* A = (!kAgg && P.agg != nullptr)
                       ? P.agg + static_cast<long long>(list) * P.L_stride + lo
                       : P.probs[slot] + static_cast<long long>(b) * P.H * P.gamma * P.L_stride + lo;
  // Alg. 2 as printed selects per speculated query and unions the sets: then everything up to
  // the threshold runs once per query over the row summed over heads only, and the kept
  // entries are collected in a bit mask of the slice.
  const int n_steps = (kAgg && kVariant && P.per_step) ? P.gamma : 1;
  const bool use_mask = kAgg && kVariant && P.per_step;
  const int w4 = n4_pad / kW;  // float4s per warp in the passes over the slice
  SearchResult res;
  bool invalid = false;
  // Searches apart: chunk scores of all queries are few (a list of 32768 positions in chunks of 16: 2048 per
  // query), so they are kept while the rows of all queries stream in one go; then every CTA of the
  // cluster gathers the scores of one query and searches them alone, all queries at once, instead of the
  // cluster searching one query after the other (9 us each, the streaming idle meanwhile: five queries of 32 such
  // lists 88 us).
  const bool apart = kAgg && kVariant && P.apart;
  const int row_room = apart ? slice_of(static_cast<int>(P.L_stride), cs, chunk) / chunk : 0;  // entries per query and CTA
  float* const scores = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(mask) +
                                                 (apart ? slice_room(slice_of(static_cast<int>(P.L_stride), cs, chunk), NT) / 8 : 0));
  bool bad = false;
  int ic = 0, ih = 0, is = 0, istep = 0, islot = 0, slot_c = 0;  // column, head, query, step and ring slots of the next piece
  for (int step = 0; step < n_steps; ++step) {
    if (kAgg && step > 0 && !apart) {
      clear();
      __syncthreads();
    }
    unsigned int kmax = 0u;

    // ---- the slice and its level-1 histogram -------------------------------------------------------
    if (!kAgg) {
      // Every thread copies exactly the float4s it will enter into the histogram, in two halves of
      // four: no barrier before the histogram, and the second half lands under the first half's pass.
      // The copies fill what lies beyond the slice with zeros.
      const int rounds = n4_pad / NT;
      const uint32_t dst = smem_u32(a) + tid * 16;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j < rounds) {
          const int left = n_loc - 4 * (j * NT + tid);
          cp_async16_zfill(dst + j * NT * 16, A + (left > 0 ? 4 * (j * NT + tid) : 0),
                           left >= 4 ? 16u : (left > 0 ? 4u * left : 0u));
        }
        if (j == 3 || j == 7) asm volatile("cp.async.commit_group;" ::: "memory");
      }
      auto take = [&](int j, unsigned int* k) {
        const uint4 v = *reinterpret_cast<const uint4*>(a + 4 * (j * NT + tid));
        k[0] = v.x;
        k[1] = v.y;
        k[2] = v.z;
        k[3] = v.w;
      };
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (half == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        const int j0 = 4 * half;
        if (rounds >= j0 + 4) {
          unsigned int k[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) take(j0 + j, k + 4 * j);
          kmax = max(kmax, checked_max<16, NT>(k, a + 4 * (j0 * NT + tid)));
          hist_add<16>(fx.hist, k);
        } else {
          for (int j = j0; j < rounds; ++j) {
            unsigned int k[4];
            take(j, k);
            kmax = max(kmax, checked_max<4, NT>(k, a + 4 * (j * NT + tid)));
            hist_add<4>(fx.hist, k);
          }
        }
      }
    } else {
      // Pieces are numbered q = piece column * R + row, i.e. in the order the adds must happen.
      // Completion is tracked per thread (commit / wait groups), so the pipeline needs no barrier.
      constexpr int kCols = kChunk / (4 * NT);
      const int n_pos4 = (n_loc + 3) & ~3;
      const int n_chunks = (n_pos4 + kChunk - 1) / kChunk;
      const int n_q = use_mask ? 1 : P.gamma;  // rows per head
      const int R = *n_heads * n_q;
      const uint32_t ring_addr = smem_u32(ring) + tid * 16;
      const float* src0 = A + 4 * tid;
      auto issue = [&]() {
        if (ic < n_chunks && R > 0) {
          const int len4 = min(kChunk, n_pos4 - ic * kChunk) >> 2;
          const float* src = src0 + static_cast<long long>(heads[ih] * P.gamma + (use_mask ? istep : is)) * P.L_stride + ic * kChunk;
          const uint32_t dst = ring_addr + islot * (kChunk * 4);
#pragma unroll
          for (int k = 0; k < kCols; ++k)
            if (tid + k * NT < len4) cp_async16(dst + k * NT * 16, src + k * NT * 4);
          if (++is == n_q) {
            is = 0;
            if (++ih == *n_heads) {
              ih = 0;
              if (++ic == n_chunks && apart && istep + 1 < n_steps) {  // on to the next query's rows without a break
                ic = 0;
                ++istep;
              }
            }
          }
          islot = (islot + 1) & (kDepth - 1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
      if (step == 0 || !apart) {
        ic = ih = is = islot = slot_c = 0;
        istep = step;
        for (int q = 0; q < kDepth - 1; ++q) issue();
      }
      // Validity of the inputs is tracked with a running minimum (a negative input, the only
      // invalid value a sum can hide) -- NaN and Inf survive into the aggregated value itself.
      float4 acc[kCols], mn[kCols];
#pragma unroll
      for (int k = 0; k < kCols; ++k) acc[k] = mn[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int c = 0; c < n_chunks; ++c) {
        const int len4 = min(kChunk, n_pos4 - c * kChunk) >> 2;
        // positions of this thread's float4s that lie beyond the slice (last float4 only)
        int cut[kCols];
#pragma unroll
        for (int k = 0; k < kCols; ++k) cut[k] = n_loc - (c * kChunk + 4 * (tid + k * NT));
        for (int r = 0; r < R; ++r) {
          issue();
          asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 1) : "memory");
          const float4* piece = reinterpret_cast<const float4*>(ring + slot_c * kChunk);
          slot_c = (slot_c + 1) & (kDepth - 1);
#pragma unroll
          for (int k = 0; k < kCols; ++k) {
            const int i4 = tid + k * NT;
            if (i4 < len4) {
              float4 x = piece[i4];
              if (cut[k] < 4) {  // values beyond kv_len are not inputs
                x.w = 0.f;
                if (cut[k] < 3) x.z = 0.f;
                if (cut[k] < 2) x.y = 0.f;
              }
              mn[k].x = fminf(mn[k].x, x.x);
              mn[k].y = fminf(mn[k].y, x.y);
              mn[k].z = fminf(mn[k].z, x.z);
              mn[k].w = fminf(mn[k].w, x.w);
              acc[k].x = acc[k].x + x.x;
              acc[k].y = acc[k].y + x.y;
              acc[k].z = acc[k].z + x.z;
              acc[k].w = acc[k].w + x.w;
            }
          }
        }
        // the column is complete: store it and feed the level-1 histogram
#pragma unroll
        for (int k = 0; k < kCols; ++k) {
          const int i4 = tid + k * NT;
          const float4 v = acc[k];
          if (i4 < len4) *reinterpret_cast<float4*>(a + c * kChunk + 4 * i4) = v;
          if (mn[k].x < 0.f || mn[k].y < 0.f || mn[k].z < 0.f || mn[k].w < 0.f) kmax = 0xffffffffu;
          const unsigned int key[4] = {__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)};
          const unsigned int m = max(max(key[0], key[1]), max(key[2], key[3]));
          // (the largest position does not bound a row of chunk scores; an infinite one voids it all the same)
          if (!chunked || m > 0x7f7fffffu) kmax = max(kmax, m);
          if (!chunked) hist_add<4>(fx.hist, key);
          acc[k] = mn[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (apart) {  // the chunks of the warp's 128 positions, one per lane
            __syncwarp();
            const int p0 = c * kChunk + 4 * (32 * warp + k * NT) + lane * chunk;
            if (lane * chunk < 128 && p0 < n_loc) {
              float s = 0.f;
              for (int e = 0; e < chunk; e += 4) {
                const float4 u = *reinterpret_cast<const float4*>(a + p0 + e);
                const int left = n_loc - (p0 + e);
                if (left > 0) s = s + u.x;
                if (left > 1) s = s + u.y;
                if (left > 2) s = s + u.z;
                if (left > 3) s = s + u.w;
              }
              scores[step * row_room + p0 / chunk] = s;
              bad |= !(s <= FLT_MAX);
            }
            __syncwarp();  // (the next query's values overwrite these)
          }
        }
      }
      if (apart) {
        bad |= kmax > 0x7f7fffffu;
        continue;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (chunked) {
        // Selection at chunk granularity: entry j of the searched row is the binary32 sum of the
        // chunk's aggregated values in ascending order (the last chunk of the list is cut at L).
        // The scores replace the head of the slice: a round reads NT chunks, then writes NT
        // entries that no later round reads.
        __syncthreads();  // the aggregated slice is complete
        for (int base = 0; base < n_srch; base += NT) {
          const int j = base + tid;
          const bool act = j < n_srch;
          float s = 0.f;
          if (act) {
            const int p0 = j * chunk;
            for (int e = 0; e < chunk; e += 4) {
              const float4 v = *reinterpret_cast<const float4*>(a + p0 + e);
              const int left = n_loc - (p0 + e);
              if (left > 0) s = s + v.x;
              if (left > 1) s = s + v.y;
              if (left > 2) s = s + v.z;
              if (left > 3) s = s + v.w;
            }
          }
          __syncthreads();
          if (act) a[j] = s;
          const unsigned int key[1] = {__float_as_uint(s)};
          kmax = max(kmax, key[0]);
          hist_add<1>(fx.hist, key);
        }
        __syncthreads();
      }
      for (int i = n_srch + tid; i < 4 * n4_pad; i += NT) {
        if (chunked || i >= n_pos4) a[i] = 0.f;
      }
    }
    kmax = __reduce_max_sync(kFull, kmax);
    if (lane == 0 && kmax != 0u) atomicMax(&fx.kmax, kmax);
    __syncthreads();
    hist_add_tiny<NT>(fx.hist, fx.kmax, a, n4_pad);

    res = search_slice<NT>(fx, sc, a, n4_pad, P.p, P.keep_all != 0, kVariant ? P.bisect_iters : 0, cs);
    invalid |= res.invalid;  // one query's invalid input voids the list
    if (use_mask) {
      // collect this query's set in the mask: a warp owns whole 32-entry words
      for (int i0 = 4 * warp * w4; i0 < 4 * (warp + 1) * w4; i0 += 32) {
        const int i = i0 + lane;
        const unsigned int m = __ballot_sync(kFull, !invalid && i < n_srch && __float_as_uint(a[i]) >= res.theta);
        if (lane == 0) mask[i0 >> 5] = (step == 0) ? m : (mask[i0 >> 5] | m);
      }
      // the next query's row overwrites the slice and the staging ring, which peers may still be reading
      csync();
    }
  }

  if (apart) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (tid == 0) fx.bad = 0;
    __syncthreads();
    if (bad) fx.bad = 1;
    csync();  // every CTA's scores are complete
    const int n_all = (L + chunk - 1) / chunk, per_e = per / chunk;
    const int n4_all = slice_room(n_all, NT) / 4;
    for (int s = rank; s < n_steps; s += cs) {
      clear();
      __syncthreads();
      unsigned int kmax = 0u;
      for (int i = tid; i < 4 * n4_all; i += NT) {
        float v = 0.f;
        if (i < n_all) {
          const int r = i / per_e;
          v = *cluster.map_shared_rank(scores + s * row_room + (i - r * per_e), r);
        }
        a[i] = v;
        const unsigned int key[1] = {__float_as_uint(v)};
        kmax = max(kmax, key[0]);
        hist_add<1>(fx.hist, key);
      }
      kmax = __reduce_max_sync(kFull, kmax);
      if (lane == 0 && kmax != 0u) atomicMax(&fx.kmax, kmax);
      __syncthreads();
      hist_add_tiny<NT>(fx.hist, fx.kmax, a, n4_all);
      res = search_slice<NT>(fx, sc, a, n4_all, P.p, P.keep_all != 0, P.bisect_iters, 1, rank);
      if (tid == 0) {
        fx.theta[s] = res.invalid ? 0xffffffffu : res.theta;
        if (s == n_steps - 1) {
          fx.masses[0] = res.total;
          fx.masses[1] = res.target;
          fx.masses[2] = res.m_gt;
          fx.masses[3] = res.m_ge;
        }
      }
      __syncthreads();
    }
    csync();  // every query has its threshold
    invalid = __any_sync(kFull, lane < cs && *cluster.map_shared_rank(&fx.bad, lane < cs ? lane : 0) != 0);
    unsigned int* const thetas = reinterpret_cast<unsigned int*>(ring);  // (the search's scratch is idle)
    if (tid < n_steps) thetas[tid] = *cluster.map_shared_rank(&fx.theta[tid], tid % cs);
    if (tid == 0) {
      const double* m = cluster.map_shared_rank(fx.masses, (n_steps - 1) % cs);
      res.total = m[0];
      res.target = m[1];
      res.m_gt = m[2];
      res.m_ge = m[3];
    }
    __syncthreads();
    for (int s = 0; s < n_steps; ++s) invalid |= thetas[s] == 0xffffffffu;
    for (int i0 = 4 * warp * w4; i0 < 4 * (warp + 1) * w4; i0 += 32) {
      const int i = i0 + lane;
      bool keep = false;
      if (i < n_srch && !invalid)
        for (int s = 0; s < n_steps; ++s) keep |= __float_as_uint(scores[s * row_room + i]) >= thetas[s];
      const unsigned int m = __ballot_sync(kFull, keep);
      if (lane == 0) mask[i0 >> 5] = m;
    }
    __syncthreads();
  }

  // ---- ordered compaction ------------------------------------------------------------------------
  // kept entries before this CTA's, and in all
  int before = 0, all = 0;
  const bool counted = res.counted && !use_mask;
  if (!counted && !invalid) {
    int wc = 0;
    for (int i0 = 4 * warp * w4; i0 < 4 * (warp + 1) * w4; i0 += 32) {
      const int i = i0 + lane;
      if (use_mask) wc += (i < n_srch) ? (mask[i0 >> 5] >> lane) & 1u : 0u;
      else wc += (i < n_srch && __float_as_uint(a[i]) >= res.theta) ? 1 : 0;
    }
    wc = __reduce_add_sync(kFull, wc);
    if (lane == 0) fx.warp_cnt[warp] = wc;
  }
  __syncthreads();
  const int wcnt = (lane < kW && !invalid) ? fx.warp_cnt[lane] : 0;
  if (!counted && cs > 1) {
    const int mine = __reduce_add_sync(kFull, wcnt);
    if (tid == 0) fx.local_kept = mine;
    csync();  // local_kept of every CTA is visible
    const int v = (lane < cs) ? *cluster.map_shared_rank(&fx.local_kept, lane) : 0;
    before = __reduce_add_sync(kFull, lane < rank ? v : 0);
    all = __reduce_add_sync(kFull, v);
  } else if (counted) {
    const int v = (lane < cs) ? fx.kept[lane] : 0;
    before = __reduce_add_sync(kFull, lane < rank ? v : 0);
    all = __reduce_add_sync(kFull, v);
  } else {
    all = __reduce_add_sync(kFull, wcnt);
  }
  // this CTA reads no peer's shared memory from here on; it leaves when the peers say the same
  __syncwarp();
  if (cs > 1) cluster_arrive_release();
  const int wbefore = __reduce_add_sync(kFull, lane < warp ? wcnt : 0);
  if (!invalid)
    emit_kept(a, use_mask ? mask : nullptr, res.theta, n_srch, chunked ? lo / chunk : lo, w4, chunk, L,
              (before + wbefore) * chunk, P.idx + out_list * P.idx_stride,
              static_cast<int>(min(P.idx_stride, static_cast<long long>(INT_MAX))));
  // the CTA that holds the row's last entry knows whether the last chunk (cut at L) is kept
  const bool last_holder = (L == 0) ? rank == 0 : (lo < L && lo + n_loc == L);
  if (last_holder && tid == 0) {
    long long count = static_cast<long long>(all) * chunk;
    if (chunked && L % chunk != 0) {
      const int i = n_srch - 1;
      if (use_mask ? ((mask[i >> 5] >> (i & 31)) & 1u) != 0u : __float_as_uint(a[i]) >= res.theta)
        count -= chunk - L % chunk;
    }
    int st = SPECATTN_ROW_OK;
    if (invalid) {
      st = SPECATTN_ROW_INVALID_PROB;
      count = 0;
    } else if (count > P.idx_stride) {
      st = SPECATTN_ROW_OVERFLOW;
    }
    P.counts[out_list] = static_cast<int>(count);
    P.status[out_list] = st;
    if (P.diag != nullptr) {
      double* d = P.diag + out_list * 4;
      d[0] = res.total;
      d[1] = res.target;
      d[2] = res.m_gt;
      d[3] = res.m_ge;
    }
  }
  __syncwarp();
  if (cs > 1) cluster_wait();  // nobody leaves while its shared memory may still be read remotely
}

#include "stream_rows.cuh"

// First launch of the two-launch form: a[i] = +0 + the contributing rows in order, for 512
// positions per CTA, so that the number of CTAs streaming the rows from HBM does not depend on
// the number of lists.  The adds are the ones of the cluster kernel (binary32, same order), so
// the bits of a[] are the same.  A negative input, which a sum could hide, poisons its
// position with NaN: the search then reports the list as invalid like the cluster kernel does.
constexpr int kAggThreads = 128;
constexpr int kAggPositions = kAggThreads * 4;
constexpr int kAggUnroll = 16;
__global__ void __launch_bounds__(kAggThreads) aggregate_rows_kernel(const __grid_constant__ SelectParams P,
                                                                  float* __restrict__ out) {
  __shared__ long long row_off[SPECATTN_MAX_ROWS_PER_LIST];
  __shared__ int n_rows;
  const int tid = threadIdx.x;
  const int list = blockIdx.y;
  const int g = list % P.G;
  const int b = (list / P.G) % P.B;
  const int slot = list / (P.G * P.B);
  long long Lll = P.kv_len[b];
  if (Lll < 0) Lll = 0;
  if (Lll > P.L_stride) Lll = P.L_stride;
  const int L = static_cast<int>(Lll);
  const int pos = blockIdx.x * kAggPositions + 4 * tid;
  if (blockIdx.x * kAggPositions >= L) return;
  if (tid == 0) {
    int n = 0;
    for (int h = 0; h < P.H; ++h) {
      if (P.has_groups && P.head_group[h] != g) continue;
      for (int s = 0; s < P.gamma; ++s) row_off[n++] = static_cast<long long>(h * P.gamma + s) * P.L_stride;
    }
    n_rows = n;
  }
  __syncthreads();
  if (pos >= L) return;
  const int R = n_rows;
  const int cut = L - pos;  // positions of this float4 that are inputs
  const float* src = P.probs[slot] + static_cast<long long>(b) * P.H * P.gamma * P.L_stride + pos;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), mn = acc;
  for (int r0 = 0; r0 < R; r0 += kAggUnroll) {
    float4 x[kAggUnroll];
#pragma unroll
    for (int k = 0; k < kAggUnroll; ++k)
      if (r0 + k < R) x[k] = __ldcs(reinterpret_cast<const float4*>(src + row_off[r0 + k]));
#pragma unroll
    for (int k = 0; k < kAggUnroll; ++k) {
      if (r0 + k < R) {
        float4 v = x[k];
        if (cut < 4) {  // values beyond kv_len are not inputs
          v.w = 0.f;
          if (cut < 3) v.z = 0.f;
          if (cut < 2) v.y = 0.f;
        }
        mn.x = fminf(mn.x, v.x);
        mn.y = fminf(mn.y, v.y);
        mn.z = fminf(mn.z, v.z);
        mn.w = fminf(mn.w, v.w);
        acc.x = acc.x + v.x;
        acc.y = acc.y + v.y;
        acc.z = acc.z + v.z;
        acc.w = acc.w + v.w;
      }
    }
  }
  const float nan = __uint_as_float(0x7fc00000u);
  if (mn.x < 0.f) acc.x = nan;
  if (mn.y < 0.f) acc.y = nan;
  if (mn.z < 0.f) acc.z = nan;
  if (mn.w < 0.f) acc.w = nan;
  *reinterpret_cast<float4*>(out + static_cast<long long>(list) * P.L_stride + pos) = acc;
  // the search kernel's CTAs may move in as this grid drains (earlier, they would take thread
  // slots from CTAs that still stream); it waits for the whole grid before reading a[]
  pdl_launch_dependents();
}

// Number of index lists of a call (0 on invalid arguments) -- shared by the entry point and
// the workspace query.
long long count_lists(const specattn_select_args& A) {
  if (A.n_draft_layers < 1 || A.n_draft_layers > SPECATTN_MAX_DRAFT_LAYERS || A.n_target_layers < 0 ||
      A.batch < 0 || A.n_groups < 1 || A.layer_map == nullptr)
    return 0;
  bool used[SPECATTN_MAX_DRAFT_LAYERS] = {false};
  int n_used = 0;
  for (int j = 0; j < A.n_target_layers; ++j) {
    const int u = A.layer_map[j];
    if (u < -1 || u >= A.n_draft_layers) return 0;
    if (u >= 0 && !used[u]) {
      used[u] = true;
      ++n_used;
    }
  }
  return static_cast<long long>(n_used) * A.batch * A.n_groups;
}

// CTAs per list of the form that sums the rows itself.
int pick_cluster(long long L_stride, long long n_lists) {
  int cs = 1;
  while (cs < 8 && (L_stride + cs - 1) / cs > 8192) cs *= 2;
  while (cs < 8 && n_lists * cs < 296 && L_stride / cs > 2048) cs *= 2;
  while (cs < kMaxCluster && (L_stride + cs - 1) / cs > kSliceMax) cs *= 2;
  return cs;
}

// CTAs per list that lies in global memory as one row: slices that fit a CTA, and more of them while
// the GPU (two CTAs per SM) has room and the slices stay long enough to pay for the cluster's
// barriers and exchanges.
int pick_cluster_row(long long L_stride, long long n_lists) {
  int cs = 1;
  while (cs < kMaxCluster && (L_stride + cs - 1) / cs > kSliceMax) cs *= 2;
  while (cs < 8 && n_lists * cs * 2 <= 296 && (L_stride + cs - 1) / cs > 4096) cs *= 2;
  return cs;
}

// CTAs per streamed list: as many as leave every CTA an SM to itself (two on one share its atomics), in slices that
// pay for the exchanges.  131072 entries, uniform / Zipf, us, in one / two / four CTAs: 32 rows 64/57, 43/40, 35/32;
// 72 rows 64/57, 45/41, 65/59; 100 rows 65/57, 66/59, 66/59.  196608 entries in two / four: 32 rows 57/51, 39/37;
// 64 rows 59/53, 59/55; 128 rows 90/82, 102/93.
int pick_cluster_stream(long long L_stride, long long n_lists, int n_sm) {
  int cs = (L_stride > kStreamMax) ? 2 : 1;
  while (cs < 4 && n_lists * cs * 2 <= n_sm && L_stride / (2 * cs) >= kSliceMax) cs *= 2;
  return cs;
}

// Clusters of cs CTAs with a whole slice each that hold their rows on this device at once (GPCs do not hold a
// multiple of every cluster size: of 148 SMs, 66 clusters of four and 30 of eight).  Asked once per device and size.
int rows_at_once(const void* kernel, int dev, int cs) {
  static std::atomic<int> known[64][kMaxCluster + 1];  // + 1; 0 = not asked yet
  int n = known[dev][cs].load(std::memory_order_relaxed);
  if (n == 0) {
    cudaLaunchConfig_t q;
    memset(&q, 0, sizeof(q));
    q.gridDim = dim3(static_cast<unsigned>(cs), 1024, 1);
    q.blockDim = dim3(512, 1, 1);
    q.dynamicSmemBytes = kFixedBytes + kSliceMax * sizeof(float) + kScratchBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cs);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    q.attrs = attr;
    q.numAttrs = 1;
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, kernel, &q) != cudaSuccess) {
      cudaGetLastError();
      fit = 0;
    }
    n = fit + 1;
    known[dev][cs].store(n, std::memory_order_relaxed);
  }
  return n - 1;
}

// The two-launch form applies to the default selection over multi-row lists of >= 2048
// positions, and pays when one cluster per list would leave SMs without a CTA: a CTA streams
// ~35 GB/s, so the cluster kernel is bound by (bytes per list) / (8 x 35 GB/s) however few the
// lists, while the search launch adds ~13 us of its own.  Measured (us, cluster / two launches, lists of 48 rows):
// 4 x 4096 positions 23 / 20; 18 x 16384 27 / 30; 8 x 32768 36 / 28; 18 x 32768 42 / 42; 32 x 32768 59 / 58;
// 4 x 131072 97 / 42; 18 x 131072 188 / 101; 18 x 196608 218 / 144.  (Lists longer than 131072 take clusters of
// sixteen, since only those hold them; their SMs stream no faster, so they count like clusters of eight.)
bool two_launch_shape(const specattn_select_args& A) {
  const bool variant = (A.per_step && A.gamma > 1) || A.bisect_iters > 0 || A.chunk > 1;
  if (variant || static_cast<long long>(A.n_draft_heads) * A.gamma <= 1 || A.L_stride < 2048 || A.L_stride % 4 != 0)
    return false;
  const long long n_lists = count_lists(A);
  if (n_lists <= 0 || A.form == SPECATTN_SELECT_FORM_CLUSTER) return false;
  if (A.form == SPECATTN_SELECT_FORM_TWO_LAUNCH) return true;  // the caller knows its batch (ragged lengths)
  return n_lists * std::min(pick_cluster(A.L_stride, n_lists), 8) < 148;
}

}  // namespace
}  // namespace specattn

using specattn::SelectParams;

extern "C" size_t specattn_select_workspace_bytes(const specattn_select_args* args) {
  if (args == nullptr || args->struct_size != sizeof(specattn_select_args)) return 0;
  if (!specattn::two_launch_shape(*args)) return 0;
  return static_cast<size_t>(specattn::count_lists(*args)) * static_cast<size_t>(args->L_stride) * sizeof(float);
}

extern "C" int specattn_select_topp(const specattn_select_args* args, void* cuda_stream) {
  specattn::NvtxRange nvtx_range("specattn_select_topp");
  if (args == nullptr) return SPECATTN_ERR_NULL;
  if (args->struct_size != sizeof(specattn_select_args)) return SPECATTN_ERR_STRUCT_SIZE;
  const specattn_select_args& A = *args;
  if (!A.draft_probs || !A.kv_len || !A.layer_map || !A.idx || !A.counts || !A.row_status)
    return SPECATTN_ERR_NULL;
  if (A.n_draft_layers < 1 || A.n_draft_layers > SPECATTN_MAX_DRAFT_LAYERS) return SPECATTN_ERR_RANGE;
  if (A.n_target_layers < 0 || A.batch < 0 || A.gamma < 1 || A.n_groups < 1) return SPECATTN_ERR_RANGE;
  if (A.n_draft_heads < 1 || A.n_draft_heads > SPECATTN_MAX_DRAFT_HEADS) return SPECATTN_ERR_RANGE;
  if (A.L_stride < 0 || A.idx_stride < 0) return SPECATTN_ERR_RANGE;
  if (!(A.p > 0.0f)) return SPECATTN_ERR_RANGE;  // also rejects NaN
  if (A.bisect_iters < 0 || A.bisect_iters > 64 || (A.per_step != 0 && A.per_step != 1)) return SPECATTN_ERR_RANGE;
  if (A.form < 0 || A.form > SPECATTN_SELECT_FORM_TWO_LAUNCH) return SPECATTN_ERR_RANGE;
  if (A.chunk < 0 || A.chunk > 64 || (A.chunk > 1 && (A.chunk < 4 || (A.chunk & (A.chunk - 1)) != 0)))
    return SPECATTN_ERR_RANGE;  // 0 / 1 = per position, else a power of two in [4, 64]
  if (A.L_stride % 4 != 0) return SPECATTN_ERR_ALIGN;
  if (A.L_stride > SPECATTN_MAX_KV_LEN) return SPECATTN_ERR_UNSUPPORTED;
  if (static_cast<long long>(A.n_draft_heads) * A.gamma > SPECATTN_MAX_ROWS_PER_LIST)
    return SPECATTN_ERR_UNSUPPORTED;

  SelectParams P;
  memset(&P, 0, sizeof(P));
  bool used[SPECATTN_MAX_DRAFT_LAYERS] = {false};
  for (int j = 0; j < A.n_target_layers; ++j) {
    const int u = A.layer_map[j];
    if (u < -1 || u >= A.n_draft_layers) return SPECATTN_ERR_RANGE;
    if (u >= 0) used[u] = true;
  }
  int n_used = 0;
  for (int u = 0; u < A.n_draft_layers; ++u) {
    if (!used[u]) continue;
    if (A.draft_probs[u] == nullptr) return SPECATTN_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(A.draft_probs[u]) % 16 != 0) return SPECATTN_ERR_ALIGN;
    P.probs[n_used] = A.draft_probs[u];
    P.layer_of[n_used] = u;
    ++n_used;
  }
  if (A.head_group != nullptr) {
    for (int h = 0; h < A.n_draft_heads; ++h) {
      if (A.head_group[h] < 0 || A.head_group[h] >= A.n_groups) return SPECATTN_ERR_RANGE;
      if (A.head_group[h] > 127) return SPECATTN_ERR_UNSUPPORTED;
      P.head_group[h] = static_cast<signed char>(A.head_group[h]);
    }
    P.has_groups = 1;
  }
  const long long n_lists = static_cast<long long>(n_used) * A.batch * A.n_groups;
  if (n_lists == 0) return SPECATTN_OK;
  if (n_lists > 65535) return SPECATTN_ERR_UNSUPPORTED;

  P.n_used = n_used;
  P.B = A.batch;
  P.H = A.n_draft_heads;
  P.gamma = A.gamma;
  P.G = A.n_groups;
  P.L_stride = A.L_stride;
  P.kv_len = A.kv_len;
  P.p = A.p;
  P.keep_all = (A.p >= 1.0f) ? 1 : 0;
  P.idx = A.idx;
  P.idx_stride = A.idx_stride;
  P.counts = A.counts;
  P.status = A.row_status;
  P.diag = A.diag;

  // two-launch form: the rows are summed into the workspace first and the search reads that sum like
  // a single-row list
  const bool two_launch = A.workspace != nullptr && specattn::two_launch_shape(A) &&
                          A.workspace_bytes >= static_cast<uint64_t>(n_lists) * A.L_stride * sizeof(float);
  if (two_launch) {
    if (reinterpret_cast<uintptr_t>(A.workspace) % 16 != 0) return SPECATTN_ERR_ALIGN;
    P.agg = static_cast<const float*>(A.workspace);
  }
  P.per_step = (A.per_step && A.gamma > 1) ? 1 : 0;  // with one query the union is the single nucleus
  P.bisect_iters = A.bisect_iters;
  P.chunk = (A.chunk > 1) ? A.chunk : 1;
  const bool variant = P.per_step || P.bisect_iters > 0 || P.chunk > 1;
  // the row is searched where it lies only if it is every group's: a group that the head does not feed has a row of
  // zeros
  const bool one_row = static_cast<long long>(A.n_draft_heads) * A.gamma == 1 && P.chunk == 1 && (!P.has_groups || A.n_groups == 1);
  const bool agg = !two_launch && !one_row;  // the CTAs sum the rows (or the chunks) themselves
  const void* const kernels[9] = {
      (const void*)specattn::select_topp_kernel<false, false, 128>, (const void*)specattn::select_topp_kernel<false, false, 512>,
      (const void*)specattn::select_topp_kernel<false, true, 512>, (const void*)specattn::select_topp_kernel<true, false, 256>,
      (const void*)specattn::select_topp_kernel<true, true, 256>, (const void*)specattn::stream_rows_kernel<false, false>,
      (const void*)specattn::stream_rows_kernel<true, false>, (const void*)specattn::stream_rows_kernel<false, true>,
      (const void*)specattn::stream_rows_kernel<true, true>};
  // Opt in to large dynamic shared memory and clusters of 16 once per device, so that later calls
  // issue nothing but the launch.
  int dev = 0;
  const int n_sm = specattn::device_sm_count();
  if (n_sm <= 0 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return SPECATTN_ERR_CUDA;
  }
  {
    static std::atomic<unsigned long long> done_mask{0};
    if (!((done_mask.load(std::memory_order_acquire) >> dev) & 1ull)) {
      for (const void* fn : kernels) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
          cudaGetLastError();
          return SPECATTN_ERR_CUDA;
        }
      }
      done_mask.fetch_or(1ull << dev, std::memory_order_release);
    }
  }
  // Rows are streamed (stream_rows.cuh) where clusters that hold them would need more than one wave (uniform / Zipf,
  // us, held / streamed: 40 rows of 98304 entries 45/39, 39/35; 72 of 65536 45/39, 31/30; 64 of 131072 62/47, 45/41;
  // 16 of 196608 51/39, 39/37 -- but 12 of them 33/27, 39/36), or where there is about a row for every SM and a
  // cluster's exchanges gain nothing (100 rows of 8192: 18/18, 18/18; of 32768 29/29, 28/25; of 65536 45/41, 41/37).
  const int row_cs = specattn::pick_cluster_row(A.L_stride, n_lists);
  const bool stream = !agg && !variant && A.L_stride > 4096 &&
                      (n_lists > specattn::rows_at_once(kernels[1], dev, row_cs) || (2 * n_lists > n_sm && n_lists <= n_sm));
  const bool small = !agg && !variant && A.L_stride <= 2048;
  const int cs = stream ? specattn::pick_cluster_stream(A.L_stride, n_lists, n_sm) : agg ? specattn::pick_cluster(A.L_stride, n_lists) : row_cs;
  const int slice = specattn::slice_of(static_cast<int>(A.L_stride), cs, (P.chunk > 4) ? P.chunk : 4);
  const int nt = small ? 128 : agg ? 256 : 512;
  if (slice > specattn::kSliceMax && !stream) return SPECATTN_ERR_UNSUPPORTED;
  // searches apart: the scores of all queries are kept, and one query's scores fit a CTA's slice
  const long long n_scores = (A.L_stride + P.chunk - 1) / P.chunk;
  const size_t score_bytes = static_cast<size_t>(A.gamma) * (slice / P.chunk) * sizeof(float);
  P.apart = (agg && P.per_step && P.chunk > 1 && A.gamma <= specattn::kMaxApart && n_scores <= specattn::kSliceMax &&
             specattn::slice_room(static_cast<int>(n_scores), nt) <= specattn::slice_room(slice, nt) && score_bytes <= 48 * 1024)
                ? 1
                : 0;
  const size_t apart_bytes = P.apart ? score_bytes : 0;
  const size_t smem = stream ? sizeof(specattn::StreamShared) : specattn::kFixedBytes + (agg ? specattn::kHeadBytes : 0) +
                      static_cast<size_t>(specattn::slice_room(slice, nt)) * sizeof(float) +
                      (agg ? specattn::kRingBytes : specattn::kScratchBytes) +
                      // the union's bit mask: one bit per entry of the slice
                      (P.per_step ? static_cast<size_t>(specattn::slice_room(slice, nt) / 8) : 0) + apart_bytes;
  const int kidx = stream ? 5 + (A.diag != nullptr ? 1 : 0) + (cs > 1 ? 2 : 0) : agg ? (variant ? 4 : 3) : (variant ? 2 : (small ? 0 : 1));
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = (stream && cs == 1) ? dim3(static_cast<unsigned>(n_lists), 1, 1) : dim3(static_cast<unsigned>(cs), static_cast<unsigned>(n_lists), 1);
  cfg.blockDim = dim3(static_cast<unsigned>(nt), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = static_cast<cudaStream_t>(cuda_stream);
  cudaLaunchAttribute attr[2];
  // the kernel may be scheduled while its predecessor drains; it waits before it reads or writes
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(cs);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = agg ? attr + 1 : attr;
  cfg.numAttrs = agg ? 1 : 2;
  if (two_launch) {
    const dim3 grid(static_cast<unsigned>((A.L_stride + specattn::kAggPositions - 1) / specattn::kAggPositions),
                    static_cast<unsigned>(n_lists), 1);
    specattn::aggregate_rows_kernel<<<grid, specattn::kAggThreads, 0, cfg.stream>>>(P, static_cast<float*>(A.workspace));
    if (cudaGetLastError() != cudaSuccess) return SPECATTN_ERR_CUDA;
    specattn::g_launch_count.fetch_add(1, std::memory_order_relaxed);
  }
  // Few clusters: ask for more shared memory than needed, so that an SM takes fewer CTAs and the
  // clusters spread over the GPU instead of filling every slot of a few SMs (co-resident CTAs
  // slow one another's passes) -- but only as far as all clusters still run at once (clusters are
  // placed GPC by GPC; 16 clusters of 8 do not fit at one CTA per SM, and a second wave costs far
  // more).  The limits are asked of the runtime once per kernel and cluster size and cached.
  {
    static const size_t pads[3] = {120 * 1024, 100 * 1024, 70 * 1024};
    static std::atomic<int> fit[64][5][5][3];  // [device][kernel, none of the streaming ones][log2 cs][pad]: clusters + 1, 0 = unknown
    int lcs = 0;
    while ((1 << lcs) < cs) ++lcs;
    for (int k = 0; k < 3 && !stream; ++k) {
      if (pads[k] <= smem) break;
      int known = fit[dev][kidx][lcs][k].load(std::memory_order_relaxed);
      if (known == 0) {
        cudaLaunchConfig_t q = cfg;
        q.dynamicSmemBytes = pads[k];
        q.gridDim = dim3(static_cast<unsigned>(cs), 1024, 1);
        q.attrs = attr + 1;
        q.numAttrs = 1;
        int n_fit = 0;
        if (cudaOccupancyMaxActiveClusters(&n_fit, kernels[kidx], &q) != cudaSuccess) {
          cudaGetLastError();
          n_fit = 0;
        }
        known = n_fit + 1;
        fit[dev][kidx][lcs][k].store(known, std::memory_order_relaxed);
      }
      if (known - 1 >= n_lists) {
        cfg.dynamicSmemBytes = pads[k];
        break;
      }
    }
  }
  void* params[1] = {&P};
  if (cudaLaunchKernelExC(&cfg, kernels[kidx], params) != cudaSuccess) {
    cudaGetLastError();
    return SPECATTN_ERR_CUDA;
  }
  specattn::g_launch_count.fetch_add(1, std::memory_order_relaxed);
  return SPECATTN_OK;
}
