// sparse_verify on warp-level tensor cores in CTAs of half an SM, a warp computing all of its query rows (up to 24) --
// included by sparse_verify.cu inside namespace specattn::{anonymous}; uses VerifyParams and the work partition there,
// gives the same operation.
//
// For calls with more units than half of the SMs (many_units).  In CTAs that take an SM whole, 128 units leave 20 SMs
// idle and 256 do not fit one each, so that every CTA walks through two or three of them, its tensor cores idle at every
// end.  Two CTAs to an SM take units of any number in halves of that size, and one's set-up, end and merge run under
// the other's tiles.  For that a CTA has half of the registers, four consumer and four producer warps, which is
// enough for the whole query block where
//   - a consumer warp takes all query rows of every fourth 16-key tile: K and V fragments are read from shared memory
//     once, not once per 16-row slab;
//   - the output is accumulated transposed,
//       S[16 rows x 16 keys] = Q K^T per slab,      O^T[128 dims x 8 rows] += V^T P^T per 8 rows,
//     where the accumulators of S are the B fragments of P^T as they lie, and the query rows are padded to eight instead
//     of sixteen in the larger product: 80 MMAs per 16 keys at 20 rows instead of 96.
// (20 rows, us, whole / half: 128 units x 2053 tokens, a call by itself, 43.3 / 36.4; 80 x 400 11.5 / 11.0; 256 x 400 26.1 / 15.4, x
// 2000 65.6 / 49.2, 512 x 400 45.7 / 37.3; the rule and its limits: half_sm.  Not for more rows: 28, 128 x 400 13.0 / 14.7; the same warps in
// whole-SM CTAs, 40 rows, 128 x 400 14.6 / 13.1, but 256 x 60 15.2 / 18.1, and 160 x 315 at 56 rows 30.4 / 36.4, since
// an end of a unit costs more.  Nor for few units, which get more parts each: 24 rows, 64 x 1228 16.4 / 19.1.)
#pragma once

namespace rows {

constexpr int kTile = 16;         // tokens per tile = one atom
constexpr int kSlots = 8;
constexpr int kConsWarps = 4, kProdWarps = 4;   // (the slots are a multiple of both: a slot is always filled and read by the same warp)
constexpr int kThreads = (kConsWarps + kProdWarps) * 32;
constexpr float kRaise = 8.f;     // the reference maximum of a row is raised when a score exceeds it by 2^8

// NT8: blocks of eight query rows.
template <int NT8>
struct VShared {
  static constexpr int kRows = 8 * NT8;
  static constexpr int kItems = 2 * NT8;            // 16 x 8 blocks of the output that a warp owns after the combine
  alignas(128) unsigned char kv[kSlots][2][kTile * kPitch];
  alignas(16) unsigned char q[2][kRows * kPitch];   // of this segment and of the next
  alignas(16) float4 scratch[kConsWarps][2 * NT8][32];
  alignas(16) float2 stat[kConsWarps][kRows];      // (maximum, sum) of every row, per warp ...
  alignas(16) float2 sum[kRows];              // ... and over the CTA (read by the cluster)
  int row_off[kRows];                         // output row of a query row inside (sequence, kv head)
  alignas(8) unsigned long long full[kSlots];
  unsigned long long empty[kSlots];
  unsigned long long q_full[2], q_empty[2];
  int unit_start[kMaxUnits + 1];
  int unit_cnt[kMaxUnits];
  Partition part;
  volatile int abort_flag;
};
template <int NT8>
constexpr size_t verify_smem() {
  static_assert(2 * (sizeof(VShared<NT8>) + 128 + 1024) <= 228 * 1024, "two CTAs per SM");
  return sizeof(VShared<NT8>) + 128;
}

// Floats of one CTA's record of a unit: per warp its blocks of the output and (maximum, sum) of its rows.
template <int NT8>
__host__ __device__ constexpr int record_floats() { return kConsWarps * (VShared<NT8>::kItems * 128 + 16 * NT8); }

// Softmax state of a warp: O^T as 16-dim x 8-row blocks; m, l of row 8 nt + lane / 4.
template <int NT8>
struct RowState {
  float acc[8][NT8][4];
  float m[NT8], l[NT8];
};

// A value per row (lane / 4 of block nt) as the two rows 2 tq, 2 tq + 1 that a lane's accumulators belong to.
__device__ __forceinline__ float2 row_to_col(float v, int tq) {
  return make_float2(__shfl_sync(0xffffffffu, v, 8 * tq), __shfl_sync(0xffffffffu, v, 8 * tq + 4));
}

// Fragments of 16 query dims: the slabs of a warp's rows.  (Half a slab: rows 8 - 15 of the fragment are zero.)
template <int NT8>
__device__ __forceinline__ void load_q(uint32_t (*f)[4], uint32_t q_addr, uint32_t q_half, int kk) {
#pragma unroll
  for (int i = 0; i < (NT8 + 1) / 2; ++i) {
    if (2 * i + 1 < NT8) {
      ldmatrix_x4(f[i], q_addr + i * 16 * kPitch + kk * 32);
    } else {
      ldmatrix_x2(f[i][0], f[i][2], q_half + i * 16 * kPitch + kk * 32);
      f[i][1] = f[i][3] = 0u;
    }
  }
}

// One tile of 16 keys.  `valid`: existing keys (rows beyond hold finite padding); `tail_begin`: index in the tile
// of the first in-flight token (>= 16: none), of which row r may see the first row_lim(r) + 1 only.
template <int NT8, class RowLim>
__device__ __forceinline__ void attend_tile(RowState<NT8>& st, uint32_t q_addr, uint32_t q_half, uint32_t k_addr, uint32_t v_addr,
                                            uint32_t turn, int valid, float scale_log2, int tq, int tail_begin, RowLim row_lim) {
  constexpr int SL = (NT8 + 1) / 2;
  float s[SL][2][4];
#pragma unroll
  for (int i = 0; i < SL; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) s[i][j][0] = s[i][j][1] = s[i][j][2] = s[i][j][3] = 0.f;
  // (fragments are loaded one step ahead of the products that use them)
  uint32_t k4[2][4], qa[2][SL][4];
  ldmatrix_x4(k4[0], k_addr);
  load_q<NT8>(qa[0], q_addr, q_half, 0);
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    if (kk < 7) {
      ldmatrix_x4(k4[(kk + 1) & 1], k_addr + (kk + 1) * 32);
      load_q<NT8>(qa[(kk + 1) & 1], q_addr, q_half, kk + 1);
    }
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      mma_bf16(s[i][0], qa[kk & 1][i], k4[kk & 1][0], k4[kk & 1][1]);
      mma_bf16(s[i][1], qa[kk & 1][i], k4[kk & 1][2], k4[kk & 1][3]);
    }
  }
  auto v_of = [&](int i) { return v_addr + ((32u * i) ^ turn); };   // block i of the output
  uint32_t v4[3][4];
  ldmatrix_x4_trans(v4[0], v_of(0));
  if (valid < kTile || tail_begin < kTile) {  // a unit's last tiles
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      const int lim = tail_begin + row_lim(nt);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int key = j * 8 + tq * 2 + i;
          if (key >= valid || (key >= tail_begin && key > lim)) s[nt >> 1][j][2 * (nt & 1) + i] = -INFINITY;
        }
    }
  }
  // The reference maximum is raised lazily: against one that is too low by less than 2^8 the weights are as
  // precise (both of their bf16 terms are floating point), and most tiles need neither shuffles nor a rescale.
  // (running maxima are kept in the scaled log2 domain: scale_log2 > 0 keeps the order)
  float mx[NT8];
  bool raise = false;
#pragma unroll
  for (int nt = 0; nt < NT8; ++nt) {
    const float(&a)[4] = s[nt >> 1][0];
    const float(&b)[4] = s[nt >> 1][1];
    const int h = 2 * (nt & 1);
    mx[nt] = fmaxf(fmaxf(a[h], a[h + 1]), fmaxf(b[h], b[h + 1])) * scale_log2;
    raise |= mx[nt] > st.m[nt] + kRaise;
  }
  if (__any_sync(0xffffffffu, raise)) {
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      float v = mx[nt];
      v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
      v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
      const float mn = fmaxf(st.m[nt], v);
      const float al = ex2(st.m[nt] - ((mn == -INFINITY) ? 0.f : mn));
      st.m[nt] = mn;
      st.l[nt] *= al;
      const float2 c = row_to_col(al, tq);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        st.acc[i][nt][0] *= c.x;
        st.acc[i][nt][1] *= c.y;
        st.acc[i][nt][2] *= c.x;
        st.acc[i][nt][3] *= c.y;
      }
    }
  }
  // P as a bf16 pair (hi, lo): the residuals are exact in fp32 and rounded once more.  Raw scores stay unscaled:
  // exp2(s c - m c) is one fused multiply-add per element.
  uint32_t phi[NT8][2], plo[NT8][2];
#pragma unroll
  for (int nt = 0; nt < NT8; ++nt) {
    const float base = (st.m[nt] == -INFINITY) ? 0.f : st.m[nt];
    float sum[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float x = ex2(fmaf(s[nt >> 1][j][2 * (nt & 1)], scale_log2, -base));
      const float y = ex2(fmaf(s[nt >> 1][j][2 * (nt & 1) + 1], scale_log2, -base));
      sum[j] = x + y;
      const uint32_t h = pack_bf16(x, y);
      phi[nt][j] = h;
      plo[nt][j] = pack_bf16(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xffff0000u));
    }
    st.l[nt] += sum[0] + sum[1];
  }
  // (the small terms of a block follow the large ones of the next: they wait for the same accumulators)
#pragma unroll
  for (int i = 0; i <= 8; ++i) {
    if (i < 7) ldmatrix_x4_trans(v4[(i + 1) % 3], v_of(i + 1));
    if (i < 8) {
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) mma_bf16(st.acc[i][nt], v4[i % 3], phi[nt][0], phi[nt][1]);
    }
    if (i > 0) {
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) mma_bf16(st.acc[i - 1][nt], v4[(i + 2) % 3], plo[nt][0], plo[nt][1]);
    }
  }
}

// Output blocks of a warp.  Item k: dims 16 (2 warp + k / NT8) ..., rows 8 (k % NT8) ...
template <int NT8>
struct Items {
  const VerifyParams& P;
  const int* row_off;
  long long row0;    // output row of (sequence, query 0, kv head)
  int warp, lane;
  __device__ __forceinline__ void store(int k, float4 v) const {
    const int g = lane >> 2, tq = lane & 3;
    const int r = 8 * (k % NT8) + 2 * tq;
    float* const o = P.out + row0 * kD + 16 * (2 * warp + k / NT8) + g;
    if (r < P.M) {
      float* const p = o + static_cast<long long>(row_off[r]) * kD;
      p[0] = v.x;
      p[8] = v.z;
    }
    if (r + 1 < P.M) {
      float* const p = o + static_cast<long long>(row_off[r + 1]) * kD;
      p[0] = v.y;
      p[8] = v.w;
    }
  }
};
__device__ __forceinline__ float lse_of(float m, float l) { return (l > 0.f) ? (m + log2f(l)) * kLn2 : -INFINITY; }

// Merge of a unit whose parts lie in one cluster: every CTA has left its blocks (rec_addr) and its rows' (maximum, sum)
// (sum_addr) in its shared memory, at the same addresses, and arrived at the cluster barrier; CTA `part` of kParts
// combines its share of the blocks from all of them, in part order, and writes it (part 0 also writes the
// LSE).  Reading is spread over all CTAs and nobody waits for more than that barrier.  (Pushing the blocks to their
// writers instead, with one remote arrival each, took 1.5 - 2.7 us longer.)  Out of line: it costs the tile loop no
// registers.  kParts is a template parameter for the sake of straight, short code.
template <int NT8, int kParts>
__device__ __noinline__ void merge_cluster(const VerifyParams& P, const int* row_off, uint32_t rec_addr, uint32_t sum_addr,
                                           int part, int u) {
  constexpr int kItems = VShared<NT8>::kItems;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tq = lane & 3;
  const uint32_t rank0 = cluster_cta_rank() - static_cast<uint32_t>(part);
  const int b = u / P.Hkv, kvh = u - b * P.Hkv;
  const Items<NT8> items{P, row_off, static_cast<long long>(b) * P.T * P.Hq + kvh * P.grp, warp, lane};
  const uint32_t mine = rec_addr + warp * kItems * 512 + lane * 16;
  const uint32_t rows = sum_addr + 2 * tq * 8;
  // (every load of the warp in flight at once: item by item, three round trips of 0.7 us each)
  constexpr int kMost = (kItems + kParts - 1) / kParts;
  const int k0 = (part + warp) % kParts;
  float4 ml[kMost][kParts], x[kMost][kParts];
  cluster_wait();
#pragma unroll
  for (int j = 0; j < kMost; ++j) {
    const int k = min(k0 + j * kParts, kItems - 1);
#pragma unroll
    for (int r = 0; r < kParts; ++r) {
      ml[j][r] = ld_cluster_v4(map_to_cta(rows + 64 * (k % NT8), rank0 + r));
      x[j][r] = ld_cluster_v4(map_to_cta(mine + 512 * k, rank0 + r));
    }
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kMost; ++j) {
    const int k = k0 + j * kParts;
    if (k >= kItems) break;
    float m0 = ml[j][0].x, m1 = ml[j][0].z;
#pragma unroll
    for (int r = 1; r < kParts; ++r) {
      m0 = fmaxf(m0, ml[j][r].x);
      m1 = fmaxf(m1, ml[j][r].z);
    }
    const float base0 = (m0 == -INFINITY) ? 0.f : m0, base1 = (m1 == -INFINITY) ? 0.f : m1;
    float l0 = 0.f, l1 = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < kParts; ++r) {
      const float a0 = ex2(ml[j][r].x - base0), a1 = ex2(ml[j][r].z - base1);
      l0 += ml[j][r].y * a0;
      l1 += ml[j][r].w * a1;
      o.x += x[j][r].x * a0;
      o.y += x[j][r].y * a1;
      o.z += x[j][r].z * a0;
      o.w += x[j][r].w * a1;
    }
    const float inv0 = (l0 > 0.f) ? 1.f / l0 : 0.f, inv1 = (l1 > 0.f) ? 1.f / l1 : 0.f;
    items.store(k, make_float4(o.x * inv0, o.y * inv1, o.z * inv0, o.w * inv1));
    if (k < NT8 && warp == 0 && lane < 4) {  // (each block of rows is item k < NT8 of one CTA: it writes the LSE)
      const int r = 8 * k + 2 * tq;
      if (r < P.M) P.lse[items.row0 + row_off[r]] = lse_of(m0, l0);
      if (r + 1 < P.M) P.lse[items.row0 + row_off[r + 1]] = lse_of(m1, l1);
    }
  }
  __syncwarp();
  cluster_arrive();  // (only reads precede it)
  cluster_wait();    // nobody leaves while its records may still be read
}

// Merge of a unit cut across CTAs i_lo ... i_hi by the warp that arrived last of those with its index: its blocks
// from all records, in CTA order (the own one included, read back from memory, so that the result does not depend
// on who arrived last).  rec(i): the warp's record of CTA i.
template <int NT8, class Rec>
__device__ __forceinline__ void merge_global(const Items<NT8>& items, int i_lo, int i_hi, Rec rec) {
  constexpr int kItems = VShared<NT8>::kItems, kHalf = NT8;   // blocks per pass over the records
  const VerifyParams& P = items.P;
  const int lane = items.lane, g = lane >> 2, tq = lane & 3;
  float m[NT8], l[NT8];
#pragma unroll
  for (int nt = 0; nt < NT8; ++nt) m[nt] = -INFINITY, l[nt] = 0.f;
  auto rows = [&](int i) { return reinterpret_cast<const float2*>(rec(i) + kItems * 32) + g; };
  for (int i = i_lo; i <= i_hi; i += 4) {   // four records' rows per round trip
    float2 ml[4][NT8];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) ml[j][nt] = __ldcg(rows(min(i + j, i_hi)) + 8 * nt);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) m[nt] = fmaxf(m[nt], ml[j][nt].x);
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    float4 o[kHalf];
#pragma unroll
    for (int k = 0; k < kHalf; ++k) o[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = i_lo; i <= i_hi; i += 2) {   // two records' blocks per round trip
      const bool two = i + 1 <= i_hi;
      const float4* const ra = rec(i);
      const float4* const rb = rec(two ? i + 1 : i);
      float2 mla[NT8], mlb[NT8];
      float4 xa[kHalf], xb[kHalf];
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) {
        mla[nt] = __ldcg(rows(i) + 8 * nt);
        mlb[nt] = __ldcg(rows(two ? i + 1 : i) + 8 * nt);
      }
#pragma unroll
      for (int k = 0; k < kHalf; ++k) {
        xa[k] = __ldcg(ra + (half * kHalf + k) * 32 + lane);
        xb[k] = __ldcg(rb + (half * kHalf + k) * 32 + lane);
      }
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) {
        const float base = (m[nt] == -INFINITY) ? 0.f : m[nt];
        const float wa = ex2(mla[nt].x - base), wb = two ? ex2(mlb[nt].x - base) : 0.f;
        if (half == 0) {
          l[nt] += mla[nt].y * wa;
          if (two) l[nt] += mlb[nt].y * wb;
        }
        const float2 ca = row_to_col(wa, tq), cb = row_to_col(wb, tq);
#pragma unroll
        for (int k = 0; k < kHalf; ++k) {
          if ((half * kHalf + k) % NT8 != nt) continue;
          o[k].x += xa[k].x * ca.x;
          o[k].y += xa[k].y * ca.y;
          o[k].z += xa[k].z * ca.x;
          o[k].w += xa[k].w * ca.y;
          if (two) {
            o[k].x += xb[k].x * cb.x;
            o[k].y += xb[k].y * cb.y;
            o[k].z += xb[k].z * cb.x;
            o[k].w += xb[k].w * cb.y;
          }
        }
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      const float2 inv = row_to_col((l[nt] > 0.f) ? 1.f / l[nt] : 0.f, tq);
#pragma unroll
      for (int k = 0; k < kHalf; ++k) {
        if ((half * kHalf + k) % NT8 != nt) continue;
        items.store(half * kHalf + k, make_float4(o[k].x * inv.x, o[k].y * inv.y, o[k].z * inv.x, o[k].w * inv.y));
      }
    }
  }
  if (items.warp == 0 && tq == 0) {
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      const int r = 8 * nt + g;
      if (r < P.M) P.lse[items.row0 + items.row_off[r]] = lse_of(m[nt], l[nt]);
    }
  }
}

template <int NT8>
__global__ void __launch_bounds__(kThreads, 2) sparse_verify_rows_kernel(const __grid_constant__ VerifyParams P) {
  using Sh = VShared<NT8>;
  constexpr int kItems = Sh::kItems;
  // Registers: a CTA is launched with 128 a thread; the producer warps hand theirs to the consumers (two warpgroups of
  // 128 threads: 168 + 88 = 152 + 104 = 2 x 128).  With 88 the producers spill, which up to 16 rows need not be.
  constexpr int kConsRegs = (NT8 == 2) ? 152 : 168, kProdRegs = 256 - kConsRegs;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Sh& sh = *reinterpret_cast<Sh*>(smem_raw);
  int* const unit_start = sh.unit_start;
  int* const unit_cnt = sh.unit_cnt;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int U = P.B * P.Hkv;

  // units with an empty list: out = 0, lse = -inf (the first global writes: the previous kernel's results, and its
  // use of the shared workspace, are complete then)
  auto empty_unit = [&](int u, int first, int step) {
    const int b = u / P.Hkv, kvh = u % P.Hkv;
    for (int e = first; e < P.M * kD; e += step) {
      const int r = e / kD, t = r / P.grp, h = kvh * P.grp + r % P.grp;
      P.out[((static_cast<long long>(b) * P.T + t) * P.Hq + h) * kD + e % kD] = 0.f;
      if (e % kD == 0) P.lse[(static_cast<long long>(b) * P.T + t) * P.Hq + h] = -INFINITY;
    }
  };
  // ---- set-up: barriers, zero padding rows of the query tile, unit prefix ---------------------
  {
    uint4* zq = reinterpret_cast<uint4*>(sh.q);
    for (int i = tid; i < static_cast<int>(sizeof(sh.q) / 16); i += kThreads) zq[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&sh.full[s], 32);  // deferred arrivals per producer lane
      mbar_init(&sh.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.q_full[i], 1);
      mbar_init(&sh.q_empty[i], kConsWarps);
    }
    mbar_fence_init();
    sh.abort_flag = 0;
    unit_start[0] = 0;
  }
  if (tid < Sh::kRows) sh.row_off[tid] = (tid / P.grp) * P.Hq + tid % P.grp;
  // Unless the caller vouched for the lists, nothing is read before the previous kernel is
  // done.  Only then may the next kernel of the stream be scheduled: a successor that starts
  // early therefore never overtakes the producer of the lists.
  if (!P.lists_stable) pdl_wait();
  pdl_launch_dependents();
  // A plan made for this launch (same units, grid, tail, dense flag) replaces the whole
  // partition below by one coalesced copy.
  const int* const plan = P.plan;
  const bool planned = plan != nullptr && plan[0] == kPlanMagic && plan[1] == U &&
                       plan[2] == static_cast<int>(gridDim.x) && (plan[3] >> 8) == P.cluster && plan[6] == P.tail &&
                       plan[7] == P.dense;
  int2 range = make_int2(0, 0), what = make_int2(0, 0);   // of this CTA, loaded together with the units
  int2 sizes = make_int2(0, 0);
  if (planned) {
    const int* const p_us = plan + kPlanHeader;
    const int* const p_cnt = p_us + (U + 1);
    const int2* const mine = reinterpret_cast<const int2*>(p_us + 2 * (U + 1) + 4 * blockIdx.x);
    range = mine[0];
    what = mine[1];
    sizes = *reinterpret_cast<const int2*>(plan + 4);
    for (int u = tid; u <= U; u += kThreads) {
      unit_start[u] = p_us[u];
      if (u < U) unit_cnt[u] = p_cnt[u];
    }
  } else {
    for (int u = tid; u < U; u += kThreads) {
      const int c = unit_count(P, u);
      unit_cnt[u] = c;
      unit_start[u + 1] = (c + kAtom - 1) / kAtom;
    }
  }
  fence_proxy_async();
  __syncthreads();
  // (every warp leaves itself the same values)
  if (!planned) {
    if (NT8 == 3) cut_units_inline<Sh, kThreads, true>(U, P.M, P.cluster);
    else cut_units<Sh, kThreads, true>(U, P.M, P.cluster);
  } else if (lane == 0) {
    sh.part.mine[0] = what.x;
    sh.part.mine[1] = part_of(what.y);
    sh.part.mine[2] = parts_of(what.y);
    sh.part.range[0] = range.x;
    sh.part.range[1] = range.y;
    sh.part.atoms = sizes.y;
    sh.part.ctas = sizes.x;
    sh.part.cluster = plan[3] & 0xff;
    sh.part.aligned = sh.part.cluster != 0;
  }
  __syncwarp();
  if (static_cast<int>(blockIdx.x) >= sh.part.ctas) {
    if (P.lists_stable) pdl_wait();
    for (int u = blockIdx.x; u < U; u += gridDim.x)
      if (unit_cnt[u] == 0) empty_unit(u, tid, kThreads);
    return;
  }

  if (warp >= kConsWarps) {
    // =========================== producer warps ===========================================
    set_max_registers_dec<kProdRegs>();
    const int pw = warp - kConsWarps;
    const int a0 = sh.part.range[0], a1 = sh.part.range[1], u_first = sh.part.mine[0];  // this CTA's atoms and the unit of the first
    const long long v_delta = P.s_kv * 2;
    int it0 = 0, seg = 0;
    int last_it = -1, q_seg = 0;   // the last tile, the last segment whose queries this warp sent for
    int a = a0, u = u_first;
    bool dead = false;
    while (a < a1 && !dead) {
      const int us = unit_start[u], ue = unit_start[u + 1];
      const int seg_hi = min(a1, ue);
      const int b = u / P.Hkv, kvh = u % P.Hkv;
      const int tiles = seg_hi - a;
      const int tok_lo = (a - us) * kAtom;
      const int tok_last = min(unit_cnt[u], (seg_hi - us) * kAtom) - 1;
      const int kvlen_b = P.kv_len[b];
      const int c_list = unit_cnt[u] - P.tail;
      const int* const list = P.dense ? nullptr
                                      : P.idx + (static_cast<long long>(b) * P.G + ((P.G == 1) ? 0 : kvh)) * P.idx_stride;
      // 16 lanes move one 256-byte row with 16-byte cp.async copies: a warp instruction fetches two rows (four
      // full 128-byte lines)
      // The query block of a unit (M rows of 256 bytes) is fetched by producer warp 0, walking the segments in order, while
      // the consumers still work on the one before it (one buffer for all segments kept this warp's tiles of the next
      // unit waiting until they were done).  The first one is fetched by the consumers themselves (see there);
      // only the barrier's phase is completed here, so that later segments find the parity they expect.
      if (pw == 0) {
        if (seg == 0) {
          if (lane == 0) mbar_arrive(&sh.q_full[0]);
        } else {
          // (The second buffer is free from the start: nothing but this wait puts its first block behind the previous
          // launch, which may have written the queries.  The first segment's K/V copies are out by now.)
          if (seg == 1 && P.lists_stable) pdl_wait();
          if (!mbar_wait(&sh.q_empty[seg & 1], ((seg >> 1) & 1u) ^ 1u, &sh.abort_flag)) { sh.abort_flag = 1; dead = true; break; }
          if (lane == 0) mbar_arrive_expect_tx(&sh.q_full[seg & 1], static_cast<uint32_t>(P.M) * kRowBytes);
          __syncwarp();
          for (int r = lane; r < P.M; r += 32)
            bulk_g2s(sh.q[seg & 1] + r * kPitch,
                     P.q + (static_cast<long long>(b) * P.T * P.Hq + kvh * P.grp + sh.row_off[r]) * kD, kRowBytes, &sh.q_full[seg & 1]);
          q_seg = seg;
        }
      }
      // Lanes 0 - 15 resolve the tokens of this warp's tile, lanes 16 - 31 those of its next one (four tiles on), to
      // the byte offset of their K row: list -> position -> block table -> page, two dependent loads, in steps so that
      // the chain stays ahead (offsets of the next two pairs of tiles, positions of the third): no load is waited for
      // between two tiles.
      auto load_pos = [&](int t) -> int {
        // token index inside the unit: the list first, then the tail.  The tail of a segment is padded to a whole tile
        // with copies of its last token, so that every row a consumer multiplies by a zero weight holds finite data.
        const int k = min(tok_lo + (t + 4 * (lane >> 4)) * kTile + (lane & 15), tok_last);
        return (k >= c_list) ? (kvlen_b + (k - c_list)) : (P.dense ? k : __ldg(list + k));
      };
      bool bad = false;
      auto offs_of = [&](int pos) -> long long {
        if (pos < 0 || pos >= kvlen_b + P.tail) { bad = true; pos = 0; }
        int lp = (P.page_shift >= 0) ? (pos >> P.page_shift) : (pos / P.page_size);
        // a position beyond the sequence's row of the block table (kv_len larger than the
        // table covers) is a bad index like any other: it reads position 0 instead
        if (lp >= P.bt_stride) { bad = true; pos = 0; lp = 0; }
        const int slot = pos - lp * P.page_size;
        long long page = P.bt ? static_cast<long long>(__ldg(P.bt + b * P.bt_stride + lp))
                              : (b * P.bt_stride + lp);
        if (page < 0 || (P.n_pages > 0 && page >= P.n_pages)) { bad = true; page = 0; }
        return (page * P.s_page + static_cast<long long>(slot) * P.s_slot) * 2;
      };
      const char* const head = reinterpret_cast<const char*>(P.kv + static_cast<long long>(kvh) * P.s_head) + (lane & 15) * 16;
      const int first = (pw - it0) & (kProdWarps - 1);
      long long off = 0, off_next = 0;
      int pos_next = 0;
      if (first < tiles) {
        const int pos = load_pos(first), pos8 = load_pos(min(first + 8, tiles - 1));
        if (first + 16 < tiles) pos_next = load_pos(first + 16);
        off = offs_of(pos);
        if (first + 8 < tiles) off_next = offs_of(pos8);
      }
#pragma unroll 1
      for (int t2 = first; t2 < tiles && !dead; t2 += 2 * kProdWarps) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const int t = t2 + kProdWarps * h;
          if (t >= tiles) break;
          const int it = it0 + t, s = it % kSlots;
          if (!mbar_wait(&sh.empty[s], ((it / kSlots) & 1u) ^ 1u, &sh.abort_flag)) { sh.abort_flag = 1; dead = true; break; }
          const uint32_t k_dst = smem_u32(sh.kv[s][0]) + (lane >> 4) * kPitch + (lane & 15) * 16;
          const int src = 16 * h + (lane >> 4);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const char* const row = head + __shfl_sync(0xffffffffu, off, src + 2 * i);
            cp_async16(k_dst + 2 * i * kPitch, row);
            cp_async16(k_dst + (kTile + 2 * i) * kPitch, row + v_delta);
          }
          // (test hook: the first tile of CTA 0 never completes, so the bounded waits run out)
          if (!(P.test_lose && blockIdx.x == 0 && it == 0)) cp_async_mbar_arrive_noinc(&sh.full[s]);
          last_it = it;
        }
        // The tiles after next are resolved when the copies went out (not before: while the ring still has free slots the
        // dependent loads would delay them).
        if (t2 + 8 < tiles) {
          off = off_next;
          if (t2 + 16 < tiles) {
            off_next = offs_of(pos_next);
            if (t2 + 24 < tiles) pos_next = load_pos(t2 + 24);
          }
        }
      }
      if (bad && P.status) atomicOr(P.status + b, SPECATTN_ROW_BAD_INDEX);
      it0 += tiles;
      a = seg_hi;
      ++seg;
      if (a == ue) {
        ++u;
        while (u < U && unit_start[u + 1] == unit_start[u]) ++u;
      }
    }
    if (sh.abort_flag) {
      // give this warp's last copies a bounded chance to land before the CTA retires (the queries of a unit that the
      // consumers will not get to among them)
      if (last_it >= 0) mbar_wait(&sh.full[last_it % kSlots], (last_it / kSlots) & 1u, nullptr);
      if (q_seg > 0) mbar_wait(&sh.q_full[q_seg & 1], (q_seg >> 1) & 1u, nullptr);
    }
    return;
  }

  // =============================== consumer warps ===========================================
  set_max_registers_inc<kConsRegs>();
  const int a0 = sh.part.range[0], a1 = sh.part.range[1], u_first = sh.part.mine[0];
  if (P.lists_stable) {
    // the first query block on its way to L2 meanwhile (only there: the previous kernel may still be writing it)
    const int b = u_first / P.Hkv, kvh = u_first % P.Hkv;
    if (tid < 2 * P.M)
      prefetch_l2(P.q + (static_cast<long long>(b) * P.T * P.Hq + kvh * P.grp + sh.row_off[tid >> 1]) * kD + (tid & 1) * 64);
    pdl_wait();
  }
  for (int v = blockIdx.x; v < U; v += gridDim.x)
    if (unit_cnt[v] == 0) empty_unit(v, tid, kConsWarps * 32);
  const int g = lane >> 2, tq = lane & 3;
  const int lm = lane >> 3, lr = lane & 7;  // ldmatrix: matrix id, row within it
  const uint32_t q_addr0 = smem_u32(sh.q) + ((lm & 1) * 8 + lr) * kPitch + (lm >> 1) * 16;
  const uint32_t q_half0 = smem_u32(sh.q) + lr * kPitch + (lm & 1) * 16;   // (of rows 0 - 7 of a slab)
  // per-lane byte offset inside a tile, for the K fragments and for the (transposed) V fragments
  const uint32_t kv_off = smem_u32(sh.kv) + ((lm >> 1) * 8 + lr) * kPitch + (lm & 1) * 16;
  // Block i of the accumulators holds dims 16 (i ^ turn / 32) ...: each warp's own share of the output, the one it
  // is left with after the combine, comes first.
  const uint32_t turn = 64u * warp;

  // A warp that meets a failed wait raises abort_flag and stops computing, but still walks through the barriers of the
  // segment it is in; at its end all consumer warps agree on whether to go on, so that they always leave together.
  int it0 = 0, seg = 0;
  int a = a0, u = u_first;
  bool ok = true;
  bool in_cluster = false;                  // the CTA's part is merged inside its cluster
  while (a < a1) {
    const int us = unit_start[u], ue = unit_start[u + 1];
    const int seg_hi = min(a1, ue);
    const int b = u / P.Hkv, kvh = u % P.Hkv;
    const int tiles = seg_hi - a;
    const int tok_lo = (a - us) * kAtom;
    const int tok_hi = min(unit_cnt[u], (seg_hi - us) * kAtom);
    const int c_list = unit_cnt[u] - P.tail;
    const long long row0 = static_cast<long long>(b) * P.T * P.Hq + kvh * P.grp;
    if (seg == 0) {
      // First query block of the CTA: the consumers copy it themselves, straight after their wait for
      // the previous kernel -- the queries are the one input that kernel may have produced.
      // Going through the producer warp (which first issues its K/V tile, then waits, then
      // starts a bulk copy) put ~2.5 us between the previous launch's end and the first product.
      for (int i = tid; i < P.M * 16; i += kConsWarps * 32) {
        const int r = i >> 4, c = i & 15;
        cp_async16(smem_u32(sh.q[0]) + r * kPitch + c * 16, P.q + (row0 + sh.row_off[r]) * kD + c * 8);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      named_bar_sync(3, kConsWarps * 32);
    } else {
      ok = mbar_wait(&sh.q_full[seg & 1], (seg >> 1) & 1u, &sh.abort_flag);
    }
    if (!ok) sh.abort_flag = 1;

    const uint32_t q_addr = q_addr0 + (seg & 1) * sizeof(sh.q[0]), q_half = q_half0 + (seg & 1) * sizeof(sh.q[0]);
    RowState<NT8> st;
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
#pragma unroll
      for (int i = 0; i < 8; ++i) st.acc[i][nt][0] = st.acc[i][nt][1] = st.acc[i][nt][2] = st.acc[i][nt][3] = 0.f;
      st.m[nt] = -INFINITY;
      st.l[nt] = 0.f;
    }
#pragma unroll 1
    for (int t = (warp - it0) & (kConsWarps - 1); ok && t < tiles; t += kConsWarps) {   // (tile it belongs to warp it % 4)
      const int it = it0 + t, s = it % kSlots;
      if (!mbar_wait(&sh.full[s], (it / kSlots) & 1u, &sh.abort_flag)) { sh.abort_flag = 1; ok = false; break; }
      const uint32_t k_addr = kv_off + s * (2 * kTile * kPitch);
      const int t0 = tok_lo + t * kTile;
      const int tail_at = P.tail ? (c_list - t0) : (1 << 20);
      const auto row_lim = [&](int nt) { return (8 * nt + g) / P.grp + P.tail_off; };
      attend_tile<NT8>(st, q_addr, q_half, k_addr, k_addr + kTile * kPitch, turn, tok_hi - t0, P.scale_log2, tq, tail_at, row_lim);
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.empty[s]);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.q_empty[seg & 1]);   // the query tile was read for the last time

    // ---- end of the segment: the key groups' shares of every row are added up -------------------
    float (&acc)[8][NT8][4] = st.acc;
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      st.l[nt] += __shfl_xor_sync(0xffffffffu, st.l[nt], 1);
      st.l[nt] += __shfl_xor_sync(0xffffffffu, st.l[nt], 2);
      if (tq == 0) sh.stat[warp][8 * nt + g] = make_float2(st.m[nt], st.l[nt]);
    }
    if (named_bar_or(3, kConsWarps * 32, !ok || sh.abort_flag)) ok = false;
#pragma unroll
    for (int nt = 0; nt < NT8; ++nt) {
      float2 ml[kConsWarps];
      float mn = -INFINITY;
#pragma unroll
      for (int j = 0; j < kConsWarps; ++j) {
        ml[j] = sh.stat[j][8 * nt + g];
        mn = fmaxf(mn, ml[j].x);
      }
      const float base = (mn == -INFINITY) ? 0.f : mn;
      const float2 c = row_to_col(ex2(st.m[nt] - base), tq);
      st.m[nt] = mn;
      st.l[nt] = 0.f;
#pragma unroll
      for (int j = 0; j < kConsWarps; ++j) st.l[nt] += ml[j].y * ex2(ml[j].x - base);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc[i][nt][0] *= c.x;
        acc[i][nt][1] *= c.y;
        acc[i][nt][2] *= c.x;
        acc[i][nt][3] *= c.y;
      }
    }
    // Two warps at a time exchange halves of what they have, two blocks of dims a turn, until each is left with its own
    // share.  (Barriers of the pair only.  Behind the last segment the ring could hold all shares at once, with one
    // barrier: a second piece of code, which cost more than the barriers, 12.8 -> 13.2 us a launch.)
#pragma unroll
    for (int w = 4; w >= 2; w >>= 1) {
      const int other = warp ^ (w / 2);
      const int pair = (w == 4) ? 4 + (warp & 1) : 6 + (warp >> 1);
#pragma unroll
      for (int i = 0; i < w; i += 2) {
#pragma unroll
        for (int k = 0; k < 2 * NT8; ++k) {
          const float(&x)[4] = acc[w + i + k / NT8][k % NT8];
          sh.scratch[warp][k][lane] = make_float4(x[0], x[1], x[2], x[3]);
        }
        named_bar_sync(pair, 64);
#pragma unroll
        for (int k = 0; k < 2 * NT8; ++k) {
          const float4 x = sh.scratch[other][k][lane];
          float(&y)[4] = acc[i + k / NT8][k % NT8];
          y[0] += x.x;
          y[1] += x.y;
          y[2] += x.z;
          y[3] += x.w;
        }
        named_bar_sync(pair, 64);
      }
    }
    const bool whole = (a == us) && (seg_hi == ue);
    // A part of a unit, this CTA's only segment, is merged inside the cluster (after a failed wait too:
    // the peers read this CTA's memory, so it leaves with them, and the result is flagged).
    if (!whole && sh.part.aligned && sh.part.cluster > 1) {
      // (in the ring: every consumer warp has met the others behind its last tile)
      float4* const rec = reinterpret_cast<float4*>(sh.kv) + warp * kItems * 32 + lane;
#pragma unroll
      for (int k = 0; k < kItems; ++k) {
        const float(&x)[4] = acc[k / NT8][k % NT8];
        rec[k * 32] = make_float4(x[0], x[1], x[2], x[3]);
      }
      if (warp == 0 && tq == 0) {
#pragma unroll
        for (int nt = 0; nt < NT8; ++nt) sh.sum[8 * nt + g] = make_float2(st.m[nt], st.l[nt]);
      }
      cluster_arrive_release();
      in_cluster = true;
      break;
    }
    if (!ok) break;
    const Items<NT8> items{P, sh.row_off, row0, warp, lane};
    if (whole) {
#pragma unroll
      for (int nt = 0; nt < NT8; ++nt) {
        const float2 inv = row_to_col((st.l[nt] > 0.f) ? 1.f / st.l[nt] : 0.f, tq);
#pragma unroll
        for (int k = nt; k < kItems; k += NT8) {
          const float(&x)[4] = acc[k / NT8][nt];
          items.store(k, make_float4(x[0] * inv.x, x[1] * inv.y, x[2] * inv.x, x[3] * inv.y));
        }
        const int r = 8 * nt + g;
        if (warp == 0 && tq == 0 && r < P.M) P.lse[row0 + sh.row_off[r]] = lse_of(st.m[nt], st.l[nt]);
      }
    } else {
      // publish this warp's share of the unit, then see whether it was the last to arrive
      const long long VN = sh.part.atoms + static_cast<long long>(kSegAtoms) * U, CN = sh.part.ctas;
      const bool al = sh.part.aligned != 0;
      const int vs = us + kSegAtoms * u;  // (where the unit's range begins)
      const auto record = [&](int i) -> float4* {
        const size_t at = static_cast<size_t>(2 * i + ((al || cta_first_atom(i, VN, CN) >= vs) ? 0 : 1)) * record_floats<NT8>();
        return reinterpret_cast<float4*>(P.partials + at) + warp * (kItems * 32 + 4 * NT8);
      };
      float4* const rec = record(blockIdx.x);
#pragma unroll
      for (int k = 0; k < kItems; ++k) {
        const float(&x)[4] = acc[k / NT8][k % NT8];
        __stcg(rec + k * 32 + lane, make_float4(x[0], x[1], x[2], x[3]));
      }
      if (tq == 0) {
#pragma unroll
        for (int nt = 0; nt < NT8; ++nt)
          __stcg(reinterpret_cast<float2*>(rec + kItems * 32) + 8 * nt + g, make_float2(st.m[nt], st.l[nt]));
      }
      __threadfence();
      __syncwarp();
      const int i_lo = al ? blockIdx.x - sh.part.mine[1] : cta_of_atom(vs + kSegAtoms, VN, CN);
      const int i_hi = al ? i_lo + sh.part.mine[2] - 1 : cta_of_atom(vs + kSegAtoms + (ue - us) - 1, VN, CN);
      unsigned int old = 0;
      if (lane == 0) old = atomicAdd(P.counters + u * kCountersPerUnit + warp, 1u);
      old = __shfl_sync(0xffffffffu, old, 0);
      if (old == static_cast<unsigned int>(i_hi - i_lo)) {
        __threadfence();
        if (lane == 0) P.counters[u * kCountersPerUnit + warp] = 0u;  // ready for the next call
        merge_global(items, i_lo, i_hi, [&](int i) -> const float4* { return record(i); });
      }
    }
    it0 += tiles;
    a = seg_hi;
    ++seg;
    if (a == ue) {
      ++u;
      while (u < U && unit_start[u + 1] == unit_start[u]) ++u;
    }
  }
  if (in_cluster) {
    const uint32_t rec = smem_u32(sh.kv), sum = smem_u32(sh.sum);
    const int mu = sh.part.mine[0], me = sh.part.mine[1], k = sh.part.mine[2];
    if (k == 2) merge_cluster<NT8, 2>(P, sh.row_off, rec, sum, me, mu);
    else merge_cluster<NT8, 4>(P, sh.row_off, rec, sum, me, mu);   // (no larger clusters: verify_grid)
  }
  if (!ok && P.status && lane == 0) atomicOr(P.status, SPECATTN_ROW_TIMEOUT);
}

}  // namespace rows
