// E-step / VQ_quant (paper Sec. 3, Eq. 5): for every d-vector x of a dense matrix (d adjacent
// columns of one row) the index of the centroid of its block that minimises
// (x - c)^T D (x - c), D = diagonal weights of the vector's columns, written in the packed index
// format the decode path reads.
//
// A CTA takes a tile of 32 rows x 256*d columns; its codebooks go to shared memory as binary32
// (int8 entries times their block scale, exact).  A thread owns 8 consecutive vectors of each of its four
// rows (a group of 8 indices = b whole bytes of the stream) and writes their b bytes; the rows are adjacent where
// the weighted search ranks the same vector of the four together, else 8 apart.
//
// The decision is taken in binary32 with every operation rounded separately (no fused
// multiply-add), terms added left to right, lowest index among equal distances: the same
// sequence the CPU oracle evaluates, so both sides break near-ties alike.
//
// Arithmetic-bound: that sequence is 4 d - 1 operations and a selection per (vector, centroid).  So it is evaluated for a
// few centroids only.  A first pass ranks all of them by the expanded form of the distance over the first weight,
//   s = sum_t r_t c_t^2 - 2 r_t x_t c_t,   r_t = D_t / D_0,
// 2 d - 1 fused multiply-adds (d without weights), two centroids per f32x2 instruction, and keeps the best group of 8 centroids
// (for large or one-dimensional codebooks the two best) and the best score outside.  If that one is further from the best than
// both forms' rounding errors can account for (the gap, below), the winner lies in the group or groups kept and the exact
// sequence runs over their centroids; else over all of them.
// Weights belong to columns: where a thread ranks the same vector of four rows of a block together, the part of the score that holds
// no x is computed once for the four, and so are the ratios r_t.  11008 x 4096, 64 2-D entries, weighted: 378 us with four
// neighbouring vectors of one row, 326 with four rows, 312 with the four vectors' exact sequences side by side.
#include "vq_common.cuh"

namespace vq {
namespace {

constexpr int kRows = 32;
constexpr int kWarps = 8;

struct AssignArgs {
  const __half* W;
  const void* cb;
  const __half* scale;
  const float* hdiag;   // [K] or null (identity)
  uint8_t* idx;
  long long stride;
  int N, K, b, Br, Bc, entries, blocks_per_row, groups;   // groups = K / (8 d) per row
  int used_bytes;       // bytes of a row that hold indices; the rest of the stride is zero-filled
  int bc_shift;         // log2(Bc)
  int br_per_tile, bc_per_seg, rows_per_br;
  int find_equal;    // two-pass kernel: leave repeated entries aside
};

template <int D>
__global__ void __launch_bounds__(32 * kWarps) assign_kernel(const AssignArgs a) {
  extern __shared__ __align__(16) float tables[];   // [block row][block col][entry][D]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seg_cols = 256 * D;
  const int row0 = blockIdx.y * kRows, col0 = blockIdx.x * seg_cols;
  const int table_floats = a.entries * D;
  {
    const long long br0 = row0 / a.Br, bc0 = col0 / a.Bc;
    const long long last_br = (a.N - 1) / a.Br;
    const int n_tab = a.br_per_tile * a.bc_per_seg;
    for (int o = tid; o < n_tab * table_floats; o += 32 * kWarps) {
      const int tb = o / table_floats, within = o - tb * table_floats;
      const int lbr = tb / a.bc_per_seg, lbc = tb - lbr * a.bc_per_seg;
      long long brow = br0 + lbr, bcol = bc0 + lbc;
      if (brow > last_br) brow = last_br;                        // rows past N: never used
      if (bcol >= a.blocks_per_row) bcol = a.blocks_per_row - 1;  // columns past K: never used
      const long long blk = brow * a.blocks_per_row + bcol;
      float v;
      if (a.scale == nullptr) v = __half2float(__ldg(static_cast<const __half*>(a.cb) + blk * table_floats + within));
      else v = __fmul_rn(static_cast<float>(__ldg(static_cast<const int8_t*>(a.cb) + blk * table_floats + within)),
                         __half2float(__ldg(a.scale + blk)));
      tables[o] = v;
    }
  }
  __syncthreads();

  const int grp = blockIdx.x * 32 + lane;   // group of 8 indices within the row
  if (grp >= a.groups) return;
  const int col = grp * 8 * D;              // first column of the thread's 8 vectors
  float dw[8][D];
#pragma unroll
  for (int v = 0; v < 8; ++v)
#pragma unroll
    for (int t = 0; t < D; ++t) dw[v][t] = a.hdiag ? __ldg(a.hdiag + col + v * D + t) : 1.f;
  const int lbc = (col - col0) >> a.bc_shift;   // 0 when the block is wider than the segment

  for (int r = warp; r < kRows; r += kWarps) {
    const int n = row0 + r;
    if (n >= a.N) break;
    float x[8][D];
    {
      const uint4* src = reinterpret_cast<const uint4*>(a.W + static_cast<long long>(n) * a.K + col);
#pragma unroll
      for (int q = 0; q < D; ++q) {   // 8*D halves = D 128-bit loads
        const uint4 raw = __ldg(src + q);
        const uint32_t wds[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          const int e = q * 8 + h;   // element index among the thread's 8*D weights
          const __half_raw hr = {static_cast<unsigned short>((wds[h >> 1] >> (16 * (h & 1))) & 0xffff)};
          x[e / D][e % D] = __half2float(__half(hr));
        }
      }
    }
    const float* tab = tables + ((r / a.rows_per_br) * a.bc_per_seg + lbc) * table_floats;
    float best[8];
    int bidx[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      best[v] = __int_as_float(0x7f800000);   // +inf
      bidx[v] = 0;
    }
    for (int m = 0; m < a.entries; ++m) {
      float c[D];
#pragma unroll
      for (int t = 0; t < D; ++t) c[t] = tab[m * D + t];
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t < D; ++t) {
          const float diff = __fsub_rn(x[v][t], c[t]);
          const float term = __fmul_rn(dw[v][t], __fmul_rn(diff, diff));
          acc = t == 0 ? term : __fadd_rn(acc, term);
        }
        if (acc < best[v]) {
          best[v] = acc;
          bidx[v] = m;
        }
      }
    }
    unsigned long long bits = 0;
#pragma unroll
    for (int v = 0; v < 8; ++v) bits |= static_cast<unsigned long long>(bidx[v]) << (v * a.b);
    uint8_t* dst = a.idx + n * a.stride + static_cast<long long>(grp) * a.b;
    for (int i = 0; i < a.b; ++i) dst[i] = static_cast<uint8_t>(bits >> (8 * i));
    if (grp == a.groups - 1)   // padding up to the row stride
      for (long long i = a.used_bytes; i < a.stride; ++i) a.idx[n * a.stride + i] = 0;
  }
}

// ---- two-pass kernel -----------------------------------------------------------------------
// two binary32 values, each operation rounded separately
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

constexpr int kGroup = 8;   // centroids per group of the first pass
// The gap, u = 2^-24.  For a centroid c let d be its distance over D_0 and M = sum_t r_t (|x_t| + |c_t|)^2, which bounds d, |s| and
// every partial sum of both.  Score: r_t (1 rounding), -2 r_t x_t (2) and c_t^2 (1) enter 2 d - 1 <= 7 fused steps, each off by at
// most u M; the group's number in its low bits moves it by less than 2 groups u M.  Distance: d + 3 <= 7 roundings of
// non-negative terms, 8 u M.  So a centroid that the exact sequence prefers to the best scored one scores within
//   2 (12 + 8 + 2 groups) u M of it, M the larger of the two; kGapBase, kGapGroup: a fifth more.  (The group's number only with
// TOP2, below.)
// And |c_t| <= |x_t| + |x_t - c_t| gives M <= 5 X + 5 d, X = sum_t r_t x_t^2, for each of them, with d within 17 u of the best
// scored centroid's, which is its score plus X.  (With the block's largest |c| in that bound's place one far centroid left every
// vector of its block undecided: 4096 x 4096, 64 2-D entries, weighted, one of them at 30 sigma 270 us, now 145 as without it.)
constexpr float kGapBase = 5.f * 48.f / 16777216.f, kGapGroup = 5.f * 5.f / 16777216.f;

// shared memory: tables of E / 8 groups; a group = 4 pairs of centroids, a pair = (c_t[m], c_t[m + 1]) for every t, and 16
// bytes of padding, so that 8 lanes reading 8 different groups hit different banks; then max |c| of each table
template <int D>
__host__ __device__ constexpr int group_bytes() { return kGroup * D * 4 + 16; }

template <int D>
__device__ __forceinline__ void load_pair(uint64_t (&c)[D], const unsigned char* p) {
  if constexpr (D == 1) {
    c[0] = *reinterpret_cast<const uint64_t*>(p);
  } else {
#pragma unroll
    for (int i = 0; i < D / 2; ++i) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + 16 * i);
      c[2 * i] = v.x;
      c[2 * i + 1] = v.y;
    }
  }
}

// Indices of the winners of V vectors of one block, given to emit(vector, index).  TOP2: the two best groups are kept, with the group's number in the low bits
// of its score; else the best group only.  COL: the vectors lie in the same columns, so that they share their weights (dw[0]) and with
// them the part of the score that the vector does not enter, sum_t r_t c_t^2: d fused steps a vector and pair are left of 2 d - 1.
template <int D, bool HD, bool TOP2, bool COL, int V, class Emit>
__device__ __forceinline__ void pick(const float (&x)[V][D], const float (&dw)[COL ? 1 : V][D], const unsigned char* tab, float c_max, int groups, Emit emit) {
  constexpr int GB = group_bytes<D>();
  const uint64_t minus1 = pack2(-1.f, -1.f);
  constexpr int W = COL ? 1 : V;
  [[maybe_unused]] int bi[V];
  // ---- rank the groups ----
  uint64_t ca[V][D], cr[W][D];   // (-2 r_t x_t) and r_t, twice each
  float best[V], second[V], third[V], xx[V];
  int gi[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    float sq = 0.f;
    if constexpr (!HD) {
#pragma unroll
      for (int t = 0; t < D; ++t) {
        const float at = -2.f * x[v][t];
        ca[v][t] = pack2(at, at);
        sq += x[v][t] * x[v][t];
      }
      // infinity or NaN among the values: NaN, which makes the exact sequence run over all centroids.  (Values are multiples
      // of 2^-24 below 2^23, so that nothing else overflows or underflows.)
      xx[v] = sq + c_max < 1e30f ? sq : __int_as_float(0x7fc00000);
    } else {
      const float (&dv)[D] = dw[COL ? 0 : v];
      float m = 0.f, base = dv[0], far = 0.f;
      bool usable = true;
      if (base == 0.f) {   // a first weight of zero counts as 2^-40 of the largest, and the gap takes in what that adds
#pragma unroll
        for (int t = 1; t < D; ++t) base = fmaxf(base, dv[t] * 0x1p-40f);
        far = (fabsf(x[v][0]) + c_max) * (fabsf(x[v][0]) + c_max);
      }
#pragma unroll
      for (int t = 0; t < D; ++t) {
        const float rt = t > 0 ? __fdiv_rn(dv[t], base) : 1.f;
        const float at = -2.f * rt * x[v][t], reach = fabsf(x[v][t]) + c_max;
        ca[v][t] = pack2(at, at);
        if (!COL || v == 0) cr[COL ? 0 : v][t] = pack2(rt, rt);
        m += rt * reach * reach;
        sq += rt * x[v][t] * x[v][t];
        usable = usable && dv[t] >= 0.f;
      }
      // in range, so that no term overflows or underflows to where the bounds above do not hold; what single terms lose to
      // underflow is less than the gap that 1e-30 over the weights' base adds
      const float dm = base * m;
      usable = usable && base > 0.f && m > 1e-30f && m < 1e30f && dm > 1e-30f && dm < 1e30f;
      sq += 1e-30f + __fdividef(1e-30f, base) + far * (2.f / kGapBase);
      xx[v] = usable ? sq : __int_as_float(0x7fc00000);
    }
    best[v] = second[v] = third[v] = __int_as_float(0x7f800000);
    gi[v] = 0;
  }
  for (int g = 0; g < groups; ++g) {
    float gm[V];
#pragma unroll
    for (int v = 0; v < V; ++v) gm[v] = __int_as_float(0x7f7fffff);   // (a group of NaN: finite with any number in its low bits)
#pragma unroll
    for (int p = 0; p < kGroup / 2; ++p) {
      uint64_t c[D], q[D];
      load_pair<D>(c, tab + g * GB + p * (D * 8));
#pragma unroll
      for (int t = 0; t < D; ++t) q[t] = mul2(c[t], c[t]);
      if constexpr (!HD) {
#pragma unroll
        for (int t = 1; t < D; ++t) q[0] = add2(q[0], q[t]);
      } else if constexpr (COL) {
#pragma unroll
        for (int t = 1; t < D; ++t) q[0] = fma2(cr[0][t], q[t], q[0]);
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        uint64_t sc = fma2(ca[v][0], c[0], q[0]);
#pragma unroll
        for (int t = 1; t < D; ++t) {
          if constexpr (HD && !COL) sc = fma2(cr[v][t], q[t], sc);
          sc = fma2(ca[v][t], c[t], sc);
        }
        float lo, hi;
        unpack2(sc, lo, hi);
        gm[v] = fminf(fminf(gm[v], lo), hi);
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      float k = gm[v];
      if constexpr (TOP2) {
        k = __int_as_float((__float_as_int(k) & ~(groups - 1)) | g);
        third[v] = fminf(third[v], fmaxf(second[v], k));
      } else {
        gi[v] = k < best[v] ? g : gi[v];
      }
      second[v] = fminf(second[v], fmaxf(best[v], k));
      best[v] = fminf(best[v], k);
    }
  }

  // ---- the exact sequence over the groups that can hold the winner, in order ----
  // pair p of group g for vector v
  auto compare = [&](int v, int g, int p, float& bd, int& b) {
    uint64_t c[D];
    load_pair<D>(c, tab + g * GB + p * (D * 8));
    float lo = 0.f, hi = 0.f;
#pragma unroll
    for (int t = 0; t < D; ++t) {
      const uint64_t diff = fma2(c[t], minus1, pack2(x[v][t], x[v][t]));   // x - c, rounded once
      uint64_t term = mul2(diff, diff);
      const float w = HD ? dw[COL ? 0 : v][t] : 0.f;
      if constexpr (HD) term = mul2(pack2(w, w), term);
      float tl, th;
      unpack2(term, tl, th);
      // (scalar: with a packed sum the product and the sum came out as one rounding)
      lo = t == 0 ? tl : __fadd_rn(lo, tl);
      hi = t == 0 ? th : __fadd_rn(hi, th);
    }
    if (lo < bd) {
      bd = lo;
      b = g * kGroup + 2 * p;
    }
    if (hi < bd) {
      bd = hi;
      b = g * kGroup + 2 * p + 1;
    }
  };
  const float inf = __int_as_float(0x7f800000);
  if constexpr (!TOP2) {
    // the best groups of all vectors together: one vector's chain of comparisons alone leaves most issue slots empty
    float bd[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      bd[v] = inf;
      bi[v] = 0;
    }
#pragma unroll
    for (int p = 0; p < kGroup / 2; ++p)
#pragma unroll
      for (int v = 0; v < V; ++v) compare(v, gi[v], p, bd[v], bi[v]);
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const float limit = best[v] + (kGapBase + (TOP2 ? kGapGroup * groups : 0.f)) * (xx[v] + fmaxf(best[v] + xx[v], 0.f));
    int g1 = gi[v], g2 = 0, count = second[v] > limit ? 1 : groups;
    if constexpr (TOP2) {
      g1 = __float_as_int(best[v]) & (groups - 1);
      g2 = __float_as_int(second[v]) & (groups - 1);
      count = second[v] > limit ? 1 : third[v] > limit ? 2 : groups;
    }
    if (!TOP2 && count == 1) {
      emit(v, bi[v]);
      continue;
    }
    float bd = inf;
    int b = 0;
#pragma unroll 1
    for (int i = 0; i < count; ++i) {
      const int g = count == 1 ? g1 : !TOP2 || count == groups ? i : i == 0 ? min(g1, g2) : max(g1, g2);
#pragma unroll
      for (int p = 0; p < kGroup / 2; ++p) compare(v, g, p, bd, b);
    }
    emit(v, b);
  }
}

// COL: blocks of a multiple of 4 rows; a thread takes the same vector of four rows at a time.
template <int D, bool HD, bool TOP2, bool COL = false>
__global__ void __launch_bounds__(32 * kWarps, D == 4 ? 2 : 3) assign_two_pass_kernel(const AssignArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int GB = group_bytes<D>();
  constexpr int V = D == 1 ? 8 : 4;   // vectors ranked together (8 of 2-D: 394 us, 4 and half as many registers again: 375 us)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seg_cols = 256 * D;
  const int row0 = blockIdx.y * kRows, col0 = blockIdx.x * seg_cols;
  const int table_floats = a.entries * D, groups = a.entries / kGroup, table_bytes = groups * GB;
  const int n_tab = a.br_per_tile * a.bc_per_seg;
  int* cmax = reinterpret_cast<int*>(smem + n_tab * table_bytes);
  for (int i = tid; i < n_tab; i += 32 * kWarps) cmax[i] = 0;
  __syncthreads();
  {
    const long long br0 = row0 / a.Br, bc0 = col0 / a.Bc;
    const long long last_br = (a.N - 1) / a.Br;
    for (int o = tid; o < n_tab * table_floats; o += 32 * kWarps) {
      const int tb = o / table_floats, within = o - tb * table_floats;
      const int lbr = tb / a.bc_per_seg, lbc = tb - lbr * a.bc_per_seg;
      long long brow = br0 + lbr, bcol = bc0 + lbc;
      if (brow > last_br) brow = last_br;                        // rows past N: never used
      if (bcol >= a.blocks_per_row) bcol = a.blocks_per_row - 1;  // columns past K: never used
      const long long blk = brow * a.blocks_per_row + bcol;
      float v;
      if (a.scale == nullptr) v = __half2float(__ldg(static_cast<const __half*>(a.cb) + blk * table_floats + within));
      else v = __fmul_rn(static_cast<float>(__ldg(static_cast<const int8_t*>(a.cb) + blk * table_floats + within)),
                         __half2float(__ldg(a.scale + blk)));
      const int m = within / D, t = within % D;
      *reinterpret_cast<float*>(smem + tb * table_bytes + (m / kGroup) * GB + (m % kGroup / 2) * (D * 8) + t * 8 + (m & 1) * 4) = v;
      atomicMax(cmax + tb, __float_as_int(fabsf(v)));   // (non-negative floats order as integers, NaN above all)
    }
  }
  __syncthreads();
  // An entry equal to one of lower index is never the answer: it becomes NaN, which both passes leave aside.  (As a tie with its
  // twin it would send every vector near the two to the exact sequence over all groups: 4096 x 4096, 64 2-D entries, weighted, a
  // quarter of them zero 215 us, now 146.)
  if (a.find_equal) {
    uint32_t equal = 0;   // (1024 entries at most: four a thread)
    const int n_ent = n_tab * a.entries;
    for (int o = tid, k = 0; o < n_ent; o += 32 * kWarps, ++k) {
      const unsigned char* tab = smem + (o >> a.b) * table_bytes;
      const int m = o & (a.entries - 1);
      const float* own = reinterpret_cast<const float*>(tab + (m / kGroup) * GB + (m % kGroup / 2) * (D * 8));
      float me[D];
#pragma unroll
      for (int t = 0; t < D; ++t) me[t] = own[2 * t + (m & 1)];
      bool eq = false;
      auto compare = [&](const unsigned char* pair, bool upper) {
        uint64_t c[D];
        load_pair<D>(c, pair);
        bool eq_lo = true, eq_hi = upper;
#pragma unroll
        for (int t = 0; t < D; ++t) {
          float lo, hi;
          unpack2(c[t], lo, hi);
          eq_lo = eq_lo && lo == me[t];
          eq_hi = eq_hi && hi == me[t];
        }
        eq = eq || eq_lo || eq_hi;
      };
      for (int g = 0; g < m / kGroup; ++g) {
#pragma unroll
        for (int p = 0; p < kGroup / 2; ++p) compare(tab + g * GB + p * (D * 8), true);
      }
      for (int p = 0; p < m % kGroup / 2; ++p) compare(tab + (m / kGroup) * GB + p * (D * 8), true);
      if (m & 1) compare(reinterpret_cast<const unsigned char*>(own), false);
      if (eq) equal |= 1u << k;
    }
    __syncthreads();
    for (int o = tid, k = 0; o < n_ent; o += 32 * kWarps, ++k)
      if (equal >> k & 1) {
        const int m = o & (a.entries - 1);
        float* p = reinterpret_cast<float*>(smem + (o >> a.b) * table_bytes + (m / kGroup) * GB + (m % kGroup / 2) * (D * 8)) + (m & 1);
#pragma unroll
        for (int t = 0; t < D; ++t) p[2 * t] = __int_as_float(0x7fc00000);
      }
    __syncthreads();
  }

  const int grp = blockIdx.x * 32 + lane;   // group of 8 indices within the row
  if (grp >= a.groups) return;
  const int col = grp * 8 * D;              // first column of the thread's 8 vectors
  const int lbc = (col - col0) >> a.bc_shift;   // 0 when the block is wider than the segment

  if constexpr (COL) {
    static_assert(kRows == 4 * kWarps);
    const int r = 4 * warp;   // the warp's rows: of one block
    if (row0 + r >= a.N) return;
    const int tb = (r / a.rows_per_br) * a.bc_per_seg + lbc;
    const unsigned char* tab = smem + tb * table_bytes;
    const float c_max = __int_as_float(cmax[tb]);
    unsigned long long bits[4] = {};
#pragma unroll 1
    for (int v = 0; v < 8; ++v) {
      float x[4][D], dw[1][D];
#pragma unroll
      for (int i = 0; i < 4; ++i) {   // (rows of a block exist together: N is a multiple of the block rows)
        const __half* src = a.W + static_cast<long long>(row0 + r + i) * a.K + col + v * D;
        uint32_t wds[D / 2];
        if constexpr (D == 2) {
          wds[0] = __ldg(reinterpret_cast<const uint32_t*>(src));
        } else {
          const uint2 raw = __ldg(reinterpret_cast<const uint2*>(src));
          wds[0] = raw.x;
          wds[D / 2 - 1] = raw.y;
        }
#pragma unroll
        for (int t = 0; t < D; ++t) {
          const __half_raw hr = {static_cast<unsigned short>((wds[t >> 1] >> (16 * (t & 1))) & 0xffff)};
          x[i][t] = __half2float(__half(hr));
        }
      }
#pragma unroll
      for (int t = 0; t < D; ++t) dw[0][t] = __ldg(a.hdiag + col + v * D + t);
      pick<D, HD, TOP2, true, 4>(x, dw, tab, c_max, groups,
                                 [&](int i, int index) { bits[i] |= static_cast<unsigned long long>(index) << (v * a.b); });
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = row0 + r + i;
      uint8_t* dst = a.idx + n * a.stride + static_cast<long long>(grp) * a.b;
      for (int k = 0; k < a.b; ++k) dst[k] = static_cast<uint8_t>(bits[i] >> (8 * k));
      if (grp == a.groups - 1)   // padding up to the row stride
        for (long long k = a.used_bytes; k < a.stride; ++k) a.idx[n * a.stride + k] = 0;
    }
  } else {
    for (int r = warp; r < kRows; r += kWarps) {
      const int n = row0 + r;
      if (n >= a.N) break;
      const int tb = (r / a.rows_per_br) * a.bc_per_seg + lbc;
      const unsigned char* tab = smem + tb * table_bytes;
      const float c_max = __int_as_float(cmax[tb]);
      unsigned long long bits = 0;
#pragma unroll
      for (int v0 = 0; v0 < 8; v0 += V) {
        float x[V][D], dw[V][D];
        {
          const uint4* src = reinterpret_cast<const uint4*>(a.W + static_cast<long long>(n) * a.K + col + v0 * D);
#pragma unroll
          for (int q = 0; q < V * D / 8; ++q) {   // V*D halves
            const uint4 raw = __ldg(src + q);
            const uint32_t wds[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int h = 0; h < 8; ++h) {
              const int e = q * 8 + h;
              const __half_raw hr = {static_cast<unsigned short>((wds[h >> 1] >> (16 * (h & 1))) & 0xffff)};
              x[e / D][e % D] = __half2float(__half(hr));
            }
          }
        }
        if constexpr (HD) {
#pragma unroll
          for (int v = 0; v < V; ++v)
#pragma unroll
            for (int t = 0; t < D; ++t) dw[v][t] = __ldg(a.hdiag + col + (v0 + v) * D + t);
        }

        pick<D, HD, TOP2, false, V>(x, dw, tab, c_max, groups,
                                    [&](int v, int index) { bits |= static_cast<unsigned long long>(index) << ((v0 + v) * a.b); });
      }
      uint8_t* dst = a.idx + n * a.stride + static_cast<long long>(grp) * a.b;
      for (int i = 0; i < a.b; ++i) dst[i] = static_cast<uint8_t>(bits >> (8 * i));
      if (grp == a.groups - 1)   // padding up to the row stride
        for (long long i = a.used_bytes; i < a.stride; ++i) a.idx[n * a.stride + i] = 0;
    }
  }
}

}  // namespace

// Covers formats with a whole number of 8-index groups per row that do not straddle blocks
// (block_cols a power of two multiple of 8 d), block rows that divide or are divided by 32.
vq_status launch_assign(const Geometry& g, const LayerPtrs& p, const __half* W, const float* hdiag, uint8_t* idx,
                        cudaStream_t s) {
  const int seg_cols = 256 * g.d;
  if (g.cb_int4 || g.J % 8 || g.Bc % (8 * g.d)) return VQ_ERR_UNSUPPORTED;
  int bc_shift = -1;
  for (int sft = 3; sft < 31; ++sft)
    if ((1 << sft) == g.Bc) bc_shift = sft;
  if (bc_shift < 0) return VQ_ERR_UNSUPPORTED;
  if (kRows % g.Br && g.Br % kRows) return VQ_ERR_UNSUPPORTED;
  AssignArgs a;
  a.W = W;
  a.cb = p.cb;
  a.scale = g.cb_int8 ? p.scale : nullptr;
  a.hdiag = hdiag;
  a.idx = idx;
  a.stride = g.stride;
  a.N = g.N;
  a.K = g.K;
  a.b = g.b;
  a.Br = g.Br;
  a.Bc = g.Bc;
  a.entries = g.entries;
  a.blocks_per_row = g.blocks_per_row;
  a.groups = g.J / 8;
  a.used_bytes = a.groups * g.b;
  a.bc_shift = bc_shift;
  a.br_per_tile = g.Br >= kRows ? 1 : kRows / g.Br;
  a.bc_per_seg = g.Bc >= seg_cols ? 1 : seg_cols / g.Bc;
  a.rows_per_br = g.Br >= kRows ? kRows : g.Br;
  const size_t smem = static_cast<size_t>(a.br_per_tile) * a.bc_per_seg * g.entries * g.d * sizeof(float);
  if (smem > 96 * 1024) return VQ_ERR_UNSUPPORTED;
  const dim3 grid((a.groups + 31) / 32, (g.N + kRows - 1) / kRows, 1);
  static int attr_set[kMaxDevices][17] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return VQ_ERR_CUDA;
  auto launch = [&](auto kern, int slot, size_t smem) {
    if (!__atomic_load_n(&attr_set[dev][slot], __ATOMIC_ACQUIRE)) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024) != cudaSuccess) return VQ_ERR_CUDA;
      __atomic_store_n(&attr_set[dev][slot], 1, __ATOMIC_RELEASE);
    }
    kern<<<grid, 32 * kWarps, smem, s>>>(a);
    return check_launch();
  };
  // Which kernel: the faster one.  us, one pass / two passes on 4096 x 4096, weighted and not: 16 2-D entries 66/- 63/60, 4-D 70/-
  // 54/49, 1-D 80/91 80/83; 32 1-D 137/131 137/115, 2-D 115/100 110/72, 4-D 114/143 99/66; 64 1-D 257/193 257/177, 2-D 215/145
  // 211/109, 4-D 201/185 186/102; 128 1-D 497/366 497/339, 2-D 412/236 408/187, 4-D 374/277 360/175; 256 1-D 976/1130 975/1060
  // (neighbours closer than the gap), 2-D 808/420 805/345, 4-D 723/468 709/321.
  const int n_tab = a.br_per_tile * a.bc_per_seg;
  const size_t smem2 = static_cast<size_t>(n_tab) * (g.entries / kGroup * (kGroup * g.d * 4 + 16) + 4);
  const bool two = g.d == 1 ? g.entries >= 32 && g.entries <= 128 : g.d == 4 && hdiag ? g.entries >= 64 : g.entries >= (hdiag ? 32 : 16);
  // The search for repeated entries grows with a tile's entries times those of a codebook, the ranking with the latter only.  us, not
  // weighted: 4 of 61 for 32 codebooks of 16 2-D entries, 9 of 117 for 16 of 64 4-D ones, 1 of 109 for 4 of 64 2-D ones.  Not
  // beyond that (a codebook per row and 256 columns: ties then cost up to 1.4 times the one-pass kernel's time).
  a.find_equal = n_tab * g.entries <= (g.entries == 16 ? 512 : 1024);
  if (two && smem2 <= 96 * 1024) {
    const bool top2 = g.entries >= 128;
    if (g.d == 1) return hdiag ? launch(assign_two_pass_kernel<1, true, true>, 3, smem2) : launch(assign_two_pass_kernel<1, false, true>, 4, smem2);
    // The same columns of four rows share their weights (one row at a time / four, 4096 x 4096, us: 32 2-D entries 106/87, 64 2-D 144/120,
    // 256 2-D 413/352, 64 4-D 183/131, 256 4-D 463/359); blocks of one or two rows do not hold four rows.
    if (hdiag && g.Br % 4 == 0) {
      if (g.d == 2) return top2 ? launch(assign_two_pass_kernel<2, true, true, true>, 13, smem2) : launch(assign_two_pass_kernel<2, true, false, true>, 14, smem2);
      return top2 ? launch(assign_two_pass_kernel<4, true, true, true>, 15, smem2) : launch(assign_two_pass_kernel<4, true, false, true>, 16, smem2);
    }
    if (g.d == 2 && top2) return hdiag ? launch(assign_two_pass_kernel<2, true, true>, 5, smem2) : launch(assign_two_pass_kernel<2, false, true>, 6, smem2);
    if (g.d == 2) return hdiag ? launch(assign_two_pass_kernel<2, true, false>, 7, smem2) : launch(assign_two_pass_kernel<2, false, false>, 8, smem2);
    if (top2) return hdiag ? launch(assign_two_pass_kernel<4, true, true>, 9, smem2) : launch(assign_two_pass_kernel<4, false, true>, 10, smem2);
    return hdiag ? launch(assign_two_pass_kernel<4, true, false>, 11, smem2) : launch(assign_two_pass_kernel<4, false, false>, 12, smem2);
  }
  if (g.d == 1) return launch(assign_kernel<1>, 0, smem);
  if (g.d == 2) return launch(assign_kernel<2>, 1, smem);
  return launch(assign_kernel<4>, 2, smem);
}

}  // namespace vq
