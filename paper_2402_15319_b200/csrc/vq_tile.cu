// Skinny GEMM on the 5th-generation tensor cores: decoded weights go to tensor memory as the A operand of
// tcgen05.mma (M = 128 weight rows, N = 16 batch rows), so one pass over the weights serves 1 to 16
// sequences (paper Sec. 3.2: packed indices -> look-up table -> product).
//
// What bounds it.  Every pair of weights costs one 32-bit shared-memory gather, 32 of them a clock and SM: 64
// weights / clk / SM at most.  So everything else is kept off the shared-memory port and out of the gathering warps:
// activations are never loaded by a warp (the tensor core reads them from shared memory as the B operand), the
// decoded tile goes from registers to tensor memory by tcgen05.st, which has its own path, and the
// accumulators live in tensor memory, which leaves registers for 16 gathering warps per SM.
// Measured: 31 to 36 weights / clk / SM for row tables (57344 x 8192, 2-D 4-bit, 16 sequences 69.0 us with four CTAs of one quad
// per SM, 55.7 here), 28 for 6 bits, where a stage of 128 x 64 weights takes 180 to 265 wavefronts of the shared-memory port: 128 gathers,
// 16 to 24 each for the indices' copy and reads, 16 for the products' B operand, 8 to 16 for activations, up to 64 for tables.
// A call costs about 4.5 us besides.  Cold code runs at the speed of its fetches: 58 KB of it instead of 35 cost 2 to 4 us a call,
// so waits carry no report, divisions are by the host's reciprocals, and what is not done in every unit stands in one place.
//
// Work.  One persistent CTA per SM.  The rows of a call's layers ("segments") are cut into tiles of 128 rows, a tile's columns
// into units of UC, four units make a step: one for each of the CTA's four quads of decoding warps, which split the columns of
// a tile among them.  A CTA takes q whole tiles; the steps of the tiles left over form one sequence that is cut into equal
// contiguous pieces, one per CTA, walked first, so that shared tiles are summed while everyone still computes whole
// ones.  (With four CTAs of one quad each per SM a tile was shared by four times as many CTAs, whose sums met in the workspace.)
//
// Roles (672 threads with row tables, else 768).  Warps 0..15 decode, four to a quad: thread = weight row = lane of tensor memory.  A thread reads its
// row's indices of a unit from the stage the copy engine filled, looks up 32 pairs (64 columns) and stores them as
// 32 columns of tensor memory, of which the quad has two such stages.  Warps 16..19 serve a quad each: they request its index and
// activation boxes by TMA (index boxes run ahead of the programmatic-dependency wait, activations come after it) and issue its
// products (one elected lane, warp-uniform control flow: with a divergent branch in place of elect.sync an issue took
// five times as long).  Warp 20 owns the tensor memory; it, or warps 20..23, add the quads' sums and store outputs or shares of them.
//
// Tables.  One 32-bit word per entry and lane, bank = lane: no conflicts whatever the indices.  Three kinds:
//   row  : 16 entries of the lane's own row; two warps' tables alternate (256-byte entry pitch), so that the index byte
//          enters the address by one byte permute;
//   warp : blocks of 4, 8, 16 or a multiple of 32 rows, every warp replicates its own rows' codebooks;
//   CTA  : blocks of a multiple of 128 rows, one table for the four warps of a quad.
// 8-bit codebooks with row tables keep the entries as exact integers in fp16 and multiply the fp32 sums of a block by its
// scale; the other tables hold fp16(scale * c), the value vq_decode_weights writes.  4-bit codebooks multiply
// the looked-up pair by the scale of the row and its group of 128 columns, the same value again.
//
// Sums.  Each quad accumulates into its own columns of tensor memory, of which it has two sets.  Four results warps (thread = weight
// row) read a fragment's sums there, add them in quad order and give the columns back, so that the decoding warps never touch a sum.  With row
// tables, whose sums are scaled block by block, the decoding warps scale and add them in shared memory and one results warp adds
// the quads'.  (So did every format once: in pieces of 4 or 8 columns where tables leave no room for 16, the decoding warps
// waiting in between, and one warp adding eight shares of a tile a column at a time.  Batch 16: 131072 x 1024, 6 bits, 32-row
// blocks 47.9 -> 31.0 us, 19712 x 5120, 128-row blocks 33.5 -> 22.7, 4-D 33.0 -> 20.9; four CTAs of one quad per SM, this kernel's
// predecessor, 32.8, 26.5, 23.8.)  A tile whose steps all belong to one CTA is rounded to fp16 and stored.  A shared
// tile's parts go to the workspace; the CTA that draws the tile's last ticket adds them in CTA order when it has done its own
// work, or beside its whole tiles (results do not depend on timing), and resets the counter.
//
// Every wait on a barrier is bounded; a wait that runs out increments a device counter, the role stops waiting for anything
// else and still arrives on every barrier it owes, so that the kernel ends.
#include <cstdio>
#include <cstdlib>
#include <type_traits>
#include <utility>

#include "vq_common.cuh"
#include "vq_device.cuh"

namespace vq {
namespace {

using namespace dev;

constexpr int kTileRows = 128;
constexpr int kStageCols = 64;        // columns a thread decodes between two hand-overs to the tensor core
constexpr int kQuads = 4;             // groups of four decoding warps
constexpr int kDecodeWarps = 4 * kQuads, kResultsWarp = kDecodeWarps + kQuads;   // (the first of the results warps)
constexpr int kAStages = 2;           // decoded stages of a quad in tensor memory, 32 columns each
constexpr int kTmemCols = 512;        // per quad 2 x 16 accumulator columns, then per quad 2 x 32 weight columns
constexpr int kAOff = 32 * kQuads;
constexpr int kMaxDepth = 4;          // unit stages of a quad at most
constexpr int kWaitTries = 1 << 18;
constexpr int kBarBytes = 640;        // barriers and the words beside them
constexpr uint32_t kMagic = 0x64646464u;   // high byte of fp16 1024.0
constexpr uint32_t kBias2 = 0x64806480u;   // fp16 pair (1152, 1152)
// tcgen05.mma kind::f16: D fp32, A and B fp16, both K-major, N = 16, M = 128
constexpr uint32_t kIdesc = (1u << 4) | ((16u / 8) << 17) | ((128u / 16) << 24);

enum TableKind { kRow = 0, kWarp = 1, kCta = 2 };

struct Segment {
  const void* cb;
  const __half* scale;
  __half* Y;
  int N;
  int tile0;   // first tile of the segment in the call's tile sequence
};

struct TileArgs {
  Segment seg[kMaxSegments];
  int n_seg;
  float* ws_part;     // [CTA][2][batch][128] partial sums
  int* ws_ticket;     // [tile], zero between calls
  int* error_flag;
  int K, batch;
  int S, steps;       // units and steps (of a unit per quad) of a tile
  unsigned steps_inv, share_inv, share1_inv, block_inv;   // 2^32 / divisor, rounded up, for divide()
  int q, extra;       // whole tiles per CTA, CTAs that take one more (calls without a workspace)
  int tail_tile0;     // the tiles left over: their steps are shared by the CTAs,
  int sharers, share, longer;  // `sharers` of them, share + 1 each for the first `longer`, share for the others
  int blocks_per_row, Br, Bc, cb_int8;
  int D;              // unit stages of a quad
  int x_bytes, x_row_bytes;    // activations of a unit; bytes of one 64-column group of them
  int red_cols;       // columns of sums handed over at a time, a multiple of 4
  const uint8_t* codes;          // normalisation: 4-bit codes, `code_row` bytes a row, a code per 2^norm_shift columns, and the
  const unsigned short* lut;     // 16 scales of every codebook block
  int code_row, norm_shift;
  int idx_off, red_off, bar_off, front_bytes;   // dynamic shared memory: activations, indices, sums, barriers, | tables
};

struct TileMaps {
  CUtensorMap idx[kMaxSegments];
  CUtensorMap x;
};

// Format policy: D columns per entry, B index bits; BR: rows that share a table word inside a warp (kWarp).
template <int D_, int B_, int TK_, int BR_, bool I4_, bool NORM_ = false>
struct Fmt {
  static constexpr int D = D_, B = B_, TK = TK_, BR = BR_;
  static constexpr bool I4 = I4_, NORM = NORM_;   // NORM: block-wise normalisation
  static constexpr int E = 1 << B;
  // Columns of a unit: 128; 256 where a row of 128 is no whole number of 16-byte pieces (5 bits) and for row tables (half as many
  // unit changes: 57344 x 8192 at batch 16 59 us with 128).
  static constexpr int UC = TK == kRow || (128 * B / (8 * D)) % 16 != 0 ? 256 : 128;
  static constexpr int RB = UC * B / (8 * D);       // bytes of a row of a unit
  static constexpr int IDX_BYTES = kTileRows * RB;
  static constexpr int STAGES = UC / kStageCols;
  static constexpr int TABLE = TK == kRow ? 4096 : E * 128;   // row: of two warps, whose 128-byte entries alternate
  static constexpr int BUFS = TK == kCta && D == 2 ? 2 : 1;
  static constexpr int TABLES = TK == kRow ? kDecodeWarps / 2 * TABLE : TK == kWarp ? kDecodeWarps * TABLE : kQuads * BUFS * TABLE;
  // OR-merged addresses need tables on multiples of their size; 4-D look-ups add (one per four weights)
  static constexpr int ALIGN = D == 4 ? 1024 : TABLE;
  // Results warps: four read the accumulators themselves; for row tables, whose sums are scaled per block, the decoding warps read
  // them and one warp adds the quads'.
  static constexpr int RW = TK == kRow ? 1 : 4;
  static constexpr int THREADS = 32 * (kResultsWarp + RW);
  static constexpr int SWIZZLE = RB == 32 ? 3 : RB == 64 ? 1 : RB == 128 ? 2 : 0;
  static_assert(RB % 16 == 0 && (TK != kRow || (B == 4 && D == 2)));
};

// ---- small device helpers ------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {   // the same, blocking for a short time
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}
// Bounded wait for phase `parity`; `tries` is the role's budget: 0 once a wait has run out, so that later ones return at once
// (the role reports it at its end: one place keeps the code small).
__device__ __forceinline__ void wait_phase(uint32_t bar, uint32_t parity, int& tries) {
  int left = tries;
#pragma unroll 1
  while (!mbar_try(bar, parity))
    if (--left <= 0) {
      tries = 0;
      break;
    }
}
__device__ __forceinline__ void results_barrier() { asm volatile("bar.sync 5, 128;" ::: "memory"); }
__device__ __forceinline__ void quad_barrier(int quad) { asm volatile("bar.sync %0, 128;" ::"r"(1 + quad) : "memory"); }
__device__ __forceinline__ void tma_box_3d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
               ::"r"(dst), "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(bar) : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// Weights, codes and scale tables: complete before the call, so read-only for the kernel, or (ORDERED: normalised calls) perhaps written
// by the kernel in front, so read behind griddepcontrol.wait only and not through the read-only path.  (volatile: not moved across the wait)
template <int BYTES, bool ORDERED>
__device__ __forceinline__ uint32_t load_weight(const void* p) {
  static_assert(BYTES == 1 || BYTES == 2 || BYTES == 4);
  if constexpr (!ORDERED) {
    if constexpr (BYTES == 1) return __ldg(static_cast<const uint8_t*>(p));
    else if constexpr (BYTES == 2) return __ldg(static_cast<const unsigned short*>(p));
    else return __ldg(static_cast<const uint32_t*>(p));
  } else {
    uint32_t v;
    if constexpr (BYTES == 1) asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p));
    else if constexpr (BYTES == 2) asm volatile("ld.global.u16 %0, [%1];" : "=r"(v) : "l"(p));
    else asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
  }
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[128 x 16] (+)= A[128 x 16] (tensor memory) * B[16 x 16] (shared memory)
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b_desc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d), "r"(a), "l"(b_desc), "r"(kIdesc), "r"(accumulate) : "memory");
}
// B operand, K-major rows of 128 bytes with the 128-byte swizzle, 8 rows (batch) per 1024-byte group
__device__ __forceinline__ uint64_t b_descriptor(uint32_t addr) {
  return (static_cast<uint64_t>(addr >> 4) & 0x3FFF) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tc_store32(uint32_t addr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
      "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// four accumulator columns of the thread's row, to be used behind tc_load_wait()
__device__ __forceinline__ void tc_load4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
template <int N>
__device__ __forceinline__ void tc_load_wait(uint32_t (&r)[N][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int i = 0; i < 4; ++i) asm volatile("" : "+r"(r[k][i]));   // used behind the wait only
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds32_now(uint32_t addr) {   // (not moved across barriers)
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float lds32f(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t mul_f16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t int8_pair(uint32_t biased, uint32_t sel) {   // (u, u') - 128 as fp16, exact
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(prmt(biased, kMagic, sel)), "r"(kBias2));
  return r;
}
__device__ __forceinline__ uint32_t scaled_pair(float s, uint32_t two) {   // fp16(s * c0), fp16(s * c1): exact products, one rounding
  const __half2 h = __floats2half2_rn(s * static_cast<float>(static_cast<int8_t>(two & 0xffu)),
                                      s * static_cast<float>(static_cast<int8_t>((two >> 8) & 0xffu)));
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t nibble_pair(uint32_t byte) {   // two signed 4-bit integers as fp16, exact
  const __half2 h = __floats2half2_rn(static_cast<float>(static_cast<int>(byte << 28) >> 28), static_cast<float>(static_cast<int>(byte << 24) >> 28));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// x / d for x * d < 2^32 and inv = ceil(2^32 / d)  (d = 1: inv = 0)
__device__ __forceinline__ int divide(int x, unsigned inv) { return inv ? static_cast<int>(__umulhi(static_cast<unsigned>(x), inv)) : x; }
// first step of CTA c's piece of the left-over tiles, and the CTA whose piece holds step x
__device__ __forceinline__ int first_step(const TileArgs& a, int c) { return min(c, a.sharers) * a.share + min(c, a.longer); }
__device__ __forceinline__ int step_owner(const TileArgs& a, int x) {
  const int n = a.longer * (a.share + 1);
  return x < n ? divide(x, a.share1_inv) : a.longer + divide(x - n, a.share_inv);
}

// A CTA's walk over its fragments (steps [s0, s1) of one tile): its piece of the left-over tiles first, then its whole tiles.
struct Walk {
  int tile, s0, s1, left, whole, whole_end;
  bool valid;

  __device__ __forceinline__ void init(const TileArgs& a, int c) {
    const int t0 = first_step(a, c), ahead = divide(t0, a.steps_inv);
    whole = c * a.q + min(c, a.extra);
    whole_end = whole + a.q + (c < a.extra ? 1 : 0);
    tile = a.tail_tile0 + ahead - 1;
    left = first_step(a, c + 1) - t0;
    next(a, t0 - ahead * a.steps);
  }
  __device__ __forceinline__ void next(const TileArgs& a, int first = 0) {
    valid = true;
    s0 = 0;
    s1 = a.steps;
    if (left > 0) {
      ++tile;
      s0 = first;
      s1 = min(a.steps, first + left);
      left -= s1 - s0;
    } else if (whole < whole_end) {
      tile = whole++;
    } else {
      valid = false;
    }
  }
  __device__ __forceinline__ bool complete(const TileArgs& a) const { return s0 == 0 && s1 == a.steps; }
  // units of the fragment that are quad k's
  __device__ __forceinline__ void range(const TileArgs& a, int k, int& u, int& end) const {
    const int u0 = kQuads * s0, n = min(kQuads * s1, a.S) - u0;
    u = u0 + n * k / kQuads;
    end = u0 + n * (k + 1) / kQuads;
  }
};
// ... and over one quad's units, fragments without any left out.
struct Units {
  Walk f;
  int u, end;
  __device__ __forceinline__ void settle(const TileArgs& a, int k) {
    while (u == end) {
      f.next(a);
      if (!f.valid) return;
      f.range(a, k, u, end);
    }
  }
  __device__ __forceinline__ void init(const TileArgs& a, const Walk& first, int k) {
    f = first;
    f.range(a, k, u, end);
    settle(a, k);
  }
  __device__ __forceinline__ void next(const TileArgs& a, int k) {
    ++u;
    settle(a, k);
  }
};

__device__ __forceinline__ int segment_of(const TileArgs& a, int tile) {
  int g = 0;
#pragma unroll
  for (int i = 1; i < kMaxSegments; ++i)
    if (i < a.n_seg && tile >= a.seg[i].tile0) g = i;
  return g;
}

// outputs of rows row .. row + 3 of one sequence
__device__ __forceinline__ void store_rows(const Segment& sg, int row, int n, float4 s) {
  __half* y = sg.Y + static_cast<long long>(n) * sg.N + row;
  const __half2 lo = __floats2half2_rn(s.x, s.y), hi = __floats2half2_rn(s.z, s.w);
  if (sg.N % 4 == 0) {   // (the rows then exist together, 8-byte aligned)
    if (row < sg.N) *reinterpret_cast<uint2*>(y) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
  } else {
    if (row < sg.N) y[0] = __low2half(lo);
    if (row + 1 < sg.N) y[1] = __high2half(lo);
    if (row + 2 < sg.N) y[2] = __low2half(hi);
    if (row + 3 < sg.N) y[3] = __high2half(hi);
  }
}

// ---- look-up tables: request a block's entries (registers), write them as table words --------------------------
template <class F>
struct Tables {
  // entries one lane requests: the whole codebook of its row (row), E / BR of one of the warp's codebooks (warp), or
  // its share of the CTA's codebook: one entry of a 2-D one (two or four threads each), 2 of a 4-D one
  static constexpr int EPL = F::TK == kRow ? 16 : F::TK == kWarp ? (F::E / F::BR) : (F::D == 4 ? 2 : 1);
  static constexpr int VALS = EPL * F::D;                 // values requested
  static constexpr int RAW = F::I4 ? (VALS + 7) / 8 : (VALS + 1) / 2;   // registers (fp16; 8-bit entries use half of them)
  uint32_t raw[RAW];
  uint32_t sc;                 // the block's scale (8-bit codebooks)
  const uint8_t* src;          // this lane's share in block column 0 of the current fragment's block row
  const unsigned short* ssrc;

  __device__ __forceinline__ void open(const TileArgs& a, const Segment& sg, int row0, int tid) {   // a fragment's rows
    const int lane = tid & 31, warp = tid >> 5;
    int brow, part;
    if constexpr (F::TK == kRow) {
      brow = min(row0 + tid, sg.N - 1) / a.Br;
      part = 0;
    } else if constexpr (F::TK == kWarp) {
      const int r = row0 + 32 * warp + (F::BR < 32 ? (lane % (32 / F::BR)) * F::BR : 0);
      brow = min(r, sg.N - 1) / a.Br;
      part = lane / (32 / F::BR) * EPL;
    } else {
      brow = row0 / a.Br;
      part = F::D == 4 ? 2 * tid : tid % F::E;
    }
    const long long blk = static_cast<long long>(brow) * a.blocks_per_row;
    const int bits = F::I4 ? 4 : a.cb_int8 ? 8 : 16;
    src = static_cast<const uint8_t*>(sg.cb) + (blk * F::E + part) * F::D * bits / 8;
    ssrc = reinterpret_cast<const unsigned short*>(sg.scale) + blk;
  }
  __device__ __forceinline__ void request(const TileArgs& a, int bcol) {
    const int bits = F::I4 ? 4 : a.cb_int8 ? 8 : 16;
    const uint8_t* p = src + static_cast<long long>(bcol) * (F::E * F::D * bits / 8);
    if constexpr (F::I4) {
      load<VALS / 2>(p);
    } else if (a.cb_int8) {
      load<VALS>(p);
      sc = load_weight<2, F::NORM>(ssrc + bcol);
    } else {
      load<VALS * 2>(p);
    }
  }
  template <int BYTES>
  __device__ __forceinline__ void load(const uint8_t* p) {
    static_assert(!F::NORM || BYTES <= 8);
    if constexpr (BYTES <= 4) raw[0] = load_weight<BYTES, F::NORM>(p);
    else if constexpr (F::NORM) {
      raw[0] = load_weight<4, true>(p);
      raw[RAW - 1] = load_weight<4, true>(p + 4);
    } else if constexpr (BYTES == 8) {
      const uint2 v = ldg64_nc(p);
      raw[0] = v.x; raw[1] = v.y;
    } else {
#pragma unroll
      for (int i = 0; i < BYTES / 16; ++i) {
        const uint4 v = ldg128_nc(p + 16 * i);
        raw[4 * i] = v.x; raw[4 * i + 1] = v.y; raw[4 * i + 2] = v.z; raw[4 * i + 3] = v.w;
      }
    }
  }
  __device__ __forceinline__ float scale() const { return __half2float(__ushort_as_half(static_cast<unsigned short>(sc))); }
  // 2-D: pair i of the requested ones as a table word
  template <bool EXACT>
  __device__ __forceinline__ uint32_t word(const TileArgs& a, int i, float s) const {
    if constexpr (F::I4) return nibble_pair((raw[i >> 2] >> (8 * (i & 3))) & 0xffu);
    else if (!a.cb_int8) return raw[i];
    else if constexpr (EXACT) return int8_pair(raw[i >> 1] ^ 0x80808080u, (i & 1) ? 0x4342u : 0x4140u);
    else return scaled_pair(s, raw[i >> 1] >> (16 * (i & 1)));
  }
  // tbl: shared address of the warp's (CTA's) table, row kind: + the half
  __device__ __forceinline__ void write(const TileArgs& a, uint32_t tbl, int tid) const {
    const int lane = tid & 31;
    const float s = !F::I4 && a.cb_int8 ? scale() : 1.f;
    if constexpr (F::TK == kRow) {
#pragma unroll
      for (int i = 0; i < EPL; ++i) sts32(tbl + i * 256 + lane * 4, word<true>(a, i, s));
    } else if constexpr (F::TK == kWarp) {
      // replicated over the rows of the block by 128-bit stores; the order of the 16-byte groups is rotated so that a
      // quarter warp writes 8 different ones
      constexpr int G = F::BR / 4, NCB = 32 / F::BR;   // 16-byte groups per codebook, codebooks of the warp
      const int c = lane % NCB, part = lane / NCB;
#pragma unroll
      for (int i = 0; i < EPL; ++i) {
        const uint32_t w = word<false>(a, i, s);
#pragma unroll
        for (int u = 0; u < G; ++u)
          sts128(tbl + (part * EPL + i) * 128 + (c * G + ((u + part) & (G - 1))) * 16, make_uint4(w, w, w, w));
      }
    } else if constexpr (F::D == 2) {
      constexpr int SHARE = 8 * F::E / 128;   // 16-byte groups per thread
      const uint32_t w = word<false>(a, 0, s);
      const int e = tid % F::E, h = tid / F::E;
#pragma unroll
      for (int i = 0; i < SHARE; ++i) sts128(tbl + e * 128 + ((lane + i + SHARE * h) & 7) * 16, make_uint4(w, w, w, w));
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t w0 = word<false>(a, 2 * i, s), w1 = word<false>(a, 2 * i + 1, s);
#pragma unroll
        for (int u = 0; u < 8; ++u) sts128(tbl + (2 * tid + i) * 128 + ((lane + u) & 7) * 16, make_uint4(w0, w1, w0, w1));
      }
    }
  }
};

// (index I of the stage's words) << 7, for tables of 128-byte entries
template <int B, int I, int NW>
__device__ __forceinline__ uint32_t entry_off(const uint32_t (&w)[NW]) {
  constexpr uint32_t MASK = ((1u << B) - 1u) << 7;
  constexpr int p = B * I, wi = p >> 5, s = p & 31;
  if constexpr (s + B > 32) return __funnelshift_r(w[wi], w[wi + 1], s - 7) & MASK;   // (s >= 25 here)
  else if constexpr (s < 7) return (w[wi] << (7 - s)) & MASK;
  else return (w[wi] >> (s - 7)) & MASK;
}

// 64 columns of the thread's row, stage J of a unit's words -> 32 fp16 pairs
template <class F, int J>
__device__ __forceinline__ void gather(uint32_t (&r)[32], const uint32_t (&w)[F::RB / 4], uint32_t tbl, uint32_t pat) {
  if constexpr (F::TK == kRow) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t even = (w[4 * J + j] & 0x0F0F0F0Fu) | pat, odd = ((w[4 * J + j] >> 4) & 0x0F0F0F0Fu) | pat;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        r[8 * j + 2 * i] = lds32(prmt(tbl, even, 0x3200u | ((4u + i) << 4)));
        r[8 * j + 2 * i + 1] = lds32(prmt(tbl, odd, 0x3200u | ((4u + i) << 4)));
      }
    }
  } else if constexpr (F::D == 2) {
    [&]<int... I>(std::integer_sequence<int, I...>) {
      ((r[I] = lds32(entry_off<F::B, 32 * J + I>(w) | tbl)), ...);
    }(std::make_integer_sequence<int, 32>{});
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t e = prmt(w[4 * J + (i >> 2)], 0u, 0x4440u | (i & 3));
      const uint2 v = lds64(e * 128u + tbl);
      r[2 * i] = v.x;
      r[2 * i + 1] = v.y;
    }
  }
}

template <class F>
__global__ void __launch_bounds__(F::THREADS, 1) tile_kernel(const __grid_constant__ TileMaps maps, const TileArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t tables = (base + a.front_bytes + F::ALIGN - 1) & ~static_cast<uint32_t>(F::ALIGN - 1);
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  {   // the host planned for dynamic shared memory that starts 1024 bytes into the CTA's window
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    if (tables + F::TABLES - raw > dyn) {   // (the same for every thread)
      if (tid == 0) atomicAdd(a.error_flag, 1);
      return;
    }
  }
  constexpr bool kExact = F::TK == kRow && !F::I4;   // 8-bit row tables hold unscaled entries: sums are scaled per block
  const int red_cols = a.red_cols;
  const int D = a.D, c = blockIdx.x;
  const bool by_block = kExact && a.cb_int8;
  const int block_units = a.Bc / F::UC;
  const int quad = warp < kDecodeWarps ? warp >> 2 : warp & 3;
  // barriers of a quad: indices and activations of a unit, decoded stages full and consumed, sums ready and read; then the CTA's
  constexpr int kQuadBars = 128;
  const uint32_t bars = base + a.bar_off, qb = bars + quad * kQuadBars;
  const uint32_t idx_full = qb, x_full = qb + 32, a_full = qb + 64, a_empty = qb + 80, d_full = qb + 96, d_empty = qb + 112;
  const uint32_t red_full = bars + kQuads * kQuadBars, red_empty = red_full + 8, tmem_slot = red_full + 16, n_last = tmem_slot + 4, ticket_word = n_last + 4, last_tile = n_last + 12;
  const uint32_t idx_at = base + a.idx_off + quad * D * F::IDX_BYTES, x_at = base + quad * D * a.x_bytes;
  const bool service = warp >= kDecodeWarps && warp < kResultsWarp;

  int tries = kWaitTries;
  Walk f;
  f.init(a, c);
  Units wi = {};   // (service warps) the next unit whose indices are to be requested
  int islot = 0, first_x = 0, first_n = 0;   // the units requested first: lane i keeps the i-th
  auto request_indices = [&]() {
    if (elect_one()) {
      const int g = segment_of(a, wi.f.tile);
      mbar_arrive_expect_tx(idx_full + 8 * islot, F::IDX_BYTES);
      tma_box_2d(idx_at + islot * F::IDX_BYTES, &maps.idx[g], wi.u * F::RB, (wi.f.tile - a.seg[g].tile0) * kTileRows, idx_full + 8 * islot);
    }
    __syncwarp();
    if (++islot == D) islot = 0;
  };
  auto request_first = [&]() {
    request_indices();
    if (lane == first_n) first_x = wi.u;
    ++first_n;
    wi.next(a, quad);
  };
  // (decoding warps) the current fragment: its tile, next unit of the quad, end, codebook block column; f: the fragment after it
  Tables<F> tb;
  const int qt = tid & 127;   // row of the tile
  int tile = f.tile, u = 0, end = 0, bcol = 0;
  bool asked = false;         // are the entries of the next block to be used on their way?
  // A normalised call reads nothing, weights, codes and scale tables included, before all in front of it on the stream is complete.
  if (warp < kDecodeWarps) {
    if (F::NORM) pdl_wait();
    f.range(a, quad, u, end);
    f.next(a);
    bcol = divide(u, a.block_inv) - 1;
    asked = u < end;
    if (asked) {
      const Segment& sg = a.seg[segment_of(a, tile)];
      tb.open(a, sg, (tile - sg.tile0) * kTileRows, qt);
      tb.request(a, bcol + 1);
    }
  } else if (service) {
    if (elect_one()) {
      for (int i = 0; i < D; ++i) {
        mbar_init(idx_full + 8 * i, 1);
        mbar_init(x_full + 8 * i, 1);
      }
      for (int i = 0; i < kAStages; ++i) {
        mbar_init(a_full + 8 * i, 4);
        mbar_init(a_empty + 8 * i, 1);
        mbar_init(d_full + 8 * i, 1);
        mbar_init(d_empty + 8 * i, F::RW);
      }
      mbar_init_fence();
    }
    __syncwarp();
    if (F::NORM) pdl_wait();
    wi.init(a, f, quad);
    if (wi.f.valid) request_first();   // (weights do not depend on the previous kernel, but for normalised calls)
  } else if (warp == kResultsWarp) {
    if (lane == 0) {
      mbar_init(red_full, kDecodeWarps);
      mbar_init(red_empty, 1);
      mbar_init_fence();
      sts32(n_last, 0u);
    }
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "n"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // The next kernel's CTAs may come as soon as this one's leave: a CTA of this kernel fills an SM, so that they take no slot
  // beside it, and their indices arrive while the last sums of this call are added.
  if (tid == 0) pdl_launch_dependents();
  const uint32_t tmem = lds32_now(tmem_slot);

  if (service) {
    // ---- service: a quad's copies and products ---------------------------------------------------------------
    int xslot = 0;
    auto request_x = [&](int u) {
      if (elect_one()) {
        mbar_arrive_expect_tx(x_full + 8 * xslot, a.x_bytes);
        tma_box_3d(x_at + xslot * a.x_bytes, &maps.x, 0, 0, u * F::STAGES, x_full + 8 * xslot);
      }
      __syncwarp();
      if (++xslot == D) xslot = 0;
    };
#pragma unroll 1
    while (first_n < D && wi.f.valid) request_first();
    pdl_wait();   // the activations belong to the previous kernel of the stream until here
#pragma unroll 1
    for (int i = 0; i < first_n; ++i) request_x(__shfl_sync(0xffffffffu, first_x, i));
    int x_next = -1;   // (u: the unit to be multiplied) the unit whose activations are to be requested
    int slot = 0, seg = 0, seg_left = 0, st = 0;
    uint32_t ph = 0, fresh = 1;
    for (;; ++st) {
      if (u == end) {
        for (; f.valid && u == end; f.next(a)) f.range(a, quad, u, end);
        if (u == end) break;
      }
      if (seg_left == 0) {
        seg_left = (by_block ? min(end, (divide(u, a.block_inv) + 1) * block_units) : end) - u;
        if (F::RW > 1) wait_phase(d_empty + 8 * (seg & 1), ((seg >> 1) & 1) ^ 1, tries);   // the sum but one before is read
      }
      wait_phase(x_full + 8 * slot, ph, tries);
#pragma unroll
      for (int j = 0; j < F::STAGES; ++j) {
        // a quad fills its two decoded stages in turn: stage j's use number is st * STAGES / 2 + j / 2
        wait_phase(a_full + 8 * (j & 1), F::STAGES == 2 ? st & 1 : (j >> 1) & 1, tries);
        __syncwarp();
        tc_fence_after();
        const uint64_t xd = b_descriptor(x_at + slot * a.x_bytes + j * a.x_row_bytes);   // (+ 2 q: 32-byte steps of K)
        const uint32_t at = tmem + kAOff + (quad * 2 + (j & 1)) * 32, dt = tmem + quad * 32 + (seg & 1) * 16;
        if (elect_one()) {   // (also after a wait that ran out: the operands are in bounds whatever they hold)
          tc_mma(dt, at, xd, fresh ^ 1u);
#pragma unroll
          for (int q = 1; q < 4; ++q) tc_mma(dt, at + 8 * q, xd + 2 * q, 1u);
          tc_commit(a_empty + 8 * (j & 1));
          if (j == F::STAGES - 1 && seg_left == 1) tc_commit(d_full + 8 * (seg & 1));
        }
        __syncwarp();
        fresh = 0;
        if (j == 0) {
          // the quad read all its indices of the unit before it handed over the first stage: the copy may be replaced
          if (wi.f.valid) {
            fence_proxy_async();   // the warps' reads (released by their arrivals) before the copy engine's writes
            request_indices();
          }
        } else if (j == 1) {
          // a stage decoded into the place of the last one of the unit before: that unit's products are complete
          if (x_next >= 0) request_x(x_next);
          x_next = -1;
          if (wi.f.valid) {
            x_next = wi.u;
            wi.next(a, quad);
          }
        }
      }
      if (--seg_left == 0) {
        ++seg;
        fresh = 1;
      }
      if (++slot == D) { slot = 0; ph ^= 1u; }
      ++u;
    }
    if (tries == 0) __nanosleep(1000000);   // gave up: let this CTA's own copies land before its shared memory goes away
  } else if (warp >= kResultsWarp && F::RW > 1) {
    // ---- results: four warps add the quads' accumulators of a fragment (thread = row), store the outputs or this CTA's share --------
    pdl_wait();   // outputs and workspace belong to earlier kernels of the stream until here
    const int first_tile = f.tile;   // (of the CTA's piece, if it has one)
    const int r = tid & 127, part_floats = a.batch * kTileRows;
    const uint32_t lane_at = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    uint32_t segs = 0;   // per quad, a byte: its sums so far
    int listed = 0;
#pragma unroll 1
    for (; f.valid; f.next(a)) {
      const Segment& sg = a.seg[segment_of(a, f.tile)];
      const int row = (f.tile - sg.tile0) * kTileRows + r, units = min(kQuads * f.s1, a.S) - kQuads * f.s0;
      const bool complete = f.complete(a);
      uint32_t has = 0;   // quads that have units of the fragment: a one in the byte
#pragma unroll
      for (int k = 0; k < kQuads; ++k)
        if (units * k / kQuads < units * (k + 1) / kQuads) has |= 1u << (8 * k);
#pragma unroll 1
      for (int k = 0; k < kQuads; ++k)
        if ((has >> (8 * k)) & 1) wait_phase(bars + k * kQuadBars + 96 + 8 * ((segs >> (8 * k)) & 1), (segs >> (8 * k + 1)) & 1, tries);
      __syncwarp();
      tc_fence_after();
      // this CTA's share of a left-over tile: slot 0 if its piece begins inside the tile, else slot 1
      float* part = a.ws_part + static_cast<long long>(c * 2 + (f.tile == first_tile ? 0 : 1)) * part_floats + r;
      __half* y = sg.Y + row;
#pragma unroll 1
      for (int n0 = 0; n0 < a.batch; n0 += 4) {
        uint32_t v[kQuads][4];
#pragma unroll
        for (int k = 0; k < kQuads; ++k) tc_load4(lane_at + k * 32 + ((segs >> (8 * k)) & 1) * 16 + n0, v[k]);
        tc_load_wait(v);
        float s[4] = {};
#pragma unroll
        for (int k = 0; k < kQuads; ++k)
          if ((has >> (8 * k)) & 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] += __uint_as_float(v[k][i]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (n0 + i < a.batch) {
            if (!complete) part[(n0 + i) * kTileRows] = s[i];
            else if (row < sg.N) y[static_cast<long long>(n0 + i) * sg.N] = __float2half_rn(s[i]);
          }
      }
      tc_fence_before();
      __syncwarp();
      if (lane < kQuads && ((has >> (8 * lane)) & 1)) mbar_arrive(bars + lane * kQuadBars + 112 + 8 * ((segs >> (8 * lane)) & 1));
      segs = (segs + has) & 0x03030303u;
      if (!complete) {
        const int first_s = (f.tile - a.tail_tile0) * a.steps, owner = step_owner(a, first_s);
        const int shares = step_owner(a, first_s + a.steps - 1) - owner + 1;   // CTAs that share the tile
        // where the first of them keeps its share: in its second slot unless its piece begins with the tile
        const int c_first = 2 * owner + (first_step(a, owner) == first_s ? 0 : 1);
        __threadfence();   // this thread's sums are visible to the GPU before the ticket is drawn
        results_barrier();
        if (tid == 32 * kResultsWarp) {
          const int ticket = atomicAdd(a.ws_ticket + f.tile, 1);
          if (ticket == shares - 1) a.ws_ticket[f.tile] = 0;   // nobody else touches the counter in this call
          sts32(ticket_word, ticket == shares - 1);
        }
        results_barrier();
        if (lds32_now(ticket_word)) {   // every share of the tile is there
          if (a.q == 0) {           // this CTA adds them when it has done its own work, by all its threads
            if (tid == 32 * kResultsWarp) sts128(last_tile + 16 * listed, make_uint4(segment_of(a, f.tile), row - r, c_first, shares));
            ++listed;
          } else {                  // whole tiles are still to come: these warps add them meanwhile
            __threadfence();
            const float* p = a.ws_part + static_cast<long long>(c_first) * part_floats + r;
            const int others = (c_first & 1 ? -1 : 0) * part_floats;   // (behind the first: in their first slots)
#pragma unroll 1
            for (int n0 = 0; n0 < a.batch; n0 += 2) {
              float s[2] = {};
#pragma unroll 1
              for (int k0 = 0; k0 < shares; k0 += 8) {   // (a load takes about 1000 clocks: sixteen at a time)
                float v[8][2];
#pragma unroll
                for (int k = 0; k < 8; ++k)
#pragma unroll
                  for (int i = 0; i < 2; ++i) {
                    v[k][i] = 0.f;
                    if (k0 + k < shares && n0 + i < a.batch)
                      v[k][i] = __ldcg(p + (2 * (k0 + k)) * part_floats + (k0 + k ? others : 0) + (n0 + i) * kTileRows);
                  }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                  s[0] += v[k][0];
                  s[1] += v[k][1];
                }
              }
#pragma unroll
              for (int i = 0; i < 2; ++i)
                if (row < sg.N && n0 + i < a.batch) y[static_cast<long long>(n0 + i) * sg.N] = __float2half_rn(s[i]);
            }
          }
        }
      }
    }
    if (tid == 32 * kResultsWarp && listed) {
      sts32(n_last, listed);
      __threadfence();   // the tickets before the shares are read
    }
  } else if (warp >= kResultsWarp) {
    // ---- results, row tables: one warp adds the quads' sums of a fragment, stores the outputs or this CTA's share of them --------
    pdl_wait();   // outputs and workspace belong to earlier kernels of the stream until here
    const int first_tile = f.tile;   // (of the CTA's piece, if it has one)
    uint32_t ph = 0;
    int listed = 0;
    for (; f.valid; f.next(a)) {
      const bool complete = f.complete(a);
      const Segment& sg = a.seg[segment_of(a, f.tile)];
      const int row = (f.tile - sg.tile0) * kTileRows + 4 * lane;
      // this CTA's share of a left-over tile: slot 0 if its piece begins inside the tile, else slot 1
      float* part = a.ws_part + (static_cast<long long>(c) * 2 + (f.tile == first_tile ? 0 : 1)) * (kTileRows * a.batch) + 4 * lane;
      int c_first = 0, shares = 1;   // CTAs that share the tile
      if (!complete) {
        const int first_s = (f.tile - a.tail_tile0) * a.steps;
        c_first = step_owner(a, first_s);
        shares = step_owner(a, first_s + a.steps - 1) - c_first + 1;
        // where the first of them keeps its share: in its second slot unless its piece begins with the tile
        c_first = 2 * c_first + (first_step(a, c_first) == first_s ? 0 : 1);
      }
      wait_phase(red_full, ph, tries);
      __syncwarp();
#pragma unroll 2
      for (int n = 0; n < a.batch; ++n) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kQuads; ++k) {
          const uint4 v = lds128(base + a.red_off + ((k * red_cols + n) * kTileRows + 4 * lane) * 4);
          s.x += __uint_as_float(v.x); s.y += __uint_as_float(v.y); s.z += __uint_as_float(v.z); s.w += __uint_as_float(v.w);
        }
        if (!complete) {
          *reinterpret_cast<float4*>(part + n * kTileRows) = s;
        } else {
          store_rows(sg, row, n, s);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(red_empty);
      ph ^= 1u;
      if (!complete) {
        __threadfence();   // this lane's sums are visible to the GPU before the ticket is drawn
        __syncwarp();
        int ticket = 0;
        if (lane == 0) {
          ticket = atomicAdd(a.ws_ticket + f.tile, 1);
          if (ticket == shares - 1) a.ws_ticket[f.tile] = 0;   // nobody else touches the counter in this call
        }
        ticket = __shfl_sync(0xffffffffu, ticket, 0);
        if (ticket == shares - 1) {   // every share of the tile is there
          if (a.q == 0) {             // this CTA adds them when it has done its own work, by all its threads
            if (lane == 0) sts128(last_tile + 16 * listed, make_uint4(segment_of(a, f.tile), row - 4 * lane, c_first, shares));
            ++listed;
          } else {                    // whole tiles are still to come: this warp adds them meanwhile
            __threadfence();
            const int part_floats = a.batch * kTileRows;
            const float* p = a.ws_part + static_cast<long long>(c_first) * part_floats + 4 * lane;
            const int others = (c_first & 1 ? -1 : 0) * part_floats;   // (behind the first: in their first slots)
#pragma unroll 1
            for (int n = 0; n < a.batch; ++n, p += kTileRows) {
              float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
              for (int k0 = 0; k0 < shares; k0 += 8) {
                float4 v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                  if (k0 + k < shares) v[k] = __ldcg(reinterpret_cast<const float4*>(p + 2 * (k0 + k) * part_floats + (k0 + k ? others : 0)));
#pragma unroll
                for (int k = 0; k < 8; ++k)
                  if (k0 + k < shares) s.x += v[k].x, s.y += v[k].y, s.z += v[k].z, s.w += v[k].w;
              }
              store_rows(sg, row, n, s);
            }
          }
        }
      }
    }
    if (lane == 0 && listed) {
      sts32(n_last, listed);
      __threadfence();   // the tickets before the shares are read
    }
  } else {
    // ---- decode ----------------------------------------------------------------------------------------------
    // One loop over units; what is not done in every unit stands in one place each (a codebook block, a running sum
    // and a fragment are whole units): the loop has to stay small enough for the instruction cache.
    const uint32_t my_table = tables + (F::TK == kRow ? (warp >> 1) * F::TABLE + (warp & 1) * 128 : F::TK == kWarp ? warp * F::TABLE : quad * F::BUFS * F::TABLE);
    const uint32_t lane_off = F::D == 4 ? (lane & 15) * 8 : lane * 4;
    const uint32_t pat = ((my_table >> 12) & 0xFu) * 0x10101010u;
    const uint32_t swz = F::RB == 32 ? ((qt >> 2) & 1) << 4 : F::RB == 64 ? ((qt >> 1) & 3) << 4 : F::RB == 128 ? (qt & 7) << 4 : 0;
    const uint32_t tmem_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t tmem_a = tmem_lane + kAOff + quad * 64, tmem_d = tmem_lane + quad * 32;
    const uint32_t red_at = base + a.red_off + (quad * red_cols * kTileRows + qt) * 4;
    uint32_t tbl = my_table + lane_off;
    int half = 0;
    uint32_t ph_i = 0, ph_red = 1;

    int block_left = 0;   // units left in the codebook block
    // The running sum, and one that is complete but not yet read (`pend_*`): it is read a unit or two later, when the tensor
    // core has caught up.
    int st = 0, seg = 0, seg_left = 0, seg_units = 0, fin_at = -1;
    bool open_sum = false, first_sum = true, more = true, pend_last = false, pend_zero = false;
    float pend_scale = 1.f, block_scale = 1.f;
    const __half* gs = nullptr;   // int4 codebooks: the scales of the thread's row
    const uint8_t* codes = nullptr;          // normalisation: the codes of the thread's row,
    const unsigned short* lut = nullptr;     // the scales of its blocks,
    uint32_t code_word = 0;                  // and the codes of the next unit, requested a unit ahead
    auto request_codes = [&](int unit) {
      if constexpr (F::NORM) {
        static_assert(!F::NORM || F::UC == 128);
        const uint8_t* p = codes + unit * (F::UC / 2 >> a.norm_shift);
        code_word = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < (F::UC / 2 >> a.norm_shift)) code_word |= load_weight<1, true>(p + i) << (8 * i);
      }
    };

#pragma unroll 1
    for (;;) {
      if (F::RW == 1 && st == fin_at) {
        // ---- read a finished sum ----
        fin_at = -1;
        const int buf = (seg - 1) & 1;
        if (!pend_zero) {
          wait_phase(d_full + 8 * buf, ((seg - 1) >> 1) & 1, tries);
          __syncwarp();
          tc_fence_after();
        }
        // (columns from the batch on are not used by anyone)
        if (first_sum) wait_phase(red_empty, ph_red, tries);
        __syncwarp();
#pragma unroll 1
        for (int n = 0; n < red_cols; n += 4) {
          uint32_t v[1][4];
          tc_load4(tmem_d + buf * 16 + n, v[0]);
          tc_load_wait(v);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t at = red_at + (n + i) * kTileRows * 4;
            const float before = lds32f(at);
            sts32f(at, fmaf(pend_scale, pend_zero ? 0.f : __uint_as_float(v[0][i]), first_sum ? 0.f : before));
          }
        }
        if (pend_last) {
          __syncwarp();
          if (lane == 0) mbar_arrive(red_full);
          ph_red ^= 1u;
        }
        tc_fence_before();
        first_sum = pend_last;
        if (!more) break;
      }
      if (seg_left == 0) {
        // ---- a sum ends (all but the first time), the next one begins ----
        if (open_sum) {
          open_sum = false;
          pend_last = u == end;
          if (F::RW == 1) {
            pend_zero = seg_units == 0;
            pend_scale = block_scale;
            if (!pend_zero) ++seg;
            fin_at = st;
          }
          if (pend_last) {   // to the next fragment
            if (!f.valid) {
              if (F::RW > 1) break;
              more = false;
              continue;
            }
            tile = f.tile;
            f.range(a, quad, u, end);
            f.next(a);
            bcol = divide(u, a.block_inv) - 1;
            block_left = 0;
          }
        }
        open_sum = true;
        seg_units = seg_left = (by_block ? min(end, (bcol + 2) * block_units) : end) - u;
        if (seg_left == 0) continue;   // nothing of the fragment is this quad's
        if (F::RW == 1 && fin_at >= 0) fin_at = st + min(F::STAGES == 2 ? 2 : 1, seg_left);
        if constexpr (F::I4) {
          const Segment& sg = a.seg[segment_of(a, tile)];
          gs = sg.scale + static_cast<long long>(min((tile - sg.tile0) * kTileRows + qt, sg.N - 1)) * (a.K / 128);
        }
        if constexpr (F::NORM) {
          const int row = min((tile - a.seg[0].tile0) * kTileRows + qt, a.seg[0].N - 1);
          codes = a.codes + static_cast<long long>(row) * a.code_row;
          lut = a.lut + static_cast<long long>(row / a.Br) * a.blocks_per_row * 16;
          request_codes(u);
        }
      }
      uint32_t nscales[F::NORM ? F::UC / 16 : 1];   // normalisation: the scale of every 16 columns, twice
      if constexpr (F::NORM) {
        const unsigned short* l = lut + divide(u, a.block_inv) * 16;
#pragma unroll
        for (int i = 0; i < F::UC / 16; ++i) nscales[i] = load_weight<2, true>(l + ((code_word >> (4 * (16 * i >> a.norm_shift))) & 15u)) * 0x10001u;
        if (seg_left > 1) request_codes(u + 1);
      }
      uint32_t scales[F::STAGES / 2];   // int4 codebooks: of the unit's groups of 128 columns
      if constexpr (F::I4) {
#pragma unroll
        for (int i = 0; i < F::STAGES / 2; ++i)
          scales[i] = __ldg(reinterpret_cast<const unsigned short*>(gs) + u * (F::UC / 128) + i) * 0x10001u;
      }
      wait_phase(idx_full + 8 * islot, ph_i, tries);
      uint32_t w[F::RB / 4];
      {
        const uint32_t row_at = idx_at + islot * F::IDX_BYTES + qt * F::RB;
#pragma unroll
        for (int i = 0; i < F::RB / 16; ++i) {   // 128-bit reads, conflict-free at every row pitch in use
          const uint4 v = lds128(row_at + ((16u * i) ^ swz));
          w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
        }
        if (++islot == D) { islot = 0; ph_i ^= 1u; }
      }
      if (block_left == 0) {   // another codebook block: its entries were requested a block ago
        ++bcol;
        block_left = (bcol + 1) * block_units - u;
        if (!asked) {
          const Segment& sg = a.seg[segment_of(a, tile)];
          tb.open(a, sg, (tile - sg.tile0) * kTileRows, qt);
          tb.request(a, bcol);
        }
        if constexpr (F::TK == kRow) {
          tb.write(a, my_table, qt);   // (a lane reads what it wrote itself)
          if (by_block) block_scale = tb.scale();
        } else if constexpr (F::TK == kWarp) {
          __syncwarp();   // every lane has left the old table
          tb.write(a, my_table, qt);
          __syncwarp();
        } else if constexpr (F::BUFS == 2) {
          tb.write(a, my_table + half * F::TABLE, qt);   // last used two blocks ago
          quad_barrier(quad);
          tbl = my_table + half * F::TABLE + lane_off;
          half ^= 1;
        } else {
          quad_barrier(quad);
          tb.write(a, my_table, qt);
          quad_barrier(quad);
        }
        fence_value(tbl);   // look-ups of the new block stay behind the writes
        // request the next block: of this fragment, or the first of the next one
        asked = false;
        if ((bcol + 1) * block_units < end) {
          tb.request(a, bcol + 1);
          asked = true;
        } else if (f.valid) {
          int nu, nend;
          f.range(a, quad, nu, nend);
          if (nu < nend) {
            const Segment& sg = a.seg[segment_of(a, f.tile)];
            tb.open(a, sg, (f.tile - sg.tile0) * kTileRows, qt);
            tb.request(a, divide(nu, a.block_inv));
            asked = true;
          }
        }
      }
      --block_left;
      auto stage = [&](auto jc) {
        constexpr int J = decltype(jc)::value;
        uint32_t r[32];
        gather<F, J>(r, w, tbl, pat);
        if constexpr (F::I4) {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = mul_f16x2(r[i], scales[J / 2]);
        }
        if constexpr (F::NORM) {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = mul_f16x2(r[i], nscales[4 * J + i / 8]);
        }
        // (the place's use number is st * STAGES / 2 + J / 2)
        wait_phase(a_empty + 8 * (J & 1), F::STAGES == 2 ? (st & 1) ^ 1 : ((J >> 1) & 1) ^ 1, tries);
        __syncwarp();
        tc_fence_after();
        tc_store32(tmem_a + (J & 1) * 32, r);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full + 8 * (J & 1));
      };
      [&]<int... J>(std::integer_sequence<int, J...>) {
        (stage(std::integral_constant<int, J>{}), ...);
      }(std::make_integer_sequence<int, F::STAGES>{});
      ++u;
      --seg_left;
      ++st;
    }
  }
  if (tries == 0 && lane == 0) atomicAdd(a.error_flag, 1);   // a wait of this warp ran out
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kResultsWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols));
  // ---- the shared tiles whose last share came from this CTA: every share is added, in CTA order ----
  const uint32_t listed = lds32_now(n_last);
  for (uint32_t i = 0; i < listed; ++i) {
    const uint4 sum = lds128(last_tile + 16 * i);
    const Segment& sg = a.seg[sum.x];
    const int r = tid & 127, row = sum.y + r, part_floats = a.batch * kTileRows;
    const float* p = a.ws_part + static_cast<long long>(sum.z) * part_floats + r;
    const int others = (sum.z & 1 ? -1 : 0) * part_floats;   // (the CTAs behind the first keep their shares in their first slots)
    constexpr int G = F::THREADS / 128;
#pragma unroll 1
    for (int n = tid >> 7; n < a.batch && tid < G * 128; n += 2 * G) {
      float s[2] = {};
#pragma unroll 1
      for (uint32_t k0 = 0; k0 < sum.w; k0 += 4) {   // (a load takes about 1000 clocks: eight at a time)
        float v[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            v[k][i] = 0.f;
            if (k0 + k < sum.w && n + i * G < a.batch)
              v[k][i] = __ldcg(p + (2 * (k0 + k)) * part_floats + (k0 + k ? others : 0) + (n + i * G) * kTileRows);
          }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          s[0] += v[k][0];
          s[1] += v[k][1];
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (row < sg.N && n + i * G < a.batch) sg.Y[static_cast<long long>(n + i * G) * sg.N + row] = __float2half_rn(s[i]);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
int env_int(const char* name, int dflt) {
#ifdef VQ_TUNING
  if (const char* e = getenv(name)) return atoi(e);
#else
  (void)name;
#endif
  return dflt;
}

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Norm {
  const void *codes, *lut;
  int cols;
};

// Without a workspace (normalised calls have none) every tile is one CTA's.
template <class F>
vq_status launch(const StreamCall& call, cudaStream_t s, const Norm* norm = nullptr) {
  auto kern = tile_kernel<F>;
  constexpr size_t kSmemCap = 227 * 1024;
  static int attr_set[kMaxDevices] = {};
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return VQ_ERR_CUDA;
  if (device_sms(&sms) != VQ_OK) return VQ_ERR_CUDA;
  if (!__atomic_load_n(&attr_set[dev], __ATOMIC_ACQUIRE)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemCap)) != cudaSuccess) return VQ_ERR_CUDA;
    __atomic_store_n(&attr_set[dev], 1, __ATOMIC_RELEASE);
  }
  const Geometry& g = call.g;
  TileArgs a = {};
  if (device_error_counter(&a.error_flag) != VQ_OK) return VQ_ERR_CUDA;
  a.n_seg = call.n_seg;
  a.K = g.K;
  a.batch = call.batch;
  a.blocks_per_row = g.blocks_per_row;
  a.Br = g.Br;
  a.Bc = g.Bc;
  a.cb_int8 = g.cb_int8;
  a.S = g.K / F::UC;   // (block columns, and so K, are whole units: tile_covers)
  a.steps = (a.S + kQuads - 1) / kQuads;
  int tiles = 0;
  long long rows_total = 0;
  for (int i = 0; i < call.n_seg; ++i) {
    a.seg[i].cb = call.cb[i];
    a.seg[i].scale = call.scale[i];
    a.seg[i].Y = call.Y[i];
    a.seg[i].N = call.N[i];
    a.seg[i].tile0 = tiles;
    tiles += (call.N[i] + kTileRows - 1) / kTileRows;
    rows_total += call.N[i];
  }
  if (static_cast<long long>(tiles) * a.S > 0x3fffffff) return VQ_ERR_UNSUPPORTED;

  // ---- shared memory: activations, indices, sums, barriers, then the tables on their boundary ----
  const int x_rows = call.batch <= 8 ? 8 : 16;
  a.x_row_bytes = x_rows * 128;
  a.x_bytes = F::STAGES * a.x_row_bytes;
  auto plan = [&](int D) {
    a.D = D;
    a.idx_off = kQuads * D * a.x_bytes;
    a.red_off = a.idx_off + kQuads * D * F::IDX_BYTES;
    a.bar_off = a.red_off + kQuads * a.red_cols * kTileRows * 4;
    a.front_bytes = a.bar_off + kBarBytes;
    // (dynamic shared memory starts 1024 bytes into the window)
    return round_up(1024 + a.front_bytes, F::ALIGN) - 1024 + F::TABLES;
  };
  // row tables: columns of sums handed over in shared memory
  a.red_cols = F::RW == 1 ? (call.batch + 3) / 4 * 4 : 0;
  int D = env_int("VQ_TD", kMaxDepth);
  while (D > 2 && plan(D) > kSmemCap) --D;
  size_t smem_bytes = plan(D);
  if (smem_bytes > kSmemCap || D < 2 || D > kMaxDepth) return VQ_ERR_UNSUPPORTED;
  if (smem_bytes < 120 * 1024) smem_bytes = 120 * 1024;   // one CTA per SM: the next kernel's go where one has left

  // ---- persistent CTAs: whole tiles first, the steps of the left-over tiles shared evenly ----
  const long long steps = static_cast<long long>(tiles) * a.steps;
  long long P = sms < kMaxStreamCtas ? sms : kMaxStreamCtas;
  if (P > steps) P = steps;
  // As many CTAs for every tile, and so one piece of one tile for each, where that costs at most half a step more than pieces
  // that end anywhere: a second piece costs its own tables, sums and share of a tile.
  if (norm && P > tiles) P = tiles;
  for (long long k = P / tiles; k >= 1 && !norm; --k)
    if (a.steps % k == 0) {
      if (2 * P * (a.steps / k) <= 2 * steps + P * env_int("VQ_SLACK", 3)) P = tiles * k;
      break;
    }
#ifdef VQ_TUNING
  if (env_int("VQ_TP", 0) && P > env_int("VQ_TP", 0)) P = env_int("VQ_TP", 0);
#endif
  a.q = static_cast<int>(tiles / P);
  const int left = static_cast<int>(tiles - a.q * P);
  const long long tail = norm ? 0 : static_cast<long long>(left) * a.steps;
  a.extra = norm ? left : 0;
  a.tail_tile0 = static_cast<int>(a.q * P);
  if (steps * a.steps >= (1LL << 31) || steps * (tail + 1) >= (1LL << 31) || static_cast<long long>(a.S) * a.S >= (1LL << 31)) return VQ_ERR_UNSUPPORTED;   // divide()
  // A tile is shared by eight CTAs at most where every CTA has whole ones.
  long long Pt = P;
  const int cap = env_int("VQ_CAP", 8);
  if (a.q > 0 && Pt > static_cast<long long>(left) * cap) Pt = static_cast<long long>(left) * cap;
  if (tail > 0 && tail < Pt) Pt = tail;
  a.sharers = static_cast<int>(Pt);
  a.share = Pt ? static_cast<int>(tail / Pt) : 0;
  a.longer = Pt ? static_cast<int>(tail % Pt) : 0;
  auto inverse = [](long long d) { return d > 1 ? static_cast<unsigned>(((1LL << 32) + d - 1) / d) : 0u; };
  a.steps_inv = inverse(a.steps);
  a.share_inv = inverse(a.share);
  a.share1_inv = inverse(a.share + 1);
  a.block_inv = inverse(g.Bc / F::UC);
  if (norm) {
    a.codes = static_cast<const uint8_t*>(norm->codes);
    a.lut = static_cast<const unsigned short*>(norm->lut);
    a.code_row = (g.K / norm->cols + 1) / 2;
    while ((1 << a.norm_shift) < norm->cols) ++a.norm_shift;
  } else {
    // counters at the start, partial sums at the end of the workspace: a call with fewer rows then never writes
    // sums where one with more rows keeps its counters
    const size_t ticket_bytes = stream_ticket_bytes(rows_total);
    if (static_cast<size_t>(tiles) * sizeof(int) > ticket_bytes) return VQ_ERR_UNSUPPORTED;
    const size_t part_ws = static_cast<size_t>(P) * 2 * kTileRows * call.batch * sizeof(float);
    const size_t total_ws = stream_workspace_bytes(rows_total, call.batch);
    if (ticket_bytes + part_ws > total_ws) return VQ_ERR_UNSUPPORTED;
    if (!call.ws || call.ws_bytes < total_ws) return VQ_ERR_WORKSPACE;
    a.ws_ticket = static_cast<int*>(call.ws);
    a.ws_part = reinterpret_cast<float*>(static_cast<char*>(call.ws) + (total_ws - part_ws));
  }

  TileMaps maps;
  for (int i = 0; i < call.n_seg; ++i) {
    const uint64_t dims[2] = {static_cast<uint64_t>(g.stride), static_cast<uint64_t>(call.N[i])};
    const uint64_t strides[1] = {static_cast<uint64_t>(g.stride)};
    const uint32_t box[2] = {F::RB, kTileRows};
    if (encode_tensor_map(&maps.idx[i], call.idx[i], 1, 2, dims, strides, box, F::SWIZZLE) != VQ_OK) return VQ_ERR_CUDA;
  }
  for (int i = call.n_seg; i < kMaxSegments; ++i) maps.idx[i] = maps.idx[0];
  {
    const uint64_t dims[3] = {64, static_cast<uint64_t>(call.batch), static_cast<uint64_t>(g.K / 64)};
    const uint64_t strides[2] = {static_cast<uint64_t>(g.K) * 2, 128};
    const uint32_t box[3] = {64, static_cast<uint32_t>(x_rows), F::STAGES};
    if (encode_tensor_map(&maps.x, call.X, 2, 3, dims, strides, box, 2) != VQ_OK) return VQ_ERR_CUDA;
  }

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(P), 1, 1);
  cfg.blockDim = dim3(F::THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = env_int("VQ_PDL", 1) ? 1 : 0;
#ifdef VQ_TUNING
  if (env_int("VQ_VERBOSE", 0)) fprintf(stderr, "tile launch: grid %d depth %d smem %zu tiles %d S %d steps %d q %d share %d+%d\n", (int)P, D, smem_bytes, tiles, a.S, a.steps, a.q, a.share, a.longer);
#endif
  if (cudaLaunchKernelEx(&cfg, kern, maps, a) != cudaSuccess) return VQ_ERR_CUDA;
  return check_launch();
}

}  // namespace

// Codebook blocks that are whole units of columns (so K is one too).
bool tile_covers(const Geometry& g) {
  if (g.d == 2 && g.b == 4) return !g.cb_int4 && g.Bc % 256 == 0;
  if (g.d == 2 && g.b == 5) return g.Bc % 256 == 0 && (g.Br % 32 == 0 || (!g.cb_int4 && (g.Br == 4 || g.Br == 8 || g.Br == 16)));
  if (g.d == 2 && g.b == 6) return g.Bc % 128 == 0 && g.Br % 32 == 0;
  return g.d == 4 && g.b == 8 && g.Bc % 128 == 0 && g.Br % kTileRows == 0 && !g.cb_int4;
}

// Which calls this kernel serves.  Its time hardly depends on the batch (one pass over the weights for 1..16 sequences), but a call
// costs about 4.5 us before and behind its look-ups, the cluster kernels' 3.3.  So it takes over above a number of weights (in 2^20,
// "line") that falls with the batch and with the columns: long rows give a CTA one long piece, where the cluster kernels stage
// activations and split K over eight CTAs at most.  One layer and a group of as many rows are planned alike, so they share their lines; the
// persistent kernel, which takes row tables of 8192 rows or of a group, is another rival than the cluster kernels and has lines of its own.
// The lines are drawn from 108394 calls (24 formats, 1024 to 28672 columns, 1.5 to 320 x 2^20 weights, one layer or three, batches 1 to 16),
// each timed here, in every other kernel, and in the library before this kernel had one CTA per SM: where nearly no call is more
// than 3 % slower than it was then, not where the mean is lower.  820 of them are (0.8 %; of calls that one kernel serves on both sides
// 1.4 % differ as much); together they take 0.70 of the time of then.  Both sides' times (us, others / here):
//   128-row blocks, 6 bits  4096 x 4096 b1 5.8/6.7, b8 8.4/7.1; 12288 x 4096 b1 10.9/12.4, b8 13.6/13.1; 19712 x 5120 b16 53/22.7
//   32-row blocks, 6 bits   6144 x 4096 b1 7.7/9.0, b16 15.0/9.8; 32768 x 1024 b1 10.9/8.8, b16 12.5/13.9
//   4-D                     49152 x 1024 b3 10.9/11.5; 19712 x 5120 b3 25.9/15.3, b8 34.2/16.3
//   row tables, 2048-column blocks, against the persistent kernel  8192 x 4096 b6 8.5/9.5; 8192 x 8192 b1 10.2/13.0, b9 16.5/13.9;
//                           24576 x 8192 b1 26.4/26.5, b6 30.3/27.8, b9 38.6/28.3
// Left: 4-D and 5 bits with 1024 to 1536 columns and 64 x 2^20 weights or more, up to 1.15 times the time of then at batch 16, in
// every kernel there is now.
constexpr unsigned char kNever = 255;
constexpr int kLineCols[5] = {1500, 2600, 3700, 4800, 5500};        // columns: below the first, the second, ..., from the last on
constexpr int kRowLineCols[5] = {1500, 2600, 4800, 5500, 10000};
struct Lines { unsigned char at[4][6]; };      // batch 1-2, 3-5, 6-8, 9-16
struct RowLines { unsigned char at[6][6]; };   // batch 1-2, 3-5, 6-7, 8, 9-10, 11-16
// against the cluster kernels: blocks of 128 k rows and 6 bits, of 32 and 64 rows and 6 bits (each: 16- and 8-bit, 4-bit codebooks), 5 bits, 4-D
constexpr Lines kTall6 = {{{128, 28, 32, 56, 64, 3}, {128, 24, 32, 56, 3, 3}, {32, 5, 20, 5, 0, 0}, {}}};
constexpr Lines kTall6Int4 = {{{80, 24, 0, 28, 0, 0}, {56, 24, 0, 28, 0, 0}, {0, 3, 0, 0, 0, 0}, {}}};
constexpr Lines kWarp6 = {{{80, 28, 32, 56, 0, 0}, {80, 24, 0, 28, 0, 0}, {56, 3, 0, 0, 0, 0}, {0, 0, 0, 3, 0, 0}}};
constexpr Lines kWarp6Int4 = {{{kNever, 56, 32, 56, 64, 0}, {128, 56, 32, 56, 0, 0}, {56, 3, 0, 28, 0, 0}, {}}};
constexpr Lines k5 = {{{12, 20, 28, 36, 3, 0}, {3, 20, 5, 5, 0, 0}, {3, 3, 3, 3, 0, 0}, {0, 3, 0, 0, 0, 0}}};
constexpr Lines k5Int4 = {{{3, 20, 3, 36, 0, 0}, {0, 3, 3, 3, 0, 0}, {0, 3, 0, 0, 0, 0}, {0, 3, 0, 0, 0, 0}}};
constexpr Lines k4D = {{{80, 24, 0, 0, 0, 0}, {80, 12, 0, 0, 0, 0}, {3, 3, 0, 0, 0, 0}, {}}};
// against the pair-table kernel: blocks of 4, of 8 and 16 rows; rows or columns that the cluster kernels do not take, 5 bits and 6
constexpr Lines kSmall4 = {{{}, {12, 0, 0, 0, 0, 0}, {12, 3, 0, 0, 0, 0}, {3, 5, 3, 0, 0, 0}}};
constexpr Lines kSmall = {{{0, 24, 24, 20, 0, 0}, {12, 24, 24, 20, 0, 0}, {12, 24, 24, 20, 0, 0}, {12, 12, 8, 8, 0, 0}}};
constexpr Lines kRagged5 = {{{12, 24, 20, 3, 0, 0}, {12, 24, 20, 3, 0, 0}, {12, 24, 20, 3, 0, 0}, {3, 5, 8, 3, 0, 0}}};
constexpr Lines kRagged6 = {{{12, 12, 0, 0, 0, 0}, {12, 0, 0, 0, 0, 0}, {8, 0, 0, 0, 0, 0}, {3, 0, 0, 0, 0, 0}}};
// row tables, blocks of 256, of up to 960 and of more columns: against the cluster kernels, against the persistent kernel
constexpr RowLines kRows[3][2] = {
    {{{{kNever, kNever, kNever, 24, 48, 56}, {0, 3, 20, 0, 5, 5}, {0, 3, 0, 0, 0, 0}, {}, {kNever, 0, 5, 0, 0, 0}, {}}},
     {{{kNever, 56, 0, 0, 0, 0}, {}, {}, {}, {}, {}}}},
    {{{{kNever, kNever, kNever, kNever, kNever, 80}, {0, kNever, 20, 24, 48, 8}, {0, 3, 20, 0, 3, 0}, {0, 3, 0, 0, 0, 0}, {0, 5, 3, 5, 0, 0}, {}}},
     {{{kNever, kNever, kNever, kNever, kNever, kNever}, {kNever, kNever, kNever, 32, kNever, kNever}, {3, 56, 40, 0, 80, kNever},
       {3, 20, 24, 0, 48, 160}, {0, 20, 28, 0, 0, 0}, {0, 5, 0, 0, 0, 0}}}},
    {{{{kNever, kNever, kNever, kNever, 56, 80}, {0, kNever, 20, 24, 48, 24}, {0, 5, 5, 0, 3, 0}, {0, 3, 0, 0, 0, 0}, {0, 5, 5, 5, 5, 0},
       {0, 5, 0, 0, 0, 0}}},
     {{{kNever, kNever, kNever, kNever, kNever, kNever}, {kNever, kNever, kNever, kNever, kNever, kNever}, {5, 20, 40, 0, 80, kNever},
       {0, 20, 24, 0, 56, 160}, {0, 56, 0, 0, 0, 0}, {0, 12, 0, 0, 0, 0}}}},
};

bool tile_preferred(const Geometry& g, const int* N, int n_seg, int batch) {
  if (!tile_covers(g)) return false;
#ifdef VQ_TUNING
  if (env_int("VQ_TILE", -1) >= 0) return env_int("VQ_TILE", 0) != 0;
#endif
  long long rows = 0;
  bool whole = blockcb_covers(g);   // do the cluster kernels take the call?
  for (int i = 0; i < n_seg; ++i) {
    rows += N[i];
    whole = whole && N[i] % kTileRows == 0;
  }
  const long long w = (rows * g.K) >> 20;   // weights of the call, in 2^20
  auto column = [&](const int (&limits)[5]) {
    int k = 0;
    while (k < 5 && g.K >= limits[k]) ++k;
    return k;
  };
  int line;
  if (g.d == 2 && g.b == 4) {
    const RowLines& l = kRows[g.Bc < 512 ? 0 : g.Bc < 1024 ? 1 : 2][n_seg > 1 || rows >= 8192];
    line = l.at[batch <= 2 ? 0 : batch <= 5 ? 1 : batch <= 7 ? 2 : batch == 8 ? 3 : batch <= 10 ? 4 : 5][column(kRowLineCols)];
  } else {
    const bool pairs = g.b == 5 && g.Br < 32;
    if (!pairs && !whole && (g.d == 4 || g.cb_int4)) return true;   // (0.2 to 0.8 of the pair-table kernel's time at every size)
    const Lines& l = pairs ? (g.Br == 4 ? kSmall4 : kSmall)
                   : !whole ? (g.b == 5 ? kRagged5 : kRagged6)
                   : g.d == 4 ? k4D
                   : g.b == 5 ? (g.cb_int4 ? k5Int4 : k5)
                   : g.Br % kTileRows == 0 ? (g.cb_int4 ? kTall6Int4 : kTall6) : (g.cb_int4 ? kWarp6Int4 : kWarp6);
    line = l.at[batch <= 2 ? 0 : batch <= 5 ? 1 : batch <= 8 ? 2 : 3][column(kLineCols)];
  }
  return line != kNever && w >= line;
}

vq_status launch_gemm_tile(const StreamCall& call, cudaStream_t s) {
  const Geometry& g = call.g;
  if (!tile_covers(g) || call.n_seg < 1 || call.n_seg > kMaxSegments) return VQ_ERR_UNSUPPORTED;
  if (g.d == 2 && g.b == 4) return launch<Fmt<2, 4, kRow, 1, false>>(call, s);
  if (g.d == 4) return launch<Fmt<4, 8, kCta, 128, false>>(call, s);
  if (g.Br % kTileRows == 0) {
    if (g.b == 6) return g.cb_int4 ? launch<Fmt<2, 6, kCta, 128, true>>(call, s) : launch<Fmt<2, 6, kCta, 128, false>>(call, s);
    return g.cb_int4 ? launch<Fmt<2, 5, kCta, 128, true>>(call, s) : launch<Fmt<2, 5, kCta, 128, false>>(call, s);
  }
  if (g.Br % 32 == 0) {
    if (g.b == 6) return g.cb_int4 ? launch<Fmt<2, 6, kWarp, 32, true>>(call, s) : launch<Fmt<2, 6, kWarp, 32, false>>(call, s);
    return g.cb_int4 ? launch<Fmt<2, 5, kWarp, 32, true>>(call, s) : launch<Fmt<2, 5, kWarp, 32, false>>(call, s);
  }
  if (g.Br == 16) return launch<Fmt<2, 5, kWarp, 16, false>>(call, s);
  if (g.Br == 8) return launch<Fmt<2, 5, kWarp, 8, false>>(call, s);
  return launch<Fmt<2, 5, kWarp, 4, false>>(call, s);
}

// Block-wise normalisation: sub-rows of 16, 32 or 64 columns, blocks of a multiple of 32 rows with 6-bit indices; one layer.
vq_status launch_gemm_tile_norm(const Geometry& g, const LayerPtrs& p, const void* norm_codes, const void* norm_lut, int norm_block_cols,
                                const __half* X, __half* Y, int batch, cudaStream_t s) {
  if (!norm_codes || !norm_lut || !tile_covers(g) || g.d != 2 || g.b != 6 || g.cb_int4) return VQ_ERR_UNSUPPORTED;
  if (norm_block_cols != 16 && norm_block_cols != 32 && norm_block_cols != 64) return VQ_ERR_UNSUPPORTED;
  // A tile is one CTA's whole: worth it where the tiles fill the SMs.  Both kernels' times in us, fitted to 20160 calls (six formats, 256 to
  // 14336 columns, 480 to 57344 rows, batches 1 to 16), with a twentieth to spare: of the 8571 calls taken 109 are more than 3 % slower than
  // in the pair-table kernel.  Sub-rows of 32, batch 1, 8-bit codebooks of 32 x 256 (pair-table kernel / here): 11008 x 4096 18.9/18.8,
  // 14336 x 4096 24.2/19.4, 37888 x 4096 59.0/34.7, 14336 x 11008 61.3/44.3; 24576 x 1024 11.6/11.8 is left to the other.
  int sms = 0;
  if (device_sms(&sms) != VQ_OK) return VQ_ERR_CUDA;
  const double rounds = ((g.N + kTileRows - 1) / kTileRows + sms - 1) / sms, cols = g.K / 1000., w = static_cast<double>(g.N) * g.K / (1 << 20);
  const double here = 2.75 + 0.06 * batch + rounds * (1.55 + (norm_block_cols == 16 ? 4.7 : 3.9) * cols);
  const double pairs = batch <= 8 ? 4.45 + 0.335 * w + 0.88 * cols : 4.85 + 0.41 * w + 0.88 * cols;
  if (1.05 * here > pairs) return VQ_ERR_UNSUPPORTED;
  StreamCall call = {};
  call.g = g;
  call.n_seg = 1;
  call.idx[0] = p.idx;
  call.cb[0] = p.cb;
  call.scale[0] = p.scale;
  call.Y[0] = Y;
  call.N[0] = g.N;
  call.X = X;
  call.batch = batch;
  const Norm norm = {norm_codes, norm_lut, norm_block_cols};
  return g.Br % kTileRows == 0 ? launch<Fmt<2, 6, kCta, 128, false, true>>(call, s, &norm) : launch<Fmt<2, 6, kWarp, 32, false, true>>(call, s, &norm);
}

}  // namespace vq
