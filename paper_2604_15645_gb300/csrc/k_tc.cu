// Tensor-core jet GEMMs for sm_103a: tcgen05.mma with operands staged in shared
// memory by TMA (cp.async.bulk.tensor, 128-byte swizzle) and FP32 accumulators in
// tensor memory, read back with tcgen05.ld for the fused epilogues.
//
// Data layout (shared with the CUDA-core path): every jet matrix is tile-major,
// [NC/256][features][256]: a tile holds 64 points, its 256 columns blocked by jet
// row ([values | d1 | d2 | d2nd], see jet.cuh).  The three GEMMs of a hidden layer are
//   forward  Z^T[fout][NC]    = W[fout][fin]   . A^T[fin][NC]       (B operand MN-major)
//   adjoint  Abar^T[fin][NC]  = W^T[fin][fout] . Zbar^T[fout][NC]   (B operand MN-major)
//   weights  dW[fout][fin]    = Zbar^T[fout][NC] . (A^T[fin][NC])^T (both K-major, split over NC)
// so a 128-row accumulator tile puts one feature in each TMEM lane and the 256
// columns of one point tile in its columns: each epilogue thread owns one feature
// of whole points and applies the tanh jet rule (or its adjoint) without any
// cross-thread exchange.  On the BF16 path the forward also adds the low half of
// the weights (all columns) and of the input's value rows (the 64 value columns).
//
// TF32 (kind::tf32) reads both operands K-major only, so its forward and adjoint take
// the jets from a point-major copy [NC][features] (written by the epilogue of the
// layer before) and add both truncation remainders: W_hi B + W_lo B + W_hi B_lo, with
// B_lo = B - tf32(B) computed in shared memory by two converter warps.
//
// Warp roles per CTA (320 threads, 384 with converters, 352 in pairs, one CTA per SM,
// persistent):
//   warp 0     TMA producer (one lane)
//   warp 1     TMEM allocator + MMA issuer (one lane)
//   warps 2-9  epilogue; warp w reads TMEM lanes 32*(w%4) .. +31 and handles the
//              points 32*((w-2)/4) .. +31 of the tile, 16 at a time
//   warps 10-11 (TF32 forward / adjoint only) B_lo converters
//   warp 10    (pairs only) output stores
// Two accumulator buffers of 256 columns let the epilogue of one tile overlap the
// MMAs of the next.  Every mbarrier wait is bounded (global timer); on expiry the
// CTA latches PINN_ERR_TIMEOUT in the status word, stops issuing work, waits for
// its own copies in flight, frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <new>
#include <type_traits>
#include <vector>

#include "fwd_route.h"
#include "jet.cuh"
#include "ptx.cuh"
#include "tc.h"

namespace pinn {

namespace {

constexpr int BM = 128;          // accumulator rows (TMEM lanes)
constexpr int BN = 256;          // accumulator columns per buffer
constexpr int EPI_WARPS = 8;     // two warps per TMEM lane quadrant, each on 32 of a tile's 64 points
constexpr uint64_t WAIT_NS = 2000000000ull;   // default bound on any single wait: 2 s

enum TcMode { TC_FWD = 0, TC_ADJ = 1, TC_DW = 2, TC_STORE = 3 };

// Shared-memory matrix descriptor (tcgen05), 128- or 64-byte swizzle, version 1.
template <int SWIZZLE = 128>
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version for tcgen05
  d |= (uint64_t)(SWIZZLE == 128 ? 2 : 4) << 61;   // SWIZZLE_128B / SWIZZLE_64B
  return d;
}
// Instruction descriptor: FP32 accumulate, A/B format (1 = BF16, 2 = TF32),
// A K-major, B K-major (b_mn = 0) or MN-major (b_mn = 1), N columns, M rows.
__host__ __device__ constexpr uint32_t make_idesc(uint32_t fmt, uint32_t b_mn, uint32_t n = BN, uint32_t m = BM) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | (b_mn << 16) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

struct TcParams {
  int M;               // valid accumulator rows (features, or dW rows)
  int N;               // valid columns (NC for fwd/adj/store, fin for dW)
  int K;               // reduction length (fin / fout for fwd / adj, NC for dW)
  int m_tiles, n_tiles, k_iters;
  int nsplit, kps;     // dW: K splits and K iterations per split
  int64_t NC;          // leading dimension of feature-major matrices
  EpiArgs e;
  float* out32;        // dW partials / selftest output
  int* status;
  int wlo_values_only; // forward: W_lo . B on the 64 value columns only (PINN_FLAG_BF16_VALUE_SPLIT)
  uint64_t wait_ns;    // bound on every mbarrier wait (WAIT_NS)
  int stall;           // test hook: the MMA issuer first waits on a barrier nothing arrives on (fused
                       // adjoint: no activation tile comes)
};

// One GEMM of a grouped launch: its tensor maps (the GEMM kernel's four, or the fused
// adjoint's three), its parameters, and the blocks of the grouped grid it owns.  Each
// GEMM keeps the CTA count and work split it has when launched alone.
struct TcGroupEntry {   // 128-byte aligned (CUtensorMap)
  CUtensorMap map[4];
  TcParams p;
  int block0;   // first block of the grouped grid that runs this GEMM
  int grid;     // its block count
};

// Orders this thread's later TMA reads of the entry's tensor maps after the writes that
// put them in global memory (the table is rewritten by the host between captures).
__device__ __forceinline__ void acquire_maps(const TcGroupEntry& g, int nmaps) {
  for (int i = 0; i < nmaps; ++i)
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&g.map[i]) : "memory");
}

// The entry that owns block b: the last one whose first block is <= b (block0 ascends).
__device__ __forceinline__ int group_of_block(const TcGroupEntry* __restrict__ tab, int n, int b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].block0 <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Where a CTA sits in the launch: the hardware indices of a single launch (read where
// used, as a plain kernel would), or its share of a grouped launch.
struct SingleGrid {
  static constexpr bool PAIR = false;
  __device__ __forceinline__ int bx() const { return (int)blockIdx.x; }
  __device__ __forceinline__ int gdim() const { return (int)gridDim.x; }
};
struct GroupShare {
  static constexpr bool PAIR = false;
  int b, g;
  __device__ __forceinline__ int bx() const { return b; }
  __device__ __forceinline__ int gdim() const { return g; }
};

// A single launch in clusters of two CTAs: neighbours, which hold two m-tiles of the same
// column tile and run their MMAs as one of 256 rows (cta_group::2), each staging half of
// the column operand.
struct PairGrid : SingleGrid {
  static constexpr bool PAIR = true;
};
// After an abort: MMAs that are still on their way read shared memory and write tensor memory
// (and, in a pair, copies and arrivals reach the other CTA).  No barrier tells when, but they
// take microseconds: wait them out (1 ms) before any of that memory is given back.
__device__ __forceinline__ void abort_settle() {
  const uint64_t t0 = gtimer();
  while (gtimer() - t0 < 1000000ull) {}
}
// Last step of a CTA of a pair: the other one arrives at this one's barriers and its MMAs
// read this one's shared memory, so neither leaves before both are done.
__device__ __forceinline__ void pair_leave(volatile int* abort_flag) {
  cluster_sync();
  if (threadIdx.x == 0 && *abort_flag) abort_settle();
  cluster_sync();
}

template <bool TF32, int MODE, bool SPLIT, bool PAIR = false>
struct Cfg {
  static constexpr int ES = TF32 ? 4 : 2;
  static constexpr int BKE = 128 / ES;            // K elements per stage (one 128-byte swizzle row)
  static constexpr int UK = TF32 ? 8 : 16;        // K per MMA instruction
  static constexpr int A_BYTES = BM * 128;        // 16 KB
  static constexpr int B_BYTES = BN * 128 / (PAIR ? 2 : 1);   // 32 KB (pair: half of the columns)
  // TF32 forward / adjoint: B from the point-major copy (K-major, 2-D map), its low
  // half computed in shared memory (one B-sized buffer).
  static constexpr bool KPM = TF32 && (MODE == TC_FWD || MODE == TC_ADJ);
  static constexpr int BLOC_BYTES = KPM ? B_BYTES : 0;
  static constexpr int CVT_WARPS = KPM ? 2 : 0;
  static constexpr int NTHREADS = 64 + 32 * (EPI_WARPS + (PAIR ? 1 : CVT_WARPS));
  // Pair: outputs leave by bulk tensor stores through these 128 x 64-point buffers.
  static constexpr int OUT_BUFS = PAIR ? 3 : 0, OUT_BYTES = BM * 128;
  // BF16 forward: low half of the input's value rows, 64 MN-major columns per stage.
  static constexpr bool VLO = (MODE == TC_FWD) && !TF32;
  // (Pair: 32 of them, and the same 32 value columns of the input for a low half of the
  // weights that is limited to the value rows: a CTA provides half of every MMA's columns.)
  static constexpr int BLO_BYTES = VLO ? TILE_PTS * 128 : 0;   // 8 KB
  static constexpr int V_BYTES = BLO_BYTES / 2;
  static constexpr int STAGE = A_BYTES * (SPLIT ? 2 : 1) + B_BYTES + BLO_BYTES;
  static constexpr int STAGES = (MODE == TC_FWD || SPLIT) ? 3 : 4;
  static_assert(STAGES * STAGE + BLOC_BYTES + OUT_BUFS * OUT_BYTES + 1024 + 256 <= 227 * 1024, "shared memory budget");
  static constexpr bool B_MN = (MODE != TC_DW) && !KPM;
  static constexpr int BOXN = 128 / ES;           // MN-major box width (columns)
  static constexpr int NBOX = BN / BOXN / (PAIR ? 2 : 1);
  static constexpr int BOX_BYTES = BKE * 128;     // one MN-major box: BKE rows of 128 bytes
  static constexpr size_t SMEM =
      (size_t)STAGES * STAGE + BLOC_BYTES + OUT_BUFS * OUT_BYTES + 1024 /*align*/ + 256 /*barriers*/;
};

// Point-major copy [NC][M] of one thread's 8 points x 4 rows of feature m: column
// c0 + 64 r + i.  Lanes hold consecutive features, so each store instruction writes
// 128 contiguous bytes.
__device__ __forceinline__ void store_pm8(float* pm, int64_t c0, int M, int m, const float v[4][8]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 8; ++i) pm[(c0 + 64 * r + i) * M + m] = v[r][i];
}

// Forward epilogue of 16 points (accumulators v[row][point]) in packed pairs: bias, tanh
// jet, BF16 rounding (hi, two points per word) and the value row's low half (lo).
template <int MODE>
__device__ __forceinline__ void fwd_pairs(const float (&v)[4][16], float bias, uint32_t (&hi)[4][8], uint32_t (&lo)[8],
                                          uint32_t keep) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    f32x2 z[4], a[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) z[r] = pack2(v[r][2 * i], v[r][2 * i + 1]);
    z[0] = add2(z[0], dup2(bias));
    jet_fwd2<MODE>(z, a);
    float x0, x1;
#pragma unroll
    for (int r = 3; r >= 0; --r) {
      unpack2(a[r], x0, x1);
      const __nv_bfloat162 q = __floats2bfloat162_rn(x0, x1);
      hi[r][i] = *reinterpret_cast<const uint32_t*>(&q) & keep;
    }
    const __nv_bfloat162 q = __floats2bfloat162_rn(x0 - __uint_as_float(hi[0][i] << 16),
                                                   x1 - __uint_as_float(hi[0][i] & 0xffff0000u));
    lo[i] = *reinterpret_cast<const uint32_t*>(&q) & keep;
  }
}

// Adjoint of 8 points in packed pairs: abar in v[row][first ..], the layer's activations as
// raw BF16 pairs in aw[row]; zbar replaces abar.
template <int MODE, int N>
__device__ __forceinline__ void adj_pairs8(float (&v)[4][N], int first, const uint32_t (&aw)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f32x2 a[4], ab[4], zb[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r] = pack2(__uint_as_float(aw[r][i] << 16), __uint_as_float(aw[r][i] & 0xffff0000u));
      ab[r] = pack2(v[r][first + 2 * i], v[r][first + 2 * i + 1]);
    }
    jet_adj_a2<MODE>(a, ab, zb);
#pragma unroll
    for (int r = 0; r < 4; ++r) unpack2(zb[r], v[r][first + 2 * i], v[r][first + 2 * i + 1]);
  }
}

// A lane of an epilogue warp holds a feature's 32 points of a jet row as two 32-byte sectors
// (a: points 0-15, b: 16-31).  After the swap within lane pairs, one access of the even
// lane and one of the odd lane cover 64 consecutive bytes: a and b are the sectors
// 16 (lane & 1) of the pair's even and of its odd feature.  (Its own inverse: loads swap back.)
// Every 128-byte line that an instruction touches takes a cycle of the L1 data path, which
// shared memory uses too: 16 lines per instruction instead of 32.  (Maxwell 5x512 forward
// launches 3.53 -> 3.40 ms.)
__device__ __forceinline__ void pair_swap(uint32_t (&a)[8], uint32_t (&b)[8]) {
  const bool odd = threadIdx.x & 1;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, odd ? a[i] : b[i], 1);
    const uint32_t keep_a = a[i];
    a[i] = odd ? y : keep_a;
    b[i] = odd ? b[i] : y;
  }
}
// Stores 32 points x 4 rows of a warp's features (w[unit][row], BF16 pairs): column pc of tile
// nb, feature m of M (M even, so a pair of lanes is valid together).
__device__ __forceinline__ void store_pairs(__nv_bfloat16* out, uint32_t (&w)[2][4][8], int m, int64_t nb, int M, int pc) {
  __nv_bfloat16* o = out + toff(m & ~1, nb * BN, M) + pc + 16 * (m & 1);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    pair_swap(w[0][r], w[1][r]);
    if (m < M) {
      st_global_256(o + 64 * r, w[0][r]);
      st_global_256(o + 64 * r + TILE_COLS, w[1][r]);
    }
  }
}
__device__ __forceinline__ void store_lo_pairs(__nv_bfloat16* out, uint32_t (&w)[2][8], int m, int64_t nb, int M, int pc) {
  __nv_bfloat16* o = out + loff(m & ~1, nb * TILE_PTS, M) + pc + 16 * (m & 1);
  pair_swap(w[0], w[1]);
  if (m < M) {
    st_global_256(o, w[0]);
    st_global_256(o + TILE_PTS, w[1]);
  }
}
// Calls f with the jet rule as a compile-time constant.
template <typename F>
__device__ __forceinline__ void with_jet_mode(int mode, F&& f) {
  if (mode == JET_NS) f(std::integral_constant<int, JET_NS>{});
  else if (mode == JET_BURGERS) f(std::integral_constant<int, JET_BURGERS>{});
  else f(std::integral_constant<int, JET_MAXWELL>{});
}

// Coordinate terms of a raw first layer's weight gradient, dW_ij = sum_points zbar x_j +
// sum over rows of direction j of zbar_j, in the adjoint epilogues.  Each warp covers 32
// points of a tile for its 32 features: lane i looks up point i's coordinates once per tile
// and the lanes exchange them by shuffles.  (Looking every point up in every lane
// took 0.56 ms more of Maxwell 5x512's four adjoint launches, 3.57 -> 3.01 ms, and 11% of a
// step of 64 networks.)
__device__ __forceinline__ void lane_coords(const EpiArgs& e, int64_t point, float x[3]) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (j < e.dterms) x[j] = point_coord(e.x_res, e.x_ic, e.x_bc, e.n_res, e.n_ic, e.n_bc, point, j);
}
template <int N>
__device__ __forceinline__ void coord_terms(const float (&v)[4][N], const float x[3], int first, int dterms, int mode,
                                            float db[4]) {
  const int nd = (mode == JET_MAXWELL) ? 3 : 2;   // rows 1..nd are first derivatives
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (j < dterms) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        db[1 + j] = fmaf(v[0][i], __shfl_sync(0xffffffffu, x[j], first + i), db[1 + j]);
        if (j < nd) db[1 + j] += v[1 + j][i];
      }
    }
}

// ---- the kernel -----------------------------------------------------------------------
// SINE (BF16 forward / adjoint): the periodic activation sin(w0 z) instead of tanh.  Its
// adjoint cannot be written in the activations (the sign of cos is lost), so the
// forward epilogue also stores the pre-activation jets Z (FP32) and the adjoint
// epilogue evaluates the rule from them.
// The body runs as CTA grid.bx() of grid.gdim() CTAs over the GEMM that p and the maps
// describe: the whole grid of a single launch, or one GEMM's share of a grouped launch.
template <bool TF32, int MODE, bool SPLIT, bool SINE, typename Grid>
__device__ __forceinline__ void tc_gemm_body(const CUtensorMap* mapA, const CUtensorMap* mapA2,
                                             const CUtensorMap* mapB, const CUtensorMap* mapBlo, const TcParams& p,
                                             const Grid grid, const CUtensorMap* mapV = nullptr,
                                             const CUtensorMap* mapO = nullptr, const CUtensorMap* mapOlo = nullptr) {
  constexpr bool PAIR = Grid::PAIR;
  static_assert(!PAIR || (MODE == TC_FWD && !TF32 && !SINE), "pairs run the BF16 tanh forward");
  using C = Cfg<TF32, MODE, SPLIT, PAIR>;
  const int rank = PAIR ? (int)(blockIdx.x & 1) : 0;
  using T = typename std::conditional<TF32, float, __nv_bfloat16>::type;
  // weight gradient with 256-row tiles: two 128-row accumulators (TMEM columns 0..255 and
  // 256..511) share each staged B operand, so the B rows are read once for 256 output
  // rows; one work item fills both accumulators (no double buffering across items)
  constexpr bool DW2 = (MODE == TC_DW) && SPLIT;
  constexpr int MROWS = DW2 ? 2 * BM : BM;                // output rows per work item
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned by offsetting the shared array itself (an integer round trip would
  // hide the address space and turn every shared access below into a generic one)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* blo = smem + C::STAGES * C::STAGE;          // TF32 B_lo buffer (BLOC_BYTES)
  uint8_t* outb = blo + C::BLOC_BYTES;                 // pair: output buffers
  uint64_t* full = reinterpret_cast<uint64_t*>(outb + C::OUT_BUFS * C::OUT_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* acc_full = empty + C::STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* lo_full = acc_empty + 2;                  // converter -> MMA: B_lo ready
  uint64_t* lo_empty = lo_full + 1;                   // MMA -> converter: B_lo consumed
  uint64_t* never = lo_empty + 1;                     // test hook (p.stall): no thread arrives on it
  uint64_t* out_full = never + 1;                     // [OUT_BUFS] epilogue -> stores: buffer written
  uint64_t* out_read = out_full + C::OUT_BUFS;        // [OUT_BUFS] stores -> epilogue: buffer read
  volatile int* abort_flag = reinterpret_cast<volatile int*>(out_read + C::OUT_BUFS);
  volatile int* inflight = abort_flag + 1;             // [STAGES]: parity+1 of an armed, unconsumed stage
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(inflight + C::STAGES));

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      inflight[s] = 0;
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], PAIR ? 2 * EPI_WARPS : 32 * EPI_WARPS);   // (pair: both CTAs' warps, at the first one's)
    }
    mbar_init(lo_full, 1);
    mbar_init(lo_empty, 1);
    mbar_init(never, 1);
    for (int b = 0; b < C::OUT_BUFS; ++b) {
      mbar_init(&out_full[b], EPI_WARPS);
      mbar_init(&out_read[b], 1);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {   // allocate 2 x 256 TMEM columns (whole warp)
    tmem_alloc<PAIR>(tmem_slot, 2 * BN);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int total = p.m_tiles * p.n_tiles * (MODE == TC_DW ? p.nsplit : 1);
  auto coords = [&](int t, int& mb, int& nb, int& k0, int& k1) {
    if (MODE != TC_DW && p.e.reverse) t = total - 1 - t;   // same tiles, last column tile first
    mb = t % p.m_tiles;
    int r = t / p.m_tiles;
    nb = r % p.n_tiles;
    if (MODE == TC_DW) {
      const int s = r / p.n_tiles;
      k0 = s * p.kps;
      k1 = min(p.k_iters, k0 + p.kps);
    } else {
      k0 = 0;
      k1 = p.k_iters;
    }
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      for (int t = grid.bx(); t < total && !*abort_flag; t += grid.gdim()) {
        int mb, nb, k0, k1;
        coords(t, mb, nb, k0, k1);
        for (int kb = k0; kb < k1; ++kb) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status, p.wait_ns)) break;
          uint8_t* sa = smem + stage * C::STAGE;
          uint8_t* sa2 = sa + C::A_BYTES;
          uint8_t* sb = sa + C::A_BYTES * (SPLIT ? 2 : 1);
          const int kx = kb * C::BKE;
          if constexpr (PAIR) {
            // both CTAs' copies complete at the first one's barrier: it issues the MMAs
            const uint32_t bar = cta_addr(&full[stage], 0);
            if (rank == 0) {
              mbar_expect_tx(&full[stage], 2 * (C::STAGE - (p.wlo_values_only ? 0 : C::V_BYTES)));
              inflight[stage] = (int)phase + 1;
            }
            tma_load_2d_pair(sa, mapA, bar, kx, mb * BM);
            tma_load_2d_pair(sa2, mapA2, bar, kx, mb * BM);
#pragma unroll
            for (int j = 0; j < C::NBOX; ++j)
              tma_load_3d_pair(sb + j * C::BOX_BYTES, mapB, bar, (C::NBOX * rank + j) * C::BOXN, kx, nb);
            tma_load_3d_pair(sb + C::B_BYTES, mapBlo, bar, rank * (TILE_PTS / 2), kx, nb);
            if (p.wlo_values_only) tma_load_3d_pair(sb + C::B_BYTES + C::V_BYTES, mapV, bar, rank * (TILE_PTS / 2), kx, nb);
            if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
            continue;
          }
          mbar_expect_tx(&full[stage], C::STAGE);
          inflight[stage] = (int)phase + 1;
          if (C::KPM) {
            // A: weights [M][K]; B: point-major jets [NC][K], columns nb*BN.. (both 2-D, K-major)
            tma_load_2d(sa, mapA, &full[stage], kx, mb * BM);
            if (SPLIT) tma_load_2d(sa2, mapA2, &full[stage], kx, mb * BM);
            tma_load_2d(sb, mapB, &full[stage], kx, nb * BN);
          } else if (C::B_MN) {
            // A: weights [M][K] (2-D); B: jet tile nb, rows kx..kx+BKE (3-D, tile-major)
            tma_load_2d(sa, mapA, &full[stage], kx, mb * BM);
            if (SPLIT) tma_load_2d(sa2, mapA2, &full[stage], kx, mb * BM);
#pragma unroll
            for (int j = 0; j < C::NBOX; ++j)
              tma_load_3d(sb + j * C::BOX_BYTES, mapB, &full[stage], j * C::BOXN, kx, nb);
            if (C::VLO) {
#pragma unroll
              for (int j = 0; j < TILE_PTS / C::BOXN; ++j)
                tma_load_3d(sb + C::B_BYTES + j * C::BOX_BYTES, mapBlo, &full[stage], j * C::BOXN, kx, nb);
            }
          } else {
            // weight gradient: K runs over jet columns, 256 / BKE K-blocks per tile
            constexpr int KPT = TILE_COLS / C::BKE;
            const int tz = kb / KPT, tx = (kb % KPT) * C::BKE;
            tma_load_3d(sa, mapA, &full[stage], tx, mb * MROWS, tz);
            if (DW2) tma_load_3d(sa2, mapA, &full[stage], tx, mb * MROWS + BM, tz);
            tma_load_3d(sb, mapB, &full[stage], tx, nb * BN, tz);
          }
          if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (PAIR)   // the last arrivals land before this CTA may leave
        for (int s = 0; s < C::STAGES; ++s) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status, p.wait_ns)) break;
          if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
        }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t MR = PAIR ? 2 * BM : BM;
      constexpr uint32_t idesc = make_idesc(TF32 ? 2u : 1u, C::B_MN ? 1u : 0u, BN, MR);
      int stage = 0;
      uint32_t phase = 0, lo_phase = 0;
      int local = 0;
      // test hook: a dependency that is never satisfied, so the bounded wait expires and
      // the whole CTA takes the abort path (status bit 1, teardown below)
      const bool stalled = p.stall && !mbar_wait(never, 0, abort_flag, p.status, p.wait_ns);
      for (int t = grid.bx(); t < total && !*abort_flag && !stalled; t += grid.gdim(), ++local) {
        int mb, nb, k0, k1;
        coords(t, mb, nb, k0, k1);
        const int buf = DW2 ? 0 : local & 1;
        const uint32_t par = DW2 ? ((uint32_t)local & 1) : ((uint32_t)(local >> 1) & 1);
        if (!mbar_wait<PAIR>(&acc_empty[buf], par ^ 1, abort_flag, p.status, p.wait_ns)) break;
        tc_fence_after();
        const uint32_t d = tmem_base + buf * BN;
        bool ok = true;
        for (int kb = k0; kb < k1; ++kb) {
          if (!mbar_wait(&full[stage], phase, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
          inflight[stage] = 0;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * C::STAGE);
          const uint32_t sa2 = sa + C::A_BYTES;
          const uint32_t sb = sa + C::A_BYTES * (SPLIT ? 2 : 1);
#pragma unroll
          for (int kk = 0; kk < C::BKE / C::UK; ++kk) {
            const uint64_t ad = make_desc(sa + kk * 32, 16, 1024);
            const uint64_t bd = C::B_MN ? make_desc(sb + kk * C::UK * 128, C::BOX_BYTES, 1024)
                                        : make_desc(sb + kk * 32, 16, 1024);
            tc_mma<TF32, PAIR>(d, ad, bd, idesc, (kb > k0 || kk > 0) ? 1u : 0u);
            if constexpr (PAIR) {
              // the same sums as below; the 64 value columns are 32 of each CTA (64-byte swizzle)
              constexpr uint32_t idesc64 = make_idesc(1u, 1u, TILE_PTS, MR);
              const uint32_t sl = sb + C::B_BYTES + kk * C::UK * 64;
              const uint64_t ad2 = make_desc(sa2 + kk * 32, 16, 1024);
              if (p.wlo_values_only) tc_mma<TF32, PAIR>(d, ad2, make_desc<64>(sl + C::V_BYTES, 512, 512), idesc64, 1u);
              else tc_mma<TF32, PAIR>(d, ad2, bd, idesc, 1u);
              tc_mma<TF32, PAIR>(d, ad, make_desc<64>(sl, 512, 512), idesc64, 1u);
              continue;
            }
            if constexpr (DW2) {
              // the second 128 output rows, same B operand, into TMEM columns 256..511
              tc_mma<TF32>(d + BN, make_desc(sa2 + kk * 32, 16, 1024), bd, idesc, (kb > k0 || kk > 0) ? 1u : 0u);
            } else if (SPLIT) {
              // low half of the weights: D += W_lo . A on every column, or on the value columns
              constexpr uint32_t idesc_v = make_idesc(TF32 ? 2u : 1u, C::B_MN ? 1u : 0u, TILE_PTS);
              tc_mma<TF32>(d, make_desc(sa2 + kk * 32, 16, 1024), bd, p.wlo_values_only ? idesc_v : idesc, 1u);
            }
            if (C::VLO) {
              // low half of the input's value rows: D[:, 0:64] += W_hi . A_lo
              constexpr uint32_t idesc64 = make_idesc(TF32 ? 2u : 1u, 1u, TILE_PTS);
              tc_mma<TF32>(d, ad, make_desc(sb + C::B_BYTES + kk * C::UK * 128, C::BOX_BYTES, 1024), idesc64, 1u);
            }
          }
          if (C::KPM) {
            // TF32: D += W_hi . B_lo once the converters have written B_lo
            if (!mbar_wait(lo_full, lo_phase, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sbl = smem_u32(blo);
#pragma unroll
            for (int kk = 0; kk < C::BKE / C::UK; ++kk)
              tc_mma<TF32>(d, make_desc(sa + kk * 32, 16, 1024), make_desc(sbl + kk * 32, 16, 1024), idesc, 1u);
            tc_commit(lo_empty);
            lo_phase ^= 1;
          }
          tc_commit<PAIR>(&empty[stage]);
          if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        tc_commit<PAIR>(&acc_full[buf]);
      }
    }
  } else if (C::KPM && warp >= 2 + EPI_WARPS) {
    // ---------------------------------------------------------------- TF32 B_lo converters
    // B_lo = B - tf32(B), elementwise over the stage's B tile (layout-agnostic), into
    // the single B_lo buffer once the MMAs of the previous stage have released it.
    const int ct = threadIdx.x - 32 * (2 + EPI_WARPS);
    int stage = 0;
    uint32_t phase = 0, lo_phase = 0;
    for (int t = grid.bx(); t < total && !*abort_flag; t += grid.gdim()) {
      int mb, nb, k0, k1;
      coords(t, mb, nb, k0, k1);
      bool ok = true;
      for (int kb = k0; kb < k1; ++kb) {
        bool got = mbar_wait(&full[stage], phase, abort_flag, p.status, p.wait_ns) &&
                   mbar_wait(lo_empty, lo_phase ^ 1, abort_flag, p.status, p.wait_ns);
        // both converter warps meet at named barrier 1 below: decide together whether to go on
        {
          uint32_t r;
          asm volatile(
              "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
              : "=r"(r)
              : "r"((uint32_t)got), "n"(32 * C::CVT_WARPS)
              : "memory");
          got = r != 0;
        }
        if (!got) { ok = false; break; }
        const float4* src = reinterpret_cast<const float4*>(smem + stage * C::STAGE + C::A_BYTES * (SPLIT ? 2 : 1));
        float4* dst = reinterpret_cast<float4*>(blo);
        // latency-bound: keep 16 shared-memory loads in flight per thread
        constexpr int U = 16, STRIDE = 32 * (C::CVT_WARPS > 0 ? C::CVT_WARPS : 1);
        static_assert((C::B_BYTES / 16) % (U * STRIDE) == 0, "converter batches cover the tile");
        for (int i0 = ct; i0 < C::B_BYTES / 16; i0 += U * STRIDE) {
          float4 x[U];
#pragma unroll
          for (int u = 0; u < U; ++u) x[u] = src[i0 + u * STRIDE];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            x[u].x -= tf32_trunc(x[u].x); x[u].y -= tf32_trunc(x[u].y);
            x[u].z -= tf32_trunc(x[u].z); x[u].w -= tf32_trunc(x[u].w);
            dst[i0 + u * STRIDE] = x[u];
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
        asm volatile("bar.sync 1, %0;" ::"n"(32 * C::CVT_WARPS) : "memory");
        if (ct == 0) mbar_arrive(lo_full);
        lo_phase ^= 1;
        if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
      }
      if (!ok) break;
    }
  } else if (PAIR && warp >= 2 + EPI_WARPS) {
    // ---------------------------------------------------------------- output stores (pair)
    if (lane == 0) {
      const int items = p.e.alo_out ? 5 : 4;              // jet rows, then the value rows' low half
      int b = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = grid.bx(); t < total && ok; t += grid.gdim()) {
        int mb, nb, k0, k1;
        coords(t, mb, nb, k0, k1);
        for (int i = 0; i < items; ++i) {
          ok = mbar_wait(&out_full[b], ph, abort_flag, p.status, p.wait_ns);
          if (!ok) break;
          tma_store_3d(i < 4 ? mapO : mapOlo, outb + b * C::OUT_BYTES, i < 4 ? TILE_PTS * i : 0, mb * BM, nb);
          bulk_commit();
          bulk_wait_read0();
          mbar_arrive(&out_read[b]);
          if (++b == C::OUT_BUFS) { b = 0; ph ^= 1; }
        }
      }
      bulk_wait0();
    }
  } else if (warp < 2 + EPI_WARPS) {
    // ---------------------------------------------------------------- epilogue
    // Warp part `part` of a lane quadrant handles points 32 part .. 32 part + 31 of the
    // tile in units of UPTS points; a unit is the four UPTS-column chunks at columns
    // pc + 64 r (jet row r), so every thread holds whole points of its feature.  A unit
    // row is one full 32-byte sector (16 BF16 or 8 FP32 values): partial-sector stores
    // would make L2 fetch the sector first.  FP32 units are small enough to double-buffer
    // the TMEM loads.
    constexpr int PARTS = EPI_WARPS / 4;                 // warps per lane quadrant
    constexpr int UPTS = TF32 ? 8 : 16;                  // points per unit
    constexpr int UNITS = TILE_PTS / (UPTS * PARTS);     // units per warp and tile
    constexpr bool PIPE = TF32;                          // double-buffered TMEM loads
    static_assert(PARTS * UNITS * UPTS == TILE_PTS && UNITS % 2 == 0, "epilogue units cover a 64-point tile");
    const int quad = warp & 3;
    const int part = (warp - 2) >> 2;
    const int row = quad * 32 + lane;
    auto unit_col = [&](int u) { return part * (UNITS * UPTS) + UPTS * u; };

    // BF16 tanh forward: both units of a warp's tile are finished before their sectors are exchanged
    // and stored; the accumulator is free as soon as it is in registers.
    constexpr bool PAIRS = !TF32 && !SINE && MODE == TC_FWD;
    // TF32 forward and adjoint: two units at a time, whose sectors lane pairs exchange; the
    // adjoint's activations of the next two units are loaded the same way before this
    // two's stores.  (One unit at a time, a line per lane: 6x256 cavity at 69,632 points, five
    // adjoint launches 1.71 -> 1.43 ms, six forward launches 1.29 -> 1.16.)
    constexpr bool PAIRS32 = TF32 && !SINE && (MODE == TC_FWD || MODE == TC_ADJ);
    [[maybe_unused]] uint32_t aw[PAIRS32 && MODE == TC_ADJ ? 2 : 1][4][8];
    [[maybe_unused]] auto load_pairs32 = [&](int t_, int u_) {
      int mb_, nb_, k0_, k1_;
      coords(t_, mb_, nb_, k0_, k1_);
      const int m_ = mb_ * BM + row;
      if (m_ < p.M) {
        const float* z = reinterpret_cast<const float*>(p.e.ain) + toff(m_ & ~1, (int64_t)nb_ * BN, p.M) +
                         unit_col(u_) + UPTS * (m_ & 1);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          ld8raw(z + 64 * r, aw[0][r]);
          ld8raw(z + 64 * r + TILE_COLS, aw[1][r]);
        }
      }
    };
    if constexpr (PAIRS32 && MODE == TC_ADJ) {
      if (grid.bx() < total) load_pairs32(grid.bx(), 0);
    }
    [[maybe_unused]] int ob = 0;                          // pair: the next output buffer, its uses' parity
    [[maybe_unused]] uint32_t oph = 0;
    bool left = false;                                   // an output buffer's wait expired
    int local = 0;
    for (int t = grid.bx(); t < total && !left; t += grid.gdim(), ++local) {
      int mb, nb, k0, k1;
      coords(t, mb, nb, k0, k1);
      const int buf = DW2 ? 0 : local & 1;
      const bool got = mbar_wait(&acc_full[buf], DW2 ? ((uint32_t)local & 1) : ((uint32_t)(local >> 1) & 1), abort_flag,
                                 p.status, p.wait_ns);
      if (__any_sync(0xffffffffu, !got)) break;   // (the warp's loads and shuffles are collective)
      tc_fence_after();
      for (int half = 0; half < (DW2 ? 2 : 1); ++half) {
      const int m = mb * MROWS + half * BM + row;
      const bool mvalid = m < p.M;
      const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + (DW2 ? half : buf) * BN;
      float db[4] = {0.f, 0.f, 0.f, 0.f};
      float xc[3] = {0.f, 0.f, 0.f};
      if (MODE == TC_ADJ && p.e.dbpart && p.e.dterms)
        lane_coords(p.e, (int64_t)nb * TILE_PTS + part * (UNITS * UPTS) + lane, xc);

      auto issue = [&](int u, float (&v)[4][UPTS]) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if constexpr (UPTS == 8) tmem_ld8_issue(tbase + unit_col(u) + 64 * r, v[r]);
          else tmem_ld16_issue(tbase + unit_col(u) + 64 * r, v[r]);
        }
      };
      // the epilogue of one unit of a valid row
      auto finish = [&](int u, float (&v)[4][UPTS]) {
        const int pc = unit_col(u);                                   // first point of the unit in its tile
        const int64_t cbase = toff(m, (int64_t)nb * BN, p.M) + pc;    // tile nb, row m
        if constexpr (MODE == TC_FWD && SINE) {
          const float bias = p.e.bias[m];
#pragma unroll
          for (int i = 0; i < UPTS; ++i) v[0][i] += bias;
          // the pre-activation jets for the adjoint, FP32 [M][NC] tile-major
          float* zo = p.e.zout + cbase;
#pragma unroll
          for (int r = 0; r < 4; ++r) st_f32<UPTS>(zo + 64 * r, v[r]);
#pragma unroll
          for (int i = 0; i < UPTS; ++i) {
            float z[4] = {v[0][i], v[1][i], v[2][i], v[3][i]}, a[4];
            jet_fwd_sine(z, a, p.e.jet_mode, p.e.omega0);
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r][i] = a[r];
          }
          T* ao = reinterpret_cast<T*>(p.e.out) + cbase;
#pragma unroll
          for (int r = 0; r < 4; ++r) st_row(ao + 64 * r, v[r]);
          if (p.e.alo_out) {
            // low half of the value rows for the next forward (BF16 rounding remainder)
            float lo[UPTS];
#pragma unroll
            for (int i = 0; i < UPTS; ++i) lo[i] = v[0][i] - __bfloat162float(__float2bfloat16_rn(v[0][i]));
            st_row(reinterpret_cast<T*>(p.e.alo_out) + loff(m, (int64_t)nb * TILE_PTS, p.M) + pc, lo);
          }
        } else if constexpr (MODE == TC_ADJ && SINE) {
          // the rule from the stored pre-activation jets z of the layer below
          const float* zr = p.e.zin + cbase;
#pragma unroll
          for (int h8 = 0; h8 < UPTS / 8; ++h8) {
            uint32_t zz[4][8];
#pragma unroll
            for (int r = 0; r < 4; ++r) ld_global_256(zr + 64 * r + 8 * h8, zz[r]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float z[4] = {__uint_as_float(zz[0][i]), __uint_as_float(zz[1][i]), __uint_as_float(zz[2][i]),
                            __uint_as_float(zz[3][i])};
              const int k = 8 * h8 + i;
              float ab[4] = {v[0][k], v[1][k], v[2][k], v[3][k]}, zb[4];
              jet_adj_sine(z, ab, zb, p.e.jet_mode, p.e.omega0);
#pragma unroll
              for (int r = 0; r < 4; ++r) v[r][k] = zb[r];
            }
          }
          if (p.e.out) {
            T* zbo = reinterpret_cast<T*>(p.e.out) + cbase;
#pragma unroll
            for (int r = 0; r < 4; ++r) st_row(zbo + 64 * r, v[r]);
          }
        } else if constexpr (MODE == TC_DW) {
          const int split = t / (p.m_tiles * p.n_tiles);
          float* dst = p.out32 + ((int64_t)split * p.M + m) * p.N;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int64_t col0 = (int64_t)nb * BN + pc + 64 * r;
            if (col0 + UPTS <= p.N && (p.N & 7) == 0) {
              st_f32<UPTS>(dst + col0, v[r]);
            } else {
              for (int j = 0; j < UPTS; ++j)
                if (col0 + j < p.N) dst[col0 + j] = v[r][j];
            }
          }
        } else if constexpr (MODE == TC_STORE) {
#pragma unroll
          for (int r = 0; r < 4; ++r) st_f32<UPTS>(p.out32 + cbase + 64 * r, v[r]);
        }
      };
      // bias gradient of the layer below (value rows) and, for a first layer on raw
      // coordinates, the coordinate terms of its weight gradient (every lane: rows past M
      // add values that nobody stores)
      [[maybe_unused]] auto bias_sums = [&](int u, const float (&v)[4][UPTS]) {
        if (!p.e.dbpart) return;
#pragma unroll
        for (int i = 0; i < UPTS; ++i) db[0] += v[0][i];
        if (p.e.dterms) coord_terms<UPTS>(v, xc, UPTS * u, p.e.dterms, p.e.jet_mode, db);
      };
      [[maybe_unused]] auto process = [&](int u, float (&v)[4][UPTS]) {
        if (mvalid) finish(u, v);
        if constexpr (MODE == TC_ADJ) bias_sums(u, v);
      };

      if constexpr (PAIRS) {
        uint32_t w[UNITS][4][8], lo[UNITS][8];
        const float bias = mvalid ? p.e.bias[m] : 0.f;
#pragma unroll
        for (int u = 0; u < UNITS; ++u) {
          float v[4][UPTS];
          issue(u, v);
          tmem_wait_ld();
          if (u == UNITS - 1) {
            tc_fence_before();
            if constexpr (PAIR) {
              __syncwarp();
              if (lane == 0) mbar_arrive_cta(&acc_empty[buf], 0);
            } else {
              mbar_arrive(&acc_empty[buf]);
            }
          }
          with_jet_mode(p.e.jet_mode,
                        [&](auto mode) { fwd_pairs<decltype(mode)::value>(v, bias, w[u], lo[u], 0xffffffffu); });
        }
        if constexpr (PAIR) {
          // 64 bytes of each row into the swizzled buffer: 16-byte chunk (32 part + 16 u + 8 q) / 8
          auto put = [&](const uint32_t (&a)[8], const uint32_t (&b)[8]) {
            const bool ok = mbar_wait(&out_read[ob], oph ^ 1, abort_flag, p.status, p.wait_ns);
            if (__any_sync(0xffffffffu, !ok)) { left = true; return; }
            const uint32_t at = smem_u32(outb + ob * C::OUT_BYTES + row * 128);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t* x = (q < 2 ? a : b) + 4 * (q & 1);
              asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at + (((part * 4 + q) ^ (row & 7)) << 4)),
                           "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3])
                           : "memory");
            }
            fence_proxy_async_smem();                   // these writes before the bulk store's reads
            __syncwarp();
            if (lane == 0) mbar_arrive(&out_full[ob]);
            if (++ob == C::OUT_BUFS) { ob = 0; oph ^= 1; }
          };
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (!left) put(w[0][r], w[1][r]);
          if (p.e.alo_out && !left) put(lo[0], lo[1]);
        } else {
          store_pairs(reinterpret_cast<T*>(p.e.out), w, m, nb, p.M, unit_col(0));
          if (p.e.alo_out) store_lo_pairs(reinterpret_cast<T*>(p.e.alo_out), lo, m, nb, p.M, unit_col(0));
        }
      } else if constexpr (PAIRS32) {
        [[maybe_unused]] const float bias = MODE == TC_FWD && mvalid ? p.e.bias[m] : 0.f;
#pragma unroll 1
        for (int u = 0; u < UNITS; u += 2) {
          float v[2][4][UPTS];
          issue(u, v[0]);
          issue(u + 1, v[1]);
          tmem_wait_ld();
          if (u + 2 == UNITS) {
            tc_fence_before();
            mbar_arrive(&acc_empty[buf]);
          }
          if constexpr (MODE == TC_ADJ) {
#pragma unroll
            for (int r = 0; r < 4; ++r) pair_swap(aw[0][r], aw[1][r]);
          }
#pragma unroll
          for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int i = 0; i < UPTS; ++i) {
              float y[4];
              if constexpr (MODE == TC_FWD) {
                const float z[4] = {v[k][0][i] + bias, v[k][1][i], v[k][2][i], v[k][3][i]};
                jet_fwd<false>(z, y, p.e.jet_mode);
              } else {
                const float ab[4] = {v[k][0][i], v[k][1][i], v[k][2][i], v[k][3][i]};
                const float av[4] = {__uint_as_float(aw[k][0][i]), __uint_as_float(aw[k][1][i]),
                                     __uint_as_float(aw[k][2][i]), __uint_as_float(aw[k][3][i])};
                jet_adj_a(av, ab, y, p.e.jet_mode);
              }
#pragma unroll
              for (int r = 0; r < 4; ++r) v[k][r][i] = y[r];
            }
            if constexpr (MODE == TC_ADJ) bias_sums(u + k, v[k]);
          }
          if constexpr (MODE == TC_ADJ) {
            if (u + 2 < UNITS) load_pairs32(t, u + 2);
            else if (t + grid.gdim() < total) load_pairs32(t + grid.gdim(), 0);
          }
          if (p.e.out_pm && mvalid) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
              store_pm8(reinterpret_cast<float*>(p.e.out_pm), (int64_t)nb * BN + unit_col(u + k), p.M, m, v[k]);
          }
          if (p.e.out) {
            float* o = reinterpret_cast<float*>(p.e.out) + toff(m & ~1, (int64_t)nb * BN, p.M) + unit_col(u) + UPTS * (m & 1);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              uint32_t (&x)[8] = reinterpret_cast<uint32_t (&)[8]>(v[0][r]);
              uint32_t (&y)[8] = reinterpret_cast<uint32_t (&)[8]>(v[1][r]);
              pair_swap(x, y);
              if (mvalid) {
                st_global_256(o + 64 * r, x);
                st_global_256(o + 64 * r + TILE_COLS, y);
              }
            }
          }
        }
      } else if constexpr (PIPE) {
        float va[4][UPTS], vb[4][UPTS];
        issue(0, va);
        tmem_wait_ld();
#pragma unroll 1
        for (int u = 0; u < UNITS; u += 2) {
          issue(u + 1, vb);
          process(u, va);
          tmem_wait_ld();
          if (u + 2 < UNITS) issue(u + 2, va);
          process(u + 1, vb);
          if (u + 2 < UNITS) tmem_wait_ld();
        }
      } else {
#pragma unroll 1
        for (int u = 0; u < UNITS; ++u) {
          float va[4][UPTS];
          issue(u, va);
          tmem_wait_ld();
          process(u, va);
        }
      }
      if (MODE == TC_ADJ && mvalid && p.e.dbpart) {
        float* dst = p.e.dbpart + ((int64_t)m * (p.n_tiles * PARTS) + nb * PARTS + part) * (1 + p.e.dterms);
        dst[0] = db[0];
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (j < p.e.dterms) dst[1 + j] = db[1 + j];
      }
      }   // half
      if constexpr (!PAIRS && !PAIRS32) {
        tc_fence_before();
        mbar_arrive(&acc_empty[buf]);
      }
    }
  }

  // ---- teardown: wait (bounded) for copies and MMAs still in flight, free TMEM ----------------
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    for (int s = 0; s < C::STAGES; ++s) {
      const int f = inflight[s];
      if (f) {
        const uint64_t t0 = gtimer();
        while (!mbar_try(&full[s], (uint32_t)(f - 1)) && gtimer() - t0 < WAIT_NS) {}
      }
    }
    if (!PAIR) abort_settle();
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) pair_leave(abort_flag);
  if (warp == 1) {
    tc_fence_after();
    tmem_free<PAIR>(tmem_base, 2 * BN);
  }
}

template <bool TF32, int MODE, bool SPLIT, bool SINE = false>
__global__ void __launch_bounds__(Cfg<TF32, MODE, SPLIT>::NTHREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA2,
              const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBlo,
              const __grid_constant__ TcParams p) {
  tc_gemm_body<TF32, MODE, SPLIT, SINE>(&mapA, &mapA2, &mapB, &mapBlo, p, SingleGrid{});
}

// The BF16 tanh forward in pairs.  Launched alone, a 128 x 256 unit of a 512-wide layer moves
// 24 KB of operands per K step and 72 KB of copies per stage through shared memory and stores
// a line per lane; at 128 bytes a cycle the sum (13,300 cycles) is its time (13,450).  As a
// pair each CTA stages half of the columns (56 KB) and its MMAs read half of them (18 KB); the
// smaller stages leave room for output buffers, from which the tile leaves by bulk tensor
// stores.  Same sums in the same order.  Forward launches, ms: Maxwell 5x512 at 294,912
// points 3.38 -> 3.09, 8x512 cavity at 1,064,960 23.4 -> 22.2.  (Pairs that store from
// registers: 3.28 and 24.3.)  Left: tensor pipe 53%, DRAM 45%; limiting the low half of the
// weights to the value rows saves nothing, and without its epilogue the unpaired kernel took
// 0.71 of its time.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Cfg<false, TC_FWD, true, true>::NTHREADS, 1)
    k_tc_fwd_pair(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA2,
                  const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBlo,
                  const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO,
                  const __grid_constant__ CUtensorMap mapOlo, const __grid_constant__ TcParams p) {
  tc_gemm_body<false, TC_FWD, true, false>(&mapA, &mapA2, &mapB, &mapBlo, p, PairGrid{}, &mapV, &mapO, &mapOlo);
}

// Grouped launch: the GEMMs of several networks (or layers) side by side, each entry of
// the device table holding one GEMM's tensor maps and parameters and its block range.
template <bool TF32, int MODE, bool SPLIT, bool SINE = false>
__global__ void __launch_bounds__(Cfg<TF32, MODE, SPLIT>::NTHREADS, 1)
    k_tc_gemm_group(const TcGroupEntry* __restrict__ tab, const int n) {
  const TcGroupEntry& g = tab[group_of_block(tab, n, (int)blockIdx.x)];
  acquire_maps(g, 4);
  tc_gemm_body<TF32, MODE, SPLIT, SINE>(&g.map[0], &g.map[1], &g.map[2], &g.map[3], g.p,
                                        GroupShare{(int)blockIdx.x - g.block0, g.grid});
}

// ---- host side ------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

// 2-D tensor map over a row-major matrix [rows][cols] (cols contiguous), box
// [box_rows][box_cols], 128-byte swizzle, zero fill out of bounds.
bool make_map(CUtensorMap* m, const void* base, bool tf32, uint64_t cols, uint64_t rows, uint32_t box_cols,
              uint32_t box_rows) {
  if (!g_encode) return false;
  const uint32_t es = tf32 ? 4 : 2;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * es};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(m, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                        const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// 3-D tensor map over a tile-major jet matrix [ntiles][rows][tcols] (tcols = 256 for
// jet matrices, 64 for value-row low halves), box [1][box_rows][box_cols], 128-byte
// swizzle, zero fill out of bounds.
bool make_map3(CUtensorMap* m, const void* base, bool tf32, uint64_t tcols, uint64_t rows, uint64_t ntiles,
               uint32_t box_cols, uint32_t box_rows, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  if (!g_encode) return false;
  const uint32_t es = tf32 ? 4 : 2;
  cuuint64_t dims[3] = {tcols, rows, ntiles};
  cuuint64_t strides[2] = {tcols * es, tcols * rows * es};
  cuuint32_t box[3] = {box_cols, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(m, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                        const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

bool tc_map3(CUtensorMap* m, const void* base, bool fp32, uint64_t tcols, uint64_t rows, uint64_t ntiles,
             uint32_t box_cols, uint32_t box_rows) {
  return make_map3(m, base, fp32, tcols, rows, ntiles, box_cols, box_rows);
}

namespace {

template <typename K>
pinn_status reserve_smem(pinn_handle* h, K kern, size_t bytes, const char* what) {
  if (allow_smem(h, reinterpret_cast<const void*>(kern), bytes) == cudaSuccess) return PINN_OK;
  snprintf(h->err, sizeof(h->err), "%s: cannot reserve %zu bytes of shared memory", what, bytes);
  return PINN_ERR_CUDA;
}

pinn_status launch_check(pinn_handle* h, const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return PINN_OK;
  snprintf(h->err, sizeof(h->err), "%s launch: %s", what, cudaGetErrorString(e));
  return PINN_ERR_CUDA;
}

// Grouped launch of n table entries (blocks in all) of one GEMM kernel variant.
template <bool TF32, int MODE, bool SPLIT, bool SINE>
pinn_status launch_group(pinn_handle* h, const TcGroupEntry* d_tab, int n, int blocks, cudaStream_t st) {
  using C = Cfg<TF32, MODE, SPLIT>;
  auto kern = k_tc_gemm_group<TF32, MODE, SPLIT, SINE>;
  pinn_status s = reserve_smem(h, kern, C::SMEM, "grouped tcgen05 kernel");
  if (s) return s;
  kern<<<blocks, C::NTHREADS, C::SMEM, st>>>(d_tab, n);
  return launch_check(h, "grouped tcgen05 kernel");
}

}  // namespace

// Tensor-core GEMMs collected from several handles (tc_batch_attach) and issued as
// grouped launches: one per kernel variant, the GEMMs with the most work first.
struct TcBatch {
  using GroupFn = pinn_status (*)(pinn_handle*, const TcGroupEntry*, int, int, cudaStream_t);
  struct Item {
    GroupFn fn;
    TcGroupEntry e;
    double work;   // tiles x K iterations: the order of the grouped grid
  };
  std::vector<Item> pending;
  std::vector<TcGroupEntry> table;   // every issued entry, in device-table order
  TcGroupEntry* d_table = nullptr;
  size_t capacity = 0;               // entries d_table holds
  int launches = 0;
};

namespace {

pinn_status batch_add(TcBatch* b, TcBatch::GroupFn fn, const CUtensorMap* maps, int nmaps, const TcParams& p,
                      int grid) {
  TcBatch::Item it{};
  it.fn = fn;
  for (int i = 0; i < nmaps; ++i) it.e.map[i] = maps[i];
  it.e.p = p;
  it.e.grid = grid;
  it.work = (double)p.m_tiles * p.n_tiles * std::max(p.k_iters, 1);
  b->pending.push_back(it);
  return PINN_OK;
}

template <bool TF32, int MODE, bool SPLIT, bool SINE = false>
pinn_status launch(pinn_handle* h, const CUtensorMap& a, const CUtensorMap& a2, const CUtensorMap& b,
                   const CUtensorMap& blo, const TcParams& p, int grid, cudaStream_t st) {
  if (h->tc_batch) {
    const CUtensorMap maps[4] = {a, a2, b, blo};
    return batch_add(h->tc_batch, &launch_group<TF32, MODE, SPLIT, SINE>, maps, 4, p, grid);
  }
  using C = Cfg<TF32, MODE, SPLIT>;
  auto kern = k_tc_gemm<TF32, MODE, SPLIT, SINE>;
  pinn_status s = reserve_smem(h, kern, C::SMEM, "tcgen05 kernel");
  if (s) return s;
  kern<<<grid, C::NTHREADS, C::SMEM, st>>>(a, a2, b, blo, p);
  return launch_check(h, "tcgen05 kernel");
}

// Whether a launch runs in pairs (not in a grouped launch, whose entries start at any block).
bool in_pairs(const pinn_handle* h, const TcParams& p) {
  return !h->tc_batch && fwd_in_pairs(p.m_tiles, p.n_tiles, p.K, p.wlo_values_only != 0, h->sm_count);
}

int grid_for(const pinn_handle* h, int tiles) { return std::max(1, std::min(tiles, std::max(h->sm_count, 1))); }

}  // namespace

void tc_init(pinn_handle* h) {
  (void)h;
  if (!g_encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
}

bool tc_layer_supported(const pinn_handle* h, int li, int64_t NC) {
  if (!g_encode || h->spec.precision == PINN_FP32 || (h->spec.flags & PINN_FLAG_CUDA_CORES)) return false;
  // the tensor-core epilogues carry the tanh jet, and (BF16) the sine jet
  if (h->act != PINN_ACT_TANH && !(h->act == PINN_ACT_SINE && h->spec.precision == PINN_BF16)) return false;
  if (NC % BN) return false;
  const int fin = h->layers[li].fin, fout = h->layers[li].fout;
  // TMA row strides must be multiples of 16 bytes: fin and fout multiples of 8 elements.
  return (fin % 8 == 0) && (fout % 8 == 0) && fin >= 16 && fout >= 16;
}

// Weight-gradient tiles have 256 output rows (two accumulators sharing B) when the
// layer has more than 256 outputs, else (or with PINN_FLAG_DW_ROWS_128) 128.  At 256
// outputs the 256-row tile is a single work item per column split, and two 128-row
// items per split balance better (measured: 0.063 -> 0.059 ms at the 6x256 cavity, and
// half as many split partials for the finalisation to sum).
static int dw_rows(const pinn_handle* h, int fout) {
  return (fout > 2 * BM && !(h->spec.flags & PINN_FLAG_DW_ROWS_128)) ? 2 * BM : BM;
}

int tc_dw_splits(const pinn_handle* h, int fout, int fin, int64_t NC) {
  const int tiles = ((fout + dw_rows(h, fout) - 1) / dw_rows(h, fout)) * ((fin + BN - 1) / BN);
  const int kblock = (h->spec.precision == PINN_TF32) ? 32 : 64;
  const int k_iters = (int)((NC + kblock - 1) / kblock);
  int ns = std::max(1, (std::max(h->sm_count, 1) + tiles - 1) / tiles);
  ns = std::min(ns, k_iters);
  const int kps = (k_iters + ns - 1) / ns;
  return (k_iters + kps - 1) / kps;   // no empty split
}

namespace {

TcParams base_params(const pinn_handle* h, int M, int N, int K, int64_t NC, int kblock, int* status) {
  TcParams p{};
  p.M = M; p.N = N; p.K = K; p.NC = NC;
  p.m_tiles = (M + BM - 1) / BM;
  p.n_tiles = (N + BN - 1) / BN;
  p.k_iters = (K + kblock - 1) / kblock;
  p.nsplit = 1; p.kps = p.k_iters;
  p.status = status;
  p.wait_ns = h->stall_ns ? h->stall_ns : WAIT_NS;
  p.stall = h->stall_ns ? 1 : 0;
  return p;
}

pinn_status map_err(pinn_handle* h, const char* what) {
  snprintf(h->err, sizeof(h->err), "cuTensorMapEncodeTiled failed for %s", what);
  return PINN_ERR_CUDA;
}

}  // namespace

namespace {

template <bool TF32>
pinn_status fwd_impl(pinn_handle* h, const void* W, const void* Wlo, const void* A, const void* Alo, int fout, int fin,
                     int64_t NC, const EpiArgs& e, cudaStream_t st) {
  using C = Cfg<TF32, TC_FWD, true>;
  CUtensorMap ma, ma2, mb, mlo;
  const uint64_t nt = (uint64_t)(NC / TILE_COLS);
  if (!make_map(&ma, W, TF32, fin, fout, C::BKE, BM) || !make_map(&ma2, Wlo, TF32, fin, fout, C::BKE, BM))
    return map_err(h, "forward weights");
  if (TF32) {
    // point-major jets [NC][fin], K-major boxes of BKE features x BN columns
    if (!make_map(&mb, A, true, fin, (uint64_t)NC, C::BKE, BN)) return map_err(h, "forward activations");
    mlo = mb;
  } else {
    if (!make_map3(&mb, A, false, TILE_COLS, fin, nt, C::BOXN, C::BKE)) return map_err(h, "forward activations");
    if (!make_map3(&mlo, Alo, false, TILE_PTS, fin, nt, C::BOXN, C::BKE))
      return map_err(h, "forward value-row low half");
  }
  TcParams p = base_params(h, fout, (int)NC, fin, NC, C::BKE, h->d_status);
  p.e = e;
  p.wlo_values_only = (!TF32 && (h->spec.flags & PINN_FLAG_BF16_VALUE_SPLIT)) ? 1 : 0;
  const int grid = grid_for(h, p.m_tiles * p.n_tiles);
  if constexpr (!TF32) {
    if (h->act == PINN_ACT_SINE) return launch<TF32, TC_FWD, true, true>(h, ma, ma2, mb, mlo, p, grid, st);
    if (in_pairs(h, p)) {
      // 32 value columns of the input and of its low half per CTA, 64-byte swizzle
      using P = Cfg<false, TC_FWD, true, true>;
      CUtensorMap mv, mo, mol;
      if (!make_map3(&mv, A, false, TILE_COLS, fin, nt, TILE_PTS / 2, C::BKE, CU_TENSOR_MAP_SWIZZLE_64B) ||
          !make_map3(&mlo, Alo, false, TILE_PTS, fin, nt, TILE_PTS / 2, C::BKE, CU_TENSOR_MAP_SWIZZLE_64B))
        return map_err(h, "paired forward value rows");
      mol = mlo;
      if (!make_map3(&mo, e.out, false, TILE_COLS, fout, nt, TILE_PTS, BM) ||
          (e.alo_out && !make_map3(&mol, e.alo_out, false, TILE_PTS, fout, nt, TILE_PTS, BM)))
        return map_err(h, "paired forward outputs");
      pinn_status s = reserve_smem(h, k_tc_fwd_pair, P::SMEM, "paired forward kernel");
      if (s) return s;
      k_tc_fwd_pair<<<grid & ~1, P::NTHREADS, P::SMEM, st>>>(ma, ma2, mb, mlo, mv, mo, mol, p);
      return launch_check(h, "paired forward");
    }
  }
  return launch<TF32, TC_FWD, true>(h, ma, ma2, mb, mlo, p, grid, st);
}

pinn_status adj_staged(pinn_handle* h, const void* WT, const void* Zbar, int fin, int fout, int64_t NC,
                       const EpiArgs& e, cudaStream_t st);

template <bool TF32>
pinn_status adj_impl(pinn_handle* h, const void* WT, const void* WTlo, const void* Zbar, int fin, int fout,
                     int64_t NC, const EpiArgs& e, cudaStream_t st) {
  // TF32: split weights and the point-major adjoint with its low half (three MMAs);
  // BF16: high halves only.
  constexpr bool SPLIT = TF32;
  if (!TF32 && h->act != PINN_ACT_SINE) return adj_staged(h, WT, Zbar, fin, fout, NC, e, st);
  using C = Cfg<TF32, TC_ADJ, SPLIT>;
  CUtensorMap ma, ma2, mb;
  if (!make_map(&ma, WT, TF32, fout, fin, C::BKE, BM)) return map_err(h, "adjoint weights");
  ma2 = ma;
  if (TF32) {
    if (!make_map(&ma2, WTlo, true, fout, fin, C::BKE, BM)) return map_err(h, "adjoint weights (low half)");
    if (!make_map(&mb, Zbar, true, fout, (uint64_t)NC, C::BKE, BN)) return map_err(h, "adjoint input");
  } else {
    if (!make_map3(&mb, Zbar, false, TILE_COLS, fout, (uint64_t)(NC / TILE_COLS), C::BOXN, C::BKE))
      return map_err(h, "adjoint input");
  }
  TcParams p = base_params(h, fin, (int)NC, fout, NC, C::BKE, h->d_status);
  p.e = e;
  const int grid = grid_for(h, p.m_tiles * p.n_tiles);
  return launch<TF32, TC_ADJ, SPLIT, !TF32>(h, ma, ma2, mb, mb, p, grid, st);
}

template <bool TF32>
pinn_status dw_impl(pinn_handle* h, const void* Zbar, const void* A, int fout, int fin, int64_t NC, int nsplit,
                    float* part, cudaStream_t st) {
  using C = Cfg<TF32, TC_DW, false>;   // (the 256-row variant stages the same boxes, twice for A)
  const bool two = dw_rows(h, fout) > BM;
  CUtensorMap ma, mb;
  const uint64_t nt = (uint64_t)(NC / TILE_COLS);
  if (!make_map3(&ma, Zbar, TF32, TILE_COLS, fout, nt, C::BKE, BM)) return map_err(h, "weight-gradient adjoint");
  if (!make_map3(&mb, A, TF32, TILE_COLS, fin, nt, C::BKE, BN)) return map_err(h, "weight-gradient activations");
  TcParams p = base_params(h, fout, fin, (int)NC, NC, C::BKE, h->d_status);
  if (two) p.m_tiles = (fout + 2 * BM - 1) / (2 * BM);
  p.nsplit = nsplit;
  p.kps = (p.k_iters + nsplit - 1) / nsplit;
  if ((p.k_iters + p.kps - 1) / p.kps != nsplit) {
    snprintf(h->err, sizeof(h->err), "weight-gradient split plan mismatch");
    return PINN_ERR_INVALID_ARG;
  }
  p.out32 = part;
  const int grid = grid_for(h, p.m_tiles * p.n_tiles * nsplit);
  if (two) return launch<TF32, TC_DW, true>(h, ma, ma, mb, mb, p, grid, st);
  return launch<TF32, TC_DW, false>(h, ma, ma, mb, mb, p, grid, st);
}

}  // namespace

pinn_status tc_gemm_fwd(pinn_handle* h, const void* W, const void* Wlo, const void* A, const void* Alo, int fout,
                        int fin, int64_t NC, const EpiArgs& e, cudaStream_t st) {
  if (h->spec.precision == PINN_TF32) return fwd_impl<true>(h, W, Wlo, A, Alo, fout, fin, NC, e, st);
  return fwd_impl<false>(h, W, Wlo, A, Alo, fout, fin, NC, e, st);
}

pinn_status tc_gemm_adj(pinn_handle* h, const void* WT, const void* WTlo, const void* Zbar, int fin, int fout,
                        int64_t NC, const EpiArgs& e, cudaStream_t st) {
  if (h->spec.precision == PINN_TF32) return adj_impl<true>(h, WT, WTlo, Zbar, fin, fout, NC, e, st);
  return adj_impl<false>(h, WT, WTlo, Zbar, fin, fout, NC, e, st);
}

pinn_status tc_gemm_dw(pinn_handle* h, const void* Zbar, const void* A, int fout, int fin, int64_t NC, int nsplit,
                       float* part, cudaStream_t st) {
  if (h->spec.precision == PINN_TF32) return dw_impl<true>(h, Zbar, A, fout, fin, NC, nsplit, part, st);
  return dw_impl<false>(h, Zbar, A, fout, fin, NC, nsplit, part, st);
}

// ==== fused adjoint + weight gradient (BF16, fan-out <= 256) ==========================
//
// For a hidden layer whose adjoint and weight gradient both run on tensor cores, the
// two GEMMs read the same two arrays for the same column tile: Zbar_l^T [fout][NC]
// and A_{l-1}^T [fin][NC].  One persistent kernel does both per work unit (fin
// m-tile mb, column tile nb):
//   adjoint  Abar^T[mb rows][256 cols] = W^T[mb rows][fout] . Zbar^T[fout][256 cols]
//            (MN-major B), then the activation-form tanh-jet adjoint in the epilogue
//   weights  dW^T[mb rows][fout] += A_{l-1}^T[mb rows][256 cols] . Zbar^T[fout][256 cols]^T
//            (both K-major over the columns), accumulated in tensor memory across all
//            of the CTA's column tiles and written once as its split partial.
// Every CTA keeps one m-tile (the grid is a multiple of the m-tile count), so its dW
// slab stays in tensor memory: 256 columns for the adjoint accumulator (single
// buffer; the epilogue copies it to registers and releases it at once) plus up to
// 256 for dW^T.  The A_{l-1} tile is staged by TMA in shared memory (two buffers)
// and serves both the dW MMAs and the epilogue, which reads it from there instead of
// global memory.  Zbar is read once from HBM per column tile (the m-tile CTAs of a
// column tile run side by side, the second read hits L2), A once, Zbar_{l-1} written
// once: the separate weight-gradient pass and its re-reads are gone.
// The epilogue works on packed pairs of points, and the next unit's Zbar is prefetched into
// L2: five launches of the 6x256 cavity at 69,632 points 0.497 -> 0.471 ms.  What bounds it
// now: no single unit (DRAM 56%, tensor pipe 37%, L1/shared memory 43%), but the time a stage
// takes to arrive: two stages of 48 KB, 3,400 cycles each under this traffic (without the
// stores 0.39 ms, with every load in L2 0.41).
//
// DW = false is the adjoint alone, for a layer whose fan-out is above 256 (its dW^T slab
// would fill tensor memory).  Two accumulators overlap the epilogue with the next unit's MMAs;
// the epilogue puts Zbar_{l-1} in the place of the staged activations and the tile leaves by
// bulk tensor stores, so no lane stores (or loads) 32-byte sectors of 32 different lines:
// 8x512 cavity at 1,064,960 points, seven launches 18.5 -> 16.5 ms, Maxwell 5x512 at 294,912,
// four 3.04 -> 2.56 ms.  (With DW = true the in-place stores were slower, 0.471 -> 0.479 ms.)
//
// Warp roles (352 threads): 0 stage producer (W^T chunk + Zbar chunk), 1 TMEM
// allocator + MMA issuer, 2-9 epilogue, 10 A tiles in, Zbar tiles out.
namespace {

constexpr int FZ_EPI = EPI_WARPS;
constexpr int FZ_NT = 64 + 32 * FZ_EPI + 32;
constexpr int FZ_WB = BM * 128;                  // W^T chunk [128 fin][64 fout]       16 KB
constexpr int FZ_BOX = 64 * 128;                 // Zbar box [64 fout][64 cols]         8 KB
constexpr int FZ_ZB = 4 * FZ_BOX;                // Zbar chunk [64 fout][256 cols]     32 KB
constexpr int FZ_STAGE = FZ_WB + FZ_ZB;          // 48 KB
constexpr int FZ_ABOX = BM * 128;                // A box [128 fin][64 cols]           16 KB
constexpr int FZ_AT = 4 * FZ_ABOX;               // A_{l-1} tile [128 fin][256 cols]   64 KB
constexpr int FZ_DW_COL = BN;                    // dW^T accumulator: TMEM columns 256..511
template <bool DW>
struct FzCfg {
  static constexpr int STAGES = DW ? 2 : 3;
  static constexpr int ABUF = DW ? 2 : 1;
  static constexpr size_t SMEM = (size_t)STAGES * FZ_STAGE + (size_t)ABUF * FZ_AT + 1024 + 256;
  static_assert(SMEM <= 227 * 1024, "fused adjoint: shared memory budget");
};

template <bool DW, typename Grid>
__device__ __forceinline__ void tc_adjdw_body(const CUtensorMap* mapW, const CUtensorMap* mapZ, const CUtensorMap* mapA,
                                              const CUtensorMap* mapO, const TcParams& p, const Grid grid) {
  constexpr int FZ_STAGES = FzCfg<DW>::STAGES, FZ_ABUF = FzCfg<DW>::ABUF;
  constexpr int ACC = DW ? 1 : 2;                // adjoint accumulators
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned by offsetting the shared array itself (an integer round trip would
  // hide the address space and turn every shared access below into a generic one)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* abase = smem + FZ_STAGES * FZ_STAGE;
  uint64_t* full = reinterpret_cast<uint64_t*>(abase + FZ_ABUF * FZ_AT);
  uint64_t* empty = full + FZ_STAGES;
  uint64_t* acc_full = empty + FZ_STAGES;
  uint64_t* acc_empty = acc_full + ACC;
  uint64_t* a_full = acc_empty + ACC;
  uint64_t* z_done = a_full + FZ_ABUF;
  uint64_t* dw_full = z_done + FZ_ABUF;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(dw_full + 1);
  volatile int* inflight = abort_flag + 1;              // [FZ_STAGES]
  volatile int* a_inflight = inflight + FZ_STAGES;      // [FZ_ABUF]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(a_inflight + FZ_ABUF));

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < FZ_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      inflight[s] = 0;
    }
    for (int b = 0; b < FZ_ABUF; ++b) {
      mbar_init(&a_full[b], 1);
      mbar_init(&z_done[b], FZ_EPI);   // one arrival per epilogue warp
      a_inflight[b] = 0;
    }
    for (int b = 0; b < ACC; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], FZ_EPI);
    }
    mbar_init(dw_full, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int total = p.m_tiles * p.n_tiles;
  auto coords = [&](int t, int& mb, int& nb) {
    if (p.e.reverse) t = total - 1 - t;
    mb = t % p.m_tiles;
    nb = t / p.m_tiles;
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- stage producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      for (int t = grid.bx(); t < total && !*abort_flag; t += grid.gdim()) {
        int mb, nb;
        coords(t, mb, nb);
        // the next unit's Zbar is brought into L2 under this unit (the m-tiles share it): two
        // stages in flight do not cover the latency of DRAM
        if (t + grid.gdim() < total) {
          int mn, nn;
          coords(t + grid.gdim(), mn, nn);
          for (int kb = mn; kb < p.k_iters; kb += p.m_tiles)
#pragma unroll
            for (int j = 0; j < 4; ++j) tma_prefetch_3d(mapZ, j * 64, kb * 64, nn);
        }
        for (int kb = 0; kb < p.k_iters; ++kb) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status, p.wait_ns)) break;
          uint8_t* sw = smem + stage * FZ_STAGE;
          uint8_t* sz = sw + FZ_WB;
          mbar_expect_tx(&full[stage], FZ_STAGE);
          inflight[stage] = (int)phase + 1;
          tma_load_2d(sw, mapW, &full[stage], kb * 64, mb * BM);
#pragma unroll
          for (int j = 0; j < 4; ++j) tma_load_3d(sz + j * FZ_BOX, mapZ, &full[stage], j * 64, kb * 64, nb);
          if (++stage == FZ_STAGES) { stage = 0; phase ^= 1; }
        }
      }
    }
  } else if (warp == 2 + FZ_EPI) {
    // ---------------------------------------------------------------- A tiles in (and Zbar tiles out)
    if (lane == 0) {
      int in = 0, out = 0;    // tiles loaded, tiles done by the epilogue
      int t_out = grid.bx();
      bool ok = true;
      // the next tile is done; staged: it leaves by bulk tensor stores
      auto next_done = [&]() {
        const int ab = out % FZ_ABUF;
        ok = mbar_wait(&z_done[ab], (uint32_t)(out / FZ_ABUF) & 1, abort_flag, p.status, p.wait_ns);
        if (!ok) return;
        if (!DW && p.e.out) {
          int mb, nb;
          coords(t_out, mb, nb);
          const uint8_t* at = abase + ab * FZ_AT;
#pragma unroll
          for (int j = 0; j < 4; ++j) tma_store_3d(mapO, at + j * FZ_ABOX, j * 64, mb * BM, nb);
          bulk_commit();
        }
        t_out += grid.gdim();
        ++out;
      };
      // (test hook, single launches: with p.stall no tile comes, and the waits for it expire)
      const bool stall = std::is_same<Grid, SingleGrid>::value && p.stall;
      for (int t = stall ? total : grid.bx(); t < total && ok && !*abort_flag; t += grid.gdim(), ++in) {
        int mb, nb;
        coords(t, mb, nb);
        const int ab = in % FZ_ABUF;
        if (in >= FZ_ABUF) {
          next_done();
          if (!ok) break;
          if (!DW) bulk_wait_read0();
        }
        mbar_expect_tx(&a_full[ab], FZ_AT);
        a_inflight[ab] = ((in / FZ_ABUF) & 1) + 1;
        uint8_t* at = abase + ab * FZ_AT;
#pragma unroll
        for (int j = 0; j < 4; ++j) tma_load_3d(at + j * FZ_ABOX, mapA, &a_full[ab], j * 64, mb * BM, nb);
        if (!DW && t + grid.gdim() < total) {   // one buffer: the next tile waits in L2
          int mn, nn;
          coords(t + grid.gdim(), mn, nn);
#pragma unroll
          for (int j = 0; j < 4; ++j) tma_prefetch_3d(mapA, j * 64, mn * BM, nn);
        }
      }
      if constexpr (!DW) {
        while (ok && out < in && !*abort_flag) next_done();
        bulk_wait0();
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc_adj = make_idesc(1u, 1u, BN);   // W^T . Zbar, B MN-major, N = 256
      constexpr uint32_t idesc_dw = make_idesc(1u, 0u, 64);    // A_{l-1} . Zbar chunk^T, both K-major, N = 64
      const uint32_t d_dw = tmem_base + FZ_DW_COL;
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int t = grid.bx(); t < total && !*abort_flag && ok; t += grid.gdim(), ++local) {
        const int ab = local % FZ_ABUF, buf = local % ACC;
        const uint32_t d_adj = tmem_base + buf * BN;
        if constexpr (DW) {
          if (!mbar_wait(&a_full[ab], (uint32_t)(local / FZ_ABUF) & 1, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
          tc_fence_after();
        }
        const uint32_t sa_t = smem_u32(abase + ab * FZ_AT);
        for (int kb = 0; kb < p.k_iters; ++kb) {
          if (!mbar_wait(&full[stage], phase, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
          inflight[stage] = 0;
          tc_fence_after();
          const uint32_t sw = smem_u32(smem + stage * FZ_STAGE);
          const uint32_t sz = sw + FZ_WB;
          // weight gradient of this 64-row fout chunk: dW^T[:, 64 kb ..] += A_tile . Zbar_chunk^T
          if constexpr (DW) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                tc_mma<false>(d_dw + 64 * kb, make_desc(sa_t + j * FZ_ABOX + kk * 32, 16, 1024),
                              make_desc(sz + j * FZ_BOX + kk * 32, 16, 1024), idesc_dw,
                              (local > 0 || j > 0 || kk > 0) ? 1u : 0u);
          }
          if (kb == 0) {
            // wait until the epilogue has copied out the accumulator's last tile
            if (!mbar_wait(&acc_empty[buf], ((uint32_t)(local / ACC) & 1) ^ 1, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
            tc_fence_after();
          }
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc_mma<false>(d_adj, make_desc(sw + kk * 32, 16, 1024), make_desc(sz + kk * 16 * 128, FZ_BOX, 1024),
                          idesc_adj, (kb > 0 || kk > 0) ? 1u : 0u);
          tc_commit(&empty[stage]);
          if (++stage == FZ_STAGES) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        tc_commit(&acc_full[buf]);
      }
      if (DW && ok && !*abort_flag) tc_commit(dw_full);
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    constexpr int PARTS = FZ_EPI / 4;
    constexpr int UPTS = 16;
    constexpr int UNITS = TILE_PTS / (UPTS * PARTS);   // 2
    const int quad = warp & 3;
    const int part = (warp - 2) >> 2;
    const int rr = quad * 32 + lane;                    // accumulator row = feature within the m-tile
    auto unit_col = [&](int u) { return part * (UNITS * UPTS) + UPTS * u; };
    const uint32_t tq = tmem_base + ((uint32_t)(quad * 32) << 16);
    int local = 0;
    int mb_cta = 0;
    for (int t = grid.bx(); t < total; t += grid.gdim(), ++local) {
      int mb, nb;
      coords(t, mb, nb);
      mb_cta = mb;
      float xc[3] = {0.f, 0.f, 0.f};
      if (p.e.dbpart && p.e.dterms) lane_coords(p.e, (int64_t)nb * TILE_PTS + part * 32 + lane, xc);
      const int ab = local % FZ_ABUF, buf = local % ACC;
      bool ok = mbar_wait(&acc_full[buf], (uint32_t)(local / ACC) & 1, abort_flag, p.status, p.wait_ns);
      if (__any_sync(0xffffffffu, !ok)) break;   // (the warp's loads and shuffles are collective)
      tc_fence_after();
      float v[UNITS][4][UPTS];
#pragma unroll
      for (int u = 0; u < UNITS; ++u)
#pragma unroll
        for (int r = 0; r < 4; ++r) tmem_ld16_issue(tq + buf * BN + unit_col(u) + 64 * r, v[u][r]);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);   // the next tile's adjoint MMAs may overwrite it now
      ok = mbar_wait(&a_full[ab], (uint32_t)(local / FZ_ABUF) & 1, abort_flag, p.status, p.wait_ns);
      if (__any_sync(0xffffffffu, !ok)) break;
      a_inflight[ab] = 0;
      uint8_t* at = abase + ab * FZ_AT;
      const int m = mb * BM + rr;
      const bool mvalid = m < p.M;
      float db[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int u = 0; u < UNITS; ++u) {
        const int pc = unit_col(u);
#pragma unroll
        for (int h8 = 0; h8 < UPTS / 8; ++h8) {
          // A_{l-1} of 8 points x 4 jet rows from the swizzled tile (staged: Zbar_{l-1} back in
          // its place): row rr of box r, 16-byte chunk (pc + 8 h8) / 8 XOR (rr mod 8)
          uint32_t aw[4][4];
          const uint32_t addr = smem_u32(at + rr * 128 + ((((pc + 8 * h8) >> 3) ^ (rr & 7)) << 4));
#pragma unroll
          for (int r = 0; r < 4; ++r)
            asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(aw[r][0]), "=r"(aw[r][1]), "=r"(aw[r][2]), "=r"(aw[r][3])
                         : "r"(addr + r * FZ_ABOX));
          with_jet_mode(p.e.jet_mode, [&](auto mode) { adj_pairs8<decltype(mode)::value>(v[u], 8 * h8, aw); });
          if (!DW && p.e.out) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              uint32_t q[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const __nv_bfloat162 x = __floats2bfloat162_rn(v[u][r][8 * h8 + 2 * i], v[u][r][8 * h8 + 2 * i + 1]);
                q[i] = *reinterpret_cast<const uint32_t*>(&x);
              }
              asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr + r * FZ_ABOX), "r"(q[0]), "r"(q[1]),
                           "r"(q[2]), "r"(q[3])
                           : "memory");
            }
          }
        }
        if (u == UNITS - 1) {   // this warp is through with the tile: its accesses before the next bulk copy's
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&z_done[ab]);
        }
        if (DW && mvalid && p.e.out) {
          __nv_bfloat16* zbo = reinterpret_cast<__nv_bfloat16*>(p.e.out) + toff(m, (int64_t)nb * BN, p.M) + pc;
#pragma unroll
          for (int r = 0; r < 4; ++r) st_row(zbo + 64 * r, v[u][r]);
        }
        if (p.e.dbpart) {   // (every lane: rows past M add zeros that nobody stores)
#pragma unroll
          for (int i = 0; i < UPTS; ++i) db[0] += v[u][0][i];
          if (p.e.dterms) coord_terms<UPTS>(v[u], xc, u * UPTS, p.e.dterms, p.e.jet_mode, db);
        }
      }
      if (mvalid && p.e.dbpart) {
        float* dst = p.e.dbpart + ((int64_t)m * (p.n_tiles * PARTS) + nb * PARTS + part) * (1 + p.e.dterms);
        dst[0] = db[0];
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (j < p.e.dterms) dst[1 + j] = db[1 + j];
      }
    }
    // this CTA's dW^T slab (its m-tile rows x all fout) as split partial (CTA index) / m_tiles
    if (DW && local > 0 && !*abort_flag && mbar_wait(dw_full, 0, abort_flag, p.status, p.wait_ns)) {
      tc_fence_after();
      const int m = mb_cta * BM + rr;
      const int split = grid.bx() / p.m_tiles;
      const int f0 = part * 128;
      for (int c = 0; c < 128; c += 16) {
        if (f0 + c >= p.K) break;
        float d[16];
        tmem_ld16_issue(tq + FZ_DW_COL + f0 + c, d);
        tmem_wait_ld();
        if (m < p.M) {
          float* dst = p.out32 + ((int64_t)split * p.K + f0 + c) * p.M + m;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (f0 + c + i < p.K) dst[(int64_t)i * p.M] = d[i];
        }
      }
    }
  }

  // ---- teardown: wait (bounded) for copies and MMAs still in flight, free TMEM ----------------
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    for (int s = 0; s < FZ_STAGES; ++s) {
      const int f = inflight[s];
      if (f) {
        const uint64_t t0 = gtimer();
        while (!mbar_try(&full[s], (uint32_t)(f - 1)) && gtimer() - t0 < WAIT_NS) {}
      }
    }
    for (int b = 0; b < FZ_ABUF; ++b) {
      const int f = a_inflight[b];
      if (f) {
        const uint64_t t0 = gtimer();
        while (!mbar_try(&a_full[b], (uint32_t)(f - 1)) && gtimer() - t0 < WAIT_NS) {}
      }
    }
    abort_settle();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * BN));
  }
}

template <bool DW>
__global__ void __launch_bounds__(FZ_NT, 1)
    k_tc_adjdw(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapZ,
               const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapO,
               const __grid_constant__ TcParams p) {
  tc_adjdw_body<DW>(&mapW, &mapZ, &mapA, &mapO, p, SingleGrid{});
}

template <bool DW>
__global__ void __launch_bounds__(FZ_NT, 1) k_tc_adjdw_group(const TcGroupEntry* __restrict__ tab, const int n) {
  const TcGroupEntry& g = tab[group_of_block(tab, n, (int)blockIdx.x)];
  acquire_maps(g, 4);
  tc_adjdw_body<DW>(&g.map[0], &g.map[1], &g.map[2], &g.map[3], g.p, GroupShare{(int)blockIdx.x - g.block0, g.grid});
}

int adjdw_grid(const pinn_handle* h, int fin, int64_t NC) {
  const int mt = (fin + BM - 1) / BM;
  const int tiles = mt * (int)(NC / TILE_COLS);
  const int per = std::max(1, std::max(h->sm_count, 1) / mt) * mt;   // a multiple of the m-tile count
  return std::max(mt, std::min(tiles, per));
}

}  // namespace

namespace {

template <bool DW>
pinn_status launch_adjdw_group(pinn_handle* h, const TcGroupEntry* d_tab, int n, int blocks, cudaStream_t st) {
  pinn_status s = reserve_smem(h, k_tc_adjdw_group<DW>, FzCfg<DW>::SMEM, "grouped fused adjoint kernel");
  if (s) return s;
  k_tc_adjdw_group<DW><<<blocks, FZ_NT, FzCfg<DW>::SMEM, st>>>(d_tab, n);
  return launch_check(h, "grouped fused adjoint");
}

template <bool DW>
pinn_status launch_adjdw(pinn_handle* h, const CUtensorMap& w, const CUtensorMap& z, const CUtensorMap& a,
                         const CUtensorMap& o, const TcParams& p, int grid, cudaStream_t st) {
  if (h->tc_batch) {
    const CUtensorMap maps[4] = {w, z, a, o};
    return batch_add(h->tc_batch, &launch_adjdw_group<DW>, maps, 4, p, grid);
  }
  pinn_status s = reserve_smem(h, k_tc_adjdw<DW>, FzCfg<DW>::SMEM, "fused adjoint kernel");
  if (s) return s;
  k_tc_adjdw<DW><<<grid, FZ_NT, FzCfg<DW>::SMEM, st>>>(w, z, a, o, p);
  return launch_check(h, "fused adjoint");
}

}  // namespace

namespace {

// The BF16 tanh adjoint of a layer whose weight gradient runs on its own (fan-out above 256).
pinn_status adj_staged(pinn_handle* h, const void* WT, const void* Zbar, int fin, int fout, int64_t NC,
                       const EpiArgs& e, cudaStream_t st) {
  CUtensorMap mw, mz, ma, mo;
  const uint64_t nt = (uint64_t)(NC / TILE_COLS);
  if (!make_map(&mw, WT, false, fout, fin, 64, BM)) return map_err(h, "adjoint weights");
  if (!make_map3(&mz, Zbar, false, TILE_COLS, fout, nt, 64, 64)) return map_err(h, "adjoint input");
  if (!make_map3(&ma, e.ain, false, TILE_COLS, fin, nt, 64, BM)) return map_err(h, "adjoint activations");
  mo = ma;
  if (e.out && !make_map3(&mo, e.out, false, TILE_COLS, fin, nt, 64, BM)) return map_err(h, "adjoint output");
  TcParams p = base_params(h, fin, (int)NC, fout, NC, 64, h->d_status);
  p.e = e;
  return launch_adjdw<false>(h, mw, mz, ma, mo, p, grid_for(h, p.m_tiles * p.n_tiles), st);
}

}  // namespace

bool tc_adjdw_supported(const pinn_handle* h, int li, int64_t NC) {
  if (h->spec.precision != PINN_BF16 || li < 1 || !tc_layer_supported(h, li, NC)) return false;
  if (h->spec.flags & PINN_FLAG_UNFUSED_ADJOINT) return false;
  if (h->act != PINN_ACT_TANH) return false;   // the fused epilogue carries the tanh jet only
  return h->layers[li].fout <= BN;   // the dW^T slab fits beside the adjoint accumulator
}

int tc_adjdw_splits(const pinn_handle* h, int fin, int64_t NC) {
  return adjdw_grid(h, fin, NC) / ((fin + BM - 1) / BM);
}

pinn_status tc_gemm_adjdw(pinn_handle* h, const void* WT, const void* Zbar, const void* Ain, int fin, int fout,
                          int64_t NC, const EpiArgs& e, float* dwpart, int nsplit, cudaStream_t st) {
  CUtensorMap mw, mz, ma, mo;
  const uint64_t nt = (uint64_t)(NC / TILE_COLS);
  if (!make_map(&mw, WT, false, fout, fin, 64, BM)) return map_err(h, "fused adjoint weights");
  if (!make_map3(&mz, Zbar, false, TILE_COLS, fout, nt, 64, 64)) return map_err(h, "fused adjoint input");
  if (!make_map3(&ma, Ain, false, TILE_COLS, fin, nt, 64, BM)) return map_err(h, "fused adjoint activations");
  mo = ma;   // (not used: this form stores from registers)
  TcParams p = base_params(h, fin, (int)NC, fout, NC, 64, h->d_status);
  p.e = e;
  p.out32 = dwpart;
  const int grid = adjdw_grid(h, fin, NC);
  if (grid / p.m_tiles != nsplit || grid > p.m_tiles * p.n_tiles) {
    snprintf(h->err, sizeof(h->err), "fused adjoint: split plan mismatch");
    return PINN_ERR_INVALID_ARG;
  }
  p.nsplit = nsplit;
  return launch_adjdw<true>(h, mw, mz, ma, mo, p, grid, st);
}

// ==== the whole hidden forward in one kernel (BF16 tanh, every width <= 256) ===========
//
// Layer by layer, a 256-wide forward launch is bound by the data it moves between L2 and
// the SMs: the weights are re-streamed for every column tile, and the jets (with their
// value-row low halves) go out and come back once per layer.  Here a CTA takes one column
// tile (64 points) through every hidden GEMM layer: the tile's jets stay in shared memory,
// in the MN-major swizzled boxes that the MMAs read as their B operand, and each
// layer's epilogue writes its outputs back into them.  What leaves the SM is A_l (for the
// reverse sweep; bulk tensor stores straight from those boxes; nothing in a loss-only
// call) and, for the last layer only, the value-row low half; what comes in is the first
// layer's input and the weights.  Per accumulator element the MMAs, their order and the
// epilogue's arithmetic are those of k_tc_gemm<FWD>, so the results are bitwise the same.
// Measured against the per-layer launches (ms): 6x256 cavity at 69,632 points 0.480 -> 0.413,
// loss only at 266,240 points 1.566 -> 1.127; 4x128 at 17,408 points 0.053 -> 0.027.  What
// bounds it now: the MMAs, 219 cycles per K step where the tensor pipe alone would take 192
// (the N = 64 ones read as much of A from shared memory as the others: 48 cycles instead of
// 32), 8,000 of about 13,500 cycles per 256-wide layer and tile, then waits for weight stages.
//
// A layer is two jobs, each with one 256-column accumulator:
//   M2 (a width above 128): the two 128-row m-tiles of one column tile, whose boxes are
//      updated in place.  Both jobs take K chunks 0 and 1 (features 0-127) first, then both
//      take chunks 2 and 3: the next layer's first half runs on what the first job's
//      epilogue wrote while the second job's epilogue is still at work, and the first job's
//      epilogue may overwrite chunks 0 and 1 once its own accumulator is complete.
//   !M2 (widths <= 128): the same m-tile of two column tiles, one in each half of the
//      boxes, so one tile's epilogue runs under the other tile's MMAs.
//
// Warp roles (384 threads): 0 weight producer, 1 TMEM allocator + MMA issuer, 2-9
// epilogue, 10 input producer, 11 store issuer.  Barriers (all waits bounded, as in
// k_tc_gemm; no role meets another at a named barrier):
//   wfull/wempty[stage]  weight ring (hi and lo chunk of 128 rows x 64 K)
//   afull[slot][chunk]   first-layer input chunk has landed
//   afree[s]             the boxes of K half s (M2) or tile s (!M2) are free for new input
//   accf[h]              job h's accumulator is complete, and the boxes its epilogue writes are read
//   accr[h]              job h's epilogue has read its accumulator
//   done[h]              job h's epilogue has written its boxes (every layer but the last)
//   sread[h]             the bulk stores have read those boxes
namespace {

constexpr int FF_NT = FZ_NT + 32;
constexpr int FF_CHUNK = 4 * FZ_BOX;              // 64 features x 256 columns: 32 KB
constexpr int FF_HI = 4 * FF_CHUNK;               // 256 features of one tile, or 128 of two: 128 KB
constexpr int FF_LO = 4 * FZ_BOX;                 // their value-row low halves: 32 KB
constexpr int FF_WST = 2 * BM * 128;              // weight stage: W_hi and W_lo chunk, 32 KB
constexpr int FF_WSTAGES = 2;
constexpr size_t FF_SMEM = (size_t)FF_HI + FF_LO + (size_t)FF_WSTAGES * FF_WST + 1024 + 256;
static_assert(FF_SMEM <= 227 * 1024, "fused forward: shared memory budget");

struct FwdAllParams {
  CUtensorMap in, in_lo;                     // first GEMM layer's input jets and low half
  CUtensorMap w[PINN_MAX_HIDDEN], wlo[PINN_MAX_HIDDEN], out[PINN_MAX_HIDDEN];
  int fin[PINN_MAX_HIDDEN], fout[PINN_MAX_HIDDEN];
  const float* bias[PINN_MAX_HIDDEN];
  __nv_bfloat16* a_last;                     // A_L, tile-major
  __nv_bfloat16* alo_last;                   // its value-row low half
  int layers, ntiles, reverse, jet_mode, wlo_values_only;
  int store;                                 // write A_l of the layers below the last
  int* status;
  uint64_t wait_ns;
  int stall;                                 // test hook: the weight producer brings nothing
};

template <bool M2>
__global__ void __launch_bounds__(FF_NT, 1) k_tc_fwd_all(const __grid_constant__ FwdAllParams p) {
  constexpr int SLOTS = M2 ? 1 : 2;               // column tiles in flight
  constexpr int SCH = M2 ? 4 : 2;                 // 64-feature chunks per slot
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* lob = smem + FF_HI;
  uint8_t* wst = lob + FF_LO;
  uint64_t* wfull = reinterpret_cast<uint64_t*>(wst + FF_WSTAGES * FF_WST);
  uint64_t* wempty = wfull + FF_WSTAGES;
  uint64_t* afull = wempty + FF_WSTAGES;          // [4]: slot * SCH + chunk
  uint64_t* afree = afull + 4;                    // [2]
  uint64_t* accf = afree + 2;                     // [2]
  uint64_t* accr = accf + 2;                      // [2]
  uint64_t* done = accr + 2;                      // [2]
  uint64_t* sread = done + 2;                     // [2]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sread + 2);
  volatile int* w_inflight = abort_flag + 1;      // [FF_WSTAGES]
  volatile int* a_inflight = w_inflight + FF_WSTAGES;   // [4]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(a_inflight + 4));

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < FF_WSTAGES; ++i) {
      mbar_init(&wfull[i], 1);
      mbar_init(&wempty[i], 1);
      w_inflight[i] = 0;
    }
    for (int i = 0; i < 4; ++i) { mbar_init(&afull[i], 1); a_inflight[i] = 0; }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&afree[i], p.store ? 2 : 1);      // the last layer's MMAs, and the store issuer
      mbar_init(&accf[i], 1);
      mbar_init(&accr[i], FZ_EPI);                // one arrival per epilogue warp
      mbar_init(&done[i], FZ_EPI);
      mbar_init(&sread[i], 1);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int g = (int)gridDim.x, L = p.layers;
  // rounds of SLOTS tiles per CTA: tiles base, base + g, ...; job h of a round exists if its
  // tile does (M2: both jobs work on the one tile)
  auto has = [&](int base, int h) { return base + (M2 ? 0 : h * g) < p.ntiles; };
  auto tile_of = [&](int base, int h) {
    const int t = base + (M2 ? 0 : h) * g;
    return p.reverse ? p.ntiles - 1 - t : t;
  };
  // whether job h of layer l has rows (an M2 layer of at most 128 rows has one m-tile)
  auto rows = [&](int l, int h) { return !M2 || h == 0 || p.fout[l] > BM; };
  // the K chunks of a layer in two halves (M2), or all at once
  constexpr int HALVES = M2 ? 2 : 1, HCH = M2 ? 2 : 4;

  if (warp == 0) {
    // ---------------------------------------------------------------- weight producer
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 0;
      bool ok = true;
      // (test hook: with p.stall it brings nothing, and the waits for its weights expire)
      for (int base = p.stall ? p.ntiles : blockIdx.x; base < p.ntiles && ok; base += SLOTS * g)
        for (int l = 0; l < L && ok; ++l) {
          const int nk = (p.fin[l] + 63) >> 6;
          for (int hh = 0; hh < 2 * HALVES && ok; ++hh) {
            const int h = hh & 1, k0 = (hh >> 1) * HCH;
            if (!has(base, h) || !rows(l, h)) continue;
            for (int kb = k0; kb < min(nk, k0 + HCH); ++kb) {
              if (!mbar_wait(&wempty[st], ph ^ 1, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
              uint8_t* sw = wst + st * FF_WST;
              mbar_expect_tx(&wfull[st], FF_WST);
              w_inflight[st] = (int)ph + 1;
              tma_load_2d(sw, &p.w[l], &wfull[st], kb * 64, (M2 ? h : 0) * BM);
              tma_load_2d(sw + BM * 128, &p.wlo[l], &wfull[st], kb * 64, (M2 ? h : 0) * BM);
              if (++st == FF_WSTAGES) { st = 0; ph ^= 1; }
            }
          }
        }
    }
  } else if (warp == 2 + FZ_EPI) {
    // ---------------------------------------------------------------- input producer
    if (lane == 0) {
      const int nk = (p.fin[0] + 63) >> 6;
      uint32_t round = 0;
      bool ok = true;
      for (int base = blockIdx.x; base < p.ntiles && ok; base += SLOTS * g, ++round) {
        // one share of the boxes at a time: the K halves of the tile (M2), or the tiles
        for (int s = 0; s < 2 && ok; ++s) {
          if (!has(base, s)) continue;
          if (round && !mbar_wait(&afree[s], (round - 1) & 1, abort_flag, p.status, p.wait_ns)) { ok = false; break; }
          const int nb = tile_of(base, s), k0 = M2 ? HCH * s : 0;
          for (int kb = k0; kb < min(nk, k0 + HCH); ++kb) {
            const int c = (M2 ? 0 : s) * SCH + kb;
            mbar_expect_tx(&afull[c], FF_CHUNK + FZ_BOX);
            a_inflight[c] = (int)(round & 1) + 1;
#pragma unroll
            for (int j = 0; j < 4; ++j) tma_load_3d(smem + c * FF_CHUNK + j * FZ_BOX, &p.in, &afull[c], j * 64, kb * 64, nb);
            tma_load_3d(lob + c * FZ_BOX, &p.in_lo, &afull[c], 0, kb * 64, nb);
          }
        }
        // the CTAs work in step, so their input loads come in bursts: the next round's input
        // is brought into L2 under this round's layers
        const int next = base + SLOTS * g;
        for (int s = 0; s < SLOTS; ++s) {
          if (next >= p.ntiles || !has(next, s)) break;
          const int nb = tile_of(next, s);
          for (int kb = 0; kb < nk; ++kb) {
#pragma unroll
            for (int j = 0; j < 4; ++j) tma_prefetch_3d(&p.in, j * 64, kb * 64, nb);
            tma_prefetch_3d(&p.in_lo, 0, kb * 64, nb);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(1u, 1u, BN), idesc64 = make_idesc(1u, 1u, TILE_PTS);
      const uint32_t idesc_lo = p.wlo_values_only ? idesc64 : idesc;
      int st = 0;
      uint32_t ph = 0, round = 0;
      int jobs[2] = {0, 0};                       // jobs issued per accumulator
      int written[2] = {0, 0};                    // those of layers below the last
      bool ok = true;
      auto wait = [&](uint64_t* bar, uint32_t par) {
        if (ok) ok = mbar_wait(bar, par, abort_flag, p.status, p.wait_ns);
        return ok;
      };
      for (int base = blockIdx.x; base < p.ntiles && ok; base += SLOTS * g, ++round)
        for (int l = 0; l < L && ok; ++l) {
          const int nk = (p.fin[l] + 63) >> 6;
          for (int hh = 0; hh < 2 * HALVES && ok; ++hh) {
            const int h = hh & 1, half = hh >> 1, k0 = half * HCH;
            if (!has(base, h)) continue;
            const int slot = M2 ? 0 : h;
            // this half's input boxes are written, and (first half) the accumulator is free
            const int src = M2 ? half : h;
            if (l > 0 && k0 < nk && (!M2 || h == 0) && !wait(&done[src], (uint32_t)(written[src] - 1) & 1)) break;
            if (half == 0 && jobs[h] && !wait(&accr[h], (uint32_t)(jobs[h] - 1) & 1)) break;
            tc_fence_after();
            const uint32_t d = tmem_base + h * BN;
            for (int kb = k0; kb < min(nk, k0 + HCH) && rows(l, h); ++kb) {
              const int c = slot * SCH + kb;
              if (l == 0) {
                if (!wait(&afull[c], round & 1)) break;
                a_inflight[c] = 0;
              }
              if (!wait(&wfull[st], ph)) break;
              w_inflight[st] = 0;
              tc_fence_after();
              const uint32_t sa = smem_u32(wst + st * FF_WST), sa2 = sa + BM * 128;
              const uint32_t sb = smem_u32(smem + c * FF_CHUNK), sl = smem_u32(lob + c * FZ_BOX);
              // descriptors advance by 32 bytes (weights) and 16 rows of 128 bytes (jets) per K step,
              // in units of 16 bytes
              const uint64_t ad = make_desc(sa, 16, 1024), ad2 = make_desc(sa2, 16, 1024);
              const uint64_t bd = make_desc(sb, FZ_BOX, 1024), bl = make_desc(sl, FZ_BOX, 1024);
              const int left = p.fin[l] - 64 * kb;   // (K steps past it are zeros)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                if (16 * kk < left) {
                  tc_mma<false>(d, ad + 2 * kk, bd + 128 * kk, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
                  tc_mma<false>(d, ad2 + 2 * kk, bd + 128 * kk, idesc_lo, 1u);
                  tc_mma<false>(d, ad + 2 * kk, bl + 128 * kk, idesc64, 1u);
                }
              tc_commit(&wempty[st]);
              if (++st == FF_WSTAGES) { st = 0; ph ^= 1; }
            }
            if (!ok) break;
            // M2: job 0 is complete after its second half; without one (K <= 128) only once
            // job 1 has read the boxes too
            if (!M2) {
              tc_commit(&accf[h]);
              if (l == L - 1) tc_commit(&afree[h]);
            } else {
              if (half == 1 && nk <= HCH && h == 1) tc_commit(&accf[0]);
              if (half == 1 && (nk > HCH || h == 1)) tc_commit(&accf[h]);
              if (l == L - 1 && h == 1) tc_commit(&afree[half]);   // both jobs are through with this half
            }
            if (half == HALVES - 1) {
              ++jobs[h];
              if (l < L - 1) ++written[h];
            }
          }
        }
    }
  } else if (warp == 3 + FZ_EPI) {
    // ---------------------------------------------------------------- store issuer
    if (lane == 0 && p.store) {
      int jobs[2] = {0, 0};
      bool ok = true;
      for (int base = blockIdx.x; base < p.ntiles && ok; base += SLOTS * g)
        for (int l = 0; l < L && ok; ++l)
          for (int h = 0; h < 2 && ok; ++h) {
            if (!has(base, h)) continue;
            if (l == L - 1) {   // no store reads these boxes any more
              mbar_arrive(&afree[h]);
              continue;
            }
            ok = mbar_wait(&done[h], (uint32_t)jobs[h] & 1, abort_flag, p.status, p.wait_ns);
            if (!ok) break;
            const int nb = tile_of(base, h);
            for (int k = 0; k < 2 && rows(l, h); ++k) {
              const int f = (M2 ? h : 0) * BM + 64 * k;
              if (f >= p.fout[l]) break;
              const uint8_t* src = smem + ((M2 ? 0 : h) * SCH + (M2 ? 2 * h : 0) + k) * FF_CHUNK;
#pragma unroll
              for (int r = 0; r < 4; ++r) tma_store_3d(&p.out[l], src + r * FZ_BOX, 64 * r, f, nb);
            }
            bulk_commit();
            bulk_wait_read0();
            mbar_arrive(&sread[h]);
            ++jobs[h];
          }
      bulk_wait0();
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    constexpr int UPTS = 16, UNITS = 2;
    const int quad = warp & 3, part = (warp - 2) >> 2;
    const int rr = quad * 32 + lane;                // accumulator row
    int jobs[2] = {0, 0}, written[2] = {0, 0};
    bool ok = true;
    for (int base = blockIdx.x; base < p.ntiles && ok; base += SLOTS * g)
      for (int l = 0; l < L && ok; ++l)
        for (int h = 0; h < 2; ++h) {
          if (!has(base, h)) continue;
          const bool last = l == L - 1;
          const int slot = M2 ? 0 : h, nb = tile_of(base, h), M = p.fout[l];
          const int m = (M2 ? h : 0) * BM + rr;
          const float bias = m < M ? p.bias[l][m] : 0.f;
          ok = mbar_wait(&accf[h], (uint32_t)jobs[h] & 1, abort_flag, p.status, p.wait_ns);
          if (__any_sync(0xffffffffu, !ok)) { ok = false; break; }   // (the warp's loads and shuffles are collective)
          ++jobs[h];
          tc_fence_after();
          uint32_t hi[UNITS][4][8], lo[UNITS][8];   // packed BF16 results: 32 points x 4 rows, value-row low halves
          if (rows(l, h)) {
            const uint32_t tq = tmem_base + ((uint32_t)(quad * 32) << 16) + h * BN + part * (UNITS * UPTS);
            const uint32_t keep = m < M ? 0xffffffffu : 0u;   // rows past the layer's width: zeros that pad the next K
            auto unit = [&](int u, auto mode) {
              float v[4][UPTS];
#pragma unroll
              for (int r = 0; r < 4; ++r) tmem_ld16_issue(tq + UPTS * u + 64 * r, v[r]);
              tmem_wait_ld();
              if (u == UNITS - 1) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accr[h]);
              }
              fwd_pairs<decltype(mode)::value>(v, bias, hi[u], lo[u], keep);
            };
            auto units = [&](auto mode) {
#pragma unroll
              for (int u = 0; u < UNITS; ++u) unit(u, mode);
            };
            with_jet_mode(p.jet_mode, units);
          } else if (lane == 0) {
            mbar_arrive(&accr[h]);
          }
          if (last) {
            if (rows(l, h)) {
              store_pairs(p.a_last, hi, m, nb, M, part * (UNITS * UPTS));
              store_lo_pairs(p.alo_last, lo, m, nb, M, part * (UNITS * UPTS));
            }
            continue;
          }
          // the bulk stores of these boxes' previous contents have read them
          if (p.store && written[h]) {
            ok = mbar_wait(&sread[h], (uint32_t)(written[h] - 1) & 1, abort_flag, p.status, p.wait_ns);
            if (__any_sync(0xffffffffu, !ok)) { ok = false; break; }
          }
          ++written[h];
          if (rows(l, h)) {
            const int c = slot * SCH + (M2 ? 2 * h : 0) + (rr >> 6);
            const uint32_t row = smem_u32(smem + c * FF_CHUNK + (rr & 63) * 128);
            const uint32_t lrow = smem_u32(lob + c * FZ_BOX + (rr & 63) * 128);
#pragma unroll
            for (int u = 0; u < UNITS; ++u)
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                const uint32_t at = (uint32_t)(((part * 4 + 2 * u + q) ^ (rr & 7)) << 4);
#pragma unroll
                for (int r = 0; r < 4; ++r)
                  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(row + r * FZ_BOX + at), "r"(hi[u][r][4 * q]),
                               "r"(hi[u][r][4 * q + 1]), "r"(hi[u][r][4 * q + 2]), "r"(hi[u][r][4 * q + 3])
                               : "memory");
                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(lrow + at), "r"(lo[u][4 * q]),
                             "r"(lo[u][4 * q + 1]), "r"(lo[u][4 * q + 2]), "r"(lo[u][4 * q + 3])
                             : "memory");
              }
            fence_proxy_async_smem();               // these writes before the MMAs' and bulk stores' reads
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&done[h]);
        }
  }

  // ---- teardown: wait (bounded) for copies and MMAs still in flight, free TMEM ----------------
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    auto drain = [&](uint64_t* bar, int f) {
      if (!f) return;
      const uint64_t t0 = gtimer();
      while (!mbar_try(bar, (uint32_t)(f - 1)) && gtimer() - t0 < WAIT_NS) {}
    };
    for (int i = 0; i < FF_WSTAGES; ++i) drain(&wfull[i], w_inflight[i]);
    for (int i = 0; i < 4; ++i) drain(&afull[i], a_inflight[i]);
    abort_settle();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * BN));
  }
}

}  // namespace

bool tc_fwd_all_supported(const pinn_handle* h, int64_t NC) {
  if (h->spec.precision != PINN_BF16 || h->act != PINN_ACT_TANH || !fwd_in_one_kernel(h->L - h->first_gemm)) return false;
  for (int li = h->first_gemm; li < h->L; ++li)
    if (!tc_layer_supported(h, li, NC) || h->layers[li].fin > 256 || h->layers[li].fout > 256) return false;
  return true;
}

pinn_status tc_gemm_fwd_all(pinn_handle* h, const TcFwdLayer* layers, int n, const void* in, const void* in_lo,
                            void* alo_last, int64_t NC, int jet_mode, int reverse, int store, cudaStream_t st) {
  FwdAllParams p;
  const uint64_t nt = (uint64_t)(NC / TILE_COLS);
  bool ok = make_map3(&p.in, in, false, TILE_COLS, layers[0].fin, nt, 64, 64) &&
            make_map3(&p.in_lo, in_lo, false, TILE_PTS, layers[0].fin, nt, 64, 64);
  bool m2 = false;
  for (int l = 0; l < n && ok; ++l) {
    const TcFwdLayer& y = layers[l];
    ok = make_map(&p.w[l], y.W, false, y.fin, y.fout, 64, BM) && make_map(&p.wlo[l], y.Wlo, false, y.fin, y.fout, 64, BM) &&
         make_map3(&p.out[l], y.out, false, TILE_COLS, y.fout, nt, 64, 64);
    p.fin[l] = y.fin; p.fout[l] = y.fout; p.bias[l] = y.bias;
    m2 = m2 || y.fin > BM || y.fout > BM;
  }
  if (!ok) return map_err(h, "fused forward");
  p.a_last = reinterpret_cast<__nv_bfloat16*>(layers[n - 1].out);
  p.alo_last = reinterpret_cast<__nv_bfloat16*>(alo_last);
  p.layers = n; p.ntiles = (int)nt; p.reverse = reverse; p.jet_mode = jet_mode;
  p.store = store;
  p.wlo_values_only = (h->spec.flags & PINN_FLAG_BF16_VALUE_SPLIT) ? 1 : 0;
  p.status = h->d_status;
  p.wait_ns = h->stall_ns ? h->stall_ns : WAIT_NS;
  p.stall = h->stall_ns ? 1 : 0;
  auto kern = m2 ? k_tc_fwd_all<true> : k_tc_fwd_all<false>;
  const pinn_status s = reserve_smem(h, kern, FF_SMEM, "fused forward kernel");
  if (s) return s;
  kern<<<grid_for(h, p.ntiles), FF_NT, FF_SMEM, st>>>(p);
  return launch_check(h, "fused forward");
}

TcBatch* tc_batch_create() { return new (std::nothrow) TcBatch(); }

void tc_batch_destroy(TcBatch* b) {
  if (!b) return;
  if (b->d_table) cudaFree(b->d_table);
  delete b;
}

void tc_batch_attach(pinn_handle* h, TcBatch* b) { h->tc_batch = b; }

void tc_batch_reset(TcBatch* b) {
  b->pending.clear();
  b->table.clear();
  b->launches = 0;
}

pinn_status tc_batch_reserve(TcBatch* b, size_t entries) {
  if (entries <= b->capacity) return PINN_OK;
  if (b->d_table) cudaFree(b->d_table);
  b->d_table = nullptr;
  b->capacity = 0;
  if (cudaMalloc(&b->d_table, entries * sizeof(TcGroupEntry)) != cudaSuccess) {
    cudaGetLastError();
    return PINN_ERR_CUDA;
  }
  b->capacity = entries;
  return PINN_OK;
}

pinn_status tc_batch_flush(TcBatch* b, pinn_handle* h, cudaStream_t st) {
  // one grouped launch per kernel variant, in the order the variants first appeared
  std::vector<TcBatch::GroupFn> fns;
  for (const TcBatch::Item& it : b->pending)
    if (std::find(fns.begin(), fns.end(), it.fn) == fns.end()) fns.push_back(it.fn);
  pinn_status s = PINN_OK;
  for (TcBatch::GroupFn fn : fns) {
    std::vector<const TcBatch::Item*> items;
    for (const TcBatch::Item& it : b->pending)
      if (it.fn == fn) items.push_back(&it);
    // the GEMMs with the most work first, so that the small ones fill the tail
    std::stable_sort(items.begin(), items.end(),
                     [](const TcBatch::Item* x, const TcBatch::Item* y) { return x->work > y->work; });
    const size_t off = b->table.size();
    if (off + items.size() > b->capacity) {
      snprintf(h->err, sizeof(h->err), "grouped launch table full (%zu entries)", b->capacity);
      s = PINN_ERR_INVALID_ARG;
      break;
    }
    int blocks = 0;
    for (const TcBatch::Item* it : items) {
      TcGroupEntry e = it->e;
      e.block0 = blocks;
      blocks += e.grid;
      b->table.push_back(e);
    }
    s = fn(h, b->d_table + off, (int)items.size(), blocks, st);
    if (s) break;
    ++b->launches;
  }
  b->pending.clear();
  return s;
}

pinn_status tc_batch_upload(TcBatch* b) {
  if (b->table.empty()) return PINN_OK;
  if (cudaMemcpy(b->d_table, b->table.data(), b->table.size() * sizeof(TcGroupEntry), cudaMemcpyHostToDevice) !=
      cudaSuccess) {
    cudaGetLastError();
    return PINN_ERR_CUDA;
  }
  return PINN_OK;
}

int tc_batch_launches(const TcBatch* b) { return b->launches; }

}  // namespace pinn

// Raw tensor-core GEMM of the library's two operand layouts, FP32 output, for
// testing the MMA core in isolation (no epilogue).
namespace {
template <bool TF32>
pinn_status selftest_impl(pinn_handle* h, int layout, int M, int N, int K, const void* d_A, const void* d_A2,
                          const void* d_B, float* d_D, int* status, cudaStream_t st, uint64_t wait_ns = 0,
                          int stall = 0) {
  using namespace pinn;
  CUtensorMap ma, ma2, mb;
  if (layout == 0) {
    // D = A B: A [M][K] row-major, B [K][N] and D [M][N] in the tile-major jet layout
    using C = Cfg<TF32, TC_STORE, false>;
    if (!make_map(&ma, d_A, TF32, K, M, C::BKE, BM) || !make_map(&ma2, d_A2 ? d_A2 : d_A, TF32, K, M, C::BKE, BM) ||
        !make_map3(&mb, d_B, TF32, TILE_COLS, K, N / TILE_COLS, C::BOXN, C::BKE))
      return PINN_ERR_CUDA;
    TcParams p = base_params(h, M, N, K, N, C::BKE, status);
    p.out32 = d_D;
    if (stall) { p.wait_ns = wait_ns; p.stall = 1; }
    const int grid = grid_for(h, p.m_tiles * p.n_tiles);
    if (d_A2) return launch<TF32, TC_STORE, true>(h, ma, ma2, mb, mb, p, grid, st);
    return launch<TF32, TC_STORE, false>(h, ma, ma, mb, mb, p, grid, st);
  }
  // D = A B^T: A [M][K] and B [N][K] in the tile-major layout (K over jet columns), D [M][N]
  using C = Cfg<TF32, TC_DW, false>;
  if (!make_map3(&ma, d_A, TF32, TILE_COLS, M, K / TILE_COLS, C::BKE, BM) ||
      !make_map3(&mb, d_B, TF32, TILE_COLS, N, K / TILE_COLS, C::BKE, BN))
    return PINN_ERR_CUDA;
  TcParams p = base_params(h, M, N, K, N, C::BKE, status);
  p.out32 = d_D;
  return launch<TF32, TC_DW, false>(h, ma, ma, mb, mb, p, grid_for(h, p.m_tiles * p.n_tiles), st);
}
}  // namespace

extern "C" PINN_API pinn_status pinn_tc_selftest(int kind, int M, int N, int K, const void* d_A, const void* d_A2,
                                                 const void* d_B, float* d_D, void* stream) {
  using namespace pinn;
  if (!d_A || !d_B || !d_D || M < 1 || N < 1 || K < 1 || kind < 0 || kind > 3) return PINN_ERR_INVALID_ARG;
  const int layout = kind & 1;
  const bool tf32 = (kind & 2) != 0;
  if (tf32 && layout == 0) return PINN_ERR_UNSUPPORTED;   // kind::tf32 takes K-major operands only
  if (K % 8 || M % 8 || N % 8) return PINN_ERR_INVALID_ARG;
  if (layout == 0 && N % TILE_COLS) return PINN_ERR_INVALID_ARG;
  if (layout == 1 && K % TILE_COLS) return PINN_ERR_INVALID_ARG;
  pinn_handle h;
  tc_init(&h);
  if (!g_encode) return PINN_ERR_UNSUPPORTED;
  if (cudaGetDevice(&h.device) != cudaSuccess ||
      cudaDeviceGetAttribute(&h.sm_count, cudaDevAttrMultiProcessorCount, h.device) != cudaSuccess)
    return PINN_ERR_CUDA;
  int* status = nullptr;
  if (cudaMalloc(&status, sizeof(int)) != cudaSuccess) return PINN_ERR_CUDA;
  cudaMemsetAsync(status, 0, sizeof(int), (cudaStream_t)stream);
  pinn_status r = tf32 ? selftest_impl<true>(&h, layout, M, N, K, d_A, d_A2, d_B, d_D, status, (cudaStream_t)stream)
                       : selftest_impl<false>(&h, layout, M, N, K, d_A, d_A2, d_B, d_D, status, (cudaStream_t)stream);
  int st = 0;
  if (r == PINN_OK) {
    if (cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream) != cudaSuccess ||
        cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
      r = PINN_ERR_CUDA;
    else if (st & 2)
      r = PINN_ERR_TIMEOUT;
  }
  cudaFree(status);
  return r;
}

extern "C" PINN_API pinn_status pinn_debug_stall(pinn_handle* h, int64_t wait_us) {
  if (!h || wait_us < 0 || wait_us > 2000000) return PINN_ERR_INVALID_ARG;
  h->stall_ns = (uint64_t)wait_us * 1000ull;
  return PINN_OK;
}

extern "C" PINN_API pinn_status pinn_debug_wait_expiry(pinn_handle* h, int M, int N, int K, const void* d_A,
                                                       const void* d_B, float* d_D, int64_t wait_us, void* stream) {
  using namespace pinn;
  if (!h || !d_A || !d_B || !d_D || M < 1 || N < 1 || K < 1 || wait_us < 1 || wait_us > 2000000)
    return PINN_ERR_INVALID_ARG;
  if (K % 8 || M % 8 || N % TILE_COLS) return PINN_ERR_INVALID_ARG;
  if (!g_encode) return PINN_ERR_UNSUPPORTED;
  // the kind-0 BF16 GEMM with its MMA issuer waiting first on a barrier that nothing
  // arrives on: the wait expires after wait_us, and the kernel latches the timeout in
  // the handle's status word and returns through its abort path
  return selftest_impl<false>(h, 0, M, N, K, d_A, nullptr, d_B, d_D, h->d_status, (cudaStream_t)stream,
                              (uint64_t)wait_us * 1000ull, 1);
}
