// CUDA-core jet GEMMs: the FP32 path (k_f32_gemm, k_f32_dw), and the BF16 fallback for
// shapes the tensor-core kernels do not take (k_simt_gemm, k_simt_dw).  Same data layout
// as the tensor-core path (tile-major jet matrices, see jet.cuh); every thread owns whole
// points, so the jet rule and its adjoint are applied locally.
#include <algorithm>

#include "internal.h"
#include "jet.cuh"
#include "ptx.cuh"

namespace pinn {

namespace {

constexpr int BM = 64, BN = TILE_COLS, BK = 16, THREADS = 256;

__device__ __forceinline__ void load_vec8(const __nv_bfloat16* p, float v[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
    v[2 * i] = f.x; v[2 * i + 1] = f.y;
  }
}


// One block per (64 features, one 256-column tile = 64 points).  Thread (ty, tx)
// owns features 4ty..4ty+3 and points 4tx..4tx+3 of the tile, i.e. the columns
// 64 r + 4 tx + j of all four jet rows r, so the jet rule is thread-local.
// EPI 0: forward (bias on value rows, activation jet, writes A and the BF16 low half;
//        with the sine activation also the pre-activation jets Z)
// EPI 1: adjoint (reads A_{l-1}, or Z_{l-1} for sine, the jet adjoint, writes Zbar_{l-1})
// EPI 2: linear adjoint (writes W^T Zbar itself: the adjoint of the input jets)
template <int EPI, bool SINE>
__global__ void __launch_bounds__(THREADS) k_simt_gemm(const float* __restrict__ Aop,
                                                       const __nv_bfloat16* __restrict__ Bop,
                                                       const __nv_bfloat16* __restrict__ Blo, int M, int K,
                                                       int64_t NP, EpiArgs e) {
  using T = __nv_bfloat16;
  __shared__ float As[BK][BM + 4];
  __shared__ float Bs[BK][BN + 4];
  const int t = threadIdx.x;
  const int ty = t >> 4, tx = t & 15;
  const int m0 = blockIdx.y * BM;
  const int64_t tile = blockIdx.x;
  const int64_t n0 = tile * BN;
  float acc[4][16];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[i][j] = 0.f;

  for (int k0 = 0; k0 < K; k0 += BK) {
    {  // A tile: 64 rows x 16 k, 4 per thread
      const int i = t >> 2, kk = (t & 3) * 4;
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + i, k = k0 + kk + q;
        As[kk + q][i] = (m < M && k < K) ? Aop[(int64_t)m * K + k] : 0.f;
      }
    }
    {  // B tile: 16 k x 256 columns, 16 per thread (value columns add the low half)
      const int kk = t >> 4, c = (t & 15) * 16;
      float v[16];
      if (k0 + kk < K) {
        load_vec8(Bop + toff(k0 + kk, n0 + c, K), v);
        load_vec8(Bop + toff(k0 + kk, n0 + c, K) + 8, v + 8);
        if (Blo && c < TILE_PTS) {
          float lo[16];
          load_vec8(Blo + loff(k0 + kk, tile * TILE_PTS + c, K), lo);
          load_vec8(Blo + loff(k0 + kk, tile * TILE_PTS + c, K) + 8, lo + 8);
          for (int q = 0; q < 16; ++q) v[q] += lo[q];
        }
      } else {
        for (int q = 0; q < 16; ++q) v[q] = 0.f;
      }
      for (int q = 0; q < 16; ++q) Bs[kk][c + q] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w};
      float b[16];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][64 * r + 4 * tx]);
        b[4 * r] = b4.x; b[4 * r + 1] = b4.y; b[4 * r + 2] = b4.z; b[4 * r + 3] = b4.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  T* out = reinterpret_cast<T*>(e.out);
  for (int i = 0; i < 4; ++i) {
    const int f = m0 + ty * 4 + i;
    if (f >= M) continue;
    float o[4][4], zz[4][4];   // [row][point]
    if (EPI == 1 && SINE) {   // sine: the pre-activation jets of the layer below
      const float* zr = e.zin + toff(f, n0 + 4 * tx, M);
      for (int r = 0; r < 4; ++r) load4<float>(zr + 64 * r, zz[r]);
    } else if (EPI == 1) {   // tanh: the output jet of the layer below (value row: hi + lo for BF16)
      const T* ar = reinterpret_cast<const T*>(e.ain) + toff(f, n0 + 4 * tx, M);
      for (int r = 0; r < 4; ++r) load4<T>(ar + 64 * r, zz[r]);
      if (e.ain_lo) {
        float lo[4];
        load4<__nv_bfloat16>(reinterpret_cast<const __nv_bfloat16*>(e.ain_lo) + loff(f, tile * TILE_PTS + 4 * tx, M), lo);
        for (int j = 0; j < 4; ++j) zz[0][j] += lo[j];
      }
    }
    const float bias = (EPI == 0) ? e.bias[f] : 0.f;
    for (int j = 0; j < 4; ++j) {
      float z[4], a[4], ab[4];
      for (int r = 0; r < 4; ++r) {
        if (EPI == 0) z[r] = acc[i][4 * r + j] + (r == 0 ? bias : 0.f);
        else { z[r] = zz[r][j]; ab[r] = acc[i][4 * r + j]; }
      }
      if (EPI == 2) {
        for (int r = 0; r < 4; ++r) o[r][j] = acc[i][4 * r + j];
      } else if (EPI == 0) {
        if constexpr (SINE) {
          jet_fwd_sine(z, a, e.jet_mode, e.omega0);
          for (int r = 0; r < 4; ++r) zz[r][j] = z[r];
        } else {
          jet_fwd<true>(z, a, e.jet_mode);
        }
        for (int r = 0; r < 4; ++r) o[r][j] = a[r];
      } else {
        if constexpr (SINE) jet_adj_sine(z, ab, a, e.jet_mode, e.omega0);
        else jet_adj_a(z, ab, a, e.jet_mode);
        for (int r = 0; r < 4; ++r) o[r][j] = a[r];
      }
    }
    if (EPI == 0 && SINE) {
      float* zrow = e.zout + toff(f, n0 + 4 * tx, M);
      for (int r = 0; r < 4; ++r) store4<float>(zrow + 64 * r, zz[r]);
    }
    T* orow = out + toff(f, n0 + 4 * tx, M);
    for (int r = 0; r < 4; ++r) store4<T>(orow + 64 * r, o[r]);
    if (EPI == 0) {
      if (e.alo_out) {
        __nv_bfloat16* lo = reinterpret_cast<__nv_bfloat16*>(e.alo_out) + loff(f, tile * TILE_PTS + 4 * tx, M);
        for (int j = 0; j < 4; ++j)
          lo[j] = __float2bfloat16_rn(o[0][j] - __bfloat162float(__float2bfloat16_rn(o[0][j])));
      }
    }
  }
}

// Split-K weight gradient: part[s][m][n] = sum_{k in split s} Aop[m][k] Bop[n][k].
constexpr int DBM = 64, DBN = 64, DBK = 32;

__global__ void __launch_bounds__(THREADS) k_simt_dw(const __nv_bfloat16* __restrict__ Aop,
                                                     const __nv_bfloat16* __restrict__ Bop, int M, int N, int64_t NC,
                                                     int64_t kchunk, float* __restrict__ part) {
  __shared__ float As[DBK][DBM + 4];
  __shared__ float Bs[DBK][DBN + 4];
  const int t = threadIdx.x;
  const int ty = t >> 4, tx = t & 15;
  const int m0 = blockIdx.y * DBM, nn0 = blockIdx.x * DBN;
  const int s = blockIdx.z;
  const int64_t kb = (int64_t)s * kchunk, ke = min(NC, kb + kchunk);
  // A split sums up to NC / nsplit jet columns (hundreds of thousands at a million
  // points): each DBK-column block is summed on its own, and the block sums are added
  // to the running total with Kahan compensation, so the rounding error stays near
  // that of a DBK-term sum instead of growing with the split's length.
  float acc[4][4], comp[4][4];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) acc[i][j] = comp[i][j] = 0.f;
  for (int64_t k0 = kb; k0 < ke; k0 += DBK) {
    const int i = t >> 2, kk = (t & 3) * 8;   // 64 rows x 32 k, 8 per thread
    {
      float v[8];
      if (m0 + i < M) load_vec8(Aop + toff(m0 + i, k0 + kk, M), v);
      else
        for (int q = 0; q < 8; ++q) v[q] = 0.f;
      for (int q = 0; q < 8; ++q) As[kk + q][i] = v[q];
    }
    {
      float v[8];
      if (nn0 + i < N) load_vec8(Bop + toff(nn0 + i, k0 + kk, N), v);
      else
        for (int q = 0; q < 8; ++q) v[q] = 0.f;
      for (int q = 0; q < 8; ++q) Bs[kk + q][i] = v[q];
    }
    __syncthreads();
    float blk[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) blk[p][q] = 0.f;
#pragma unroll
    for (int k = 0; k < DBK; ++k) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) blk[p][q] = fmaf(a[p], b[q], blk[p][q]);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {   // Kahan: acc + blk with the lost low part kept in comp
        const float y = blk[p][q] - comp[p][q];
        const float t = acc[p][q] + y;
        comp[p][q] = (t - acc[p][q]) - y;
        acc[p][q] = t;
      }
    __syncthreads();
  }
  for (int p = 0; p < 4; ++p) {
    const int m = m0 + ty * 4 + p;
    if (m >= M) continue;
    for (int q = 0; q < 4; ++q) {
      const int n = nn0 + tx * 4 + q;
      if (n < N) part[((int64_t)s * M + m) * N + n] = acc[p][q];
    }
  }
}

// ==== FP32 storage ======================================================================
//
// Bound by the FP32 FMA pipe (80 TFLOP/s).  Kernels that wait for each K step's own global
// loads and spend an issue slot per FMA beside the shared-memory loads run at 30 (forward,
// adjoint) and 17 TFLOP/s (weight gradient).  Here operands arrive through a multi-stage
// cp.async ring and each thread keeps 64 accumulators; the forward and the adjoint use the
// packed fma.rn.f32x2: two IEEE FMAs per instruction, the rounding and the K order of scalar
// FMAs, at half the issue slots.  Results are bitwise those of the 4-wide kernels.  Measured
// on the 6x256 cavity at 17,408 points (ms per step, before -> after): forward 1.57 -> 1.02
// (54 TFLOP/s, FMA pipe 80% busy), adjoint 1.36 -> 0.88, weight gradient 2.92 -> 1.44.

// 16- / 4-byte asynchronous copies global -> shared; `ok` false writes zeros (nothing is read).
__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int FPTS = 32;             // points per block: half a 64-point tile
constexpr int FCOLS = 4 * FPTS;      // its jet columns
constexpr int FBK = 16;              // K per stage
constexpr int FSTAGES = 4;

template <int FM>
constexpr size_t f32_smem() { return (size_t)FSTAGES * FBK * (FM + FCOLS) * sizeof(float); }

// One block per (FM features, half a point tile); a thread owns 8 features x 2 points x 4
// jet rows as 32 packed accumulators (the two points of a row are one f32x2).  At is the
// left operand transposed, [K][M], so both operands are copied as they lie; rows of At
// that are no multiple of 16 bytes (M % 4) take 4-byte copies.  EPI as in k_simt_gemm.
template <int FM, int EPI, bool SINE>
__global__ void __launch_bounds__(2 * FM, FM == 128 ? 2 : 4)
    k_f32_gemm(const float* __restrict__ At, const float* __restrict__ Bop, int M, int K, EpiArgs e) {
  constexpr int NT = 2 * FM;
  extern __shared__ __align__(16) float fsm[];
  float* As = fsm;                                  // [FSTAGES][FBK][FM]
  float* Bs = fsm + FSTAGES * FBK * FM;             // [FSTAGES][FBK][FCOLS], column = 32 r + point
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * FM;
  const int64_t tile = blockIdx.x >> 1;
  const int half = blockIdx.x & 1;
  const float* Bt = Bop + tile * K * TILE_COLS + FPTS * half;
  const bool vec = (M & 3) == 0;
  const int nk = (K + FBK - 1) / FBK;

  auto load = [&](int kt) {
    if (kt < nk) {
      float* a = As + (kt % FSTAGES) * FBK * FM;
      float* b = Bs + (kt % FSTAGES) * FBK * FCOLS;
      const int k0 = kt * FBK;
      if (vec) {
#pragma unroll
        for (int i = t; i < FBK * FM / 4; i += NT) {
          const int kk = i / (FM / 4), c = 4 * (i % (FM / 4));
          const bool ok = k0 + kk < K && m0 + c < M;
          cp16(a + kk * FM + c, ok ? At + (int64_t)(k0 + kk) * M + m0 + c : At, ok);
        }
      } else {
        for (int i = t; i < FBK * FM; i += NT) {
          const int kk = i / FM, c = i % FM;
          const bool ok = k0 + kk < K && m0 + c < M;
          cp4(a + kk * FM + c, ok ? At + (int64_t)(k0 + kk) * M + m0 + c : At, ok);
        }
      }
#pragma unroll
      for (int i = t; i < FBK * FCOLS / 4; i += NT) {
        const int kk = i >> 5, r = (i >> 3) & 3, q = 4 * (i & 7);
        const bool ok = k0 + kk < K;
        cp16(b + kk * FCOLS + FPTS * r + q, ok ? Bt + (int64_t)(k0 + kk) * TILE_COLS + TILE_PTS * r + q : Bt, ok);
      }
    }
    cp_commit();
  };

  f32x2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[i][r] = 0ull;
#pragma unroll
  for (int s = 0; s < FSTAGES - 1; ++s) load(s);
  for (int kt = 0; kt < nk; ++kt) {
    cp_wait<FSTAGES - 2>();
    __syncthreads();
    load(kt + FSTAGES - 1);
    const float* a = As + (kt % FSTAGES) * FBK * FM + 4 * ty;
    const float* b = Bs + (kt % FSTAGES) * FBK * FCOLS + 2 * tx;
#pragma unroll
    for (int kk = 0; kk < FBK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(a + kk * FM);
      const float4 a1 = *reinterpret_cast<const float4*>(a + kk * FM + FM / 2);
      f32x2 bb[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) bb[r] = *reinterpret_cast<const f32x2*>(b + kk * FCOLS + FPTS * r);
      const f32x2 av[8] = {dup2(a0.x), dup2(a0.y), dup2(a0.z), dup2(a0.w), dup2(a1.x), dup2(a1.y), dup2(a1.z), dup2(a1.w)};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[i][r] = fma2(av[i], bb[r], acc[i][r]);
    }
  }

  float* out = reinterpret_cast<float*>(e.out);
  const int pc = FPTS * half + 2 * tx;              // first of the thread's two points in the tile
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int f = m0 + (i < 4 ? 0 : FM / 2) + 4 * ty + (i & 3);
    if (f >= M) continue;
    const int64_t o = toff(f, tile * TILE_COLS, M) + pc;
    float v[4][2], zz[4][2];                        // [row][point]
#pragma unroll
    for (int r = 0; r < 4; ++r) unpack2(acc[i][r], v[r][0], v[r][1]);
    if constexpr (EPI == 1) {   // the jets of the layer below: outputs (tanh) or pre-activations (sine)
      const float* src = SINE ? e.zin + o : reinterpret_cast<const float*>(e.ain) + o;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float2 q = *reinterpret_cast<const float2*>(src + TILE_PTS * r);
        zz[r][0] = q.x; zz[r][1] = q.y;
      }
    }
    if constexpr (EPI == 0) {
      const float bias = e.bias[f];
#pragma unroll
      for (int j = 0; j < 2; ++j) v[0][j] += bias;
      if constexpr (SINE) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          *reinterpret_cast<float2*>(e.zout + o + TILE_PTS * r) = make_float2(v[r][0], v[r][1]);
      }
    }
    if constexpr (EPI != 2) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float x[4] = {v[0][j], v[1][j], v[2][j], v[3][j]};
        float y[4];
        if constexpr (EPI == 0) {
          if constexpr (SINE) jet_fwd_sine(x, y, e.jet_mode, e.omega0);
          else jet_fwd<false>(x, y, e.jet_mode);
        } else {
          const float z[4] = {zz[0][j], zz[1][j], zz[2][j], zz[3][j]};
          if constexpr (SINE) jet_adj_sine(z, x, y, e.jet_mode, e.omega0);
          else jet_adj_a(z, x, y, e.jet_mode);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r][j] = y[r];
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) *reinterpret_cast<float2*>(out + o + TILE_PTS * r) = make_float2(v[r][0], v[r][1]);
  }
}

// Split-K weight gradient, part[s][m][n] = sum over the columns of split s of A[m][k] B[n][k]
// (both tile-major, K contiguous): 64 x 64 outputs per block, 8 x TJ per thread (TJ = 8: two
// warps per block, four blocks per SM).  Both operands keep their layout in shared memory: with a
// row pitch of 36 floats the 16-byte reads along K of eight neighbouring rows fall on
// distinct banks.  Every DBK columns are summed on their own and added to the running total
// with Kahan compensation, as in k_simt_dw and in the same order: the rounding error stays
// near that of a 32-term sum however long the split is, and repeated training steps stay
// bitwise what they were.
constexpr int WT = 64, WBK = DBK, WPITCH = WBK + 4, WSTAGES = 3;
constexpr size_t W_SMEM = (size_t)WSTAGES * 2 * WT * WPITCH * sizeof(float);

template <int TJ>
__global__ void __launch_bounds__(512 / TJ, TJ == 8 ? 4 : 2) k_f32_dw(const float* __restrict__ Aop, const float* __restrict__ Bop,
                                                       int M, int N, int64_t NC, int64_t kchunk,
                                                       float* __restrict__ part) {
  extern __shared__ __align__(16) float fsm[];
  constexpr int NT = 512 / TJ, CX = WT / TJ;             // threads; threads along the columns
  const int t = threadIdx.x, tx = t % CX, ty = t / CX;   // rows ty + 8 i, columns tx + CX j
  const int n0 = blockIdx.x * WT, m0 = blockIdx.y * WT, s = blockIdx.z;
  const int64_t kb = (int64_t)s * kchunk, ke = min(NC, kb + kchunk);
  const int nk = ke > kb ? (int)((ke - kb) / WBK) : 0;   // NC and kchunk are multiples of 32

  auto load = [&](int kt) {
    if (kt < nk) {
      float* a = fsm + (kt % WSTAGES) * 2 * WT * WPITCH;
      float* b = a + WT * WPITCH;
      const int64_t k0 = kb + (int64_t)kt * WBK;
#pragma unroll
      for (int i = t; i < WT * WBK / 4; i += NT) {
        const int row = i >> 3, q = 4 * (i & 7);
        const bool oa = m0 + row < M, ob = n0 + row < N;
        cp16(a + row * WPITCH + q, oa ? Aop + toff(m0 + row, k0 + q, M) : Aop, oa);
        cp16(b + row * WPITCH + q, ob ? Bop + toff(n0 + row, k0 + q, N) : Bop, ob);
      }
    }
    cp_commit();
  };

  float acc[8][TJ], comp[8][TJ];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) acc[i][j] = comp[i][j] = 0.f;
#pragma unroll
  for (int q = 0; q < WSTAGES - 1; ++q) load(q);
  for (int kt = 0; kt < nk; ++kt) {
    float blk[8][TJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < TJ; ++j) blk[i][j] = 0.f;
    cp_wait<WSTAGES - 2>();
    __syncthreads();
    load(kt + WSTAGES - 1);
    const float* a = fsm + (kt % WSTAGES) * 2 * WT * WPITCH + ty * WPITCH;
    const float* b = fsm + (kt % WSTAGES) * 2 * WT * WPITCH + (WT + tx) * WPITCH;
#pragma unroll 2
    for (int k = 0; k < WBK; k += 2) {
      float2 bv[TJ];
#pragma unroll
      for (int j = 0; j < TJ; ++j) bv[j] = *reinterpret_cast<const float2*>(b + CX * j * WPITCH + k);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 av = *reinterpret_cast<const float2*>(a + 8 * i * WPITCH + k);
#pragma unroll
        for (int j = 0; j < TJ; ++j) blk[i][j] = fmaf(av.x, bv[j].x, blk[i][j]);
#pragma unroll
        for (int j = 0; j < TJ; ++j) blk[i][j] = fmaf(av.y, bv[j].y, blk[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < TJ; ++j) {   // Kahan: acc + blk with the lost low part kept in comp
        const float y = blk[i][j] - comp[i][j];
        const float u = acc[i][j] + y;
        comp[i][j] = (u - acc[i][j]) - y;
        acc[i][j] = u;
      }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + ty + 8 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < TJ; ++j) {
      const int n = n0 + tx + CX * j;
      if (n < N) part[((int64_t)s * M + m) * N + n] = acc[i][j];
    }
  }
}

template <int TJ>
cudaError_t f32_dw_launch(pinn_handle* h, const void* Aop, const void* Bop, int M, int N, int64_t NC, int nsplit,
                          int64_t kchunk, float* part, cudaStream_t st) {
  const cudaError_t err = allow_smem(h, reinterpret_cast<const void*>(k_f32_dw<TJ>), W_SMEM);
  if (err != cudaSuccess) return err;
  dim3 grid((N + WT - 1) / WT, (M + WT - 1) / WT, nsplit);
  k_f32_dw<TJ><<<grid, 512 / TJ, W_SMEM, st>>>((const float*)Aop, (const float*)Bop, M, N, NC, kchunk, part);
  return cudaGetLastError();
}

template <int FM, int EPI, bool SINE>
cudaError_t f32_gemm_launch(pinn_handle* h, const float* At, const void* Bop, int M, int K, int64_t NP, const EpiArgs& e,
                            cudaStream_t st) {
  auto kern = k_f32_gemm<FM, EPI, SINE>;
  const cudaError_t err = allow_smem(h, reinterpret_cast<const void*>(kern), f32_smem<FM>());
  if (err != cudaSuccess) return err;
  kern<<<dim3((unsigned)(NP / FPTS), (M + FM - 1) / FM), 2 * FM, f32_smem<FM>(), st>>>(At, (const float*)Bop, M, K, e);
  return cudaGetLastError();
}

// 128-feature blocks read each jet column half as often as 64-feature ones; they are
// taken once they fill two blocks on every SM, below that the smaller blocks spread
// the work over more SMs.
template <int EPI, bool SINE>
cudaError_t f32_gemm(pinn_handle* h, const float* At, const void* Bop, int M, int K, int64_t NP, const EpiArgs& e,
                     cudaStream_t st) {
  if (M > 64 && (NP / FPTS) * ((M + 127) / 128) >= 2 * (int64_t)h->sm_count)
    return f32_gemm_launch<128, EPI, SINE>(h, At, Bop, M, K, NP, e, st);
  return f32_gemm_launch<64, EPI, SINE>(h, At, Bop, M, K, NP, e, st);
}

}  // namespace

cudaError_t launch_simt_gemm_fwd(pinn_handle* h, const float* W, const float* WT, const void* Bop, int M, int K,
                                 int64_t NP, const EpiArgs& e, int prec, cudaStream_t st) {
  if (prec != PINN_BF16)
    return e.act ? f32_gemm<0, true>(h, WT, Bop, M, K, NP, e, st) : f32_gemm<0, false>(h, WT, Bop, M, K, NP, e, st);
  dim3 grid((unsigned)(NP / TILE_PTS), (M + BM - 1) / BM);
  const __nv_bfloat16* B = (const __nv_bfloat16*)Bop;
  const __nv_bfloat16* Blo = (const __nv_bfloat16*)e.alo_in;
  if (e.act) k_simt_gemm<0, true><<<grid, THREADS, 0, st>>>(W, B, Blo, M, K, NP, e);
  else k_simt_gemm<0, false><<<grid, THREADS, 0, st>>>(W, B, Blo, M, K, NP, e);
  return cudaGetLastError();
}

cudaError_t launch_simt_gemm_adj(pinn_handle* h, const float* WT, const float* W, const void* Bop, int M, int K,
                                 int64_t NP, const EpiArgs& e, int prec, cudaStream_t st) {
  if (prec != PINN_BF16)
    return e.act ? f32_gemm<1, true>(h, W, Bop, M, K, NP, e, st) : f32_gemm<1, false>(h, W, Bop, M, K, NP, e, st);
  dim3 grid((unsigned)(NP / TILE_PTS), (M + BM - 1) / BM);
  const __nv_bfloat16* B = (const __nv_bfloat16*)Bop;
  if (e.act) k_simt_gemm<1, true><<<grid, THREADS, 0, st>>>(WT, B, nullptr, M, K, NP, e);
  else k_simt_gemm<1, false><<<grid, THREADS, 0, st>>>(WT, B, nullptr, M, K, NP, e);
  return cudaGetLastError();
}

cudaError_t launch_simt_gemm_lin(pinn_handle* h, const float* WT, const float* W, const void* Bop, int M, int K,
                                 int64_t NP, void* out, int prec, cudaStream_t st) {
  EpiArgs e{};
  e.out = out;
  if (prec != PINN_BF16) return f32_gemm<2, false>(h, W, Bop, M, K, NP, e, st);
  dim3 grid((unsigned)(NP / TILE_PTS), (M + BM - 1) / BM);
  k_simt_gemm<2, false><<<grid, THREADS, 0, st>>>(WT, (const __nv_bfloat16*)Bop, nullptr, M, K, NP, e);
  return cudaGetLastError();
}

cudaError_t launch_simt_gemm_dw(pinn_handle* h, const void* Aop, const void* Bop, int M, int N, int64_t NC, int nsplit,
                                float* part, int prec, cudaStream_t st) {
  const int64_t per = (NC + nsplit - 1) / nsplit;
  const int64_t kchunk = (per + DBK - 1) / DBK * DBK;
  if (prec != PINN_BF16) {
    // Short splits (a few stages per block, few blocks) are bound by latency: twice the
    // threads per block, half the columns each (4x64 network at 4,608 points: 13 us per launch
    // against 17; at 17,408 points and 256 wide 0.28 ms against 0.24).
    return kchunk <= 8 * DBK ? f32_dw_launch<4>(h, Aop, Bop, M, N, NC, nsplit, kchunk, part, st)
                             : f32_dw_launch<8>(h, Aop, Bop, M, N, NC, nsplit, kchunk, part, st);
  }
  dim3 grid((N + DBN - 1) / DBN, (M + DBM - 1) / DBM, nsplit);
  k_simt_dw<<<grid, THREADS, 0, st>>>((const __nv_bfloat16*)Aop, (const __nv_bfloat16*)Bop, M, N, NC, kchunk, part);
  return cudaGetLastError();
}

}  // namespace pinn
