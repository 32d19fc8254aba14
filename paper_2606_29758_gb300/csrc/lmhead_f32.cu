// f32 LM-head forward/backward on the CUDA cores.
//
// The tensor cores have no full-f32 mode (tf32 keeps a 10-bit mantissa), so f32
// inputs run here with exact f32 products and f32 accumulation, every element of Z, and of a dH or dW
// that is not split, over its k in increasing order. Split gradients (few tiles: launch_grad) add up 2, 4
// or 8 shares of k that way and then the shares in that order; whether they are split follows from the
// sizes of the whole call and the number of SMs. One tiled kernel computes C(m, n) = sum_k A(m, k) B(k, n) for
// operands whose k or whose m (n) is contiguous (Z = H W^T, dH = dZ W and dW = dZ^T H) and
// hands blocks of its tile to an epilogue: the forward's per-row (max, sum of exp) over 64
// columns (rows reduced across the 8 lanes that share them with warp shuffles), the
// backward's dZ, or a plain store.
#include <type_traits>

#include "internal.h"
#include "ps_common.cuh"

namespace psk {

constexpr int kSB = 64;   // columns per (max, sum) partial of the forward

// One operand: MN rows (A's m, B's n) by K, 16-byte aligned, ld % 4 == 0. K-major: element (i, k) at
// p[i ld + k], readable up to the next multiple of 4 of K; MN-major: at p[k ld + i], readable up to the
// next multiple of 4 of MN (what lies there never reaches an output: k past K reads as 0, and rows past
// MN are not stored).
struct Operand {
  const float* p;
  int64_t ld;
};

// (a.x b.x + c.x, a.y b.y + c.y), each one rounding: two FMAs per instruction.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  uint64_t ua, ub, uc, ud;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ua) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(ub) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(uc) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(ud) : "l"(ua), "l"(ub), "l"(uc));
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(ud));
  return d;
}

// A tile of TM x TN outputs by WM x WN warps, in k steps of BK. A warp owns 16 GM x 32 GN outputs, its lanes (ly, lx)
// of 4 x 8 the rows 4 ly + i + 16 g and the columns 4 lx + j + 32 h (i, j < 4) of them, so that its operands are 16-byte
// shared loads; neighbouring lanes differ in ly. PD: k steps whose global loads are in flight while one is computed (they
// wait in registers; shared memory holds two steps).
template <int TM_, int TN_, int WM_, int WN_, int BK_, int PD_, int MIN_BLOCKS>
struct SimtCfg {
  static constexpr int TM = TM_, TN = TN_, WN = WN_, BK = BK_, PD = PD_, kMinBlocks = MIN_BLOCKS;
  static constexpr int kThreads = 32 * WM_ * WN_;
  static constexpr int GM = TM / (16 * WM_), GN = TN / (32 * WN_);   // 4 x 4 blocks per thread
};
// The FP32 pipes are what bounds a product of many tiles; FFMA2 leaves issue slots for the shared loads
// (the same kernel on single FMAs was 7-20% slower). 6330 rows at d = 768, V = 8192 (79.6 GFLOP each): Z
// 1322 us on large tiles and 1452 on medium ones, dH 1425 and dW 1436 us on medium ones (large: 1839, 1581),
// i.e. 55-60 TFLOP/s of the 80.5 that 152 SMs x 128 lanes have at 2070 MHz. (With 2 x 16 lanes to a warp,
// and on medium tiles 8 x 4 outputs to a thread, Z 1334 / 1580, dH 1564, dW 1497; unpipelined 64 x 64 tiles with
// scalar loads 3960, 2500 and 3390 us. 8 x 16 and 16 x 8 outputs to a thread: Z 1349 and 1414, dH 1539 and 1497, dW
// 1643 and 1634.) Few tiles are bound by the latency of their k steps instead.
using SimtLarge = SimtCfg<64, 128, 2, 2, 16, 1, 3>;
using SimtMedium = SimtCfg<64, 64, 4, 1, 16, 2, 3>;
using SimtSmall = SimtCfg<32, 64, 2, 2, 32, 2, 3>;

// The T x BK slab of an operand that starts at row i0 and k0, through registers into s[BK][T + 4].
template <int T, int BK, int THREADS, bool KMAJOR>
struct SlabLoader {
  static constexpr int kVec = T * BK / 4 / THREADS;   // float4 per thread
  static_assert(T * BK % (4 * THREADS) == 0, "whole vectors per thread");
  float4 v[kVec];
  __device__ __forceinline__ void load(const Operand& o, int64_t i0, int64_t mn, int64_t k0, int64_t K, int tid) {
#pragma unroll
    for (int e = 0; e < kVec; ++e) {
      const int idx = tid + e * THREADS;
      v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (KMAJOR) {
        const int64_t i = i0 + idx / (BK / 4), k = k0 + idx % (BK / 4) * 4;
        if (i < mn && k < K) {
          v[e] = *reinterpret_cast<const float4*>(o.p + i * o.ld + k);
          if (k + 1 >= K) v[e].y = 0.f;
          if (k + 2 >= K) v[e].z = 0.f;
          if (k + 3 >= K) v[e].w = 0.f;
        }
      } else {
        const int64_t k = k0 + idx / (T / 4), i = i0 + idx % (T / 4) * 4;
        if (k < K && i < mn) v[e] = *reinterpret_cast<const float4*>(o.p + k * o.ld + i);
      }
    }
  }
  __device__ __forceinline__ void store(float (*s)[T + 4], int tid) const {
#pragma unroll
    for (int e = 0; e < kVec; ++e) {
      const int idx = tid + e * THREADS;
      if (KMAJOR) {
        const int i = idx / (BK / 4), k = idx % (BK / 4) * 4;
        s[k][i] = v[e].x;
        s[k + 1][i] = v[e].y;
        s[k + 2][i] = v[e].z;
        s[k + 3][i] = v[e].w;
      } else {
        *reinterpret_cast<float4*>(&s[idx / (T / 4)][idx % (T / 4) * 4]) = v[e];
      }
    }
  }
};

// Grid (column tiles, row tiles, ranks). With ranks > 1 (SPLIT: a cluster along z) each CTA of a cluster
// takes a share of the k steps, and the partial tiles, added in rank order, are read from the ranks'
// shared memory by the rank that stores their rows.
template <class Cfg, bool A_K, bool B_K, class Epi, bool SPLIT>
__global__ void __launch_bounds__(Cfg::kThreads, Cfg::kMinBlocks)
    simt_gemm_kernel(int64_t M, int64_t N, int64_t K, Operand A, Operand B, typename Epi::Params ep, uint32_t* clear) {
  wait_for_previous_kernel();
  // the call's first kernel zeroes the status (no CTA of this one sets a bit)
  if (clear != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) clear_status(clear);
  constexpr int TM = Cfg::TM, TN = Cfg::TN, BK = Cfg::BK, PD = Cfg::PD, GM = Cfg::GM, GN = Cfg::GN;
  struct Slabs {
    float a[2][BK][TM + 4];
    float b[2][BK][TN + 4];
  };
  __shared__ __align__(16) unsigned char smem[sizeof(Slabs)];
  Slabs& sm = *reinterpret_cast<Slabs*>(smem);
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int r0 = warp / Cfg::WN * 16 * GM + 4 * ((lane & 1) | ((lane >> 4) << 1));   // the thread's first row and column
  const int c0 = warp % Cfg::WN * 32 * GN + 4 * ((lane >> 1) & 7);                   // of the tile
  const int64_t m0 = static_cast<int64_t>(blockIdx.y) * TM;
  const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TN;
  int64_t kfirst = 0, steps = (K + BK - 1) / BK;
  if (SPLIT) {
    const int64_t all = steps, ranks = gridDim.z, rank = blockIdx.z;
    kfirst = all * rank / ranks;
    steps = all * (rank + 1) / ranks - kfirst;
  }
  float2 acc[4 * GM][2 * GN];
#pragma unroll
  for (int i = 0; i < 4 * GM; ++i)
#pragma unroll
    for (int j = 0; j < 2 * GN; ++j) acc[i][j] = make_float2(0.f, 0.f);

  SlabLoader<TM, BK, Cfg::kThreads, A_K> la[PD];
  SlabLoader<TN, BK, Cfg::kThreads, B_K> lb[PD];
  auto load = [&](int slot, int64_t step) {
    la[slot].load(A, m0, M, (kfirst + step) * BK, step < steps ? K : 0, tid);
    lb[slot].load(B, n0, N, (kfirst + step) * BK, step < steps ? K : 0, tid);
  };
#pragma unroll
  for (int s = 0; s < PD; ++s) load(s, s);
  la[0].store(sm.a[0], tid);
  lb[0].store(sm.b[0], tid);
  __syncthreads();
  for (int64_t t0 = 0; t0 < steps; t0 += PD) {
#pragma unroll
    for (int u = 0; u < PD; ++u) {
      const int64_t t = t0 + u;
      if (t >= steps) break;
      const int buf = static_cast<int>(t & 1);
      load(u, t + PD);   // slot u held step t, which is in shared memory by now
#pragma unroll
      for (int k = 0; k < BK; ++k) {
        float4 a[GM], b[GN];
#pragma unroll
        for (int g = 0; g < GM; ++g) a[g] = *reinterpret_cast<const float4*>(&sm.a[buf][k][r0 + 16 * g]);
#pragma unroll
        for (int h = 0; h < GN; ++h) b[h] = *reinterpret_cast<const float4*>(&sm.b[buf][k][c0 + 32 * h]);
#pragma unroll
        for (int g = 0; g < GM; ++g) {
          const float av[4] = {a[g].x, a[g].y, a[g].z, a[g].w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < GN; ++h) {
              const float2 aa = make_float2(av[i], av[i]);
              acc[4 * g + i][2 * h] = ffma2(aa, make_float2(b[h].x, b[h].y), acc[4 * g + i][2 * h]);
              acc[4 * g + i][2 * h + 1] = ffma2(aa, make_float2(b[h].z, b[h].w), acc[4 * g + i][2 * h + 1]);
            }
        }
      }
      if (t + 1 < steps) {   // step t + 1 into the other buffer, last read before the previous barrier
        la[(u + 1) % PD].store(sm.a[buf ^ 1], tid);
        lb[(u + 1) % PD].store(sm.b[buf ^ 1], tid);
      }
      __syncthreads();
    }
  }

  if constexpr (SPLIT) {
    static_assert(TM * TN * sizeof(float) <= sizeof(Slabs), "a partial tile lies over the slabs");
    float(*part)[TN] = reinterpret_cast<float(*)[TN]>(smem);
#pragma unroll
    for (int i = 0; i < 4 * GM; ++i)
#pragma unroll
      for (int h = 0; h < GN; ++h)
        *reinterpret_cast<float4*>(&part[r0 + (i & 3) + 16 * (i >> 2)][c0 + 32 * h]) =
            make_float4(acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x, acc[i][2 * h + 1].y);
    cluster_sync_all();   // every rank's partial is in its shared memory
    const int ranks = gridDim.z, rank = blockIdx.z;
    const uint32_t base = smem_addr(smem);
    for (int e = tid; e < TM / ranks * (TN / 4); e += Cfg::kThreads) {
      const int r = rank * (TM / ranks) + e / (TN / 4), c = e % (TN / 4) * 4;
      float4 v = ld_cluster_v4(mapa_shared(base + (r * TN + c) * 4, 0));
      for (int k = 1; k < ranks; ++k) {
        const float4 x = ld_cluster_v4(mapa_shared(base + (r * TN + c) * 4, k));
        v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
      }
      Epi::store4(ep, M, N, m0 + r, n0 + c, v);
    }
    cluster_sync_all();   // no rank exits while another reads its partial
  } else {
#pragma unroll
    for (int g = 0; g < GM; ++g) {
      float block[4][GN][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < GN; ++h) {
          block[i][h][0] = acc[4 * g + i][2 * h].x;
          block[i][h][1] = acc[4 * g + i][2 * h].y;
          block[i][h][2] = acc[4 * g + i][2 * h + 1].x;
          block[i][h][3] = acc[4 * g + i][2 * h + 1].y;
        }
      Epi::tile(ep, M, N, m0 + r0 + 16 * g, n0 + c0, block);
    }
  }
}

struct SimtFwdEpi {
  struct Params {
    const int32_t* tok;
    float2* part;   // [ceil(N / 64)][M]
    float* ztok;
    int tok_base;   // token ids are global; W holds vocabulary rows [tok_base, tok_base + N)
  };
  // a warp has 64 columns, from a multiple of 64 on; the 8 lanes of a row differ in bits 1 to 3 of their number
  static __device__ __forceinline__ void tile(const Params& p, int64_t M, int64_t N, int64_t r0, int64_t c0,
                                              float (&acc)[4][2][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t row = r0 + i;
      float x[8];
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        x[j] = (c0 + (j >> 2) * 32 + (j & 3) < N) ? acc[i][j >> 2][j & 3] * kLog2e : -INFINITY;
        mx = fmaxf(mx, x[j]);
      }
      const int t = row < M ? __ldg(p.tok + row) - p.tok_base : -1;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t c = c0 + (j >> 2) * 32 + (j & 3);
        if (c < N && c == t) p.ztok[row] = acc[i][j >> 2][j & 3];
      }
#pragma unroll
      for (int o = 8; o >= 2; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) s += exp2f(x[j] - mx);
#pragma unroll
      for (int o = 8; o >= 2; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if ((c0 & 63) == 0 && row < M && c0 < N) p.part[(c0 >> 6) * M + row] = make_float2(mx, s);
    }
  }
};

struct SimtDzEpi {
  struct Params {
    const int32_t* tok;
    const float* lse;
    const float* coef;
    float* dz;       // 16-byte aligned, ldz % 4 == 0
    int64_t ldz;
    int tok_base;
  };
  template <int GN>
  static __device__ __forceinline__ void tile(const Params& p, int64_t M, int64_t N, int64_t r0, int64_t c0,
                                              float (&acc)[4][GN][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t row = r0 + i;
      if (row >= M) continue;
      const int t = __ldg(p.tok + row) - p.tok_base;
      const float l = __ldg(p.lse + row), c = __ldg(p.coef + row);
#pragma unroll
      for (int h = 0; h < GN; ++h) {
        const int64_t col = c0 + 32 * h;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = c * ((col + j == t ? 1.f : 0.f) - expf(acc[i][h][j] - l));
        float* dst = p.dz + row * p.ldz + col;
        if (col + 4 <= N) {
          *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (col + j < N) dst[j] = v[j];
        }
      }
    }
  }
};

struct SimtStoreEpi {
  struct Params {
    float* out;     // 16-byte aligned, ld % 4 == 0, and N % 4 == 0: whole vectors
    int64_t ld;
    int accumulate;
  };
  static __device__ __forceinline__ void store4(const Params& p, int64_t M, int64_t N, int64_t row, int64_t col,
                                                float4 v) {
    if (row >= M || col >= N) return;
    float4* d = reinterpret_cast<float4*>(p.out + row * p.ld + col);
    if (p.accumulate) {
      const float4 o = *d;
      v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
    }
    *d = v;
  }
  template <int GN>
  static __device__ __forceinline__ void tile(const Params& p, int64_t M, int64_t N, int64_t r0, int64_t c0,
                                              float (&acc)[4][GN][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int h = 0; h < GN; ++h)
        store4(p, M, N, r0 + i, c0 + 32 * h, make_float4(acc[i][h][0], acc[i][h][1], acc[i][h][2], acc[i][h][3]));
  }
};

template <class Cfg>
static int64_t simt_tiles(int64_t M, int64_t N) {
  return ((M + Cfg::TM - 1) / Cfg::TM) * ((N + Cfg::TN - 1) / Cfg::TN);
}

template <class Cfg, bool A_K, bool B_K, class Epi>
static int launch_simt_cfg(int64_t M, int64_t N, int64_t K, int ranks, Operand A, Operand B,
                           const typename Epi::Params& ep, cudaStream_t s, uint32_t* clear = nullptr) {
  dim3 grid(static_cast<unsigned>((N + Cfg::TN - 1) / Cfg::TN), static_cast<unsigned>((M + Cfg::TM - 1) / Cfg::TM),
            static_cast<unsigned>(ranks));
  if constexpr (std::is_same<Epi, SimtStoreEpi>::value) {
    if (ranks > 1) {
      if (launch_after(simt_gemm_kernel<Cfg, A_K, B_K, Epi, true>, grid, Cfg::kThreads, 0, s, 1,
                       static_cast<unsigned>(ranks), true, M, N, K, A, B, ep, nullptr) == cudaSuccess)
        return PS_OK;
      cudaGetLastError();   // the stream's SMs do not take such a cluster: not split
      grid.z = 1;
    }
  }
  return launch_after(simt_gemm_kernel<Cfg, A_K, B_K, Epi, false>, grid, Cfg::kThreads, 0, s, 1, 1, clear == nullptr, M, N,
                      K, A, B, ep, clear) == cudaSuccess
             ? PS_OK
             : PS_ERR_CUDA;
}

// M tiles of 64 rows past the grid's y limit are refused.
static bool simt_fits(int64_t M) { return (M + kSB - 1) / kSB <= 65535; }

// Z = H W^T: large tiles from three per two SMs on (measured, large / medium: 256 tiles 73 / 78 us, 216
// tiles 30 / 25 us), medium ones below (small ones were never faster).
template <class Epi>
static int launch_z(int64_t M, int64_t N, int64_t K, Operand A, Operand B, const typename Epi::Params& ep,
                    cudaStream_t s, uint32_t* clear) {
  if (M == 0 || N == 0) return PS_OK;
  if (!simt_fits(M)) return PS_ERR_UNSUPPORTED;
  if (2 * simt_tiles<SimtLarge>(M, N) >= 3 * num_sms_current())
    return launch_simt_cfg<SimtLarge, true, true, Epi>(M, N, K, 1, A, B, ep, s, clear);
  return launch_simt_cfg<SimtMedium, true, true, Epi>(M, N, K, 1, A, B, ep, s, clear);
}

// dH = dZ W (its k steps are the vocabulary) and dW = dZ^T H (the rows) may have few tiles: the CTAs of a cluster
// then share the k steps where that shortens the longest SM's queue. n tiles on an SM take about 2.2, 2.5, 3, 4, 5,
// ... times the steps of one (three are resident), and the exchange costs about 60 such steps. Measured, 1 / 2 / 4 / 8
// ranks (us): dH at d = 768, V = 8192, 200 rows 233 / 160 / 108 / 78, 560 rows 235 / 215 / 154 / 170, 1200 rows 388 /
// 326 / 335 / 333, 2500 rows 754 / 719 / 652 / 664; dW unsplit / by this rule, 8000 rows: d = 128, V = 1024 208 / 53,
// d = 256, V = 3000 373 / 276, and (282 tiles, not split) d = 128, V = 9000 371 against 387 split.
// Below 32 tiles, small ones with 8 ranks (dH of 560 rows, d = 128, V = 1024: 8.2 us against 11.8 on medium tiles and
// 31 unsplit), and small ones too where an unsplit product would leave half of the SMs idle (dW there: 8.2 against
// 16.2 us).
// m_call: the rows of the whole call (dH) or of the whole vocabulary (dW), which decide, so that dH does not depend on
// how the call is cut into chunks and a vocabulary shard's dW rows are the whole head's.
template <bool A_K, bool B_K>
static int launch_grad(int64_t M, int64_t N, int64_t K, int64_t m_call, Operand A, Operand B,
                       const SimtStoreEpi::Params& ep, cudaStream_t s) {
  if (M == 0 || N == 0) return PS_OK;
  if (!simt_fits(M)) return PS_ERR_UNSUPPORTED;
  const int64_t tiles = simt_tiles<SimtMedium>(m_call, N);
  const int sms = num_sms_current();
  int ranks = 1;
  if (tiles < 32) {
    while (ranks < 8 && K >= 8 * ranks * SimtSmall::BK) ranks *= 2;
    return launch_simt_cfg<SimtSmall, A_K, B_K, SimtStoreEpi>(M, N, K, ranks, A, B, ep, s);
  }
  auto cost = [&](int r) {
    const int64_t n = (tiles * r + sms - 1) / sms, tenths = n == 1 ? 22 : n == 2 ? 25 : 10 * n;
    return tenths * ((K + SimtMedium::BK - 1) / SimtMedium::BK) / r + (r > 1 ? 600 : 0);
  };
  const int64_t most = A_K ? 4 * sms : 3 * sms / 2;   // from there on the exchanges cost what the last round gains
  for (int r = 2; r <= 8 && K >= 4 * r * SimtMedium::BK && tiles < most; r *= 2)
    if (cost(r) < cost(ranks)) ranks = r;
  if (ranks == 1 && 2 * tiles < sms) return launch_simt_cfg<SimtSmall, A_K, B_K, SimtStoreEpi>(M, N, K, 1, A, B, ep, s);
  return launch_simt_cfg<SimtMedium, A_K, B_K, SimtStoreEpi>(M, N, K, ranks, A, B, ep, s);
}

int fwd_splits_f32(int V) { return (V + kSB - 1) / kSB; }

int fwd_gemm_f32(int64_t N, int d, int V, const float* Hpk, const float* W, const int32_t* tok, float2* part,
                 float* ztok, uint32_t* status, cudaStream_t s, int tok_base) {
  return launch_z<SimtFwdEpi>(N, V, d, Operand{Hpk, d}, Operand{W, d}, SimtFwdEpi::Params{tok, part, ztok, tok_base},
                              s, status);
}

int bwd_chunk_f32(int64_t rc, int d, int V, const float* Hpk, const float* W, const int32_t* tok,
                  const float* lse, const float* coef, float* dH, float* dW, int dw_accumulate, float* dz,
                  int64_t ldz, uint32_t* status, cudaStream_t s, int tok_base, int dh_accumulate, int64_t n_call, int64_t v_call, bool clear) {
  int r = launch_z<SimtDzEpi>(rc, V, d, Operand{Hpk, d}, Operand{W, d},
                              SimtDzEpi::Params{tok, lse, coef, dz, ldz, tok_base}, s, clear ? status : nullptr);
  if (r != PS_OK) return r;
  if (dH) {  // dH(m=i, n=c) = sum_v dz[i][v] W[v][c]
    r = launch_grad<true, false>(rc, d, V, n_call, Operand{dz, ldz}, Operand{W, d},
                                 SimtStoreEpi::Params{dH, d, dh_accumulate}, s);
    if (r != PS_OK) return r;
  }
  if (dW) {  // dW(m=v, n=c) = sum_i dz[i][v] H[i][c]
    r = launch_grad<false, false>(V, d, rc, v_call, Operand{dz, ldz}, Operand{Hpk, d},
                                  SimtStoreEpi::Params{dW, d, dw_accumulate}, s);
  }
  return r;
}

}  // namespace psk
