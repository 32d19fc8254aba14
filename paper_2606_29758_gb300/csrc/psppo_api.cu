// C ABI of libpsppo: argument checks, workspace layout, and the SIMT kernels of the
// pass (cutoff sampling, packing, forward finalisation). The GEMM-shaped steps live
// in lmhead_bf16.cu (tensor cores) and lmhead_f32.cu (CUDA cores).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <climits>
#include <cstdint>

#include "ps_nvtx.h"
#include "internal.h"
#include "ps_common.cuh"
#include "psppo.h"
#include "psppo_diag.h"

namespace psk {

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int num_sms_current() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 1;
  return n;
}

int device_is_sm103() {
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  return major == 10 && minor == 3;
}

static int check_ws(const void* ws, size_t ws_bytes, size_t need) {
  if (ws == nullptr || (reinterpret_cast<uintptr_t>(ws) & 255)) return PS_ERR_WORKSPACE;
  return ws_bytes < need ? PS_ERR_WORKSPACE : PS_OK;
}
// The workspace checked and its status zeroed. (Calls whose first kernel zeroes it use check_ws alone.)
static int begin_call(void* ws, size_t ws_bytes, size_t need, cudaStream_t s) {
  const int rc = check_ws(ws, ws_bytes, need);
  if (rc != PS_OK) return rc;
  if (cudaMemsetAsync(ws, 0, kWsHeader, s) != cudaSuccess) return PS_ERR_CUDA;
  return PS_OK;
}

// An error before such a first kernel was launched: the status is zeroed here instead.
int refused(int rc, void* ws, cudaStream_t s) {
  cudaMemsetAsync(ws, 0, kWsHeader, s);
  return rc;
}

static uint32_t* status_word(void* ws) { return static_cast<uint32_t*>(ws); }
// A second word of the header, zeroed with the status at the call's start: a count of finished blocks.
static uint32_t* ticket_word(void* ws) { return static_cast<uint32_t*>(ws) + 1; }

constexpr uint64_t kCutoffKeyTag = 0x5053505030303031ull;  // "PSPP0001"

// ================================================================== K1: cutoff sampler
// Saturating scans of the masses give U[h]; S[t] = 2^62 - U[t-1]; a completion's bucket is the first h with its draw x
// below U[h], looked for by bisection in the tile of steps whose U span x (a thread per draw; with the thread of every
// bucket going through all draws a prompt of 512 completions and 100 steps took 33 us instead of 8.5).
// A prompt's steps are shared by blockIdx.y of the grid: what costs is a step's f64 division (an SM of GB300 does
// two FP64 operations a clock), so one CTA per prompt took 81 us for 2 prompts x 16384 steps and 36 us for one of
// 7220, against 14 and 8.4 us with 64 and 29 CTAs each. Every CTA adds up the whole row of masses itself
// (integers, from L2) rather than wait for the CTAs before it; kSampMaxParts bounds that reading.
constexpr int kSampThreads = 256;
constexpr int kSampMaxParts = 64;
constexpr uint64_t kSatCap = kOne62 + 1;   // any prefix above 2^62 is invalid; saturate just past it

__device__ __forceinline__ uint64_t sat_add(uint64_t a, uint64_t b) {
  const uint64_t s = a + b;  // a, b <= kSatCap so no wrap
  return s > kSatCap ? kSatCap : s;
}

__global__ void __launch_bounds__(kSampThreads)
    sample_cutoffs_kernel(int K, int T_max, const uint64_t* __restrict__ q, const int32_t* __restrict__ L,
                          uint64_t seed, uint64_t step, int64_t traj_base, int mode, int32_t* __restrict__ H,
                          int32_t* __restrict__ n, float* __restrict__ w_tab, uint32_t* status) {
  extern __shared__ uint64_t xs[];  // [K] draws
  constexpr int kWarps = kSampThreads / 32;
  __shared__ uint64_t warp_tot[kWarps], warp_before[kWarps], u_s[kSampThreads];
  const int p = blockIdx.x;
  const int tid = threadIdx.x;
  const bool first_part = blockIdx.y == 0;
  const int64_t wrow = static_cast<int64_t>(p) * T_max;
  // this CTA's steps [t_begin, t_end): whole tiles of kSampThreads
  const int64_t tiles = (T_max + kSampThreads - 1) / kSampThreads;
  const int t_begin = static_cast<int>(tiles * blockIdx.y / gridDim.y * kSampThreads);
  const int t_end = min(T_max, static_cast<int>(tiles * (blockIdx.y + 1) / gridDim.y * kSampThreads));

  for (int j = tid; j < K; j += blockDim.x) {
    const int k = p * K + j;
    if (first_part) {
      const int Lk = L[k];
      if (Lk < 1 || Lk > T_max) raise_status(status, PS_DEV_BAD_LENGTH);
      if (mode == PS_MODE_FULL) {
        H[k] = Lk;
        n[k] = Lk;
      }
    }
    if (mode != PS_MODE_FULL) {
      uint64_t c[4] = {static_cast<uint64_t>(traj_base + k), step, 0ull, 0ull};
      philox4x64_10(c, seed, kCutoffKeyTag);
      xs[j] = c[0] >> 2;
    }
  }
  if (mode == PS_MODE_FULL) {
    for (int t = t_begin + tid; t < t_end; t += blockDim.x) w_tab[wrow + t] = 1.0f;
    return;
  }
  const int lane = tid & 31, wid = tid >> 5;
  // Total mass U[T] and the mass before this CTA's steps (saturating). Exact mode requires U[T] = 2^62; in the
  // H = 0 mode the deficit 2^62 - U[T] is Pr(H = 0) and the survival is S[t] = U[T] - U[t-1].
  uint64_t part = 0, before = 0;
#pragma unroll 4
  for (int t = tid; t < T_max; t += kSampThreads) {
    const uint64_t m = q[wrow + t];
    part = sat_add(part, m > kOne62 ? kSatCap : m);
    if (t < t_begin) before = part;   // (a tile lies on one side of t_begin)
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    part = sat_add(part, __shfl_xor_sync(0xffffffffu, part, o));
    before = sat_add(before, __shfl_xor_sync(0xffffffffu, before, o));
  }
  if (lane == 0) {
    warp_tot[wid] = part;
    warp_before[wid] = before;
  }
  __syncthreads();
  uint64_t mass = 0, carry = 0;
  for (int w = 0; w < kWarps; ++w) {
    mass = sat_add(mass, warp_tot[w]);
    carry = sat_add(carry, warp_before[w]);
  }
  if (first_part) {
    if (tid == 0 && (mass > kOne62 || (mode == PS_MODE_TRUNC && mass != kOne62))) raise_status(status, PS_DEV_BAD_PMF);
    for (int j = tid; j < K; j += blockDim.x)   // a draw at or above U[T]
      if (xs[j] >= mass) {
        H[p * K + j] = 0;
        n[p * K + j] = 0;
      }
  }
  const uint64_t total = mass > kOne62 ? kOne62 : mass;

  for (int base = t_begin; base < t_end; base += kSampThreads) {
    __syncthreads();
    const int t = base + tid;  // 0-based: bucket h = t + 1
    uint64_t m = t < T_max ? q[wrow + t] : 0ull;
    if (m > kOne62) {
      raise_status(status, PS_DEV_BAD_PMF);
      m = kSatCap;
    }
    uint64_t v = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v = sat_add(v, y);
    }
    if (lane == 31) warp_tot[wid] = v;
    __syncthreads();
    const uint64_t tile_from = carry;
    uint64_t prior = carry;          // up to this warp
    for (int w = 0; w < kWarps; ++w) {
      if (w < wid) prior = sat_add(prior, warp_tot[w]);
      carry = sat_add(carry, warp_tot[w]);
    }
    const uint64_t incl = sat_add(prior, v);  // U[h]
    const uint64_t left = __shfl_up_sync(0xffffffffu, v, 1);
    const uint64_t excl = lane > 0 ? sat_add(prior, left) : prior;   // U[h-1]
    u_s[tid] = incl;
    __syncthreads();
    if (t < T_max) {
      // S[t+1] = U[T] - U[t]; weight 2^62 / S (f64 divide, rounded once to f32)
      float wt;
      if (excl >= total) {
        wt = INFINITY;
        if (excl > kOne62) raise_status(status, PS_DEV_BAD_PMF);
      } else {
        const double S = __ull2double_rn(total - excl);
        wt = __double2float_rn(__ddiv_rn(4611686018427387904.0, S));
      }
      w_tab[wrow + t] = wt;
    }
    for (int j = kSampThreads - 1 - tid; j < K; j += kSampThreads) {   // from the last thread on: a short trace leaves it free
      const uint64_t x = xs[j];
      if (x < tile_from || x >= carry) continue;
      const int k = p * K + j, Lk = L[k];
      int lo = 0, hi = kSampThreads - 1;   // the first step with x < u_s; the last one is carry
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (x < u_s[mid]) hi = mid;
        else lo = mid + 1;
      }
      const bool valid = u_s[lo] <= kOne62;   // a bucket past 2^62 (an invalid row) decides nothing
      const int h = base + lo + 1;
      H[k] = valid ? h : 0;
      n[k] = valid ? min(h, Lk) : 0;
    }
  }
}

// ================================================================== K2: packing
// Workspace after the header: off_L [B+1] int64, A [B] f64, N (int64).
struct PackWs {
  int64_t* off_L;
  double* A;
  int64_t* N;
};
static PackWs pack_ws(void* ws, int B) {
  uint8_t* base = static_cast<uint8_t*>(ws) + kWsHeader;
  PackWs w;
  w.off_L = reinterpret_cast<int64_t*>(base);
  base += align_up(sizeof(int64_t) * (B + 1), 256);
  w.A = reinterpret_cast<double*>(base);
  base += align_up(sizeof(double) * B, 256);
  w.N = reinterpret_cast<int64_t*>(base);
  return w;
}

// CTA 0: scans of L and n. The others: group advantages, a warp per prompt (sequential f64 sums per group, no FMA
// contraction, so the result is the correctly rounded sequence of the stated operations; the divisions, one per
// completion, by its lanes). Latency-bound: with one CTA that scanned through 20 barriers and a thread per prompt
// that divided one completion after another it took 14.6 us for 2 prompts x 16, now 4.1.
constexpr int kMetaThreads = 1024;
constexpr int kAdvWarps = 4;   // per CTA: more would wait for each other's double operations
__global__ void __launch_bounds__(kMetaThreads)
    pack_meta_kernel(int P, int K, int T_max, const int32_t* __restrict__ L, const int32_t* __restrict__ n,
                     const float* __restrict__ R, int adv_mode, int64_t capacity, int32_t* __restrict__ cu_seqlens,
                     PackWs w, uint32_t* status) {
  constexpr int kWarps = kMetaThreads / 32;
  const int B = P * K;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (blockIdx.x == 0) {
    __shared__ int64_t warp_l[kWarps], warp_n[kWarps];
    int64_t carry_l = 0, carry_n = 0;
    if (threadIdx.x == 0) clear_status(status);   // the call's first kernel; only this CTA sets bits
    __syncthreads();
    for (int base = 0; base < B; base += kMetaThreads) {
      const int k = base + threadIdx.x;
      int64_t lk = 0, nk = 0;
      if (k < B) {
        lk = L[k];
        nk = n[k];
        if (lk < 1 || lk > T_max || nk < 0 || nk > lk) {
          raise_status(status, PS_DEV_BAD_LENGTH);
          lk = lk < 0 ? 0 : lk;
          nk = nk < 0 ? 0 : (nk > lk ? lk : nk);
        }
      }
      int64_t sl = lk, sn = nk;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t yl = __shfl_up_sync(0xffffffffu, sl, o), yn = __shfl_up_sync(0xffffffffu, sn, o);
        if (lane >= o) {
          sl += yl;
          sn += yn;
        }
      }
      if (lane == 31) {
        warp_l[wid] = sl;
        warp_n[wid] = sn;
      }
      __syncthreads();
      // the warps' sums, scanned by every warp for itself
      int64_t tl = warp_l[lane], tn = warp_n[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t yl = __shfl_up_sync(0xffffffffu, tl, o), yn = __shfl_up_sync(0xffffffffu, tn, o);
        if (lane >= o) {
          tl += yl;
          tn += yn;
        }
      }
      const int64_t before_l = __shfl_sync(0xffffffffu, tl, wid - 1), before_n = __shfl_sync(0xffffffffu, tn, wid - 1);
      if (wid > 0) {
        sl += before_l;
        sn += before_n;
      }
      if (k < B) {
        w.off_L[k] = carry_l + sl - lk;
        const int64_t cu = carry_n + sn - nk;
        cu_seqlens[k] = static_cast<int32_t>(cu > INT32_MAX ? INT32_MAX : cu);
      }
      carry_l += __shfl_sync(0xffffffffu, tl, 31);
      carry_n += __shfl_sync(0xffffffffu, tn, 31);
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      w.off_L[B] = carry_l;
      int64_t N = carry_n;
      if (N > capacity || N > INT32_MAX || carry_l > INT32_MAX) {
        raise_status(status, PS_DEV_CAPACITY);
        N = 0;  // write no rows
      }
      cu_seqlens[B] = static_cast<int32_t>(carry_n > INT32_MAX ? INT32_MAX : carry_n);
      *w.N = N;
    }
    return;
  }
  if (wid >= kAdvWarps) return;
  const int warps = (gridDim.x - 1) * kAdvWarps;
  for (int p = (blockIdx.x - 1) * kAdvWarps + wid; p < P; p += warps) {
    const float* Rp = R + static_cast<int64_t>(p) * K;
    double* Ap = w.A + static_cast<int64_t>(p) * K;
    double s = 0.0;
    for (int j = 0; j < K; ++j) s = __dadd_rn(s, static_cast<double>(Rp[j]));
    const double mu = __ddiv_rn(s, static_cast<double>(K));
    if (adv_mode == PS_ADV_CENTERED) {
      for (int j = lane; j < K; j += 32) Ap[j] = __dsub_rn(static_cast<double>(Rp[j]), mu);
      continue;
    }
    double ss = 0.0;
    for (int j = 0; j < K; ++j) {
      const double dv = __dsub_rn(static_cast<double>(Rp[j]), mu);
      ss = __dadd_rn(ss, __dmul_rn(dv, dv));
    }
    const double sigma = __dsqrt_rn(__ddiv_rn(ss, static_cast<double>(K)));
    const double den = __dadd_rn(sigma, 1e-6);
    for (int j = lane; j < K; j += 32) Ap[j] = __ddiv_rn(__dsub_rn(static_cast<double>(Rp[j]), mu), den);
  }
}

// One warp per packed row: lane 0 locates (k, t) by binary search over cu_seqlens and
// writes the row's scalars; the warp copies the hidden row with 16-byte accesses.
constexpr int kPackThreads = 256;
__global__ void __launch_bounds__(kPackThreads)
    pack_rows_kernel(int B, int K, int T_max, const int32_t* __restrict__ cu_seqlens, PackWs w,
                     const float* __restrict__ w_tab, const int32_t* __restrict__ tok_full,
                     const float* __restrict__ oldlogp_full, const uint4* __restrict__ hid_full, int64_t row_vec,
                     int32_t* __restrict__ src_row, int32_t* __restrict__ row_traj, int32_t* __restrict__ row_pos,
                     int32_t* __restrict__ tok, float* __restrict__ oldlogp, float* __restrict__ wout,
                     float* __restrict__ adv, uint4* __restrict__ hid_packed) {
  wait_for_previous_kernel();
  const int64_t N = *w.N;
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < N; i += warps) {
    int64_t src = 0;
    if (lane == 0) {
      int lo = 0, hi = B - 1;  // largest k with cu_seqlens[k] <= i
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cu_seqlens[mid] <= i) lo = mid;
        else hi = mid - 1;
      }
      const int k = lo;
      const int t = static_cast<int>(i - cu_seqlens[k]) + 1;
      src = w.off_L[k] + t - 1;
      if (src_row) src_row[i] = static_cast<int32_t>(src);
      if (row_traj) row_traj[i] = k;
      if (row_pos) row_pos[i] = t;
      tok[i] = tok_full[src];
      oldlogp[i] = oldlogp_full[src];
      wout[i] = w_tab[static_cast<int64_t>(k / K) * T_max + (t - 1)];
      adv[i] = __double2float_rn(w.A[k]);
    }
    if (hid_full == nullptr) continue;
    src = __shfl_sync(0xffffffffu, src, 0);
    const uint4* s = hid_full + src * row_vec;
    uint4* d = hid_packed + i * row_vec;
    int64_t c = lane;
    for (; c + 96 < row_vec; c += 128) {
      const uint4 v0 = s[c], v1 = s[c + 32], v2 = s[c + 64], v3 = s[c + 96];
      d[c] = v0;
      d[c + 32] = v1;
      d[c + 64] = v2;
      d[c + 96] = v3;
    }
    for (; c < row_vec; c += 32) d[c] = s[c];
  }
}

// ================================================================== K4: forward finalize
constexpr int kFinThreads = 256;

// One packed row of the forward (Eq. 1 through the head, the loss of Eq. truncated_update_Ghat):
// from the row's logsumexp in base 2, lse2 = m + log2(S) (m the base-2 maximum, S the sum of
// 2^(x - m) over the vocabulary), and its chosen logit zt. Returns the row's loss term.
__device__ __forceinline__ double finalize_row(int64_t i, float m, float S, float zt, int t, int V,
                                               const float* __restrict__ oldlogp, const float* __restrict__ adv,
                                               const float* __restrict__ w, double eps, double loss_scale,
                                               float* __restrict__ lse, float* __restrict__ logp,
                                               float* __restrict__ ratio, float* __restrict__ coef,
                                               float* __restrict__ row_loss, uint32_t* status) {
  const double l = (static_cast<double>(m) + log2(static_cast<double>(S))) * 0.6931471805599453;
  double lp;
  if (t < 0 || t >= V) {
    raise_status(status, PS_DEV_BAD_TOKEN);
    lp = NAN;
  } else {
    lp = static_cast<double>(zt) - l;
  }
  const double r = exp(lp - static_cast<double>(oldlogp[i]));
  const double A = adv[i], wt = w[i];
  // min and clip as the definition has them: a NaN ratio (a non-finite input or a bad token
  // id) gives a NaN surrogate, which fmin / fmax alone would replace by the other operand
  const double clipped = r != r ? r : fmin(fmax(r, 1.0 - eps), 1.0 + eps);
  const double ra = r * A, ca = clipped * A;
  const double sur = (ra != ra || ca != ca) ? NAN : fmin(ra, ca);
  const double rl = -loss_scale * wt * sur;
  const bool bind = (A > 0.0 && r > 1.0 + eps) || (A < 0.0 && r < 1.0 - eps);
  lse[i] = static_cast<float>(l);
  logp[i] = static_cast<float>(lp);
  ratio[i] = static_cast<float>(r);
  coef[i] = bind ? 0.f : static_cast<float>(-loss_scale * wt * A * r);
  if (row_loss) row_loss[i] = static_cast<float>(rl);
  return rl;
}

// The (max, sum) pairs of `count` parts of a row's vocabulary (stride `stride` between parts),
// merged into one pair: m = max m_s, S = sum S_s 2^(m_s - m).
__device__ __forceinline__ float2 merge_parts(const float2* __restrict__ part, int count, int64_t stride) {
  float m = -INFINITY;
  for (int s = 0; s < count; ++s) m = fmaxf(m, part[static_cast<int64_t>(s) * stride].x);
  float S = 0.f;
  for (int s = 0; s < count; ++s) {
    const float2 pr = part[static_cast<int64_t>(s) * stride];
    S += pr.y * exp2f(pr.x - m);
  }
  return make_float2(m, S);
}

// A block of the forward's finalize (and of the shard statistics' merge) takes 8, 16 or 32 rows. Its threads find the
// maximum m of each row's parts and copy the parts, chunk by chunk, into a ring in shared memory; all warps but the
// first turn every x into 2^(x - m), and a lane of warp 0 per row adds the products of the chunk before up in
// vocabulary order, as merge_parts does, whatever the batch around the row. (Sums over slices of the parts, rescaled and merged,
// need one reading but left the lse 0.2 to 0.8% further from 64 bits: a mean error of 2.139e-5 instead of 2.134e-5 over
// 185 rows at V = 152064.) Bound by reading the parts twice, the second time mostly from L2 (a row of the 152k
// vocabulary has 1188, 9.5 KB; once where the ring holds them all), and for few rows by the 2.5 us that 1188 dependent
// additions take. Whole kernel at V = 152064: 185 rows 16 us, 8000 rows 32, 106000 rows 329; V = 2000: 7.8, 9.2 and 33.
// (The same sum by one thread per row that reads its parts twice: 204, 230 and 8.0, 9.2 at 185 and 8000 rows.)
constexpr int kMergeBatch = 6;                     // parts per thread and chunk
constexpr int kMergeStages = 4;                    // two in flight, one converted, one added up
template <int R, int THREADS>
struct MergeCfg {
  static constexpr int kRows = R, kThreads = THREADS;
  static constexpr int kMakers = THREADS - 32;                 // the threads that copy and convert
  static constexpr int kChunk = kMakers * kMergeBatch;         // elements of a chunk
  static constexpr int kParts = kChunk / R, kSlices = kMakers / R;   // its parts, and the threads per row
  static_assert(kMakers % R == 0 && kParts * R == kChunk, "whole parts");
};

__device__ __forceinline__ void cp_async_8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The merged (max, sum) of the block's `rows` <= R rows, row i's in lane i of warp 0. part: the first row's first part,
// `count` parts `stride` apart. Every thread of the block calls it. Shared memory: min(chunks, kMergeStages) chunks.
template <class C>
__device__ __forceinline__ float2 merge_parts_block(const float2* part, int count, int64_t stride, int rows) {
  extern __shared__ __align__(16) float2 ring[];
  constexpr int R = C::kRows, kSlices = C::kSlices, kParts = C::kParts, kMakers = C::kMakers;
  __shared__ float max_s[C::kThreads / 32][R];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int maker = static_cast<int>(threadIdx.x) - 32, r = threadIdx.x % R;
  const bool live = r < rows;
  const int chunks = (count + kParts - 1) / kParts;
  const bool held = chunks <= kMergeStages;   // every part stays in the ring
  auto fetch = [&](int k) {   // this thread's parts of chunk k
    int c = k * kParts + maker / R;
    const float2* p = part + c * stride + r;
    float2* to = ring + k % kMergeStages * C::kChunk + maker;
#pragma unroll
    for (int j = 0; j < kMergeBatch; ++j, c += kSlices, p += kSlices * stride, to += kMakers)
      if (live && c < count) cp_async_8(to, p);
    cp_async_commit();
  };
  if (maker >= 0)
    for (int k = 0; k < (held ? chunks : 2); ++k) fetch(k);
  float m = -INFINITY;
  if (held) {
    cp_async_wait<0>();
    if (maker >= 0 && live)
#pragma unroll 6
      for (int c = maker / R, e = maker; c < count; c += kSlices, e += kMakers) m = fmaxf(m, ring[e].x);
  } else if (live) {
    constexpr int kAll = C::kThreads / R, kFly = 12;
    int c = threadIdx.x / R;
    const float2* p = part + c * stride + r;
    for (; c + (kFly - 1) * kAll < count; c += kFly * kAll, p += kFly * kAll * stride) {
      float x[kFly];
#pragma unroll
      for (int j = 0; j < kFly; ++j) x[j] = p[j * (kAll * stride)].x;
#pragma unroll
      for (int j = 0; j < kFly; ++j) m = fmaxf(m, x[j]);
    }
#pragma unroll 4
    for (; c < count; c += kAll, p += kAll * stride) m = fmaxf(m, p->x);
  }
#pragma unroll
  for (int o = 16; o >= R; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane < R) max_s[warp][lane] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < C::kThreads / 32; ++w) m = fmaxf(m, max_s[w][r]);
  float S = 0.f;
  for (int k = 0; k <= chunks; ++k) {   // chunk k is converted and chunk k - 1 added
    if (maker >= 0) {
      if (k < chunks) {
        if (!held) {
          fetch(k + 2);   // where chunk k - 2 was, added in the round before
          cp_async_wait<2>();
        }
        const int c = k * kParts + maker / R;
        float2* v = ring + k % kMergeStages * C::kChunk + maker;
#pragma unroll
        for (int j = 0; j < kMergeBatch; ++j)
          if (live && c + j * kSlices < count) v[j * kMakers].x = exp2f(v[j * kMakers].x - m);
      }
    } else if (k > 0 && lane < R) {
      const float2* b = ring + (k - 1) % kMergeStages * C::kChunk + lane;
      const int n = min(kParts, count - (k - 1) * kParts);
      // 10 parts at a time, the next 10 loaded under their additions
      float2 x[10], y[10];
      auto take = [&](float2(&to)[10], int c) {
        if (c + 10 <= n) {
#pragma unroll
          for (int j = 0; j < 10; ++j) to[j] = b[(c + j) * R];
        }
      };
      auto add = [&](const float2(&of)[10]) {
#pragma unroll
        for (int j = 0; j < 10; ++j) S = fmaf(of[j].y, of[j].x, S);
      };
      int c = 0;
      take(x, 0);
      for (; c + 10 <= n; c += 10) {
        take(y, c + 10);
        add(x);
        c += 10;
        if (c + 10 > n) break;
        take(x, c + 10);
        add(y);
      }
      for (; c < n; ++c) S = fmaf(b[c * R].y, b[c * R].x, S);
    }
    __syncthreads();
  }
  return make_float2(m, S);
}

template <class C, class Kernel, class... Args>
static int launch_merge_cfg(Kernel kern, int64_t N, int count, cudaStream_t s, Args... args) {
  const int chunks = (count + C::kParts - 1) / C::kParts;
  const size_t smem = sizeof(float2) * C::kChunk * (chunks < kMergeStages ? chunks : kMergeStages);
  // more than the 48 KB that a launch may have without asking (the kernel's own arrays included)
  if (smem > 45 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               static_cast<int>(smem)) != cudaSuccess)
    return PS_ERR_CUDA;
  return launch_after(kern, dim3(static_cast<unsigned>((N + C::kRows - 1) / C::kRows)), C::kThreads, smem, s, 1, 1, true,
                      N, args...) == cudaSuccess
             ? PS_OK
             : PS_ERR_CUDA;
}
// Launches the kernel that `pick` gives for a MergeCfg. Few rows are spread over the SMs, 8 to a block; then a warp
// finalises more of them (its double arithmetic costs the same for 32 rows as for 8). Small blocks leave an SM 8 rings
// and 8 adding warps, which pays once there are enough of them: 60000 rows at V = 152064 take 195 us with 128 threads
// and 203 with 512, at V = 32000 51 and 81, at V = 2000 23 and 46. A row of one chunk wants no more threads either
// (600 rows, V = 2000: 7.7 and 8.3 us; 250 parts: 10.1 and 9.7).
template <class Pick, class... Args>
static int launch_merge(Pick pick, int64_t N, int count, cudaStream_t s, Args... args) {
  const int64_t sms = num_sms_current();
  auto go = [&](auto cfg) { return launch_merge_cfg<decltype(cfg)>(pick(cfg), N, count, s, args...); };
  const bool one_chunk = count <= MergeCfg<8, 128>::kParts;
  if (N <= 8 * 2 * sms) return one_chunk ? go(MergeCfg<8, 128>()) : go(MergeCfg<8, 512>());
  if (N <= 16 * 2 * sms && !one_chunk) return go(MergeCfg<16, 512>());
  if (N <= 32 * 2 * sms && !one_chunk) return go(MergeCfg<32, 512>());
  return go(MergeCfg<32, 128>());
}

// Sum of v over the block in a fixed order (warp shuffles, then warp 0 over the warps' sums), in thread 0.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double ws_sum[32];
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws_sum[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < (blockDim.x >> 5) ? ws_sum[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

// The block's sum of row losses goes where its rows' first parts were (nobody else reads them), and
// the last block to finish (`ticket`, zeroed at the call's start, counts them) adds the sums up: one
// launch less than a separate reduction, and the same order of addition whichever block is last.
template <class C>
__global__ void __launch_bounds__(C::kThreads, 1024 / C::kThreads)
    fwd_finalize_kernel(int64_t N, int V, int splits, float2* __restrict__ part, const float* __restrict__ ztok,
                        const int32_t* __restrict__ tok, const float* __restrict__ oldlogp,
                        const float* __restrict__ adv, const float* __restrict__ w, double eps, double loss_scale,
                        double* __restrict__ loss, float* __restrict__ lse, float* __restrict__ logp,
                        float* __restrict__ ratio, float* __restrict__ coef, float* __restrict__ row_loss,
                        uint32_t* ticket, uint32_t* status) {
  __shared__ bool last;
  wait_for_previous_kernel();
  constexpr int R = C::kRows;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * R, i = i0 + threadIdx.x;
  const int rows = static_cast<int>(N - i0 < R ? N - i0 : R);
  const float2 ms = merge_parts_block<C>(part + i0, splits, N, rows);
  if (threadIdx.x < 32) {
    double rl = 0.0;
    if (threadIdx.x < rows)
      rl = finalize_row(i, ms.x, ms.y, ztok[i], tok[i], V, oldlogp, adv, w, eps, loss_scale, lse, logp, ratio, coef,
                        row_loss, status);
#pragma unroll
    for (int o = R / 2; o >= 1; o >>= 1) rl += __shfl_down_sync(0xffffffffu, rl, o);
    if (threadIdx.x == 0) {
      *reinterpret_cast<double*>(part + i0) = rl;
      __threadfence();
      last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v = 0.0;
  for (int64_t b = threadIdx.x; b < gridDim.x; b += blockDim.x)
    v += __ldcg(reinterpret_cast<const double*>(part + b * R));
  v = block_sum(v);
  if (threadIdx.x == 0) *loss = v;
}

// A vocabulary shard's statistics: its vocabulary tiles' (max, sum) pairs merged per row, and the
// chosen logit where the row's token lies in the shard ([tok_base, tok_base + Vs)), -inf elsewhere.
template <class C>
__global__ void __launch_bounds__(C::kThreads, 1024 / C::kThreads)
    stats_merge_kernel(int64_t N, int splits, const float2* __restrict__ part, const float* __restrict__ ztok_ws,
                       const int32_t* __restrict__ tok, int64_t tok_base, int Vs, float2* __restrict__ stats,
                       float* __restrict__ ztok) {
  wait_for_previous_kernel();
  constexpr int R = C::kRows;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * R, i = i0 + threadIdx.x;
  const int rows = static_cast<int>(N - i0 < R ? N - i0 : R);
  const float2 ms = merge_parts_block<C>(part + i0, splits, N, rows);
  if (threadIdx.x >= rows) return;
  stats[i] = ms;
  const int64_t t = static_cast<int64_t>(tok[i]) - tok_base;
  ztok[i] = (t >= 0 && t < Vs) ? ztok_ws[i] : -INFINITY;
}

// The forward finalize from the statistics of S vocabulary shards ([S][ld] each): their (max, sum)
// pairs merged as one row's tiles are, and the chosen logit from the shard that holds the token (the
// largest of the S values, the others being -inf).
__global__ void __launch_bounds__(kFinThreads)
    stats_finalize_kernel(int64_t N, int S, int64_t ld, int V, const float2* __restrict__ stats,
                          const float* __restrict__ ztok,
                          const int32_t* __restrict__ tok, const float* __restrict__ oldlogp,
                          const float* __restrict__ adv, const float* __restrict__ w, double eps, double loss_scale,
                          float* __restrict__ lse, float* __restrict__ logp, float* __restrict__ ratio,
                          float* __restrict__ coef, float* __restrict__ row_loss, double* __restrict__ block_loss,
                          uint32_t* status) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * kFinThreads + threadIdx.x;
  double rl = 0.0;
  if (i < N) {
    const float2 ms = merge_parts(stats + i, S, ld);
    float zt = -INFINITY;
    for (int r = 0; r < S; ++r) zt = fmaxf(zt, ztok[static_cast<int64_t>(r) * ld + i]);
    rl = finalize_row(i, ms.x, ms.y, zt, tok[i], V, oldlogp, adv, w, eps, loss_scale, lse, logp, ratio, coef,
                      row_loss, status);
  }
  rl = block_sum(rl);
  if (threadIdx.x == 0) block_loss[blockIdx.x] = rl;
}

__global__ void __launch_bounds__(1024) loss_reduce_kernel(int64_t nblocks, const double* __restrict__ part,
                                                           double* __restrict__ loss) {
  wait_for_previous_kernel();
  double v = 0.0;
  for (int64_t b = threadIdx.x; b < nblocks; b += 1024) v += part[b];
  v = block_sum(v);
  if (threadIdx.x == 0) *loss = v;
}

// Forward workspace: header | ztok [N] f32 | 8 ceil(N / 256) bytes, unused (they keep the layout, and so
// what a given workspace holds) | part [S][N] float2. The
// (max, sum of exp) partials come last: S is as many as the workspace holds, up to two per
// 256-column vocabulary tile (bf16: one per column group of the forward's epilogue, so the
// vocabulary ranges per row are S / 2; at one range per tile every unit of the forward GEMM is one
// tile, the schedule that keeps W traffic lowest). f32 always uses one partial per 64-column tile.
struct FwdWs {
  float2* part;
  float* ztok;
  int splits;       // S that fits (0 if not even one)
  size_t bytes;     // bytes used with that S
};
static int fwd_full_splits(int V, int dtype) {
  return dtype == PS_DTYPE_BF16 ? fwd_tile_splits_bf16(V) * fwd_partials_per_split_bf16() : fwd_splits_f32(V);
}
// Partials per vocabulary range, and the fewest partials a forward can run with.
static int fwd_group(int dtype) { return dtype == PS_DTYPE_BF16 ? fwd_partials_per_split_bf16() : 1; }
static size_t fwd_fixed_bytes(int64_t N) {
  const int64_t nb = (N + kFinThreads - 1) / kFinThreads;
  return kWsHeader + align_up(sizeof(float) * N, 256) + align_up(sizeof(double) * (nb > 0 ? nb : 1), 256);
}
// the partials are the last region: no padding after them, so S partials need exactly this much
static size_t fwd_part_bytes(int64_t N, int S) { return sizeof(float2) * static_cast<size_t>(S) * N; }
// Layout for a workspace of ws_bytes (SIZE_MAX: the full-size layout).
static FwdWs fwd_ws(void* ws, int64_t N, int V, int dtype, size_t ws_bytes) {
  const int full = fwd_full_splits(V, dtype);
  const size_t fixed = fwd_fixed_bytes(N);
  FwdWs f;
  uint8_t* base = static_cast<uint8_t*>(ws);
  f.ztok = reinterpret_cast<float*>(base + kWsHeader);
  f.part = reinterpret_cast<float2*>(base + fixed);
  const int g = fwd_group(dtype);
  int S = full;
  if (ws_bytes != SIZE_MAX && N > 0) {
    const size_t room = ws_bytes > fixed ? ws_bytes - fixed : 0;
    const size_t fit = room / (sizeof(float2) * static_cast<size_t>(N));
    if (fit < static_cast<size_t>(S)) S = static_cast<int>(fit) / g * g;   // whole vocabulary ranges
    if (dtype != PS_DTYPE_BF16 && S < full) S = 0;   // the f32 kernel needs every partial
  }
  f.splits = S;
  f.bytes = fixed + fwd_part_bytes(N, S > 0 ? S : g);
  return f;
}

static size_t elem_size(int dtype) { return dtype == PS_DTYPE_BF16 ? 2 : 4; }
static bool dtype_ok(int dtype) { return dtype == PS_DTYPE_BF16 || dtype == PS_DTYPE_F32; }
static bool d_ok(int d, int dtype) { return d >= 8 && (dtype == PS_DTYPE_BF16 ? d % 8 == 0 : d % 4 == 0); }
static bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
static int64_t ldz_for(int V) { return (static_cast<int64_t>(V) + 7) / 8 * 8; }

}  // namespace psk

using namespace psk;

// ============================================================================= C ABI
extern "C" {

const char* ps_status_string(int status) {
  switch (status) {
    case PS_OK: return "ok";
    case PS_ERR_INVALID_ARG: return "invalid argument";
    case PS_ERR_UNSUPPORTED: return "unsupported dtype, shape or device";
    case PS_ERR_WORKSPACE: return "workspace too small or misaligned";
    case PS_ERR_CAPACITY: return "packed rows exceed capacity";
    case PS_ERR_DEVICE_DATA: return "invalid device data (masses, lengths or token ids)";
    case PS_ERR_TIMEOUT: return "a bounded wait inside a kernel ran out";
    case PS_ERR_CUDA: return "CUDA runtime error";
    default: return "unknown status";
  }
}

int ps_version(void) { return 100; }

int ps_workspace_status(const void* ws, ps_stream_t stream, uint32_t* bits) {
  if (ws == nullptr) return PS_ERR_INVALID_ARG;
  uint32_t v = 0;
  if (cudaMemcpyAsync(&v, ws, sizeof(v), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return PS_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return PS_ERR_CUDA;
  if (bits) *bits = v;
  if (v & PS_DEV_TIMEOUT) return PS_ERR_TIMEOUT;
  if (v & PS_DEV_CAPACITY) return PS_ERR_CAPACITY;
  if (v) return PS_ERR_DEVICE_DATA;
  return PS_OK;
}

size_t ps_sample_cutoffs_workspace_size(int, int, int) { return kWsHeader; }

int ps_sample_cutoffs(int P, int K, int T_max, const uint64_t* q, const int32_t* L, uint64_t seed, uint64_t step,
                      int64_t traj_base, int mode, int32_t* H, int32_t* n, float* w_tab, void* ws, size_t ws_bytes,
                      ps_stream_t stream) {
  NvtxRange nvtx_range("ps_sample_cutoffs");
  if (P < 1 || K < 1 || K > 8192 || T_max < 1 || T_max > (1 << 24) || traj_base < 0) return PS_ERR_INVALID_ARG;
  if (static_cast<int64_t>(P) * K > INT32_MAX) return PS_ERR_INVALID_ARG;
  if (mode != PS_MODE_TRUNC && mode != PS_MODE_FULL && mode != PS_MODE_TRUNC_ZERO) return PS_ERR_INVALID_ARG;
  if ((mode != PS_MODE_FULL && q == nullptr) || !L || !H || !n || !w_tab) return PS_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = begin_call(ws, ws_bytes, ps_sample_cutoffs_workspace_size(P, K, T_max), s);
  if (rc != PS_OK) return rc;
  const size_t smem = sizeof(uint64_t) * K;
  if (smem > 47 * 1024 && cudaFuncSetAttribute(sample_cutoffs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               static_cast<int>(smem)) != cudaSuccess)
    return PS_ERR_CUDA;
  // parts of a prompt: one per tile of steps while that leaves no more than two CTAs per SM
  int64_t parts = (T_max + kSampThreads - 1) / kSampThreads;
  const int64_t most = 2 * static_cast<int64_t>(num_sms_current()) / P;
  if (parts > most) parts = most > 0 ? most : 1;
  if (parts > kSampMaxParts) parts = kSampMaxParts;
  const dim3 grid(static_cast<unsigned>(P), static_cast<unsigned>(parts));
  sample_cutoffs_kernel<<<grid, kSampThreads, smem, s>>>(K, T_max, q, L, seed, step, traj_base, mode, H, n, w_tab,
                                                      status_word(ws));
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

size_t ps_pack_prefixes_workspace_size(int P, int K) {
  const int B = P * K;
  return kWsHeader + align_up(sizeof(int64_t) * (B + 1), 256) + align_up(sizeof(double) * B, 256) + 256;
}

int ps_pack_prefixes(int P, int K, int T_max, int d, int dtype, const int32_t* L, const int32_t* n, const float* R,
                     int adv_mode, const float* w_tab, const int32_t* tok_full, const float* oldlogp_full,
                     const void* hid_full, int64_t capacity, int32_t* cu_seqlens, int32_t* src_row,
                     int32_t* row_traj, int32_t* row_pos, int32_t* tok, float* oldlogp, float* w, float* adv,
                     void* hid_packed, int64_t* h_num_rows, void* ws, size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_pack_prefixes");
  if (P < 1 || K < 1 || T_max < 1 || capacity < 0 || !dtype_ok(dtype)) return PS_ERR_INVALID_ARG;
  if (static_cast<int64_t>(P) * K > (1 << 24)) return PS_ERR_INVALID_ARG;
  if (adv_mode != PS_ADV_CENTERED && adv_mode != PS_ADV_GROUP_NORM) return PS_ERR_INVALID_ARG;
  if (!L || !n || !R || !w_tab || !tok_full || !oldlogp_full || !cu_seqlens || !tok || !oldlogp || !w || !adv)
    return PS_ERR_INVALID_ARG;
  if (hid_full != nullptr) {
    if (!hid_packed || !d_ok(d, dtype) || !al16(hid_full) || !al16(hid_packed)) return PS_ERR_INVALID_ARG;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int rc = check_ws(ws, ws_bytes, ps_pack_prefixes_workspace_size(P, K));
  if (rc != PS_OK) return rc;
  const int B = P * K;
  PackWs pw = pack_ws(ws, B);
  const int sms = num_sms_current();
  const int adv_ctas = P < kAdvWarps * sms ? (P + kAdvWarps - 1) / kAdvWarps : sms;
  pack_meta_kernel<<<1 + adv_ctas, kMetaThreads, 0, s>>>(P, K, T_max, L, n, R, adv_mode, capacity, cu_seqlens, pw,
                                                         status_word(ws));
  if (cudaGetLastError() != cudaSuccess) return refused(PS_ERR_CUDA, ws, s);
  const int64_t row_vec = hid_full ? static_cast<int64_t>(d) * elem_size(dtype) / 16 : 0;
  const int grid = sms * 8;
  if (launch_after(pack_rows_kernel, dim3(static_cast<unsigned>(grid)), kPackThreads, 0, s, 1, 1, true, B, K, T_max,
                   cu_seqlens, pw, w_tab, tok_full, oldlogp_full, static_cast<const uint4*>(hid_full), row_vec, src_row,
                   row_traj, row_pos, tok, oldlogp, w, adv, static_cast<uint4*>(hid_packed)) != cudaSuccess)
    return PS_ERR_CUDA;
  if (h_num_rows) {
    // straight into the caller's word (its low half: both hosts are little-endian), so that a page-locked one
    // is copied to without the driver's staging
    *h_num_rows = 0;
    if (cudaMemcpyAsync(h_num_rows, cu_seqlens + B, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
      return PS_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return PS_ERR_CUDA;
  }
  return PS_OK;
}

size_t ps_lmhead_ppo_fwd_workspace_size(int64_t N, int d, int V, int dtype) {
  if (N < 0 || V < 1 || !dtype_ok(dtype)) return 0;
  (void)d;
  return fwd_ws(nullptr, N, V, dtype, SIZE_MAX).bytes;
}

}  // extern "C"

// Layout of the logit store of N rows: [N][ldz] 2-byte values (f16 e after the forward, bf16 dZ after
// the backward's conversion), then the slice maxima [ceil(V / 32)][N] f32 at a 256-byte boundary.
struct StoreLayout {
  int64_t ldz;
  size_t scale_off;
  size_t bytes;
};
static StoreLayout store_layout(int64_t N, int V) {
  StoreLayout L;
  L.ldz = ldz_for(V);
  L.scale_off = align_up(static_cast<size_t>(N) * static_cast<size_t>(L.ldz) * 2, 256);
  L.bytes = L.scale_off + sizeof(float) * static_cast<size_t>((V + 31) / 32) * static_cast<size_t>(N);
  return L;
}

static int lmhead_fwd_impl(int64_t N, int d, int V, int dtype, const void* Hpk, const void* W, const int32_t* tok,
                           const float* oldlogp, const float* adv, const float* w, double eps, double loss_scale,
                           double* loss, float* lse, float* logp, float* ratio, float* coef, float* row_loss,
                           void* store, size_t store_bytes, void* ws, size_t ws_bytes, ps_stream_t stream) {
  if (N < 0 || N > INT32_MAX || V < 1 || !dtype_ok(dtype) || !d_ok(d, dtype)) return PS_ERR_INVALID_ARG;
  if (!(eps >= 0.0) || !loss || (N > 0 && (!Hpk || !W || !tok || !oldlogp || !adv || !w || !lse || !logp ||
                                           !ratio || !coef)))
    return PS_ERR_INVALID_ARG;
  if (N > 0 && (!al16(Hpk) || !al16(W))) return PS_ERR_INVALID_ARG;
  if (store != nullptr) {
    if (dtype != PS_DTYPE_BF16) return PS_ERR_UNSUPPORTED;
    if (!al16(store)) return PS_ERR_INVALID_ARG;
    if (store_bytes < store_layout(N, V).bytes) return PS_ERR_WORKSPACE;
  }
  if (dtype == PS_DTYPE_BF16 && !device_is_sm103()) return PS_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  FwdWs f = fwd_ws(ws, N, V, dtype, ws_bytes);
  if (N > 0 && f.splits < 1) return PS_ERR_WORKSPACE;
  int rc = N == 0 ? begin_call(ws, ws_bytes, f.bytes, s) : check_ws(ws, ws_bytes, f.bytes);
  if (rc != PS_OK) return rc;
  if (N == 0) return cudaMemsetAsync(loss, 0, sizeof(double), s) == cudaSuccess ? PS_OK : PS_ERR_CUDA;
  int splits;
  if (dtype == PS_DTYPE_BF16) {
    const int g = fwd_partials_per_split_bf16();
    const int ranges = choose_fwd_splits_bf16(N, d, V, num_sms_current(), f.splits / g);
    if (store) {
      const StoreLayout L = store_layout(N, V);
      float* scale = reinterpret_cast<float*>(static_cast<uint8_t*>(store) + L.scale_off);
      rc = fwd_gemm_store_bf16(N, d, V, Hpk, W, tok, f.part, f.ztok, ranges, store, L.ldz, scale, status_word(ws),
                               s);
    } else {
      rc = fwd_gemm_bf16(N, d, V, Hpk, W, tok, f.part, f.ztok, ranges, status_word(ws), s);
    }
    splits = ranges * g;   // the partials the finalize merges
  } else {
    splits = fwd_splits_f32(V);
    rc = fwd_gemm_f32(N, d, V, static_cast<const float*>(Hpk), static_cast<const float*>(W), tok, f.part, f.ztok,
                      status_word(ws), s);
  }
  if (rc != PS_OK) return refused(rc, ws, s);
  return launch_merge([](auto cfg) { return fwd_finalize_kernel<decltype(cfg)>; }, N, splits, s, V, splits, f.part,
                      f.ztok, tok, oldlogp, adv, w, eps, loss_scale, loss, lse, logp, ratio, coef, row_loss, ticket_word(ws),
                      status_word(ws));
}

// The backward from a logit store of V vocabulary columns whose first is global token id tok_base.
// v_call: the whole head's vocabulary.
static int bwd_from_store_impl(int64_t N, int d, int V, int64_t tok_base, int64_t v_call, int dtype, const void* Hpk, const void* W,
                               const int32_t* tok, const float* lse, const float* logp, const float* coef,
                               void* store, size_t store_bytes, float* dH, float* dW, int flags, void* ws,
                               size_t ws_bytes, ps_stream_t stream) {
  if (N < 0 || N > INT32_MAX || V < 1 || !dtype_ok(dtype) || !d_ok(d, dtype)) return PS_ERR_INVALID_ARG;
  if (flags & ~(PS_DW_ACCUMULATE | PS_DH_ACCUMULATE)) return PS_ERR_INVALID_ARG;
  if (dtype != PS_DTYPE_BF16) return PS_ERR_UNSUPPORTED;
  if (N > 0 && (!Hpk || !W || !tok || !lse || !logp || !coef || !store)) return PS_ERR_INVALID_ARG;
  if ((N > 0 && (!al16(Hpk) || !al16(W) || !al16(store))) || (dH && !al16(dH)) || (dW && !al16(dW)))
    return PS_ERR_INVALID_ARG;
  if (N > 0 && store_bytes < store_layout(N, V).bytes) return PS_ERR_WORKSPACE;
  if (!device_is_sm103()) return PS_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = N == 0 ? begin_call(ws, ws_bytes, kWsHeader, s) : check_ws(ws, ws_bytes, kWsHeader);
  if (rc != PS_OK) return rc;
  if (N == 0) {
    if (dW && !(flags & PS_DW_ACCUMULATE))
      return cudaMemsetAsync(dW, 0, sizeof(float) * static_cast<size_t>(V) * d, s) == cudaSuccess ? PS_OK
                                                                                                : PS_ERR_CUDA;
    return PS_OK;
  }
  // the conversion into dZ (HBM-bound), then dH and dW over all rows. Running the conversion of later
  // rows on a second stream under the dH GEMM of earlier rows (the GEMM's one CTA per SM leaves room
  // for conversion blocks) measured 1-2% slower at the 7B workload (backward 272.7 / 273.0 against
  // 267.3 / 269.2 ms, back to back), so the parts run in turn.
  const StoreLayout L = store_layout(N, V);
  const float* scale = reinterpret_cast<const float*>(static_cast<const uint8_t*>(store) + L.scale_off);
  rc = dz_from_store_bf16(N, V, store, L.ldz, scale, N, tok, lse, logp, coef, status_word(ws), s,
                          static_cast<int>(tok_base));
  if (rc != PS_OK) return refused(rc, ws, s);
  return bwd_grads_bf16(N, d, V, Hpk, W, dH, dW, (flags & PS_DW_ACCUMULATE) ? 1 : 0, store, L.ldz, status_word(ws),
                        s, (flags & PS_DH_ACCUMULATE) ? 1 : 0, N, v_call);
}

extern "C" {

int ps_lmhead_ppo_fwd(int64_t N, int d, int V, int dtype, const void* Hpk, const void* W, const int32_t* tok,
                      const float* oldlogp, const float* adv, const float* w, double eps, double loss_scale,
                      double* loss, float* lse, float* logp, float* ratio, float* coef, float* row_loss, void* ws,
                      size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_fwd");
  return lmhead_fwd_impl(N, d, V, dtype, Hpk, W, tok, oldlogp, adv, w, eps, loss_scale, loss, lse, logp, ratio, coef,
                         row_loss, nullptr, 0, ws, ws_bytes, stream);
}

size_t ps_lmhead_logit_store_size(int64_t N, int V) {
  if (N < 0 || N > INT32_MAX || V < 1) return 0;
  return store_layout(N, V).bytes;
}

int ps_lmhead_ppo_fwd_store(int64_t N, int d, int V, int dtype, const void* Hpk, const void* W, const int32_t* tok,
                            const float* oldlogp, const float* adv, const float* w, double eps, double loss_scale,
                            double* loss, float* lse, float* logp, float* ratio, float* coef, float* row_loss,
                            void* store, size_t store_bytes, void* ws, size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_fwd_store");
  if (store == nullptr) return PS_ERR_INVALID_ARG;
  return lmhead_fwd_impl(N, d, V, dtype, Hpk, W, tok, oldlogp, adv, w, eps, loss_scale, loss, lse, logp, ratio, coef,
                         row_loss, store, store_bytes, ws, ws_bytes, stream);
}

size_t ps_lmhead_ppo_bwd_from_store_workspace_size(void) { return kWsHeader; }

int ps_lmhead_ppo_bwd_from_store(int64_t N, int d, int V, int dtype, const void* Hpk, const void* W,
                                 const int32_t* tok, const float* lse, const float* logp, const float* coef,
                                 void* store, size_t store_bytes, float* dH, float* dW, int flags, void* ws,
                                 size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_bwd_from_store");
  return bwd_from_store_impl(N, d, V, 0, V, dtype, Hpk, W, tok, lse, logp, coef, store, store_bytes, dH, dW, flags, ws,
                             ws_bytes, stream);
}

int ps_lmhead_ppo_bwd_vocab_shard_from_store(int64_t N, int d, int Vs, int64_t v0, int V, int dtype, const void* Hpk,
                                             const void* W_shard, const int32_t* tok, const float* lse,
                                             const float* logp, const float* coef, void* store, size_t store_bytes,
                                             float* dH, float* dW_shard, int flags, void* ws, size_t ws_bytes,
                                             ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_bwd_vocab_shard_from_store");
  if (Vs < 1 || v0 < 0 || V < 1 || v0 + Vs > V) return PS_ERR_INVALID_ARG;
  return bwd_from_store_impl(N, d, Vs, v0, V, dtype, Hpk, W_shard, tok, lse, logp, coef, store, store_bytes, dH,
                             dW_shard, flags, ws, ws_bytes, stream);
}

size_t ps_lmhead_logit_stats_workspace_size(int64_t N, int d, int Vs, int dtype) {
  return ps_lmhead_ppo_fwd_workspace_size(N, d, Vs, dtype);
}

}  // extern "C"

static int logit_stats_impl(int64_t N, int d, int Vs, int64_t v0, int dtype, const void* Hpk, const void* W_shard,
                            const int32_t* tok, float* stats, float* ztok, void* store, size_t store_bytes, void* ws,
                            size_t ws_bytes, ps_stream_t stream) {
  if (N < 0 || N > INT32_MAX || Vs < 1 || v0 < 0 || v0 + Vs > INT32_MAX || !dtype_ok(dtype) || !d_ok(d, dtype))
    return PS_ERR_INVALID_ARG;
  if (N > 0 && (!Hpk || !W_shard || !tok || !stats || !ztok)) return PS_ERR_INVALID_ARG;
  if (N > 0 && (!al16(Hpk) || !al16(W_shard) || (reinterpret_cast<uintptr_t>(stats) & 7))) return PS_ERR_INVALID_ARG;
  if (store != nullptr) {
    if (dtype != PS_DTYPE_BF16) return PS_ERR_UNSUPPORTED;
    if (!al16(store)) return PS_ERR_INVALID_ARG;
    if (store_bytes < store_layout(N, Vs).bytes) return PS_ERR_WORKSPACE;
  }
  if (dtype == PS_DTYPE_BF16 && !device_is_sm103()) return PS_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  FwdWs f = fwd_ws(ws, N, Vs, dtype, ws_bytes);
  if (N > 0 && f.splits < 1) return PS_ERR_WORKSPACE;
  int rc = N == 0 ? begin_call(ws, ws_bytes, f.bytes, s) : check_ws(ws, ws_bytes, f.bytes);
  if (rc != PS_OK || N == 0) return rc;
  int splits;
  if (dtype == PS_DTYPE_BF16) {
    const int g = fwd_partials_per_split_bf16();
    const int ranges = choose_fwd_splits_bf16(N, d, Vs, num_sms_current(), f.splits / g);
    if (store) {
      const StoreLayout L = store_layout(N, Vs);
      float* scale = reinterpret_cast<float*>(static_cast<uint8_t*>(store) + L.scale_off);
      rc = fwd_gemm_store_bf16(N, d, Vs, Hpk, W_shard, tok, f.part, f.ztok, ranges, store, L.ldz, scale,
                               status_word(ws), s, static_cast<int>(v0));
    } else {
      rc = fwd_gemm_bf16(N, d, Vs, Hpk, W_shard, tok, f.part, f.ztok, ranges, status_word(ws), s,
                         static_cast<int>(v0));
    }
    splits = ranges * g;   // the partials the merge reads
  } else {
    splits = fwd_splits_f32(Vs);
    rc = fwd_gemm_f32(N, d, Vs, static_cast<const float*>(Hpk), static_cast<const float*>(W_shard), tok, f.part,
                      f.ztok, status_word(ws), s, static_cast<int>(v0));
  }
  if (rc != PS_OK) return refused(rc, ws, s);
  return launch_merge([](auto cfg) { return stats_merge_kernel<decltype(cfg)>; }, N, splits, s, splits, f.part, f.ztok,
                      tok, v0, Vs, reinterpret_cast<float2*>(stats), ztok);
}

extern "C" {

int ps_lmhead_logit_stats(int64_t N, int d, int Vs, int64_t v0, int dtype, const void* Hpk, const void* W_shard,
                          const int32_t* tok, float* stats, float* ztok, void* ws, size_t ws_bytes,
                          ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_logit_stats");
  return logit_stats_impl(N, d, Vs, v0, dtype, Hpk, W_shard, tok, stats, ztok, nullptr, 0, ws, ws_bytes, stream);
}

int ps_lmhead_logit_stats_store(int64_t N, int d, int Vs, int64_t v0, int dtype, const void* Hpk,
                                const void* W_shard, const int32_t* tok, float* stats, float* ztok, void* store,
                                size_t store_bytes, void* ws, size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_logit_stats_store");
  if (store == nullptr) return PS_ERR_INVALID_ARG;
  return logit_stats_impl(N, d, Vs, v0, dtype, Hpk, W_shard, tok, stats, ztok, store, store_bytes, ws, ws_bytes,
                          stream);
}

size_t ps_lmhead_ppo_fwd_from_stats_workspace_size(int64_t N) {
  if (N < 0) return 0;
  const int64_t nb = (N + kFinThreads - 1) / kFinThreads;
  return kWsHeader + align_up(sizeof(double) * static_cast<size_t>(nb > 0 ? nb : 1), 256);
}

int ps_lmhead_ppo_fwd_from_stats(int64_t N, int S, int64_t ld, int V, const float* stats, const float* ztok,
                                 const int32_t* tok,
                                 const float* oldlogp, const float* adv, const float* w, double eps,
                                 double loss_scale, double* loss, float* lse, float* logp, float* ratio, float* coef,
                                 float* row_loss, void* ws, size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_fwd_from_stats");
  if (N < 0 || N > INT32_MAX || S < 1 || ld < N || V < 1 || !(eps >= 0.0) || !loss) return PS_ERR_INVALID_ARG;
  if (N > 0 && (!stats || !ztok || !tok || !oldlogp || !adv || !w || !lse || !logp || !ratio || !coef))
    return PS_ERR_INVALID_ARG;
  if (N > 0 && (reinterpret_cast<uintptr_t>(stats) & 7)) return PS_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = begin_call(ws, ws_bytes, ps_lmhead_ppo_fwd_from_stats_workspace_size(N), s);
  if (rc != PS_OK) return rc;
  if (N == 0) return cudaMemsetAsync(loss, 0, sizeof(double), s) == cudaSuccess ? PS_OK : PS_ERR_CUDA;
  const int64_t nb = (N + kFinThreads - 1) / kFinThreads;
  double* block_loss = reinterpret_cast<double*>(static_cast<uint8_t*>(ws) + kWsHeader);
  stats_finalize_kernel<<<static_cast<unsigned>(nb), kFinThreads, 0, s>>>(
      N, S, ld, V, reinterpret_cast<const float2*>(stats), ztok, tok, oldlogp, adv, w, eps, loss_scale, lse, logp, ratio,
      coef, row_loss, block_loss, status_word(ws));
  if (cudaGetLastError() != cudaSuccess) return PS_ERR_CUDA;
  return launch_after(loss_reduce_kernel, dim3(1), 1024, 0, s, 1, 1, true, nb, block_loss, loss) == cudaSuccess
             ? PS_OK
             : PS_ERR_CUDA;
}

size_t ps_lmhead_ppo_bwd_workspace_size(int64_t N, int d, int V, int dtype, int64_t chunk_rows) {
  if (N < 0 || V < 1 || !dtype_ok(dtype)) return 0;
  (void)d;
  int64_t rows = chunk_rows <= 0 ? N : chunk_rows;
  if (rows > N) rows = N;
  rows = (rows + 127) / 128 * 128;
  if (rows < 128) rows = 128;
  return kWsHeader + static_cast<size_t>(rows) * ldz_for(V) * elem_size(dtype);
}

}  // extern "C"

// The backward over a head of V vocabulary rows whose first is global token id tok_base (0 for the
// whole head, v0 for one shard of a vocabulary-parallel head of v_call rows in all).
static int lmhead_bwd_impl(int64_t N, int d, int V, int64_t tok_base, int64_t v_call, int dtype, const void* Hpk, const void* W,
                           const int32_t* tok, const float* lse, const float* coef, float* dH, float* dW, int flags,
                           void* ws, size_t ws_bytes, ps_stream_t stream) {
  if (N < 0 || N > INT32_MAX || V < 1 || !dtype_ok(dtype) || !d_ok(d, dtype)) return PS_ERR_INVALID_ARG;
  if (flags & ~(PS_DW_ACCUMULATE | PS_DH_ACCUMULATE)) return PS_ERR_INVALID_ARG;
  if (N > 0 && (!Hpk || !W || !tok || !lse || !coef)) return PS_ERR_INVALID_ARG;
  if ((N > 0 && (!al16(Hpk) || !al16(W))) || (dH && !al16(dH)) || (dW && !al16(dW))) return PS_ERR_INVALID_ARG;
  if (dtype == PS_DTYPE_BF16 && !device_is_sm103()) return PS_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const size_t need = ps_lmhead_ppo_bwd_workspace_size(N, d, V, dtype, 128);
  int rc = N == 0 ? begin_call(ws, ws_bytes, need, s) : check_ws(ws, ws_bytes, need);
  if (rc != PS_OK) return rc;
  if (N == 0) {
    if (dW && !(flags & PS_DW_ACCUMULATE))
      return cudaMemsetAsync(dW, 0, sizeof(float) * static_cast<size_t>(V) * d, s) == cudaSuccess ? PS_OK
                                                                                                : PS_ERR_CUDA;
    return PS_OK;
  }
  const int64_t ldz = ldz_for(V);
  const size_t es = elem_size(dtype);
  int64_t chunk = static_cast<int64_t>((ws_bytes - kWsHeader) / (static_cast<size_t>(ldz) * es)) / 128 * 128;
  if (chunk < 1) return PS_ERR_WORKSPACE;
  // As few chunks as the workspace allows, of equal size (a multiple of 128 rows): a short last
  // chunk would cost a whole pass over dW for little work.
  const int64_t nchunks = (N + chunk - 1) / chunk;
  chunk = ((N + nchunks - 1) / nchunks + 127) / 128 * 128;
  if (chunk >= N) chunk = N;
  void* dz = static_cast<uint8_t*>(ws) + kWsHeader;
  for (int64_t r0 = 0; r0 < N; r0 += chunk) {
    const int64_t rcn = (N - r0) < chunk ? (N - r0) : chunk;
    const int acc = (r0 > 0 || (flags & PS_DW_ACCUMULATE)) ? 1 : 0;
    const int hacc = (flags & PS_DH_ACCUMULATE) ? 1 : 0;
    if (dtype == PS_DTYPE_BF16) {
      const uint16_t* h = static_cast<const uint16_t*>(Hpk) + r0 * d;
      rc = bwd_chunk_bf16(rcn, d, V, h, W, tok + r0, lse + r0, coef + r0, dH ? dH + r0 * d : nullptr, dW, acc, dz,
                          ldz, status_word(ws), s, static_cast<int>(tok_base), hacc, N, v_call, r0 == 0);
    } else {
      const float* h = static_cast<const float*>(Hpk) + r0 * d;
      rc = bwd_chunk_f32(rcn, d, V, h, static_cast<const float*>(W), tok + r0, lse + r0, coef + r0,
                         dH ? dH + r0 * d : nullptr, dW, acc, static_cast<float*>(dz), ldz, status_word(ws), s,
                         static_cast<int>(tok_base), hacc, N, v_call, r0 == 0);
    }
    if (rc != PS_OK) return r0 == 0 ? refused(rc, ws, s) : rc;
  }
  return PS_OK;
}

extern "C" {

int ps_lmhead_ppo_bwd(int64_t N, int d, int V, int dtype, const void* Hpk, const void* W, const int32_t* tok,
                      const float* lse, const float* coef, float* dH, float* dW, int flags, void* ws,
                      size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_bwd");
  return lmhead_bwd_impl(N, d, V, 0, V, dtype, Hpk, W, tok, lse, coef, dH, dW, flags, ws, ws_bytes, stream);
}

int ps_lmhead_ppo_bwd_vocab_shard(int64_t N, int d, int Vs, int64_t v0, int V, int dtype, const void* Hpk,
                                  const void* W_shard, const int32_t* tok, const float* lse, const float* coef,
                                  float* dH, float* dW_shard, int flags, void* ws, size_t ws_bytes,
                                  ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_ppo_bwd_vocab_shard");
  if (Vs < 1 || v0 < 0 || V < 1 || v0 + Vs > V) return PS_ERR_INVALID_ARG;
  return lmhead_bwd_impl(N, d, Vs, v0, V, dtype, Hpk, W_shard, tok, lse, coef, dH, dW_shard, flags, ws, ws_bytes,
                         stream);
}

// ----------------------------------------------------------------------------- diagnostics
int ps_diag_gemm_bf16(int M, int N, int K, int a_mn_major, int b_mn_major, const void* A, int64_t lda,
                      const void* B, int64_t ldb, float* C, int64_t ldc, int accumulate, int variant, void* ws,
                      size_t ws_bytes, ps_stream_t stream) {
  if (M < 1 || N < 1 || K < 1 || !A || !B || !C || ldc < N || ldc % 4 || !al16(C)) return PS_ERR_INVALID_ARG;
  if (lda < (a_mn_major ? M : K) || ldb < (b_mn_major ? N : K) || lda % 8 || ldb % 8) return PS_ERR_INVALID_ARG;
  if (!device_is_sm103()) return PS_ERR_UNSUPPORTED;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = begin_call(ws, ws_bytes, kWsHeader, s);
  if (rc != PS_OK) return rc;
  return gemm_bf16(M, N, K, a_mn_major, b_mn_major, A, lda, B, ldb, C, ldc, accumulate, variant, status_word(ws), s);
}

int ps_diag_choose_splitk(int64_t M, int64_t N, int num_kb, int narrow_too, int sms, int pairs, int fours, int eights,
                          int* ranks, int* halves) {
  if (M < 1 || N < 1 || num_kb < 1 || sms < 1 || !ranks || !halves) return PS_ERR_INVALID_ARG;
  const int at_once[3] = {pairs, fours, eights};
  const SplitK k = choose_splitk(M, N, num_kb, narrow_too != 0, sms, at_once);
  *ranks = k.ranks;
  *halves = k.halves;
  return PS_OK;
}

int ps_diag_wait_timeout(uint64_t timeout_ns, void* ws, size_t ws_bytes, ps_stream_t stream) {
  if (timeout_ns > 10000000000ull) return PS_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int rc = begin_call(ws, ws_bytes, kWsHeader, s);
  if (rc != PS_OK) return rc;
  return wait_timeout_probe(timeout_ns, status_word(ws), s);
}

}  // extern "C"
