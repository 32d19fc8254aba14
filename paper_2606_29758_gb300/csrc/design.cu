// Cutoff-distribution design on the device (the step upstream of the sampler).
//
//  ps_lmhead_score_proxy: per token, the output-head score proxy of Appendix D,
//      gamma = ||h||^2 (1 - 2 p(o) + ||p||^2),
//  and log p(o), from one pass of the LM-head GEMM (the forward's schedule) whose epilogue keeps
//  two running exponential sums (||p||^2 from the two-logsumexp identity).
//  ps_design_cutoffs: per prompt, the group average of gamma at each step (Section 3.3), timestep
//  weights w = gamma_bar * u, the budgeted monotone xi of Appendix F (closed form + pooling of
//  adjacent violators + the xi <= 1 cap), or one of the Section 4 variants, and the integer
//  masses the sampler takes (the deficit is Pr(H = 0)).
//
// The design arithmetic is sequential float64 with explicitly rounded operations (no FMA
// contraction), so the masses are reproducible bit for bit.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <climits>
#include <cstdint>

#include "ps_nvtx.h"
#include "internal.h"
#include "ps_common.cuh"
#include "psppo.h"

namespace psk {

static size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// ================================================================== score proxy
__global__ void row_sqnorm_kernel(int64_t N, int d, int is_bf16, const void* __restrict__ H,
                                  float* __restrict__ out, uint32_t* status) {
  if (blockIdx.x == 0 && threadIdx.x == 0) clear_status(status);   // the call's first kernel
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); i < N; i += warps) {
    float acc = 0.f;
    if (is_bf16) {
      const uint4* r = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(H) + i * d);
      for (int c = lane; c < d / 8; c += 32) {
        const uint4 v = r[c];
        const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float a = __uint_as_float(w4[k] << 16), b = __uint_as_float(w4[k] & 0xFFFF0000u);
          acc = fmaf(a, a, fmaf(b, b, acc));
        }
      }
    } else {
      const float* r = static_cast<const float*>(H) + i * d;
      for (int c = lane; c < d; c += 32) acc = fmaf(r[c], r[c], acc);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[i] = acc;
  }
}

// 16 lanes per row: the partial sums of the row's vocabulary parts, and the merge of its sorted lists (at most
// 16, a lane each, the largest head taken 16 times; equal logits lower column first). A row's closing
// arithmetic is a lane's of one warp: the f64 exponentials and logarithms are what bounds the kernel, and a
// warp's FP64 instruction costs the same for 2 rows as for 32. 21840 rows with 16 lists: 67 us, against 113
// with a thread per row that inserted the lists' entries one by one.
constexpr int kProxyRows = 32;
__global__ void __launch_bounds__(16 * kProxyRows)
    proxy_finalize_kernel(int64_t N, int V, int splits, const float4* __restrict__ part,
                          const float* __restrict__ ztok, const float* __restrict__ hn, const int32_t* __restrict__ tok,
                          float* __restrict__ gamma, float* __restrict__ logp, int topk_k,
                          const float2* __restrict__ topk_part, int32_t* __restrict__ top_idx,
                          float* __restrict__ top_prob, uint32_t* status) {
  __shared__ double s1_s[kProxyRows], s2_s[kProxyRows], tot_s[kProxyRows];
  __shared__ float m_s[kProxyRows];
  wait_for_previous_kernel();
  const int sub = threadIdx.x & 15, r = threadIdx.x >> 4;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * kProxyRows + r;
  const bool live = i < N;
  float m = -INFINITY;
  if (live)
    for (int s = sub; s < splits; s += 16) m = fmaxf(m, part[static_cast<int64_t>(s) * N + i].x);
#pragma unroll
  for (int o = 8; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  double S1 = 0.0, S2 = 0.0;
  if (live)
    for (int s = sub; s < splits; s += 16) {
      const float4 pr = part[static_cast<int64_t>(s) * N + i];
      const double f = exp2(static_cast<double>(pr.x) - m);
      S1 += pr.y * f;
      S2 += pr.z * f * f;
    }
#pragma unroll
  for (int o = 8; o >= 1; o >>= 1) {
    S1 += __shfl_xor_sync(0xffffffffu, S1, o);
    S2 += __shfl_xor_sync(0xffffffffu, S2, o);
  }
  if (sub == 0) {
    s1_s[r] = S1;
    s2_s[r] = S2;
    m_s[r] = m;
  }
  __syncthreads();
  if (threadIdx.x < kProxyRows) {
    const int64_t row = static_cast<int64_t>(blockIdx.x) * kProxyRows + threadIdx.x;
    const double a1 = s1_s[threadIdx.x], a2 = s2_s[threadIdx.x];
    if (row < N) {
      const int t = tok[row];
      if (t < 0 || t >= V) {
        raise_status(status, PS_DEV_BAD_TOKEN);
        gamma[row] = NAN;
        if (logp) logp[row] = NAN;
      } else {
        // S1, S2: sums over the other columns; e_o = 2^(x_o - m) for the chosen one
        const double x = static_cast<double>(ztok[row]) * 1.4426950408889634 - m_s[threadIdx.x];
        const double eo = exp2(x);
        const double tot = eo + a1;
        gamma[row] = static_cast<float>(static_cast<double>(hn[row]) * ((a1 * a1 + a2) / (tot * tot)));
        if (logp) logp[row] = static_cast<float>((x - log2(tot)) * 0.6931471805599453);
        tot_s[threadIdx.x] = tot;
      }
    }
  }
  if (topk_k == 0) return;
  __syncthreads();
  // the lists' heads: (logit, column), the next entry loaded ahead
  const float2* lst = topk_part + (static_cast<int64_t>(sub) * N + i) * 16;
  const bool has = live && sub < splits;
  const float2 none = make_float2(-INFINITY, __int_as_float(-1));
  float2 head = has ? lst[0] : none, next = has ? lst[1] : none;
  int at = 2;
  float mine_v = -INFINITY;
  int mine_id = -1;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    float v = head.x;
    int id = __float_as_int(head.y);
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, v, o);
      const int oid = __shfl_xor_sync(0xffffffffu, id, o);
      if (ov > v || (ov == v && oid < id)) {
        v = ov;
        id = oid;
      }
    }
    if (sub == j) {
      mine_v = v;
      mine_id = id;
    }
    if (__float_as_int(head.y) == id) {   // this list's head was taken
      head = next;
      next = has && at < 16 ? lst[at] : none;
      ++at;
    }
  }
  const int t = live ? tok[i] : -1;
  if (t < 0 || t >= V || sub >= topk_k) return;
  top_idx[i * topk_k + sub] = mine_id;
  top_prob[i * topk_k + sub] = static_cast<float>(exp2(static_cast<double>(mine_v) * 1.4426950408889634 - m) / tot_s[r]);
}

// ================================================================== reward uncertainty
// One warp per (prompt, step t): the group's completions that reach t contribute their top-k
// next-token probabilities with coefficient p_hat / |G_t| (success) or -(1 - p_hat) / |B_t|
// (failure); u_t = 1/2 - 1/2 (sum over distinct tokens |sum of contributions| + |other mass|). Bound by the
// comparisons of all pairs of entries: a lane compares four of its own with four others per shared load (2
// prompts of 8 completions, 3240 steps, top 16: 44 us, against 99 one pair at a time).
constexpr int kUncWarps = 4;
constexpr int kUncOwn = 4;
__host__ __device__ inline int unc_entries(int K, int topk) { return (K * topk + 3) / 4 * 4; }   // whole vectors
__global__ void __launch_bounds__(kUncWarps * 32)
    uncertainty_kernel(int P, int K, int T_max, const int32_t* __restrict__ L, const float* __restrict__ R,
                       int topk, const int32_t* __restrict__ top_idx, const float* __restrict__ top_prob,
                       const int64_t* __restrict__ off, float* __restrict__ u) {
  extern __shared__ __align__(16) uint8_t smem[];
  wait_for_previous_kernel();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int cap = unc_entries(K, topk);
  int32_t* etok = reinterpret_cast<int32_t*>(smem) + wid * cap;
  double* eval = reinterpret_cast<double*>(smem + sizeof(int32_t) * kUncWarps * cap) + wid * cap;
  const int64_t task = static_cast<int64_t>(blockIdx.x) * kUncWarps + wid;
  if (task >= static_cast<int64_t>(P) * T_max) return;
  const int p = static_cast<int>(task / T_max);
  const int t = static_cast<int>(task % T_max);   // 0-based step
  int nG = 0, gA = 0, bA = 0, Tp = 0;
  for (int j = 0; j < K; ++j) {
    const int k = p * K + j;
    const bool g = R[k] >= 0.5f;
    nG += g;
    gA += (g && L[k] > t);
    bA += (!g && L[k] > t);
    Tp = max(Tp, L[k]);
  }
  if (t >= Tp) {
    if (lane == 0) u[static_cast<int64_t>(p) * T_max + t] = 0.f;
    return;
  }
  const double phat = static_cast<double>(nG) / K;
  const double cg = gA > 0 ? phat / gA : 0.0, cb = bA > 0 ? -(1.0 - phat) / bA : 0.0;
  // entries of the alive completions, in completion order
  int E = 0;
  double other = 0.0;
  for (int j = 0; j < K; ++j) {
    const int k = p * K + j;
    if (L[k] <= t) continue;
    const double c = R[k] >= 0.5f ? cg : cb;
    const int64_t row = off[k] + t;
    double tot = 0.0;
    for (int i = lane; i < topk; i += 32) {
      etok[E + i] = top_idx[row * topk + i];
      const double pv = top_prob[row * topk + i];
      eval[E + i] = c * pv;
      tot += pv;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    other += c * (1.0 - tot);
    E += topk;
  }
  __syncwarp();
  // each distinct token's contributions in completion order, summed by the lane of its first entry
  double acc = 0.0;
  for (int e0 = lane; e0 < E; e0 += 32 * kUncOwn) {
    int tk[kUncOwn];
    bool own[kUncOwn];   // the entry exists and no earlier one has its token
    double sum[kUncOwn];
#pragma unroll
    for (int i = 0; i < kUncOwn; ++i) {
      own[i] = e0 + 32 * i < E;
      tk[i] = own[i] ? etok[e0 + 32 * i] : 0;
      sum[i] = 0.0;
    }
    for (int f0 = 0; f0 < E; f0 += 4) {
      const int4 v = *reinterpret_cast<const int4*>(etok + f0);
#pragma unroll
      for (int i = 0; i < kUncOwn; ++i) {
        unsigned hit = (v.x == tk[i] ? 1u : 0u) | (v.y == tk[i] ? 2u : 0u) | (v.z == tk[i] ? 4u : 0u) |
                       (v.w == tk[i] ? 8u : 0u);
        if (hit != 0u && own[i]) {
          for (; hit != 0u; hit &= hit - 1u) {
            const int f = f0 + __ffs(hit) - 1;
            if (f < e0 + 32 * i) own[i] = false;
            else if (f < E) sum[i] += eval[f];   // (entries past E pad the last four)
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kUncOwn; ++i)
      if (own[i]) acc += fabs(sum[i]);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    const double l1 = acc + fabs(other);
    u[static_cast<int64_t>(p) * T_max + t] = static_cast<float>(fmin(0.5, fmax(0.0, 0.5 - 0.5 * l1)));
  }
}

// One warp: exclusive scan of L.
__global__ void group_offsets_kernel(int B, const int32_t* __restrict__ L, int64_t* __restrict__ off,
                                     uint32_t* status) {
  const int lane = threadIdx.x;
  if (lane == 0) clear_status(status);   // the call's first kernel
  int64_t carry = 0;
  for (int k0 = 0; k0 < B; k0 += 32) {
    const int64_t n = k0 + lane < B ? L[k0 + lane] : 0;
    int64_t v = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (k0 + lane < B) off[k0 + lane] = carry + v - n;
    carry += __shfl_sync(0xffffffffu, v, 31);
  }
}

// ================================================================== design
constexpr int kDesignThreads = 256;
constexpr int kDesignWarps = kDesignThreads / 32;

// Prefixes that the capped design tries side by side, a lane of a warp each, on a stack of T_max blocks each: the
// workspace has these of bW, bs and bn per prompt. The arrays of one prefix tried by the whole CTA (2 T_max entries
// each, a few of each kind) lie in the same place.
constexpr int kCapLanes = 32;
struct DesignWs {
  double* w;       // [P][T_max] weights
  double* xi;      // [P][T_max]
  double* bW;      // [P][T_max][kCapLanes] block weights, one stack per lane (interleaved)
  double* bs;      // [P][T_max][kCapLanes] block scores sqrt(W / n)
  int32_t* bn;     // [P][T_max][kCapLanes] block lengths
};

// True when the block (Wc, nc) violates the order against the block (Wp, np) below it, i.e. when
// sqrt(Wp / np) < sqrt(Wc / nc) with both quotients and roots rounded to double, exactly as the
// sequential definition decides it. The cross products Wp nc and Wc np settle every case whose
// quotients differ by more than 2^-40 relative (then the rounded roots are ordered the same way): their difference's
// exponent is then at most 39 below a's (compared as integers: a double comparison takes 64 cycles).
__device__ __forceinline__ bool pav_violates_double(double Wp, int np, double Wc, int nc) {
  const double a = __dmul_rn(Wp, static_cast<double>(nc));
  const double b = __dmul_rn(Wc, static_cast<double>(np));
  const double d = __dsub_rn(b, a);
  const int ea = __double2hiint(a) >> 20, eb = __double2hiint(b) >> 20;   // biased exponents (no sign: sums of weights)
  if (ea > 123 && eb > 123 && ea < 1923 && eb < 1923 && (__double2hiint(d) >> 20 & 0x7ff) >= ea - 39)
    return __double2hiint(d) >= 0;
  return __dsqrt_rn(__ddiv_rn(Wp, static_cast<double>(np))) < __dsqrt_rn(__ddiv_rn(Wc, static_cast<double>(nc)));
}
// The same, with the products taken in float first (each within 2^-22), which settles quotients that differ by more
// than 2^-19: an SM of GB300 does two FP64 operations a clock, so double operations, let alone the near-ties'
// divisions and square roots, are slow (the design of 8 prompts of 15350 steps: 1.71 ms, without the float test 1.86).
__device__ __forceinline__ bool pav_violates(double Wp, int np, double Wc, int nc) {
  const float fa = static_cast<float>(Wp) * static_cast<float>(nc), fb = static_cast<float>(Wc) * static_cast<float>(np);
  if (fa > 1e-30f && fb > 1e-30f && fa < 1e30f && fb < 1e30f) {
    if (fb > fa * (1.0f + 0x1p-19f)) return true;
    if (fb < fa * (1.0f - 0x1p-19f)) return false;
  }
  return pav_violates_double(Wp, np, Wc, nc);
}

// Float-float numbers (an unevaluated sum hi + lo of two floats, about 44 significant bits). Knuth's TwoSum
// and the Dekker renormalisation.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return FF{s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const float lo = a.lo + b.lo;
  const FF s = two_sum(a.hi, b.hi);
  const float e = s.lo + lo;
  const float h = s.hi + e;
  return FF{h, e - (h - s.hi)};
}
__device__ __forceinline__ FF ff_select(bool c, FF a, FF b) { return FF{c ? a.hi : b.hi, c ? a.lo : b.lo}; }

__device__ __forceinline__ FF ff_shfl_up(FF v, int o) {
  return FF{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
}
// a - b as a float (a relative error of about 2^-23 of the difference beside the sums' own).
__device__ __forceinline__ float ff_diff(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }

// About 1 ulp (PTX sqrt.approx.ftz.f32).
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------- pooling by convex-hull links
// Pooling adjacent violators over weights w[s..T) one after another leaves, after t of them, blocks whose
// means fall from left to right: the segments of the least concave majorant of the prefix sums. The last
// block starts at link(t) = argmin_{a < t} (S_t - S_a) / (t - a), which every t can look for by itself, so the
// CTA finds the links of kWin positions at a time (below) and no longer walks the chain of decisions with one
// thread, whose every step costs 0.3 us or more: a dependent FP64 addition takes 64 cycles on GB300, and a
// divergent loop's turn some 50 before its work. The design kernel, 8 prompts, T = 15350: 13.7 ms with the
// one-thread walks (4.5 ms once their loops had no branches and decided in floats), 1.69 ms now; 2 prompts,
// T = 3240: 2.59 against 0.33 ms. What is left, at T = 15350: 0.35 ms for each search of links, 0.1 for each
// prefix sum, 0.7 for the sums by the links (rounds of a barrier and an FP64 addition), 0.1 for their check.
constexpr int kWin = kDesignThreads;
constexpr int kHullSmem = 14336;       // hull vertices in shared memory (deeper ones in the workspace)
constexpr size_t kDesignDynSmem = kHullSmem * (sizeof(float2) + sizeof(int32_t));

// S[u], u = 0..n: the sums of the first u values (float-float), times sign. value(i) is the i-th one. The sums before a
// window are carried in three floats, so that what a sum is off by does not grow with the windows before it: 2^-47
// relative, measured up to 2^22 values of one size or of eleven decades (in two floats, warp after warp: 2^-45 at 2^14
// values and 2^-41 at 2^22). At most it is the 14 float-float additions behind it, 2^-46 each.
template <class F>
__device__ void ff_prefix_sums(F value, int n, float sign, float2* S) {
  __shared__ float2 warp_s[kDesignWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float c0 = 0.f, c1 = 0.f, c2 = 0.f;
  if (tid == 0) S[0] = make_float2(0.f, 0.f);
  for (int i0 = 0; i0 < n; i0 += kDesignThreads) {
    const int i = i0 + tid;
    FF v{0.f, 0.f};
    if (i < n) v = value(i);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const FF y = ff_shfl_up(v, o);
      if (lane >= o) v = ff_add(y, v);
    }
    if (lane == 31) warp_s[wid] = make_float2(v.hi, v.lo);
    __syncthreads();
    FF before{0.f, 0.f}, all{0.f, 0.f};   // the window's sums before this warp, and the whole window's
    for (int k = 0; k < kDesignWarps; ++k) {
      if (k == wid) before = all;
      all = ff_add(all, FF{warp_s[k].x, warp_s[k].y});
    }
    v = ff_add(FF{c0, c1}, ff_add(before, v));
    if (i < n) S[i + 1] = make_float2(sign * v.hi, sign * v.lo);
    // (c0, c1, c2) += all: TwoSums down the three floats, then renormalised
    const FF s0 = two_sum(c0, all.hi), s1 = two_sum(c1, all.lo), s2 = two_sum(s1.hi, s0.lo);
    c2 += s1.lo + s2.lo;
    c0 = s0.hi + s2.hi;
    const float r = s2.hi - (c0 - s0.hi);
    c1 = r + c2;
    c2 -= c1 - r;
    __syncthreads();
  }
}

// link[u] = argmin over v < u of (S[u] - S[v]) / (u - v) (the nearest v on ties), u = 1..n. The hull of
// S[0..lo] is kept as a stack of its vertices; a window's positions lo < u <= lo + kWin look at every v of the
// window themselves (at most 256 steps) and at the hull by bisection (along it the slope to u falls, then
// rises); the walk from the window's end along the links then gives the next hull. Compared in float, so a
// link may be another whose slope is within about 2^-22 of the smallest.
__device__ void hull_links(const float2* S, int n, int32_t* link, float2* hull_S, int32_t* hull, int32_t* hull_deep) {
  __shared__ float2 win_S[kWin + 1];
  __shared__ int win_link[kWin], win_at[kWin], path[kWin];
  __shared__ int path_n, path_base;
  const int tid = threadIdx.x;
  auto vertex = [&](int i) { return i < kHullSmem ? hull[i] : hull_deep[i]; };
  auto vertex_S = [&](int i, int v) { return i < kHullSmem ? hull_S[i] : S[v]; };
  if (tid == 0) {
    hull[0] = 0;
    hull_S[0] = S[0];
  }
  int depth = 1;
  for (int lo = 0; lo < n; lo += kWin) {
    const int m = min(kWin, n - lo);
    for (int i = tid; i <= m; i += kDesignThreads) win_S[i] = S[lo + i];
    __syncthreads();
    if (tid < m) {
      const int u = lo + 1 + tid;
      const float2 Su = win_S[tid + 1];
      int best = u - 1, at = -1;
      float bd = ff_diff(Su, win_S[tid]), bn = 1.f;
      float nv = 1.f;
      for (int k = tid - 1; k >= 0; --k) {
        const float dv = ff_diff(Su, win_S[k]);
        nv += 1.f;
        if (dv * bn < bd * nv) {
          bd = dv;
          bn = nv;
          best = lo + k;
        }
      }
      int l = 0, r = depth - 1;   // the top vertex is lo itself
      while (l < r) {
        const int mid = (l + r) >> 1;
        const int a = vertex(mid), b = vertex(mid + 1);
        const float2 Sa = vertex_S(mid, a), Sb = vertex_S(mid + 1, b);
        if (ff_diff(Sb, Sa) * static_cast<float>(u - a) > ff_diff(Su, Sa) * static_cast<float>(b - a)) l = mid + 1;
        else r = mid;
      }
      if (l < depth - 1) {
        const int a = vertex(l);
        if (ff_diff(Su, vertex_S(l, a)) * bn < bd * static_cast<float>(u - a)) {
          best = a;
          at = l;
        }
      }
      win_link[tid] = best;
      win_at[tid] = at;
      link[u] = best;
    }
    __syncthreads();
    if (tid == 0) {
      int cnt = 0, u = lo + m, base = depth;
      while (u > lo) {
        path[cnt++] = u;
        const int i = u - lo - 1;
        if (win_at[i] >= 0) base = win_at[i] + 1;
        u = win_link[i];
      }
      path_n = cnt;
      path_base = base;
    }
    __syncthreads();
    depth = path_base + path_n;
    for (int i = tid; i < path_n; i += kDesignThreads) {
      const int v = path[path_n - 1 - i], j = path_base + i;
      if (j < kHullSmem) {
        hull[j] = v;
        hull_S[j] = win_S[v - lo];
      } else {
        hull_deep[j] = v;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- capped design: locating the prefix
// The capped design saturates the smallest prefix s whose suffix design (w[s..T), budget B - s)
// starts at or below 1. Whether a prefix qualifies is not monotone in s, so it cannot be bisected;
// instead the links of the weights taken from the right give the first block [t, T - link) of every suffix
// design at once. With D(t) = sum over a suffix's blocks of n_m s_m = sqrt(n_m W_m), which is its first block's
// term plus D at that block's end, the suffix design starts at g(t) = (B - t) s_front / D(t). status[t] records
// whether g(t) is clearly above 1 (0), clearly below (2) or within kCapBand of 1 (1); all but the first kind are then
// decided by the exact rounded sequence of the definition, in increasing order, until one passes.
// The first block's mean is the largest slope from t, hence at least Q_t / (T - t) with Q_t the sum of the
// suffix. A float-float sum is off by 2^-42 of itself at most (ff_prefix_sums), so the block's weight, the difference of
// two, by 2^-41 (T - t) / n relative: 2^-17 at the largest T of 2^24 (2^-22 with the 2^-47 that is measured), 2^-27 at
// 2^14. Its root halves that; D, an addition per window, is off by 2^-30, and roots, products and the comparison add a
// few 2^-24: inside kCapBand at every T.
constexpr double kCapBand = 0x1p-16;

// S, link: of the weights from the right, u = T - t, S negated. D [T + 1] scratch.
__device__ void cap_status(const float2* S, const int32_t* link, int T, double B, float2* D, float* status) {
  __shared__ float2 acc_s[kWin];
  __shared__ int ptr_s[kWin];
  const int tid = threadIdx.x;
  const float hi_band = static_cast<float>(1.0 + kCapBand), lo_band = static_cast<float>(1.0 - kCapBand);
  // B - t as a float: B's whole part less t is exact, so the sum is within an ulp
  const int B_whole = static_cast<int>(B);
  const float B_rest = static_cast<float>(B - static_cast<double>(B_whole));
  for (int lo = 0; lo < T; lo += kWin) {
    const int m = min(kWin, T - lo), u = lo + 1 + tid;
    int ptr = 0;
    float n = 1.f, r = 0.f;
    FF acc{0.f, 0.f};
    if (tid < m) {
      ptr = link[u];
      n = static_cast<float>(u - ptr);
      r = sqrt_approx(n * ff_diff(S[ptr], S[u]));
      acc.hi = r;
    }
    // sums along the links inside the window, twice as far each round
    while (__syncthreads_or(ptr > lo)) {
      acc_s[tid] = make_float2(acc.hi, acc.lo);
      ptr_s[tid] = ptr;
      __syncthreads();
      if (ptr > lo) {
        const int i = ptr - lo - 1;
        acc = ff_add(acc, FF{acc_s[i].x, acc_s[i].y});
        ptr = ptr_s[i];
      }
    }
    if (tid < m) {
      if (ptr > 0) {
        const float2 rest = D[ptr];
        acc = ff_add(acc, FF{rest.x, rest.y});
      }
      D[u] = make_float2(acc.hi, acc.lo);
      const int t = T - u;
      const float num = (static_cast<float>(B_whole - t) + B_rest) * r, den = acc.hi * n;
      status[t] = num > hi_band * den ? 0.f : (num < lo_band * den ? 2.f : 1.f);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- pooling in the definition's arithmetic
// first[t], W[t] for s < t <= T: the last block [first[t], t) after the weights w[s..t) have been pooled one after
// another, and its sum as the definition adds it: the new weight c, then W_prev + c for each block that it
// violates the order with, from the nearest on. A block below the last one is the last one of an earlier t, so
// the sums of a window of kWin positions are taken together where the links say which blocks they merge; and every
// decision is then checked on the sums themselves (pav_violates), which by induction over t makes the result the
// sequential one whatever the links were. Up to kBatch windows are pooled and then checked together; from the first of
// them with a decision that differs (its link came from slopes that the float sums cannot tell apart: near-ties, or
// weights far below the sums before them) they are done again and checked one by one, and in a window the first
// position that differs is redone alone and those after it again. After kMaxRepairs of these one thread does the
// window's rest, and whole windows: kSerial, and twice as many each time that the links, tried again, are wrong again.
// 8 prompts of 15000 steps: 1.4 ms without a wrong link, 1.6 to 2.0 with some dozens (half to nine tenths of the steps'
// weights spread over ten decades; 5.4 to 7.6 when a repair had everything after it pooled again, and with 4 repairs
// and 8 windows 1.7 to 6.0), 11 where nearly all are wrong (weights within 1e-7 of each other; then 31, and 15 by one
// thread from the start on).
constexpr int kBatch = 16;
constexpr int kMaxRepairs = 12;
constexpr int kSerial = 2;
struct Pooled {
  const double* w;
  int s, T;
  const int32_t* link;   // [T - s + 1], relative to s
  int32_t* first;        // [T + 1]
  double* W;             // [T + 1]

  __device__ void run() const {   // (the whole CTA)
    __shared__ double w_s[kWin], W_s[kWin];
    __shared__ int first_s[kWin], ready_s[kWin];
    __shared__ int wrong_s;
    const int tid = threadIdx.x;
    int repairs_left = kMaxRepairs, serial_left = 0, serial_next = kSerial;
    int size = kBatch / 4;   // windows of a batch
    bool one_by_one = false;
    for (int b0 = s, b1; b0 < T; b0 = b1) {
      b1 = min(T, b0 + kWin * size);
      int unclean = 0, redo = b0;
      for (int checked = one_by_one ? 1 : 0; checked < 2; ++checked) {
        for (int lo = checked ? redo : b0; lo < b1; lo += kWin) {
          const int t = lo + 1 + tid, end = min(T, lo + kWin);
          const bool mine = t <= T;
          const double wt = mine ? w[t - 1] : 0.0;
          const int target = mine ? s + link[t - s] : t;
          auto sum = [&](int j) { return j > lo ? W_s[j - lo - 1] : W[j]; };
          auto start = [&](int j) { return j > lo ? first_s[j - lo - 1] : first[j]; };
          // positions k0..k1 as the definition does them, on those before them (one thread)
          auto serial = [&](int k0, int k1) {
            int j = k0 - 1, f = j > s ? start(j) : s;
            double Wj = j > s ? sum(j) : 0.0;   // [f, j) is the last block after k0 - 1 weights, Wj its sum
            for (int k = k0; k <= k1; ++k) {
              double c = w_s[k - lo - 1];
              j = k - 1;
              while (j > s) {
                const double below = f > s ? sum(f) : 0.0;   // the block before it, loaded under the decision
                const int below_f = f > s ? start(f) : s;
                if (!pav_violates_double(Wj, j - f, c, k - j)) break;
                c = __dadd_rn(Wj, c);
                j = f;
                Wj = below;
                f = below_f;
              }
              W_s[k - lo - 1] = Wj = c;
              first_s[k - lo - 1] = f = j;
            }
          };
          w_s[tid] = wt;
          int from = lo + 1;
          if (checked && serial_left > 0) {
            __syncthreads();
            if (tid == 0) serial(from, end);
            __syncthreads();
            from = end + 1;
            ++unclean;
            --serial_left;
          }
          while (from <= end) {
            // positions from..end by the links
            bool done = !mine || t < from;
            double c = wt;
            int j = t - 1;
            if (!done) ready_s[tid] = 0;
            if (tid == 0) wrong_s = end + 1;
            __syncthreads();
            while (true) {
              bool fresh = false;
              if (!done) {
                while (j > target) {
                  const int k = j - lo - 1;
                  if (k < 0) {
                    c = __dadd_rn(W[j], c);
                    j = first[j];
                  } else {
                    if (!ready_s[k]) break;
                    c = __dadd_rn(W_s[k], c);
                    j = first_s[k];
                  }
                }
                if (j <= target) {
                  W_s[tid] = c;
                  first_s[tid] = j;
                  done = fresh = true;
                }
              }
              __syncthreads();
              if (fresh) ready_s[tid] = 1;
              if (!__syncthreads_or(!done)) break;
            }
            if (!checked) break;
            if (mine && t >= from && !right(t, wt, sum, start)) atomicMin(&wrong_s, t);
            __syncthreads();
            const int wrong = wrong_s;
            __syncthreads();
            if (wrong > end) {
              if (from == lo + 1) {
                repairs_left = kMaxRepairs;
                serial_next = kSerial;
              }
              break;
            }
            unclean += from == lo + 1;
            if (repairs_left > 0) {
              --repairs_left;
              from = wrong + 1;
            } else {
              serial_left = serial_next;
              serial_next *= 2;
              from = end + 1;
            }
            if (tid == 0) serial(wrong, from - 1);
            __syncthreads();
          }
          if (mine) {
            W[t] = W_s[tid];
            first[t] = first_s[tid];
          }
          __syncthreads();
        }
        if (checked) break;
        // the batch's first window with a wrong decision
        if (tid == 0) wrong_s = b1 + 1;
        __syncthreads();
        for (int t = b0 + 1 + tid; t <= b1; t += kDesignThreads)
          if (!right(t, w[t - 1], [&](int j) { return W[j]; }, [&](int j) { return first[j]; })) {
            atomicMin(&wrong_s, t);
            break;
          }
        __syncthreads();
        redo = wrong_s > b1 ? b1 : b0 + (wrong_s - b0 - 1) / kWin * kWin;
        __syncthreads();
      }
      one_by_one = 4 * unclean >= size;
      size = unclean > 0 ? kBatch / 4 : min(kBatch, 2 * size);
    }
  }
  // Whether first[t] is where the definition's decisions lead from w[t - 1] = c.
  template <class Sum, class Start>
  __device__ __forceinline__ bool right(int t, double c, const Sum& sum, const Start& start) const {
    const int f = start(t);
    int j = t - 1;
    while (j > f) {
      const double Wj = sum(j);
      const int fj = start(j);
      if (!pav_violates(Wj, j - fj, c, t - j)) return false;
      c = __dadd_rn(Wj, c);
      j = fj;
    }
    return j <= s || !pav_violates(sum(j), j - start(j), c, t - j);
  }
  // The blocks after all weights, last one first: their ends in `ends`; returns their number (the whole CTA).
  // A position is a block's end if no later one's block reaches over it.
  __device__ int blocks(int32_t* ends) const {
    __shared__ int min_s[kDesignWarps], cnt_s[kDesignWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int reach = T, count = 0;   // the smallest start among positions further right, and the ends found there
    for (int t0 = T; t0 > s; t0 -= kDesignThreads) {
      const int t = t0 - tid;   // thread order runs from right to left
      const int f = t > s ? first[t] : T;
      int low = f;              // smallest start among this and the earlier threads of the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, low, o);
        if (lane >= o) low = min(low, y);
      }
      if (lane == 31) min_s[wid] = low;
      int right = __shfl_up_sync(0xffffffffu, low, 1);   // ... among the earlier threads alone
      if (lane == 0) right = T;
      __syncthreads();
      right = min(right, reach);
      for (int k = 0; k < kDesignWarps; ++k) {
        if (k < wid) right = min(right, min_s[k]);
        reach = min(reach, min_s[k]);
      }
      const bool end = t > s && right >= t;
      const unsigned mask = __ballot_sync(0xffffffffu, end);
      if (lane == 0) cnt_s[wid] = __popc(mask);
      __syncthreads();
      int at = count + __popc(mask & ((1u << lane) - 1u));
      for (int k = 0; k < kDesignWarps; ++k) {
        if (k < wid) at += cnt_s[k];
        count += cnt_s[k];
      }
      if (end) ends[at] = t;
      __syncthreads();
    }
    return count;
  }
};

// Pools w[0..T) one weight after another into one lane's stack (element m of the stack at index m * kCapLanes), each
// block sum added as the definition adds it. The last block stays in registers, and memory is read only when a merge
// uncovers the block below. (Traces that get here are nearly flat: the float test would only add to the double one.)
// Returns the number of blocks.
__device__ __noinline__ int pav_stack(const double* w, int T, double* bW, int32_t* bn) {
  int nb = 0, nt = 0;
  double Wt = 0.0, wnext = T > 0 ? w[0] : 0.0;
  for (int t = 0; t < T; ++t) {
    if (t + 16 < T) asm volatile("prefetch.global.L1 [%0];" ::"l"(w + t + 16));
    double Wc = wnext;
    if (t + 1 < T) wnext = w[t + 1];
    int nc = 1;
    while (nb > 0 && pav_violates_double(Wt, nt, Wc, nc)) {
      Wc = __dadd_rn(Wt, Wc);
      nc += nt;
      --nb;
      if (nb > 0) {
        Wt = bW[static_cast<int64_t>(nb - 1) * kCapLanes];
        nt = bn[static_cast<int64_t>(nb - 1) * kCapLanes];
      }
    }
    if (nb > 0) {
      bW[static_cast<int64_t>(nb - 1) * kCapLanes] = Wt;
      bn[static_cast<int64_t>(nb - 1) * kCapLanes] = nt;
    }
    Wt = Wc;
    nt = nc;
    ++nb;
  }
  if (nb > 0) {
    bW[static_cast<int64_t>(nb - 1) * kCapLanes] = Wt;
    bn[static_cast<int64_t>(nb - 1) * kCapLanes] = nt;
  }
  return nb;
}

// Timestep weights of the OPTIMIZED and HEURISTIC designs, before the floor: w_t = gamma_bar_t * u_t with
// gamma_bar_t = (1/K) sum over the completions that reach t, and the largest of each kWeightSteps steps. A
// division costs tens of FP64 operations, of which an SM of GB300 does two a clock, so the steps are spread over
// the chip: 17 us for 8 prompts of 16 completions and 15350 steps. Traces of one such part are weighed by the design
// kernel itself, a launch less (heuristic design of 20 steps: 11.6 us, 15 with the launch).
constexpr int kWeightSteps = 512;
// A prompt's rows before its first completion (with_rows) and its horizon, the longest completion (the whole CTA).
struct Group {
  long long base;
  int horizon;
};
__device__ __forceinline__ Group group_of(int p, int K, const int32_t* __restrict__ L, bool with_rows) {
  __shared__ long long red_l[kDesignWarps];
  __shared__ int red_i[kDesignWarps];
  const int tid = threadIdx.x;
  Group g{0, 0};
  if (with_rows)
    for (int k = tid; k < p * K; k += kDesignThreads) g.base += L[k];
  for (int j = tid; j < K; j += kDesignThreads) g.horizon = max(g.horizon, L[p * K + j]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    g.base += __shfl_xor_sync(0xffffffffu, g.base, o);
    g.horizon = max(g.horizon, __shfl_xor_sync(0xffffffffu, g.horizon, o));
  }
  if ((tid & 31) == 0) {
    red_l[tid >> 5] = g.base;
    red_i[tid >> 5] = g.horizon;
  }
  __syncthreads();
  g.base = 0;
  for (int i = 0; i < kDesignWarps; ++i) {
    g.base += red_l[i];
    g.horizon = max(g.horizon, red_i[i]);
  }
  return g;
}
// The weights of the steps [t0, t1) into w; returns the largest of this thread's.
__device__ __forceinline__ double design_weights(int p, int K, int T_max, const int32_t* __restrict__ L,
                                                 const float* __restrict__ gamma, const float* __restrict__ u,
                                                 long long base, int t0, int t1, double* __restrict__ w,
                                                 uint32_t* status) {
  double wmax = 0.0;
  for (int t = t0 + static_cast<int>(threadIdx.x); t < t1; t += kDesignThreads) {
    double acc = 0.0;
    long long off = base;
    for (int j = 0; j < K; ++j) {
      const int n = L[p * K + j];
      if (t < n) acc = __dadd_rn(acc, static_cast<double>(gamma[off + t]));
      off += n;
    }
    double v = __ddiv_rn(acc, static_cast<double>(K));
    if (u) v = __dmul_rn(v, static_cast<double>(u[static_cast<int64_t>(p) * T_max + t]));
    if (!isfinite(v)) raise_status(status, PS_DEV_NONFINITE);
    w[t] = v;
    wmax = fmax(wmax, v);
  }
  return wmax;
}
__global__ void __launch_bounds__(kDesignThreads)
    design_weights_kernel(int K, int T_max, const int32_t* __restrict__ L, const float* __restrict__ gamma,
                          const float* __restrict__ u, DesignWs ws, uint32_t* status) {
  __shared__ double red_d[kDesignWarps];
  const int p = blockIdx.x, tid = threadIdx.x;
  const Group g = group_of(p, K, L, true);
  const int Tp = min(max(g.horizon, 1), T_max);
  double wmax = design_weights(p, K, T_max, L, gamma, u, g.base, blockIdx.y * kWeightSteps,
                               min(Tp, static_cast<int>(blockIdx.y + 1) * kWeightSteps),
                               ws.w + static_cast<int64_t>(p) * T_max, status);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
  if ((tid & 31) == 0) red_d[tid >> 5] = wmax;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < kDesignWarps; ++i) wmax = fmax(wmax, red_d[i]);
    ws.bW[static_cast<int64_t>(p) * T_max * kCapLanes + blockIdx.y] = wmax;   // free until the pooling
  }
}

// One CTA per prompt (and, OPTIMIZED, 172 KB of shared memory each): registers are not what limits residency. gamma, u:
// the weights are taken here; nullptr: design_weights_kernel has taken them, or the strategy has none.
template <bool OPTIMIZED>
__global__ void __launch_bounds__(kDesignThreads, 1)
    design_kernel(int K, int T_max, const int32_t* __restrict__ L, const float* __restrict__ gamma,
                  const float* __restrict__ u, double budget, int strategy, double param, uint64_t* __restrict__ q,
                  double* __restrict__ xi_out, DesignWs ws, uint32_t* status) {
  const int p = blockIdx.x;
  const int tid = threadIdx.x;
  __shared__ double red_d[kDesignThreads / 32];
  __shared__ unsigned long long red_u[kDesignThreads / 32];
  __shared__ unsigned long long red_b[kDesignThreads / 32];
  __shared__ int red_i[kDesignThreads / 32];
  __shared__ double lam_s;
  __shared__ int decided_s, found_s;
  __shared__ int cand_s[kCapLanes], nb_s[kCapLanes];
  __shared__ double den_s;
  extern __shared__ __align__(16) float2 dyn_smem[];    // the hull's vertices (kDesignDynSmem bytes)
  const int lane = tid & 31, wid = tid >> 5;
  double* w = ws.w + static_cast<int64_t>(p) * T_max;
  double* xi = ws.xi + static_cast<int64_t>(p) * T_max;

  const Group group = group_of(p, K, L, gamma != nullptr);
  if (tid == 0 && (group.horizon < 1 || group.horizon > T_max)) raise_status(status, PS_DEV_BAD_LENGTH);
  const int Tp = min(max(group.horizon, 1), T_max);
  const double Bp = fmin(budget, static_cast<double>(Tp));

  if (OPTIMIZED || strategy == PS_DESIGN_HEURISTIC) {
    // the floor under the weights: the largest of them, taken here or from the weights kernel's parts
    double wmax = 0.0;
    if (gamma != nullptr) {
      wmax = design_weights(p, K, T_max, L, gamma, u, group.base, 0, Tp, w, status);
    } else {
      const double* parts = ws.bW + static_cast<int64_t>(p) * T_max * kCapLanes;
      for (int c = tid; c * kWeightSteps < Tp; c += kDesignThreads) wmax = fmax(wmax, parts[c]);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
    if (lane == 0) red_d[wid] = wmax;
    __syncthreads();
    double wm = 0.0;
    for (int i = 0; i < kDesignThreads / 32; ++i) wm = fmax(wm, red_d[i]);
    const double fl = __dmul_rn(1e-12, wm);
    for (int t = tid; t < Tp; t += kDesignThreads) w[t] = wm > 0.0 ? (w[t] > fl ? w[t] : fl) : 1.0;
    __syncthreads();
    if constexpr (OPTIMIZED) {
      // The smallest saturated prefix s whose suffix design (budget B - s) starts at or below 1, decided by
      // the definition's exact rounded sequence: for a candidate s, w[s..T) is pooled, the blocks' scores are
      // s_m = sqrt(W_m / n_m), den = sum_m n_m s_m in block order, and it passes if (B - s) s_1 / den <= 1.
      // Candidates, in increasing order: the prefixes whose status is not clearly above 1. As a rule the first or
      // second passes. The whole CTA tries them one by one until that has taken the steps of two whole traces; the
      // rest go 32 at a time, a lane each: a budget at or above the horizon puts every suffix that is flat to 2^-16
      // into the band, hundreds of them, and where the weights fall slowly none passes before the last. (4000
      // steps that fall by 3e-6 in all, budget 4000: 0.44 s so, 15.8 s one by one.)
      const int64_t stacks = static_cast<int64_t>(p) * T_max * kCapLanes;
      const int64_t pitch = 2 * static_cast<int64_t>(T_max);   // at least T + 1
      double* fW = ws.bW + stacks;
      double* fs = ws.bs + stacks;
      int32_t* fn = ws.bn + stacks;
      float2* S = reinterpret_cast<float2*>(fW);
      float2* D = reinterpret_cast<float2*>(fW + pitch);
      double* blockW = fW + 2 * pitch;      // Pooled::W
      double* score = fs;
      double* term = fs + pitch;
      int32_t* link = fn;
      int32_t* first = fn + pitch;
      int32_t* ends = fn + 2 * pitch;
      int32_t* hull_deep = fn + 3 * pitch;
      float2* hull_S = dyn_smem;
      int32_t* hull = reinterpret_cast<int32_t*>(hull_S + kHullSmem);
      float* status = reinterpret_cast<float*>(xi);            // xi is written last
      const double inv = 1.0 / (wm > 0.0 ? wm : 1.0);
      auto scaled = [&](int t) {   // w[t] over the largest weight: in [1e-12, 1]
        const double v = w[t] * inv;
        const float hi = static_cast<float>(v);
        return FF{hi, static_cast<float>(v - static_cast<double>(hi))};
      };
      ff_prefix_sums([&](int i) { return scaled(Tp - 1 - i); }, Tp, -1.f, S);
      hull_links(S, Tp, link, hull_S, hull, hull_deep);
      cap_status(S, link, Tp, Bp, D, status);
      // The next prefixes from `from` on that are to be tried, at most `most` of them, into cand_s in increasing
      // order; returns their number (the whole CTA). above: those whose status is clearly above 1 instead.
      auto candidates = [&](int from, int most, bool above) {
        int count = 0;
        for (int t0 = from; t0 < Tp && count < most; t0 += kDesignThreads) {
          const int t = t0 + tid;
          const bool take = t < Tp && (status[t] == 0.f) == above;
          const unsigned mask = __ballot_sync(0xffffffffu, take);
          if (lane == 0) red_i[wid] = __popc(mask);
          __syncthreads();
          int at = count + __popc(mask & ((1u << lane) - 1u));
          for (int k = 0; k < kDesignWarps; ++k) {
            if (k < wid) at += red_i[k];
            count += red_i[k];
          }
          if (take && at < most) cand_s[at] = t;
          __syncthreads();
        }
        return min(count, most);
      };
      int nb = 0;
      // Pools w[s..T) and tests the prefix; block m's end is ends[nb - 1 - m].
      auto passes = [&](int s) {
        ff_prefix_sums([&](int i) { return scaled(s + i); }, Tp - s, 1.f, S);
        hull_links(S, Tp - s, link, hull_S, hull, hull_deep);
        const Pooled pool{w, s, Tp, link, first, blockW};
        pool.run();
        nb = pool.blocks(ends);
        for (int m = tid; m < nb; m += kDesignThreads) {
          const int e = ends[nb - 1 - m];
          const double n = static_cast<double>(e - first[e]);
          const double sc = __dsqrt_rn(__ddiv_rn(blockW[e], n));
          score[m] = sc;
          term[m] = __dmul_rn(n, sc);
        }
        __syncthreads();
        if (tid == 0) {
          double den = 0.0;
          int m = 0;
          for (; m + 8 <= nb; m += 8) {
            double v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = term[m + j];
#pragma unroll
            for (int j = 0; j < 8; ++j) den = __dadd_rn(den, v[j]);
          }
          for (; m < nb; ++m) den = __dadd_rn(den, term[m]);
          den_s = den;
        }
        __syncthreads();
        return __ddiv_rn(__dmul_rn(__dsub_rn(Bp, static_cast<double>(s)), score[0]), den_s) <= 1.0;
      };
      // The first of cand_s[0..n) that passes, -1 if none does; lane l of warp 0 pools for cand_s[l].
      auto first_passing = [&](int n) {
        if (wid == 0) nb_s[lane] = lane < n ? pav_stack(w + cand_s[lane], Tp - cand_s[lane], fW + lane, fn + lane) : 0;
        __syncthreads();
        for (int l = 0; l < n; ++l)
          for (int m = tid; m < nb_s[l]; m += kDesignThreads) {
            const int64_t at = static_cast<int64_t>(m) * kCapLanes + l;
            fs[at] = __dsqrt_rn(__ddiv_rn(fW[at], static_cast<double>(fn[at])));
          }
        __syncthreads();
        if (wid == 0) {
          bool ok = false;
          if (lane < n) {
            double den = 0.0;
            for (int64_t m = 0, at = lane; m < nb_s[lane]; ++m, at += kCapLanes)
              den = __dadd_rn(den, __dmul_rn(static_cast<double>(fn[at]), fs[at]));
            ok = __ddiv_rn(__dmul_rn(__dsub_rn(Bp, static_cast<double>(cand_s[lane])), fs[lane]), den) <= 1.0;
          }
          const unsigned m = __ballot_sync(0xffffffffu, ok);
          if (lane == 0) found_s = m != 0u ? cand_s[__ffs(m) - 1] : -1;
        }
        __syncthreads();
        return found_s;
      };
      int found = -1, from = 0;
      if (isfinite(wm)) {   // (an infinite weight has no design: PS_DEV_NONFINITE)
        for (int64_t steps = 0; found < 0 && candidates(from, 1, false) == 1;) {
          const int t = cand_s[0];
          steps += Tp - t;
          if (steps > 2 * static_cast<int64_t>(Tp)) break;
          if (passes(t)) found = t;
          from = t + 1;
        }
        // (the last prefix always passes, so those clearly above 1 are tried only if the statuses were wrong)
        for (int above = 0; above < 2 && found < 0; ++above, from = 0)
          for (int n; found < 0 && (n = candidates(from, kCapLanes, above != 0)) > 0;) {
            from = cand_s[n - 1] + 1;
            found = first_passing(n);
            if (found >= 0) passes(found);   // its blocks
          }
      }
      __syncthreads();
      if (found < 0) {
        for (int t = tid; t < Tp; t += kDesignThreads) xi[t] = 1.0;
      } else {
        const double Bs = __dsub_rn(Bp, static_cast<double>(found));
        for (int t = tid; t < found; t += kDesignThreads) xi[t] = 1.0;
        // short blocks by a thread each, long ones by a warp
        auto fill = [&](int m, int t_first, int t_step, bool want_long) {
          const int b1 = ends[nb - 1 - m], b0 = first[b1];
          if ((b1 - b0 >= 64) != want_long) return;
          const double v = __ddiv_rn(__dmul_rn(Bs, score[m]), den_s);
          for (int t = b0 + t_first; t < b1; t += t_step) xi[t] = v;
        };
        for (int m = tid; m < nb; m += kDesignThreads) fill(m, 0, 1, false);
        for (int m = wid; m < nb; m += kDesignWarps) fill(m, lane, 32, true);
      }
    } else {
      // Heuristic: closed form B sqrt(w_t) / sum_j sqrt(w_j) (the sum in step order), a running
      // minimum, then the cap at 1. The roots and quotients are taken in parallel.
      for (int t = tid; t < Tp; t += kDesignThreads) xi[t] = __dsqrt_rn(w[t]);
      __syncthreads();
      if (tid == 0) {
        double tot = 0.0;
        int t = 0;
        for (; t + 8 <= Tp; t += 8) {
          double v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = xi[t + j];
#pragma unroll
          for (int j = 0; j < 8; ++j) tot = __dadd_rn(tot, v[j]);
        }
        for (; t < Tp; ++t) tot = __dadd_rn(tot, xi[t]);
        den_s = tot;
      }
      __syncthreads();
      const double tot = den_s;
      // the running minimum over 256 steps at a time: a scan in each warp, then the minima before it
      double run = INFINITY;
      for (int t0 = 0; t0 < Tp; t0 += kDesignThreads) {
        const int t = t0 + tid;
        double v = t < Tp ? __ddiv_rn(__dmul_rn(Bp, xi[t]), tot) : INFINITY;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double y = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v = fmin(y, v);
        }
        if (lane == 31) red_d[wid] = v;
        __syncthreads();
        for (int i = 0; i < wid; ++i) run = fmin(run, red_d[i]);
        if (t < Tp) xi[t] = fmin(fmin(run, v), 1.0);
        for (int i = wid; i < kDesignWarps; ++i) run = fmin(run, red_d[i]);
        __syncthreads();
      }
    }
  } else if (strategy == PS_DESIGN_UNIFORM) {
    for (int t = tid; t < Tp; t += kDesignThreads)
      xi[t] = __ddiv_rn(static_cast<double>(Tp - t), static_cast<double>(Tp));
  } else if (strategy == PS_DESIGN_FIXED) {
    for (int t = tid; t < Tp; t += kDesignThreads) xi[t] = (t + 1 <= param) ? 1.0 : 0.0;
  } else {  // PS_DESIGN_TIME_PRIOR: xi_t = exp(-lam t), sum_t xi_t = budget, lam by bisection
    auto budget_at = [&](double lam) {
      double part = 0.0;
      for (int t = tid; t < Tp; t += kDesignThreads) part += exp(-lam * t);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      __syncthreads();
      if (lane == 0) red_d[wid] = part;
      __syncthreads();
      double tot = 0.0;
      for (int i = 0; i < kDesignThreads / 32; ++i) tot += red_d[i];
      return tot;
    };
    // Whether the budget at lam exceeds Bp. The sum is (1 - e^(-lam T)) / (1 - e^-lam), which one thread has in
    // microseconds, where the sum over T steps keeps an SM's FP64 lanes busy for T / 200 us. Both are off by at
    // most (T / 256 + 32) 2^-53 relative (the longest chain of additions, and a few roundings), so outside
    // twice that band the closed form decides as the sum would; inside it, the sum decides.
    constexpr int kClosedFormFrom = 2048;
    auto over = [&](double lam) {
      if (Tp >= kClosedFormFrom) {
        __syncthreads();
        if (tid == 0) {
          const double est = expm1(-lam * Tp) / expm1(-lam);
          const double band = (Tp / kDesignThreads + 32) * 0x1p-52 * Bp;
          decided_s = est > Bp + band ? 1 : est < Bp - band ? 0 : -1;
        }
        __syncthreads();
        if (decided_s >= 0) return decided_s != 0;
      }
      return budget_at(lam) > Bp;
    };
    if (static_cast<double>(Tp) <= Bp) {
      if (tid == 0) lam_s = 0.0;
    } else {
      double lo = 0.0, hi = 1.0;
      for (int it = 0; it < 64 && over(hi); ++it) hi *= 2.0;
      for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (mid <= lo || mid >= hi) break;   // lo and hi are adjacent doubles: nothing changes any more
        if (over(mid)) lo = mid;
        else hi = mid;
      }
      if (tid == 0) lam_s = hi;
    }
    __syncthreads();
    for (int t = tid; t < Tp; t += kDesignThreads) xi[t] = exp(-lam_s * t);
  }
  __syncthreads();

  // masses q_h = floor((xi_h - xi_{h+1}) 2^62); excess over 2^62 comes off the largest mass
  uint64_t* qp = q + static_cast<int64_t>(p) * T_max;
  unsigned long long sum = 0, best = 0;
  int besti = INT_MAX;
  for (int t = tid; t < T_max; t += kDesignThreads) {
    uint64_t v = 0;
    if (t < Tp) {
      const double d = __dsub_rn(xi[t], t + 1 < Tp ? xi[t + 1] : 0.0);
      v = d > 0.0 ? __double2ull_rz(floor(__dmul_rn(d, 4611686018427387904.0))) : 0ull;
    }
    qp[t] = v;
    if (xi_out) xi_out[static_cast<int64_t>(p) * T_max + t] = t < Tp ? xi[t] : 0.0;
    sum += v;
    if (v > best || (v == best && t < besti)) {
      best = v;
      besti = t;
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, besti, o);
    if (ob > best || (ob == best && oi < besti)) {
      best = ob;
      besti = oi;
    }
  }
  __syncthreads();
  if (lane == 0) {
    red_u[wid] = sum;
    red_b[wid] = best;
    red_i[wid] = besti;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long s = 0, b = 0;
    int bi = INT_MAX;
    for (int i = 0; i < kDesignThreads / 32; ++i) {
      s += red_u[i];
      const unsigned long long v = red_b[i];
      if (v > b || (v == b && red_i[i] < bi)) {
        b = v;
        bi = red_i[i];
      }
    }
    if (s > kOne62 && bi < T_max) qp[bi] -= (s - kOne62);
  }
}

// ---------------------------------------------------------------- reward binarisation (Appendix G)
constexpr uint64_t kRewardKeyTag = 0x5053505052574431ull;  // "PSPPRWD1"
constexpr double kLn2d = 0.6931471805599453;              // the double nearest ln 2
constexpr double kTwo53 = 9007199254740992.0;

// sigma(r) = 1 / (1 + e^-r) by one fixed sequence of correctly rounded double operations:
// z = -r clamped to [-40, 40], k = floor(z / ln2 + 1/2), f = z - k ln2, e^f by Horner's rule
// over its Taylor series to degree 16, e^z = e^f 2^k (exact scaling), sigma = 1 / (1 + e^z).
// No step is left to the compiler's choice (no contraction into FMAs), so the value is the
// same double wherever the sequence is repeated. The clamp moves sigma by less than 4.3e-18.
__device__ double sigmoid_fixed_dev(double r) {
  if (r != r) return 0.0;
  double z = -r;
  z = z > 40.0 ? 40.0 : (z < -40.0 ? -40.0 : z);
  const double k = floor(__dadd_rn(__ddiv_rn(z, kLn2d), 0.5));
  const double f = __dsub_rn(z, __dmul_rn(k, kLn2d));
  double p = 1.0;
  for (int n = 16; n >= 1; --n) p = __dadd_rn(1.0, __ddiv_rn(__dmul_rn(f, p), static_cast<double>(n)));
  const double two_k = __longlong_as_double(static_cast<long long>(static_cast<int>(k) + 1023) << 52);
  return __ddiv_rn(1.0, __dadd_rn(1.0, __dmul_rn(p, two_k)));
}

// y_k = 1 when the trajectory's 53-bit Philox uniform lies below sigma(R_k), else 0.
__global__ void binarize_rewards_kernel(int B, const float* __restrict__ R, uint64_t seed, uint64_t step,
                                        int64_t traj_base, float* __restrict__ y) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= B) return;
  uint64_t c[4] = {static_cast<uint64_t>(traj_base + k), step, 0ull, 0ull};
  philox4x64_10(c, seed, kRewardKeyTag);
  const double m = static_cast<double>(c[0] >> 11);
  const double s = sigmoid_fixed_dev(static_cast<double>(R[k]));
  y[k] = m < __dmul_rn(s, kTwo53) ? 1.0f : 0.0f;
}

}  // namespace psk

using namespace psk;

extern "C" {

// Score-proxy workspace: header | ztok [N] f32 | hn [N] f32 | part [S][N] float4 (S as many as fit,
// up to one per 256-column vocabulary tile) -- with top-k: part [S][N] float4 and topk [S][N][16]
// float2 for S <= 16 contiguous vocabulary ranges.
static size_t proxy_fixed(int64_t N) { return kWsHeader + al256(sizeof(float) * N) * 2; }
static size_t proxy_per_split(int64_t N, int topk) {
  return (sizeof(float4) + (topk > 0 ? sizeof(float2) * 16 : 0)) * static_cast<size_t>(N);
}
static int proxy_max_splits(int V, int topk) { return topk > 0 ? 16 : fwd_tile_splits_bf16(V); }

size_t ps_lmhead_score_proxy_workspace_size(int64_t N, int d, int V, int dtype, int topk) {
  if (N < 0 || V < 1 || d < 8 || dtype != PS_DTYPE_BF16 || topk < 0 || topk > 16) return 0;
  int S = proxy_max_splits(V, topk);
  if (S > fwd_tile_splits_bf16(V)) S = fwd_tile_splits_bf16(V);
  return proxy_fixed(N) + proxy_per_split(N, topk) * S;
}

int ps_lmhead_score_proxy(int64_t N, int d, int V, int dtype, const void* Hrows, const void* W, const int32_t* tok,
                          float* gamma, float* logp, int topk, int32_t* top_idx, float* top_prob, void* ws,
                          size_t ws_bytes, ps_stream_t stream) {
  NvtxRange nvtx_range("ps_lmhead_score_proxy");
  if (N < 0 || N > INT32_MAX || V < 1 || d < 8 || d % 8 || topk < 0 || topk > 16) return PS_ERR_INVALID_ARG;
  if (dtype != PS_DTYPE_BF16) return PS_ERR_UNSUPPORTED;
  if (N > 0 && (!Hrows || !W || !tok || !gamma)) return PS_ERR_INVALID_ARG;
  if (N > 0 && topk > 0 && (!top_idx || !top_prob)) return PS_ERR_INVALID_ARG;
  if (N > 0 && ((reinterpret_cast<uintptr_t>(Hrows) & 15) || (reinterpret_cast<uintptr_t>(W) & 15)))
    return PS_ERR_INVALID_ARG;
  if (!device_is_sm103()) return PS_ERR_UNSUPPORTED;
  if (ws == nullptr || (reinterpret_cast<uintptr_t>(ws) & 255)) return PS_ERR_WORKSPACE;
  const size_t fixed = proxy_fixed(N);
  int S = proxy_max_splits(V, topk);
  if (S > fwd_tile_splits_bf16(V)) S = fwd_tile_splits_bf16(V);
  if (N > 0) {
    const size_t room = ws_bytes > fixed ? ws_bytes - fixed : 0;
    const size_t fit = room / proxy_per_split(N, topk);
    if (fit < static_cast<size_t>(S)) S = static_cast<int>(fit);
    if (S < 1) return PS_ERR_WORKSPACE;
  }
  if (ws_bytes < fixed) return PS_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (N == 0) return cudaMemsetAsync(ws, 0, kWsHeader, s) == cudaSuccess ? PS_OK : PS_ERR_CUDA;
  uint8_t* base = static_cast<uint8_t*>(ws);
  float* ztok = reinterpret_cast<float*>(base + kWsHeader);
  float* hn = reinterpret_cast<float*>(base + kWsHeader + al256(sizeof(float) * N));
  float4* part = reinterpret_cast<float4*>(base + fixed);
  float2* tpart = reinterpret_cast<float2*>(base + fixed + sizeof(float4) * static_cast<size_t>(S) * N);
  uint32_t* status = static_cast<uint32_t*>(ws);
  row_sqnorm_kernel<<<num_sms_current() * 8, 256, 0, s>>>(N, d, 1, Hrows, hn, status);
  if (cudaGetLastError() != cudaSuccess) return refused(PS_ERR_CUDA, ws, s);
  // With the top-k lists, as many vocabulary ranges as the workspace holds (up to 16): shorter
  // ranges keep the CTAs of a band closer together along W (16 ranges measured 4% faster than
  // the 11 the forward's chooser picks at 7B). Without them, the forward's per-tile schedule.
  int splits, rc;
  if (topk > 0) {
    const int per_range = proxy_topk_lists_bf16(N, d, S), ranges = S / per_range;
    splits = ranges * per_range;
    rc = proxy_topk_gemm_bf16(N, d, V, Hrows, W, tok, part, tpart, ztok, ranges, per_range, status, s);
  } else {
    splits = choose_fwd_splits_bf16(N, d, V, num_sms_current(), S);
    rc = proxy_gemm_bf16(N, d, V, Hrows, W, tok, part, ztok, splits, status, s);
  }
  if (rc != PS_OK) return rc;
  return launch_after(proxy_finalize_kernel, dim3(static_cast<unsigned>((N + kProxyRows - 1) / kProxyRows)), 16 * kProxyRows,
                      0, s, 1, 1, true, N, V, splits, part, ztok, hn, tok, gamma, logp, topk, tpart, top_idx, top_prob,
                      status) == cudaSuccess
             ? PS_OK
             : PS_ERR_CUDA;
}

size_t ps_reward_uncertainty_workspace_size(int P, int K) {
  if (P < 1 || K < 1) return 0;
  return kWsHeader + al256(sizeof(int64_t) * static_cast<size_t>(P) * K);
}

int ps_binarize_rewards(int B, const float* R, uint64_t seed, uint64_t step, int64_t traj_base, float* y,
                        ps_stream_t stream) {
  NvtxRange nvtx_range("ps_binarize_rewards");
  if (B < 1 || traj_base < 0 || !R || !y) return PS_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  binarize_rewards_kernel<<<(B + 255) / 256, 256, 0, s>>>(B, R, seed, step, traj_base, y);
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

int ps_reward_uncertainty(int P, int K, int T_max, const int32_t* L, const float* R, int topk,
                          const int32_t* top_idx, const float* top_prob, float* u, void* ws, size_t ws_bytes,
                          ps_stream_t stream) {
  NvtxRange nvtx_range("ps_reward_uncertainty");
  if (P < 1 || K < 1 || K > 64 || T_max < 1 || topk < 1 || topk > 16) return PS_ERR_INVALID_ARG;
  if (!L || !R || !top_idx || !top_prob || !u) return PS_ERR_INVALID_ARG;
  if (ws == nullptr || (reinterpret_cast<uintptr_t>(ws) & 255) ||
      ws_bytes < ps_reward_uncertainty_workspace_size(P, K))
    return PS_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int64_t* off = reinterpret_cast<int64_t*>(static_cast<uint8_t*>(ws) + kWsHeader);
  group_offsets_kernel<<<1, 32, 0, s>>>(P * K, L, off, static_cast<uint32_t*>(ws));
  if (cudaGetLastError() != cudaSuccess) return refused(PS_ERR_CUDA, ws, s);
  const size_t smem = (sizeof(int32_t) + sizeof(double)) * kUncWarps * unc_entries(K, topk);
  if (cudaFuncSetAttribute(uncertainty_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(smem)) != cudaSuccess)
    return PS_ERR_CUDA;
  const int64_t tasks = static_cast<int64_t>(P) * T_max;
  return launch_after(uncertainty_kernel, dim3(static_cast<unsigned>((tasks + kUncWarps - 1) / kUncWarps)), kUncWarps * 32,
                      smem, s, 1, 1, true, P, K, T_max, L, R, topk, top_idx, top_prob, off, u) == cudaSuccess
             ? PS_OK
             : PS_ERR_CUDA;
}

static DesignWs design_ws(void* ws, int P, int T_max) {
  uint8_t* b = static_cast<uint8_t*>(ws) + kWsHeader;
  const size_t pt = static_cast<size_t>(P) * T_max;
  DesignWs d;
  d.w = reinterpret_cast<double*>(b);
  b += al256(sizeof(double) * pt);
  d.xi = reinterpret_cast<double*>(b);
  b += al256(sizeof(double) * pt);
  d.bW = reinterpret_cast<double*>(b);
  b += al256(sizeof(double) * pt * kCapLanes);
  d.bs = reinterpret_cast<double*>(b);
  b += al256(sizeof(double) * pt * kCapLanes);
  d.bn = reinterpret_cast<int32_t*>(b);
  return d;
}

size_t ps_design_cutoffs_workspace_size(int P, int K, int T_max) {
  if (P < 1 || K < 1 || T_max < 1) return 0;
  const size_t pt = static_cast<size_t>(P) * T_max;
  return kWsHeader + al256(sizeof(double) * pt) * 2 + al256(sizeof(double) * pt * kCapLanes) * 2 +
         al256(sizeof(int32_t) * pt * kCapLanes);
}

int ps_design_cutoffs(int P, int K, int T_max, const int32_t* L, const float* gamma_full, const float* u,
                      double budget, int strategy, double param, uint64_t* q, double* xi, void* ws, size_t ws_bytes,
                      ps_stream_t stream) {
  NvtxRange nvtx_range("ps_design_cutoffs");
  if (P < 1 || K < 1 || T_max < 1 || T_max > (1 << 24) || !L || !q) return PS_ERR_INVALID_ARG;
  if (static_cast<int64_t>(P) * K > INT32_MAX) return PS_ERR_INVALID_ARG;
  if (strategy < PS_DESIGN_OPTIMIZED || strategy > PS_DESIGN_FIXED) return PS_ERR_INVALID_ARG;
  const bool uses_gamma = strategy == PS_DESIGN_OPTIMIZED || strategy == PS_DESIGN_HEURISTIC;
  if (uses_gamma && !gamma_full) return PS_ERR_INVALID_ARG;
  if ((uses_gamma || strategy == PS_DESIGN_TIME_PRIOR) && !(budget > 0.0)) return PS_ERR_INVALID_ARG;
  if (strategy == PS_DESIGN_FIXED && !(param >= 1.0)) return PS_ERR_INVALID_ARG;
  if (ws == nullptr || (reinterpret_cast<uintptr_t>(ws) & 255) ||
      ws_bytes < ps_design_cutoffs_workspace_size(P, K, T_max))
    return PS_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(ws, 0, kWsHeader, s) != cudaSuccess) return PS_ERR_CUDA;
  const DesignWs d = design_ws(ws, P, T_max);
  uint32_t* status = static_cast<uint32_t*>(ws);
  const float* gamma = uses_gamma ? gamma_full : nullptr;
  if (uses_gamma && T_max > kWeightSteps) {
    const dim3 grid(static_cast<unsigned>(P), static_cast<unsigned>((T_max + kWeightSteps - 1) / kWeightSteps));
    design_weights_kernel<<<grid, kDesignThreads, 0, s>>>(K, T_max, L, gamma, u, d, status);
    if (cudaGetLastError() != cudaSuccess) return PS_ERR_CUDA;
    gamma = nullptr;
  }
  if (strategy == PS_DESIGN_OPTIMIZED) {
    if (cudaFuncSetAttribute(design_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kDesignDynSmem)) != cudaSuccess)
      return PS_ERR_CUDA;
    design_kernel<true><<<P, kDesignThreads, kDesignDynSmem, s>>>(K, T_max, L, gamma, u, budget, strategy, param, q, xi, d,
                                                                  status);
  } else {
    design_kernel<false><<<P, kDesignThreads, 0, s>>>(K, T_max, L, gamma, u, budget, strategy, param, q, xi, d, status);
  }
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

}  // extern "C"
