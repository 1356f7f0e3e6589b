// The compact-pattern fitter (Sec. 3.2 "Fitting", Eq. "fit-objective"; Algorithm 1's fitting loop; appendix
// "Selection, fitting, and installation" and "Compact fitting and storage").
//
//   target     P = rows of the mean attention map, causal entries floored at 1e-9, each row scaled to sum one
//   marginals  eta_abs(j) = sum_{i>=j} P(i,j),  eta_rel(d) = sum_{i-j=d} P(i,j),  and sum_{ij} P log P
//   Fit        alpha = 0, rho(d) = log max(eta_rel(d)/(T-d), 1e-9); J Adam steps on
//              L = (1/T)[sum_i log Z(i) - eta_abs.alpha - eta_rel.rho],  whose gradient is
//              (fitted marginal - target marginal)/T
//   accept     kappa = mean row KL(P || P^) = L + (1/T) sum P log P   (rows of P sum to one)
//
// Nothing of size T x T is formed after the target has been read once.  Beyond 128 positions the Adam steps run in
// saf_fit_fft.cu, where the three sums of a step are fp64 transforms; the kernel here serves the shortest sequences and goes
// on with the heads that leave the transforms' bounds.  A thread-block cluster per head runs all Adam steps in one launch,
// exchanging vectors of length T through distributed shared memory (normalisers) and L2 (parameters), with two cluster barriers
// per step:
//   pass A   rows:      Z(i) = sum_{d<=i} R(d) A(i-d),  W(i) = 1 / Z(i)
//   pass B   marginals: c(j) = A(j) sum_d R(d) W(j+d)  and  g(d) = R(d) sum_j A(j) W(j+d),
//            followed in the same thread by the Adam update of alpha(j) / rho(d) (fp64 state)
// with A = exp(alpha), R = exp(rho) taken once per parameter and step: the pattern's factorisation turns the three sums
// into causal convolutions / correlations, one fp32 multiply-add per causal pair and sum instead of an exponential.
// All terms are positive, so the sums keep the relative accuracy of their terms.  The plain products cannot leave
// fp32's range while every parameter and normaliser is inside the bounds below; a head that leaves them goes on in the
// log form (one exp2 per pair, referred to the previous step's normaliser), in the same kernel.
#include <cuda_runtime.h>
#include <cstdint>
#include <cmath>
#include <algorithm>
#include "saf_internal.h"

namespace saf {

namespace {

constexpr double LOG2E_D = 1.4426950408889634074;
constexpr double LN2_D = 0.6931471805599453094;
__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------ target marginals
// One CTA of NT threads walks rows blockIdx.x, blockIdx.x + gridDim.x, ... of head blockIdx.y.  Thread t owns the
// columns t, t + NT, ...: their column sums stay in registers over all rows of the CTA; the diagonal sums live in
// shared memory (for a given row every thread touches different distances, rows are separated by the CTA barrier of
// the row-sum reduction).  256 threads with up to 32 columns each measured fastest (loading the next row ahead of
// the reduction costs registers, hence resident CTAs, and measured slower).
// Row pieces specialised on the number KK of column chunks that reach the diagonal, so that the chunks above it
// cost nothing and the loads of a row still issue back to back.
template <int NT, int KK>
__device__ __forceinline__ void marg_load(const float* __restrict__ r, int row, int tid, float floor_v, float* dst) {
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    const int j = tid + k * NT;
    dst[k] = (j <= row) ? fmaxf(__ldg(r + j), floor_v) : 0.0f;
  }
}
template <int KK>
__device__ __forceinline__ float marg_sum(const float* cur) {
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < KK; ++k) s += cur[k];
  return s;
}
template <int NT, int KK>
__device__ __forceinline__ void marg_consume(const float* cur, float inv, float* col, float* dg, float& ent, int i,
                                             int tid) {
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    if (tid + k * NT <= i) {
      const float p = cur[k] * inv;
      col[k] += p;
      dg[-k * NT] += p;
      ent = fmaf(p, __log2f(p), ent);
    }
  }
}
// (quarters of the NCH chunks: case q serves rows whose last chunk index is below (q+1) NCH/4; one case per chunk
// count measured slower: more registers, fewer resident CTAs)
#define SAF_MARG_DISPATCH(q, CALL)                         \
  switch (q) {                                             \
    case 0: { constexpr int KK = G; CALL; } break;         \
    case 1: { constexpr int KK = 2 * G; CALL; } break;     \
    case 2: { constexpr int KK = 3 * G; CALL; } break;     \
    default: { constexpr int KK = NCH; CALL; } break;      \
  }

template <int NT, int NCH>
__global__ void __launch_bounds__(NT)
saf_fit_marginals_kernel(const float* __restrict__ Abar, float floor_v, double* __restrict__ eta_abs,
                         double* __restrict__ eta_rel, double* __restrict__ plogp, int T) {
  extern __shared__ float sm_f[];
  float* diag = sm_f;                          // [T]
  constexpr int NW = NT / 32;
  constexpr int G = (NCH >= 4) ? NCH / 4 : NCH;
  __shared__ float red[2][NW];
  __shared__ double redd[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int h = blockIdx.y;
  const float* A = Abar + static_cast<size_t>(h) * T * T;
  for (int d = tid; d < T; d += NT) diag[d] = 0.0f;
  float col[NCH];
#pragma unroll
  for (int k = 0; k < NCH; ++k) col[k] = 0.0f;
  float ent = 0.0f;                            // sum p log2 p of this thread (scaled to nats at the end)
  double ent_d = 0.0;
  float cur[NCH];
  int i = blockIdx.x;
  if (i < T) {
    SAF_MARG_DISPATCH((i / NT) / G, (marg_load<NT, KK>(A + static_cast<size_t>(i) * T, i, tid, floor_v, cur)));
  }
  __syncthreads();
  int par = 0, nrow = 0;
  for (; i < T; i += gridDim.x, par ^= 1, ++nrow) {
    const int q = (i / NT) / G;
    float s = 0.0f;
    SAF_MARG_DISPATCH(q, (s = marg_sum<KK>(cur)));
    s = warp_sum(s);
    if (lane == 0) red[par][warp] = s;
    __syncthreads();                           // also: the previous row's diagonal updates are complete
    float tot = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) tot += red[par][w];
    const float inv = 1.0f / tot;
    float* dg = diag + (i - tid);
    SAF_MARG_DISPATCH(q, (marg_consume<NT, KK>(cur, inv, col, dg, ent, i, tid)));
    if ((nrow & 63) == 63) {                   // keep the fp32 partial short
      ent_d += static_cast<double>(ent);
      ent = 0.0f;
    }
    const int inext = i + gridDim.x;
    if (inext < T) {
      SAF_MARG_DISPATCH((inext / NT) / G, (marg_load<NT, KK>(A + static_cast<size_t>(inext) * T, inext, tid, floor_v, cur)));
    }
  }
  ent_d += static_cast<double>(ent);
  __syncthreads();
  double* ea = eta_abs + static_cast<size_t>(h) * T;
  double* er = eta_rel + static_cast<size_t>(h) * T;
#pragma unroll
  for (int k = 0; k < NCH; ++k) {
    const int j = tid + k * NT;
    if (j < T && col[k] != 0.0f) atomicAdd(ea + j, static_cast<double>(col[k]));
  }
  for (int d = tid; d < T; d += NT)
    if (diag[d] != 0.0f) atomicAdd(er + d, static_cast<double>(diag[d]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ent_d += __shfl_xor_sync(0xffffffffu, ent_d, o);
  if (lane == 0) redd[warp] = ent_d;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < NW; ++w) t += redd[w];
    atomicAdd(plogp + h, t * LN2_D);
  }
}
#undef SAF_MARG_DISPATCH

// ------------------------------------------------------------------------------------------------ Fit
constexpr int FX = 256;            // x values of a block: 8 consecutive ones per lane
constexpr int FPIECE = 64;         // terms of a chain of fp32 additions
constexpr int FPAD = 288;          // floats kept neutral in front of A and behind A, R and W
// Bounds (log2) inside which the product form is used: every factor and product of two stays within 2^+-120, sums of
// 16384 of them below 2^127, so nothing overflows and nothing is flushed.
constexpr float A_LO = -50.0f, A_HI = 50.0f, R_LO = -70.0f, R_HI = 50.0f;
constexpr float Z_LO = 8.6736174e-19f, Z_HI = 1.1258999e15f;      // 2^-60, 2^50

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 2^x of an fp64 exponent, rounded to fp32 once.  (The same A(j) and R(d) enter a whole row, column or diagonal of terms,
// so that their own rounding does not average out: with ex2.approx of the fraction the loss was off by 1e-8.)
__device__ __forceinline__ float exp2_f32(double x) { return static_cast<float>(exp2(x)); }

// Layout of a vector in shared memory.  A lane reads 8 consecutive values plus a sliding window in 16-byte pieces, so
// lanes are 32 bytes apart: PADDED inserts 16 bytes after every 32, which makes those reads conflict-free (lanes 48
// bytes apart) and keeps the pieces at constant offsets.  Indices of a piece: a multiple of 4.
template <bool PADDED>
__device__ __forceinline__ int fit_phys(int i) { return PADDED ? i + ((i >> 3) << 2) : i; }
template <bool PADDED>
__device__ __forceinline__ constexpr int fit_off(int d) { return PADDED ? d + (d >= 0 ? (d >> 3) : -((7 - d) >> 3)) * 4 : d; }

__device__ __forceinline__ void ld4(const float* p, float* v) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

// acc[k] += sum over y in [y0, y1) of u(y) * w(x + k -/+ y) for this lane's x .. x+7 (MODE 0: minus, with one u; MODE 1:
// plus, with two u and two accumulators).  y0, y1: multiples of 16; xl = the lane's x (a multiple of 8).  Per 16 values
// of y: 4 window pieces and 4 (8) uniform pieces for 128 (256) multiply-adds.  LOG: the vectors hold logarithms and a
// term is 2^(u + w + c).
template <int MODE, bool PADDED, bool LOG>
__device__ __forceinline__ void fit_accumulate(const float* __restrict__ u0, const float* __restrict__ u1,
                                               const float* __restrict__ w, int xl, int y0, int y1, const float* c0,
                                               const float* c1, float* acc0, float* acc1) {
  float win[24];
  const float* wp = w + fit_phys<PADDED>(MODE == 0 ? xl - y0 : xl + y0);
  if (y0 < y1) {
    // the two pieces that consecutive steps share
    ld4(wp + fit_off<PADDED>(0), MODE == 0 ? win + 16 : win);
    ld4(wp + fit_off<PADDED>(4), MODE == 0 ? win + 20 : win + 4);
  }
  for (int ye = y0; ye < y1;) {
    // (pieces of FPIECE values of y are summed on their own, so that no chain of fp32 additions gets long)
    const int yb = ye;
    ye = min(y1, yb + FPIECE);
    float s0[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, s1[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
    for (int y = yb; y < ye; y += 16) {
      if (MODE == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ld4(wp + fit_off<PADDED>(-16 + 4 * q), win + 4 * q);
      } else {
#pragma unroll
        for (int q = 2; q < 6; ++q) ld4(wp + fit_off<PADDED>(4 * q), win + 4 * q);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a[4], b[4];
        ld4(u0 + y + 4 * q, a);
        if (MODE == 1) ld4(u1 + fit_phys<PADDED>(y) + fit_off<PADDED>(4 * q), b);
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float wv = win[MODE == 0 ? 16 + k - (4 * q + t) : k + 4 * q + t];
            if (LOG) {
              s0[k] += ex2f((a[t] + c0[k]) + wv);
              if (MODE == 1) s1[k] += ex2f((b[t] + c1[k]) + wv);
            } else {
              s0[k] = fmaf(a[t], wv, s0[k]);
              if (MODE == 1) s1[k] = fmaf(b[t], wv, s1[k]);
            }
          }
      }
      if (MODE == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) win[16 + k] = win[k];
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) win[k] = win[16 + k];
      }
      wp += (MODE == 0 ? -1 : 1) * (PADDED ? 24 : 16);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      acc0[k] += s0[k];
      if (MODE == 1) acc1[k] += s1[k];
    }
  }
}

// The x blocks of 256 that a CTA owns in one pass and the segments its NW warps work on.  The 16-wide y chunks of the
// CTA's blocks are numbered through (in rounds of RB blocks) and split evenly over the warps; warp w's part of block b
// goes to slot w + b of the partial sums (both only ever move up, so no two segments meet in a slot).
struct FitPlan {
  int count;                                     // blocks
  int total[64];                                 // chunks of round r
  short xb[64], first[64], n[64];                // block number, first chunk within its round, chunks
  signed char lo[64], hi[64];                    // warps whose segments touch the block
};

// One cluster = one head.  A head's x blocks go to the cluster's CTAs in snake order by descending work.  Bound: fp32
// multiply-adds (128 per clock and SM), 1.5 T^2 per head and step.  Measured (36 heads, T = 4096, 400 steps): 23.4 ms =
// 58 us per step on 108 SMs, against 100.2 ms for one exponential per pair and sum in two launches per step; 57 % of those
// SMs' multiply-add peak over everything.  One head of 256 positions: 6.0 us per
// step (two cluster barriers, L2 round trips of the parameters, fp64 Adam).  Heads of more than 128 positions start in
// saf_fit_fft_kernel (13.6 us a step of the 36) and come here only from there, or where its state or clusters have no room.
template <int NW, bool PADDED, int RB>
__global__ void __launch_bounds__(NW * 32, 1)
saf_fit_kernel(FitState s, int steps, const double* __restrict__ plogp, float* __restrict__ alpha_out,
               float* __restrict__ rho_out, float* __restrict__ logZ_out, long long out_stride,
               double* __restrict__ loss_out, double* __restrict__ kl_out) {
  extern __shared__ float4 sm_f4[];
  constexpr int NT = NW * 32;
  // a parameter (set in pass B, read after its barrier) or a normaliser (pass A) of this head has left the bounds
  __shared__ int out_par, out_z;
  __shared__ double redd[NW], part_loss[16];
  __shared__ float redf[NW];
  __shared__ FitPlan plan[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = s.T;
  uint32_t cs, rank;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(cs));
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int h = blockIdx.x / cs;
  const size_t o = static_cast<size_t>(h) * T;
  const int Tr = (T + 15) & ~15;
  const int nA = fit_phys<PADDED>(FPAD + Tr + FPAD), nW = fit_phys<PADDED>(Tr + FPAD);
  float* Abase = reinterpret_cast<float*>(sm_f4);
  float* A = Abase + fit_phys<PADDED>(FPAD);     // A[-FPAD .. Tr+FPAD)
  float* W = Abase + nA;                         // W[0 .. Tr+FPAD)
  float* R = W + nW;                             // R[0 .. Tr+FPAD), unpadded
  float* part = R + Tr + FPAD;                   // [NW + RB][2][FX] partial sums
  const int nxb = (T + FX - 1) / FX;
  bool slow = false;
  // a head that the transform form has finished, or the step at which it handed it over (1: nothing done yet)
  const int t0 = s.resume ? s.resume[h] : 1;
  if (t0 < 0) return;
  const bool fresh = t0 <= 1;

  if (tid < 2) {                                 // plan[0]: pass A, plan[1]: pass B
    FitPlan& p = plan[tid];
    int cnt = 0;
    for (int k = 0; k < nxb; ++k) {              // k: blocks in descending order of work
      const int r = k / static_cast<int>(cs), i = k % static_cast<int>(cs);
      if (((r & 1) ? static_cast<int>(cs) - 1 - i : i) != static_cast<int>(rank)) continue;
      const int xb = tid == 0 ? nxb - 1 - k : k;
      p.xb[cnt] = static_cast<short>(xb);
      p.n[cnt] = static_cast<short>(((tid == 0 ? min(T, (xb + 1) * FX) : T - xb * FX) + 15) >> 4);
      ++cnt;
    }
    p.count = cnt;
    for (int i0 = 0, r = 0; i0 < cnt; i0 += RB, ++r) {
      const int i1 = min(cnt, i0 + RB);
      int tot = 0;
      for (int i = i0; i < i1; ++i) {
        p.first[i] = static_cast<short>(tot);
        tot += p.n[i];
      }
      p.total[r] = tot;
      for (int i = i0; i < i1; ++i) {
        int lo = 0, hi = NW - 1;
        while ((lo + 1) * tot / NW <= p.first[i]) ++lo;
        while (hi * tot / NW >= p.first[i] + p.n[i]) --hi;
        p.lo[i] = static_cast<signed char>(lo);
        p.hi[i] = static_cast<signed char>(hi);
      }
    }
  }
  // neutral elements around the vectors
  auto fill_pads = [&](float v) {
    for (int i = tid; i < FPAD; i += NT) A[fit_phys<PADDED>(i - FPAD)] = v;
    for (int i = T + tid; i < Tr + FPAD; i += NT) {
      A[fit_phys<PADDED>(i)] = v;
      W[fit_phys<PADDED>(i)] = v;
      R[i] = v;
    }
  };
  // to the log form: parameters from their fp64 values, normalisers as they stand (any nearby reference will do)
  auto go_slow = [&]() {
    slow = true;
    fill_pads(-INFINITY);
    for (int i = tid; i < T; i += NT) {
      A[fit_phys<PADDED>(i)] = static_cast<float>(__ldcg(s.alpha + o + i) * LOG2E_D);
      R[i] = static_cast<float>(__ldcg(s.rho + o + i) * LOG2E_D);
      W[fit_phys<PADDED>(i)] = __log2f(W[fit_phys<PADDED>(i)]);
    }
    cluster_sync_all();                          // nobody's next normalisers may arrive before this is done
  };
  auto raise_flag = [&](int* flag) {
    const uint32_t a = smem_addr(flag);
    for (uint32_t r = 0; r < cs; ++r)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(a, r)), "r"(1) : "memory");
  };

  // ---- start: alpha = 0, rho(d) = log max(eta_rel(d)/(T-d), 1e-9), Adam moments zero, and a first reference for the
  // normalisers: the upper bound max rho (alpha = 0)
  if (tid == 0) out_par = out_z = 0;
  float mx = -INFINITY;
  bool bad = false;
  for (int d = tid; d < T; d += NT) {
    const double r = fresh ? log(fmax(s.eta_rel[o + d] / static_cast<double>(T - d), 1e-9)) : s.rho[o + d];
    const double a = fresh ? 0.0 : s.alpha[o + d];
    const float r2 = static_cast<float>(r * LOG2E_D), a2 = static_cast<float>(a * LOG2E_D);
    mx = fmaxf(mx, r2);
    if (!(r2 >= R_LO && r2 <= R_HI && a2 >= A_LO && a2 <= A_HI)) bad = true;
    if (!fresh && !(fabsf(s.wref[o + d]) <= A_HI)) bad = true;
    R[d] = exp2_f32(r * LOG2E_D);
    A[fit_phys<PADDED>(d)] = exp2_f32(a * LOG2E_D);
    if (!fresh) continue;
    // (each block's state is written and later read by its owner in pass B only, except for the fp64 parameters)
    const int k = d / FX, kr = k / static_cast<int>(cs), ki = k % static_cast<int>(cs);
    if (((kr & 1) ? static_cast<int>(cs) - 1 - ki : ki) == static_cast<int>(rank)) {
      s.rho[o + d] = r;
      s.alpha[o + d] = 0.0;
      s.m_a[o + d] = 0.0; s.v_a[o + d] = 0.0; s.m_r[o + d] = 0.0; s.v_r[o + d] = 0.0;
    }
  }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, k));
  if (lane == 0) redf[warp] = mx;
  bad = __syncthreads_or(bad);
  mx = redf[0];
#pragma unroll
  for (int w = 1; w < NW; ++w) mx = fmaxf(mx, redf[w]);
  fill_pads(0.0f);
  auto wstart = [&](int i) { return fresh ? -mx : s.wref[o + i]; };
  for (int i = tid; i < T; i += NT) W[fit_phys<PADDED>(i)] = bad ? wstart(i) : ex2f(wstart(i));
  cluster_sync_all();
  if (bad) {                                     // (the same decision in every CTA of the cluster)
    go_slow();
    for (int i = tid; i < T; i += NT) W[fit_phys<PADDED>(i)] = wstart(i);
    cluster_sync_all();
  }

  double acc = 0.0;                              // this thread's part of T * loss
  // pass A over this CTA's blocks; `last`: the normalisers of the final parameters (results are written)
  auto pass_a = [&](bool last) {
    const FitPlan& p = plan[0];
    for (int i0 = 0, rd = 0; i0 < p.count; i0 += RB, ++rd) {
      const int nb = min(RB, p.count - i0), tot = p.total[rd];
      const int k0 = warp * tot / NW, k1 = (warp + 1) * tot / NW;
      if (i0 > 0) __syncthreads();
      for (int b = 0; b < nb; ++b) {
        const int first = p.first[i0 + b];
        const int y0 = (max(k0, first) - first) << 4, y1 = (min(k1, first + p.n[i0 + b]) - first) << 4;
        if (warp < p.lo[i0 + b] || warp > p.hi[i0 + b]) continue;   // (a warp without chunks in between adds zeros)
        const int xl = p.xb[i0 + b] * FX + 8 * lane;
        float a8[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (!slow) {
          fit_accumulate<0, PADDED, false>(R, nullptr, A, xl, y0, y1, nullptr, nullptr, a8, nullptr);
        } else {
          float c8[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) c8[q] = xl + q < T ? W[fit_phys<PADDED>(xl + q)] : -INFINITY;
          fit_accumulate<0, PADDED, true>(R, nullptr, A, xl, y0, y1, c8, nullptr, a8, nullptr);
        }
        float4* dst = reinterpret_cast<float4*>(part + (warp + b) * 2 * FX + 8 * lane);
        dst[0] = make_float4(a8[0], a8[1], a8[2], a8[3]);
        dst[1] = make_float4(a8[4], a8[5], a8[6], a8[7]);
      }
      __syncthreads();
      for (int q = tid; q < nb * FX; q += NT) {
        const int b = q / FX, i = i0 + b, x = p.xb[i] * FX + (q & (FX - 1));
        if (x >= T) continue;
        double S = 0.0;
#pragma unroll 4
        for (int w = p.lo[i]; w <= p.hi[i]; ++w) S += part[(w + b) * 2 * FX + (q & (FX - 1))];
        float* slot = W + fit_phys<PADDED>(x);
        float out;
        double lz;
        bool in = true;
        if (slow) {
          out = *slot - __log2f(static_cast<float>(S));
          lz = -static_cast<double>(out) * LN2_D;
        } else {
          in = S >= Z_LO && S <= Z_HI;
          out = static_cast<float>(1.0 / S);
          lz = last ? log(S) : 0.0;
        }
        if (in) {
          const uint32_t a = smem_addr(slot);
          for (uint32_t r = 0; r < cs; ++r) st_cluster_f32(cluster_addr(a, r), out);
        } else {
          raise_flag(&out_z);
        }
        if (last) {
          logZ_out[static_cast<size_t>(h) * out_stride + x] = static_cast<float>(lz);
          if (slow || in) acc += lz;
        }
      }
    }
    cluster_sync_all();
  };

  double p1 = 1.0, p2 = 1.0;
  for (int t = 1; t < t0; ++t) {
    p1 *= 0.9;
    p2 *= 0.999;
  }
  for (int t = max(t0, 1); t <= steps + 1; ++t) {
    const bool last = t == steps + 1;
    if (t > max(t0, 1)) {
      // the parameters of this step, from the owners of their blocks
      if (!slow && out_par) {
        go_slow();
      } else {
        for (int i = tid; i < T; i += NT) {
          A[fit_phys<PADDED>(i)] = __ldcg(s.a2 + o + i);
          R[i] = __ldcg(s.r2 + o + i);
        }
        __syncthreads();
      }
    }
    pass_a(last);
    if (!slow && out_z) {
      acc = 0.0;
      go_slow();
      pass_a(last);
    }
    if (last) break;
    p1 *= 0.9;
    p2 *= 0.999;
    const double ib1 = 1.0 / (1.0 - p1), ib2 = 1.0 / (1.0 - p2), iT = 1.0 / static_cast<double>(T);
    const FitPlan& p = plan[1];
    for (int i0 = 0, rd = 0; i0 < p.count; i0 += RB, ++rd) {
      const int nb = min(RB, p.count - i0), tot = p.total[rd];
      const int k0 = warp * tot / NW, k1 = (warp + 1) * tot / NW;
      if (i0 > 0) __syncthreads();
      for (int b = 0; b < nb; ++b) {
        const int first = p.first[i0 + b];
        const int y0 = (max(k0, first) - first) << 4, y1 = (min(k1, first + p.n[i0 + b]) - first) << 4;
        if (warp < p.lo[i0 + b] || warp > p.hi[i0 + b]) continue;   // (a warp without chunks in between adds zeros)
        const int xl = p.xb[i0 + b] * FX + 8 * lane;
        float c8[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, g8[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (!slow) {
          fit_accumulate<1, PADDED, false>(R, A, W, xl, y0, y1, nullptr, nullptr, c8, g8);
        } else {
          float ca[8], cr[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            ca[q] = A[fit_phys<PADDED>(xl + q)];
            cr[q] = R[xl + q];
          }
          fit_accumulate<1, PADDED, true>(R, A, W, xl, y0, y1, ca, cr, c8, g8);
        }
        float4* dst = reinterpret_cast<float4*>(part + (warp + b) * 2 * FX + 8 * lane);
        dst[0] = make_float4(c8[0], c8[1], c8[2], c8[3]);
        dst[1] = make_float4(c8[4], c8[5], c8[6], c8[7]);
        dst[FX / 4] = make_float4(g8[0], g8[1], g8[2], g8[3]);
        dst[FX / 4 + 1] = make_float4(g8[4], g8[5], g8[6], g8[7]);
      }
      __syncthreads();
      // one Adam step in fp64 on Eq. "fit-objective": gradient = (fitted marginal - target marginal) / T
#pragma unroll 2
      for (int q = tid; q < nb * 2 * FX; q += NT) {
        const int b = q / (2 * FX), i = i0 + b, x = p.xb[i] * FX + (q & (FX - 1));
        const bool is_rho = (q & FX) != 0;
        if (x >= T) continue;
        double* par = (is_rho ? s.rho : s.alpha) + o + x;
        double* mm = (is_rho ? s.m_r : s.m_a) + o + x;
        double* vv = (is_rho ? s.v_r : s.v_a) + o + x;
        const double eta = (is_rho ? s.eta_rel : s.eta_abs)[o + x];
        const double m0 = *mm, v0 = *vv, x_old = *par;
        double S = 0.0;
#pragma unroll 4
        for (int w = p.lo[i]; w <= p.hi[i]; ++w) S += part[(w + b) * 2 * FX + (q & (2 * FX - 1))];
        if (!slow) S *= is_rho ? R[x] : A[fit_phys<PADDED>(x)];
        const double g = (S - eta) * iT;
        const double m = 0.9 * m0 + 0.1 * g;
        const double v = 0.999 * v0 + 0.001 * g * g;
        *mm = m;
        *vv = v;
        const double pnew = x_old - s.lr * (m * ib1) / (sqrt(v * ib2) + 1e-8);
        *par = pnew;
        const double e = pnew * LOG2E_D;
        (is_rho ? s.r2 : s.a2)[o + x] = slow ? static_cast<float>(e) : exp2_f32(e);
        if (!slow && !(e >= (is_rho ? R_LO : A_LO) && e <= (is_rho ? R_HI : A_HI))) raise_flag(&out_par);
      }
    }
    cluster_sync_all();
  }

  // ---- results: L = (1/T)[sum_i log Z(i) - eta_abs.alpha - eta_rel.rho], kappa = L + (1/T) sum P log P
  const size_t oo = static_cast<size_t>(h) * static_cast<size_t>(out_stride);
  for (int k = static_cast<int>(rank) * NT + tid; k < T; k += static_cast<int>(cs) * NT) {
    const double a = __ldcg(s.alpha + o + k), r = __ldcg(s.rho + o + k);
    // L at the parameters as the sums saw them, to fp32: first-order in that rounding, log Z and the linear terms cancel
    const float a32 = A[fit_phys<PADDED>(k)], r32 = R[k];
    acc -= s.eta_abs[o + k] * (slow ? a32 * LN2_D : log(static_cast<double>(a32))) +
           s.eta_rel[o + k] * (slow ? r32 * LN2_D : log(static_cast<double>(r32)));
    alpha_out[oo + k] = static_cast<float>(a);
    rho_out[oo + k] = static_cast<float>(r);
  }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, k);
  if (lane == 0) redd[warp] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < NW; ++w) t += redd[w];
    st_cluster_f64(cluster_addr(smem_addr(part_loss + rank), 0), t);
  }
  cluster_sync_all();
  if (rank == 0 && tid == 0) {
    double t = 0.0;
    for (uint32_t r = 0; r < cs; ++r) t += part_loss[r];
    const double loss = t / static_cast<double>(T);
    if (loss_out) loss_out[h] = loss;
    if (kl_out) kl_out[h] = loss + plogp[h] / static_cast<double>(T);
  }
}

}  // namespace

// ------------------------------------------------------------------------------------------------ launchers
int fit_max_T() { return 16384; }

// Up to 128 positions the direct sums stay: the two are within 5 % of one another for the head counts of a model (us a step, direct /
// transforms: one head of 64 5.4 / 5.3, 100 5.1 / 5.3, 128 5.6 / 5.4, 36 of 100 5.2 / 5.3; 150 of 100, more than there are SMs,
// 10.1 / 5.4), beyond it the transforms are faster (160 5.8 / 5.3, 256 6.2 / 5.4, 1024 9.1 / 7.5, 4096 22.8 / 10.1).
bool fit_has_transforms(int T) { return T > 128; }

cudaError_t launch_fit_marginals(const float* Abar, float floor_v, double* eta_abs, double* eta_rel, double* plogp,
                                 int Hf, int T, int num_sms, cudaStream_t st) {
  // CTAs per head: one resident wave over all heads, but at least 32 rows each so that the final flush
  // (2T atomics per CTA) stays small beside the rows read
  const size_t smem = static_cast<size_t>(T) * sizeof(float);
#define SAF_MARG(NT, N)                                                                                          \
  do {                                                                                                           \
    auto kern = saf_fit_marginals_kernel<NT, N>;                                                                 \
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,                      \
                                         static_cast<int>(smem));                                                \
    if (e != cudaSuccess) return e;                                                                              \
    int occ = 1;                                                                                                 \
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, smem);                                     \
    if (e != cudaSuccess) return e;                                                                              \
    int nb = (std::max(occ, 1) * num_sms) / Hf;             /* one resident wave over all heads */               \
    nb = std::max(1, std::min(nb, (T + 31) / 32));                                                               \
    kern<<<dim3(nb, Hf), NT, smem, st>>>(Abar, floor_v, eta_abs, eta_rel, plogp, T);                             \
  } while (0)
  if (T <= 128 * 2) SAF_MARG(128, 2);
  else if (T <= 256 * 4) SAF_MARG(256, 4);
  else if (T <= 256 * 8) SAF_MARG(256, 8);
  else if (T <= 256 * 16) SAF_MARG(256, 16);
  else if (T <= 256 * 32) SAF_MARG(256, 32);
  else if (T <= 512 * 32) SAF_MARG(512, 32);
  else return cudaErrorInvalidValue;
#undef SAF_MARG
  return cudaGetLastError();
}

namespace {

template <int NW, bool PADDED, int RB>
size_t fit_smem(int T) {
  const size_t Tr = (T + 15) & ~15;
  auto ph = [](size_t i) { return PADDED ? i + ((i >> 3) << 2) : i; };
  return (ph(2 * FPAD + Tr) + ph(Tr + FPAD) + Tr + FPAD + 2 * (NW + RB) * FX) * sizeof(float);
}

template <int NW, bool PADDED, int RB, typename... Args>
cudaError_t launch_fit_clusters(const FitState& s, int Hf, cudaStream_t st, Args... args) {
  auto kern = saf_fit_kernel<NW, PADDED, RB>;
  const size_t smem = fit_smem<NW, PADDED, RB>(s.T);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(NW * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // Cluster size: the shortest of (waves of clusters) x (a head's multiply-adds over its CTAs + a fixed cost per step).
  // Clusters stay inside a GPC, so fewer than 148 / size fit at once (measured with one CTA per SM: 74 of two, 45 of
  // three, 33 of four, 26 of five, 22 of six, 15 of eight, 9 of ten, 7 of 12 to 16): 36 heads run faster on three CTAs each,
  // in one wave, than on four.  Sizes above the portable eight are for few heads and long sequences: one head of 8192
  // 44 us a step on 16 CTAs, 80 on 8 (51 with one exponential per pair on all SMs); of 16384 154 and 305.
  const int nxb = (s.T + FX - 1) / FX;
  double best = 0.0;
  int best_cs = 0;
  for (int cs = 1; cs <= std::min(16, nxb); ++cs) {
    attr[0].val.clusterDim.x = cs;
    cfg.gridDim = dim3(static_cast<unsigned>(Hf) * cs);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      continue;
    }
    const double waves = (Hf + n - 1) / n;
    const double cost = waves * (1.5 * s.T * static_cast<double>(s.T) / 128.0 / cs + 5000.0);
    if (best_cs == 0 || cost < best) {
      best = cost;
      best_cs = cs;
    }
  }
  if (best_cs == 0) return cudaErrorInvalidConfiguration;
  attr[0].val.clusterDim.x = best_cs;
  cfg.gridDim = dim3(static_cast<unsigned>(Hf) * best_cs);
  return cudaLaunchKernelEx(&cfg, kern, s, args...);
}

}  // namespace

cudaError_t launch_fit(FitState& s, int Hf, int steps, const double* plogp, float* alpha_out, float* rho_out,
                       float* logZ_out, long long out_stride, double* loss_out, double* kl_out, cudaStream_t st) {
  if (s.resume) {
    bool launched = false;
    const cudaError_t e = launch_fit_fft(s, Hf, steps, plogp, alpha_out, rho_out, logZ_out, out_stride, loss_out, kl_out, st, &launched);
    if (e != cudaSuccess) return e;
    if (!launched) s.resume = nullptr;
  }
  // up to 8192 positions the padded vectors fit beside the partial sums of 16 warps, up to 12288 beside those of 12; the
  // longest sequences keep them unpadded (two-way bank conflicts on the window reads)
  if (s.T <= 8192)
    return launch_fit_clusters<16, true, 16>(s, Hf, st, steps, plogp, alpha_out, rho_out, logZ_out, out_stride, loss_out, kl_out);
  if (s.T <= 12288)
    return launch_fit_clusters<12, true, 2>(s, Hf, st, steps, plogp, alpha_out, rho_out, logZ_out, out_stride, loss_out, kl_out);
  return launch_fit_clusters<12, false, 2>(s, Hf, st, steps, plogp, alpha_out, rho_out, logZ_out, out_stride, loss_out, kl_out);
}

}  // namespace saf
