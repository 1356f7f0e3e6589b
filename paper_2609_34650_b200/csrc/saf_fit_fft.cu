// The fitter's Adam steps with the three sums of a step as fp64 transforms (Sec. 3.2 "Fitting"; the paper's fitter, too,
// obtains its normalisers by FFT).  With A = exp(alpha), R = exp(rho), W = 1/Z, vectors zero beyond T:
//   Z(i) = sum_d R(d) A(i-d),   c(j) = sum_i R(i-j) W(i),   g(d) = sum_j A(j) W(j+d)
// are a causal convolution and two correlations.  A length-M transform (M a power of two >= T) of real vectors at the
// points z_k = exp(-2 pi i (k + 1/4) / M) gives them without zero padding to 2M: z_k^M = -i, so the part of a product
// that wraps around lands in the imaginary part (the "right-angle" convolution),
//   Re IDFT(A^ R^) = Z,   Re IDFT(conj(R^) W^) = c,   Re IDFT(conj(A^) W^) = g:
// six complex fp64 transforms of length M per step, about 5 M log2 M operations each, against 1.5 T^2 multiply-adds.
//
// One cluster of C CTAs per head, all steps in one launch.  M = C L; index n = n2 + L n1, frequency k = k1 + C k2.  CTA q
// owns the positions with n2 in [q L/C, (q+1) L/C) for every n1 (parameters, normalisers, Adam) and, as k1 = q, the
// frequencies k = q mod C: a transform is a C-point sum over n1 in the owner's registers, one exchange through distributed
// shared memory, and an L-point FFT inside a CTA (and the reverse for the inverses).  Four exchanges, each with a cluster
// barrier, per step:
//   1  A, R out -> A^, R^, their product, its inverse     2  back to the owners: Z, W
//   3  W out    -> W^, two products, two inverses         4  back to the owners: c, g, Adam
// The L-point FFT: a thread holds 8 points, radix-8 passes in place (decimation in frequency forward, in time backward, so
// that no reordering is needed), the last pass radix 2 or 4 where log2 L is no multiple of three.  After the first pass a
// sub-transform lies inside a warp.  16-byte pads behind every 8 points keep all passes free of bank conflicts.
//
// Bound: latency.  A few warps per scheduler work through chains of dependent fp64 operations (fp64 pipe 13 % busy on the SMs of
// one head, 24 % with 36), barriers and exchanges.  36 heads of 4096 positions, 400 steps: 13.6 us a step against 59.3 with the
// direct fp32 sums on 108 SMs; one head: 9.4 against 22.8.  Registers decide much of it: the 512-point kernel of eight-CTA
// clusters spilled 160 bytes a thread and thrashed L1 with them (with less L1 it lost another 12 %); with the owner twiddles in
// shared memory, the references of the normalisers written out and the peers' addresses computed where they are used, 24 bytes are
// left (36 x 4096: 6.29 -> 5.91 ms for the whole fit, 1 x 8192: 7.61 -> 6.59, 36 x 8192: 19.6 -> 17.8).  The larger ones have 128
// registers a thread and still spill: 68 bytes with 1024 points in clusters of four, 408 and 416 with 1024 and 2048 in
// clusters of eight (8193 positions and up).  Clusters of up to four keep all of the above in registers (with them moved out they
// measured 1-6 % slower).
//
// Accuracy.  An output's error is up to about 4.5 2^-53 of the 2-norms of its two factors, whatever its own size (measured, T =
// 4096).  The pattern does not change under alpha(j) -> alpha(j) - k j, rho(d) -> rho(d) - k d, Z(i) -> e^{-k i} Z(i), and
// Adam's trajectory drifts along this direction (|A||R| reached 2^27 min Z and |A||W| 2^29 min g after 400 steps of 4096
// positions), so every step uses the k that makes the last step's log Z level (2^19 and 2^12).  A head stays here while every
// Z is at least 2^-28 |A||R| and every marginal, or the target it is compared with, at least 2^-28 of A(j) |R||W| or R(d) |A||W|,
// so that no error exceeds 1.5e-7 of these (the direct fp32 sums: 1.4e-7 in the mean, 8e-7 at most); a head that leaves the
// bounds, or whose targets are not finite, is handed to saf_fit_kernel, which has no such restriction, at the step it has
// reached.  Its state before that step is still there: the steps write to two copies in turn.
#include <cuda_runtime.h>
#include <cstdint>
#include <cmath>
#include <algorithm>
#include "saf_fit_math.cuh"
#include "saf_internal.h"

namespace saf {

namespace {

using cd = double2;

constexpr double LN2_D = 0.6931471805599453094;
constexpr float GUARD = 3.7252903e-9f;          // 2^-28

// cos, sin of 2 pi m / 32
__host__ __device__ constexpr double cos32(int m) {
  m &= 31;
  if (m > 16) m = 32 - m;
  const int q = m <= 8 ? m : 16 - m;
  const double c = q == 0 ? 1.0 : q == 1 ? 0.98078528040323044912618 : q == 2 ? 0.92387953251128675612818
                 : q == 3 ? 0.83146961230254523707879 : q == 4 ? 0.70710678118654752440084
                 : q == 5 ? 0.55557023301960222474283 : q == 6 ? 0.38268343236508977172846
                 : q == 7 ? 0.19509032201612826784828 : 0.0;
  return m <= 8 ? c : -c;
}
__host__ __device__ constexpr double sin32(int m) { return cos32(m - 8); }

__device__ __forceinline__ cd cmul(cd a, cd b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ cd cmulc(cd a, cd b) {                      // a conj(b)
  return make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ cd cadd(cd a, cd b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ cd csub(cd a, cd b) { return make_double2(a.x - b.x, a.y - b.y); }

template <bool INV>
__device__ __forceinline__ cd rot90(cd a) {                            // times -i (INV: i)
  return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}
template <bool INV>
__device__ __forceinline__ cd rot45(cd a) {                            // times e^{-i pi/4} (INV: its conjugate)
  constexpr double h = cos32(4);
  return INV ? make_double2(h * (a.x - a.y), h * (a.x + a.y)) : make_double2(h * (a.x + a.y), h * (a.y - a.x));
}

__host__ __device__ constexpr int rev8(int k) { return (k & 1) << 2 | (k & 2) | k >> 2; }
// 8-point DFT in place; slot k holds residue rev8(k).  The inverse undoes it up to the factor 8.
__device__ __forceinline__ void bf8_fwd(cd* x) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const cd u = x[j];
    x[j] = cadd(u, x[j + 4]);
    x[j + 4] = csub(u, x[j + 4]);
  }
  x[5] = rot45<false>(x[5]);
  x[6] = rot90<false>(x[6]);
  x[7] = rot90<false>(rot45<false>(x[7]));
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
#pragma unroll
    for (int j = h; j < h + 2; ++j) {
      const cd u = x[j];
      x[j] = cadd(u, x[j + 2]);
      x[j + 2] = csub(u, x[j + 2]);
    }
    x[h + 3] = rot90<false>(x[h + 3]);
  }
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const cd u = x[j];
    x[j] = cadd(u, x[j + 1]);
    x[j + 1] = csub(u, x[j + 1]);
  }
}
__device__ __forceinline__ void bf8_inv(cd* x) {
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const cd u = x[j];
    x[j] = cadd(u, x[j + 1]);
    x[j + 1] = csub(u, x[j + 1]);
  }
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
    x[h + 3] = rot90<true>(x[h + 3]);
#pragma unroll
    for (int j = h; j < h + 2; ++j) {
      const cd u = x[j];
      x[j] = cadd(u, x[j + 2]);
      x[j + 2] = csub(u, x[j + 2]);
    }
  }
  x[5] = rot45<true>(x[5]);
  x[6] = rot90<true>(x[6]);
  x[7] = rot90<true>(rot45<true>(x[7]));
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const cd u = x[j];
    x[j] = cadd(u, x[j + 4]);
    x[j + 4] = csub(u, x[j + 4]);
  }
}
// the last pass over 8 consecutive points: radix 2 or 4
template <int RADIX, bool INV>
__device__ __forceinline__ void bf_last(cd* x) {
  if (RADIX == 4 && !INV) {
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
#pragma unroll
      for (int j = h; j < h + 2; ++j) {
        const cd u = x[j];
        x[j] = cadd(u, x[j + 2]);
        x[j + 2] = csub(u, x[j + 2]);
      }
      x[h + 3] = rot90<false>(x[h + 3]);
    }
  }
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const cd u = x[j];
    x[j] = cadd(u, x[j + 1]);
    x[j + 1] = csub(u, x[j + 1]);
  }
  if (RADIX == 4 && INV) {
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
      x[h + 3] = rot90<true>(x[h + 3]);
#pragma unroll
      for (int j = h; j < h + 2; ++j) {
        const cd u = x[j];
        x[j] = cadd(u, x[j + 2]);
        x[j + 2] = csub(u, x[j + 2]);
      }
    }
  }
}

__device__ __forceinline__ uint32_t smem_a(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
// FRESH: computed at each use, not hoisted out of the steps' loop and held
template <bool FRESH>
__device__ __forceinline__ uint32_t peer(uint32_t addr, uint32_t rank) {
  uint32_t r;
  if (FRESH) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  else asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer(uint32_t a, cd v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, int v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
template <int C>
__device__ __forceinline__ void all_sync() {
  if (C == 1) __syncthreads();
  else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int LOGL, int C>
struct FftCfg {
  static constexpr int L = 1 << LOGL, G = L / 8, NT = 2 * G, NW = NT / 32;
  static constexpr int N2 = L / C;                                     // positions n2 that a CTA owns
  static constexpr bool SPLIT = C == 8;                                // a thread owns alpha or rho, not both
  static constexpr int UN = SPLIT ? 1 : 4 / C;                         // n2 of a thread (and vector)
  static constexpr int NV = SPLIT ? 1 : 2;                             // vectors of a thread
  static constexpr int BUF = L + L / 8;                                // padded points
  static constexpr int NTW = (LOGL - 1) / 3 * 3 * G;                   // twiddle bases (none for a pass of sub-length 8)
  static constexpr int SMEM = (3 * BUF + 2 * L + NTW + (SPLIT ? 2 * N2 : 0)) * 16;
};

// Twiddle bases in shared memory: w, w^2, w^4 of thread t and pass q (sub-length N = L / 8^q, w = e^{-2 pi i p / N}) at
// [3 q + e][t].  (In registers they push the kernel into spills.)
template <int LOGL, int G>
__device__ __forceinline__ void twiddle_init(cd* tab, int tid) {
  for (int i = tid; i < (LOGL - 1) / 3 * 3 * G; i += 2 * G) {
    const int e = i / G, q = e / 3, n = (1 << LOGL) >> (3 * q), t = i - e * G;
    double sn, cs;
    sincospi(-2.0 * static_cast<double>((t & (n / 8 - 1)) << (e - 3 * q)) / n, &sn, &cs);
    tab[i] = make_double2(cs, sn);
  }
}

__device__ __forceinline__ int pad8(int i) { return i + (i >> 3); }

// Between two passes: the first exchange crosses warps (barrier of the G threads that share the transform), the others do not.
template <int G>
__device__ __forceinline__ void pass_sync(int q, int group) {
  if (q == 0 && G > 32) asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(G) : "memory");
  else __syncwarp();
}

// Forward transform of buf by G threads (t = 0..G-1); the results stay in x: slot k = point 8t + k of the permuted spectrum.
template <int LOGL, int G>
__device__ __forceinline__ void fft_forward(cd* buf, cd* x, const cd* tw, int t, int group) {
  constexpr int NP = LOGL / 3, LAST = 1 << (LOGL % 3);
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int s = (1 << LOGL) >> (3 * q + 3);
    const int i0 = (t & ~(s - 1)) * 8 + (t & (s - 1));
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = buf[pad8(i0 + s * k)];
    bf8_fwd(x);
    if (s == 1) break;                                     // (the last pass: no twiddles, results stay in registers)
    const cd w1 = tw[3 * q * G + t], w2 = tw[(3 * q + 1) * G + t], w4 = tw[(3 * q + 2) * G + t], w3 = cmul(w1, w2);
    x[1] = cmul(x[1], w4);                                 // slot k holds residue rev8(k)
    x[2] = cmul(x[2], w2);
    x[3] = cmul(x[3], cmul(w2, w4));
    x[4] = cmul(x[4], w1);
    x[5] = cmul(x[5], cmul(w1, w4));
    x[6] = cmul(x[6], w3);
    x[7] = cmul(x[7], cmul(w3, w4));
#pragma unroll
    for (int k = 0; k < 8; ++k) buf[pad8(i0 + s * k)] = x[k];
    pass_sync<G>(q, group);
  }
  if (LAST > 1) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = buf[pad8(8 * t + k)];
    bf_last<LAST, false>(x);
  }
}
// Inverse (times L) of x (slot k = point 8t + k) through buf; slot k ends as point t + G k in natural order.
template <int LOGL, int G>
__device__ __forceinline__ void fft_inverse(cd* buf, cd* x, const cd* tw, int t, int group) {
  constexpr int NP = LOGL / 3, LAST = 1 << (LOGL % 3);
  if (LAST > 1) {
    bf_last<LAST, true>(x);
#pragma unroll
    for (int k = 0; k < 8; ++k) buf[pad8(8 * t + k)] = x[k];
    pass_sync<G>(1, group);
  }
#pragma unroll
  for (int q = NP - 1; q >= 0; --q) {
    const int s = (1 << LOGL) >> (3 * q + 3);
    const int i0 = (t & ~(s - 1)) * 8 + (t & (s - 1));
    if (s > 1) {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = buf[pad8(i0 + s * k)];
      const cd w1 = tw[3 * q * G + t], w2 = tw[(3 * q + 1) * G + t], w4 = tw[(3 * q + 2) * G + t], w3 = cmul(w1, w2);
      x[1] = cmulc(x[1], w4);
      x[2] = cmulc(x[2], w2);
      x[3] = cmulc(x[3], cmul(w2, w4));
      x[4] = cmulc(x[4], w1);
      x[5] = cmulc(x[5], cmul(w1, w4));
      x[6] = cmulc(x[6], w3);
      x[7] = cmulc(x[7], cmul(w3, w4));
    }
    bf8_inv(x);
    if (q > 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) buf[pad8(i0 + s * k)] = x[k];
      pass_sync<G>(q - 1, group);
    }
  }
}

template <int LOGL, int C>
__global__ void __launch_bounds__(FftCfg<LOGL, C>::NT, LOGL <= 9 ? 3 : LOGL == 10 ? 2 : 1)
saf_fit_fft_kernel(FitState s, int steps, const double* __restrict__ plogp, float* __restrict__ alpha_out,
                   float* __restrict__ rho_out, float* __restrict__ logZ_out, long long out_stride,
                   double* __restrict__ loss_out, double* __restrict__ kl_out) {
  using F = FftCfg<LOGL, C>;
  constexpr int L = F::L, G = F::G, NT = F::NT, NW = F::NW, N2 = F::N2, UN = F::UN, NV = F::NV;
  extern __shared__ double2 sm_d2[];
  cd* const FA = sm_d2;                          // A^, later conj(A^) W^ in place
  cd* const FR = FA + F::BUF;
  cd* const FW = FR + F::BUF;                    // A^ R^ on its way back, then W
  cd* const TZ = FW + F::BUF;                    // [C][N2] back at the owners: Z, later c
  cd* const TG = TZ + L;                         // g
  cd* const tw = TG + L;                         // twiddle bases
  cd* const own = tw + F::NTW;                   // owner twiddles [2][N2] (registers where a thread has both vectors)
  __shared__ float nrm[4][8 * NW];               // partial |A|^2, |R|^2, |W|^2, slope of log Z of every warp of the cluster
  __shared__ double lossp[8 * NW];
  __shared__ int flag[2];                        // raised between barriers 2 and 3, 4 and 1
  // Where half of the threads own alpha and the normalisers, that half has twice the other's fp64 work (and the first
  // warps always sit on the same schedulers): every second CTA of an SM, by its hardware warp slots, swaps the halves
  // (36 x 4096 -2.4 %, one head -5 %; the values do not depend on it).
  __shared__ int swapped;
  if (F::SPLIT) {
    if (threadIdx.x == 0) {
      uint32_t slot;
      asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
      swapped = slot / NW & 1;
    }
    __syncthreads();
  }
  const int tid = F::SPLIT && swapped ? threadIdx.x ^ G : threadIdx.x, lane = tid & 31, warp = tid >> 5, T = s.T;
  uint32_t rank = 0;
  if (C > 1) asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int h = blockIdx.x / C;
  const size_t o = static_cast<size_t>(h) * T;
  const int group = tid / G, t = tid - group * G;          // group 0, 1: the CTA's two transforms of a phase
  const double invM = 1.0 / (static_cast<double>(L) * C);
  twiddle_init<LOGL, G>(tw, tid);
  const int my_vec = F::SPLIT ? tid / N2 : 0;              // vector of local index v: my_vec + v
  // n2 of local index u (within the CTA's share), position of element (u, n1)
  auto n2l = [&](int u) { return F::SPLIT ? tid - my_vec * N2 : tid + u * NT; };
  auto pos = [&](int u, int n1) { return static_cast<int>(rank) * N2 + n2l(u) + L * n1; };
  // owner twiddles e^{-2 pi i n2 (k1 + 1/4) / M}: of k1 = 0, and the factor from one k1 to the next
  cd owr[2 * UN];
#pragma unroll
  for (int k = 0; k < 2 * UN; ++k) {
    const int u = k % UN;
    double sn, cs;
    sincospi((k < UN ? -0.5 : -2.0) * pos(u, 0) / (static_cast<double>(L) * C), &sn, &cs);
    owr[k] = make_double2(cs, sn);
    if (F::SPLIT) own[k * N2 + n2l(u)] = owr[k];
  }
  // C-point sum of an owner's real values, twiddled, to the CTAs of the residues
  auto send = [&](cd* buf, const double* x, int u) {
    const int slot = pad8(static_cast<int>(rank) * N2 + n2l(u));
    const cd fs = F::SPLIT ? own[N2 + n2l(u)] : owr[UN + u];
    cd f = F::SPLIT ? own[n2l(u)] : owr[u], y[C];
    if constexpr (C == 8) {                                // e^{-2 pi i n / 32}, then an 8-point DFT
#pragma unroll
      for (int n = 0; n < C; ++n) y[n] = make_double2(x[n] * cos32(n), -x[n] * sin32(n));
      bf8_fwd(y);
    } else {
#pragma unroll
      for (int k = 0; k < C; ++k) {
        y[k] = make_double2(0.0, 0.0);
#pragma unroll
        for (int n = 0; n < C; ++n) {
          const int m = n * (4 * k + 1) * (8 / C);
          y[k].x = fma(x[n], cos32(m), y[k].x);
          y[k].y = fma(x[n], -sin32(m), y[k].y);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const cd v = cmul(y[C == 8 ? rev8(k) : k], f);
      if (k + 1 < C) f = cmul(f, fs);
      if (C == 1) buf[slot] = v;
      else st_peer(peer<F::SPLIT>(smem_a(buf + slot), k), v);
    }
  };
  // and back: real parts of the inverse at the owner's positions (scaled by 1 / M)
  auto receive = [&](const cd* buf, double* x, int u) {
    const cd fs = F::SPLIT ? own[N2 + n2l(u)] : owr[UN + u];
    cd f = F::SPLIT ? own[n2l(u)] : owr[u], y[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      y[C == 8 ? rev8(k) : k] = cmulc(buf[k * N2 + n2l(u)], f);
      if (k + 1 < C) f = cmul(f, fs);
    }
    if constexpr (C == 8) {
      bf8_inv(y);
#pragma unroll
      for (int n = 0; n < C; ++n) x[n] = invM * fma(y[n].x, cos32(n), -y[n].y * sin32(n));
    } else {
#pragma unroll
      for (int n = 0; n < C; ++n) {
        x[n] = 0.0;
#pragma unroll
        for (int k = 0; k < C; ++k) {
          const int m = n * (4 * k + 1) * (8 / C);
          x[n] = fma(y[k].x, cos32(m), fma(-y[k].y, sin32(m), x[n]));
        }
        x[n] *= invM;
      }
    }
  };
  // an inverse transform's points t + G k to their owners
  auto give_back = [&](cd* buf, const cd* x) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = t + G * k, q = i / N2;
      cd* dst = buf + static_cast<int>(rank) * N2 + (i - q * N2);
      if (C == 1) *dst = x[k];
      else st_peer(peer<F::SPLIT>(smem_a(dst), q), x[k]);
    }
  };
  auto raise = [&](int which) {
    if (C == 1) flag[which] = 1;
    else
      for (int r = 0; r < C; ++r) st_peer(peer<F::SPLIT>(smem_a(flag + which), r), 1);
  };
  auto give_norm = [&](int which, float v) {               // v: this thread's part
    v = wsum(v);
    if (C == 1) {
      if (lane == 0) nrm[which][warp] = v;
    } else if (lane < C) {
      st_peer(peer<F::SPLIT>(smem_a(&nrm[which][rank * NW + warp]), lane), v);
    }
  };
  auto norm2 = [&](int which) {
    float v = 0.0f;
    for (int i = lane; i < C * NW; i += 32) v += nrm[which][i];
    return wsum(v);
  };

  // ---- start: alpha = 0, rho(d) = log max(eta_rel(d)/(T-d), 1e-9), Adam moments zero
  double val[NV][UN][C];                                   // exp of this thread's parameters (0 beyond T)
  if (tid < 2) flag[tid] = 0;
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int n = 0; n < C; ++n) {
        const int i = pos(u, n);
        val[v][u][n] = 0.0;
        if (i >= T) continue;
        const bool is_rho = my_vec + v;
        const double x = is_rho ? log(fmax(s.eta_rel[o + i] / static_cast<double>(T - i), 1e-9)) : 0.0;
        (is_rho ? s.rho : s.alpha)[o + i] = x;
        (is_rho ? s.m_r : s.m_a)[o + i] = 0.0;
        (is_rho ? s.v_r : s.v_a)[o + i] = 0.0;
        val[v][u][n] = is_rho ? exp(x) : 1.0;
        if (F::SPLIT && !is_rho) s.wref[o + i] = 0.0f;
      }
  double tilt = 0.0;                                       // k: A(j) = exp(alpha(j) - k j), R(d) = exp(rho(d) - k d)
  // log2 of the last normalisers' reciprocals, without tilt (straight to memory where registers are short)
  float wlog[F::SPLIT ? 1 : UN * C];
#pragma unroll
  for (int k = 0; k < (F::SPLIT ? 1 : UN * C); ++k) wlog[k] = 0.0f;
  all_sync<C>();

  double acc = 0.0;                                        // this thread's part of T * loss
  double p1 = 1.0, p2 = 1.0;
  bool failed = false;
  int step = 1;
  for (;; ++step) {
    const bool last = step == steps + 1;
    // ---- 1: A, R out
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float nv = 0.0f;
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        send(my_vec + v ? FR : FA, val[v][u], u);
#pragma unroll
        for (int n = 0; n < C; ++n) nv = fmaf(static_cast<float>(val[v][u][n]), static_cast<float>(val[v][u][n]), nv);
      }
      if (F::SPLIT) {                                      // (a warp's threads may own either vector)
        give_norm(0, my_vec ? 0.0f : nv);
        give_norm(1, my_vec ? nv : 0.0f);
      } else {
        give_norm(v, nv);
      }
    }
    all_sync<C>();
    if (flag[1]) {
      --step;                                              // the marginals of the step before were out of bounds
      failed = true;
      break;
    }
    cd x[8];
    fft_forward<LOGL, G>(group ? FR : FA, x, tw, t, group);
    {
      cd* const mine = group ? FR : FA;
#pragma unroll
      for (int k = 0; k < 8; ++k) mine[pad8(8 * t + k)] = x[k];
    }
    __syncthreads();
    if (group == 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = cmul(x[k], FR[pad8(8 * t + k)]);
      fft_inverse<LOGL, G>(FW, x, tw, t, 0);
      give_back(TZ, x);
    }
    all_sync<C>();
    // ---- 2: Z, W
    const float na = sqrtf(norm2(0)), nr = sqrtf(norm2(1));
    float slope = 0.0f;                                    // sum of (i - (T-1)/2) log2 Z
    double w[UN][C];
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int n = 0; n < C; ++n) w[u][n] = 0.0;
    if (!F::SPLIT || my_vec == 0) {
      // (1e-30 .. 1e30: rcp64 and the fp32 logarithm)
      const double lim = fmax(static_cast<double>(GUARD) * na * nr, 1e-30);
      const float ft = static_cast<float>(tilt / LN2_D);
      bool ok = na * nr > 0.0f;
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        double z[C];
        receive(TZ, z, u);
        bool in_bounds = true;
#pragma unroll
        for (int n = 0; n < C; ++n) {
          const bool in = pos(u, n) < T;
          z[n] = in ? z[n] : 1.0;
          in_bounds = in_bounds && (!in || (z[n] >= lim && z[n] < 1e30));
          const double r = rcp64(z[n]);
          w[u][n] = in ? r : 0.0;
          const float lg = __log2f(static_cast<float>(z[n])), fi = static_cast<float>(pos(u, n));
          slope = fmaf(fi - 0.5f * (T - 1), lg, slope);    // (beyond T: log 1)
          z[n] = -lg - ft * fi;
        }
        if (in_bounds) {
#pragma unroll
          for (int n = 0; n < C; ++n) {
            if (!F::SPLIT) wlog[F::SPLIT ? 0 : u * C + n] = static_cast<float>(z[n]);
            else if (pos(u, n) < T) s.wref[o + pos(u, n)] = static_cast<float>(z[n]);
          }
        }
        ok = ok && in_bounds;
        if (!last) send(FW, w[u], u);
      }
      if (!ok) raise(0);
      if (last) {
#pragma unroll
        for (int u = 0; u < UN; ++u)
#pragma unroll
          for (int n = 0; n < C; ++n) {
            const int i = pos(u, n);
            if (i >= T) continue;
            const double lz = fma(tilt, static_cast<double>(i), -log(w[u][n]));
            logZ_out[static_cast<size_t>(h) * out_stride + i] = static_cast<float>(lz);
            acc += lz;
          }
      }
    }
    {
      float nw = 0.0f;
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int n = 0; n < C; ++n) nw = fmaf(static_cast<float>(w[u][n]), static_cast<float>(w[u][n]), nw);
      give_norm(2, nw);
      give_norm(3, slope);
    }
    all_sync<C>();
    if (flag[0]) {
      failed = true;
      break;
    }
    if (last) break;
    // ---- 3: c and g
    if (group == 0) {
      fft_forward<LOGL, G>(FW, x, tw, t, 0);
#pragma unroll
      for (int k = 0; k < 8; ++k) FW[pad8(8 * t + k)] = x[k];
    }
    __syncthreads();
    {
      cd* const mine = group ? FA : FR;
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = cmulc(group ? FW[pad8(8 * t + k)] : x[k], mine[pad8(8 * t + k)]);
      fft_inverse<LOGL, G>(mine, x, tw, t, group);
      give_back(group ? TG : TZ, x);
    }
    // ---- 4: one Adam step in fp64 on Eq. "fit-objective": gradient = (fitted marginal - target marginal) / T
    p1 *= 0.9;
    p2 *= 0.999;
    if (T > 1) tilt += LN2_D * norm2(3) * (12.0 / (static_cast<double>(T) * (static_cast<double>(T) * T - 1.0)));
    const double ib1 = 1.0 / (1.0 - p1), ib2 = 1.0 / (1.0 - p2), iT = 1.0 / static_cast<double>(T);
    // A thread's eight parameters in two halves (alpha and rho, or n1 below and from 4 on): the first half's state is on its
    // way while the cluster meets, the second's while the first is worked on.
    const size_t from = o + ((step - 1) & 1) * s.second, to = o + (step & 1) * s.second;
    double st[2][4][4];
    auto load_state = [&](int half) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = F::SPLIT ? 0 : e / C, n = F::SPLIT ? 4 * half + e : e % C, i = pos(u, n);
        const bool is_rho = F::SPLIT ? my_vec : half, in = i < T;
        st[half][e][0] = in ? ((is_rho ? s.rho : s.alpha) + from)[i] : 0.0;
        st[half][e][1] = in ? ((is_rho ? s.m_r : s.m_a) + from)[i] : 0.0;
        st[half][e][2] = in ? ((is_rho ? s.v_r : s.v_a) + from)[i] : 0.0;
        st[half][e][3] = in ? ((is_rho ? s.eta_rel : s.eta_abs) + o)[i] : 0.0;
      }
    };
    load_state(0);
    all_sync<C>();
    const double nw = static_cast<double>(GUARD) * sqrtf(norm2(2)), lim_c = nw * nr, lim_g = nw * na;
    bool ok = lim_c > 0.0 && lim_g > 0.0;
    double S[UN][C];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const bool is_rho = F::SPLIT ? my_vec : half;
      if (half == 0) load_state(1);
      if (half == 0 || !F::SPLIT) {
#pragma unroll
        for (int u = 0; u < UN; ++u) receive(is_rho ? TG : TZ, S[u], u);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = F::SPLIT ? 0 : e / C, n = F::SPLIT ? 4 * half + e : e % C, i = pos(u, n);
        double& value = val[F::SPLIT ? 0 : half][u][n];
        const double fitted = S[u][n] * value;
        const double g = (fitted - st[half][e][3]) * iT;
        const double m = fma(0.9, st[half][e][1], 0.1 * g);
        const double q = fma(0.999, st[half][e][2], 0.001 * g * g);
        // (fmax drops a NaN, which q holds: NaN and infinite targets go to the direct sums, which pass them on to the whole head)
        ok = ok && fmax(fitted, st[half][e][3]) >= (is_rho ? lim_g : lim_c) * value && q < 1e300;
        const double pnew = fma(-s.lr * (m * ib1), rcp64(sqrt64(q * ib2) + 1e-8), st[half][e][0]);
        const double ex = exp64(fma(-tilt, static_cast<double>(i), pnew));
        value = i < T ? ex : 0.0;
        if (i < T) {
          ((is_rho ? s.rho : s.alpha) + to)[i] = pnew;
          ((is_rho ? s.m_r : s.m_a) + to)[i] = m;
          ((is_rho ? s.v_r : s.v_a) + to)[i] = q;
        }
      }
    }
    if (!ok) raise(1);
  }

  if (failed) {
    // the parameters are those before this step; a reference for the normalisers goes along (of this step or the last)
    if (!F::SPLIT) {
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int n = 0; n < C; ++n)
          if (pos(u, n) < T) s.wref[o + pos(u, n)] = wlog[F::SPLIT ? 0 : u * C + n];
    }
    if (!(step & 1)) {                                     // the state before the step, from the second copy to the first
#pragma unroll
      for (int v = 0; v < NV; ++v)
        for (int u = 0; u < UN; ++u)
          for (int n = 0; n < C; ++n) {
            const int i = pos(u, n);
            if (i >= T) continue;
            double* const a[3] = {my_vec + v ? s.rho : s.alpha, my_vec + v ? s.m_r : s.m_a, my_vec + v ? s.v_r : s.v_a};
            for (int k = 0; k < 3; ++k) a[k][o + i] = a[k][o + s.second + i];
          }
    }
    if (rank == 0 && tid == 0) s.resume[h] = step;
    return;                                                // (nothing of the cluster's is written behind its last barrier)
  }
  // ---- results: L = (1/T)[sum_i log Z(i) - eta_abs.alpha - eta_rel.rho], kappa = L + (1/T) sum P log P
  const size_t oo = static_cast<size_t>(h) * static_cast<size_t>(out_stride);
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int n = 0; n < C; ++n) {
        const int i = pos(u, n);
        if (i >= T) continue;
        const bool is_rho = my_vec + v;
        const double x = (is_rho ? s.rho : s.alpha)[o + (steps & 1) * s.second + i];
        acc -= (is_rho ? s.eta_rel : s.eta_abs)[o + i] * x;
        (is_rho ? rho_out : alpha_out)[oo + i] = static_cast<float>(x);
      }
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, k);
  if (lane == 0) {
    if (C == 1) lossp[warp] = acc;
    else st_peer(peer<F::SPLIT>(smem_a(lossp + rank * NW + warp), 0), acc);
  }
  all_sync<C>();
  if (rank == 0 && tid == 0) {
    double sum = 0.0;
    for (int r = 0; r < C * NW; ++r) sum += lossp[r];
    const double loss = sum / static_cast<double>(T);
    if (loss_out) loss_out[h] = loss;
    if (kl_out) kl_out[h] = loss + plogp[h] / static_cast<double>(T);
    s.resume[h] = -1;
  }
}

// go: launch; else ask how many clusters fit at once
template <int LOGL, int C, typename... Args>
cudaError_t fft_launch(int* active, bool go, const FitState& s, int Hf, cudaStream_t st, Args... args) {
  using F = FftCfg<LOGL, C>;
  auto kern = saf_fit_fft_kernel<LOGL, C>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(Hf) * C);
  cfg.blockDim = dim3(F::NT);
  cfg.dynamicSmemBytes = F::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!go) return cudaOccupancyMaxActiveClusters(active, kern, &cfg);
  return cudaLaunchKernelEx(&cfg, kern, s, args...);
}

template <typename... Args>
cudaError_t fft_dispatch(int logl, int c, int* active, bool go, const FitState& s, int Hf, cudaStream_t st, Args... args) {
#define SAF_FFT(LL, CC) if (logl == LL && c == CC) return fft_launch<LL, CC>(active, go, s, Hf, st, args...)
  SAF_FFT(8, 1); SAF_FFT(9, 1); SAF_FFT(9, 2); SAF_FFT(9, 4); SAF_FFT(9, 8); SAF_FFT(10, 4); SAF_FFT(10, 8); SAF_FFT(11, 8);
#undef SAF_FFT
  return cudaErrorInvalidValue;
}

__global__ void saf_fit_math_kernel(int which, int n, const double* __restrict__ x, double* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = which == 0 ? rcp64(x[i]) : which == 1 ? sqrt64(x[i]) : exp64(x[i]);
}

}  // namespace

cudaError_t launch_fit_math(int which, int n, const double* x, double* y, cudaStream_t st) {
  saf_fit_math_kernel<<<(n + 255) / 256, 256, 0, st>>>(which, n, x, y);
  return cudaGetLastError();
}

// One transform of 512 points (128 threads, three CTAs per SM) per CTA and as many CTAs as that takes, up to eight: us a step of
// one head, clusters of 1 / 2 / 4 / 8: 1024 positions 9.2 / 7.5, 2048 14.8 / 11.4 / 8.4, 4096 - / 18.3 / 12.8 / 9.9.  With
// more heads of 4096 than fit at once (48 clusters of eight), 71 clusters of four do; rounds of them are weighed 18 : 15 (us a step,
// four / eight: 48 heads 20.0 / 14.8, 49 20.0 / 22.5, 71 20.3 / 27.0, 72 31.6 / 27.1, 142 40.2 / 44.1, 143 49.9 / 44.3, 150
// 50.5 / 51.3, 240 69.5 / 77.8).  Other lengths have one cluster size each.
// *launched: false where no such cluster can be resident (then nothing was launched and the direct sums, which run in any
// cluster size, serve all heads).
cudaError_t launch_fit_fft(const FitState& s, int Hf, int steps, const double* plogp, float* alpha_out, float* rho_out,
                           float* logZ_out, long long out_stride, double* loss_out, double* kl_out, cudaStream_t st, bool* launched) {
  int logm = 8;
  while ((1 << logm) < s.T) ++logm;
  int lc = std::max(0, std::min(3, logm - 9));
  auto dispatch = [&](int lc, int* active) {
    return fft_dispatch(logm - lc, 1 << lc, active, active == nullptr, s, Hf, st, steps, plogp, alpha_out, rho_out, logZ_out, out_stride,
                        loss_out, kl_out);
  };
  auto resident = [&](int lc) {
    int n = 0;
    if (dispatch(lc, &n) == cudaSuccess) return n;
    cudaGetLastError();
    return 0;
  };
  int n = resident(lc);
  if (logm == 12) {
    const int n4 = resident(2);
    if (n4 > 0 && (n < 1 || (Hf > n && 18 * ((Hf + n4 - 1) / n4) < 15 * ((Hf + n - 1) / n)))) {
      lc = 2;
      n = n4;
    }
  }
  *launched = n > 0;
  return n > 0 ? dispatch(lc, nullptr) : cudaSuccess;
}

}  // namespace saf
