// Backward of the hybrid causal attention layer on sm_100a, head dimension 128 (96 runs here too: TMA zero-fills
// features 96..127): one persistent kernel, one work item per (batch, head, 128-key block J), looping over the
// 128-query tiles I >= J.  TMEM (512 columns): dV 128, dK 128, X = S^T then P^T, Y = dP^T then dQ.
//   S(t)  = K_J Q_t^T -> X          dP(t) = V_J dO_t^T -> Y                      (operands in smem)
//   P^T   = exp2(c S^T - lse) over X (bf16 pairs),  dS^T = P^T o (dP^T - delta) -> smem
//   dV_J += P^T dO_t (A from TMEM),  dQ_t = dS K_J -> Y (A = the smem dS^T tile read M-major),  dK_J += dS^T Q_t (A = the
//   same smem tile, K-major)
// Issue order of a tile: dP(t) | dV(t), S(t+1) | dQ(t), dK(t).  S(t+1) is queued behind the MMA that consumes P(t), so
// the exponentials of tile t+1 run while tile t's dS, dQ and dK are in flight, and dK(t) runs while dQ(t) is drained
// out of Y; MMAs of one thread execute in order, which is all that protects X, Y and the dS tile.
//
// What bounds it: the five MMAs of a tile are 2900 clk of tensor pipe (512 with A in TMEM, 600 with both operands in
// smem) and the chain through Y (dP, dS, dQ, drain) is about as long.  The 64-query half tiles that this replaces went
// through one S / dP buffer in sequence, two full round trips a tile.
//
// Row terms: LSE and delta reach the compute warps as fp32 vectors with each Q tile (columns of S^T are queries, so a
// value is a broadcast load).  Appendix E.2 (key-block programs accumulate dV and dK; dQ here comes out of the same loop
// and is accumulated across key blocks with TMA reduce-adds).  Frozen items (Sec. 3.3: dV = P^^T dO, no query/key
// gradients) use the tensor-core form (Hankel band x scaled dO, see the forward) or generate P^^T tiles with one
// exponential per element; their dO tiles go through the Q stages.
//
// CTA = 896 threads: warps 0-15 compute (TMEM lane = key row; four warps per lane quarter, 32 query columns each),
// warps 16-23 dQ drain (two per lane quarter, 64 feature columns each), warp 24 TMA producer, warp 25 tcgen05 issuer and
// TMEM owner.  Registers: 512 x 80 + 256 x 72 + 128 x 40 = the 896 x 72 of the launch.  Every wait is bounded.
#include <cuda_bf16.h>
#include "ptx.cuh"
#include "saf_internal.h"

SAF_SPAN_DEFINE(bwd128)

#ifdef SAF_TRACE
__device__ unsigned long long g_saf_trace_bwd128[3][16384];
#define TRB(role, id)                                                                                  \
  do {                                                                                                 \
    if (blockIdx.x == 0 && (threadIdx.x & 31) == 0 && tr_n < 16380)                                    \
      g_saf_trace_bwd128[role][tr_n++] = (static_cast<unsigned long long>(id) << 48) | (clock64() & 0xffffffffffffULL); \
  } while (0)
extern "C" int saf_debug_read_trace_bwd128(unsigned long long* out) {
  return static_cast<int>(cudaMemcpyFromSymbol(out, g_saf_trace_bwd128, sizeof(g_saf_trace_bwd128)));
}
#else
#define TRB(role, id)
#endif

namespace saf {

namespace {

constexpr float LOG2E_W = 1.4426950408889634f;

struct W128 {
  static constexpr int PANEL = 128 * 64 * 2;         // [128 rows][64 cols] bf16, 16 KB
  static constexpr int TILE = 2 * PANEL;
  static constexpr int NS = 2;                       // stages of Q (frozen items: of dO)
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = TILE;
  static constexpr int OFF_Q = 2 * TILE;
  static constexpr int OFF_DO = OFF_Q + NS * TILE;   // one dO tile; tensor-core frozen form: bands, 4 KB per stage
  static constexpr int OFF_DS = OFF_DO + TILE;       // [query half][128 key rows][64 queries]; general frozen form: tables
  static constexpr int OFF_DQ = OFF_DS + TILE;       // fp32 staging boxes of the drain warps, 8 x [32 rows][32 floats]
  static constexpr int OFF_AUX = OFF_DQ + 8 * 4096;  // NS x { -LSE log2 e [128], -delta [128] }
  static constexpr int OFF_BAR = OFF_AUX + NS * 1024;
  static constexpr int NBAR = 2 + 2 * NS + 2 + 9;
  static constexpr int SMEM = OFF_BAR + NBAR * 8 + 16;
  static constexpr int TMEM_COLS = 512;
  static constexpr int COL_DV = 0, COL_DK = 128, COL_X = 256, COL_Y = 384;
  static constexpr int NTHREADS = 896;
};
static_assert(W128::SMEM <= 227 * 1024, "shared memory");

enum W128Site { W_KV_EMPTY = 81, W_Q_EMPTY, W_KV_FULL, W_Q_FULL, W_P_FULL, W_ACC_FREE, W_DQ_FREE, W_S_FULL,
                W_DP_FULL, W_DQ_FULL, W_ACC_FULL, W_PFREE, W_DO_EMPTY, W_DO_FULL, W_DS_FULL, W_ALIGN };

__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Work item `it` and whether it takes the tensor-core frozen form, fetched one item ahead of its use.
struct ItemW {
  WorkItem w;
  bool fast;
};
__device__ __forceinline__ ItemW load_item_w(const BwdParams& p, int it, int it_end) {
  ItemW v;
  v.w = WorkItem{0, 0, 0, KIND_ORDINARY};
  v.fast = false;
  if (it < it_end) {
    const int4 raw = __ldg(reinterpret_cast<const int4*>(p.items + it));
    v.w = WorkItem{raw.x, raw.y, raw.z, raw.w};
    v.fast = raw.w != KIND_ORDINARY && p.band_b != nullptr && __ldg(p.fast_ok + raw.y) != 0 &&
             __ldg(p.ovf + raw.y) != p.call_id;
  }
  return v;
}

}  // namespace

__global__ void __launch_bounds__(W128::NTHREADS, 1)
saf_bwd128_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                  const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mdo,
                  const __grid_constant__ CUtensorMap mdot, const __grid_constant__ CUtensorMap mdq,
                  const BwdParams p) {
  using C = W128;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* kv_full = bars;
  uint64_t* kv_empty = bars + 1;
  uint64_t* q_full = bars + 2;                   // [NS] Q tile and its row terms (frozen: dO tile, band)
  uint64_t* q_empty = q_full + C::NS;            // [NS]
  uint64_t* do_full = q_empty + C::NS;
  uint64_t* do_empty = do_full + 1;
  uint64_t* s_full = do_empty + 1;
  uint64_t* dp_full = s_full + 1;
  uint64_t* p_full = dp_full + 1;                // P^T written (16 warp arrivals)
  uint64_t* ds_full = p_full + 1;                // dS^T written (16 warp arrivals)
  uint64_t* dq_full = ds_full + 1;
  uint64_t* dq_free = dq_full + 1;               // dQ is in the drain warps' registers (8 warp arrivals)
  uint64_t* acc_full = dq_free + 1;
  uint64_t* acc_free = acc_full + 1;             // 16 compute warps
  uint64_t* pfree = acc_free + 1;                // general frozen form: the P^^T tile has been consumed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pfree + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const WaitCtx wc{abort_flag, p.status, p.wait_limit_ns};
  SAF_SPAN(bwd128, 0);
#ifdef SAF_TRACE
  int tr_n = 0;
#endif
  const int nblk = p.nblk;
  if ((smem_u32(smem) & 1023u) != 0) {           // (the swizzled tiles need it; there is no room for a slack)
    if (tid == 0) atomicCAS(p.status, 0, (DEV_TIMEOUT << 24) | (W_ALIGN << 16) | static_cast<int>(blockIdx.x & 0xffff));
    return;
  }

  if (tid == 0) {
    *abort_flag = 0;
    mbar_init(kv_full, 1);
    mbar_init(kv_empty, 1);
    for (int s = 0; s < C::NS; ++s) {
      mbar_init(q_full + s, 1);
      mbar_init(q_empty + s, 1);
    }
    mbar_init(do_full, 1);
    mbar_init(do_empty, 1);
    mbar_init(s_full, 1);
    mbar_init(dp_full, 1);
    mbar_init(p_full, 16);
    mbar_init(ds_full, 16);
    mbar_init(dq_full, 1);
    mbar_init(dq_free, 8);
    mbar_init(acc_full, 1);
    mbar_init(acc_free, 16);
    mbar_init(pfree, 1);
    mbar_fence_init();
  }
  const int it_begin = p.cta_offsets[blockIdx.x], it_end = p.cta_offsets[blockIdx.x + 1];
  if (warp == 25) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 24 && lane == 0) {
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
    tma_prefetch_desc(&mq);
    tma_prefetch_desc(&mdo);
    tma_prefetch_desc(&mdot);
    if (it_begin < it_end) prefetch_l1(p.items + it_begin);
  }
  const uint32_t tmem = *tmem_slot;
  // The prologue above overlapped the previous kernel's tail.  Of global memory it touches only what no kernel writes, the
  // tensor maps and the work list (pdl_wait in ptx.cuh): their first use would otherwise miss behind the wait.
  pdl_launch_dependents();
  pdl_wait();

  if (warp >= 24) {
    reg_dec<40>();
    if (warp == 24) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0) {
        uint32_t nkv = 0, nq = 0, ndo = 0;
        bool ok = true, bands_open = false;
        ItemW nxt = load_item_w(p, it_begin, it_end);
        for (int it = it_begin; it < it_end && ok; ++it) {
          const WorkItem w = nxt.w;
          const bool fast = nxt.fast;
          nxt = load_item_w(p, it + 1, it_end);
          const bool ord = w.kind == KIND_ORDINARY;
          const size_t bh = static_cast<size_t>(w.b) * p.H + w.h;
          const int qh = (ord && p.qslot) ? p.qslot[w.h] : w.h;          // head index in the Q tensor
          auto load_tile = [&](const CUtensorMap* m, int off, uint64_t* bar, int row0, int head) {
            for (int pn = 0; pn < 2; ++pn)
              tma_load_4d(smem + off + pn * C::PANEL, m, bar, pn * 64, row0, head, w.b);
          };
          if (ord) {
            const int kh = p.qslot ? p.qslot[w.h] : w.h / p.kv_group;    // ... in the K tensor
            ok = mbar_wait(kv_empty, (nkv & 1) ^ 1, wc, W_KV_EMPTY);
            if (!ok) break;
            mbar_expect_tx(kv_full, 2 * C::TILE);
            load_tile(&mk, C::OFF_K, kv_full, w.blk * BLK, kh);
            load_tile(&mv, C::OFF_V, kv_full, w.blk * BLK, w.h / p.kv_group);
            ++nkv;
            if (bands_open) {
              // the bands (in the dO tile's place) of the last frozen tiles have been consumed
              for (uint32_t n = nq > C::NS ? nq - C::NS : 0; n < nq && ok; ++n)
                ok = mbar_wait(q_empty + n % C::NS, (n / C::NS) & 1, wc, W_Q_EMPTY);
              if (!ok) break;
              bands_open = false;
            }
          } else if (fast && !bands_open) {
            // the last dO tile has been consumed
            if (ndo > 0) ok = mbar_wait(do_empty, (ndo - 1) & 1, wc, W_DO_EMPTY);
            if (!ok) break;
            bands_open = true;
          }
          const int fo = fast ? p.hord[w.h] : 0;
          const uint8_t* bands = static_cast<const uint8_t*>(p.band_b) + static_cast<size_t>(w.h) * p.nblkp * 4096;
          for (int I = w.blk; I < nblk; ++I, ++nq) {
            const uint32_t s = nq % C::NS;
            ok = mbar_wait(q_empty + s, ((nq / C::NS) & 1) ^ 1, wc, W_Q_EMPTY);
            if (!ok) break;
            const int qoff = C::OFF_Q + s * C::TILE;
            if (ord) {
              mbar_expect_tx(q_full + s, C::TILE + 1024);
              load_tile(&mq, qoff, q_full + s, I * BLK, qh);
              uint8_t* aux = smem + C::OFF_AUX + s * 1024;
              const size_t vec = (bh * nblk + I) * 512;
              bulk_load(aux, static_cast<const uint8_t*>(p.q_ext) + vec, 512, q_full + s);
              bulk_load(aux + 512, static_cast<const uint8_t*>(p.do_ext) + vec, 512, q_full + s);
              ok = mbar_wait(do_empty, (ndo & 1) ^ 1, wc, W_DO_EMPTY);
              if (!ok) break;
              mbar_expect_tx(do_full, C::TILE);
              load_tile(&mdo, C::OFF_DO, do_full, I * BLK, w.h);
              ++ndo;
            } else if (fast) {
              // tensor-core form: the Hankel band of distance block (I - J) and the scaled dO tile
              mbar_expect_tx(q_full + s, C::TILE + 4096);
              bulk_load(smem + C::OFF_DO + s * 4096, bands + static_cast<size_t>(I - w.blk) * 4096, 4096, q_full + s);
              load_tile(&mdot, qoff, q_full + s, I * BLK, fo);
            } else {
              mbar_expect_tx(q_full + s, C::TILE);
              load_tile(&mdo, qoff, q_full + s, I * BLK, w.h);
            }
          }
        }
      }
    } else if (warp == 25) {
      // ---------------------------------------------------------------- tcgen05 issuer
      // The whole warp walks the loops (warp-uniform operands); one elected lane issues.
      const bool leader = elect_one() != 0;
      const uint32_t sb = smem_u32(smem);
      constexpr uint32_t id_s = umma_idesc_bf16(128, 128, 0, 0);     // S^T, dP^T: both operands K-major
      // (head dimension 96 runs here with features 96..127 zero-filled by TMA: the gradient MMAs produce only 96
      // columns and the score MMAs skip the two empty k-steps)
      const uint32_t id_acc = umma_idesc_bf16(128, p.d_real, 0, 1);  // dV, dK: A K-major, B MN-major
      const uint32_t id_dq = umma_idesc_bf16(128, p.d_real, 1, 1);   // dQ: A (dS^T tile) M-major, B MN-major
      const uint32_t id_hk = umma_idesc_f16(128, p.d_real, 0, 1);    // fp16 band x fp16 scaled dO
      const int nk16 = p.d_real / 16;
      // descriptor halves for smem offset 0: 128B-swizzled K-major tiles (k-step +32 B inside a 64-wide panel), MN-major
      // tiles whose two 64-wide halves are a panel apart (k-step +2048 B), and the Hankel band
      const uint64_t d_k = umma_smem_desc(sb, 16, 1024, UMMA_LAYOUT_SW128);
      const uint64_t d_m = umma_smem_desc(sb, C::PANEL, 1024, UMMA_LAYOUT_SW128);
      const uint64_t d_band = umma_smem_desc(sb, 128, 128, UMMA_LAYOUT_NONE);
      const uint32_t lo_k = desc_lo(d_k), hi_k = desc_hi(d_k), lo_m = desc_lo(d_m), hi_m = desc_hi(d_m);
      const uint32_t lo_b = desc_lo(d_band), hi_b = desc_hi(d_band);
      const uint32_t t_x = tmem + C::COL_X, t_y = tmem + C::COL_Y;
      uint32_t nkv = 0, nq = 0, ndo = 0, nitem = 0, np = 0, nds = 0;
      bool ok = true;
      auto q_wait = [&](uint32_t pos) {
        return mbar_wait_warp(q_full + pos % C::NS, (pos / C::NS) & 1, wc, W_Q_FULL);
      };
      // (scores) d = a b^T over the features; a, b: smem offsets of K-major tiles
      auto issue_kk = [&](uint32_t d, uint32_t a_off, uint32_t b_off, uint64_t* bar) {
        if (leader) {
#pragma unroll
          for (int kc = 0; kc < 8; ++kc) {
            if (kc >= nk16) break;
            const uint32_t off = ((kc >> 2) * C::PANEL + (kc & 3) * 32) >> 4;
            umma_ss2(d, lo_k + (a_off >> 4) + off, hi_k, lo_k + (b_off >> 4) + off, hi_k, id_s, kc > 0);
          }
          umma_commit(bar);
        }
        __syncwarp();
      };
      ItemW nxt = load_item_w(p, it_begin, it_end);
      for (int it = it_begin; it < it_end && ok; ++it, ++nitem) {
        const WorkItem w = nxt.w;
        const bool fast = nxt.fast;
        nxt = load_item_w(p, it + 1, it_end);
        const int nt = nblk - w.blk;
        if (w.kind == KIND_ORDINARY) {
          ok = mbar_wait_warp(kv_full, nkv++ & 1, wc, W_KV_FULL) && q_wait(nq);
          if (!ok) break;
          tc_fence_after();
          issue_kk(t_x, C::OFF_K, C::OFF_Q + (nq % C::NS) * C::TILE, s_full);
          for (int t = 0; t < nt && ok; ++t, ++nq) {
            // dP(t): the dQ that was in Y is out
            ok = mbar_wait_warp(do_full, ndo & 1, wc, W_DO_FULL) && mbar_wait_warp(dq_free, (ndo & 1) ^ 1, wc, W_DQ_FREE);
            if (!ok) break;
            ++ndo;
            tc_fence_after();
            TRB(0, 1);
            issue_kk(t_y, C::OFF_V, C::OFF_DO, dp_full);
            TRB(0, 2);
            // dV(t), S(t+1)
            ok = (t > 0 || mbar_wait_warp(acc_free, (nitem & 1) ^ 1, wc, W_ACC_FREE)) &&
                 (t + 1 == nt || q_wait(nq + 1)) && mbar_wait_warp(p_full, np++ & 1, wc, W_P_FULL);
            if (!ok) break;
            tc_fence_after();
            TRB(0, 3);
            if (leader) {
#pragma unroll
              for (int kc = 0; kc < 8; ++kc)
                umma_ts2(tmem + C::COL_DV, t_x + 32 * (kc >> 1) + 8 * (kc & 1), lo_m + (C::OFF_DO >> 4) + 128 * kc, hi_m, id_acc,
                         kc > 0 || t > 0 ? 1u : 0u);
              umma_commit(do_empty);
            }
            __syncwarp();
            if (t + 1 < nt) issue_kk(t_x, C::OFF_K, C::OFF_Q + ((nq + 1) % C::NS) * C::TILE, s_full);
            TRB(0, 4);
            // dQ(t), dK(t)
            ok = mbar_wait_warp(ds_full, nds++ & 1, wc, W_DS_FULL);
            if (!ok) break;
            tc_fence_after();
            TRB(0, 5);
            if (leader) {
#pragma unroll
              for (int kc = 0; kc < 8; ++kc)
                umma_ss2(t_y, lo_m + (C::OFF_DS >> 4) + 128 * kc, hi_m, lo_m + (C::OFF_K >> 4) + 128 * kc, hi_m, id_dq, kc > 0);
              umma_commit(dq_full);
            }
            __syncwarp();
            const uint32_t q_lo = lo_m + ((C::OFF_Q + (nq % C::NS) * C::TILE) >> 4);
            if (leader) {
#pragma unroll
              for (int kc = 0; kc < 8; ++kc)
                umma_ss2(tmem + C::COL_DK, lo_k + (C::OFF_DS >> 4) + (((kc >> 2) * C::PANEL + (kc & 3) * 32) >> 4), hi_k,
                         q_lo + 128 * kc, hi_m, id_acc, kc > 0 || t > 0 ? 1u : 0u);
              umma_commit(q_empty + nq % C::NS);
              if (t + 1 == nt) umma_commit(kv_empty);
            }
            __syncwarp();
            TRB(0, 6);
          }
        } else {
          // frozen item: dV only.  Tensor-core form: A = Hankel band, B = scaled dO tile; general form: A = the P^^T tile
          // the compute warps wrote into X.
          for (int t = 0; t < nt && ok; ++t, ++nq) {
            const uint32_t s = nq % C::NS;
            ok = q_wait(nq) && (t > 0 || mbar_wait_warp(acc_free, (nitem & 1) ^ 1, wc, W_ACC_FREE)) &&
                 (fast || mbar_wait_warp(p_full, np++ & 1, wc, W_P_FULL));
            if (!ok) break;
            tc_fence_after();
            const uint32_t do_lo = lo_m + ((C::OFF_Q + s * C::TILE) >> 4);
            const uint32_t band_lo = lo_b + ((C::OFF_DO + s * 4096) >> 4);
            if (leader) {
              if (fast) {
#pragma unroll
                for (int kc = 0; kc < 8; ++kc)
                  umma_ss2(tmem + C::COL_DV, band_lo + 16 * kc, hi_b, do_lo + 128 * kc, hi_m, id_hk, kc > 0 || t > 0 ? 1u : 0u);
              } else {
#pragma unroll
                for (int kc = 0; kc < 8; ++kc)
                  umma_ts2(tmem + C::COL_DV, t_x + 32 * (kc >> 1) + 8 * (kc & 1), do_lo + 128 * kc, hi_m, id_acc,
                           kc > 0 || t > 0 ? 1u : 0u);
                umma_commit(pfree);
              }
              umma_commit(q_empty + s);
            }
            __syncwarp();
          }
        }
        if (!ok) break;
        if (leader) umma_commit(acc_full);
        __syncwarp();
      }
    }
  } else if (warp >= 16) {
    // ------------------------------------------------------------------ dQ drain warps
    // A warp takes 32 query rows x 64 features into registers at once, so that Y is free again, and sends them as
    // two [32][32] boxes through its own staging box.
    const int q4 = warp & 3, hh = (warp - 16) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    uint8_t* box = smem + C::OFF_DQ + (warp - 16) * 4096;
    const uint32_t stage_row = smem_u32(box) + lane * 128;
    uint32_t ndq = 0;
    bool ok = true;
    for (int it = it_begin; it < it_end && ok; ++it) {
      const WorkItem w = p.items[it];
      if (w.kind != KIND_ORDINARY) continue;
      const int qh = p.qslot ? p.qslot[w.h] : w.h;      // head index in the dQ accumulator
      for (int I = w.blk; I < nblk; ++I) {
        ok = mbar_wait_warp(dq_full, ndq++ & 1, wc, W_DQ_FULL);
        if (!ok) break;
        tc_fence_after();
        uint32_t r[2][32];
        tmem_ld32(tmem + lane_base + C::COL_Y + 64 * hh, r[0]);
        tmem_ld32(tmem + lane_base + C::COL_Y + 64 * hh + 32, r[1]);
        tmem_wait_ld();
        tc_fence_before();
        warp_arrive(dq_free);                           // the tensor core may overwrite Y
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int col = 64 * hh + 32 * k;
          if (col >= p.d_real) break;                   // head dimension 96: the fourth box does not exist
          if (lane == 0) bulk_wait_group_read0();       // the box's previous contents have been read
          __syncwarp();
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const uint32_t chunk = static_cast<uint32_t>(g ^ (lane & 7)) * 16;
            st_shared_v4w(stage_row + chunk, __float_as_uint(__uint_as_float(r[k][4 * g]) * p.scale),
                          __float_as_uint(__uint_as_float(r[k][4 * g + 1]) * p.scale),
                          __float_as_uint(__uint_as_float(r[k][4 * g + 2]) * p.scale),
                          __float_as_uint(__uint_as_float(r[k][4 * g + 3]) * p.scale));
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_reduce_add_4d(&mdq, box, col, I * BLK + 32 * q4, qh, w.b);
            bulk_commit_group();
          }
        }
      }
    }
    if (lane == 0) bulk_wait_group0();                  // all reduce-adds have landed before the kernel ends
  } else {
    // ------------------------------------------------------------------ compute warps (16 x 32 threads)
    // warp = 4 cq + q4: lane quarter q4 (TMEM lane = key row), query columns 32 cq .. 32 cq + 31 of the tile
    reg_inc<80>();
    const int q4 = warp & 3, cq = warp >> 2;
    const int rowl = q4 * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const uint32_t t_x = tmem + lane_base + C::COL_X + 32 * cq;
    const uint32_t t_y = tmem + lane_base + C::COL_Y + 32 * cq;
    float* r2raw = reinterpret_cast<float*>(smem + C::OFF_DS);     // [256] rho' over the tile's band of distances
    float* z2s = r2raw + 256;                                      // [128] logZ' of the tile's queries
    uint32_t ns = 0, nacc = 0, nq = 0, npf = 0;
    bool ok = true;
    // A warp whose wait was abandoned keeps walking (without storing) to the next agreement barrier, where all
    // sixteen leave together; none is ever left alone at a named barrier.
    ItemW nxt = load_item_w(p, it_begin, it_end);
    for (int it = it_begin; it < it_end; ++it) {
      const WorkItem w = nxt.w;
      const bool fast = nxt.fast;                        // (the next item is fetched under the epilogue's wait)
      const bool ord = w.kind == KIND_ORDINARY;
      const int nt = nblk - w.blk;
      int key = w.blk * BLK + rowl;
      float dv_mul = 1.0f;
      if (named_bar_or(1, 512, !ok)) break;
      if (fast) {
        // tensor-core form: nothing to do per tile; lane m holds key 127-m, scaled by a(j) below
        key = w.blk * BLK + 127 - rowl;
        dv_mul = (key < p.T) ? p.avec[static_cast<size_t>(w.h) * p.Tp + key] * (1.0f / HK_BAND_SCALE) : 0.0f;
        nq += nt;
      } else if (ord) {
        const uint64_t c2 = pk2(p.scale_log2, p.scale_log2);
        for (int t = 0; t < nt; ++t, ++nq, ++ns) {
          const uint32_t aux = smem_u32(smem + C::OFF_AUX) + (nq % C::NS) * 1024 + cq * 128;
          if (warp == 0) TRB(1, 11);
          // (the Q tile's barrier also covers its row terms: this thread reads them, so it waits for it itself)
          if (!mbar_wait_warp(q_full + nq % C::NS, (nq / C::NS) & 1, wc, W_Q_FULL)) ok = false;
          if (!mbar_wait_warp(s_full, ns & 1, wc, W_S_FULL)) ok = false;
          tc_fence_after();
          if (warp == 0) TRB(1, 12);
          uint32_t rs[32];
          tmem_ld32(t_x, rs);
          tmem_wait_ld();
          {
            uint32_t pk[16];
#pragma unroll
            for (int e4 = 0; e4 < 8; ++e4) {
              float z[4];
              ld_shared_v4f(aux + e4 * 16, z[0], z[1], z[2], z[3]);       // -LSE log2 e of four queries
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const int e = 2 * e4 + k;
                float p0, p1;
                upk2(fma2(pk2(__uint_as_float(rs[2 * e]), __uint_as_float(rs[2 * e + 1])), c2, pk2(z[2 * k], z[2 * k + 1])), p0, p1);
                p0 = ex2_approx(p0);
                p1 = ex2_approx(p1);
                if (t == 0) {                              // diagonal tile: query index >= key index
                  const int qa = 32 * cq + 2 * e;
                  if (qa < rowl) p0 = 0.0f;
                  if (qa + 1 < rowl) p1 = 0.0f;
                }
                rs[2 * e] = __float_as_uint(p0);
                rs[2 * e + 1] = __float_as_uint(p1);
                pk[e] = pack_bf16x2(p0, p1);
              }
            }
            tmem_st16(t_x, pk);                            // bf16 pairs re-use columns this warp has consumed
          }
          tmem_wait_st();
          tc_fence_before();
          warp_arrive(p_full);
          if (warp == 0) TRB(1, 13);
          if (!mbar_wait_warp(dp_full, ns & 1, wc, W_DP_FULL)) ok = false;
          tc_fence_after();
          if (warp == 0) TRB(1, 14);
          // dS^T row (this key) -> smem panel of this query half, 128-byte swizzle (chunk ^= row & 7).  (The MMAs that read
          // the tile's previous contents were issued before dP(t): they have completed.)
          const uint32_t rowaddr = smem_u32(smem + C::OFF_DS + (cq >> 1) * C::PANEL) + rowl * 128;
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            uint32_t rd[16], dk[8];
            tmem_ld16(t_y + 16 * hf, rd);
            tmem_wait_ld();
#pragma unroll
            for (int e4 = 0; e4 < 4; ++e4) {
              float z[4];
              ld_shared_v4f(aux + 512 + hf * 64 + e4 * 16, z[0], z[1], z[2], z[3]);     // -delta of four queries
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const int e = 2 * e4 + k;
                float d0, d1;
                upk2(mul2(add2(pk2(__uint_as_float(rd[2 * e]), __uint_as_float(rd[2 * e + 1])), pk2(z[2 * k], z[2 * k + 1])),
                          pk2(__uint_as_float(rs[16 * hf + 2 * e]), __uint_as_float(rs[16 * hf + 2 * e + 1]))),
                     d0, d1);
                dk[e] = pack_bf16x2(d0, d1);
              }
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              const uint32_t chunk = static_cast<uint32_t>((4 * (cq & 1) + 2 * hf + g) ^ (rowl & 7));
              st_shared_v4w(rowaddr + chunk * 16, dk[4 * g], dk[4 * g + 1], dk[4 * g + 2], dk[4 * g + 3]);
            }
          }
          fence_proxy_async_smem();
          tc_fence_before();
          warp_arrive(ds_full);
          if (warp == 0) TRB(1, 15);
        }
      } else {
        // ---------------- frozen head, general form: P^^T tiles, one exponential per element
        nq += nt;
        const float* alpha_h = p.alpha + static_cast<size_t>(w.h) * p.Tp;
        const float* rho_h = p.rho + static_cast<size_t>(w.h) * p.Tp;
        const float* logz_h = p.logZ + static_cast<size_t>(w.h) * p.Tp;
        const float a2 = (key < p.T) ? alpha_h[key] * LOG2E_W : -INFINITY;
        bool leave = false;
        for (int t = 0; t < nt; ++t) {
          if (named_bar_or(1, 512, !ok)) {                 // previous tile's table readers are done; agree to go on
            ok = false;
            leave = true;
            break;
          }
          const int d = t * BLK - 127 + tid;               // band entry x = tid: distance of (query - key + 127)
          if (tid < 256) r2raw[tid] = (tid < 255 && d >= 0 && d < p.T) ? rho_h[d] * LOG2E_W : -INFINITY;
          if (tid < 128) {
            const int qi = (w.blk + t) * BLK + tid;
            z2s[tid] = (qi < p.T) ? logz_h[qi] * LOG2E_W : INFINITY;
          }
          named_bar_sync(2, 512);
          if (t > 0) {                                     // the previous P^^T tile has been consumed
            if (!mbar_wait_warp(pfree, npf & 1, wc, W_PFREE)) ok = false;
            ++npf;
            tc_fence_after();
          }
          const int q0 = 32 * cq;
          const float* rb = r2raw + (q0 - rowl + 127);
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e)
            pk[e] = pack_bf16x2(ex2_approx(a2 + rb[2 * e] - z2s[q0 + 2 * e]),
                                ex2_approx(a2 + rb[2 * e + 1] - z2s[q0 + 2 * e + 1]));
          tmem_st16(t_x, pk);
          tmem_wait_st();
          tc_fence_before();
          warp_arrive(p_full);
        }
        if (leave) break;
        // keep the barrier in step: absorb the completion of the last tile
        if (!mbar_wait_warp(pfree, npf & 1, wc, W_PFREE)) ok = false;
        ++npf;
      }
      // ---------------- epilogue: this warp's 32 feature columns of dV and (ordinary items) dK
      nxt = load_item_w(p, it + 1, it_end);              // its load latency passes under the wait for the last MMAs
      if (!mbar_wait_warp(acc_full, nacc & 1, wc, W_ACC_FULL)) ok = false;
      ++nacc;
      tc_fence_after();
      // The rows go through 2 KB of the idle dS tile per warp, so that a store instruction covers eight rows with 64
      // consecutive bytes each instead of 32 rows with 16 (written row by row from the registers, 64 KB per gradient kept
      // the load/store unit busy for ~12000 clk an item: 0.889 ms against 0.836 on 8x12x4096x128, 25 % frozen).
      const int ncol = p.d_real;                           // 128, or 96 (row length of the gradient tensors)
      const int kvh = w.h / p.kv_group;
      const uint32_t box = smem_u32(smem + C::OFF_DS) + warp * 2048;
      const uint32_t put = box + lane * 64, swz = (lane >> 1) & 3;    // chunk ^= (row >> 1) & 3: conflict-free both ways
      const int grow = lane >> 2, gch = lane & 3;          // reading: row 8 i + grow, 16-byte chunk gch
#pragma unroll 1
      for (int which = 0; which < (ord ? 2 : 1); ++which) {
        uint32_t r[32];
        tmem_ld32(tmem + lane_base + (which == 0 ? C::COL_DV : C::COL_DK) + 32 * cq, r);
        tmem_wait_ld();
        if (which == 1 || !ord) {
          tc_fence_before();
          warp_arrive(acc_free);                           // the accumulators may be overwritten
        }
        if (32 * cq >= ncol) continue;
        const float mul = which == 0 ? dv_mul : p.scale;
        const int hk = (which == 1 && p.qslot) ? p.qslot[w.h] : kvh;
        const int nhk = (which == 1 && p.qslot) ? p.n_ord : p.H / p.kv_group;
        const size_t head = (static_cast<size_t>(w.b) * nhk + hk) * p.T;
        void* base = which == 0 ? p.dV : p.dK;
#pragma unroll
        for (int half = 0; half < 2; ++half) {             // fp32: 16 columns at a time; bf16: all 32 in the first round
          if (half == 1 && !p.grad_f32) break;
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
              v[k] = p.grad_f32 ? __float_as_uint(__uint_as_float(r[16 * half + 4 * c + k]) * mul)
                                : pack_bf16x2(__uint_as_float(r[8 * c + 2 * k]) * mul, __uint_as_float(r[8 * c + 2 * k + 1]) * mul);
            st_shared_v4w(put + ((c ^ swz) * 16), v[0], v[1], v[2], v[3]);
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int rr = 8 * i + grow, rk = q4 * 32 + rr;
            const int row = w.blk * BLK + (fast ? 127 - rk : rk);
            float x0, x1, x2, x3;
            ld_shared_v4f(box + rr * 64 + ((gch ^ ((rr >> 1) & 3)) * 16), x0, x1, x2, x3);
            if (row >= p.T || !ok) continue;
            if (p.grad_f32) {
              float* dst = static_cast<float*>(base) + (head + row) * ncol + 32 * cq + 16 * half + 4 * gch;
              if (p.kv_group > 1) red_add_v4(dst, x0, x1, x2, x3);      // shared head: sum over its query heads
              else *reinterpret_cast<float4*>(dst) = make_float4(x0, x1, x2, x3);
            } else {
              *reinterpret_cast<float4*>(static_cast<__nv_bfloat16*>(base) + (head + row) * ncol + 32 * cq + 8 * gch) =
                  make_float4(x0, x1, x2, x3);
            }
          }
        }
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  __syncwarp();
  if (*abort_flag) {
    // A wait gave up: let copies and MMAs that are still in flight land before the CTA's
    // shared memory and TMEM are released.
    for (int i = 0; i < 64; ++i) __nanosleep(20000);
  }
  tc_fence_before();
  __syncthreads();
  SAF_SPAN(bwd128, 1);
  if (warp == 25) tmem_dealloc(tmem, C::TMEM_COLS);
}

cudaError_t launch_bwd128(const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mq, const CUtensorMap& mdo,
                          const CUtensorMap& mdot, const CUtensorMap& mdq, const BwdParams& p, int grid,
                          cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(saf_bwd128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, W128::SMEM);
  if (e != cudaSuccess) return e;
  return launch_pdl(PDL_BWD, saf_bwd128_kernel, dim3(grid), dim3(W128::NTHREADS), W128::SMEM, st, mk, mv, mq, mdo, mdot, mdq, p);
}

}  // namespace saf
