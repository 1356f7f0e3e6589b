// Forward of the hybrid causal attention layer on sm_100a, two chains of tiles per work item: one persistent kernel for
// ordinary (flash-style online softmax) and frozen (pattern rebuilt from alpha/rho/logZ) heads.
//
// One CTA per SM, 512 threads: warps 0-3 softmax of query block 0 of the item, warps 4-7 of query block 1 (one thread
// per query row = TMEM lane, all 128 scores of a tile in registers), warps 8-11 epilogue, warp 12 TMA producer,
// warp 13 tcgen05 issuer and TMEM owner.  Registers are moved to the softmax warps (192 a thread) from the others (64):
// 256 x 192 + 256 x 64 = the 512 x 128 of the launch.
//
// Why this shape: a 128x128 tile of an ordinary head costs 1024 clk of special-function unit (16 ex2/clk/SM) and, at
// D = 128, 1024 clk of tensor pipe.  With one score buffer per CTA the two alternate; with the two query blocks
// of an item sharing each K/V tile, the tensor pipe works on one block while the other is in its softmax, and
// each K/V tile is loaded once for 256 queries.  TMEM: S/P of the two blocks [0,128) [128,256), O [256,256+D) and
// [256+D,256+2D).
//
// Ordinary item (b,h,q1): query blocks q1 and (pair) q1-1; for J = 0..: S_t = Q_t K_J^T, row max / lazy rescale / exp2 /
//   row sum in registers, P_t -> TMEM as bf16 over S_t, O_t += P_t V_J; the next score MMA of a block is queued
//   directly behind the MMA that consumes its P (MMAs of one thread execute in order).  The first scores of the next
//   item go out as soon as block 0 of this one has its last P V MMA, so no softmax warp idles between items.
// Split item: one query block, its even key tiles in the first chain and the odd ones in the second, each with running
//   maximum, row sum and accumulator of its own; chain 1 hands maximum and sum to chain 0, which forms the factors
//   with which the epilogue adds the two accumulators.  It takes half the time of a pair of its length (a pair of tiles 2.2 us
//   either way) but loads every K and V tile for one block: for grids whose longest items would set the time.
// Frozen item, tensor-core form (pattern tables prepared and the head's flag set): with global maxima,
//   O = diag(w) R (diag(a) V), R(i,j) = r(i-j).  A tile of R with reversed rows is a Hankel matrix that the tensor
//   core reads straight from a 4 KB band table (no-swizzle descriptor, both strides 128 bytes), so a tile is two bulk
//   copies of bands, one TMA load of the a-scaled V tile and 16 MMAs; the epilogue scales the finished rows by w(i)
//   (TMEM lane m holds query 127-m of the block).
// Frozen item, general form: P^(i,j) = exp(alpha(j) + rho(i-j) - logZ(i)) for j <= i (Eq. "compact-prior" with the
//   stored normaliser) generated into TMEM by the softmax warps, O_t += P^ V_J.  The exponential is factorised per
//   tile as w(i) a(j) r(i-j) with a = exp(alpha - max_tile alpha), r = exp(rho - max_band rho),
//   w = exp(max alpha + max rho - logZ(i)); a tile whose exponent range would leave fp32 falls back to one exp per
//   element.
#include <cuda_bf16.h>
#include "ptx.cuh"
#include "saf_internal.h"

#ifdef SAF_TRACE
__device__ unsigned long long g_saf_trace_fwd128[3][16384];
#define TRF(role, id)                                                                                  \
  do {                                                                                                 \
    if (blockIdx.x == 0 && (threadIdx.x & 31) == 0 && tr_n < 16380)                                    \
      g_saf_trace_fwd128[role][tr_n++] = (static_cast<unsigned long long>(id) << 48) | (clock64() & 0xffffffffffffULL); \
  } while (0)
extern "C" int saf_debug_read_trace_fwd128(unsigned long long* out) {
  return static_cast<int>(cudaMemcpyFromSymbol(out, g_saf_trace_fwd128, sizeof(g_saf_trace_fwd128)));
}
#else
#define TRF(role, id)
#endif

SAF_SPAN_DEFINE(fwd128)

namespace saf {

namespace {

constexpr float LOG2E_F = 1.4426950408889634f;
constexpr float LN2_F = 0.6931471805599453f;

struct FwdCfg {
  static constexpr int D = 128;                         // (96 runs here with features 96..127 zero-filled by TMA)
  static constexpr int NPANEL = D / 64;                 // 64-column bf16 panels: 128-byte rows, one swizzle atom
  static constexpr int PANEL_BYTES = 128 * 64 * 2;      // 16 KB
  static constexpr int TILE_BYTES = NPANEL * PANEL_BYTES;
  static constexpr int NS = 4;                          // ring of K and V tiles (K_0 V_0 K_1 V_1 ...)
  static constexpr int OFF_Q = 0;                       // Q of the two query blocks (general frozen form: tables)
  static constexpr int OFF_KV = 2 * TILE_BYTES;
  static constexpr int OFF_BAND = OFF_KV + NS * TILE_BYTES;   // 2 x 4 KB of Hankel bands per ring stage
  static constexpr int OFF_LINV = OFF_BAND + NS * 8192;       // [2][128] 1 / row sum
  static constexpr int OFF_XM = OFF_LINV + 2 * 128 * 4;       // [128] split items: chain 1's reference
  static constexpr int OFF_BAR = OFF_XM + 128 * 4;
  static constexpr int NRING = 4;                       // work-item records in flight
  static constexpr int CLAIM_AHEAD = 4;
  static constexpr int NBAR = 2 * NS + 15 + 2 * NRING;
  static constexpr int OFF_RING = (OFF_BAR + NBAR * 8 + 16 + 15) / 16 * 16;
  static constexpr int SMEM = OFF_RING + NRING * 16 + 1024;   // + slack for 1024-byte alignment
  static constexpr int TMEM_COLS = 512;
  static constexpr int COL_S = 0, COL_O = 256;          // + 128 t, + D t
  static constexpr int NTHREADS = 512;
};
constexpr int TAB_FLOATS = 784;                         // one tile's tables of the general frozen form (two buffers)
static_assert(2 * TAB_FLOATS * 4 <= FwdCfg::TILE_BYTES, "the tables fit into a query tile");

enum FwdSite { SITE_Q_EMPTY = 1, SITE_KV_EMPTY, SITE_Q_FULL, SITE_KV_FULL, SITE_P_FULL, SITE_O_FREE, SITE_S_FULL,
               SITE_O_FULL, SITE_L_FULL, SITE_RING_EMPTY, SITE_RING_FULL, SITE_X_FULL };

constexpr int RING_FAST = 1 << 8;
constexpr int RING_END = -1;

// A work item as the roles see it: two chains of score MMA, softmax and P V MMA.  n1 = key tiles of query block `blk`
// (chain 1), n0 = key tiles of query block blk - 1 (chain 0; 0: the item has one query block).  Split: both chains work on
// block `blk`, chain 0 on its even key tiles and chain 1 on the odd ones.  tiles = key tiles loaded.
struct ItemView {
  int b, h, blk, kind, n0, n1, tiles;
  bool fast, split;
};

template <bool SPLIT>
__device__ __forceinline__ bool ring_take(const int4* ring, uint64_t* ring_full, uint64_t* ring_empty, uint32_t n,
                                          const WaitCtx& wc, ItemView& v) {
  const uint32_t slot = n % FwdCfg::NRING;
  if (!mbar_wait_warp_compact(ring_full + slot, (n / FwdCfg::NRING) & 1, wc, SITE_RING_FULL)) return false;
  const int4 raw = ring[slot];
  warp_arrive(ring_empty + slot);
  v.b = raw.x;
  v.h = raw.y;
  v.blk = raw.z;
  v.kind = raw.w < 0 ? RING_END : (raw.w & 0x7f);
  v.fast = raw.w >= 0 && (raw.w & RING_FAST) != 0;
  v.split = SPLIT && raw.w >= 0 && (raw.w & KIND_SPLIT) != 0;
  v.tiles = raw.z + 1;
  v.n1 = v.split ? v.tiles >> 1 : v.tiles;
  v.n0 = v.split ? v.tiles - v.n1 : (raw.w & KIND_PAIR) ? raw.z : 0;
  return true;
}

}  // namespace

// SPLIT: the list holds split items (the issuer's extra conditions cost lists without them 1.6 %, 4x32x4096x128 on shared heads)
template <bool SPLIT>
__global__ void __launch_bounds__(FwdCfg::NTHREADS, 1)
saf_fwd_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
               const __grid_constant__ CUtensorMap mv, const __grid_constant__ CUtensorMap mvt, const FwdParams p) {
  using C = FwdCfg;
  constexpr int D = C::D;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* kv_full = bars;                      // [NS]
  uint64_t* kv_empty = kv_full + C::NS;          // [NS]
  uint64_t* q_full = kv_empty + C::NS;           // [2] Q of block t has landed
  uint64_t* q_empty = q_full + 2;                // [2] the item's last use of Q t's memory has completed
  uint64_t* s_full = q_empty + 2;                // [2] scores of block t (general form: buffer t may be written)
  uint64_t* p_full = s_full + 2;                 // [2] P of block t written (4 warp arrivals)
  uint64_t* o_full = p_full + 2;                 // [2] last MMA into O_t has completed
  uint64_t* o_free = o_full + 2;                 // [2] epilogue has read O_t (4 warp arrivals)
  uint64_t* l_full = o_free + 2;                 // [2] 1 / row sum of block t written (4 warp arrivals)
  uint64_t* x_full = l_full + 2;                 // split items: row sums and references of chain 1 written (4 warp arrivals)
  uint64_t* ring_full = x_full + 1;              // [NRING] record n has been published by the producer
  uint64_t* ring_empty = ring_full + C::NRING;   // [NRING] issuer + 8 softmax warps + 4 epilogue warps have copied it
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ring_empty + C::NRING);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int4* ring = reinterpret_cast<int4*>(smem + C::OFF_RING);
  float* linv = reinterpret_cast<float*>(smem + C::OFF_LINV);
  float* xm = reinterpret_cast<float*>(smem + C::OFF_XM);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const WaitCtx wc{abort_flag, p.status, p.wait_limit_ns};
  SAF_SPAN(fwd128, 0);
#ifdef SAF_TRACE
  int tr_n = 0;
#endif

  if (tid == 0) {
    *abort_flag = 0;
    for (int s = 0; s < C::NS; ++s) {
      mbar_init(kv_full + s, 1);
      mbar_init(kv_empty + s, 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(q_full + t, 1);
      mbar_init(q_empty + t, 1);
      mbar_init(s_full + t, 1);
      mbar_init(p_full + t, 4);
      mbar_init(o_full + t, 1);
      mbar_init(o_free + t, 4);
      mbar_init(l_full + t, 4);
    }
    mbar_init(x_full, 4);
    for (int k = 0; k < C::NRING; ++k) {
      mbar_init(ring_full + k, 1);
      mbar_init(ring_empty + k, 13);
    }
    mbar_fence_init();
  }
  if (warp == 13) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the prologue above overlapped the previous kernel's tail; global memory is touched only from here on
  // On a grid that fills much of the chip the next kernel is let in only once the one in front has ended: let in before, a queue of
  // passes runs two kernels deep and its waiting CTAs hold back the one in front; updates on few CTAs want it at once.  us at once /
  // behind the wait, forwards of 1xHxTx128: 32 CTAs 11.4 / 11.1, 40 11.6 / 11.2, 48 11.8 / 11.7, 56 13.1 / 12.2, 64 12.4 / 11.7, 96 17.0 /
  // 16.1, on shared heads 15.5 / 14.4; updates: 24 33.0 / 34.3, 32 33.2 / 34.5, 36 59.8 / 60.8, 48 35.2 / 35.9, 56 36.6 / 36.6, 72 to
  // 128 the same (52.5 / 52.3, 50.8 / 50.8).
  const bool at_once = gridDim.x <= 48;
  if (at_once) pdl_launch_dependents();
  pdl_wait();
  if (!at_once) pdl_launch_dependents();

  // (each warpgroup sets its register share at the top of its own branch)
  if (warp >= 12) {
    reg_dec<64>();
    if (warp == 12) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0) {
        tma_prefetch_desc(&mq);
        tma_prefetch_desc(&mk);
        tma_prefetch_desc(&mv);
        tma_prefetch_desc(&mvt);
        uint32_t n = 0;                            // ring position
        uint32_t nq0 = 0, nq1 = 0;                 // uses of the two Q areas
        bool ok = true;
        bool drop_load = p.selftest_drop_load != 0;   // (see FwdParams)
        // Claim the next item of the queue and publish it to the other roles.  Claimed CLAIM_AHEAD tiles before the current
        // item's last, but behind the loads of its first two: the claim's global round trips and the loads of Q_0 and K_0
        // behind it then fit under the tiles that are left (claimed behind the item's last load they cost ~13000 clk an item).
        int4 next;
        uint32_t nclaim = 0;
        bool claimed = false;
        auto claim = [&] {
          const uint32_t slot = nclaim % C::NRING;
          ok = mbar_wait_compact(ring_empty + slot, ((nclaim / C::NRING) & 1) ^ 1, wc, SITE_RING_EMPTY);
          if (!ok) return;
          ++nclaim;
          claimed = true;
          // (a CTA's first item is its own number; a grid of one item per CTA does not touch the queue)
          const int grid = static_cast<int>(gridDim.x);
          const int idx = nclaim == 1 ? static_cast<int>(blockIdx.x) : p.n_items <= grid ? p.n_items : grid + atomicAdd(p.queue, 1);
          next = make_int4(0, 0, 0, RING_END);
          if (idx < p.n_items) {
            next = __ldg(reinterpret_cast<const int4*>(p.items + idx));
            if ((next.w & 0x7f) != KIND_ORDINARY && p.band_f != nullptr && __ldg(p.fast_ok + next.y) != 0 &&
                __ldg(p.ovf + next.y) != p.call_id)
              next.w |= RING_FAST;
          }
          if (next.w >= 0 && (next.w & 0x7f) == KIND_ORDINARY) {
            // (its Q tiles are read by no other item, so nobody has brought them into L2)
            const int hq = p.qslot ? p.qslot[next.y] : next.y;
            for (int pn = 0; pn < C::NPANEL; ++pn) {
              if (next.w & KIND_PAIR) tma_prefetch_4d(&mq, pn * 64, (next.z - 1) * BLK, hq, next.x);
              tma_prefetch_4d(&mq, pn * 64, next.z * BLK, hq, next.x);
            }
          }
          ring[slot] = next;
          mbar_arrive(ring_full + slot);                 // (release: the record is visible to whoever sees the phase)
        };
        for (;;) {
          if (!claimed) claim();
          if (!ok || next.w < 0) break;
          const int4 rec = next;
          claimed = false;
          const int b = rec.x, h = rec.y, n1 = rec.z + 1;
          const bool fast = (rec.w & RING_FAST) != 0, pair = (rec.w & KIND_PAIR) != 0;
          auto load_kv = [&](const CUtensorMap* m, int j, int head) {
            const uint32_t s = n % C::NS;
            ok = mbar_wait_compact(kv_empty + s, ((n / C::NS) & 1) ^ 1, wc, SITE_KV_EMPTY);
            if (!ok) return;
            ++n;
            if (drop_load) {
              drop_load = false;
              return;
            }
            mbar_expect_tx(kv_full + s, C::TILE_BYTES);
            for (int pn = 0; pn < C::NPANEL; ++pn)
              tma_load_4d(smem + C::OFF_KV + s * C::TILE_BYTES + pn * C::PANEL_BYTES, m, kv_full + s, pn * 64, j * BLK, head, b);
          };
          if (fast) {
            // tensor-core form: per tile the scaled V tile and the Hankel bands of distance blocks q1 - J, q1 - 1 - J
            const int ord = p.hord[h];
            const uint8_t* bands = static_cast<const uint8_t*>(p.band_f) + static_cast<size_t>(h) * p.nblkp * 4096;
            for (int j = 0; j < n1; ++j) {
              const uint32_t s = n % C::NS;
              ok = mbar_wait_compact(kv_empty + s, ((n / C::NS) & 1) ^ 1, wc, SITE_KV_EMPTY);
              if (!ok) break;
              const int d = n1 - 1 - j;
              const bool two = pair && d > 0;
              mbar_expect_tx(kv_full + s, C::TILE_BYTES + (two ? 8192 : 4096));
              for (int pn = 0; pn < C::NPANEL; ++pn)
                tma_load_4d(smem + C::OFF_KV + s * C::TILE_BYTES + pn * C::PANEL_BYTES, &mvt, kv_full + s, pn * 64, j * BLK,
                            ord, b);
              bulk_load(smem + C::OFF_BAND + s * 8192 + 4096, bands + static_cast<size_t>(d) * 4096, 4096, kv_full + s);
              if (two) bulk_load(smem + C::OFF_BAND + s * 8192, bands + static_cast<size_t>(d - 1) * 4096, 4096, kv_full + s);
              ++n;
              if (!claimed && j + C::CLAIM_AHEAD >= n1 && (j > 0 || n1 == 1)) claim();
              if (!ok) break;
            }
            if (!ok) break;
            continue;
          }
          const int hv = h / p.kv_group;
          if ((rec.w & 0x7f) == KIND_ORDINARY) {
            const int hq = p.qslot ? p.qslot[h] : h, hk = p.qslot ? hq : hv;
            // Q_0 and K_0 first: chain 0's first scores are issued before this item's predecessor has finished with Q_1
            // (a split item has its block's Q in both areas)
            const bool split = SPLIT && (rec.w & KIND_SPLIT) != 0;
            if (pair || split) {
              ok = mbar_wait_compact(q_empty, (nq0 & 1) ^ 1, wc, SITE_Q_EMPTY);
              if (!ok) break;
              mbar_expect_tx(q_full, C::TILE_BYTES);
              for (int pn = 0; pn < C::NPANEL; ++pn)
                tma_load_4d(smem + C::OFF_Q + pn * C::PANEL_BYTES, &mq, q_full, pn * 64, (split ? rec.z : rec.z - 1) * BLK, hq, b);
              ++nq0;
            }
            load_kv(&mk, 0, hk);
            if (!ok) break;
            ok = mbar_wait_compact(q_empty + 1, (nq1 & 1) ^ 1, wc, SITE_Q_EMPTY);
            if (!ok) break;
            mbar_expect_tx(q_full + 1, C::TILE_BYTES);
            for (int pn = 0; pn < C::NPANEL; ++pn)
              tma_load_4d(smem + C::OFF_Q + C::TILE_BYTES + pn * C::PANEL_BYTES, &mq, q_full + 1, pn * 64, rec.z * BLK, hq, b);
            ++nq1;
            // K_0 V_0 K_1 V_1 ...; split: K_0 K_1 V_0 K_2 V_1 ... V_last, in the order of the two chains
            load_kv(split ? &mk : &mv, split ? 1 : 0, split ? hk : hv);
            for (int j = split ? 2 : 1;; ++j) {
              if (ok && split) load_kv(&mv, j - 2, hv);
              if (ok && !claimed && j + C::CLAIM_AHEAD > n1 && (j > 1 || j == n1)) claim();
              if (j == n1 || !ok) break;
              load_kv(&mk, j, hk);
              if (ok && !split) load_kv(&mv, j, hv);
            }
            if (ok && split) load_kv(&mv, n1 - 1, hv);
          } else {
            // general frozen form: the Q areas hold the tables of the softmax warps; an area counts as used by this item
            if (pair) {
              ok = mbar_wait_compact(q_empty, (nq0 & 1) ^ 1, wc, SITE_Q_EMPTY);
              ++nq0;
            }
            if (ok) ok = mbar_wait_compact(q_empty + 1, (nq1 & 1) ^ 1, wc, SITE_Q_EMPTY);
            ++nq1;
            for (int j = 0; j < n1 && ok; ++j) load_kv(&mv, j, hv);
          }
          if (!ok) break;                            // (a given-up item is the last: its tile sequence is broken)
        }
      }
    } else if (warp == 13) {
      // ---------------------------------------------------------------- tcgen05 issuer
      // The whole warp walks the loops (warp-uniform operands); one elected lane issues.
      const bool leader = elect_one() != 0;
      const uint32_t sb = smem_u32(smem);
      constexpr uint32_t idesc_s = umma_idesc_bf16(128, 128, 0, 0);
      // (head dimension 96 runs here with features 96..127 zero-filled by TMA: its MMAs skip the two empty k-steps of
      // the scores and produce only 96 output columns)
      const uint32_t idesc_o = umma_idesc_bf16(128, p.d_real, 0, 1);
      const int nk16 = p.d_real / 16;
      const uint32_t idesc_hk = umma_idesc_f16(128, p.d_real, 0, 1);  // tensor-core frozen form: fp16 band x fp16 scaled V
      // descriptor halves for smem offset 0: K-major tiles (k-step +32 B within a 64-column panel) and
      // the MN-major V tile (k-step +2048 B, LBO = panel stride)
      const uint64_t d_kmaj = umma_smem_desc(sb, 16, 1024, UMMA_LAYOUT_SW128);
      const uint64_t d_mn = umma_smem_desc(sb, C::PANEL_BYTES, 1024, UMMA_LAYOUT_SW128);
      const uint32_t lo_k = desc_lo(d_kmaj), hi_k = desc_hi(d_kmaj), lo_m = desc_lo(d_mn), hi_m = desc_hi(d_mn);
      // Hankel band: no-swizzle K-major, core matrices 128 bytes apart in both directions
      const uint64_t d_band = umma_smem_desc(sb, 128, 128, UMMA_LAYOUT_NONE);
      const uint32_t lo_b = desc_lo(d_band), hi_b = desc_hi(d_band);
      auto kv_wait = [&](uint32_t pos) {
        return mbar_wait_warp_compact(kv_full + pos % C::NS, (pos / C::NS) & 1, wc, SITE_KV_FULL);
      };
      // (the warp converges behind every burst: without that the two bursts of block 0 took 1560 clk instead of 1050)
      auto issue_qk = [&](uint32_t t, uint32_t pos) {
        const uint32_t q_lo = lo_k + ((C::OFF_Q + t * C::TILE_BYTES) >> 4);
        const uint32_t k_lo = lo_k + ((C::OFF_KV + (pos % C::NS) * C::TILE_BYTES) >> 4);
        if (leader) {
#pragma unroll
          for (int kc = 0; kc < D / 16; ++kc) {
            if (kc >= nk16) break;
            const uint32_t off = ((kc >> 2) * C::PANEL_BYTES + (kc & 3) * 32) >> 4;
            umma_ss2(tmem + C::COL_S + 128 * t, q_lo + off, hi_k, k_lo + off, hi_k, idesc_s, kc > 0);
          }
          umma_commit(s_full + t);
        }
        __syncwarp();
      };
      auto issue_pv = [&](uint32_t t, uint32_t pos, uint32_t acc0) {
        const uint32_t v_lo = lo_m + ((C::OFF_KV + (pos % C::NS) * C::TILE_BYTES) >> 4);
        if (leader) {
#pragma unroll
          for (int kc = 0; kc < 8; ++kc)
            umma_ts2(tmem + C::COL_O + D * t, tmem + C::COL_S + 128 * t + 8 * kc, v_lo + 128 * kc, hi_m, idesc_o,
                     kc > 0 ? 1u : acc0);
        }
        __syncwarp();
      };
      // (One copy of each burst and wait, the block t a run-time value: with the bursts inlined per block and case the
      // kernel's code was 133 KB, and every item boundary fetched instructions for ~10000 clk.)
      uint32_t n = 0, nrec = 0;
      uint32_t ph_q = 0, ph_p = 0, ph_o = 3;       // bit t: parity of the next phase of q_full[t], p_full[t], o_free[t]
      auto wait_t = [&](uint64_t* bar, uint32_t& ph, uint32_t t, int site) {
        const bool r = mbar_wait_warp_compact(bar + t, (ph >> t) & 1, wc, site);
        ph ^= 1u << t;
        return r;
      };
      bool early = false;                          // block 0's first scores of `cur` are already issued
      ItemView cur;
      bool ok = ring_take<SPLIT>(ring, ring_full, ring_empty, nrec++, wc, cur);
      while (ok && cur.kind != RING_END) {
        ItemView nxt;
        bool have_next = false;
        const int n0 = cur.n0, n1 = cur.n1, tiles = cur.tiles;
        const bool split = SPLIT && cur.split;
        if (cur.fast) {
          for (int j = 0; j < n1 && ok; ++j, ++n) {
            ok = kv_wait(n);
            const uint32_t s = n % C::NS;
            const uint32_t band_lo = lo_b + ((C::OFF_BAND + s * 8192) >> 4);
            const uint32_t v_lo = lo_m + ((C::OFF_KV + s * C::TILE_BYTES) >> 4);
            const uint32_t acc0 = j > 0 ? 1u : 0u;
#pragma unroll 1
            for (uint32_t t = j < n0 ? 0 : 1; t < 2 && ok; ++t) {
              if (j == 0) ok = wait_t(o_free, ph_o, t, SITE_O_FREE);
              if (!ok) break;
              tc_fence_after();
              if (leader) {
#pragma unroll
                for (int kc = 0; kc < 8; ++kc)
                  umma_ss2(tmem + C::COL_O + D * t, band_lo + 256 * t + 16 * kc, hi_b, v_lo + 128 * kc, hi_m, idesc_hk,
                           kc > 0 ? 1u : acc0);
                if (j == (t ? n1 : n0) - 1) umma_commit(o_full + t);
              }
              __syncwarp();
            }
            if (leader) umma_commit(kv_empty + s);
            __syncwarp();
          }
        } else {
          const bool ord = cur.kind == KIND_ORDINARY;
          if (ord) {
            // first scores
#pragma unroll 1
            for (uint32_t t = n0 > 0 && !early ? 0 : 1; t < 2 && ok; ++t) {
              const uint32_t k0 = split ? n + t : n;
              ok = wait_t(q_full, ph_q, t, SITE_Q_FULL) && kv_wait(k0);
              if (!ok) break;
              tc_fence_after();
              issue_qk(t, k0);
              if (leader && (t ? n1 : n0) == 1) umma_commit(q_empty + t);
            }
            if (leader) {
              umma_commit(kv_empty + n % C::NS);
              if (split) umma_commit(kv_empty + (n + 1) % C::NS);
            }
            early = false;
          } else if (leader) {
            // general frozen form: P^ written by the softmax warps, one P V per block and tile; s_full says that a
            // block's P^ buffer may be written (everything issued before has completed)
            if (n0 > 0) umma_commit(s_full);
            umma_commit(s_full + 1);
          }
          __syncwarp();
          const int steps = split ? n0 : n1;                        // (split: chain 0 has the odd tile, or as many)
          for (int j = 0; j < steps && ok; ++j) {
            uint32_t pv = ord ? n + 2 * j + 1 : n + j;             // ring position of V_j; K_{j+1} follows
            const uint32_t acc0 = j > 0 ? 1u : 0u;
            // the tiles' loads land long before P is ready: test their barriers first, so that only one test
            // stands between "P is ready" and the MMAs that wait for it
            if (!split) ok = kv_wait(pv) && (!ord || j + 1 == n1 || kv_wait(pv + 1));
#pragma unroll 1
            for (uint32_t t = j < n0 ? 0 : 1; t < 2 && ok; ++t) {
              const int nt = t ? n1 : n0;
              if (split) {
                // tile J = 2 j + t of the block: V_J, followed by K_{J+2}
                if (j == nt) break;
                const int J = 2 * j + static_cast<int>(t);
                pv = J + 1 < tiles ? n + 2 + 2 * J : n + 2 * tiles - 1;
                ok = kv_wait(pv) && (j + 1 == nt || kv_wait(pv + 1));
                if (!ok) break;
              }
              if (j == 0) ok = wait_t(o_free, ph_o, t, SITE_O_FREE);
              if (ok) ok = wait_t(p_full, ph_p, t, SITE_P_FULL);
              if (!ok) break;
              tc_fence_after();
              TRF(0, 2 + 2 * t);
              issue_pv(t, pv, acc0);
              if (leader && (t == 1 || split)) umma_commit(kv_empty + pv % C::NS);
              uint32_t pos = pv + 1;
              bool qk = ord && j + 1 < nt, last_qk = j + 2 == nt;
              if (j + 1 == nt) {
                if (leader) {
                  umma_commit(o_full + t);
                  if (!ord) umma_commit(q_empty + t);
                }
                __syncwarp();
                if (ord && t == 0) {
                  // block 0 is through: its first scores of the next item go out now
                  ok = ring_take<SPLIT>(ring, ring_full, ring_empty, nrec++, wc, nxt);
                  if (!ok) break;
                  have_next = true;
                  if (nxt.kind == KIND_ORDINARY && nxt.n0 > 0) {
                    pos = n + 2 * tiles;
                    ok = wait_t(q_full, ph_q, 0, SITE_Q_FULL) && kv_wait(pos);
                    if (!ok) break;
                    tc_fence_after();
                    early = qk = true;
                    last_qk = nxt.n0 == 1;
                  }
                }
              } else if (!ord && leader) {
                umma_commit(s_full + t);
              }
              __syncwarp();
              if (qk) {
                issue_qk(t, pos);                        // executes after P V: same thread, in order
                if (leader) {
                  if ((t == 1 || split) && !(j + 1 == nt)) umma_commit(kv_empty + pos % C::NS);
                  if (last_qk) umma_commit(q_empty + t);
                }
              }
              __syncwarp();
              TRF(0, 3 + 2 * t);
            }
          }
          n += ord ? 2 * tiles : tiles;
        }
        if (!ok) break;
        if (have_next) cur = nxt;
        else ok = ring_take<SPLIT>(ring, ring_full, ring_empty, nrec++, wc, cur);
      }
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------------ softmax warps (2 x 128 threads)
    reg_inc<192>();
    const int q4 = warp & 3, t = warp >> 2;
    const int rowl = q4 * 32 + lane;                   // query row within the block = TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const uint32_t t_s = tmem + lane_base + C::COL_S + 128 * t;       // scores, then bf16 pairs of P in the first 64
    const uint32_t t_o = tmem + lane_base + C::COL_O + D * t;
    const int wg_bar = 1 + t, wg_bar2 = 3 + t;
    uint32_t ns = 0, nof = 0, nx = 0;                  // phases of s_full[t]; items of this chain so far; split ones
    bool ok = true;
    // A softmax warp whose wait was abandoned keeps walking (without storing) until the next
    // agreement barrier, where its four leave together; none is ever left alone at a barrier.
    for (uint32_t nrec = 0;; ++nrec) {
      ItemView w;
      if (!ring_take<SPLIT>(ring, ring_full, ring_empty, nrec, wc, w)) {
        ok = false;
        w.kind = KIND_ORDINARY; w.n0 = w.n1 = w.tiles = 0; w.fast = w.split = false; w.b = w.h = w.blk = 0;
      }
      if (named_bar_or(wg_bar, 128, !ok) || w.kind == RING_END) break;
      const int nt = t == 0 ? w.n0 : w.n1;
      if (nt == 0) continue;
      const int blk = SPLIT && w.split ? w.blk : nt - 1;
      const int row = blk * BLK + rowl;
      if (w.fast) {
        ++nof;
        continue;
      }
      if (w.kind == KIND_ORDINARY) {
        float m_ref = -INFINITY;
        uint64_t l2a = 0, l2b = 0;                     // packed pairs of partial row sums
        const float c = p.scale_log2;
        const uint64_t c2 = pk2(c, c);
        const int j_diag = !(SPLIT && w.split) ? blk : (blk & 1) == t ? blk >> 1 : -1;   // this chain's tile on the diagonal
        for (int j = 0; j < nt; ++j) {
          if (q4 == 0) TRF(1 + t, 11);
          // (the completion of this score MMA also covers the block's previous P V MMA, issued before it)
          if (!mbar_wait_warp_compact(s_full + t, ns & 1, wc, SITE_S_FULL)) ok = false;
          ++ns;
          tc_fence_after();
          if (q4 == 0) TRF(1 + t, 12);
          uint32_t r[4][32];
          tmem_ld32(t_s, r[0]);
          tmem_ld32(t_s + 32, r[1]);
          tmem_wait_ld();
          tmem_ld32(t_s + 64, r[2]);
          tmem_ld32(t_s + 96, r[3]);
          if (j == j_diag) {
#pragma unroll
            for (int e = 0; e < 64; ++e)
              if (e > rowl) r[e >> 5][e & 31] = 0xff800000u;          // -inf above the diagonal
          }
          // (four chains of three-input maxima: two chains of 64 two-input ones cost ~300 clk of latency a tile)
          float mx[4];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            mx[2 * k] = fmaxf(__uint_as_float(r[k][0]), __uint_as_float(r[k][1]));
            mx[2 * k + 1] = fmaxf(__uint_as_float(r[k][2]), __uint_as_float(r[k][3]));
          }
#pragma unroll
          for (int e = 4; e < 32; e += 4)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mx[k] = max3(mx[k], __uint_as_float(r[k >> 1][e + 2 * (k & 1)]), __uint_as_float(r[k >> 1][e + 2 * (k & 1) + 1]));
          tmem_wait_ld();
          if (j == j_diag) {
#pragma unroll
            for (int e = 64; e < 128; ++e)
              if (e > rowl) r[e >> 5][e & 31] = 0xff800000u;
          }
#pragma unroll
          for (int e = 0; e < 32; e += 4)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mx[k] = max3(mx[k], __uint_as_float(r[2 + (k >> 1)][e + 2 * (k & 1)]), __uint_as_float(r[2 + (k >> 1)][e + 2 * (k & 1) + 1]));
          if (q4 == 0) TRF(1 + t, 13);
          const float m_new = fmaxf(m_ref, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * c);
          if (j == 0) {
            m_ref = m_new;
          } else {
            const bool need = (m_new - m_ref) > 8.0f;
            if (__any_sync(0xffffffffu, need)) {
              const float f = need ? ex2_approx(m_ref - m_new) : 1.0f;
              l2a = mul2(l2a, pk2(f, f));
              l2b = mul2(l2b, pk2(f, f));
              if (need) m_ref = m_new;
#pragma unroll 1
              for (int cc = 0; cc < D / 16; ++cc) {
                uint32_t o[16];
                tmem_ld16(t_o + 16 * cc, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * f);
                tmem_st16(t_o + 16 * cc, o);
              }
            }
          }
          // (the second chain of a split block does not start at key 0: all its scores of a row so far may be -inf, by overflow of
          // Q K^T; they count zero then, and a finite maximum later scales sums and accumulator, zeros so far, by zero)
          const float neg_m = SPLIT && m_ref == -INFINITY ? 0.0f : -m_ref;
          const uint64_t nm2 = pk2(neg_m, neg_m);
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const uint64_t x2 = fma2(pk2(__uint_as_float(r[cc][2 * e]), __uint_as_float(r[cc][2 * e + 1])), c2, nm2);
              float a0, a1;
              upk2(x2, a0, a1);
              a0 = ex2_approx(a0);
              a1 = ex2_approx(a1);
              const uint64_t a2 = pk2(a0, a1);
              if (e & 1) l2b = add2(l2b, a2);
              else l2a = add2(l2a, a2);
              pk[e] = pack_bf16x2(a0, a1);
            }
            tmem_st16(t_s + 16 * cc, pk);
          }
          if (q4 == 0) TRF(1 + t, 14);
          tmem_wait_st();
          tc_fence_before();
          warp_arrive(p_full + t);
          if (q4 == 0) TRF(1 + t, 15);
        }
        float la, lb, lc, ld;
        upk2(l2a, la, lb);
        upk2(l2b, lc, ld);
        const float l = (la + lb) + (lc + ld);
        // the epilogue has read the previous item's row sums once it has released O_t
        if (nof > 0 && !mbar_wait_warp_compact(o_free + t, (nof - 1) & 1, wc, SITE_O_FREE)) ok = false;
        float m_all = m_ref, l_all = l;
        if (!SPLIT || !w.split) {
          linv[t * 128 + rowl] = 1.0f / l;
          warp_arrive(l_full + t);
        } else if (t == 1) {
          // chain 1 hands its row sums and references to chain 0, which forms the two accumulators' factors
          linv[128 + rowl] = l;
          xm[rowl] = m_ref;
          warp_arrive(x_full);
        } else {
          if (!mbar_wait_warp_compact(x_full, nx++ & 1, wc, SITE_X_FULL)) ok = false;
          const float l1 = linv[128 + rowl], m1 = xm[rowl];
          m_all = fmaxf(m_ref, m1);
          const float f0 = ex2_approx(m_ref - m_all), f1 = ex2_approx(m1 - m_all);   // (NaN where no chain has a finite score)
          l_all = fmaf(f0, l, f1 * l1);
          linv[rowl] = f0 / l_all;
          linv[128 + rowl] = f1 / l_all;
          warp_arrive(l_full);
        }
        if (p.LSE != nullptr && row < p.T && ok && !(SPLIT && w.split && t == 1))
          p.LSE[(static_cast<size_t>(w.b) * p.H + w.h) * p.T + row] = (m_all + log2f(l_all)) * LN2_F;
      } else {
        // ---------------- frozen head, general form: generate P^ tiles
        const int wt = tid & 127;
        const float* alpha_h = p.alpha + static_cast<size_t>(w.h) * p.Tp;
        const float* rho_h = p.rho + static_cast<size_t>(w.h) * p.Tp;
        const float z2 = (row < p.T) ? p.logZ[static_cast<size_t>(w.h) * p.Tp + row] * LOG2E_F : INFINITY;
        // A tile's table entries are fetched one tile ahead and its tables are made while the previous tile's P^ V is
        // still running.  Fetched and filled behind that wait, a tile was one serial chain (4 heads x 8192 x 128, one
        // head of this form, so that its last item sets the time: 184 us, 154 with the fetch ahead, 142 with both).
        float a_next = 0.0f, r_next[2] = {0.0f, 0.0f};
        auto fetch = [&](int j) {
          const int key = j * BLK + wt;
          a_next = key < p.T ? alpha_h[key] : -INFINITY;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int x = wt + 128 * k, d = (blk - j) * BLK - 127 + x;     // band covers distances d0 .. d0+254
            r_next[k] = x < 255 && d >= 0 && d < p.T ? rho_h[d] : -INFINITY;
          }
        };
        // P^ buffer free (first tile: everything issued before this item has completed, which also frees the tables'
        // memory); the four warps agree whether to go on.  Past the agreement of tile j every reader of tile j - 1's
        // tables is done with them, so two buffers suffice.
        auto p_free = [&]() {
          if (!mbar_wait_warp_compact(s_full + t, ns & 1, wc, SITE_S_FULL)) ok = false;
          ++ns;
          tc_fence_after();
          if (named_bar_or(wg_bar, 128, !ok)) ok = false;
          return ok;
        };
        fetch(0);
        bool stay = p_free();
        for (int j = 0; j < nt && stay; ++j) {
          float* tab = reinterpret_cast<float*>(smem + C::OFF_Q + t * C::TILE_BYTES) + (j & 1) * TAB_FLOATS;
          float* aJ = tab;                             // [128] a of the tile's keys
          float* rband = tab + 128;                    // [256] r of the tile's distances
          float* a2raw = tab + 384;                    // [128]
          float* r2raw = tab + 512;                    // [256]
          float* red = tab + 768;                      // [8]
          const float a2 = a_next * LOG2E_F, r2[2] = {r_next[0] * LOG2E_F, r_next[1] * LOG2E_F};
          a2raw[wt] = a2;
          r2raw[wt] = r2[0];
          r2raw[wt + 128] = r2[1];
          float ma = a2, mr = fmaxf(r2[0], r2[1]);
          if (j + 1 < nt) fetch(j + 1);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
            mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
          }
          if (lane == 0) {
            red[q4] = ma;
            red[4 + q4] = mr;
          }
          named_bar_sync(wg_bar2, 128);
          ma = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
          mr = fmaxf(fmaxf(red[4], red[5]), fmaxf(red[6], red[7]));
          const float ew = ma + mr - z2;               // -inf for rows beyond T
          aJ[wt] = ex2_approx(a2 - ma);
          rband[wt] = ex2_approx(r2[0] - mr);
          rband[wt + 128] = ex2_approx(r2[1] - mr);
          // (agreement on the form: the factorised one would overflow or flush for some row)
          const bool exact = named_bar_or(wg_bar2, 128, ew > 100.0f);
          if (j > 0 && !(stay = p_free())) break;
#pragma unroll 1
          for (int cc = 0; cc < 4; ++cc) {
            uint32_t pk[16];
            if (!exact) {
              const float wv = ex2_approx(ew);
              const float* rb = rband + rowl + 127;    // rb[-k] = r(distance of key k in this tile)
#pragma unroll
              for (int e4 = 0; e4 < 8; ++e4) {
                const int k0 = 32 * cc + 4 * e4;
                const float4 a4 = *reinterpret_cast<const float4*>(aJ + k0);
                const float p0 = wv * a4.x * rb[-k0], p1 = wv * a4.y * rb[-k0 - 1];
                const float p2 = wv * a4.z * rb[-k0 - 2], p3 = wv * a4.w * rb[-k0 - 3];
                pk[2 * e4] = pack_bf16x2(p0, p1);
                pk[2 * e4 + 1] = pack_bf16x2(p2, p3);
              }
            } else {
              const float* rb = r2raw + rowl + 127;
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const int k0 = 32 * cc + 2 * e;
                const float p0 = ex2_approx(a2raw[k0] + rb[-k0] - z2);
                const float p1 = ex2_approx(a2raw[k0 + 1] + rb[-k0 - 1] - z2);
                pk[e] = pack_bf16x2(p0, p1);
              }
            }
            tmem_st16(t_s + 16 * cc, pk);
          }
          tmem_wait_st();
          tc_fence_before();
          fence_proxy_async_smem();                    // the tables' memory is a TMA destination of a later item
          warp_arrive(p_full + t);
        }
        if (!stay) break;
      }
      ++nof;
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps
    reg_dec<64>();
    const int q4 = warp & 3;
    const int rowl = q4 * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    uint32_t nof0 = 0, nof1 = 0, nl0 = 0, nl1 = 0;
    bool ok = true;
    for (uint32_t nrec = 0; ok; ++nrec) {
      ItemView w;
      ok = ring_take<SPLIT>(ring, ring_full, ring_empty, nrec, wc, w);
      if (!ok || w.kind == RING_END) break;
      if (SPLIT && w.split) {
        // both accumulators of the block, each times its factor
        ok = mbar_wait_warp_compact(l_full, nl0++ & 1, wc, SITE_L_FULL);
        if (!ok) break;
        const float f0 = linv[rowl], f1 = linv[128 + rowl];
        ok = mbar_wait_warp_compact(o_full, nof0++ & 1, wc, SITE_O_FULL) && mbar_wait_warp_compact(o_full + 1, nof1++ & 1, wc, SITE_O_FULL);
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_o = tmem + lane_base + C::COL_O;
        const int row = w.blk * BLK + rowl;
        const int64_t off = w.b * p.o_strides[0] + w.h * p.o_strides[1] + static_cast<int64_t>(row) * p.o_strides[2];
#pragma unroll 1
        for (int cc = 0; cc < D / 16; ++cc) {
          uint32_t r0[16], r1[16];
          tmem_ld16(t_o + 16 * cc, r0);
          tmem_ld16(t_o + D + 16 * cc, r1);
          tmem_wait_ld();
          if (cc == D / 16 - 1) {
            tc_fence_before();
            warp_arrive(o_free);
            warp_arrive(o_free + 1);
          }
          if (row < p.T && 16 * cc < p.d_real) {
#pragma unroll
            for (int e = 0; e < 16; ++e) r0[e] = __float_as_uint(fmaf(__uint_as_float(r0[e]), f0, __uint_as_float(r1[e]) * f1));
            if (p.o_f32) {
              uint4* orow = reinterpret_cast<uint4*>(static_cast<float*>(p.O) + off + 16 * cc);
#pragma unroll
              for (int g = 0; g < 4; ++g) orow[g] = make_uint4(r0[4 * g], r0[4 * g + 1], r0[4 * g + 2], r0[4 * g + 3]);
            } else {
              uint4* orow = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.O) + off + 16 * cc);
#pragma unroll
              for (int g = 0; g < 2; ++g) {
                uint4 o;
                o.x = pack_bf16x2(__uint_as_float(r0[8 * g + 0]), __uint_as_float(r0[8 * g + 1]));
                o.y = pack_bf16x2(__uint_as_float(r0[8 * g + 2]), __uint_as_float(r0[8 * g + 3]));
                o.z = pack_bf16x2(__uint_as_float(r0[8 * g + 4]), __uint_as_float(r0[8 * g + 5]));
                o.w = pack_bf16x2(__uint_as_float(r0[8 * g + 6]), __uint_as_float(r0[8 * g + 7]));
                orow[g] = o;
              }
            }
          }
        }
        continue;
      }
#pragma unroll 1
      for (int t = 0; t < 2 && ok; ++t) {
        const int nt = t == 0 ? w.n0 : w.n1;
        if (nt == 0) continue;
        const int blk = nt - 1;
        int row = blk * BLK + rowl;
        float f = 1.0f;
        if (w.fast) {
          row = blk * BLK + 127 - rowl;                // tensor-core form: lane m holds query 127-m, scaled by w(i)
          f = (row < p.T) ? p.wvec[static_cast<size_t>(w.h) * p.Tp + row] * (1.0f / (HK_BAND_SCALE * HK_A_SCALE)) : 0.0f;
        } else if (w.kind == KIND_ORDINARY) {
          ok = mbar_wait_warp_compact(l_full + t, (t == 0 ? nl0++ : nl1++) & 1, wc, SITE_L_FULL);
          if (!ok) break;
          f = linv[t * 128 + rowl];
        }
        ok = mbar_wait_warp_compact(o_full + t, (t == 0 ? nof0++ : nof1++) & 1, wc, SITE_O_FULL);
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_o = tmem + lane_base + C::COL_O + D * t;
        const int64_t off = w.b * p.o_strides[0] + w.h * p.o_strides[1] + static_cast<int64_t>(row) * p.o_strides[2];
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          uint32_t r[32];
          tmem_ld32(t_o + 32 * cc, r);
          tmem_wait_ld();
          if (cc == D / 32 - 1) {
            tc_fence_before();
            warp_arrive(o_free + t);                   // the accumulator and linv may be overwritten
          }
          if (row < p.T && 32 * cc < p.d_real) {
            if (p.o_f32) {
              float* orow = static_cast<float*>(p.O) + off + 32 * cc;
#pragma unroll
              for (int g = 0; g < 8; ++g)
                *reinterpret_cast<float4*>(orow + 4 * g) =
                    make_float4(__uint_as_float(r[4 * g + 0]) * f, __uint_as_float(r[4 * g + 1]) * f,
                                __uint_as_float(r[4 * g + 2]) * f, __uint_as_float(r[4 * g + 3]) * f);
            } else {
              __nv_bfloat16* orow = static_cast<__nv_bfloat16*>(p.O) + off + 32 * cc;
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                uint4 o;
                o.x = pack_bf16x2(__uint_as_float(r[8 * g + 0]) * f, __uint_as_float(r[8 * g + 1]) * f);
                o.y = pack_bf16x2(__uint_as_float(r[8 * g + 2]) * f, __uint_as_float(r[8 * g + 3]) * f);
                o.z = pack_bf16x2(__uint_as_float(r[8 * g + 4]) * f, __uint_as_float(r[8 * g + 5]) * f);
                o.w = pack_bf16x2(__uint_as_float(r[8 * g + 6]) * f, __uint_as_float(r[8 * g + 7]) * f);
                *reinterpret_cast<uint4*>(orow + 8 * g) = o;
              }
            }
          }
        }
        if (w.kind != KIND_ORDINARY && p.LSE != nullptr && row < p.T)
          p.LSE[(static_cast<size_t>(w.b) * p.H + w.h) * p.T + row] = 0.0f;
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
  SAF_SPAN(fwd128, 1);
  if (warp == 13) tmem_dealloc(tmem, C::TMEM_COLS);
  if (tid == 0 && p.n_items > static_cast<int>(gridDim.x)) {
    // this CTA claims nothing more; the last CTA to get here rewinds the queue for the next launch
    __threadfence();
    if (atomicAdd(p.queue + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      p.queue[0] = 0;
      p.queue[1] = 0;
      __threadfence();
    }
  }
}

cudaError_t launch_fwd(int D, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                       const CUtensorMap& mvt, const CUtensorMap& mo, const FwdParams& p, int grid, cudaStream_t st) {
  if (D == 64) return launch_fwd64(mq, mk, mv, mvt, mo, p, grid, st);   // head dimension 64 has its own kernel
  auto kern = p.split ? saf_fwd_kernel<true> : saf_fwd_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdCfg::SMEM);
  if (e != cudaSuccess) return e;
  return launch_pdl(PDL_FWD128, kern, dim3(grid), dim3(FwdCfg::NTHREADS), FwdCfg::SMEM, st, mq, mk, mv,
                    mvt, p);
}

}  // namespace saf
