// A run of prefill chunks of a bf16 layer (F = 64) as ONE kernel, for units with many queries or many units: a cluster of
// A + N thread blocks carries one (batch row, KV head) unit through all chunks of the run.
//
//   A attention blocks   Eq. 14 for the chunk's queries, two query tiles of 128 rows (two heads x 64 tokens each) at a time
//   N scoring blocks     Eq. 10 for their tiles of E, two groups of 256 threads on a tile each; then, every block for itself,
//                        the selection (Eq. 12) and dH = phi^T V of the folded pairs; each adds the d / N columns of dH
//                        it owns to H in memory and copies their bf16 operand rows to all blocks
//
// What bounds it: as three dependent launches a chunk of 64 tokens of 64 units took 34.5 us (d = 128, 896 pairs): attention
// 24 us beside scoring and selection 25 us, then the fold 8.5 us, each with its own set-up.  Here the set-up happens
// once, the fold runs beside the attention, and only the moves of pairs wait for it: 27 us a chunk in a run (chunks of 256
// tokens, 16 units: 51 -> 30 us).  Per chunk the cluster meets at an
// mbarrier that counts the scores (scoring blocks), at a cluster barrier (A) when every block has read all it needs of
// the old memories, and at one when the new memories are written.
// Every wait on an mbarrier is bounded; a wait that runs out sets bit 512 of the status word.
#pragma once
#include <cuda.h>

#include "lola_generic.cuh"
#include "lola_run_tc.cuh"
#include "lola_score2_tc.cuh"
#include "lola_select.cuh"
#include "lola_tc.cuh"

namespace lola {

constexpr int kTeamThreads = 576;
constexpr int kTeamMaxE = 2048;      // eligible pairs of a unit
constexpr int kTeamMaxN = 256;       // tokens per chunk

struct TeamMaps {
  tc::SlotMaps gk, gv;
  CUtensorMap wk, wv, q, k, v, out;
};

struct TeamAttMisc {
  uint64_t bars[20];
  float s_vec[128];
  float hx[2][2][128];               // [query tile][half][row]: row maxima of the two halves of a key tile, then the denominators
  uint32_t tmem_slot;
  int abort_word;
};
struct TeamScoreMisc {
  alignas(16) unsigned key[kTeamMaxE];   // score bits of E
  short cand[kTeamMaxE];             // scratch of the selection
  unsigned char mark[kTeamMaxE];
  short fold[kTeamMaxN];             // E indices of the folded pairs
  short dst[kTeamMaxN];              // per leaving pair: slot it takes, or -1
  SelectScratch sel;
  alignas(16) float s[128];          // the normaliser state, fp32 (the same in every scoring block)
  float ssp[2][128];
  float2 phx[2][2][128];             // fold: maximum and sum of a thread's 32 features
  uint64_t bars[16];
  uint32_t tmem_slot;
  int abort_word;
};

template <int DPL>
struct TeamSmem {
  static constexpr int d = DPL * 32;
  // attention block
  static constexpr uint32_t q = 0;                                   // 2 x [kblk][128][128B]; the outputs on their way out
  static constexpr uint32_t stage0 = 65536;                          // 2 x (K 32 KB + V 32 KB)
  static constexpr uint32_t st_v = 32768, stage_bytes = 65536;
  static constexpr uint32_t aht = stage0 + 2 * stage_bytes;          // H^T operand image [2 j blocks][d][128B]
  static constexpr uint32_t aht_blk = d * 128;
  static constexpr uint32_t amisc = aht + 32768;
  static constexpr uint32_t atotal = amisc + (uint32_t)sizeof(TeamAttMisc);
  // scoring block
  static constexpr uint32_t wt = 0;                                  // W^T, K-major [kblk][64][128B]
  static constexpr uint32_t ht = 16384;                              // [H^T ; s_hi ; s_lo], K-major [2 j blocks][d + 16][128B]
  static constexpr uint32_t ht_blk = (d + 16) * 128;
  static constexpr uint32_t grp0 = ht + 36864;                       // per group K tile 32 KB, V tile 32 KB; then the fold's tiles
  static constexpr uint32_t fold_k = grp0, fold_v = grp0 + 32768;    // K_S then phi [2][128][128B]; [V_S | 1] [kblk + 1][128][128B], pairs in rows 0-63
  static constexpr uint32_t hrow0 = fold_v + 3 * 16384;              // this block's columns of H, fp32 [128][d / N]: 48 KB here ...
  static constexpr uint32_t smisc = grp0 + 2 * 65536;
  static constexpr uint32_t hrow1 = (smisc + (uint32_t)sizeof(TeamScoreMisc) + 127) / 128 * 128;   // ... the rest here
  static constexpr uint32_t stotal = hrow1 + 16384;
  static constexpr uint32_t bytes = 232448;                          // all of an SM's shared memory; the base is aligned at run time
};
static_assert(TeamSmem<4>::atotal <= 232448 && TeamSmem<4>::stotal <= 232448 && TeamSmem<4>::ht % 1024 == 0 && TeamSmem<4>::grp0 % 1024 == 0, "shared memory");

// barriers of an attention block: queries there / free, key and value stages full / empty, scores there, weights ready,
// output products complete, the scoring blocks' rows of the H image there
enum { TA_QFULL = 0, TA_QFREE = 1, TA_KFULL = 2, TA_VFULL = 4, TA_KEMPTY = 6, TA_VEMPTY = 8, TA_SFULL = 10, TA_PREADY = 12, TA_ODONE = 14, TA_H = 16, TA_N = 17 };
// ... of a scoring block (one of each pair per group): tiles full / empty, [P | den] complete; scores of all; fold product;
// the others' rows of the H image; U complete
enum { TS_KFULL = 0, TS_VFULL = 2, TS_KEMPTY = 4, TS_VEMPTY = 6, TS_S = 8, TS_SCORES = 10, TS_FOLD = 11, TS_H = 12, TS_U = 13, TS_N = 15 };

// LONG: for chunks of more than 64 tokens, and for runs with chunks whose fold takes phi in three parts (see k_prefill_run)
template <int DPL, bool LONG>
__global__ void __launch_bounds__(kTeamThreads, 1)
k_prefill_team(Layer L, Call c, int n_chunks, const __grid_constant__ TeamMaps M, const uint4* wt_image, int A) {
  using S = TeamSmem<DPL>;
  constexpr int d = DPL * 32, kblk = d / 64, D = 128;
  constexpr float kLog2e = 1.4426950408889634f;
  typedef __nv_bfloat16 T;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = tc::smem_u32(sm);
  TeamAttMisc& XA = *reinterpret_cast<TeamAttMisc*>(sm + S::amisc);
  TeamScoreMisc& X = *reinterpret_cast<TeamScoreMisc*>(sm + S::smisc);

  const int K = (int)tc::cluster_size(), rank = (int)tc::cluster_rank(), N = K - A, sr = rank - A;
  const bool att = rank < A;
  const int unit = blockIdx.x / K, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gr = warp >> 3, hf = (warp >> 2) & 1, wq = warp & 3;
  const int t = wq * 32 + lane;                       // row of a tile = tensor-memory lane
  const int lam = L.lam, eta = L.eta, g = L.g, n = c.n;
  const bool want_out = c.out != nullptr;
  const uint32_t bar0 = sbase + (att ? S::amisc + (uint32_t)offsetof(TeamAttMisc, bars) : S::smisc + (uint32_t)offsetof(TeamScoreMisc, bars));
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  int* abort_word = att ? &XA.abort_word : &X.abort_word;
  uint32_t* tmem_slot = att ? &XA.tmem_slot : &X.tmem_slot;
  volatile int* abw = abort_word;
  bool ok = true;
  auto WAIT = [&](int i, uint32_t parity) { ok = tc::mbar_wait(BAR(i), parity, abw) && ok; };
  float* scu = L.score + (size_t)unit * (lam + L.cmax);
  float* Hg = L.H + (size_t)unit * D * d;

  if (tid == 0) {
    if (att)
      for (int i = 0; i < TA_N; ++i) tc::mbar_init(BAR(i), i == TA_QFREE ? 2u : i == TA_PREADY || i == TA_PREADY + 1 ? 256u : 1u);
    else
      for (int i = 0; i < TS_N; ++i) tc::mbar_init(BAR(i), 1u);
    tc::mbar_init_fence();
    tc::grid_dep_launch_dependents();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, 512);
  if (!att)
    for (int i = tid; i < kblk * 512; i += kTeamThreads) *reinterpret_cast<uint4*>(sm + S::wt + i * 16) = wt_image[(size_t)h * kblk * 512 + i];
  tc::grid_dep_wait();                                // everything before this kernel in the stream is complete
  const bool fits = (uint32_t)(sm - smem_raw) + max(S::atotal, S::stotal) <= S::bytes;   // (a misaligned window cannot happen)
  if (!fits && tid == 0) atomicOr(L.status, 512);
  // an earlier kernel failed: do nothing.  All blocks of a cluster take the first one's word for it
  if (tid == 0) *abort_word = state_failed(L) || !fits ? 1 : 0;
  // H -> bf16 operand image, s (scoring blocks: and its two bf16 rows)
  if (fits) {
    const uint32_t img = att ? S::aht : S::ht, blk = att ? S::aht_blk : S::ht_blk;
    for (int it = tid; it < d * 16; it += kTeamThreads) {
      const int cc = it % d, jc = it / d;
      float hv[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) hv[j] = Hg[(size_t)(jc * 8 + j) * d + cc];
      *reinterpret_cast<uint4*>(sm + img + (jc >> 3) * blk + tc::sw128_off(cc, jc & 7)) = tc::pack8_bf16(hv);
    }
  }
  auto put_s = [&](int j, float sv) {
    const T hi = __float2bfloat16_rn(sv), lo = __float2bfloat16_rn(sv - __bfloat162float(hi));
    const int ch = (j & 63) >> 3;
    X.s[j] = sv;
    *reinterpret_cast<T*>(sm + S::ht + (j >> 6) * S::ht_blk + tc::sw128_off(d, ch) + (j & 7) * 2) = hi;
    *reinterpret_cast<T*>(sm + S::ht + (j >> 6) * S::ht_blk + tc::sw128_off(d + 1, ch) + (j & 7) * 2) = lo;
  };
  if (fits) {
    if (att) {
      if (tid < D) XA.s_vec[tid] = L.s[(size_t)unit * D + tid];
    } else {
      if (tid < D) put_s(tid, L.s[(size_t)unit * D + tid]);
      for (int i = tid; i < 2 * 14 * 8; i += kTeamThreads)   // operand rows d + 2 .. d + 15
        *reinterpret_cast<uint4*>(sm + S::ht + (i / 112) * S::ht_blk + tc::sw128_off(d + 2 + (i / 8) % 14, i % 8)) = make_uint4(0, 0, 0, 0);
    }
  }
  tc::fence_async_all();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  if (tc::cluster_failed(sbase + S::amisc + (uint32_t)offsetof(TeamAttMisc, abort_word))) {   // (and the barriers of all blocks are initialised)
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
    return;
  }
  if (tid == 0) *abw = 0;
  __syncthreads();

  const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
  // query tiles of a chunk: blocks of 64 tokens (the last first: they see the most keys) x pairs of head pairs
  const int ntb = (n + 63) / 64, nqt = (g + 1) / 2, nqc = (nqt + 1) / 2, items = want_out ? ntb * nqc : 0;
  int n_seen = c.n_seen;
  // running counts; every role keeps its own
  uint32_t ke = 0, ve = 0, ni = 0;                    // attention: entries of the key ring and of the value ring, items
  uint32_t cs[2] = {0, 0};                            // attention: score products of the query tiles
  uint32_t ph_h = 0;                                  // phases of TA_H / TS_H
  uint32_t en = 0, ph_sc = 0, ph_f = 0;               // scoring: tiles of this group; phases of TS_SCORES, TS_FOLD

#pragma unroll 1
  for (int chunk = 0; chunk < n_chunks; ++chunk) {
    plan_call(L, c, n_seen, n, false);
    const int cg = c.count_g, cw = c.att_wn, att_g = c.att_g, nE = cg + c.r;
    const bool sel = c.mode == UPD_SELECT;
    const int nF = sel ? nE - lam : 0;
    const int nGB = (cg + 63) / 64, nRB = (cw + 63) / 64;

    if (att) {
      if (warp == 17) {
        // =============================== TMA producer ===============================
        // an item's queries and, as an entry of the key ring, W^T: neither depends on the memories
        auto start_item = [&](int it, int ch) {
          if (ni > 0) WAIT(TA_QFREE, (ni - 1) & 1);
          if (!ok) return;                             // (a wait gave up: nothing more is requested)
          ++ni;
          const int qt0 = (it % nqc) * 2, nw = min(2, nqt - qt0), tok0 = (ntb - 1 - it / nqc) * 64;
          tc::mbar_expect_tx(BAR(TA_QFULL), (uint32_t)nw * kblk * 16384u);
#pragma unroll 1
          for (int x = 0; x < nw * 2; ++x) {
            const int hl = qt0 * 2 + x, head = hl < g ? h * g + hl : L.Hq;   // (a head index outside the tensor reads as zeros)
#pragma unroll
            for (int cb = 0; cb < kblk; ++cb)
              tc::tma_load_5d(sbase + S::q + (uint32_t)(x >> 1) * 32768u + (uint32_t)cb * 16384u + (uint32_t)(x & 1) * 8192u, &M.q, cb * 64, head, tok0, b, ch, BAR(TA_QFULL));
          }
          const uint32_t st = ke & 1;
          if (ke >= 2) WAIT(TA_KEMPTY + st, ((ke >> 1) & 1) ^ 1);
          if (!ok) return;
          tc::mbar_expect_tx(BAR(TA_KFULL + st), (uint32_t)kblk * 8192u);
          tc::bulk_copy_g2s(sbase + S::stage0 + st * S::stage_bytes, wt_image + (size_t)h * kblk * 512, kblk * 8192u, BAR(TA_KFULL + st));
          ++ke;
        };
        if (tc::elect_one()) {
          if (chunk == 0 && rank < items) start_item(rank, 0);
#pragma unroll 1
          for (int it = rank; it < items; it += A) {
            const int tb = ntb - 1 - it / nqc, NT = (nGB + nRB + tb + 2) / 2;
#pragma unroll 1
            for (int kt = 0; kt < NT; ++kt) {
#pragma unroll 1
              for (int isv = 0; isv < 2; ++isv) {
                const uint32_t e = isv ? ve : ke, st = e & 1, bar = BAR((isv ? TA_VFULL : TA_KFULL) + st);
                if (e >= 2) WAIT((isv ? TA_VEMPTY : TA_KEMPTY) + st, ((e >> 1) & 1) ^ 1);
                if (!ok) break;
                tc::mbar_expect_tx(bar, (uint32_t)kblk * 16384u);
                const uint32_t dst = sbase + S::stage0 + st * S::stage_bytes + (isv ? S::st_v : 0u);
                const bool whole = kt * 2 + 1 < nGB;
                if (whole) tc::tma_load_slots(dst, isv ? &M.gv : &M.gk, kt, unit, bar);
#pragma unroll 1
                for (int hb = whole ? 2 : 0; hb < 2; ++hb) {
                  const int blk = kt * 2 + hb;
#pragma unroll
                  for (int cb = 0; cb < kblk; ++cb) {
                    const uint32_t dd = dst + (uint32_t)cb * 16384u + (uint32_t)hb * 8192u;
                    if (blk < nGB) tc::tma_load_3d(dd, isv ? &M.gv.block : &M.gk.block, cb * 64, blk * 64, unit, bar);
                    else if (blk < nGB + nRB) tc::tma_load_3d(dd, isv ? &M.wv : &M.wk, cb * 64, (blk - nGB) * 64, unit, bar);
                    else tc::tma_load_5d(dd, isv ? &M.v : &M.k, cb * 64, h, (blk - nGB - nRB) * 64, b, chunk, bar);   // (beyond the chunk: zeros)
                  }
                }
                if (isv) ++ve; else ++ke;
              }
            }
            if (it + A < items) start_item(it + A, chunk);
          }
        }
        __syncwarp();
        tc::cluster_arrive();                          // (A)
        if (chunk + 1 < n_chunks && rank < items && tc::elect_one()) start_item(rank, chunk + 1);
        __syncwarp();
      } else if (warp == 16) {
        // =============================== MMA issuer ===============================
        const uint32_t idesc_s = tc::make_idesc_bf16(128, 128, false, false), idesc_pv = tc::make_idesc_bf16(128, d, false, true);
        const uint64_t dq = tc::make_desc_sw128(sbase + S::q, 16, 1024), dk = tc::make_desc_sw128(sbase + S::stage0, 16, 1024);
        const uint64_t dv = tc::make_desc_sw128(sbase + S::stage0 + S::st_v, 16384, 1024), dh = tc::make_desc_sw128(sbase + S::aht, 16, 1024);
        auto issue_s = [&](int w, uint32_t st) {
#pragma unroll
          for (int ks = 0; ks < d / 16; ++ks) {
            const uint64_t off = (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
            tc::mma_bf16_ss(tmem + (uint32_t)w * 128u, dq + (uint64_t)(w * 2048) + off, dk + (uint64_t)(st * (S::stage_bytes >> 4)) + off, idesc_s, ks > 0);
          }
          tc::mma_commit(BAR(TA_SFULL + w));
        };
        // U_w = Q_w W over the score columns of the item's query tiles
        auto issue_u = [&](int it) {
          const int nw = min(2, nqt - (it % nqc) * 2);
          const uint32_t st = ke & 1;
          WAIT(TA_QFULL, ni & 1);
          ++ni;
          WAIT(TA_KFULL + st, (ke >> 1) & 1);
          ++ke;
          tc::fence_after_sync();
          for (int w = 0; w < nw; ++w) {
#pragma unroll
            for (int ks = 0; ks < d / 16; ++ks)
              tc::mma_bf16_ss(tmem + (uint32_t)w * 128u, dq + (uint64_t)(w * 2048) + (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4),
                              dk + (uint64_t)(st * (S::stage_bytes >> 4)) + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4), tc::make_idesc_bf16(128, 64, false, false), ks > 0);
            tc::mma_commit(BAR(TA_SFULL + w));
          }
          tc::mma_commit(BAR(TA_KEMPTY + st));
        };
        if (lane == 0) {
          if (chunk == 0 && rank < items) issue_u(rank);
#pragma unroll 1
          for (int it = rank; it < items; it += A) {
            const int tb = ntb - 1 - it / nqc, NT = (nGB + nRB + tb + 2) / 2, nw = min(2, nqt - (it % nqc) * 2);
            WAIT(TA_KFULL + (ke & 1), (ke >> 1) & 1);
            for (int w = 0; w < nw; ++w) {
              WAIT(TA_PREADY + w, cs[w] & 1);                               // phi(Q_w) in tensor memory
              tc::fence_after_sync();
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks)                           // the linear term is the first thing in O_w
                tc::mma_bf16_ts(tmem + 256u + (uint32_t)w * 128u, tmem + (uint32_t)w * 128u + 64u + ks * 8,
                                dh + (uint64_t)(((ks >> 2) * S::aht_blk + (ks & 3) * 32) >> 4), tc::make_idesc_bf16(128, d, false, false), ks > 0);
              tc::mma_commit(BAR(TA_ODONE + w));
              issue_s(w, ke & 1);                                           // (the tensor pipe runs in order: phi is consumed first)
            }
            tc::mma_commit(BAR(TA_KEMPTY + (ke & 1)));
            ++ke;
#pragma unroll 1
            for (int kt = 0; kt < NT; ++kt) {
              const uint32_t vs = ve & 1, ks2 = ke & 1;
              WAIT(TA_VFULL + vs, (ve >> 1) & 1);
              if (kt + 1 < NT) WAIT(TA_KFULL + ks2, (ke >> 1) & 1);
              for (int w = 0; w < nw; ++w) {
                WAIT(TA_PREADY + w, (cs[w] + (uint32_t)kt + 1u) & 1);
                tc::fence_after_sync();
                const uint32_t to = tmem + 256u + (uint32_t)w * 128u, tp = tmem + (uint32_t)w * 128u;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                  tc::mma_bf16_ts(to, tp + (uint32_t)(ks >> 2) * 64u + (ks & 3) * 8, dv + (uint64_t)(vs * (S::stage_bytes >> 4)) + (uint64_t)((ks * 2048) >> 4), idesc_pv, 1u);
                tc::mma_commit(BAR(TA_ODONE + w));
                if (kt + 1 < NT) issue_s(w, ks2);
              }
              tc::mma_commit(BAR(TA_VEMPTY + vs));
              ++ve;
              if (kt + 1 < NT) { tc::mma_commit(BAR(TA_KEMPTY + ks2)); ++ke; }
            }
            for (int w = 0; w < nw; ++w) cs[w] += (uint32_t)NT + 1u;
            if (it + A < items) issue_u(it + A);
          }
        }
        __syncwarp();
        tc::cluster_arrive();                          // (A)
        if (lane == 0 && chunk + 1 < n_chunks && rank < items) issue_u(rank);
        if (lane == 0 && sel) {                        // the new rows of the H image
          tc::mbar_expect_tx(BAR(TA_H), (uint32_t)d * 256u);
          WAIT(TA_H, ph_h & 1);
          ++ph_h;
        }
        __syncwarp();
      } else {
        // =============================== softmax, two threads per query row ===============================
        // thread (query tile w, row t, half hf) owns the 64 keys [64 hf, 64 hf + 64) of every key tile, half of the
        // feature map in the linear term and half of the output columns
        const int w = gr, tok = t & 63;
        const float sl2 = L.scale * kLog2e;
        const float grow_by = LONG && n > kLagMaxN ? 0.f : kLag;   // the stabiliser moves only when it must grow by more than 2^grow_by
        const uint32_t tm_s = tmem + (uint32_t)w * 128u + lane_addr, tm_sb = tm_s + (uint32_t)hf * 64u;
        const uint32_t tm_o = tmem + 256u + (uint32_t)w * 128u + lane_addr;
        constexpr int HC = d / 2;
        const int pair_bar = 1 + w * 4 + wq;           // the two warps that share this row quadrant (64 threads)
        bool told = false;                             // (A) is passed on
#pragma unroll 1
        for (int it = rank; it < items; it += A) {
          const int tb = ntb - 1 - it / nqc, tok0 = tb * 64, qt0 = (it % nqc) * 2, nw = min(2, nqt - qt0), NT = (nGB + nRB + tb + 2) / 2;
          if (w >= nw) continue;
          const uint32_t c0s = cs[0];                  // (this thread's query tile: its count)
          cs[0] += (uint32_t)NT + 1u;
          WAIT(TA_SFULL + w, c0s & 1);                 // U = Q W is in the first 64 score columns
          tc::fence_after_sync();
          float m_used = 0.f, l;                       // log2 units; m >= 0 is the stabiliser max(0, max z)
          {
            // this thread's half of phi(q) with weight exp(0 - m), m = 0: bf16 pairs into columns 64 + 32 hf .. of S_w
            float e[64];
            tc::tmem_ld64(tm_s, e);
            const float em = (c.att_flags & 1) ? 0.f : 1.0f, sgn = hf ? -kLog2e : kLog2e;   // (0: the queries do not see H, s)
            float scale;
            if (L.phi_kind == 1) {
#pragma unroll
              for (int i = 0; i < 64; ++i) e[i] = tc::fast_exp2(e[i] * sgn);
              scale = em;
            } else {
              float m0 = -CUDART_INF_F, m1 = -CUDART_INF_F;
#pragma unroll
              for (int i = 0; i < 64; i += 2) { m0 = fmaxf(m0, e[i] * sgn); m1 = fmaxf(m1, e[i + 1] * sgn); }
              const float mm = fmaxf(m0, m1);
              float s0 = 0.f, s1 = 0.f;
#pragma unroll
              for (int i = 0; i < 64; i += 2) {
                e[i] = tc::fast_exp2(fmaf(e[i], sgn, -mm)); s0 += e[i];
                e[i + 1] = tc::fast_exp2(fmaf(e[i + 1], sgn, -mm)); s1 += e[i + 1];
              }
              scale = em / (s0 + s1);
            }
            float ld0 = 0.f, ld1 = 0.f;
#pragma unroll
            for (int i = 0; i < 64; i += 2) {
              e[i] *= scale;
              e[i + 1] *= scale;
              ld0 = fmaf(e[i], XA.s_vec[hf * 64 + i], ld0);
              ld1 = fmaf(e[i + 1], XA.s_vec[hf * 64 + i + 1], ld1);
            }
            l = ld0 + ld1;                             // this half of the normaliser phi . s starts the sum of the weights
            uint32_t pk[32];
#pragma unroll
            for (int j = 0; j < 64; j += 2) pk[j >> 1] = pack_bf16x2(e[j], e[j + 1]);
            tc::tmem_st32u(tm_s + 64 + hf * 32, pk);
          }
          tc::fence_before_sync();
          tc::mbar_arrive(BAR(TA_PREADY + w));
#pragma unroll 1
          for (int kt = 0; kt < NT; ++kt) {
            // valid leading columns of this thread's 64-key block of the tile, for this row
            const int blk = 2 * kt + hf;
            int lim;
            if (blk < nGB) lim = att_g - blk * 64;
            else if (blk < nGB + nRB) lim = cw - (blk - nGB) * 64;
            else if (blk < nGB + nRB + tb) lim = 64;   // an earlier block of the chunk
            else if (blk == nGB + nRB + tb) lim = min(n - tok0, tok + 1);
            else lim = 0;
            lim = max(0, min(64, lim));
            WAIT(TA_SFULL + w, (c0s + (uint32_t)kt + 1u) & 1);
            tc::fence_after_sync();
            float sv[64];
            tc::tmem_ld64(tm_sb, sv);
            float mx0 = -CUDART_INF_F, mx1 = -CUDART_INF_F;
            if (lim == 64) {
#pragma unroll
              for (int j = 0; j < 64; j += 4) {
                mx0 = tc::max3(mx0, sv[j], sv[j + 1]);
                mx1 = tc::max3(mx1, sv[j + 2], sv[j + 3]);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 64; ++j) {
                sv[j] = j < lim ? sv[j] : -CUDART_INF_F;   // masked keys get weight 2^(-inf) = 0 below
                mx0 = fmaxf(mx0, sv[j]);
              }
            }
            XA.hx[w][hf][t] = fmaxf(mx0, mx1);
            tc::named_bar_sync(pair_bar, 64);          // (also: both halves hold their scores in registers now)
            const float m_tile = fmaxf(XA.hx[w][0][t], XA.hx[w][1][t]) * sl2;
            const bool grow = m_tile > m_used + grow_by;
            if (__any_sync(0xffffffffu, grow)) {       // rare; tensor-memory accesses are warp-wide: every lane takes part
              const float m_new = grow ? m_tile : m_used, alpha = tc::fast_exp2(m_used - m_new);
              l *= alpha;
              m_used = m_new;
              WAIT(TA_ODONE + w, (c0s + (uint32_t)kt) & 1);   // the product of the tile before (or the linear term) is complete
              tc::fence_after_sync();
#pragma unroll 1
              for (int c0 = 0; c0 < HC; c0 += 8) {     // this thread's half of the row's output columns
                float ov[8];
                tc::tmem_ld8(tm_o + hf * HC + c0, ov);
#pragma unroll
                for (int j = 0; j < 8; ++j) ov[j] *= alpha;
                tc::tmem_st8(tm_o + hf * HC + c0, ov);
              }
            }
            // weights 2^(z - m) <= 2^8 as bf16 pairs over the first half of this thread's S columns
            const uint64_t sl22 = tc::pack_f2(sl2, sl2), nm2 = tc::pack_f2(-m_used, -m_used);
            uint64_t lacc = tc::pack_f2(0.f, 0.f);
            uint32_t pk[32];
#pragma unroll
            for (int j = 0; j < 64; j += 2) {
              float x0, x1;
              tc::unpack_f2(tc::fma2(tc::pack_f2(sv[j], sv[j + 1]), sl22, nm2), x0, x1);
              const float p0 = tc::fast_exp2(x0), p1 = tc::fast_exp2(x1);
              lacc = tc::add2(lacc, tc::pack_f2(p0, p1));
              pk[j >> 1] = pack_bf16x2(p0, p1);
            }
            tc::tmem_st32u(tm_sb, pk);
            float l0, l1;
            tc::unpack_f2(lacc, l0, l1);
            l += l0 + l1;
            tc::fence_before_sync();
            tc::mbar_arrive(BAR(TA_PREADY + w));
          }
          // ---- the two halves of the row's denominator meet (the extra barrier: the partner has read this row's last
          // maxima before the slot is reused)
          tc::named_bar_sync(pair_bar, 64);
          XA.hx[w][hf][t] = l;
          tc::named_bar_sync(pair_bar, 64);
          const float lden = XA.hx[w][hf ^ 1][t];
          WAIT(TA_ODONE + w, (c0s + (uint32_t)NT) & 1);
          tc::fence_after_sync();
          if (it + A >= items) {                       // (A): this query tile has read all it needs of the memories
            told = true;
            __syncwarp();
            tc::cluster_arrive();
          }
          // the outputs leave from the query tile's own buffer, in the layout of a TMA box ([head slot][64-column block]
          // [64 tokens][128 bytes], 128-byte swizzle)
          const float inv = 1.0f / (XA.hx[w][hf][t] + lden);
          const int hs = t >> 6;
#pragma unroll
          for (int c0 = 0; c0 < HC; c0 += 32) {
            float ov[32];
            tc::tmem_ld32(tm_o + hf * HC + c0, ov);
#pragma unroll
            for (int q8 = 0; q8 < 4; ++q8) {
              const int cc = hf * HC + c0 + q8 * 8;
              uint4 o;
              o.x = pack_bf16x2(ov[q8 * 8 + 0] * inv, ov[q8 * 8 + 1] * inv);
              o.y = pack_bf16x2(ov[q8 * 8 + 2] * inv, ov[q8 * 8 + 3] * inv);
              o.z = pack_bf16x2(ov[q8 * 8 + 4] * inv, ov[q8 * 8 + 5] * inv);
              o.w = pack_bf16x2(ov[q8 * 8 + 6] * inv, ov[q8 * 8 + 7] * inv);
              *reinterpret_cast<uint4*>(sm + S::q + w * 32768 + (hs * kblk + (cc >> 6)) * 8192 + tc::sw128_off(tok, (cc & 63) >> 3)) = o;
            }
          }
          tc::fence_async_smem();
          tc::fence_before_sync();
          tc::named_bar_sync(9 + w, 256);
          if (t == 0 && hf == 0) {
            for (int s2 = 0; s2 < 2; ++s2) {
              const int hl2 = (qt0 + w) * 2 + s2;
              if (hl2 >= g || !ok) continue;           // (rows of tokens >= n lie outside the tensor: not written)
#pragma unroll
              for (int cb = 0; cb < kblk; ++cb)
                tc::tma_store_5d(&M.out, sbase + S::q + (uint32_t)w * 32768u + (uint32_t)(s2 * kblk + cb) * 8192u, cb * 64, h * g + hl2, tok0, b, chunk);
            }
            tc::bulk_commit_group();
            tc::bulk_wait_group_read();                // the buffer is read: the next queries may come
            tc::mbar_arrive(BAR(TA_QFREE));
            if (nw == 1) tc::mbar_arrive(BAR(TA_QFREE));
          }
          __syncwarp();
        }
        __syncwarp();
        if (!told) tc::cluster_arrive();               // (A)
      }
      tc::cluster_wait();
      if (warp < 16) {
        // a warp per incoming token (half a warp each for key and value): the pair whose ring slot it takes first moves
        // into the sparse cache if it stays
        const int ch = lane & 15;
        const bool isv = lane >= 16;
#pragma unroll 1
        for (int ci = rank * 16 + warp; ci < n; ci += A * 16) {
          const int p = n_seen + ci, slot = p % eta, i = p - eta - c.r_pos0;
          const int to = i < 0 || i >= c.r ? -1 : sel ? __ldcg(L.move_dst + (size_t)unit * L.cmax + i) : c.mode == UPD_APPEND ? cg + i : -1;
          const bool enters = ci >= n - eta;
          if (ch < d / 8 && ok) {
            T* ring = (T*)(isv ? L.wv : L.wk) + ((size_t)unit * eta + slot) * d + ch * 8;
            uint4 o4, n4;
            if (to >= 0) o4 = __ldcg(reinterpret_cast<const uint4*>(ring));
            if (enters) n4 = *reinterpret_cast<const uint4*>((const T*)(isv ? c.v : c.k) + (((size_t)(chunk * L.B + b) * n + ci) * L.Hkv + h) * d + ch * 8);
            if (to >= 0) *reinterpret_cast<uint4*>((T*)(isv ? L.gv : L.gk) + ((size_t)unit * lam + to) * d + ch * 8) = o4;
            if (enters) *reinterpret_cast<uint4*>(ring) = n4;
          }
        }
      }
    } else {
      const ScoreBlocks SB(cg, c.r, c.r_pos0, eta);    // what is scored: the sparse cache and the leaving pairs
      const int n_score = sel ? SB.tiles() : 0, ring0 = SB.s0;
      if (warp >= 16) {
        // =============================== tiles of group warp - 16 ===============================
        if (tc::elect_one()) {
          const int gp = warp - 16;
#pragma unroll 1
          for (int tile = sr + gp * N; tile < n_score; tile += 2 * N, ++en) {
            if (en >= 1) WAIT(TS_KEMPTY + gp, (en - 1) & 1);
            if (!ok) break;
            score_issue_tile<DPL>(sbase + S::grp0 + (uint32_t)gp * 65536u, &M.gk, &M.wk, tile, SB, eta, unit, BAR(TS_KFULL + gp));
            if (en >= 1) WAIT(TS_VEMPTY + gp, (en - 1) & 1);
            if (!ok) break;
            score_issue_tile<DPL>(sbase + S::grp0 + (uint32_t)gp * 65536u + 32768u, &M.gv, &M.wv, tile, SB, eta, unit, BAR(TS_VFULL + gp));
          }
        }
        __syncwarp();
        tc::fence_before_sync();
        tc::cluster_arrive();                          // (A)
        tc::cluster_wait();
        if (warp == 16 && lane == 0 && sel && N > 1) { // the other blocks' new rows of the H image
          tc::mbar_expect_tx(BAR(TS_H), (uint32_t)(d - d / N) * 256u);
          WAIT(TS_H, ph_h & 1);
          ++ph_h;
        }
        __syncwarp();
      } else if (!sel) {
        tc::cluster_arrive();                          // (A)
        tc::cluster_wait();
        if (sr == 0 && c.mode == UPD_APPEND)
          for (int i = tid; i < c.r; i += 512)
            if (ok) {
              L.gpos[(size_t)unit * lam + cg + i] = c.r_pos0 + i;
              scu[cg + i] = CUDART_NAN_F;
            }
      } else {
        // =============================== scoring, two groups ===============================
        const uint64_t dw = tc::make_desc_sw128(sbase + S::wt, 16, 1024), dh = tc::make_desc_sw128(sbase + S::ht, 16, 1024);
        const uint32_t id_u = tc::make_idesc_bf16(128, 64, false, false), id_p = tc::make_idesc_bf16(128, d + 16, false, false);
        const uint32_t tm_u = tmem + (uint32_t)gr * 256u, tm_p = tm_u + 64u;
        const bool lead = (tid & 255) == 0;
        auto sync = [&] { tc::named_bar_sync(1 + gr, 256); };
        auto sync_all = [] { tc::named_bar_sync(3, 512); };
        // U = K W of a tile is issued behind [P | den] of the group's tile before (the tensor pipe runs in order, so the
        // feature map there is consumed first).  The key tile's barrier is the issuing thread's alone: it may complete
        // again before a late warp has looked at it
        auto issue_u = [&](uint32_t e) {
          WAIT(TS_KFULL + gr, e & 1);
          tc::fence_after_sync();
          const uint64_t dk = tc::make_desc_sw128(sbase + S::grp0 + (uint32_t)gr * 65536u, 16, 1024);
#pragma unroll
          for (int ks = 0; ks < d / 16; ++ks)
            tc::mma_bf16_ss(tm_u, dk + (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), dw + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4), id_u, ks > 0);
          tc::mma_commit(BAR(TS_U + gr));
          tc::mma_commit(BAR(TS_KEMPTY + gr));
        };
        const int tile0 = sr + gr * N;
        if (lead && tile0 < n_score) issue_u(en);
#pragma unroll 1
        for (int tile = tile0; tile < n_score; tile += 2 * N, ++en) {
          const uint32_t par = en & 1;
          // member of E this row holds (-1: none)
          const int blk = 2 * tile + (t >> 6), ro = t & 63;
          int e = -1;
          if (blk < nGB) { if (blk * 64 + ro < cg) e = blk * 64 + ro; }
          else if (blk < nGB + SB.nR1) { const int i = (blk - nGB) * 64 + ro; if (i < SB.len1) e = cg + i; }
          else { const int i = SB.len1 + (blk - nGB - SB.nR1) * 64 + ro; if (i < c.r) e = cg + i; }
          WAIT(TS_U + gr, par);
          tc::fence_after_sync();
          {
            uint32_t u[64], pk2[32];
            tc::tmem_ld64u(tm_u + lane_addr, u);
            tc::phi_half(u, hf != 0, L.phi_kind == 1, pk2);
            tc::fence_before_sync();
            sync();                                    // both threads of a row have read U: its columns take the feature map
            tc::tmem_st32u(tm_u + lane_addr + hf * 32, pk2);
          }
          tc::fence_before_sync();
          sync();
          tc::fence_after_sync();
          if (lead) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)
              tc::mma_bf16_ts(tm_p, tm_u + ks * 8, dh + (uint64_t)(((ks >> 2) * S::ht_blk + (ks & 3) * 32) >> 4), id_p, ks > 0);
            tc::mma_commit(BAR(TS_S + gr));
            if (tile + 2 * N < n_score) issue_u(en + 1);
          }
          WAIT(TS_VFULL + gr, par);
          WAIT(TS_S + gr, par);
          tc::fence_after_sync();
          constexpr int HC = d / 2;
          uint64_t ninv2 = 0, accA = tc::pack_f2(0.f, 0.f), accB = accA;
          const uint8_t* vt = sm + S::grp0 + gr * 65536 + 32768;
#pragma unroll
          for (int c0 = 0; c0 < HC; c0 += 32) {
            uint32_t p[32];
            if (c0 == 0) {
              uint32_t dn[2];
              tc::tmem_ld32u_and2(tm_p + lane_addr + hf * HC, p, tm_p + lane_addr + d, dn);
              const float den = __uint_as_float(dn[0]) + __uint_as_float(dn[1]), inv = den > 0.f ? 1.0f / den : 0.f;
              ninv2 = tc::pack_f2(-inv, -inv);
            } else {
              tc::tmem_ld32u(tm_p + lane_addr + hf * HC + c0, p);
            }
#pragma unroll
            for (int q8 = 0; q8 < 4; ++q8) {
              const int cc = hf * HC + c0 + q8 * 8;
              const uint4 raw = *reinterpret_cast<const uint4*>(vt + (cc >> 6) * 16384 + tc::sw128_off(t, (cc & 63) >> 3));
              const uint64_t d01 = tc::fma2(tc::pack_u2(p[q8 * 8 + 0], p[q8 * 8 + 1]), ninv2, tc::pack_u2(raw.x << 16, raw.x & 0xffff0000u));
              const uint64_t d23 = tc::fma2(tc::pack_u2(p[q8 * 8 + 2], p[q8 * 8 + 3]), ninv2, tc::pack_u2(raw.y << 16, raw.y & 0xffff0000u));
              const uint64_t d45 = tc::fma2(tc::pack_u2(p[q8 * 8 + 4], p[q8 * 8 + 5]), ninv2, tc::pack_u2(raw.z << 16, raw.z & 0xffff0000u));
              const uint64_t d67 = tc::fma2(tc::pack_u2(p[q8 * 8 + 6], p[q8 * 8 + 7]), ninv2, tc::pack_u2(raw.w << 16, raw.w & 0xffff0000u));
              accA = tc::fma2(d01, d01, accA);
              accB = tc::fma2(d23, d23, accB);
              accA = tc::fma2(d45, d45, accA);
              accB = tc::fma2(d67, d67, accB);
            }
          }
          float a0, a1, a2, a3;
          tc::unpack_f2(accA, a0, a1);
          tc::unpack_f2(accB, a2, a3);
          const float ss = (a0 + a1) + (a2 + a3);
          if (hf == 1) X.ssp[gr][t] = ss;
          tc::fence_before_sync();
          sync();                                      // both halves are done with the value tile and with P
          tc::fence_after_sync();
          if (lead) tc::mbar_arrive(BAR(TS_VEMPTY + gr));
          if (hf == 0) {
            const float sc = sqrtf(ss + X.ssp[gr][t]);
            const uint32_t sb = __float_as_uint(sc), ka = sbase + S::smisc + (uint32_t)offsetof(TeamScoreMisc, key);
            const int e0 = __shfl_sync(0xffffffffu, e, 0);
            if (__all_sync(0xffffffffu, e >= 0 && e == e0 + lane && (e0 & 3) == 0)) {
              // four scores a message, each of the four lanes that hold them for every fourth block
              const int l4 = lane & ~3;
              const uint4 q4 = make_uint4(__shfl_sync(0xffffffffu, sb, l4), __shfl_sync(0xffffffffu, sb, l4 + 1), __shfl_sync(0xffffffffu, sb, l4 + 2),
                                          __shfl_sync(0xffffffffu, sb, l4 + 3));
              for (int r = lane & 3; r < N; r += 4) tc::st_async_v4(tc::map_rank(ka + (uint32_t)(e0 + l4) * 4u, (uint32_t)(A + r)), q4, tc::map_rank(BAR(TS_SCORES), (uint32_t)(A + r)));
            } else if (e >= 0) {
              for (int r = 0; r < N; ++r) tc::st_async_u32(tc::map_rank(ka + (uint32_t)e * 4u, (uint32_t)(A + r)), sb, tc::map_rank(BAR(TS_SCORES), (uint32_t)(A + r)));
            }
            if (ok && e >= 0) scu[e < cg ? e : lam + (e - cg)] = sc;
          }
        }
        if (tid == 0) tc::mbar_expect_tx(BAR(TS_SCORES), (uint32_t)nE * 4u);
        WAIT(TS_SCORES, ph_sc & 1);                    // the scores of all blocks are here
        ++ph_sc;
        const int dK = d / N, dKs = 31 - __clz(dK), c0 = sr * dK, part = dK / 4;   // (N is a power of two)
        auto hrow = [&](int i) { return i < 96 * 128 * 4 ? S::hrow0 + (uint32_t)i : S::hrow1 + (uint32_t)(i - 96 * 128 * 4); };   // byte i of [128][dK] (a row is in one part)
        const int hm = min(8, dK / 4) - 1;             // 16-byte piece p of row j lies at piece p ^ (j & hm): rows and columns without bank conflicts
        constexpr int PPR = d / 4;                     // 16-byte pieces of a pair: key, then value
        constexpr int NP = kUp2Batch * PPR / 512;
        const int isv = (tid % PPR) / (PPR / 2), ch = tid % (PPR / 2);
        auto gather = [&](int f0) {                    // the folded pairs' keys and values into the fold's tiles
          const int nb = min(kUp2Batch, nF - f0);
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            const int row = tid / PPR + q * (512 / PPR);
            const int e = X.fold[f0 + min(row, nb - 1)];
            int slot = ring0 + e - cg;
            if (slot >= eta) slot -= eta;
            const T* src = (e < cg ? (const T*)(isv ? L.gv : L.gk) + ((size_t)unit * lam + e) * d : (const T*)(isv ? L.wv : L.wk) + ((size_t)unit * eta + slot) * d) + ch * 8;
            const uint32_t dst = sbase + (isv ? S::fold_v : S::fold_k) + (uint32_t)(ch >> 3) * 16384u, sz = row < nb ? 16u : 0u;
            tc::cp_async16(dst + tc::sw128_off(row, ch & 7), src, sz);
            if (!isv) tc::cp_async16(dst + tc::sw128_off(row + 64, ch & 7), src, sz);   // again, for the second parts of phi
          }
        };
        // (one group selects: half as many threads wait for each other; 832 of 896 pairs 5200 cycles, by both 6250)
        if (gr == 0)
          select_lists<256>(X.key, [&](int e) { return e < cg ? __ldcg(L.gpos + (size_t)unit * lam + e) : c.r_pos0 + (e - cg); }, X.cand, X.mark, nE, nF, cg,
                            X.fold, X.sel, tid, sync,
                            [&](int i, int to) {
                              X.dst[i] = (short)to;
                              if (sr == 0 && ok) L.move_dst[(size_t)unit * L.cmax + i] = to;   // (read by the attention blocks)
                            },
                            sync_all);
        else
          sync_all();
        // (both groups are through with their tiles: the buffers may be written)
        gather(0);
#pragma unroll 1
        for (int i = tid; i < dK * 32; i += 512)       // this block's columns of H
          tc::cp_async16(sbase + hrow((i ^ ((i >> (dKs - 2)) & hm)) * 16), Hg + (size_t)(i >> (dKs - 2)) * d + c0 + (i & (dK / 4 - 1)) * 4);
        if (sr == 0 && tid == 0 && ok) {
          L.thr[(size_t)unit * 2 + 0] = __uint_as_float(X.sel.min_keep);
          L.thr[(size_t)unit * 2 + 1] = __uint_as_float(X.sel.max_fold);
        }
        // ---- Eq. 13: dH = phi(K_S)^T [V_S | 1], 64 pairs at a time, phi in two or three bf16 parts against the same values
        const bool three = LONG && fold_in_three(c);
        float ds_sum = 0.f;
        const uint32_t tm_fu = tmem, tm_fp = tmem + 64u;
#pragma unroll 1
        for (int f0 = 0; f0 < nF; f0 = LONG ? f0 + kUp2Batch : nF) {
          const int nb = min(kUp2Batch, nF - f0);
          if (LONG && f0 > 0) gather(f0);                      // (the first ones are on their way since the selection)
          if (tid < 64) {                              // the column of ones and its 15 empty neighbours
            uint4 one = make_uint4(0, 0, 0, 0);
            if (tid < nb) one.x = 0x3f80u;
            *reinterpret_cast<uint4*>(sm + S::fold_v + kblk * 16384 + tc::sw128_off(tid, 0)) = one;
            *reinterpret_cast<uint4*>(sm + S::fold_v + kblk * 16384 + tc::sw128_off(tid, 1)) = make_uint4(0, 0, 0, 0);
          }
          tc::cp_async_wait_all();
          tc::fence_async_smem();
          tc::fence_before_sync();
          if (!LONG || f0 + kUp2Batch >= nF) tc::cluster_arrive();   // (A)
          sync_all();
          tc::fence_after_sync();
          if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < d / 16; ++ks)
              tc::mma_bf16_ss(tm_fu, tc::make_desc_sw128(sbase + S::fold_k + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024),
                              dw + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4), id_u, ks > 0);
            tc::mma_commit(BAR(TS_FOLD));
          }
          WAIT(TS_FOLD, ph_f & 1);
          ++ph_f;
          tc::fence_after_sync();
          {                                            // rows 0-63 the pairs' first parts, 64-127 the second ones; 32 features a thread
            const bool ek = L.phi_kind == 1;
            uint32_t u[32];
            uint64_t x2[16];
            float m, sum, f = 1.0f;
            tc::tmem_ld32u(tm_fu + lane_addr + gr * 32, u);
            tc::phi_quarter_f32(u, hf != 0, ek, x2, m, sum);
            if (!ek) {
              X.phx[gr][hf][t] = make_float2(m, sum);
              tc::named_bar_sync(4 + hf * 4 + wq, 64); // the two warps that share these features' rows
              const float2 o = X.phx[gr ^ 1][hf][t];
              const float mm = fmaxf(m, o.x), a = tc::fast_exp2(m - mm);
              f = a / fmaf(sum, a, o.y * tc::fast_exp2(o.x - mm));
            }
            const uint64_t f2 = tc::pack_f2(f, f);
            // (the third parts, if taken, in the rows of the value tile that hold no pair)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t pk[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                x2[q * 4 + e] = tc::mul2(x2[q * 4 + e], f2);
                pk[e] = tc::phi_part(x2[q * 4 + e], t >= 64);
              }
              *reinterpret_cast<uint4*>(sm + S::fold_k + hf * 16384 + tc::sw128_off(t, gr * 4 + q)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
            if (LONG && three && t >= 64) {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(sm + S::fold_v + hf * 16384 + tc::sw128_off(t, gr * 4 + q)) =
                    make_uint4(tc::phi_third(x2[q * 4]), tc::phi_third(x2[q * 4 + 1]), tc::phi_third(x2[q * 4 + 2]), tc::phi_third(x2[q * 4 + 3]));
            }
          }
          tc::fence_async_smem();
          tc::fence_before_sync();
          sync_all();
          tc::fence_after_sync();
          if (tid == 0) {
            tc::fold_product<DPL, LONG>(tm_fp, sbase + S::fold_k, sbase + S::fold_v, three);
            tc::mma_commit(BAR(TS_FOLD));
          }
          WAIT(TS_FOLD, ph_f & 1);
          ++ph_f;
          tc::fence_after_sync();
          // the batch's dH into this block's columns of H, in shared memory (batches are added up here: see fold_product)
          const int p0 = (gr * 2 + hf) * (part / 4);
          const uint32_t tcol = tm_fp + lane_addr + (uint32_t)(c0 + p0 * 4);
          auto add_h = [&](int q, float a, float b, float cc, float e) {
            float4* to = reinterpret_cast<float4*>(sm + hrow((t * (dK / 4) + ((p0 + q) ^ (t & hm))) * 16));
            const float4 o = *to;
            *to = make_float4(o.x + a, o.y + b, o.z + cc, o.w + e);
          };
          if (part == 32) {
            float p[32];
            tc::tmem_ld32(tcol, p);
#pragma unroll
            for (int q = 0; q < 8; ++q) add_h(q, p[q * 4], p[q * 4 + 1], p[q * 4 + 2], p[q * 4 + 3]);
          } else {
#pragma unroll 1
            for (int q = 0; q < part / 4; ++q) {
              float p[4];
              tc::tmem_ld4(tcol + q * 4, p);
              add_h(q, p[0], p[1], p[2], p[3]);
            }
          }
          if (gr == 0 && hf == 0) {
            float ds[2];
            tc::tmem_ld2(tm_fp + lane_addr + d, ds);
            ds_sum += ds[0];
          }
        }
        // the new columns of H into memory and, rounded, into the operand image: here at once, in the other blocks when all
        // have read the old one (A).  A thread has 8 rows of one column, 16 bytes of the image, and lanes have neighbouring
        // columns of H (a row each took 9 us)
        if (gr == 0 && hf == 0) {
          const float sv = X.s[t] + ds_sum;
          put_s(t, sv);
          if (sr == 0 && ok) L.s[(size_t)unit * D + t] = sv;
        }
        tc::fence_before_sync();
        sync_all();
#pragma unroll 1
        for (int it = tid; it < dK * 16; it += 512) {
          const int cc = it & (dK - 1), jc = it >> dKs;
          const float* hr = reinterpret_cast<const float*>(sm + hrow(jc * 8 * dK * 4)) + (cc & 3);
          float* hg = Hg + (size_t)(jc * 8) * d + c0 + cc;
          float hv[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) hv[j] = hr[j * dK + ((cc >> 2) ^ (j & hm)) * 4];
          if (ok) {
#pragma unroll
            for (int j = 0; j < 8; ++j) hg[j * d] = hv[j];
          }
          *reinterpret_cast<uint4*>(sm + S::ht + (jc >> 3) * S::ht_blk + tc::sw128_off(c0 + cc, jc & 7)) = tc::pack8_bf16(hv);
        }
        tc::fence_async_smem();
        sync_all();
        tc::cluster_wait();                            // (A)
        if (warp == 0) {                               // its rows of the image to every block: a lane per block and half of the features
          const int r = lane >> 1;
          const uint32_t jb = (uint32_t)lane & 1u, off = (uint32_t)c0 * 128u;
          if (r < K && r != rank)
            tc::bulk_copy_s2peer(tc::map_rank(sbase + (r < A ? S::aht + jb * S::aht_blk : S::ht + jb * S::ht_blk) + off, (uint32_t)r), sbase + S::ht + jb * S::ht_blk + off,
                                 (uint32_t)dK * 128u,
                                 tc::map_rank(sbase + (r < A ? S::amisc + (uint32_t)offsetof(TeamAttMisc, bars) + 8u * TA_H : S::smisc + (uint32_t)offsetof(TeamScoreMisc, bars) + 8u * TS_H), (uint32_t)r));
          __syncwarp();
        }
        if (sr == 0) {
          if (warp == 1)
            for (int r = 0; r < A; ++r)
              tc::st_cluster_v4(tc::map_rank(sbase + S::amisc + (uint32_t)offsetof(TeamAttMisc, s_vec) + (uint32_t)lane * 16u, (uint32_t)r), *reinterpret_cast<const uint4*>(&X.s[lane * 4]));
          for (int i = tid; i < c.r; i += 512) {
            const int to = X.dst[i];
            if (to >= 0 && ok) {
              L.gpos[(size_t)unit * lam + to] = c.r_pos0 + i;
              scu[to] = __uint_as_float(X.key[cg + i]);
            }
          }
        }
      }
    }
    if (warp < 16) tc::fence_async_all();              // what was written is read by TMA and tensor cores next
    tc::fence_before_sync();
    __syncwarp();
    tc::cluster_arrive();
    tc::cluster_wait();
    if (warp >= 16 || (warp & 7) == 0) tc::fence_async_all();
    tc::fence_after_sync();
    n_seen += n;
  }
  if (!ok) *abw = 1;
  __syncthreads();
  if (*abw != 0) __nanosleep(200000);                 // (after a failure: copies on their way into this block's memory arrive first)
  if (tid == 0 && *abw != 0) atomicOr(L.status, 512);
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace lola
