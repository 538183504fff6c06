// A run of prefill chunks of a bf16 layer (F = 64) as ONE kernel: a cluster of K thread blocks carries one (batch row,
// KV head) unit through all chunks of the run.
//
// What bounds it: the chain score -> select -> fold of a unit, which is serial from chunk to chunk and nearly all
// latency (a unit's chunk is 0.17 GFLOP).  As three dependent launches it took 24 us (d = 64) to 34 us (d = 128) a
// chunk with most SMs idle at small batches: every launch sets up its operands again (H, W, tensor memory, 4 - 5 us),
// runs through 50 - 65 KB of cold code and hands lists over through memory.  Here the set-up happens once per run and
// the code stays in the instruction cache: 13 us (d = 64) and 18.6 us (d = 128) a chunk of 8 units.  Each block has two
// groups of 256 threads that work side by side:
//
//   score group (warps 0-7)       the tiles of E this block owns: U = K W, feature map, [P | den] = phi [H | s_hi s_lo],
//                                 Eq. 10; the scores go to all blocks of the cluster.  Then, in every block for itself,
//                                 the selection (Eq. 12) and dH = phi^T V of the folded pairs; each block adds the d / K
//                                 columns of dH it owns to H in memory and sends their bf16 operand rows to the others.
//   attention group (warps 8-15)  Eq. 14 for the query items this block owns (an item is one query head x 32 tokens;
//                                 NQ / 32 items): all key tiles are streamed, Z = K Q^T (keys are the rows of
//                                 the product, so 32 or 64 queries fill the tensor cores' M = 128), softmax weights
//                                 into the Pr^T operand, O^T += V^T Pr^T; the linear term H^T phi(Q)^T comes first.
//   warp 16 key / value tiles by TMA,  warp 17 Z products and queries,  warp 18 O^T products
//
// A block streams the tiles it scores first, so one copy of a tile in shared memory serves both groups.  Per chunk the
// cluster meets three times: an mbarrier that counts the scores that have arrived, a cluster barrier (A) when every block
// has read all it needs of the old memories (the attention groups then move the pairs while the score groups fold), and
// one when the new memories are written.
// Rows of the stream in 64-row blocks: sparse-cache slots, ring slots, the chunk itself; two blocks are a tile.
// K is the largest of 8, 4, 2 whose clusters are all resident; chunks with more than 2 K query items go to k_prefill_team.
// Every wait on an mbarrier is bounded; a wait that runs out sets bit 256 of the status word.
#pragma once
#include <cuda.h>

#include "lola_generic.cuh"
#include "lola_select.cuh"
#include "lola_tc.cuh"
#include "lola_update2_tc.cuh"

namespace lola {

constexpr int kRunThreads = 608;
// eligible pairs of a unit (shared memory: the scores and the scratch of the selection)
constexpr int run_max_e(int nq) { return nq == 32 ? 1280 : 1024; }
constexpr int kRunMaxN = 64;         // tokens per chunk (and folds: one batch of them)

template <int NQ>
struct RunMisc {
  alignas(16) unsigned key[run_max_e(NQ)];   // score bits of E
  short cand[run_max_e(NQ)];         // scratch of the selection
  unsigned char mark[run_max_e(NQ)];
  short fold[kRunMaxN];              // E indices of the folded pairs
  short dst[kRunMaxN];               // per leaving pair: slot it takes, or -1
  SelectScratch sel;
  float s[128];                      // the normaliser state, fp32 (the same in every block)
  float ssp[128];
  float2 phx[2][128];                // fold: maximum and sum of a thread's 32 features
  union {
    float redm[4][64];               // per row quadrant: column maxima of a tile
    float l_s[4][64];                // after the last tile: sums of the weights
  };
  float m[64];                       // stabiliser of every query (log2 units)
  float lden[2][64];                 // phi(q) . s, the two halves of the features
  float inv[64];
  int grow[3][2];
  uint64_t bars[23];
  uint32_t tmem_slot;
  int abort_word;
};

template <int DPL, int NQ>
struct RunSmem {
  static constexpr uint32_t wt = 0;                                 // W^T, K-major [kblk][64][128B]
  static constexpr uint32_t ht = 16384;                             // [H^T ; s_hi ; s_lo], K-major [2 j blocks][d + 16][128B];
  static constexpr uint32_t ht_blk = (DPL * 32 + 16) * 128;
  static constexpr uint32_t q = ht + 36864;                         // queries, K-major [kblk][NQ][128B]
  static constexpr uint32_t pt = q + NQ * 256;                      // phi(Q), K-major [2][NQ][128B]; then the weights [128 keys][128B]
  static constexpr uint32_t stage0 = pt + 16384;                    // 2 x (K tile 32 KB, V tile 32 KB); then the fold's tiles
  static constexpr uint32_t st_v = 32768, stage_bytes = 65536;
  static constexpr uint32_t fold_k = stage0, fold_v = stage0 + 32768;   // K_S then phi [2][128][128B]; [V_S | 1] [kblk + 1][128][128B], pairs in rows 0-63
  static constexpr uint32_t fold_h = fold_v + 3 * 16384;            // dH, this block's columns, fp32 [128][d / K + 4]
  static constexpr uint32_t misc = stage0 + 2 * stage_bytes;
  static_assert(fold_h + 128 * (DPL * 16 + 4) * 4 <= misc, "the fold's tiles");
  static constexpr uint32_t total = misc + (uint32_t)sizeof(RunMisc<NQ>);
  static constexpr uint32_t bytes = 232448;                         // all of an SM's shared memory; the base is aligned at run time
};
static_assert(RunSmem<4, 64>::total <= 232448 && RunSmem<4, 32>::total <= 232448, "shared memory");

// The order in which block `rank` streams the tiles of a pass: the ones it scores (t = rank, rank + K, .. < n_score)
// first, then the others.
struct TileOrder {
  int rank, K, n_score, n_tiles, t;
  bool own;
  __device__ __forceinline__ TileOrder(int rank_, int K_, int n_score_, int n_tiles_) : rank(rank_), K(K_), n_score(n_score_), n_tiles(n_tiles_), t(rank_), own(true) {
    if (t >= n_score) { own = false; t = -1; next(); }
  }
  __device__ __forceinline__ bool done() const { return t >= n_tiles; }
  __device__ __forceinline__ void next() {
    if (own) {
      t += K;
      if (t < n_score) return;
      own = false;
      t = -1;
    }
    ++t;
    while (t < n_score && (t & (K - 1)) == rank) ++t;   // (K is a power of two)
  }
};

// Reduces N values per lane (N = 16) over the 32 lanes; lane l returns the result of column l >> 1.
template <bool MAX>
__device__ __forceinline__ float cols_reduce16(const float (&v)[16], int lane) {
  float a[8];
  const bool u4 = lane & 16, u3 = lane & 8, u2 = lane & 4, u1 = lane & 2;
  auto comb = [](float x, float y) { return MAX ? fmaxf(x, y) : x + y; };
#pragma unroll
  for (int j = 0; j < 8; ++j) a[j] = comb(u4 ? v[j + 8] : v[j], __shfl_xor_sync(0xffffffffu, u4 ? v[j] : v[j + 8], 16));
#pragma unroll
  for (int j = 0; j < 4; ++j) a[j] = comb(u3 ? a[j + 4] : a[j], __shfl_xor_sync(0xffffffffu, u3 ? a[j] : a[j + 4], 8));
#pragma unroll
  for (int j = 0; j < 2; ++j) a[j] = comb(u2 ? a[j + 2] : a[j], __shfl_xor_sync(0xffffffffu, u2 ? a[j] : a[j + 2], 4));
  a[0] = comb(u1 ? a[1] : a[0], __shfl_xor_sync(0xffffffffu, u1 ? a[0] : a[1], 2));
  return comb(a[0], __shfl_xor_sync(0xffffffffu, a[0], 1));
}

struct RunMaps {
  tc::SlotMaps gk, gv;
  CUtensorMap wk, wv, q, k, v;
};

// barriers
enum { R_KFULL = 0, R_VFULL = 2, R_KEMPTY = 4, R_VEMPTY = 6, R_ZFULL = 8, R_ZFREE = 10, R_PT = 12, R_O = 14, R_LIN = 16, R_OFREE = 17, R_QFULL = 18,
       R_UQ = 19, R_PHIQ = 20, R_S = 21, R_SCORES = 22, R_N = 23 };

// THREE: a kernel for runs with chunks whose fold takes phi in three parts (fold_in_three; its code costs the others up to 1 us a
// chunk)
template <int DPL, int NQ, bool THREE>
__global__ void __launch_bounds__(kRunThreads, 1)
k_prefill_run(Layer L, Call c, int n_chunks, const __grid_constant__ RunMaps M, const uint4* wt_image) {
  using S = RunSmem<DPL, NQ>;
  constexpr int d = DPL * 32, kblk = d / 64, D = 128, HQ = NQ / 2;
  constexpr float kLog2e = 1.4426950408889634f;
  constexpr float kGrow = 64.0f;                      // log2 units of a score from which the stabiliser moves
  typedef __nv_bfloat16 T;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = tc::smem_u32(sm);
  typedef RunMisc<NQ> Misc;
  Misc& X = *reinterpret_cast<Misc*>(sm + S::misc);
  volatile int* abw = &X.abort_word;
  const uint32_t bar0 = sbase + S::misc + (uint32_t)offsetof(Misc, bars);
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  bool ok = true;
  auto WAIT = [&](int i, uint32_t parity) { ok = tc::mbar_wait(BAR(i), parity, abw) && ok; };

  const int K = (int)tc::cluster_size(), rank = (int)tc::cluster_rank();
  const int unit = blockIdx.x / K, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gtid = tid & 255, wq = warp & 3, hf = (warp >> 2) & 1;
  const int t = wq * 32 + lane;                       // row of a tile = tensor-memory lane
  const int lam = L.lam, eta = L.eta, g = L.g, n = c.n;
  const bool want_out = c.out != nullptr;
  const float sl2 = L.scale * kLog2e;
  const int ntb = (n + 31) / 32, items = g * ntb;
  constexpr int IP = NQ / 32;                         // items of a block: rank * IP ..
  // Buffers of the weights operand.  32 queries fill half of its 128-byte rows, so tiles take turns in the two halves and the
  // weights of a tile are made while the product of the one before runs
  constexpr uint32_t NB = NQ == 32 ? 2 : 1;
  const int it0 = rank * IP;
  float* scu = L.score + (size_t)unit * (lam + L.cmax);
  float* Hg = L.H + (size_t)unit * D * d;

  if (tid == 0) {
    X.abort_word = 0;
    for (int i = 0; i < 6; ++i) X.grow[i / 2][i & 1] = 0;
    for (int i = 0; i < R_N; ++i)
      tc::mbar_init(BAR(i), (i >= R_KEMPTY && i < R_ZFULL) ? 2u : (i == R_ZFREE || i == R_ZFREE + 1 || i == R_PT || i == R_PT + 1 || i == R_OFREE) ? 256u
                            : i == R_PHIQ ? (uint32_t)NQ * 2u : 1u);
    tc::mbar_init_fence();
    tc::grid_dep_launch_dependents();
  }
  if (warp == 0) tc::tmem_alloc(&X.tmem_slot, 512);
  for (int i = tid; i < kblk * 512; i += kRunThreads) *reinterpret_cast<uint4*>(sm + S::wt + i * 16) = wt_image[(size_t)h * kblk * 512 + i];
  tc::grid_dep_wait();                                // everything before this kernel in the stream is complete
  // an earlier kernel failed: do nothing; all blocks of a cluster take the first one's word for it (a misaligned window
  // cannot happen)
  const bool fits = (uint32_t)(sm - smem_raw) + S::total <= S::bytes;
  if (tid == 0) X.abort_word = state_failed(L) || !fits ? 1 : 0;
  if (!fits && tid == 0) atomicOr(L.status, 256);
  // H -> bf16 operand image, s -> its two bf16 rows
  for (int it = tid; it < d * 16 && fits; it += kRunThreads) {
    const int cc = it % d, jc = it / d;
    float hv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) hv[j] = Hg[(size_t)(jc * 8 + j) * d + cc];
    *reinterpret_cast<uint4*>(sm + S::ht + (jc >> 3) * S::ht_blk + tc::sw128_off(cc, jc & 7)) = tc::pack8_bf16(hv);
  }
  auto put_s = [&](int j, float sv) {
    const T hi = __float2bfloat16_rn(sv), lo = __float2bfloat16_rn(sv - __bfloat162float(hi));
    const int ch = (j & 63) >> 3;
    X.s[j] = sv;
    *reinterpret_cast<T*>(sm + S::ht + (j >> 6) * S::ht_blk + tc::sw128_off(d, ch) + (j & 7) * 2) = hi;
    *reinterpret_cast<T*>(sm + S::ht + (j >> 6) * S::ht_blk + tc::sw128_off(d + 1, ch) + (j & 7) * 2) = lo;
  };
  if (tid < D && fits) put_s(tid, L.s[(size_t)unit * D + tid]);
  for (int i = tid; i < 2 * 14 * 8; i += kRunThreads)   // operand rows d + 2 .. d + 15
    *reinterpret_cast<uint4*>(sm + S::ht + (i / 112) * S::ht_blk + tc::sw128_off(d + 2 + (i / 8) % 14, i % 8)) = make_uint4(0, 0, 0, 0);
  tc::fence_async_all();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = X.tmem_slot;
  if (tc::cluster_failed(sbase + S::misc + (uint32_t)offsetof(Misc, abort_word))) {
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
    return;
  }
  if (tid == 0) X.abort_word = 0;
  __syncthreads();

  const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
  const uint32_t tm_z = tmem, tm_u = tmem + 2 * NQ, tm_p = tm_u + 64, tm_o = tm_p + 144;
  auto stage_k = [&](uint32_t i) { return S::stage0 + (i & 1) * S::stage_bytes; };
  auto stage_v = [&](uint32_t i) { return S::stage0 + (i & 1) * S::stage_bytes + S::st_v; };
  uint32_t seq0 = 0;                                  // tiles streamed before this chunk
  uint32_t ph_s = 0, ph_sc = 0;                       // score group: phases of R_S, R_SCORES
  uint32_t nit = 0;                                   // attention group: tiles so far
  int n_seen = c.n_seen;

#pragma unroll 1
  for (int chunk = 0; chunk < n_chunks; ++chunk) {
    plan_call(L, c, n_seen, n, false);
    const int cg = c.count_g, cw = c.att_wn, nE = cg + c.r;
    const bool sel = c.mode == UPD_SELECT;
    const int nF = sel ? nE - lam : 0;
    const int nGB = (cg + 63) / 64, nRB = (cw + 63) / 64;
    const int n_score = sel ? (nGB + nRB + 1) / 2 : 0;
    const int n_tiles = want_out ? (nGB + nRB + (n + 63) / 64 + 1) / 2 : 0;
    const int ring0 = c.r_pos0 % eta;                  // ring slot of the oldest leaving pair
    uint32_t seq = seq0;                               // tiles streamed so far (every role counts for itself)
    seq0 += (uint32_t)(want_out ? n_tiles : n_score > rank ? (n_score - rank + K - 1) / K : 0);

    if (warp == 16) {
      // =============================== key and value tiles ===============================
      if (tc::elect_one()) {
#pragma unroll 1
        for (TileOrder o(rank, K, n_score, n_tiles); o.own || !o.done(); o.next(), ++seq) {
            const uint32_t st = seq & 1, par = ((seq >> 1) & 1) ^ 1;
            if (seq >= 2) WAIT(R_KEMPTY + st, par);
            if (!ok) break;                            // (a wait gave up: nothing more is requested)
#pragma unroll 1
            for (int isv = 0; isv < 2; ++isv) {
              if (isv && seq >= 2) WAIT(R_VEMPTY + st, par);
              if (!ok) break;
              const uint32_t dst = sbase + (isv ? stage_v(seq) : stage_k(seq)), bar = BAR((isv ? R_VFULL : R_KFULL) + st);
              tc::mbar_expect_tx(bar, (uint32_t)kblk * 16384u);
              if (o.t * 2 + 1 < nGB) {
                tc::tma_load_slots(dst, isv ? &M.gv : &M.gk, o.t, unit, bar);
                continue;
              }
#pragma unroll 1
              for (int hb = 0; hb < 2; ++hb) {
                const int blk = o.t * 2 + hb;
#pragma unroll
                for (int cb = 0; cb < kblk; ++cb) {
                  const uint32_t dd = dst + (uint32_t)cb * 16384u + (uint32_t)hb * 8192u;
                  if (blk < nGB) tc::tma_load_3d(dd, isv ? &M.gv.block : &M.gk.block, cb * 64, blk * 64, unit, bar);
                  else if (blk < nGB + nRB) tc::tma_load_3d(dd, isv ? &M.wv : &M.wk, cb * 64, (blk - nGB) * 64, unit, bar);
                  else tc::tma_load_5d(dd, isv ? &M.v : &M.k, cb * 64, h, (blk - nGB - nRB) * 64, b, chunk, bar);   // (beyond the chunk: zeros)
                }
              }
            }
        }
      }
      __syncwarp();
    } else if (warp == 17) {
      // =============================== queries, Z = K Q^T ===============================
      if (tc::elect_one()) {
        const uint64_t dq = tc::make_desc_sw128(sbase + S::q, 16, 1024), dw = tc::make_desc_sw128(sbase + S::wt, 16, 1024);
        const uint32_t idz = tc::make_idesc_bf16(128, NQ, false, false);
        if (!want_out)
          for (TileOrder o(rank, K, n_score, 0); o.own; o.next(), ++seq) {   // (the score group alone reads the tiles)
            WAIT(R_KFULL + (seq & 1), (seq >> 1) & 1);
            tc::mbar_arrive(BAR(R_KEMPTY + (seq & 1)));
          }
        // the queries of chunk ch2: loaded once the last Z product has read the ones before; U_Q = Q W over the Z buffers
        // once the attention group is through with the chunk (rows beyond NQ are whatever follows the queries in shared
        // memory; not read).  Neither depends on the memories
        auto load_q = [&](int ch2) {
          tc::mbar_expect_tx(BAR(R_QFULL), (uint32_t)IP * kblk * 4096u);
#pragma unroll
          for (int j = 0; j < IP; ++j) {
            const int it = it0 + j, hl = it / ntb;
            const int head = it < items ? h * g + hl : L.Hq;   // (a head index outside the tensor reads as zeros)
#pragma unroll
            for (int cb = 0; cb < kblk; ++cb)
              tc::tma_load_5d(sbase + S::q + (uint32_t)(cb * NQ * 128 + j * 4096), &M.q, cb * 64, head, (it - hl * ntb) * 32, b, ch2, BAR(R_QFULL));
          }
        };
        auto issue_uq = [&](uint32_t ph) {
          WAIT(R_QFULL, ph & 1);
          tc::fence_after_sync();
#pragma unroll
          for (int ks = 0; ks < d / 16; ++ks)
            tc::mma_bf16_ss(tm_z, dq + (uint64_t)(((ks >> 2) * (NQ * 128) + (ks & 3) * 32) >> 4), dw + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4),
                            tc::make_idesc_bf16(128, 64, false, false), ks > 0);
          tc::mma_commit(BAR(R_UQ));
        };
        if (want_out) {
          if (chunk == 0) { load_q(0); issue_uq(0); }
          WAIT(R_PHIQ, chunk & 1);                     // U_Q is read
#pragma unroll 1
          for (TileOrder o(rank, K, n_score, n_tiles); o.own || !o.done(); o.next(), ++seq) {
            const uint32_t st = seq & 1, z = seq & 1;
            WAIT(R_KFULL + st, (seq >> 1) & 1);
            if (seq >= 2) WAIT(R_ZFREE + z, ((seq >> 1) & 1) ^ 1);
            tc::fence_after_sync();
            const uint64_t dk = tc::make_desc_sw128(sbase + stage_k(seq), 16, 1024);
#pragma unroll
            for (int ks = 0; ks < d / 16; ++ks)
              tc::mma_bf16_ss(tm_z + z * NQ, dk + (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4),
                              dq + (uint64_t)(((ks >> 2) * (NQ * 128) + (ks & 3) * 32) >> 4), idz, ks > 0);
            tc::mma_commit(BAR(R_ZFULL + z));
            tc::mma_commit(BAR(R_KEMPTY + st));
            if (!o.own) tc::mbar_arrive(BAR(R_KEMPTY + st));
          }
          if (chunk + 1 < n_chunks) {
            WAIT(R_ZFULL + ((seq - 1) & 1), ((seq - 1) >> 1) & 1);
            load_q(chunk + 1);
            WAIT(R_OFREE, chunk & 1);
            issue_uq((uint32_t)chunk + 1);
          }
        }
      }
      __syncwarp();
    } else if (warp == 18) {
      // =============================== O^T products ===============================
      if (tc::elect_one()) {
        const uint64_t dh = tc::make_desc_sw128(sbase + S::ht, 16, 1024), dp = tc::make_desc_sw128(sbase + S::pt, 16, 1024);
        if (!want_out)
          for (TileOrder o(rank, K, n_score, 0); o.own; o.next(), ++seq) {
            WAIT(R_VFULL + (seq & 1), (seq >> 1) & 1);
            tc::mbar_arrive(BAR(R_VEMPTY + (seq & 1)));
          }
        if (want_out) {
          WAIT(R_PHIQ, chunk & 1);                     // (phi(Q), made at the end of the chunk before)
          tc::fence_after_sync();
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            tc::mma_bf16_ss(tm_o, dh + (uint64_t)(((ks >> 2) * S::ht_blk + (ks & 3) * 32) >> 4), dp + (uint64_t)(((ks >> 2) * (NQ * 128) + (ks & 3) * 32) >> 4),
                            tc::make_idesc_bf16(128, NQ, false, false), ks > 0);
          tc::mma_commit(BAR(R_LIN));
#pragma unroll 1
          for (TileOrder o(rank, K, n_score, n_tiles); o.own || !o.done(); o.next(), ++seq) {
            const uint32_t st = seq & 1, pb = seq & (NB - 1);
            WAIT(R_VFULL + st, (seq >> 1) & 1);
            WAIT(R_PT + pb, (seq / NB) & 1);
            tc::fence_after_sync();
            const uint64_t dv = tc::make_desc_sw128(sbase + stage_v(seq), 16384, 1024);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              tc::mma_bf16_ss(tm_o, dv + (uint64_t)((ks * 2048) >> 4), dp + (uint64_t)((ks * 2048 + pb * 64) >> 4), tc::make_idesc_bf16(128, NQ, true, true), 1u);
            tc::mma_commit(BAR(R_O + pb));
            tc::mma_commit(BAR(R_VEMPTY + st));
            if (!o.own) tc::mbar_arrive(BAR(R_VEMPTY + st));
          }
        }
      }
      __syncwarp();
    } else if (warp >= 8) {
      // =============================== attention group ===============================
      // phi(Q): thread (query row t, half hf of the features), bf16 into its operand rows
      auto make_phiq = [&](uint32_t ph) {
        if (wq < NQ / 32) {
          WAIT(R_UQ, ph & 1);
          tc::fence_after_sync();
          uint32_t u[64], pk2[32];
          tc::tmem_ld64u(tm_z + lane_addr, u);
          tc::phi_half(u, hf != 0, L.phi_kind == 1, pk2);
          if (c.att_flags & 1) {                       // the queries do not see H, s
#pragma unroll
            for (int i = 0; i < 32; ++i) pk2[i] = 0u;
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<uint4*>(sm + S::pt + hf * (NQ * 128) + tc::sw128_off(t, q)) = make_uint4(pk2[4 * q], pk2[4 * q + 1], pk2[4 * q + 2], pk2[4 * q + 3]);
          tc::fence_async_smem();
          tc::fence_before_sync();
          tc::mbar_arrive(BAR(R_PHIQ));
        }
      };
      if (want_out) {
        if (chunk == 0) { make_phiq(0); tc::named_bar_sync(2, 256); }
        int tok0[HQ / 16];                             // first token of this thread's groups of 16 queries
#pragma unroll
        for (int sb = 0; sb < HQ / 16; ++sb) tok0[sb] = ((it0 + ((hf * HQ + sb * 16) >> 5)) % ntb) * 32 + ((hf * HQ + sb * 16) & 31);
        if (gtid < NQ * 2) {                           // phi(q) . s, half of the features each; stabiliser max(0, max z)
          const int r = gtid % NQ, half = gtid / NQ;
          float a0 = 0.f, a1 = 0.f;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint4 raw = *reinterpret_cast<const uint4*>(sm + S::pt + half * (NQ * 128) + tc::sw128_off(r, q));
            const float* sv = &X.s[half * 64 + q * 8];
            a0 = fmaf(bf16lo_f(raw.x), sv[0], a0); a1 = fmaf(bf16hi_f(raw.x), sv[1], a1);
            a0 = fmaf(bf16lo_f(raw.y), sv[2], a0); a1 = fmaf(bf16hi_f(raw.y), sv[3], a1);
            a0 = fmaf(bf16lo_f(raw.z), sv[4], a0); a1 = fmaf(bf16hi_f(raw.z), sv[5], a1);
            a0 = fmaf(bf16lo_f(raw.w), sv[6], a0); a1 = fmaf(bf16hi_f(raw.w), sv[7], a1);
          }
          X.lden[half][r] = a0 + a1;
          if (half == 0) X.m[r] = 0.f;
        }
        tc::named_bar_sync(2, 256);
        uint64_t lpart[HQ / 2];                        // sums of the weights, packed pairs
#pragma unroll
        for (int j = 0; j < HQ / 2; ++j) lpart[j] = 0;
        const uint64_t sl22 = tc::pack_f2(sl2, sl2);
        const uint32_t nit0 = nit;
#pragma unroll 1
        for (TileOrder o(rank, K, n_score, n_tiles); o.own || !o.done(); o.next(), ++nit) {
          const uint32_t z = nit & 1, slot3 = nit % 3u, pb = nit & (NB - 1);
          // what this thread's key row is: visible to every query, to none, or to the chunk's tokens from its own on
          const int blk = 2 * o.t + (t >> 6), ro = t & 63;
          int first = 1 << 20;                         // first token that sees the row
          if (blk < nGB) { if (blk * 64 + ro < c.att_g) first = 0; }
          else if (blk < nGB + nRB) { if ((blk - nGB) * 64 + ro < cw) first = 0; }
          else first = (blk - nGB - nRB) * 64 + ro;
          const bool partial = __any_sync(0xffffffffu, first > 0);
          if (t == 0) X.grow[(nit + 1) % 3u][hf] = 0;
          WAIT(R_ZFULL + z, (nit >> 1) & 1);
          tc::fence_after_sync();
          float v[HQ / 16][16];
          float mx = 0.f;
#pragma unroll
          for (int sb = 0; sb < HQ / 16; ++sb) {
            tc::tmem_ld16(tm_z + z * NQ + lane_addr + hf * HQ + sb * 16, v[sb]);
            if (partial) {
#pragma unroll
              for (int j = 0; j < 16; ++j) v[sb][j] = first <= tok0[sb] + j ? v[sb][j] : -CUDART_INF_F;
            }
#pragma unroll
            for (int j = 0; j < 16; j += 2) mx = tc::max3(mx, v[sb][j], v[sb][j + 1]);
          }
          tc::fence_before_sync();
          tc::mbar_arrive(BAR(R_ZFREE + z));           // Z is in registers
          // The weights keep their relative precision whatever the stabiliser is (bf16 has fp32's range), so it stays 0
          // until a score could overflow the sums: one comparison a tile instead of a maximum per query
          if (__any_sync(0xffffffffu, mx * sl2 > kGrow) && lane == 0) X.grow[slot3][hf] = 1;
          tc::named_bar_sync(4 + hf, 128);             // the four warps of these columns
          const bool grow = *reinterpret_cast<volatile int*>(&X.grow[slot3][hf]) != 0;
          // the product that read this buffer is complete (for the first tile: the linear term, whose phi(Q) lies there)
          if (nit == nit0) WAIT(R_LIN, chunk & 1);
          if (nit >= NB) WAIT(R_O + pb, (nit / NB - 1) & 1);
          if (grow) {                                  // rare, uniform over the four warps
            if (NB > 1 && nit > 0) WAIT(R_O + (pb ^ 1), ((nit - 1) / NB) & 1);   // O^T is moved: the product before, too
            tc::fence_after_sync();
#pragma unroll
            for (int sb = 0; sb < HQ / 16; ++sb) {
              const float cm = cols_reduce16<true>(v[sb], lane) * sl2;
              if (!(lane & 1)) X.redm[wq][hf * HQ + sb * 16 + (lane >> 1)] = cm;
            }
            tc::named_bar_sync(4 + hf, 128);
#pragma unroll
            for (int sb = 0; sb < HQ / 16; ++sb) {
              float ov[16];
              tc::tmem_ld16(tm_o + lane_addr + hf * HQ + sb * 16, ov);
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int col = hf * HQ + sb * 16 + j;
                const float mo = X.m[col], mn = fmaxf(fmaxf(mo, fmaxf(X.redm[0][col], X.redm[1][col])), fmaxf(X.redm[2][col], X.redm[3][col]));
                const float alpha = tc::fast_exp2(mo - mn);
                ov[j] *= alpha;
                float l0, l1;
                tc::unpack_f2(lpart[sb * 8 + j / 2], l0, l1);
                lpart[sb * 8 + j / 2] = j & 1 ? tc::pack_f2(l0, l1 * alpha) : tc::pack_f2(l0 * alpha, l1);
              }
#pragma unroll
              for (int j = 0; j < 16; j += 8) tc::tmem_st8(tm_o + lane_addr + hf * HQ + sb * 16 + j, *reinterpret_cast<float(*)[8]>(&ov[j]));
            }
            tc::named_bar_sync(4 + hf, 128);
            if (t < HQ) {
              const int col = hf * HQ + t;
              const float mo = X.m[col], mn = fmaxf(fmaxf(mo, fmaxf(X.redm[0][col], X.redm[1][col])), fmaxf(X.redm[2][col], X.redm[3][col]));
              const float alpha = tc::fast_exp2(mo - mn);
              X.lden[0][col] *= alpha;
              X.lden[1][col] *= alpha;
              X.m[col] = mn;
            }
            tc::named_bar_sync(4 + hf, 128);
          }
          // weights (bf16) of this key for HQ queries: consecutive in its row of the operand
#pragma unroll
          for (int j = 0; j < HQ; j += 8) {
            uint32_t pk[4];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              const uint64_t m2 = *reinterpret_cast<const uint64_t*>(&X.m[hf * HQ + j + i]) ^ 0x8000000080000000ull;
              float x0, x1;
              tc::unpack_f2(tc::fma2(tc::pack_f2(v[j / 16][j % 16 + i], v[j / 16][j % 16 + i + 1]), sl22, m2), x0, x1);
              const float p0 = tc::fast_exp2(x0), p1 = tc::fast_exp2(x1);
              lpart[(j + i) / 2] = tc::add2(lpart[(j + i) / 2], tc::pack_f2(p0, p1));
              pk[i / 2] = pack_bf16x2(p0, p1);
            }
            *reinterpret_cast<uint4*>(sm + S::pt + tc::sw128_off(t, (int)pb * 4 + ((hf * HQ + j) >> 3))) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
          tc::fence_async_smem();
          tc::fence_before_sync();
          tc::mbar_arrive(BAR(R_PT + pb));
        }
        // ---- the sums of the weights, then the outputs
#pragma unroll
        for (int sb = 0; sb < HQ / 16; ++sb) {
          float lv[16];
#pragma unroll
          for (int j = 0; j < 8; ++j) tc::unpack_f2(lpart[sb * 8 + j], lv[2 * j], lv[2 * j + 1]);
          const float l = cols_reduce16<false>(lv, lane);
          if (!(lane & 1)) X.l_s[wq][hf * HQ + sb * 16 + (lane >> 1)] = l;
        }
        tc::named_bar_sync(2, 256);
        if (gtid < NQ) X.inv[gtid] = 1.0f / (((X.l_s[0][gtid] + X.l_s[1][gtid]) + (X.l_s[2][gtid] + X.l_s[3][gtid])) + (X.lden[0][gtid] + X.lden[1][gtid]));
        WAIT(R_O + ((nit - 1) & (NB - 1)), ((nit - 1) / NB) & 1);   // O^T is complete
        tc::fence_after_sync();
        tc::named_bar_sync(2, 256);
#pragma unroll
        for (int sb = 0; sb < HQ / 16; ++sb) {
          float v[16];
          tc::tmem_ld16(tm_o + lane_addr + hf * HQ + sb * 16, v);
          const int col0 = hf * HQ + sb * 16, it = it0 + (col0 >> 5), hl = it / ntb;
          if (t < d && it < items && ok) {
            T* op = (T*)c.out + (((size_t)(chunk * L.B + b) * n + tok0[sb]) * L.Hq + h * g + hl) * d + t;
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (tok0[sb] + j < n) op[(size_t)j * L.Hq * d] = __float2bfloat16_rn(v[j] * X.inv[col0 + j]);
          }
        }
        tc::fence_before_sync();
        tc::mbar_arrive(BAR(R_OFREE));
      }
      tc::fence_async_all();
      tc::named_bar_arrive(3, 512);                    // this block's tiles are no longer needed
      tc::fence_before_sync();
      tc::cluster_arrive();                            // (A) this warp has read all it needs of the old memories
      if (want_out && chunk + 1 < n_chunks) make_phiq((uint32_t)chunk + 1);
      tc::cluster_wait();                              // (A)
      // a warp per incoming token (half a warp each for key and value): the pair whose ring slot it takes first moves
      // into the sparse cache if it stays
      const int ch = lane & 15;
      const bool isv = lane >= 16;
#pragma unroll 1
      for (int ci = rank * 8 + (warp - 8); ci < n; ci += K * 8) {
        const int p = n_seen + ci, slot = p % eta, i = p - eta - c.r_pos0;
        const int to = i >= 0 && i < c.r ? X.dst[i] : -1;
        const bool enters = ci >= n - eta;
        if (ch < d / 8 && ok) {
          T* ring = (T*)(isv ? L.wv : L.wk) + ((size_t)unit * eta + slot) * d + ch * 8;
          uint4 o4, n4;
          if (to >= 0) o4 = __ldcg(reinterpret_cast<const uint4*>(ring));
          if (enters) n4 = *reinterpret_cast<const uint4*>((const T*)(isv ? c.v : c.k) + (((size_t)(chunk * L.B + b) * n + ci) * L.Hkv + h) * d + ch * 8);
          if (to >= 0) *reinterpret_cast<uint4*>((T*)(isv ? L.gv : L.gk) + ((size_t)unit * lam + to) * d + ch * 8) = o4;
          if (enters) *reinterpret_cast<uint4*>(ring) = n4;
        }
        if (to >= 0 && lane == 0 && ok) {
          L.gpos[(size_t)unit * lam + to] = c.r_pos0 + i;
          scu[to] = sel ? __uint_as_float(X.key[cg + i]) : CUDART_NAN_F;
        }
      }
    } else {
      // =============================== score group ===============================
      if (sel) {
        const uint64_t dw = tc::make_desc_sw128(sbase + S::wt, 16, 1024), dh = tc::make_desc_sw128(sbase + S::ht, 16, 1024);
        const uint32_t id_u = tc::make_idesc_bf16(128, 64, false, false), id_p = tc::make_idesc_bf16(128, d + 16, false, false);
        auto sync = [] { tc::named_bar_sync(1, 256); };
#pragma unroll 1
        for (int tile = rank; tile < n_score; tile += K, ++seq) {
          const uint32_t st = seq & 1, par = (seq >> 1) & 1;
          // member of E this row holds (-1: none)
          const int blk = 2 * tile + (t >> 6), ro = t & 63;
          int e = -1;
          if (blk < nGB) { if (blk * 64 + ro < cg) e = blk * 64 + ro; }
          else if (blk < nGB + nRB) {
            int i = (blk - nGB) * 64 + ro - ring0;
            if (i < 0) i += eta;
            if ((blk - nGB) * 64 + ro < cw && i < c.r) e = cg + i;
          }
          // (the key tile's barrier may complete again before a late warp has looked at it: the issuing warp alone must wait)
          if (warp == 0) WAIT(R_KFULL + st, par); else tc::mbar_try_wait(BAR(R_KFULL + st), par);
          tc::fence_after_sync();
          if (warp == 0 && tc::elect_one()) {
            const uint64_t dk = tc::make_desc_sw128(sbase + stage_k(seq), 16, 1024);
#pragma unroll
            for (int ks = 0; ks < d / 16; ++ks)
              tc::mma_bf16_ss(tm_u, dk + (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4), dw + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4), id_u, ks > 0);
            tc::mma_commit(BAR(R_S));
            tc::mma_commit(BAR(R_KEMPTY + st));
          }
          WAIT(R_S, ph_s & 1);
          ++ph_s;
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
          if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)
              tc::mma_bf16_ts(tm_p, tm_u + ks * 8, dh + (uint64_t)(((ks >> 2) * S::ht_blk + (ks & 3) * 32) >> 4), id_p, ks > 0);
            tc::mma_commit(BAR(R_S));
          }
          WAIT(R_VFULL + st, par);
          WAIT(R_S, ph_s & 1);
          ++ph_s;
          tc::fence_after_sync();
          constexpr int HC = d / 2;
          uint64_t ninv2 = 0, accA = tc::pack_f2(0.f, 0.f), accB = accA;
          const uint8_t* vt = sm + stage_v(seq);
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
          if (hf == 1) X.ssp[t] = ss;
          tc::fence_before_sync();
          sync();                                      // both halves are done with the value tile and with P
          tc::fence_after_sync();
          if (tid == 0) tc::mbar_arrive(BAR(R_VEMPTY + st));
          if (hf == 0) {
            const float sc = sqrtf(ss + X.ssp[t]);
            const uint32_t sb = __float_as_uint(sc), ka = sbase + S::misc + (uint32_t)offsetof(Misc, key);
            const int e0 = __shfl_sync(0xffffffffu, e, 0);
            if (__all_sync(0xffffffffu, e >= 0 && e == e0 + lane && (e0 & 3) == 0)) {
              // four scores a message, each of the four lanes that hold them for every fourth block (single scores kept
              // the receiving blocks busy for 1 us)
              const int l4 = lane & ~3;
              const uint4 q4 = make_uint4(__shfl_sync(0xffffffffu, sb, l4), __shfl_sync(0xffffffffu, sb, l4 + 1), __shfl_sync(0xffffffffu, sb, l4 + 2),
                                          __shfl_sync(0xffffffffu, sb, l4 + 3));
              for (int r = lane & 3; r < K; r += 4) tc::st_async_v4(tc::map_rank(ka + (uint32_t)(e0 + l4) * 4u, (uint32_t)r), q4, tc::map_rank(BAR(R_SCORES), (uint32_t)r));
            } else if (e >= 0) {
              for (int r = 0; r < K; ++r) tc::st_async_u32(tc::map_rank(ka + (uint32_t)e * 4u, (uint32_t)r), sb, tc::map_rank(BAR(R_SCORES), (uint32_t)r));
            }
            if (ok && e >= 0) scu[e < cg ? e : lam + (e - cg)] = sc;
          }
        }
        if (tid == 0) tc::mbar_expect_tx(BAR(R_SCORES), (uint32_t)nE * 4u);
        WAIT(R_SCORES, ph_sc & 1);                     // the scores of all blocks are here
        ++ph_sc;
        constexpr int PPR = d / 4;                     // 16-byte pieces of a pair: key, then value
        constexpr int NP = kUp2Batch * PPR / 256;
        uint4 val[NP];                                 // the folded pairs, on their way as soon as they are known
        const int isv = (tid % PPR) / (PPR / 2), ch = tid % (PPR / 2);
        select_lists<256>(X.key, [&](int e) { return e < cg ? __ldcg(L.gpos + (size_t)unit * lam + e) : c.r_pos0 + (e - cg); }, X.cand, X.mark, nE, nF, cg,
                          X.fold, X.sel, tid, sync, [&](int i, int to) { X.dst[i] = (short)to; }, [&] {
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            const int row = tid / PPR + q * (256 / PPR);
            val[q] = make_uint4(0, 0, 0, 0);
            if (row < nF) {
              const int e = X.fold[row];
              int slot = ring0 + e - cg;
              if (slot >= eta) slot -= eta;
              const T* base = e < cg ? (const T*)(isv ? L.gv : L.gk) + ((size_t)unit * lam + e) * d : (const T*)(isv ? L.wv : L.wk) + ((size_t)unit * eta + slot) * d;
              val[q] = __ldcg(reinterpret_cast<const uint4*>(base + ch * 8));
            }
          }
        });
        if (rank == 0 && tid == 0 && ok) {
          L.thr[(size_t)unit * 2 + 0] = __uint_as_float(X.sel.min_keep);
          L.thr[(size_t)unit * 2 + 1] = __uint_as_float(X.sel.max_fold);
        }
        // ---- Eq. 13: dH = phi(K_S)^T [V_S | 1], phi in two or three bf16 parts against the same values
        const bool three = THREE && fold_in_three(c);
        const int dK = d / K, dKs = 31 - __clz(dK), c0 = rank * dK, part = dK / 2, ld = dK + 4;
        float* stg = reinterpret_cast<float*>(sm + S::fold_h);   // [128][ld]
        float hv[8];
        auto load_h = [&](int it) {
#pragma unroll
          for (int j = 0; j < 8; ++j) hv[j] = Hg[(size_t)((it >> dKs) * 8 + j) * d + c0 + (it & (dK - 1))];
        };
        {
          tc::named_bar_sync(3, 512);                  // the attention group is done with the stages, which the tiles lie over
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            const int row = tid / PPR + q * (256 / PPR);
            uint8_t* dst = sm + (isv ? S::fold_v : S::fold_k) + (ch >> 3) * 16384;
            *reinterpret_cast<uint4*>(dst + tc::sw128_off(row, ch & 7)) = val[q];
            if (!isv) *reinterpret_cast<uint4*>(dst + tc::sw128_off(row + 64, ch & 7)) = val[q];   // again, for the second parts of phi
          }
          if (tid < 64) {                              // the column of ones and its 15 empty neighbours
            uint4 one = make_uint4(0, 0, 0, 0);
            if (tid < nF) one.x = 0x3f80u;
            *reinterpret_cast<uint4*>(sm + S::fold_v + kblk * 16384 + tc::sw128_off(tid, 0)) = one;
            *reinterpret_cast<uint4*>(sm + S::fold_v + kblk * 16384 + tc::sw128_off(tid, 1)) = make_uint4(0, 0, 0, 0);
          }
          tc::fence_async_smem();
          tc::fence_before_sync();
          tc::cluster_arrive();                        // (A)
          sync();
          tc::fence_after_sync();
          if (warp == 0 && tc::elect_one()) {
#pragma unroll
            for (int ks = 0; ks < d / 16; ++ks)
              tc::mma_bf16_ss(tm_u, tc::make_desc_sw128(sbase + S::fold_k + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024),
                              dw + (uint64_t)(((ks >> 2) * 8192 + (ks & 3) * 32) >> 4), id_u, ks > 0);
            tc::mma_commit(BAR(R_S));
          }
          WAIT(R_S, ph_s & 1);
          ++ph_s;
          tc::fence_after_sync();
          {
            // lanes t and t + 64 hold the same pair and take 32 features of their half each: first parts into rows 0-63, second
            // ones into 64-127; the third ones, if taken, into the rows of the value tile that hold no pair
            const bool ek = L.phi_kind == 1;
            const int pr = t & 63, qh = t >> 6;
            uint32_t u[32];
            uint64_t x2[16];
            float m, sum, f = 1.0f;
            tc::tmem_ld32u(tm_u + lane_addr + qh * 32, u);
            tc::phi_quarter_f32(u, hf != 0, ek, x2, m, sum);
            if (!ek) {
              X.phx[hf][t] = make_float2(m, sum);
              tc::named_bar_sync(6 + hf * 2 + (wq & 1), 64);   // the two warps that share these pairs
              const float2 o = X.phx[hf][t ^ 64];
              const float mm = fmaxf(m, o.x), a = tc::fast_exp2(m - mm);
              f = a / fmaf(sum, a, o.y * tc::fast_exp2(o.x - mm));
            }
            const uint64_t f2 = tc::pack_f2(f, f);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t p1[4], p2[4], p3[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                float a, b;
                tc::unpack_f2(tc::mul2(x2[q * 4 + e], f2), a, b);
                p1[e] = tc::next_part(a, b);
                p2[e] = tc::next_part(a, b);
                if (THREE) p3[e] = tc::next_part(a, b);
              }
              const uint32_t off = tc::sw128_off(pr, qh * 4 + q), dst = S::fold_k + hf * 16384;
              *reinterpret_cast<uint4*>(sm + dst + off) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
              *reinterpret_cast<uint4*>(sm + dst + 8192 + off) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
              if (THREE && three) *reinterpret_cast<uint4*>(sm + S::fold_v + hf * 16384 + 8192 + off) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
            }
          }
          tc::fence_async_smem();
          tc::fence_before_sync();
          sync();
          tc::fence_after_sync();
          if (warp == 0 && tc::elect_one()) {
            tc::fold_product<DPL, THREE>(tm_p, sbase + S::fold_k, sbase + S::fold_v, three);
            tc::mma_commit(BAR(R_S));
          }
          if (tid < dK * 16) load_h(tid);
          WAIT(R_S, ph_s & 1);
          ++ph_s;
          tc::fence_after_sync();
          // dH, this block's columns, through shared memory
#pragma unroll 1
          for (int q = 0; q < part; q += 4) {
            float p[4];
            tc::tmem_ld4(tm_p + lane_addr + c0 + hf * part + q, p);
            *reinterpret_cast<float4*>(stg + t * ld + hf * part + q) = make_float4(p[0], p[1], p[2], p[3]);
          }
          if (hf == 0) {
            float ds[2];
            tc::tmem_ld2(tm_p + lane_addr + d, ds);
            const float sv = X.s[t] + ds[0];
            put_s(t, sv);
            if (rank == 0 && ok) L.s[(size_t)unit * D + t] = sv;
          }
        }
        // this block's columns of dH into H (fp32, in memory) and, rounded, into the operand image: here at once, in the
        // other blocks when all have read the old one (A).  A thread has 8 rows of one column, 16 bytes of the image, and
        // lanes have neighbouring columns of H
        sync();
#pragma unroll 1
        for (int it = tid; it < dK * 16; it += 256) {
          const int cc = it & (dK - 1), jc = it >> dKs;
          if (it != tid) load_h(it);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            hv[j] += stg[(jc * 8 + j) * ld + cc];
            if (ok) Hg[(size_t)(jc * 8 + j) * d + c0 + cc] = hv[j];
          }
          *reinterpret_cast<uint4*>(sm + S::ht + (jc >> 3) * S::ht_blk + tc::sw128_off(c0 + cc, jc & 7)) = tc::pack8_bf16(hv);
        }
        sync();
        tc::cluster_wait();                            // (A)
        for (int i = tid; i < dK * 16; i += 256) {
          const uint32_t off = S::ht + (uint32_t)((i >> 3) & 1) * S::ht_blk + (uint32_t)(c0 + (i >> 4)) * 128u + (uint32_t)(i & 7) * 16u;
          const uint4 v = *reinterpret_cast<const uint4*>(sm + off);
          for (int r = 1; r < K; ++r) tc::st_cluster_v4(tc::map_rank(sbase + off, (uint32_t)((rank + r) & (K - 1))), v);
        }
      } else {
        for (int i = tid; i < c.r; i += 256) X.dst[i] = (short)(c.mode == UPD_APPEND ? cg + i : -1);
        tc::named_bar_sync(3, 512);
        tc::cluster_arrive();
        tc::cluster_wait();                            // (A)
      }
    }
    if (warp >= 16) {
      tc::fence_before_sync();
      tc::cluster_arrive();
      tc::cluster_wait();                              // (A)
    }
    if (warp < 16) tc::fence_async_all();              // what was written is read by TMA and tensor cores next
    tc::fence_before_sync();
    tc::cluster_arrive();
    tc::cluster_wait();
    if (warp >= 16 || warp == 0) tc::fence_async_all();
    tc::fence_after_sync();
    n_seen += n;
  }
  if (!ok) *abw = 1;
  __syncthreads();
  if (X.abort_word != 0) __nanosleep(200000);         // (after a failure: copies on their way into this block's memory arrive first)
  if (tid == 0 && X.abort_word != 0) atomicOr(L.status, 256);
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace lola
