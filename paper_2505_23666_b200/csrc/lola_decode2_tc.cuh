// The generation step (Eq. 11-14) as ONE kernel for bf16 layers with F = 64, one CTA per (batch row, KV head)
// unit; the unit's memories are streamed once from HBM by TMA and everything that depends on them is computed on
// the way.  Rows of the stream: the occupied sparse-cache slots, then (from the next multiple of 64) the window
// ring slots, in tiles of 128 rows; rows that hold no pair are masked.  Per tile:
//     [U | Z] = K_tile [W | Q^T]          tcgen05.mma  M=128, N=80,   K=d   (pre-activations, q.k)
//     phi = feature map of U, rounded to bf16
//     [P | den] = phi [H | s_hi s_lo]      tcgen05.mma  M=128, N=d+16, K=128 (s split in two bf16 parts)
//     score = || P / den - v ||            for sparse-cache rows and the evicted pair (Eq. 10)
//     O^T += V_tile^T Pr^T                 tcgen05.mma  M=d(128), N=16, K=128 (Eq. 14 numerator),
//                                          Pr = exp(z - m) with a running maximum per query row
// The linear term uses the state after the fold: phi(q)^T H_old (an MMA that initialises O^T with weight
// exp(0 - m), the m = max(0, .) stabiliser) plus (phi(q) . phi_fold) v_fold.
// While the caches still fill (UPD_NONE, UPD_APPEND) no row is scored and nothing is folded; the leaving pair, if
// there is one, takes the next free slot.
//
// The work is organised as a pipeline of roles:
//
//   feature group (warps 0-7)   per tile: q.k columns and their warp maxima into shared memory, the
//                               feature map of U into tensor memory; no barrier inside the group
//   score group   (warps 8-15)  per tile: running maxima and softmax weights (bf16) into the Pr^T operand,
//                               Eq. 10 from [P | den] and the value tile, the running sums of the weights,
//                               and per row quadrant (a pair of warps) the lowest-scored pair so far
//   warp 16, one thread         issues [P | den] = phi [H | s] (and the linear term H^T phi(Q)^T once)
//   warp 17, one thread         issues O^T += V^T Pr^T; value-tile loads
//   warp 18, one thread         issues [U | Z] = K [W | Q^T]; key-tile loads
//
// The two groups work on different tiles at the same time: [U | Z] and phi are double-buffered in
// tensor memory, so while the score group is busy with tile t the feature group already works on
// tile t + 1 and the tensor core on the products between them.  Every hand-over is an mbarrier; every
// wait is bounded, and a wait that runs out raises the block's abort word (bit 8 of the status word).
//
// The pair to fold is only known after the last tile.  Every row is therefore attended by the O^T products;
// each quadrant keeps (q.k, stabiliser, value row, feature row) of its lowest-scored pair, and the epilogue
// takes the overall lowest out of O^T and the weight sums again (its bf16 weight times its bf16 value row is
// exact in fp32, so what is subtracted is what the product added, up to the rounding of the running sum).  Where the folded
// pair held all but 1 / 256 of a row's weight, that rounding is too much, and the row is attended again without the pair.
// The score group's warps only meet their quadrant partner inside a tile (a 64-thread barrier); a slow warp
// holds up its partner and the hand-over to the O^T product, not the other quadrants.
//
// SPLIT: a cluster of K blocks per unit.  A unit is a chain of up to 7 tiles of 2 us between 6 us of set-up and 3 us of
// epilogue, so where there are fewer units than SMs the tiles are dealt out (block k: tiles k, k + K, ..).  Everything
// a tile adds is a sum or a minimum: O^T, the weight sums and the lowest pairs stay where they are, and after one
// cluster barrier each block reads the lowest pair of all (a second round trip fetches its rows) and folds its rows
// of H, block 0 adds up the outputs, the last block moves the pairs.
#pragma once
#include <cuda.h>

#include "lola_generic.cuh"
#include "lola_tc.cuh"

namespace lola {

constexpr int kDecQ = 8;          // query rows per unit the kernel carries (group size g <= 8)
constexpr int kDecNarrowTiles = 16;  // tiles of a unit up to which a step on full caches takes 16-bit operands

template <int DPL>
struct DecodeSmem {
  static constexpr int d = DPL * 32;
  static constexpr int kblk = d / 64;
  static constexpr uint32_t b1_blk = 80 * 128;                       // one K block of [W^T ; Q]: 80 rows
  static constexpr uint32_t b1 = 0;                                  // [kblk][80][128B]
  static constexpr uint32_t ht_blk = (d + 16) * 128;                 // one j block of [H^T ; s_hi ; s_lo ; ...]
  static constexpr uint32_t ht = 2 * b1_blk;                         // K-major: [2 j blocks][d + 16 rows][128B]
  static constexpr uint32_t phiq = ht + 2 * (128 + 16) * 128;        // phi(Q), K-major: [2 j blocks][16][128B] (WIDE: fp32 [128][QR])
  static constexpr uint32_t stage0 = phiq + 4096;
  static constexpr uint32_t st_k = 0;                                // K tile [kblk][128][128B]
  static constexpr uint32_t st_v = 32768;                            // V tile [kblk][128 keys][128B]
  static constexpr uint32_t st_pt = 65536;                           // Pr^T, K-major: [2 key blocks][16][128B]
  static constexpr uint32_t stage_bytes = 65536 + 4096;
  static constexpr uint32_t misc = stage0 + 2 * stage_bytes;         // small arrays, see Decode2Misc
  static constexpr uint32_t total = misc + 28672;
  static constexpr uint32_t bytes = total + 1024;                    // slack to align the base to 1024
};

constexpr int kDec2Threads = 608;      // 16 compute warps + 3 issuing warps
constexpr float kDec2Lazy = 8.0f;      // log2 units the running maximum may lag behind before O^T is rescaled

__device__ __forceinline__ int ld_global_i32(const int* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

struct Decode2Misc {
  union {
    float qf[kDecQ][128];        // query rows, fp32
    uint4 peer_rows[8][32];      // SPLIT, after the tiles: feature row and value row of each block's lowest pair
  };
  float phiq_f[kDecQ][128];      // phi(q) as fp32 (rounded to bf16 unless WIDE)
  float u_s[kDecQ][64];
  float knew[128], vnew[128];
  float s_f[128];                // the normaliser state s, fp32
  uint4 ring_kv[2 * 16];         // the pair that leaves the window (key chunks, then value chunks), bf16
  uint4 new_kv[2 * 16];          // the new pair, bf16
  alignas(16) float zn[kDecQ];
  alignas(16) float lden[kDecQ];
  alignas(16) float dotL[kDecQ];
  alignas(16) float redmax[2][4][kDecQ];
  float m_s[1][kDecQ];           // running maxima after the last tile (log2 units)
  float z_s[2][kDecQ][128];      // q.k of the tile's rows (log2 units)
  float ssp[2][128];             // partial squared errors of the second half of the value columns (by tile parity)
  float l_s[4][kDecQ];
  // the lowest-scored pair each of the four row quadrants has seen (its warp keeps the key in registers)
  unsigned long long wb_key[4];
  float wb_a1[4], wb_a2[4];      // the two lowest scores of the quadrant
  float phi_fold[128];           // WIDE: feature row of the folded pair, fp32
  int wb_row[4];
  float wb_z[4][kDecQ];          // q.k of that row (log2 units) ...
  float wb_m[4][kDecQ];          // ... and the stabiliser its weights were taken at
  uint4 wb_v[4][16];             // value row, bf16
  uint4 wb_phi[4][16];           // feature row, bf16
  // SPLIT: of each block's lowest pair its key, score and the runner-up's; its row, and whether the block failed; and per
  // query row its q.k, the stabiliser its weights were taken at, the block's maximum and sum of weights
  uint4 peer_key[8], peer_row[8];
  float peer_f[8][4][kDecQ];
  int redo;                      // rows of whose weight the folded pair held nearly all (decode_redo_row), a bit each
  int failed;
  uint64_t bars[20];
  uint32_t tmem_slot;
  int abort_word;
};
static_assert(sizeof(Decode2Misc) <= 28672, "misc region too small");

// Loads of one tile: two half tiles of 64 rows; a half tile is a block of sparse-cache slots, a block
// of ring slots, or nothing (a box that lies entirely outside the ring tensor reads as zeros).
template <int DPL>
__device__ __forceinline__ void decode_issue_tile(uint32_t dst, const tc::SlotMaps* tm_g, const CUtensorMap* tm_w, int tile,
                                                  int nGB, int nRB, int unit, uint32_t bar) {
  constexpr int kblk = DPL / 2;
  tc::mbar_expect_tx(bar, (uint32_t)kblk * 16384u);
  if (tile * 2 + 1 < nGB) {
    tc::tma_load_slots(dst, tm_g, tile, unit, bar);
    return;
  }
#pragma unroll
  for (int hb = 0; hb < 2; ++hb) {
    const int blk = tile * 2 + hb;
    const bool from_g = blk < nGB;
    const CUtensorMap* tm = from_g ? &tm_g->block : tm_w;
    const int row = from_g ? blk * 64 : min(blk - nGB, nRB) * 64;
#pragma unroll
    for (int cb = 0; cb < kblk; ++cb)
      tc::tma_load_3d(dst + (uint32_t)cb * 16384u + (uint32_t)hb * 8192u, tm, cb * 64, row, unit, bar);
  }
}

// The tile loader as a real function: the issuing threads reach it from many places, and every inlined copy
// would add to an instruction footprint that four different roles already share.
template <int DPL>
__device__ __noinline__ void decode2_issue_tile(uint32_t dst, const tc::SlotMaps* tm_g, const CUtensorMap* tm_w, int tile, int nGB, int nRB,
                                                int unit, uint32_t bar) {
  decode_issue_tile<DPL>(dst, tm_g, tm_w, tile, nGB, nRB, unit, bar);
}

// Outputs of the rows of a bit mask again, from all their pairs but the folded one, fp32 on the CUDA cores (the score
// group's 256 threads).  Taking a weight out of O^T leaves 2^-24 of that weight behind, too much where little else is left.  A
// warp has every eighth pair.  No slot that the step writes is read.  A function of its own, and its operands gathered only
// where it is called: the epilogue runs once, from a cold instruction cache.
struct RedoRows {
  const __nv_bfloat16 *q, *gk, *gv, *wk, *wv, *vL;
  __nv_bfloat16* out;
  float* part;                   // [8][d], shared memory
  uint32_t lin0, lin1;           // WIDE: the linear term [d][QR] in shared memory, of blocks whose number of tiles is even, odd
  const uint8_t* ht;             // else: the operand image H^T
  uint32_t ht_blk;
  int g, qr, cg, cw, s_ev, rowL, K, tiles;
  float sl2;
};
template <int DPL, bool WIDE, bool SPLIT>
__device__ __noinline__ void decode_redo_rows(Decode2Misc& X, const RedoRows& R, int rows) {
  typedef __nv_bfloat16 T;
  constexpr int d = DPL * 32;
  const int gtid = threadIdx.x & 255, warp = gtid >> 5, lane = gtid & 31;
#pragma unroll 1
  for (int r = 0; r < R.g; ++r) {
    if (!((rows >> r) & 1)) continue;
    float q[DPL], acc[DPL], m = 0.f, l = 0.f;
#pragma unroll
    for (int e = 0; e < DPL; ++e) { q[e] = __bfloat162float(R.q[r * d + lane * DPL + e]); acc[e] = 0.f; }
#pragma unroll 1
    for (int i = warp; i < R.cg + R.cw; i += 8) {
      if (i == R.rowL || (i == R.cg + R.s_ev && R.rowL >= R.cg)) continue;   // the folded pair
      const T *kp = R.gk + (size_t)i * d, *vp = R.gv + (size_t)i * d;
      if (i == R.cg + R.s_ev) {                        // the pair that leaves the window and stays
        kp = reinterpret_cast<const T*>(X.ring_kv);
        vp = kp + d;
      } else if (i >= R.cg) {
        kp = R.wk + (size_t)(i - R.cg) * d;
        vp = R.wv + (size_t)(i - R.cg) * d;
      }
      float z = 0.f;
#pragma unroll
      for (int e = 0; e < DPL; ++e) z = fmaf(q[e], __bfloat162float(kp[lane * DPL + e]), z);
      z = warp_sum(z) * R.sl2;
      const float mn = fmaxf(m, z), a = tc::fast_exp2(m - mn), p = tc::fast_exp2(z - mn);
      l = fmaf(l, a, p);
#pragma unroll
      for (int e = 0; e < DPL; ++e) acc[e] = fmaf(p, __bfloat162float(vp[lane * DPL + e]), acc[e] * a);
      m = mn;
    }
#pragma unroll
    for (int e = 0; e < DPL; ++e) R.part[warp * d + lane * DPL + e] = acc[e];
    if (lane == 0) { X.ssp[0][warp] = m; X.ssp[1][warp] = l; }
    tc::named_bar_sync(11, 256);
    if (gtid < d) {
      float lin = 0.f, mf = X.zn[r];
      if (!WIDE) {
#pragma unroll 1
        for (int j = 0; j < 128; j += 8) {
          const uint4 raw = *reinterpret_cast<const uint4*>(R.ht + (j >> 6) * R.ht_blk + tc::sw128_off(gtid, (j & 63) >> 3));
          const float* pq = &X.phiq_f[r][j];
          lin = fmaf(pq[0], bf16lo_f(raw.x), lin); lin = fmaf(pq[1], bf16hi_f(raw.x), lin);
          lin = fmaf(pq[2], bf16lo_f(raw.y), lin); lin = fmaf(pq[3], bf16hi_f(raw.y), lin);
          lin = fmaf(pq[4], bf16lo_f(raw.z), lin); lin = fmaf(pq[5], bf16hi_f(raw.z), lin);
          lin = fmaf(pq[6], bf16lo_f(raw.w), lin); lin = fmaf(pq[7], bf16hi_f(raw.w), lin);
        }
      }
      for (int k = 0; WIDE && k < R.K; ++k) {          // (the blocks' shares of H's rows)
        const uint32_t at = (max(1, (R.tiles - k + R.K - 1) / R.K) & 1 ? R.lin1 : R.lin0) + (uint32_t)(gtid * R.qr + r) * 4u;
        lin += __uint_as_float(tc::ld_cluster_u32(SPLIT ? tc::map_rank(at, (uint32_t)k) : at));
      }
      for (int i = 0; i < 8; ++i) mf = fmaxf(mf, X.ssp[0][i]);
      const float pn = tc::fast_exp2(X.zn[r] - mf), e = tc::fast_exp2(-mf), dot = X.dotL[r];
      float num = fmaf(pn, X.vnew[gtid], e * fmaf(dot, __bfloat162float(R.vL[gtid]), lin)), den = fmaf(e, X.lden[r] + dot, pn);
      for (int i = 0; i < 8; ++i) {
        const float a = tc::fast_exp2(X.ssp[0][i] - mf);
        num = fmaf(a, R.part[i * d + gtid], num);
        den = fmaf(a, X.ssp[1][i], den);
      }
      if (X.abort_word == 0) R.out[r * d + gtid] = __float2bfloat16_rn(num / den);
    }
    tc::named_bar_sync(11, 256);                       // (the next row takes the same shared memory)
  }
}

// WIDE: Eq. 14 and the fold with nothing rounded to 16 bits, for the steps that always had it so: while the caches fill,
// sparse caches that are no whole number of 64-slot blocks, units of more than 16 tiles.  The softmax weights enter O^T in two
// bf16 parts (the second one in the operand rows that would be zero: no further product), the linear term phi(q)^T H is taken
// in fp32 on the CUDA cores by the feature group behind its last tile, while the score group still works on that tile, and
// the folded pair's feature row is made again in fp32.
// STEADY (neither WIDE nor SPLIT): caches full and lambda a whole number of 64-slot blocks (the geometry is then a constant of the layer;
// the general kernel keeps more of it in registers and spills in the tile loop, 3.5% at 512 units of 7 tiles).
// ahead: the SMs' number; the unit that many further on is likely the next one of this SM.
template <int DPL, int QR, bool WIDE, bool SPLIT>
__global__ void __launch_bounds__(kDec2Threads, 1)
k_decode2_tc(Layer L, Call c, const __grid_constant__ tc::SlotMaps tm_gk, const __grid_constant__ tc::SlotMaps tm_gv,
             const __grid_constant__ CUtensorMap tm_wk, const __grid_constant__ CUtensorMap tm_wv, const uint4* wt_image, int ahead) {
  using S = DecodeSmem<DPL>;
  constexpr int d = DPL * 32;
  constexpr int kblk = d / 64;
  constexpr int F = 64, D = 128;
  constexpr bool STEADY = !WIDE && !SPLIT;
  constexpr int HC = d / 2;                  // value columns per thread of a row pair
  constexpr int QH = QR / 2;                 // query rows per thread of a row pair
  constexpr float kLog2e = 1.4426950408889634f;
  typedef __nv_bfloat16 T;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = tc::smem_u32(sm);
  Decode2Misc& X = *reinterpret_cast<Decode2Misc*>(sm + S::misc);

  const int K = SPLIT ? (int)tc::cluster_size() : 1, rank = SPLIT ? (int)tc::cluster_rank() : 0;
  const int unit = SPLIT ? blockIdx.x / K : blockIdx.x, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int role = warp < 8 ? 0 : (warp < 16 ? 1 : warp - 14);   // 0 feature, 1 score, 2 / 3 / 4 issuing threads
  const int gtid = tid & 255;                // index inside a compute group
  const int gw = warp & 7;
  const int wq = gw & 3;                     // tensor-memory lane quadrant of this warp (= warp % 4)
  const int hf = gw >> 2;                    // which half of the row's work this thread does
  const int t = wq * 32 + lane;              // row of the tile = tensor-memory lane
  const int lam = L.lam, eta = L.eta, g = L.g;
  const int cg = STEADY ? lam : c.count_g;   // occupied slots (all lam of them when a pair is to be folded)
  const int cw = STEADY ? eta : min(eta, c.n_seen);   // pairs in the window
  const bool sel = STEADY || c.mode == UPD_SELECT;
  const int nGB = STEADY ? lam / 64 : (cg + 63) / 64, nRB = (cw + 63) / 64;
  const int NT = max(1, SPLIT ? ((nGB + nRB + 1) / 2 - rank + K - 1) / K : (nGB + nRB + 1) / 2);   // tiles of this block
  auto gt = [&](int tile) { return SPLIT ? rank + tile * K : tile; };     // ... and which of the unit's they are
  const int ring0 = STEADY ? lam : nGB * 64;                // row of ring slot 0
  const int s_ev = c.n_seen % eta;           // ring slot of the pair that leaves = slot the new pair takes
  const int pos_ev = c.n_seen - eta;
  const float sl2 = L.scale * kLog2e;        // q.k in log2 units
  float* scu = L.score + (size_t)unit * (lam + L.cmax);
  volatile int* abw = &X.abort_word;

  const uint32_t bars = sbase + S::misc + (uint32_t)offsetof(Decode2Misc, bars);
  auto bar_kfull = [&](int i) { return bars + 8u * (uint32_t)i; };
  auto bar_vfull = [&](int i) { return bars + 16u + 8u * (uint32_t)i; };
  auto bar_u = [&](int i) { return bars + 32u + 8u * (uint32_t)i; };
  auto bar_phidone = [&](int i) { return bars + 48u + 8u * (uint32_t)i; };
  const uint32_t bar_p = bars + 64u, bar_pfree = bars + 72u;
  auto bar_ptready = [&](int i) { return bars + 80u + 8u * (uint32_t)i; };
  auto bar_o = [&](int i) { return bars + 96u + 8u * (uint32_t)i; };
  const uint32_t bar_w = bars + 112u, bar_phiq = bars + 120u, bar_ht = bars + 128u;
  auto bar_uread = [&](int i) { return bars + 136u + 8u * (uint32_t)i; };
  auto stage_k = [&](int i) { return sbase + S::stage0 + (uint32_t)i * S::stage_bytes + S::st_k; };
  auto stage_v = [&](int i) { return sbase + S::stage0 + (uint32_t)i * S::stage_bytes + S::st_v; };
  auto stage_pt = [&](int i) { return S::stage0 + (uint32_t)i * S::stage_bytes + S::st_pt; };   // offset from sm

  // what the set-up of a unit does without anything the kernels before this one leave
  auto init_bars = [&] {                     // one thread; W^T goes straight into its operand rows
    for (int i = 0; i < 19; ++i) {
      const bool group = (i == 6 || i == 7 || i == 9 || i == 10 || i == 11 || i >= 15);
      tc::mbar_init(bars + 8u * i, i == 16 ? 512u : (group ? 256u : 1u));   // (16: H^T written, by both groups)
    }
    tc::mbar_init_fence();
    tc::mbar_expect_tx(bar_w, (uint32_t)kblk * 8192u);
    for (int kb = 0; kb < kblk; ++kb)
      tc::bulk_copy_g2s(sbase + S::b1 + (uint32_t)kb * S::b1_blk, wt_image + ((size_t)h * kblk + kb) * 512, 8192u, bar_w);
  };
  auto first_tiles = [&] {                   // (that thread) the first two tiles start to stream
    for (int i = 0; i < min(NT, 2); ++i) {
      decode2_issue_tile<DPL>(stage_k(i), &tm_gk, &tm_wk, gt(i), nGB, nRB, unit, bar_kfull(i));
      decode2_issue_tile<DPL>(stage_v(i), &tm_gv, &tm_wv, gt(i), nGB, nRB, unit, bar_vfull(i));
    }
  };
  auto clear = [&] {
    if (role < 2) {
      // rows d+2 .. d+15 of both j blocks of H^T, phi(Q) and both Pr^T tiles: zero
      for (int i = tid; i < 2 * 14 * 8; i += 512) {
        const int jb = i / (14 * 8), r = (i / 8) % 14, ch = i % 8;
        *reinterpret_cast<uint4*>(sm + S::ht + jb * S::ht_blk + tc::sw128_off(d + 2 + r, ch)) = make_uint4(0, 0, 0, 0);
      }
      for (int i = tid; i < 256; i += 512) {
        *reinterpret_cast<uint4*>(sm + S::phiq + i * 16) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(sm + stage_pt(0) + i * 16) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(sm + stage_pt(1) + i * 16) = make_uint4(0, 0, 0, 0);
      }
    }
  };
  // The start of a unit is one request for H and two key and value tiles by all SMs at once, so these come into the L2
  // ahead of time: here where the step before still runs, for the SM's next unit below
  auto prefetch_unit = [&](int u) {
    const uint32_t rows = (uint32_t)min(cg, 256) * (uint32_t)(d * 2);
    tc::prefetch_l2(L.H + (size_t)u * D * d, D * d * 4);
    if (rows) {
      tc::prefetch_l2((const T*)L.gk + (size_t)u * lam * d, rows);
      tc::prefetch_l2((const T*)L.gv + (size_t)u * lam * d, rows);
    }
  };
  if (rank == 0 && tid == 0) prefetch_unit(unit);
  if (tid == 0) { X.abort_word = 0; X.redo = 0; }
  if (SPLIT) {                               // (few units: this block is here before the step before it ends)
    if (tid == 17 * 32) init_bars();
    if (warp == 0) tc::tmem_alloc(&X.tmem_slot, 512);
    clear();
  }
  tc::grid_dep_wait();                       // everything before this step in the stream is complete
  if (SPLIT && tid == 17 * 32) first_tiles();
  // everything the prologue needs from global memory is requested first, so that the round trips overlap
  const int pre_status = *reinterpret_cast<volatile const int*>(L.status);   // (acted on below: an earlier kernel failed: do nothing)
  float pre_s = 0.f, pre_k = 0.f, pre_v = 0.f;
  uint4 pre_q = make_uint4(0, 0, 0, 0);
  if (tid < D) pre_s = L.s[(size_t)unit * D + tid];
  if (tid < 16 * (d / 8) && tid / (d / 8) < g)
    pre_q = *reinterpret_cast<const uint4*>((const T*)c.q + ((size_t)b * L.Hq + h * g + tid / (d / 8)) * d + (tid % (d / 8)) * 8);
  uint4 pre_ring = make_uint4(0, 0, 0, 0), pre_new = pre_ring;
  if (tid >= 384 && tid < 384 + 2 * (d / 8)) {
    const int i = tid - 384, ch = i % (d / 8);
    const bool is_k = i < d / 8;
    pre_ring = *reinterpret_cast<const uint4*>((is_k ? (const T*)L.wk : (const T*)L.wv) + ((size_t)unit * eta + s_ev) * d + ch * 8);
    pre_new = *reinterpret_cast<const uint4*>((is_k ? (const T*)c.k : (const T*)c.v) + ((size_t)b * L.Hkv + h) * d + ch * 8);
  }
  if (tid >= 256 && tid < 256 + d) {
    pre_k = ldf<T>((const T*)c.k + ((size_t)b * L.Hkv + h) * d + (tid - 256));
    pre_v = ldf<T>((const T*)c.v + ((size_t)b * L.Hkv + h) * d + (tid - 256));
  }
  // H (fp32 [D][d]) straight into registers: compute thread x gathers, for DPL items (column c, 8 consecutive j),
  // the eight values H[j][c]; lanes = consecutive columns, so every load of a warp is one 128-byte line.  They
  // become the bf16 operand image H^T below; no staging buffer, so both stages stream key and value tiles from
  // the start
  float pre_h[DPL][8];
  if (tid < 512) {
    const float* Hg = L.H + (size_t)unit * D * d;
#pragma unroll
    for (int n = 0; n < DPL; ++n) {
      const int it = tid + 512 * n, cc = it % d, jc = it / d;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) pre_h[n][jj] = Hg[(size_t)(jc * 8 + jj) * d + cc];
    }
  }

  if (tid == 0) {
    tc::grid_dep_launch_dependents();
    X.failed = pre_status;                   // (one thread's view for all)
  }
  if (!SPLIT) {
    if (tid == 17 * 32) { init_bars(); first_tiles(); }
    if (warp == 0) tc::tmem_alloc(&X.tmem_slot, 512);
    clear();
  }

  // ---- operands that stay for the whole unit (compute warps)
  if (role < 2) {
    // rows d, d+1: s as the sum of two bf16 parts (phi . s_hi + phi . s_lo keeps the fp32 normaliser)
    if (tid < D) {
      const float sv = pre_s;
      X.s_f[tid] = sv;
      const __nv_bfloat16 hi = __float2bfloat16_rn(sv);
      const __nv_bfloat16 lo = __float2bfloat16_rn(sv - __bfloat162float(hi));
      const int ch = (tid & 63) >> 3;
      *reinterpret_cast<T*>(sm + S::ht + (tid >> 6) * S::ht_blk + tc::sw128_off(d, ch) + (tid & 7) * 2) = hi;
      *reinterpret_cast<T*>(sm + S::ht + (tid >> 6) * S::ht_blk + tc::sw128_off(d + 1, ch) + (tid & 7) * 2) = lo;
    }
    // query rows: B1 rows 64..79 (rows >= g are zero) and an fp32 copy
    constexpr int per_row = d / 8;
    if (tid < 16 * per_row) {
      const int r = tid / per_row, ch = tid % per_row;
      const uint4 val = pre_q;
      *reinterpret_cast<uint4*>(sm + S::b1 + (ch >> 3) * S::b1_blk + tc::sw128_off(64 + r, ch & 7)) = val;
      if (r < QR) {
        const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&val);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float2 ff = __bfloat1622float2(v2[q]);
          X.qf[r][ch * 8 + 2 * q] = ff.x;
          X.qf[r][ch * 8 + 2 * q + 1] = ff.y;
        }
      }
    }
    if (tid >= 384 && tid < 384 + 2 * (d / 8)) {
      X.ring_kv[tid - 384] = pre_ring;
      X.new_kv[tid - 384] = pre_new;
    }
    if (tid >= 256 && tid < 256 + d) {
      X.knew[tid - 256] = pre_k;
      X.vnew[tid - 256] = pre_v;
    }
    tc::fence_async_smem();
  }
  __syncthreads();
  // The state's status word is set: leave the memories as they are.  (SPLIT: the blocks agree on it after the tiles)
  if (!SPLIT && X.failed != 0) {
    if (tid == 17 * 32) {                            // (what is on its way into shared memory arrives first)
      tc::mbar_wait(bar_w, 0, abw);
      for (int i = 0; i < min(NT, 2); ++i) { tc::mbar_wait(bar_kfull(i), 0, abw); tc::mbar_wait(bar_vfull(i), 0, abw); }
    }
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(X.tmem_slot, 512);
    return;
  }
  // (0) this block runs, and its query rows' copy is no longer needed (score group: once that is so)
  if (SPLIT && role != 1) tc::cluster_arrive();

  const uint32_t tmem = X.tmem_slot;
  const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
  auto tm_uz = [&](int i) { return tmem + (uint32_t)i * 96u; };          // [U | Z]: 80 columns, two buffers
  const uint32_t tm_o = tmem + 176u;                                       // O^T: lanes = value column, 16 columns = query rows
  auto tm_phi = [&](int i) { return tmem + 192u + (uint32_t)i * 64u; };   // phi tile, bf16 pairs: 64 columns, two buffers
  const uint32_t tm_p = tmem + 320u;                                       // [P | den]: d + 16 columns
  const uint32_t idesc1 = tc::make_idesc_bf16(128, 80, false, false);
  const uint32_t idesc2 = tc::make_idesc_bf16(128, d + 16, false, false);
  const uint32_t idesc0 = tc::make_idesc_bf16(128, 16, false, false);
  const uint32_t idesc3 = tc::make_idesc_bf16(128, 16, true, false);
  bool ok = true;

  if (role < 2) {
    // H -> bf16 H^T, K-major: row c, 64 j per 128-byte row, two j blocks (lanes = consecutive columns: no conflicts)
#pragma unroll
    for (int n = 0; n < DPL; ++n) {
      const int it = tid + 512 * n, cc = it % d, jc = it / d;
      *reinterpret_cast<uint4*>(sm + S::ht + (jc >> 3) * S::ht_blk + tc::sw128_off(cc, jc & 7)) = tc::pack8_bf16(pre_h[n]);
    }
    tc::fence_async_smem();
    tc::mbar_arrive(bar_ht);
  }

  if (role == 2) {
    // =================== [P | den] products ===================
    if (lane == 0) {
      // operand descriptor: the address field (units of 16 bytes) takes the offset of a K step
      const uint64_t dht = tc::make_desc_sw128(sbase + S::ht, 16, 1024);
      for (int tile = 0; tile < NT; ++tile) {
        const int i = tile & 1;
        ok = tc::mbar_wait(bar_phidone(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;   // phi(tile) is in tensor memory
        tc::fence_after_sync();
        if (tile == 0) {
          ok = tc::mbar_wait(bar_ht, 0, abw) && ok;                              // H^T is in place
        } else {
          ok = tc::mbar_wait(bar_pfree, (uint32_t)(tile - 1) & 1u, abw) && ok;   // [P | den] of the tile before is read
        }
        tc::fence_after_sync();
        const uint32_t tph = tm_phi(i);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          tc::mma_bf16_ts(tm_p, tph + ks * 8, dht + (uint64_t)(((ks >> 2) * S::ht_blk + (ks & 3) * 32) >> 4), idesc2, ks > 0);
        tc::mma_commit(bar_p);
        if (tile == 0) {
          // O^T starts as the linear term H^T phi(Q)^T, with weight exp(0 - m), m = 0 so far; the first O^T
          // product waits for it (WIDE: starts empty)
          ok = tc::mbar_wait(bar_phiq, 0, abw) && ok;
          tc::fence_after_sync();
          if (!WIDE && rank == 0) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)
              tc::mma_bf16_ss(tm_o, tc::make_desc_sw128(sbase + S::ht + (ks >> 2) * S::ht_blk + (ks & 3) * 32, 16, 1024),
                              tc::make_desc_sw128(sbase + S::phiq + (ks >> 2) * 2048 + (ks & 3) * 32, 16, 1024), idesc0, ks > 0);
          }
          tc::mma_commit(bar_o(0));
        }
      }
    }
    __syncwarp();
  } else if (role == 4) {
    // =================== [U | Z] products, key tiles ===================
    if (lane == 0) {
      const uint64_t dk0 = tc::make_desc_sw128(stage_k(0), 16, 1024), dk1 = tc::make_desc_sw128(stage_k(1), 16, 1024);
      const uint64_t db1 = tc::make_desc_sw128(sbase + S::b1, 16, 1024);
      ok = tc::mbar_wait(bar_w, 0, abw) && ok;
      for (int tile = 0; tile < NT; ++tile) {
        const int i = tile & 1;
        if (!SPLIT && tile == 2 && unit + ahead < (int)gridDim.x) prefetch_unit(unit + ahead);
        ok = tc::mbar_wait(bar_kfull(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;
        if (tile >= 2)                               // the feature group has read [U | Z] of tile - 2
          ok = tc::mbar_wait(bar_uread(i), (uint32_t)((tile - 2) >> 1) & 1u, abw) && ok;
        tc::fence_after_sync();
        const uint64_t dk = i ? dk1 : dk0;
        const uint32_t tmu = tm_uz(i);
#pragma unroll
        for (int ks = 0; ks < d / 16; ++ks)
          tc::mma_bf16_ss(tmu, dk + (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4),
                          db1 + (uint64_t)(((ks >> 2) * S::b1_blk + (ks & 3) * 32) >> 4), idesc1, ks > 0);
        tc::mma_commit(bar_u(i));
        if (tile + 2 < NT) {                         // the tile after next streams into this buffer once the product has read it
          ok = tc::mbar_wait(bar_u(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;
          decode2_issue_tile<DPL>(stage_k(i), &tm_gk, &tm_wk, gt(tile + 2), nGB, nRB, unit, bar_kfull(i));
        }
      }
    }
    __syncwarp();
  } else if (role == 3) {
    // =================== O^T products, value tiles ===================
    if (lane == 0) {
      const uint64_t dv0 = tc::make_desc_sw128(stage_v(0), 16384, 1024), dv1 = tc::make_desc_sw128(stage_v(1), 16384, 1024);
      const uint64_t dp0 = tc::make_desc_sw128(sbase + stage_pt(0), 16, 1024), dp1 = tc::make_desc_sw128(sbase + stage_pt(1), 16, 1024);
      for (int tile = 0; tile < NT; ++tile) {
        const int i = tile & 1;
        ok = tc::mbar_wait(bar_ptready(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;
        if (tile == 0) ok = tc::mbar_wait(bar_o(0), 0, abw) && ok;   // the linear term is in O^T
        tc::fence_after_sync();
        const uint64_t dv = i ? dv1 : dv0, dp = i ? dp1 : dp0;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          tc::mma_bf16_ss(tm_o, dv + (uint64_t)((ks * 2048) >> 4), dp + (uint64_t)(((ks >> 2) * 2048 + (ks & 3) * 32) >> 4), idesc3, (!WIDE && (!SPLIT || rank == 0)) || tile > 0 || ks > 0);
        const int ev = tile + 1;                                      // completion event of this product
        tc::mma_commit(bar_o(ev & 1));
        ok = tc::mbar_wait(bar_o(ev & 1), (uint32_t)(ev >> 1) & 1u, abw) && ok;
        if (tile + 2 < NT) decode2_issue_tile<DPL>(stage_v(i), &tm_gv, &tm_wv, gt(tile + 2), nGB, nRB, unit, bar_vfull(i));
      }
    }
    __syncwarp();
  } else if (role == 0) {
    // =================== feature group ===================
    // this thread's query rows: [hf * QH, hf * QH + QH)
    const bool exp_kind = L.phi_kind == 1;
    for (int tile = 0; tile < NT; ++tile) {
      const int i = tile & 1;
      const int R = gt(tile) * 128 + t;
      const bool valid = STEADY ? (R < lam || R - lam < eta) : (R < ring0 ? R < cg : R - ring0 < cw);
      ok = tc::mbar_wait(bar_u(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;
      tc::fence_after_sync();
      // [U | Z] of this row in one round trip to tensor memory: this thread's q.k columns (log2 units after
      // scaling; their warp maxima go to the score group, which turns them into weights) and all of U
      float z[QH], wm[QH];
      uint32_t pk2[32];
      {
        uint32_t u[64], zraw[QH];
        if (QH == 4) tc::tmem_ld64u_and4(tm_uz(i) + lane_addr, u, tm_uz(i) + lane_addr + 64 + hf * QH, reinterpret_cast<uint32_t(&)[4]>(zraw));
        else tc::tmem_ld64u_and2(tm_uz(i) + lane_addr, u, tm_uz(i) + lane_addr + 64 + hf * QH, reinterpret_cast<uint32_t(&)[2]>(zraw));
        tc::fence_before_sync();
        tc::mbar_arrive(bar_uread(i));               // [U | Z] of this tile is in registers: the buffer may take tile + 2
#pragma unroll
        for (int r = 0; r < QH; ++r) {
          z[r] = valid ? __uint_as_float(zraw[r]) * sl2 : -CUDART_INF_F;
          wm[r] = warp_max_redux(z[r]);
        }
        // this thread's half of the feature map: hf = 0: softmax(u), hf = 1: softmax(-u)
        tc::phi_half(u, hf != 0, exp_kind, pk2);
      }
      if (tile >= 2) {                               // the score group is done with the buffers of tile - 2
        ok = tc::mbar_wait(bar_ptready(i), (uint32_t)((tile - 2) >> 1) & 1u, abw) && ok;
        tc::fence_after_sync();
      }
      // bf16 pairs into tensor memory: the A operand of the second product (K index = feature j)
      tc::tmem_st32u(tm_phi(i) + lane_addr + hf * 32, pk2);
#pragma unroll
      for (int r = 0; r < QH; ++r) {
        X.z_s[i][hf * QH + r][t] = z[r];
        if (lane == 0) X.redmax[i][wq][hf * QH + r] = wm[r];
      }
      tc::fence_before_sync();
      tc::mbar_arrive(bar_phidone(i));               // (release: the shared-memory writes above are visible to whoever acquires it)
    }
    if constexpr (WIDE) {
      // the linear term of this block's rows of H (those it folds into later), before the fold, in fp32: a warp has d / 8
      // value columns, its lanes the columns times 32 / (d / 8) shares of the rows
      ok = tc::mbar_wait(bar_phiq, 0, abw) && ok;
      const float* phiq_t = reinterpret_cast<const float*>(sm + S::phiq);   // [feature][QR] (rows >= g are zero)
      constexpr int CW = d / 8, P = 32 / CW;
      const int cc = gw * CW + lane % CW, jper = (D + K - 1) / K, j0 = min(D, rank * jper), j1 = min(D, j0 + jper);
      const float* Hc = L.H + (size_t)unit * D * d + cc;
      float acc[QR];
#pragma unroll
      for (int r = 0; r < QR; ++r) acc[r] = 0.f;
#pragma unroll 1
      for (int j = j0 + lane / CW; j < j1; j += 8 * P) {
        float hv[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) hv[q] = j + q * P < j1 ? __ldcg(Hc + (size_t)(j + q * P) * d) : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4* pq = reinterpret_cast<const float4*>(phiq_t + min(j + q * P, D - 1) * QR);
#pragma unroll
          for (int r = 0; r < QR; r += 4) {
            const float4 p = pq[r / 4];
            acc[r] = fmaf(hv[q], p.x, acc[r]); acc[r + 1] = fmaf(hv[q], p.y, acc[r + 1]);
            acc[r + 2] = fmaf(hv[q], p.z, acc[r + 2]); acc[r + 3] = fmaf(hv[q], p.w, acc[r + 3]);
          }
        }
      }
      // [d][QR], in the key tile of the stage the last tile does not use
      float* lin = reinterpret_cast<float*>(sm + S::stage0 + (uint32_t)(NT & 1) * S::stage_bytes + S::st_k) + cc * QR;
#pragma unroll
      for (int r = 0; r < QR; ++r) {
#pragma unroll
        for (int o = CW; o < 32; o <<= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
      }
      if (lane < CW)
#pragma unroll
        for (int r = 0; r < QR; r += 4) *reinterpret_cast<float4*>(lin + r) = make_float4(acc[r], acc[r + 1], acc[r + 2], acc[r + 3]);
      if (SPLIT) tc::named_bar_arrive(13, 512);      // the score group adds it to O^T
    }
  } else {
    // =================== score group ===================
    // first: what the linear term needs.  u = q W on the CUDA cores (g rows only) from the W^T operand image
    ok = tc::mbar_wait(bar_w, 0, abw) && ok;
    for (int i = gtid; i < g * F; i += 256) {
      const int r = i >> 6, f = i & 63;
      float a0 = 0.f, a1 = 0.f;
#pragma unroll
      for (int ch = 0; ch < d / 8; ++ch) {
        uint4 raw = *reinterpret_cast<const uint4*>(sm + S::b1 + (ch >> 3) * S::b1_blk + tc::sw128_off(f, ch & 7));
        const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float2 ww = __bfloat1622float2(w2[q]);
          a0 = fmaf(X.qf[r][ch * 8 + 2 * q], ww.x, a0);
          a1 = fmaf(X.qf[r][ch * 8 + 2 * q + 1], ww.y, a1);
        }
      }
      X.u_s[r][f] = a0 + a1;
    }
    tc::named_bar_sync(2, 256);
    // phi(q), its normaliser phi(q) . s and q . k_new
    if (gw < g) {
      const int r = gw;
      float u0 = X.u_s[r][lane], u1 = X.u_s[r][lane + 32];
      float p0, p1, n0, n1;
      if (L.phi_kind == 1) {
        p0 = expf(u0); p1 = expf(u1); n0 = expf(-u0); n1 = expf(-u1);
      } else {
        float mx = warp_max(fmaxf(u0, u1)), mn = warp_min(fminf(u0, u1));
        p0 = expf(u0 - mx); p1 = expf(u1 - mx); n0 = expf(mn - u0); n1 = expf(mn - u1);
        float s1 = warp_sum(p0 + p1), s2 = warp_sum(n0 + n1);
        p0 /= s1; p1 /= s1; n0 /= s2; n1 /= s2;
      }
      float vals[4] = {p0, p1, n0, n1};
      if constexpr (!WIDE) {
#pragma unroll
        for (int q = 0; q < 4; ++q) vals[q] = round_bf16f(vals[q]);
      }
      int js[4] = {lane, lane + 32, 64 + lane, 96 + lane};
      float ld = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = js[q];
        X.phiq_f[r][j] = vals[q];
        if constexpr (WIDE) reinterpret_cast<float*>(sm + S::phiq)[j * QR + r] = vals[q];
        else *reinterpret_cast<T*>(sm + S::phiq + (j >> 6) * 2048 + tc::sw128_off(r, (j & 63) >> 3) + (j & 7) * 2) = __float2bfloat16_rn(vals[q]);
        ld = fmaf(vals[q], X.s_f[j], ld);
      }
      ld = warp_sum(ld);
      float zz = 0.f;
      for (int j = lane; j < d; j += 32) zz = fmaf(X.qf[r][j], X.knew[j], zz);
      zz = warp_sum(zz);
      if (lane == 0) { X.lden[r] = ld; X.zn[r] = zz * sl2; }
    }
    tc::fence_async_smem();
    tc::mbar_arrive(bar_phiq);                       // phi(Q) is in its operand rows
    if (SPLIT) tc::cluster_arrive();                 // (0)

    // running maxima of q.k per query row (log2 units; every valid row counts, also the one that will be
    // folded: any m >= the true maximum leaves Eq. 14 unchanged) and this thread's share of the sums
    float lpart[QH], m_run[QR];
    unsigned long long w_key = ~0ull;                // lowest (score, then youngest) pair of this warp's rows so far
    float w_a1 = CUDART_INF_F, w_a2 = CUDART_INF_F;  // the two lowest scores of this warp's rows so far
#pragma unroll
    for (int r = 0; r < QR; ++r) m_run[r] = 0.f;
#pragma unroll
    for (int r = 0; r < QH; ++r) lpart[r] = 0.f;
    // token position of this thread's row, fetched one tile ahead (its round trip to the L2 would otherwise sit
    // in front of the lowest-score reduction of every tile)
    const int* gpos_u = L.gpos + (size_t)unit * lam;
    int pos_next = gt(0) * 128 + t < cg ? ld_global_i32(gpos_u + gt(0) * 128 + t) : pos_ev;
    for (int tile = 0; tile < NT; ++tile) {
      const int i = tile & 1;
      const int R = gt(tile) * 128 + t;
      const bool is_g = R < cg;
      const int slot = R - ring0;
      const bool scored = sel && (is_g || slot == s_ev);
      const int pos = pos_next;
      pos_next = (tile + 1 < NT && R + K * 128 < cg) ? ld_global_i32(gpos_u + R + K * 128) : pos_ev;
      const uint8_t* vtile = sm + S::stage0 + (size_t)i * S::stage_bytes + S::st_v;
      uint8_t* ptile = sm + stage_pt(i);

      ok = tc::mbar_wait(bar_vfull(i), (uint32_t)(tile >> 1) & 1u, abw) && ok;
      ok = tc::mbar_wait(bar_p, (uint32_t)tile & 1u, abw) && ok;   // (its commit follows the feature group's arrival: z_s, redmax are visible)
      if (tile >= 2) {                               // the Pr^T operand of tile - 2 was consumed by its O^T product
        const int ev = tile - 1;
        ok = tc::mbar_wait(bar_o(ev & 1), (uint32_t)(ev >> 1) & 1u, abw) && ok;
      }
      tc::fence_after_sync();
      // ---- softmax weights of the tile (bf16; the sums use the rounded weights) into the Pr^T operand
      float pw[QH];
      {
        const bool valid = is_g || ((STEADY || slot >= 0) && slot < cw);
        float m_new[QR];
        bool moved = false;
#pragma unroll
        for (int r = 0; r < QR; ++r) {
          m_new[r] = fmaxf(fmaxf(m_run[r], fmaxf(X.redmax[i][0][r], X.redmax[i][1][r])),
                           fmaxf(X.redmax[i][2][r], X.redmax[i][3][r]));
          moved = moved || (m_new[r] > m_run[r] + kDec2Lazy);
        }
        // The stabiliser only follows the maximum when it has run away by more than 2^kDec2Lazy: any m within
        // that distance of the true maximum leaves Eq. 14 unchanged (weights up to 2^kDec2Lazy are exact in
        // bf16's and fp32's range), and moving it means waiting for the O^T product of the tile before.
        if (moved) {                                 // uniform over the group, rare
          float alpha[QR];
#pragma unroll
          for (int r = 0; r < QR; ++r) alpha[r] = tc::fast_exp2(m_run[r] - m_new[r]);
#pragma unroll
          for (int r = 0; r < QH; ++r) lpart[r] *= hf ? alpha[QH + r] : alpha[r];
          if (hf == 0) {
            // O^T so far (the products up to the tile before, or the linear term) moves to the new maximum
            ok = tc::mbar_wait(bar_o(tile & 1), (uint32_t)(tile >> 1) & 1u, abw) && ok;
            tc::fence_after_sync();
            // (WIDE: the columns of the weights' second parts follow those of the first)
#pragma unroll
            for (int p = 0; p < (WIDE ? QR / 4 : 1); ++p) {
              float ov[8];
              tc::tmem_ld8(tm_o + lane_addr + p * 8, ov);
#pragma unroll
              for (int r = 0; r < (WIDE ? 8 : QR); ++r) ov[r] *= alpha[r % QR];
              tc::tmem_st8(tm_o + lane_addr + p * 8, ov);
            }
          }
          // all rows move together
#pragma unroll
          for (int r = 0; r < QR; ++r) m_run[r] = m_new[r];
        }
#pragma unroll
        for (int r = 0; r < QH; ++r) {
          const int rr = hf * QH + r;
          const float mr = hf ? m_run[QH + r] : m_run[r];
          const float w = valid ? tc::fast_exp2(X.z_s[i][rr][t] - mr) : 0.f;
          const uint32_t pb = pack_bf16x2(w, 0.f);
          pw[r] = bf16lo_f(pb);
          *reinterpret_cast<unsigned short*>(ptile + (t >> 6) * 2048 + tc::sw128_off(rr, (t & 63) >> 3) + (t & 7) * 2) = (unsigned short)pb;
          if constexpr (WIDE) {
            const uint32_t pl = pack_bf16x2(w - pw[r], 0.f);
            pw[r] += bf16lo_f(pl);
            *reinterpret_cast<unsigned short*>(ptile + (t >> 6) * 2048 + tc::sw128_off(QR + rr, (t & 63) >> 3) + (t & 7) * 2) = (unsigned short)pl;
          }
        }
      }
      // ---- Eq. 10: this thread's half of the value columns
      float ss;
      {
        // packed pairs: d = v - P / den, four running sums of squares (columns 4k, 4k+1 | 4k+2, 4k+3)
        uint64_t ninv2 = 0;
        uint64_t accA = tc::pack_f2(0.f, 0.f), accB = accA;
#pragma unroll
        for (int c0 = 0; c0 < HC; c0 += 32) {
          uint32_t p[32];
          if (c0 == 0) {                                 // the two parts of the denominator come with the first columns
            uint32_t dn[2];
            tc::tmem_ld32u_and2(tm_p + lane_addr + hf * HC, p, tm_p + lane_addr + d, dn);
            const float den = __uint_as_float(dn[0]) + __uint_as_float(dn[1]);
            const float inv = den > 0.f ? 1.0f / den : 0.f;
            ninv2 = tc::pack_f2(-inv, -inv);
          } else {
            tc::tmem_ld32u(tm_p + lane_addr + hf * HC + c0, p);
          }
          if (c0 + 32 >= HC) {                 // [P | den] is read: the next tile's product may overwrite it
            tc::fence_before_sync();
            tc::mbar_arrive(bar_pfree);
          }
#pragma unroll
          for (int q8 = 0; q8 < 4; ++q8) {
            const int cc = hf * HC + c0 + q8 * 8;
            const uint4 raw = *reinterpret_cast<const uint4*>(vtile + (cc >> 6) * 16384 + tc::sw128_off(t, (cc & 63) >> 3));
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
        ss = (a0 + a1) + (a2 + a3);
      }
      // every row stays in O^T and in the sums; the one pair that is folded in the end is taken out again
      // after the last tile, so nothing here needs the other quadrants
#pragma unroll
      for (int r = 0; r < QH; ++r) lpart[r] += pw[r];
      if (hf == 1) X.ssp[i][t] = ss;
      tc::named_bar_sync(4 + wq, 64);                // the two warps of this row quadrant
      if (hf == 0) {
        const float score = sqrtf(ss + X.ssp[i][t]);
        if (scored && ok && (!SPLIT || X.failed == 0)) scu[is_g ? R : lam] = score;
        // lowest score of the quadrant's rows in this tile (ties: the younger pair) and the runner-up;
        // scores are norms (>= 0): their bit patterns order like unsigned integers
        const unsigned sb = scored ? __float_as_uint(score) : 0xffffffffu;
        const unsigned smin = __reduce_min_sync(0xffffffffu, sb);
        const unsigned tb_ = (sb == smin && scored) ? (unsigned)(0x7fffffff - pos) : 0xffffffffu;
        const unsigned tmin = __reduce_min_sync(0xffffffffu, tb_);
        const bool is_min = scored && sb == smin && tb_ == tmin;
        const unsigned s2 = __reduce_min_sync(0xffffffffu, is_min ? 0xffffffffu : sb);
        const float c1 = smin == 0xffffffffu ? CUDART_INF_F : __uint_as_float(smin);
        const float c2 = s2 == 0xffffffffu ? CUDART_INF_F : __uint_as_float(s2);
        w_a2 = fminf(fmaxf(w_a1, c1), fminf(w_a2, c2));
        w_a1 = fminf(w_a1, c1);
        const unsigned long long k = smin != 0xffffffffu ? (((unsigned long long)smin << 32) | tmin) : ~0ull;
        if (k < w_key) {                             // (uniform over the warp) a new lowest pair of this quadrant:
          w_key = k;                                 // keep what the fold and Eq. 14 need of it
          const int src = __ffs(__ballot_sync(0xffffffffu, is_min)) - 1;
          uint32_t pr[32];
#pragma unroll
          for (int half = 0; half < 2; ++half) {     // its feature row, read back from tensor memory
            tc::tmem_ld32u(tm_phi(i) + lane_addr + half * 32, pr);
            if (is_min) {
              uint4* dst = &X.wb_phi[wq][half * 8];
#pragma unroll
              for (int q = 0; q < 8; ++q) dst[q] = make_uint4(pr[4 * q], pr[4 * q + 1], pr[4 * q + 2], pr[4 * q + 3]);
            }
          }
          if (lane < d / 8)                          // its value row: one 16-byte piece per lane
            X.wb_v[wq][lane] = *reinterpret_cast<const uint4*>(vtile + (lane >> 3) * 16384 + tc::sw128_off(wq * 32 + src, lane & 7));
          if (is_min) {
            X.wb_row[wq] = R;
#pragma unroll
            for (int r = 0; r < QR; ++r) {
              X.wb_z[wq][r] = X.z_s[i][r][t];
              X.wb_m[wq][r] = m_run[r];
            }
          }
        }
      }
      tc::fence_async_smem();
      tc::fence_before_sync();
      tc::mbar_arrive(bar_ptready(i));
    }
    if (hf == 0 && lane == 0) { X.wb_key[wq] = w_key; X.wb_a1[wq] = w_a1; X.wb_a2[wq] = w_a2; }
#pragma unroll
    for (int r = 0; r < QH; ++r) {
      float ls = warp_sum(lpart[r]);
      if (lane == 0) X.l_s[wq][hf * QH + r] = ls;
    }
    if (gtid == 0) {
#pragma unroll
      for (int r = 0; r < QR; ++r) X.m_s[0][r] = m_run[r];
    }
    if constexpr (SPLIT) {
      // the block's lowest pair, maxima and sums to every block: a warp per block
      tc::named_bar_sync(2, 256);
      int lq = 0;
      unsigned long long best = X.wb_key[0];
#pragma unroll
      for (int i = 1; i < 4; ++i)
        if (X.wb_key[i] < best) { best = X.wb_key[i]; lq = i; }
      float second = X.wb_a2[lq];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i != lq) second = fminf(second, X.wb_a1[i]);
      tc::cluster_wait();                            // (0)
      if (gw < K) {
        auto to = [&](uint32_t off) { return tc::map_rank(sbase + S::misc + off, (uint32_t)gw); };
        const int q = lane & 7, what = lane >> 3;
        const float f = what == 0 ? X.wb_z[lq][q] : what == 1 ? X.wb_m[lq][q] : what == 2 ? X.m_s[0][q] : (X.l_s[0][q] + X.l_s[1][q]) + (X.l_s[2][q] + X.l_s[3][q]);
        tc::st_cluster_u32(to((uint32_t)offsetof(Decode2Misc, peer_f) + (uint32_t)(rank * 128 + lane * 4)), __float_as_uint(f));
        tc::st_cluster_v4(to((uint32_t)offsetof(Decode2Misc, peer_rows) + (uint32_t)(rank * 512 + lane * 16)), (lane < 16 ? X.wb_phi : X.wb_v)[lq][lane & 15]);
        if (lane == 0)
          tc::st_cluster_v4(to((uint32_t)offsetof(Decode2Misc, peer_key) + (uint32_t)rank * 16u),
                            make_uint4((unsigned)best, (unsigned)(best >> 32), __float_as_uint(X.wb_a1[lq]), __float_as_uint(second)));
        if (lane == 1)
          tc::st_cluster_v4(to((uint32_t)offsetof(Decode2Misc, peer_row) + (uint32_t)rank * 16u),
                            make_uint4((unsigned)X.wb_row[lq], X.abort_word != 0 || (rank == 0 && X.failed != 0) ? 1u : 0u, 0u, 0u));
      }
    }
  }

  const bool exact = WIDE && sel;            // the folded pair's feature row in fp32 (phi_of_key)
  // the weight of a pair as the O^T product used it
  auto used_weight = [](float z, float m) {
    const float w = tc::fast_exp2(z - m), hi = round_bf16f(w);
    return WIDE ? hi + round_bf16f(w - hi) : hi;
  };
  auto redo_rows = [&](int rows, int rowL, const T* vL) {
    RedoRows R;
    const size_t row = ((size_t)b * L.Hq + h * g) * d;
    R.q = (const T*)c.q + row; R.out = (T*)c.out + row; R.vL = vL;
    R.gk = (const T*)L.gk + (size_t)unit * lam * d; R.gv = (const T*)L.gv + (size_t)unit * lam * d;
    R.wk = (const T*)L.wk + (size_t)unit * eta * d; R.wv = (const T*)L.wv + (size_t)unit * eta * d;
    R.part = reinterpret_cast<float*>(sm + S::phiq);
    R.lin0 = sbase + S::stage0 + S::st_k; R.lin1 = R.lin0 + S::stage_bytes;
    R.g = g; R.qr = QR; R.cg = cg; R.cw = cw; R.s_ev = s_ev; R.rowL = rowL; R.K = K; R.tiles = (nGB + nRB + 1) / 2; R.sl2 = sl2;
    R.ht = sm + S::ht; R.ht_blk = S::ht_blk;
    decode_redo_rows<DPL, WIDE, SPLIT>(X, R, rows);
  };
  // this thread's row of O^T (WIDE: both parts and the linear term, which is a summand of score 0), score group
  auto read_o = [&](float (&o)[QR]) {
    float ov[8];
    tc::tmem_ld8(tm_o + lane_addr, ov);
    if constexpr (WIDE) {
      float lo[8];
      if (QR == 8) tc::tmem_ld8(tm_o + lane_addr + 8, lo);
      const float* lin = reinterpret_cast<const float*>(sm + S::stage0 + (uint32_t)(NT & 1) * S::stage_bytes + S::st_k) + min(t, d - 1) * QR;
#pragma unroll
      for (int r = 0; r < QR; ++r) o[r] = fmaf(tc::fast_exp2(-X.m_s[0][r]), lin[r], ov[r] + (QR == 8 ? lo[r] : ov[(r + 4) & 7]));
    } else {
#pragma unroll
      for (int r = 0; r < QR; ++r) o[r] = ov[r];
    }
  };
  // H += phi_fold v_fold^T for rows [j0, j0 + jn), by the feature group: the additions happen at the L2, nothing is read
  // back (as bulk reductions from shared memory the block had to stay 1.6 us longer for them to be read)
  auto fold_rows = [&](int j0, int jn, const __nv_bfloat16* phiL, const __nv_bfloat16* vL) {
    constexpr int per_row = d / 4;
    const int c4 = tid % per_row * 4;
    const uint2 vv = *reinterpret_cast<const uint2*>(vL + c4);
    const float v0 = bf16lo_f(vv.x), v1 = bf16hi_f(vv.x), v2 = bf16lo_f(vv.y), v3 = bf16hi_f(vv.y);
    float* Hgw = L.H + (size_t)unit * D * d + c4;
#pragma unroll 4
    for (int j = j0 + tid / per_row; j < j0 + jn; j += 256 / per_row) {
      const float pj = exact ? X.phi_fold[j] : __bfloat162float(phiL[j]);
      tc::red_add_v4(Hgw + (size_t)j * d, make_float4(pj * v0, pj * v1, pj * v2, pj * v3));
    }
  };
  // The folded pair's feature row comes from the bf16 operand.  WIDE: it is recomputed in fp32 from the folded key (feature
  // group; X.phi_fold): u = k W on the CUDA cores (64 features x 4 threads), then one warp's feature map, about 1 us
  // behind the last tile
  auto phi_of_key = [&](const T* kr) {
    const int f = tid >> 2, part = tid & 3;
    uint4 kraw[d / 32];
#pragma unroll
    for (int q = 0; q < d / 32; ++q) kraw[q] = __ldcg(reinterpret_cast<const uint4*>(kr + (part * (d / 32) + q) * 8));
    float a = 0.f;
#pragma unroll
    for (int q = 0; q < d / 32; ++q) {
      const int ch = part * (d / 32) + q;
      const uint4 wraw = *reinterpret_cast<const uint4*>(sm + S::b1 + (ch >> 3) * S::b1_blk + tc::sw128_off(f, ch & 7));
      const uint32_t kk[4] = {kraw[q].x, kraw[q].y, kraw[q].z, kraw[q].w}, ww[4] = {wraw.x, wraw.y, wraw.z, wraw.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        a = fmaf(bf16lo_f(kk[e]), bf16lo_f(ww[e]), a);
        a = fmaf(bf16hi_f(kk[e]), bf16hi_f(ww[e]), a);
      }
    }
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    if (part == 0) X.u_s[0][f] = a;
    tc::named_bar_sync(10, 256);
    if (gw == 0) {
      const float u0 = X.u_s[0][lane], u1 = X.u_s[0][lane + 32];
      float p0, p1, n0, n1;
      if (L.phi_kind == 1) {
        p0 = expf(u0); p1 = expf(u1); n0 = expf(-u0); n1 = expf(-u1);
      } else {
        const float mx = warp_max(fmaxf(u0, u1)), mn = warp_min(fminf(u0, u1));
        p0 = expf(u0 - mx); p1 = expf(u1 - mx); n0 = expf(mn - u0); n1 = expf(mn - u1);
        const float s1 = warp_sum(p0 + p1), s2 = warp_sum(n0 + n1);
        p0 /= s1; p1 /= s1; n0 /= s2; n1 /= s2;
      }
      X.phi_fold[lane] = p0; X.phi_fold[lane + 32] = p1; X.phi_fold[64 + lane] = n0; X.phi_fold[96 + lane] = n1;
    }
    tc::named_bar_sync(10, 256);
    if (rank == 0) tc::named_bar_arrive(12, 512);    // X.phi_fold is there, and the key is read: its slot may be written
  };

  if constexpr (SPLIT) {
    // ---- the blocks have told each other their lowest pairs; block 0 also reads the O^T parts of the others, which wait
    // for that at a second barrier
    const uint32_t free_stage = S::stage0 + (uint32_t)(NT & 1) * S::stage_bytes;
    if (role == 1) {
      ok = tc::mbar_wait(bar_o(NT & 1), (uint32_t)(NT >> 1) & 1u, abw) && ok;
      tc::fence_after_sync();
      if constexpr (WIDE) tc::named_bar_sync(13, 512);
      if (gw < 4 && t < d) {                         // [d][QR], in the free stage's Pr^T tile
        float ov[QR];
        read_o(ov);
#pragma unroll
        for (int r = 0; r < QR; r += 4)
          *reinterpret_cast<float4*>(sm + free_stage + S::st_pt + (t * QR + r) * 4) = make_float4(ov[r], ov[r + 1], ov[r + 2], ov[r + 3]);
      }
    } else {
      tc::cluster_wait();                            // (0)
    }
    if (!ok) *abw = 1;
    __syncwarp();
    tc::fence_before_sync();
    tc::cluster_arrive();
    tc::cluster_wait();
    if (role < 2) {
      // the pair to fold: lowest (score, then youngest) of all
      uint4 win = X.peer_key[0];
      int wr = 0;
      bool okb = true;
      float kept = CUDART_INF_F;                     // lowest score but that
      for (int k = 0; k < K; ++k) {
        const uint4 p = X.peer_key[k];
        okb = okb && X.peer_row[k].y == 0u;
        if (k > 0) {
          const bool less = p.y < win.y || (p.y == win.y && p.x < win.x);
          kept = fminf(kept, __uint_as_float(less ? win.z : p.z));
          if (less) { win = p; wr = k; }
        }
      }
      kept = fminf(kept, __uint_as_float(win.w));
      const bool fold = okb && sel;
      const int rowL = sel ? (int)X.peer_row[wr].x : cg;
      const __nv_bfloat16* phiL = reinterpret_cast<const __nv_bfloat16*>(&X.peer_rows[wr][0]);
      const __nv_bfloat16* vL = reinterpret_cast<const __nv_bfloat16*>(&X.peer_rows[wr][16]);
      if (role == 0) {
        // ---- Eq. 13, this block's rows of H
        if (exact) phi_of_key((unsigned)rowL < (unsigned)cg ? (const T*)L.gk + ((size_t)unit * lam + rowL) * d : (const T*)L.wk + ((size_t)unit * eta + s_ev) * d);
        tc::cluster_arrive();
        if (fold) {
          const int jper = (D + K - 1) / K, j0 = min(D, rank * jper), jn = min(jper, D - j0);
          fold_rows(j0, jn, phiL, vL);
          if (tid < jn) atomicAdd(L.s + (size_t)unit * D + j0 + tid, exact ? X.phi_fold[j0 + tid] : __bfloat162float(phiL[j0 + tid]));
        }
      } else if (rank == 0) {
        // ---- Eq. 14: a thread has one value column of four query rows
        const int cc = gtid % d, r0 = gtid / d * 4;
        const bool mine = r0 < QR && r0 < g;
        uint4 op[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (mine && k < K) {
            // (a block's O^T part lies in the stage its last tile did not use)
            const int ntk = max(1, ((nGB + nRB + 1) / 2 - k + K - 1) / K);
            op[k] = tc::ld_cluster_v4(tc::map_rank(sbase + S::stage0 + (uint32_t)(ntk & 1) * S::stage_bytes + S::st_pt + (uint32_t)(cc * QR + r0) * 4u, k));
          }
        // a warp per query row: what its output takes of each block's O^T, of the folded and of the new value.  (All
        // of this runs once and from a cold instruction cache: short code is what counts)
        float* coef = &X.redmax[0][0][0];            // [block][row]
        if (exact) tc::named_bar_sync(12, 512);
        if (gw < g) {
          const int r = gw;
          float dot = 0.f;                           // phi(q) . phi_fold
          if (sel)
            for (int j = lane; j < D; j += 32) dot = fmaf(X.phiq_f[r][j], WIDE ? X.phi_fold[j] : __bfloat162float(phiL[j]), dot);
          dot = warp_sum(dot);
          const float m = lane < K ? X.peer_f[lane][2][r] : -CUDART_INF_F, zn = X.zn[r];
          const float mf = fmaxf(warp_max(m), zn), am = tc::fast_exp2(m - mf);
          float den = warp_sum(lane < K ? am * X.peer_f[lane][3][r] : 0.f);
          // the folded pair leaves the softmax part again, with the weight its tile's product used
          const float wm = X.peer_f[wr][1][r];
          const float pL = sel ? used_weight(X.peer_f[wr][0][r], wm) * tc::fast_exp2(wm - mf) : 0.f;
          const float pn = tc::fast_exp2(zn - mf), e = tc::fast_exp2(-mf);
          den = den - pL + pn + e * (X.lden[r] + dot);
          const float inv = 1.0f / den;
          if (lane < K) coef[lane * kDecQ + r] = am * inv;
          __syncwarp();
          if (lane == 0) {
            const bool redo = sel && !(pL <= 256.f * den);
            if (redo) atomicOr(&X.redo, 1 << r);
            X.dotL[r] = redo ? dot : sel ? fmaf(e, dot, -pL) * inv : 0.f;
            if (!redo) X.zn[r] = pn * inv;
          }
        }
        tc::named_bar_sync(11, 256);
        const int redo = X.redo;
        if (__builtin_expect(redo != 0, 0)) redo_rows(redo, rowL, vL);
        if (mine && okb) {
          const float vLc = sel ? __bfloat162float(vL[cc]) : 0.f, vn = X.vnew[cc];
          float4 o = *reinterpret_cast<const float4*>(&X.dotL[r0]);
          const float4 bn = *reinterpret_cast<const float4*>(&X.zn[r0]);
          o = make_float4(fmaf(o.x, vLc, bn.x * vn), fmaf(o.y, vLc, bn.y * vn), fmaf(o.z, vLc, bn.z * vn), fmaf(o.w, vLc, bn.w * vn));
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k < K) {
              const float4 a = *reinterpret_cast<const float4*>(coef + k * kDecQ + r0);
              o.x = fmaf(a.x, __uint_as_float(op[k].x), o.x); o.y = fmaf(a.y, __uint_as_float(op[k].y), o.y);
              o.z = fmaf(a.z, __uint_as_float(op[k].z), o.z); o.w = fmaf(a.w, __uint_as_float(op[k].w), o.w);
            }
          const float ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (r0 + r < g && !((redo >> (r0 + r)) & 1)) ((T*)c.out)[((size_t)b * L.Hq + h * g + r0 + r) * d + cc] = __float2bfloat16_rn(ov[r]);
        }
        __syncwarp();
        tc::cluster_arrive();
      } else {
        tc::cluster_arrive();
        if (rank == K - 1) {
          // ---- the pairs move: no block reads the memories any more (exact: once all have read the folded key)
          if (exact) tc::cluster_wait();
          const bool moves = sel ? rowL < cg : c.mode == UPD_APPEND;
          constexpr int nch = d / 8;
          if (okb) {
            if (gtid < 2 * nch && moves)
              *reinterpret_cast<uint4*>((gtid < nch ? (T*)L.gk : (T*)L.gv) + ((size_t)unit * lam + rowL) * d + (gtid % nch) * 8) = X.ring_kv[gtid];
            if (gtid >= 32 && gtid < 32 + 2 * nch) {
              const int i = gtid - 32;
              *reinterpret_cast<uint4*>((i < nch ? (T*)L.wk : (T*)L.wv) + ((size_t)unit * eta + s_ev) * d + (i % nch) * 8) = X.new_kv[i];
            }
            if (gtid == 64 && moves) {
              L.gpos[(size_t)unit * lam + rowL] = pos_ev;
              scu[rowL] = sel ? __ldcg(scu + lam) : CUDART_NAN_F;
            }
            if (gtid == 96 && sel) {                 // lowest kept / highest folded score of this update
              L.thr[(size_t)unit * 2 + 0] = kept;
              L.thr[(size_t)unit * 2 + 1] = __uint_as_float(win.z);
            }
          }
          __syncwarp();
        }
      }
      if (!(exact && role == 1 && rank == K - 1)) tc::cluster_wait();
    } else {
      tc::cluster_arrive();
      tc::cluster_wait();
    }
  }
  // ---- after the last tile the two compute groups split the rest: the feature group folds (Eq. 13), the score
  // group writes the outputs (Eq. 14) and the memories; the issuing warps go straight to the end
  if (!SPLIT && role < 2) {
    tc::fence_before_sync();
    tc::named_bar_sync(9, 512);                      // the score group has finished the last tile
    tc::fence_after_sync();
    // the pair to fold: lowest (score, then youngest) over the four quadrants
    int lt = 0;
    {
      unsigned long long best = X.wb_key[0];
#pragma unroll
      for (int i = 1; i < 4; ++i)
        if (X.wb_key[i] < best) { best = X.wb_key[i]; lt = i; }
    }
    const __nv_bfloat16* phiL = reinterpret_cast<const __nv_bfloat16*>(&X.wb_phi[lt][0]);
    const __nv_bfloat16* vL = reinterpret_cast<const __nv_bfloat16*>(&X.wb_v[lt][0]);
    // the stage the last tile did not use is free once the O^T product of the tile before the last is complete
    const uint32_t free_stage = S::stage0 + (uint32_t)(NT & 1) * S::stage_bytes;
    if (role == 0) {
      // ---- Eq. 13
      const bool okb = X.abort_word == 0;
      if (exact) {
        const int rowL = X.wb_row[lt];
        phi_of_key((unsigned)rowL < (unsigned)cg ? (const T*)L.gk + ((size_t)unit * lam + rowL) * d : (const T*)L.wk + ((size_t)unit * eta + s_ev) * d);
      }
      if (okb && sel) fold_rows(0, D, phiL, vL);
      if (okb && sel && tid < D) atomicAdd(L.s + (size_t)unit * D + tid, exact ? X.phi_fold[tid] : __bfloat162float(phiL[tid]));
    } else {
      auto dot_fold = [&] {                          // phi(q) . phi_fold
        if (gw < g) {
          const int r = gw;
          float a = 0.f;
          if (!WIDE || sel)
            for (int j = lane; j < D; j += 32) a = fmaf(X.phiq_f[r][j], WIDE ? X.phi_fold[j] : __bfloat162float(phiL[j]), a);
          a = warp_sum(a);
          if (lane == 0) X.dotL[r] = sel ? a : 0.f;
          if (sel && lane == 0) {
            const float m0 = X.m_s[0][r], mf = fmaxf(m0, X.zn[r]), wm = X.wb_m[lt][r];
            const float pL = used_weight(X.wb_z[lt][r], wm) * tc::fast_exp2(wm - mf);
            const float l0 = (X.l_s[0][r] + X.l_s[1][r]) + (X.l_s[2][r] + X.l_s[3][r]);
            const float den = fmaf(tc::fast_exp2(m0 - mf), l0, -pL) + tc::fast_exp2(X.zn[r] - mf) + tc::fast_exp2(-mf) * (X.lden[r] + a);
            if (!(pL <= 256.f * den)) atomicOr(&X.redo, 1 << r);
          }
        }
      };
      if constexpr (!WIDE) dot_fold();
      // O^T is complete with the product of the last tile
      ok = tc::mbar_wait(bar_o(NT & 1), (uint32_t)(NT >> 1) & 1u, abw) && ok;
      tc::fence_after_sync();
      float* opart = reinterpret_cast<float*>(sm + free_stage + S::st_pt);   // [128][QR], in the free stage's Pr^T tile
      if (gw < 4) {
        float ov[QR];
        read_o(ov);
#pragma unroll
        for (int r = 0; r < QR; ++r) opart[t * QR + r] = ov[r];
      }
      if constexpr (WIDE) {
        if (exact) tc::named_bar_sync(12, 512);      // the feature group has read the folded key and made its feature row
        dot_fold();
      }
      tc::named_bar_sync(11, 256);
      const bool okb = X.abort_word == 0;
      const int redo = X.redo;
      if (__builtin_expect(redo != 0, 0)) redo_rows(redo, X.wb_row[lt], vL);
      // ---- Eq. 14: thread (query row r, value column cc)
      if (okb) {
        for (int i = gtid; i < g * d; i += 256) {
          const int r = i / d, cc = i % d;
          if ((redo >> r) & 1) continue;
          const float m0 = X.m_s[0][r];              // the score group left the final maxima there
          const float mf = fmaxf(m0, X.zn[r]);
          const float a0 = tc::fast_exp2(m0 - mf);
          float l0 = 0.f;
#pragma unroll
          for (int w = 0; w < 4; ++w) l0 += X.l_s[w][r];
          // the folded pair leaves the softmax part again: its weight as the tile's product used it (taken at the
          // stabiliser of that tile), brought to the final stabiliser like everything else in O^T
          const float vLc = sel ? __bfloat162float(vL[cc]) : 0.f;
          const float pL = sel ? used_weight(X.wb_z[lt][r], X.wb_m[lt][r]) * tc::fast_exp2(X.wb_m[lt][r] - m0) : 0.f;
          float num = a0 * fmaf(-pL, vLc, opart[cc * QR + r]);
          float den = a0 * (l0 - pL);
          const float pn = tc::fast_exp2(X.zn[r] - mf);
          num = fmaf(pn, X.vnew[cc], num);
          den += pn;
          const float e = tc::fast_exp2(-mf);
          num = fmaf(e * X.dotL[r], vLc, num);
          den = fmaf(e, X.lden[r] + X.dotL[r], den);
          ((T*)c.out)[((size_t)b * L.Hq + h * g + r) * d + cc] = __float2bfloat16_rn(num / den);
        }
        // ---- the evicted pair takes the folded member's slot (nothing moves when it is folded itself), or the
        // next free one while there is room, and the new pair enters the window ring; both were fetched at the start
        const int rowL = sel ? X.wb_row[lt] : cg;
        const bool moves = sel ? rowL < cg : c.mode == UPD_APPEND;
        constexpr int nch = d / 8;
        if (gtid < 2 * nch && moves) {
          T* dst = (gtid < nch ? (T*)L.gk : (T*)L.gv) + ((size_t)unit * lam + rowL) * d;
          *reinterpret_cast<uint4*>(dst + (gtid % nch) * 8) = X.ring_kv[gtid];
        }
        if (gtid >= 32 && gtid < 32 + 2 * nch) {
          const int i = gtid - 32;
          T* dst = (i < nch ? (T*)L.wk : (T*)L.wv) + ((size_t)unit * eta + s_ev) * d;
          *reinterpret_cast<uint4*>(dst + (i % nch) * 8) = X.new_kv[i];
        }
        if (gtid == 64 && moves) {
          L.gpos[(size_t)unit * lam + rowL] = pos_ev;
          scu[rowL] = sel ? scu[lam] : CUDART_NAN_F;   // never scored while the cache still has room
        }
        if (gtid == 96 && sel) {
          // lowest kept / highest folded score of this update
          float second = X.wb_a2[lt];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i != lt) second = fminf(second, X.wb_a1[i]);
          L.thr[(size_t)unit * 2 + 0] = second;
          L.thr[(size_t)unit * 2 + 1] = X.wb_a1[lt];
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid == 0 && X.abort_word != 0) atomicOr(L.status, 8);
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// Writes, once per layer, W^T of every KV head as the K-major 128-byte-swizzled operand image the
// decode kernel copies into shared memory: per head [d/64 K blocks][64 rows f][128 bytes = 64 i].
template <int DPL>
__global__ void k_prep_wt_image(const __nv_bfloat16* W, __nv_bfloat16* image, int Hkv) {
  constexpr int d = DPL * 32, F = 64;
  const int h = blockIdx.x;
  for (int i = threadIdx.x; i < d * F; i += blockDim.x) {
    const int j = i / F, f = i % F;
    const size_t off = (size_t)h * (d / 64) * 8192 + (size_t)(j >> 6) * 8192 + tc::sw128_off(f, (j & 63) >> 3) + (j & 7) * 2;
    image[off / 2] = W[(size_t)h * d * F + i];
  }
}

}  // namespace lola
