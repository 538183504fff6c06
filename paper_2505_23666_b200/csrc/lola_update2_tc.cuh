// Eq. 12 and Eq. 13 of the chunkwise update (bf16 layer, F = 64), one CTA per unit.  Steps 1-2 run in the
// scoring kernel's last block of a unit (select_body), steps 3-4 are k_apply_tc:
//   1. exact top-lambda of the eligible set by (score descending, older first);
//   2. ordered compaction into the pairs to fold and, per leaving pair, the slot it takes (select_lists);
//   3. the folded pairs are gathered into operand tiles, phi(K_S) is recomputed
//      (tcgen05.mma K_S W, feature map with one thread pair per row, rounded to bf16) and
//      [dH | ds] = phi(K_S)^T [V_S | 1]   (tcgen05.mma, M = 128 features, N = d + 16, K = folded pairs)
//      is added to H, s in memory, 64 pairs at a time.  Eq. 13 folds phi(k) itself into the fp32 state: phi
//      goes in as two or three bf16 parts (fold_in_three; the first in operand rows 0..63, the second in rows
//      64..127, the third in the rows of the value tile that hold no pair), each against the same value rows;
//   4. leaving pairs that stay move into the freed slots; the incoming pairs enter the window ring.
// Every wait on an mbarrier is bounded; a wait that runs out sets bit 32 of the status word.
#pragma once
#include <cuda.h>

#include "lola_generic.cuh"
#include "lola_select.cuh"
#include "lola_tc.cuh"

namespace lola {

constexpr int kUp2Threads = 512;
constexpr int kUp2MaxE = 4096;      // eligible pairs this kernel handles (scores and positions in shared memory)
constexpr int kUp2MaxFold = 512;    // leaving (and hence folded) pairs per call
constexpr uint32_t kUp2MiscBytes = 45056;
constexpr int kUp2Batch = 64;       // folded pairs per product (half an operand tile: the other half holds the second parts)

template <int DPL>
struct Update2Smem {
  static constexpr int d = DPL * 32;
  static constexpr int kblk = d / 64;
  static constexpr uint32_t b1 = 0;                        // W^T, K-major: [kblk][64][128B]
  static constexpr uint32_t kt = 16384;                    // K_S tile, K-major [kblk][128][128B]; then phi tile [2][128][128B]
  static constexpr uint32_t vt = kt + 32768;               // [V_S | 1], MN-major: [kblk + 1 column blocks][128 rows][128B], pairs in rows 0-63
  static constexpr uint32_t misc = vt + 3 * 16384;
  static constexpr uint32_t hs = misc + kUp2MiscBytes;     // dH of the unit, fp32, rows padded by 4 floats
  static constexpr uint32_t hs_row = (d + 4) * 4;
  static constexpr uint32_t total = hs + 128 * hs_row;
  static constexpr uint32_t bytes = total + 1024;
};

// shared memory of the selection
struct SelectMisc {
  alignas(16) unsigned key[kUp2MaxE];   // score bits
  int pos[kUp2MaxE];                // positions
  int cand[kUp2MaxE];
  unsigned char mark[kUp2MaxE];     // 1: the pair folds
  int fold_e[kUp2MaxFold];          // E indices of the folded pairs, ascending
  SelectScratch scratch;
};

// A key row and its value row.
struct RowPair { const __nv_bfloat16 *k, *v; };
struct RowCopy { RowPair from, to; };   // from.k == nullptr: nothing to copy

// small shared arrays of the apply kernel: where every row comes from and goes to, worked out once per row
struct ApplyMisc {
  RowPair fold[kUp2MaxFold];        // the folded pairs
  RowCopy move[kUp2MaxFold];        // leaving pair i into the sparse cache, if it stays
  RowCopy roll[kUp2MaxFold];        // incoming pairs into the window ring
  int dst[kUp2MaxFold];             // per leaving pair: the sparse-cache slot it takes, or -1
  uint64_t bar;
  uint32_t tmem_slot;
};
static_assert(sizeof(ApplyMisc) <= kUp2MiscBytes, "misc region too small");

// Copies n rows of d elements with threads t0, t0 + 1, .. of nt: 16-byte pieces, all loads of a batch before its
// stores (one round trip to memory per batch).  A function of its own and addresses from the table: the kernel is one
// long pass through its code, and fetching that code costs more than running it (inlined four times with the address
// arithmetic of every piece this part alone was 60 KB).
template <int DPL>
__device__ __noinline__ void copy_rows(const RowCopy* rows, int n, int t0, int nt) {
  constexpr int nch = DPL * 4, kBatch = 8;
#pragma unroll 1
  for (int base = t0; base < n * nch * 2; base += nt * kBatch) {
    uint4 tmp[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int i = base + k * nt, w = i / (2 * nch), ch = i % nch;
      const __nv_bfloat16* p = w < n ? ((i / nch) & 1 ? rows[w].from.v : rows[w].from.k) : nullptr;
      if (p) tmp[k] = *reinterpret_cast<const uint4*>(p + ch * 8);
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int i = base + k * nt, w = i / (2 * nch), ch = i % nch;
      if (w < n && rows[w].from.k)
        *reinterpret_cast<uint4*>(const_cast<__nv_bfloat16*>((i / nch) & 1 ? rows[w].to.v : rows[w].to.k) + ch * 8) = tmp[k];
    }
  }
}

// Steps 1-2 for one unit with a block of kUp2Threads threads; `sm` holds a SelectMisc.  The lists go to the
// state's work-list arrays (the memories are only read, so this may run beside the attention kernel).
__device__ __forceinline__ void select_body(const Layer& L, const Call& c, uint8_t* sm, const int unit) {
  SelectMisc& X = *reinterpret_cast<SelectMisc*>(sm);
  const int tid = threadIdx.x, lam = L.lam;
  const int cg = c.count_g, nE = cg + c.r, nF = nE - lam;             // 1 <= nF <= min(r, kUp2MaxFold)
  const float* scu = L.score + (size_t)unit * (lam + L.cmax);
  const size_t lo = (size_t)unit * L.cmax;
  for (int e = tid; e < nE; e += kUp2Threads) {
    X.key[e] = __float_as_uint(e < cg ? scu[e] : scu[lam + (e - cg)]);
    X.pos[e] = e < cg ? L.gpos[(size_t)unit * lam + e] : c.r_pos0 + (e - cg);
  }
  __syncthreads();
  if (tid < 256)                                       // (faster than with all threads; see select_lists)
    select_lists<256>(X.key, [&](int e) { return X.pos[e]; }, X.cand, X.mark, nE, nF, cg,
                      X.fold_e, X.scratch, tid, [] { tc::named_bar_sync(5, 256); }, [&](int i, int to) { L.move_dst[lo + i] = to; }, [] {});
  __syncthreads();
  // the lists leave through the state's work-list arrays
  for (int i = tid; i < nF; i += kUp2Threads) L.fold_idx[lo + i] = X.fold_e[i];
  if (tid == 0) {
    L.thr[(size_t)unit * 2 + 0] = __uint_as_float(X.scratch.min_keep);
    L.thr[(size_t)unit * 2 + 1] = __uint_as_float(X.scratch.max_fold);
  }
}

// Steps 3-4 from the lists of the selection.  Calls that fold nothing run only the moves and the window roll:
// nothing leaves the window yet (UPD_NONE), or every leaving pair still finds a free slot (UPD_APPEND; then the
// list of moves is known without a selection: pair i takes slot count_g + i).
// THREE: the fold takes phi in three parts (fold_in_three); otherwise 64 pairs fold at most.
template <int DPL, bool THREE>
__global__ void __launch_bounds__(kUp2Threads, 1) k_apply_tc(Layer L, Call c, const uint4* wt_image) {
  if (state_failed(L)) return;                        // an earlier kernel failed: do nothing
  using S = Update2Smem<DPL>;
  constexpr int d = DPL * 32;
  constexpr int kblk = d / 64;
  constexpr int D = 128;
  constexpr int nch = d / 8;
  typedef __nv_bfloat16 T;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = tc::smem_u32(sm);
  ApplyMisc& X = *reinterpret_cast<ApplyMisc*>(sm + S::misc);
  const int unit = blockIdx.x, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lam = L.lam, eta = L.eta;
  const bool fold = c.mode == UPD_SELECT;
  const int cg = c.count_g, nF = fold ? cg + c.r - lam : 0;           // folding: 1 <= nF <= min(r, kUp2MaxFold)
  const int n_roll = min(c.n, eta);                                   // incoming pairs that enter the ring
  float* scu = L.score + (size_t)unit * (lam + L.cmax);
  const uint32_t bar = sbase + S::misc + (uint32_t)offsetof(ApplyMisc, bar);
  uint32_t ph = 0;
  bool ok = true;

  if (tid == 0) { tc::mbar_init(bar, 1); tc::mbar_init_fence(); }
  if (fold && warp == 0) tc::tmem_alloc(&X.tmem_slot, 256);
  // launched early (programmatic dependent launch): the zeroed operand tiles need nothing from memory
  if (tid == 0) tc::grid_dep_launch_dependents();
  if (fold)
    for (int i = tid; i < (32768 + 3 * 16384) / 16; i += kUp2Threads)
      *reinterpret_cast<uint4*>(sm + S::kt + i * 16) = make_uint4(0, 0, 0, 0);
  tc::grid_dep_wait();                               // the attention kernel has read the memories this kernel changes
  // everything the set-up needs from global memory is requested at once (one round trip): the work lists, the W^T
  // image; thread i then works out where folded pair i, leaving pair i and incoming pair i lie
  {
    const size_t lo = (size_t)unit * L.cmax;
    int e = 0, dst = c.mode == UPD_APPEND ? cg + tid : -1;
    uint4 pre_w[kblk];
    if (fold) {
      if (tid < nF) e = L.fold_idx[lo + tid];
      if (tid < c.r) dst = L.move_dst[lo + tid];
      const uint4* img = wt_image + (size_t)h * kblk * 512;
#pragma unroll
      for (int q = 0; q < kblk; ++q) pre_w[q] = img[tid + q * kUp2Threads];
#pragma unroll
      for (int q = 0; q < kblk; ++q) *reinterpret_cast<uint4*>(sm + S::b1 + (tid + q * kUp2Threads) * 16) = pre_w[q];
    }
    if (tid < c.r) {
      const T *kp, *vp;
      locate_leaving<T>(L, c, unit, b, h, c.r_pos0 + tid, kp, vp);
      const size_t o = ((size_t)unit * lam + (dst >= 0 ? dst : 0)) * d;
      X.move[tid].from.k = dst >= 0 ? kp : nullptr;
      X.move[tid].from.v = vp;
      X.move[tid].to.k = (const T*)L.gk + o;
      X.move[tid].to.v = (const T*)L.gv + o;
      X.dst[tid] = dst;
    }
    if (tid < nF) {
      const T *kp, *vp;
      locate_eligible<T>(L, c, unit, b, h, e, kp, vp);
      X.fold[tid].k = kp;
      X.fold[tid].v = vp;
    }
    if (tid < n_roll) {
      const int ci = c.n - n_roll + tid;
      const size_t o = ((size_t)unit * eta + (c.n_seen + ci) % eta) * d, q = (((size_t)b * c.n + ci) * L.Hkv + h) * d;
      X.roll[tid].from.k = (const T*)c.k + q;
      X.roll[tid].from.v = (const T*)c.v + q;
      X.roll[tid].to.k = (const T*)L.wk + o;
      X.roll[tid].to.v = (const T*)L.wv + o;
    }
  }
  __syncthreads();
  // leaving pairs that stay go into the freed slots, then into the slots beyond count_g
  auto do_movers = [&](int t0, int nt) {
    copy_rows<DPL>(X.move, c.r, t0, nt);
    for (int i = t0; i < c.r; i += nt)
      if (X.dst[i] >= 0) {
        L.gpos[(size_t)unit * lam + X.dst[i]] = c.r_pos0 + i;
        scu[X.dst[i]] = fold ? scu[lam + i] : CUDART_NAN_F;          // never scored while the cache still has room
      }
  };
  if (!fold) {
    do_movers(tid, kUp2Threads);
    __syncthreads();                                                 // ring rows are read above before they are replaced
    copy_rows<DPL>(X.roll, n_roll, tid, kUp2Threads);                // the window takes the chunk's last eta tokens
    return;
  }
  const uint32_t tmem = X.tmem_slot;
  const uint32_t tm_u = tmem, tm_d = tmem + 64;
  const int wq = warp & 3, hf = (warp >> 2) & 1;
  const int t = wq * 32 + lane;
  const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
  float ds_sum = 0.f;
  for (int f0 = 0; f0 < nF; f0 = THREE ? f0 + kUp2Batch : nF) {
    const int nb = min(kUp2Batch, nF - f0);
    const bool last = !THREE || f0 + kUp2Batch >= nF;
    // ---- 3. gather the folded pairs into the operand tiles (rows beyond the batch are zero)
    // (the tiles start out zero; a later batch clears its own rest.)  All loads of a thread before its stores
    {
      constexpr int kG = kUp2Batch * nch * 2 / kUp2Threads;
      uint4 val[kG];
#pragma unroll
      for (int q = 0; q < kG; ++q) {
        const int i = tid + q * kUp2Threads, row = i / (2 * nch), rem = i % (2 * nch), isv = rem / nch, ch = rem % nch;
        val[q] = make_uint4(0, 0, 0, 0);
        if (row < nb) val[q] = *reinterpret_cast<const uint4*>((isv ? X.fold[f0 + row].v : X.fold[f0 + row].k) + ch * 8);
      }
#pragma unroll
      for (int q = 0; q < kG; ++q) {
        const int i = tid + q * kUp2Threads, row = i / (2 * nch), rem = i % (2 * nch), isv = rem / nch, ch = rem % nch;
        if (row >= nb && (!THREE || f0 == 0)) continue;
        *reinterpret_cast<uint4*>(sm + (isv ? S::vt : S::kt) + (ch >> 3) * 16384 + tc::sw128_off(row, ch & 7)) = val[q];
      }
    }
    const int rows = THREE && f0 > 0 ? kUp2Batch : nb;
    if (tid < rows)                                                  // the column of ones (block kblk, column 0)
      *reinterpret_cast<T*>(sm + S::vt + kblk * 16384 + tc::sw128_off(tid, 0)) = __float2bfloat16_rn(tid < nb ? 1.0f : 0.0f);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
#pragma unroll
      for (int ks = 0; ks < d / 16; ++ks)
        tc::mma_bf16_ss(tm_u, tc::make_desc_sw128(sbase + S::kt + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024),
                        tc::make_desc_sw128(sbase + S::b1 + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024),
                        tc::make_idesc_bf16(128, 64, false, false), ks > 0);
      tc::mma_commit(bar);
    }
    // the upper half of the block moves the staying pairs meanwhile (the gathers have read every slot and ring
    // row the fold needs; the movers only read ring rows and write freed or new slots)
    if (tid >= 256) { if (last) do_movers(tid - 256, kUp2Threads - 256); }
    else ok = tc::mbar_wait(bar, ph) && ok;
    ph ^= 1;
    tc::fence_after_sync();
    if (tid < 256) {                                                 // one thread pair per row: half of the feature map each
      const bool ek = L.phi_kind == 1;
      uint32_t u[64];
      uint64_t x2[32];
      tc::tmem_ld64u(tm_u + lane_addr, u);                           // (warp-wide: every lane takes part)
      if (t < 64) {
        const uint64_t inv2 = tc::phi_half_f32(u, hf != 0, ek, x2);
        // phi tile over the key tile (consumed): row = folded pair (first parts) and 64 + folded pair (second parts),
        // 64 features per 128-byte row and block; third parts behind the value rows
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
          uint32_t p1[4], p2[4], p3[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float x, y;
            tc::unpack_f2(ek ? x2[ch * 4 + e] : tc::mul2(x2[ch * 4 + e], inv2), x, y);
            p1[e] = tc::next_part(x, y);
            p2[e] = tc::next_part(x, y);
            if (THREE) p3[e] = tc::next_part(x, y);
          }
          const uint32_t off = (uint32_t)hf * 16384u;
          *reinterpret_cast<uint4*>(sm + S::kt + off + tc::sw128_off(t, ch)) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
          *reinterpret_cast<uint4*>(sm + S::kt + off + tc::sw128_off(t + 64, ch)) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
          if (THREE) *reinterpret_cast<uint4*>(sm + S::vt + off + tc::sw128_off(t + 64, ch)) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
        }
      }
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
      // (rows of no pair hold the feature map of a zero key against a zero value row)
      tc::fold_product<DPL, THREE>(tm_d, sbase + S::kt, sbase + S::vt, true);
      tc::mma_commit(bar);
    }
    if (last && tid >= 256) copy_rows<DPL>(X.roll, n_roll, tid - 256, kUp2Threads - 256);   // the movers' reads of the ring ended at the barrier above
    else ok = tc::mbar_wait(bar, ph) && ok;                          // (not the last: all wait, the tiles are written again)
    ph ^= 1;
    tc::fence_after_sync();
    if (tid < 256 && ok) {                                           // row j = t, columns [hf * d/2, +d/2)
      // dH from tensor memory into the (padded) rows of the staging area, where the batches are added up (see fold_product)
      constexpr int HC = d / 2;
      float* Hrow = reinterpret_cast<float*>(sm + S::hs + (size_t)t * S::hs_row) + hf * HC;
#pragma unroll
      for (int c0 = 0; c0 < HC; c0 += 32) {
        float p[32];
        tc::tmem_ld32(tm_d + lane_addr + hf * HC + c0, p);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float4* to = reinterpret_cast<float4*>(Hrow + c0 + q * 4);
          float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
          if (THREE && f0 > 0) o = *to;
          *to = make_float4(o.x + p[q * 4], o.y + p[q * 4 + 1], o.z + p[q * 4 + 2], o.w + p[q * 4 + 3]);
        }
      }
      if (hf == 0) {
        float ds[2];
        tc::tmem_ld2(tm_d + lane_addr + d, ds);
        ds_sum += ds[0];
        if (last) L.s[(size_t)unit * D + t] += ds_sum;
      }
    }
  }
  // (the lower half alone: the upper half is still rolling the window)
  if (tid < 256) tc::named_bar_sync(2, 256);
  if (tid < 256 && ok) {
    // H += dH: 16-byte reductions performed at the L2, a warp covers 512 consecutive bytes (nothing is read back)
    float4* Hg4 = reinterpret_cast<float4*>(L.H + (size_t)unit * D * d);
    for (int i = tid; i < D * (d / 4); i += 256) {
      const int row = i / (d / 4), c4 = i % (d / 4);
      atomicAdd(Hg4 + i, *reinterpret_cast<const float4*>(sm + S::hs + (size_t)row * S::hs_row + (size_t)c4 * 16));
    }
  }
  if (!ok && tid == 0) atomicOr(L.status, 32);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

}  // namespace lola
