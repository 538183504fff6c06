// The generation step (Eq. 11-14) of an fp32 layer with F = 64 as one kernel: a cluster of K thread blocks per (batch row,
// KV head) unit, all arithmetic in fp32 on the CUDA cores.
//
// What bounds it: latency.  A step of the tiny layer reads 160 KB a unit and takes 2 MFMA; what counts is how many times
// the blocks meet and how long the chains between are.  The pairs a step may see (sparse cache, then the ring from its
// oldest slot on) are dealt out one by one (block k: pairs k, k + K, ..), so that all blocks score and attend equally many,
// and everything a block finds out is sent to the others in ONE exchange:
//   * its lowest-scored pair (Eq. 12: one pair leaves, one is folded), with score, key product, feature and value row.  That
//     pair is left out of the block's softmax sums; of all these pairs the lowest is folded and the others are summands
//     of Eq. 14 like any block's.  Nothing is ever taken out of a sum again.
//   * its stabiliser, sum of weights and weighted values per query row (Eq. 14 without that pair), for the block that finishes the row
// Behind it every block adds its D / K rows of the fold to H and s (Eq. 13), block r mod K finishes query row r, the block that
// holds the leaving pair moves it.
// Both products, [u] = [K; Q] W and [P] = phi [K; Q] H, are split over the inner dimension: a warp has d / 8 rows of W (in
// registers before the step ahead is complete) and 16 rows of H in registers, all pairs pass by as broadcasts, and the eight
// parts meet in shared memory.
// A pair's rows come in tiles of TR, two in flight.
// Measured: 8 units of 128 + 64 pairs, d = 64: 9.0 us a step (26 as two rounds of k_unit_run, where scoring, fold and attention
// follow each other with a cluster barrier between each and one block attends); of 16.5 K cycles loads take 1.4, the products 5,
// the feature map 2.3, scores and selection 2, the exchange 2.5, the outputs 2.  With W and H in shared memory, rows
// interleaved for packed fp32 instructions (which run at half the rate of plain ones), it was 13.1 us.
#pragma once
#include "lola_generic.cuh"
#include "lola_tc.cuh"

namespace lola {

constexpr int kStepThreads = 256;
constexpr int kStepQ = 8;              // query rows per unit the kernel carries
// The stabiliser of Eq. 14 (any will do) stays 0 until a weight would exceed 2^8: most blocks' sums then meet without a factor,
// whose rounding a whole block's values would share.  (Error of the outputs for scores below 2: 1.03e-7 - 1.06e-7 of their norm, with
// a stabiliser that follows every score 1.05e-7 - 1.11e-7; a lag of 64 is no better, and values from 1e11 on overflowed with it.)
constexpr float kStepLag = 5.545177f;

template <int DPL>
struct StepMsg {                       // what a block tells the others
  unsigned key_lo, key_hi;             // lowest pair: score bits above (2^31 - 1 - position); all ones: none
  unsigned second;                     // lowest score but that
  unsigned failed;
  int row, pad[3];                     // the pair's place in the unit's list
  float z[kStepQ];                     // its q.k
  float m[kStepQ], l[kStepQ];          // stabiliser and sum of weights of the block's other pairs
  float phi[128], v[DPL * 32];         // the pair's rows
};

template <int DPL>
struct StepSmem {
  static constexpr int d = DPL * 32, TR = 2048 / d, NJ = TR + kStepQ;
  alignas(16) float part[8][NJ][d];    // products, an eighth of the inner dimension each
  alignas(16) float xk[2][TR][d + 4];
  alignas(16) float xv[2][TR][d];
  alignas(16) float xq[kStepQ][d];
  alignas(16) float phi[NJ][128];      // scored rows of the tile, then the queries
  alignas(16) float phiq[kStepQ][128];
  alignas(16) float lin[kStepQ][d];    // phi(q)^T H
  alignas(16) float kv_new[2][d];
  alignas(16) float s[128];
  float den[NJ], sc[TR], lden[kStepQ], zn[kStepQ];
  float z[kStepQ][TR];
  int pos[2][TR];
  alignas(16) StepMsg<DPL> msg;
  alignas(16) float o[kStepQ][d];      // weighted values of the block's other pairs
  alignas(16) StepMsg<DPL> peer[8];
  alignas(16) float peer_o[16][d];     // [block x rows finished here]
  float lev_score;
  uint64_t bar;
  int abort_word, failed;
};
static_assert(sizeof(StepSmem<2>) <= 232448 && sizeof(StepSmem<4>) <= 232448, "shared memory");

template <int DPL>
__global__ void __launch_bounds__(kStepThreads, 1) k_unit_step(Layer L, Call c) {
  typedef StepSmem<DPL> S;
  typedef StepMsg<DPL> Msg;
  constexpr int d = DPL * 32, d4 = d / 4, TR = S::TR, NC = d / 32, WR = d / 8;   // NC: columns of a lane
  extern __shared__ __align__(16) uint8_t smem_raw[];
  S& X = *reinterpret_cast<S*>(smem_raw);
  const int K = (int)tc::cluster_size(), rank = (int)tc::cluster_rank();
  const int unit = blockIdx.x / K, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lam = L.lam, eta = L.eta, g = L.g;
  const int cg = c.count_g, cw = min(eta, c.n_seen), NL = cg + cw;
  const bool sel = c.mode == UPD_SELECT;
  const int ring0 = (c.n_seen - cw) % eta, s_ev = c.n_seen % eta;
  const int n_own = (NL - rank + K - 1) / K, n_tiles = max(1, (n_own + TR - 1) / TR);
  const int n_scored = sel ? (cg + 1 - rank + K - 1) / K : 0;   // the first of them (the leaving pair is the oldest of the ring)
  const int mover = cg % K;                            // the block that holds the leaving pair
  const uint32_t sbase = tc::smem_u32(smem_raw), bar = tc::smem_u32(&X.bar);
  volatile int* abw = &X.abort_word;
  const size_t gofs = (size_t)unit * lam * d, wofs = (size_t)unit * eta * d;
  const size_t qofs = ((size_t)b * L.Hq + h * g) * d, kofs = ((size_t)b * L.Hkv + h) * d;
  const int* gpos = L.gpos + (size_t)unit * lam;
  float* scu = L.score + (size_t)unit * (lam + L.cmax);

  if (tid == 0) {
    X.abort_word = 0;
    tc::mbar_init(bar, 1);
    tc::mbar_init_fence();
    tc::grid_dep_launch_dependents();
  }
  float2 wr[WR];                                       // rows [warp WR, + WR) of W, features 2 lane, 2 lane + 1
#pragma unroll
  for (int j = 0; j < WR; ++j) wr[j] = *reinterpret_cast<const float2*>((const float*)L.W + ((size_t)h * d + warp * WR + j) * 64 + 2 * lane);
  __syncthreads();
  if (K > 1) tc::cluster_arrive();                     // this block runs and its barrier is set up
  tc::grid_dep_wait();                                 // everything before this step in the stream is complete

  // what is kept in registers is requested first
  const int pre_status = tid == 0 ? *reinterpret_cast<volatile const int*>(L.status) : 0;
  float hr[16][NC];                                    // rows [16 warp, + 16) of H, columns NC lane ..
  {
    const float* Hg = L.H + ((size_t)unit * 128 + warp * 16) * d + NC * lane;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if constexpr (NC == 2) { const float2 x = *reinterpret_cast<const float2*>(Hg + j * d); hr[j][0] = x.x; hr[j][1] = x.y; }
      else { const float4 x = *reinterpret_cast<const float4*>(Hg + j * d); hr[j][0] = x.x; hr[j][1] = x.y; hr[j][2] = x.z; hr[j][3] = x.w; }
    }
  }
  float4 lev = make_float4(0.f, 0.f, 0.f, 0.f);        // what the ring slot of the new pair holds
  if (rank == mover && tid < 2 * d4) lev = *reinterpret_cast<const float4*>((const float*)(tid < d4 ? L.wk : L.wv) + wofs + (size_t)s_ev * d + tid % d4 * 4);
  // queries, new pair and s go with the first tile
  for (int i = tid; i < (kStepQ + 2) * d4 + 32; i += kStepThreads) {
    const int r = i / d4, c4 = i % d4 * 4;
    if (r < kStepQ) tc::cp_async16(tc::smem_u32(&X.xq[r][c4]), (const float*)c.q + qofs + (r < g ? r * d + c4 : 0), r < g ? 16u : 0u);
    else if (r < kStepQ + 2) tc::cp_async16(tc::smem_u32(&X.kv_new[r - kStepQ][c4]), (const float*)(r == kStepQ ? c.k : c.v) + kofs + c4);
    else tc::cp_async16(tc::smem_u32(&X.s[(i - (kStepQ + 2) * d4) * 4]), L.s + (size_t)unit * 128 + (i - (kStepQ + 2) * d4) * 4);
  }

  // the lowest-scored pair so far: (score, then the younger) as one number, the lowest score but that
  unsigned long long low = ~0ull;
  unsigned second = 0xffffffffu;
  int low_row = -1;
  // warp r: query row r, its stabiliser, this lane's part of the sum of weights, weighted values and what their last addition lost
  float acc[NC], lost[NC], m = 0.f, l = 0.f, lsum = 0.f;
#pragma unroll
  for (int i = 0; i < NC; ++i) acc[i] = lost[i] = 0.f;

#pragma unroll 1
  for (int t = 0; t < n_tiles; ++t) {
    const int buf = t & 1, rows = min(TR, n_own - t * TR);
    const int nj = max(0, min(TR, n_scored - t * TR)); // scored rows: the first ones
    const int jobs = nj + (t == 0 ? g : 0);
    // pairs of the next tile (of the first, too, at the start); those beyond the block's share read as zeros
#pragma unroll 1
    for (int t2 = t == 0 ? 0 : t + 1; t2 <= t + 1 && t2 < n_tiles; ++t2) {
#pragma unroll
      for (int i = tid; i < TR * d4; i += kStepThreads) {
        const int row = i / d4, c4 = i % d4 * 4, e = rank + (t2 * TR + row) * K;
        int slot = ring0 + e - cg;
        if (slot >= eta) slot -= eta;
        const bool in = e < NL, isg = e < cg;
        const size_t at = in ? (isg ? gofs + (size_t)e * d + c4 : wofs + (size_t)slot * d + c4) : 0;
        tc::cp_async16(tc::smem_u32(&X.xk[t2 & 1][row][c4]), (const float*)(isg ? L.gk : L.wk) + at, in ? 16u : 0u);
        tc::cp_async16(tc::smem_u32(&X.xv[t2 & 1][row][c4]), (const float*)(isg ? L.gv : L.wv) + at, in ? 16u : 0u);
      }
      if (tid < TR) {
        const int e = rank + (t2 * TR + tid) * K;
        if (e < cg) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(&X.pos[t2 & 1][tid])), "l"(gpos + e) : "memory");
        else X.pos[t2 & 1][tid] = c.r_pos0;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (t + 1 < n_tiles) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (t == 0 && tid == 0) X.failed = pre_status;     // (an earlier kernel failed: leave the memories as they are)
    __syncthreads();
    // ---- u = x W
#pragma unroll 1
    for (int r0 = 0; r0 < jobs; r0 += 4) {
      float a[4][2];
      float* to[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int j = min(r0 + r, jobs - 1);
        const float* x = (j < nj ? X.xk[buf][j] : X.xq[j - nj]) + warp * WR;
        to[r] = &X.part[warp][j][2 * lane];
        a[r][0] = a[r][1] = 0.f;
#pragma unroll
        for (int k = 0; k < WR; k += 4) {
          const float4 xx = *reinterpret_cast<const float4*>(x + k);
          a[r][0] = fmaf(xx.x, wr[k].x, a[r][0]); a[r][1] = fmaf(xx.x, wr[k].y, a[r][1]);
          a[r][0] = fmaf(xx.y, wr[k + 1].x, a[r][0]); a[r][1] = fmaf(xx.y, wr[k + 1].y, a[r][1]);
          a[r][0] = fmaf(xx.z, wr[k + 2].x, a[r][0]); a[r][1] = fmaf(xx.z, wr[k + 2].y, a[r][1]);
          a[r][0] = fmaf(xx.w, wr[k + 3].x, a[r][0]); a[r][1] = fmaf(xx.w, wr[k + 3].y, a[r][1]);
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) *reinterpret_cast<float2*>(to[r]) = make_float2(a[r][0], a[r][1]);
    }
    // ---- q.k of all pairs of the tile (t = 0: and of the new pair), eight lanes each
    const int zrows = rows + (t == 0 ? 1 : 0);
#pragma unroll 1
    for (int r = 0; r < g; ++r)
#pragma unroll 1
      for (int i0 = warp * 4; i0 < zrows; i0 += kStepThreads / 8) {
        const int row = min(i0 + (lane >> 3), zrows - 1);
        const float* x = row < rows ? X.xk[buf][row] : X.kv_new[0];
        float a = 0.f;
#pragma unroll
        for (int q = 0; q < d4; q += 8) {
          const float4 y = *reinterpret_cast<const float4*>(&X.xq[r][(q + (lane & 7)) * 4]), kx = *reinterpret_cast<const float4*>(x + (q + (lane & 7)) * 4);
          a = fmaf(y.x, kx.x, fmaf(y.y, kx.y, fmaf(y.z, kx.z, fmaf(y.w, kx.w, a))));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((lane & 7) == 0) *(row < rows ? &X.z[r][row] : &X.zn[r]) = a * L.scale;
      }
    __syncthreads();
    // ---- feature map: three rows of a warp side by side
#pragma unroll 1
    for (int j0 = warp; j0 < jobs; j0 += 24) {
      float p[3][4], s1[3], s2[3], dn[3];              // features 2 lane, 2 lane + 1 of both halves
      const float2 sa = *reinterpret_cast<const float2*>(&X.s[2 * lane]), sb = *reinterpret_cast<const float2*>(&X.s[64 + 2 * lane]);
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int j = min(j0 + 8 * r, jobs - 1);
        float2 u = *reinterpret_cast<const float2*>(&X.part[0][j][2 * lane]);
#pragma unroll
        for (int q = 1; q < 8; ++q) { const float2 e = *reinterpret_cast<const float2*>(&X.part[q][j][2 * lane]); u.x += e.x; u.y += e.y; }
        float mx = 0.f, mn = 0.f;
        if (L.phi_kind != 1) { mx = warp_max_redux(fmaxf(u.x, u.y)); mn = -warp_max_redux(fmaxf(-u.x, -u.y)); }
        p[r][0] = expf(u.x - mx); p[r][1] = expf(u.y - mx); p[r][2] = expf(mn - u.x); p[r][3] = expf(mn - u.y);
        s1[r] = p[r][0] + p[r][1];
        s2[r] = p[r][2] + p[r][3];
      }
      if (L.phi_kind != 1) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int r = 0; r < 3; ++r) { s1[r] += __shfl_xor_sync(0xffffffffu, s1[r], o); s2[r] += __shfl_xor_sync(0xffffffffu, s2[r], o); }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const float i1 = 1.0f / s1[r], i2 = 1.0f / s2[r];
          p[r][0] *= i1; p[r][1] *= i1; p[r][2] *= i2; p[r][3] *= i2;
        }
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int j = min(j0 + 8 * r, jobs - 1);       // (a row that is not there: the last one's values again)
        *reinterpret_cast<float2*>(&X.phi[j][2 * lane]) = make_float2(p[r][0], p[r][1]);
        *reinterpret_cast<float2*>(&X.phi[j][64 + 2 * lane]) = make_float2(p[r][2], p[r][3]);
        dn[r] = fmaf(p[r][0], sa.x, p[r][1] * sa.y) + fmaf(p[r][2], sb.x, p[r][3] * sb.y);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < 3; ++r) dn[r] += __shfl_xor_sync(0xffffffffu, dn[r], o);
      if (lane < 3) X.den[min(j0 + 8 * lane, jobs - 1)] = lane == 0 ? dn[0] : lane == 1 ? dn[1] : dn[2];
    }
    __syncthreads();
    // ---- phi H
#pragma unroll 1
    for (int r0 = 0; r0 < jobs; r0 += 4) {
      float a[4][NC];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float* x = &X.phi[min(r0 + r, jobs - 1)][warp * 16];
#pragma unroll
        for (int i = 0; i < NC; ++i) a[r][i] = 0.f;
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
          const float4 xx = *reinterpret_cast<const float4*>(x + k);
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            a[r][i] = fmaf(xx.x, hr[k][i], a[r][i]); a[r][i] = fmaf(xx.y, hr[k + 1][i], a[r][i]);
            a[r][i] = fmaf(xx.z, hr[k + 2][i], a[r][i]); a[r][i] = fmaf(xx.w, hr[k + 3][i], a[r][i]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float* to = &X.part[warp][min(r0 + r, jobs - 1)][NC * lane];
        if constexpr (NC == 2) *reinterpret_cast<float2*>(to) = make_float2(a[r][0], a[r][1]);
        else *reinterpret_cast<float4*>(to) = make_float4(a[r][0], a[r][1], a[r][2], a[r][3]);
      }
    }
    __syncthreads();
    // ---- the parts meet: Eq. 10 of a pair, the linear term of a query; three rows of a warp side by side
#pragma unroll 1
    for (int j0 = warp; j0 < jobs; j0 += 24) {
      float err[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int j = min(j0 + 8 * r, jobs - 1);
        const float dn = X.den[j], inv = dn > 0.f ? 1.0f / dn : 0.f;
        const float* v = j < nj ? &X.xv[buf][j][NC * lane] : &X.lin[j - nj][NC * lane];
        float a[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) a[i] = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
          for (int i = 0; i < NC; i += 2) { const float2 e = *reinterpret_cast<const float2*>(&X.part[q][j][NC * lane + i]); a[i] += e.x; a[i + 1] += e.y; }
        err[r] = 0.f;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          if (j >= nj) X.lin[j - nj][NC * lane + i] = a[i];
          const float x = fmaf(a[i], inv, -v[i]);
          err[r] = fmaf(x, x, err[r]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < 3; ++r) err[r] += __shfl_xor_sync(0xffffffffu, err[r], o);
      const int jl = min(j0 + 8 * lane, jobs - 1);
      if (lane < 3 && jl < nj) X.sc[jl] = sqrtf(lane == 0 ? err[0] : lane == 1 ? err[1] : err[2]);
    }
    if (t == 0) {                                      // (the feature rows' places are the next tile's)
      for (int i = tid; i < g * 32; i += kStepThreads) *reinterpret_cast<float4*>(&X.phiq[i >> 5][(i & 31) * 4]) = *reinterpret_cast<const float4*>(&X.phi[nj + (i >> 5)][(i & 31) * 4]);
      if (tid < g) X.lden[tid] = X.den[nj + tid];
    }
    __syncthreads();
    // ---- the tile's lowest pair, by every warp for itself
    const int e = rank + (t * TR + lane) * K;          // this lane's pair
    unsigned hi = 0xffffffffu, lo = 0xffffffffu;
    if (lane < nj) { hi = __float_as_uint(X.sc[lane]); lo = (unsigned)(0x7fffffff - X.pos[buf][lane]); }
    const unsigned whi = __reduce_min_sync(0xffffffffu, hi), wlo = __reduce_min_sync(0xffffffffu, hi == whi ? lo : 0xffffffffu);
    const unsigned long long tkey = ((unsigned long long)whi << 32) | wlo;
    const bool is_min = lane < nj && hi == whi && lo == wlo, newc = nj > 0 && tkey < low;
    const int src = __ffs(__ballot_sync(0xffffffffu, is_min)) - 1;
    second = min(second, __reduce_min_sync(0xffffffffu, is_min ? 0xffffffffu : hi));
    second = min(second, (unsigned)((newc ? low : tkey) >> 32));
    const int out = newc ? src : -1;                   // the row that stays out of the sums
    if (lane < nj && warp == 7 && X.failed == 0) {
      if (lane != out) scu[e < cg ? e : lam] = X.sc[lane];   // (the lowest pair's at the end: its slot may be taken)
      if (e == cg) X.lev_score = X.sc[lane];
    }
    // ---- Eq. 14: warp r has query row r
    if (warp < g) {
      const float zz = lane < rows && lane != out ? X.z[warp][lane] : -CUDART_INF_F;
      const float zo = newc && low != ~0ull ? X.msg.z[warp] : -CUDART_INF_F;    // the lowest pair so far joins the others
      const float mx = fmaxf(zo, warp_max_redux(zz)), mn = mx > m + kStepLag ? mx : m, alpha = expf(m - mn), p = expf(zz - mn), po = expf(zo - mn);
      l = fmaf(l, alpha, lane == 0 ? p + po : p);
      m = mn;
      if (t + 1 == n_tiles) lsum = warp_sum(l);
      // (four sums side by side: one long one rounds more, 1.36e-7 of the outputs' norm against 1.05e-7; tiles are added with
      // Kahan's correction, and the sum of weights stays in its lanes: seven tiles 1.17e-7 -> 1.04e-7, 20 at d = 128 1.50e-7 -> 1.04e-7)
      float a4[4][NC];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < NC; ++i) a4[q][i] = 0.f;
      auto add_values = [&](int but) {                 // (no pair: weight 0, values 0)
#pragma unroll
        for (int r0 = 0; r0 < TR; r0 += 4)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float w = __shfl_sync(0xffffffffu, p, r0 + q);
            if (r0 + q == but) continue;
#pragma unroll
            for (int i = 0; i < NC; i += 2) {
              const float2 v = *reinterpret_cast<const float2*>(&X.xv[buf][r0 + q][NC * lane + i]);
              a4[q][i] = fmaf(w, v.x, a4[q][i]);
              a4[q][i + 1] = fmaf(w, v.y, a4[q][i + 1]);
            }
          }
      };
      if (out < 0 || whi < 0x7f800000u) add_values(-1);
      else add_values(out);                            // its score is no number, so its value need not be finite: a weight of 0 would not keep it out
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        float y = (a4[0][i] + a4[1][i]) + (a4[2][i] + a4[3][i]);
        if (po != 0.f) y = fmaf(po, X.msg.v[NC * lane + i], y);
        const float a = acc[i] * alpha;
        y = fmaf(lost[i], alpha, y);
        acc[i] = a + y;
        lost[i] = fabsf(acc[i]) < CUDART_INF_F ? y - (acc[i] - a) : 0.f;
      }
    }
    if (n_tiles > 1) __syncthreads();                  // (the pair that joined has been read)
    if (newc) {
      if (warp == 7 && lane == 0 && low != ~0ull && X.failed == 0) scu[low_row < cg ? low_row : lam] = __uint_as_float((unsigned)(low >> 32));
      low = tkey;
      low_row = rank + (t * TR + src) * K;
      if (tid >= 128) X.msg.phi[tid - 128] = X.phi[src][tid - 128];
      else if (tid < d) X.msg.v[tid] = X.xv[buf][src][tid];
      if (tid >= 96 && tid < 96 + g) X.msg.z[tid - 96] = X.z[tid - 96][src];   // (d = 128: these threads have a value, too)
    }
    if (t + 1 < n_tiles) __syncthreads();
  }
  if (warp < g) {
#pragma unroll
    for (int i = 0; i < NC; i += 2) *reinterpret_cast<float2*>(&X.o[warp][NC * lane + i]) = make_float2(acc[i], acc[i + 1]);
    if (lane == 0) { X.msg.m[warp] = m; X.msg.l[warp] = lsum; }
  }
  if (tid == 224) {
    X.msg.key_lo = (unsigned)low;
    X.msg.key_hi = (unsigned)(low >> 32);
    X.msg.second = second;
    X.msg.failed = X.failed != 0 || *abw != 0 ? 1u : 0u;
    X.msg.row = low_row;
  }
  const int per = (g + K - 1) / K;                     // query rows a block finishes: k, k + K, ..
  auto finished_by = [&](int k) { return k < g ? (g - k + K - 1) / K : 0; };
  if (K > 1 && tid == 0) tc::mbar_expect_tx(bar, (uint32_t)K * ((uint32_t)sizeof(Msg) + (uint32_t)finished_by(rank) * 4u * d));
  __syncthreads();
  // ---- the exchange: a warp per block (a block alone was not launched as a cluster and takes no cluster instructions)
  if (K > 1) {
    tc::cluster_wait();
    if (warp < K) {
      const uint32_t peer = tc::map_rank(sbase, (uint32_t)warp), to_bar = peer + (bar - sbase);
      const uint32_t to = peer + (uint32_t)offsetof(S, peer) + (uint32_t)(rank * sizeof(Msg)), to_o = peer + (uint32_t)offsetof(S, peer_o) + (uint32_t)(rank * per * d * 4);
      const uint4* from = reinterpret_cast<const uint4*>(&X.msg);
#pragma unroll
      for (int i = 0; i < (int)sizeof(Msg) / 16; i += 32)
        if (i + lane < (int)sizeof(Msg) / 16) tc::st_async_v4(to + 16u * (uint32_t)(i + lane), from[i + lane], to_bar);
#pragma unroll 1
      for (int r = warp, q = 0; r < g; r += K, ++q)
        if (lane < d4) tc::st_async_v4(to_o + 16u * (uint32_t)(q * d4 + lane), *reinterpret_cast<const uint4*>(&X.o[r][lane * 4]), to_bar);
    }
  } else {
    for (int i = tid; i < (int)sizeof(Msg) / 16; i += kStepThreads) reinterpret_cast<uint4*>(&X.peer[0])[i] = reinterpret_cast<const uint4*>(&X.msg)[i];
    for (int i = tid; i < g * d4; i += kStepThreads) reinterpret_cast<uint4*>(&X.peer_o[0][0])[i] = reinterpret_cast<const uint4*>(&X.o[0][0])[i];
    __syncthreads();
  }
  bool ok = K > 1 ? tc::mbar_wait(bar, 0, abw) : true;
  // ---- the pair to fold: the lowest (score, then the younger) of all, by every warp for itself
  const int k8 = lane & 7;
  const unsigned khi = k8 < K ? X.peer[k8].key_hi : 0xffffffffu, klo = k8 < K ? X.peer[k8].key_lo : 0xffffffffu;
  ok = !__any_sync(0xffffffffu, !ok || (k8 < K && X.peer[k8].failed != 0u));
  const unsigned whi = __reduce_min_sync(0xffffffffu, khi), wlo = __reduce_min_sync(0xffffffffu, khi == whi ? klo : 0xffffffffu);
  const int wr_ = __ffs(__ballot_sync(0xffffffffu, khi == whi && klo == wlo)) - 1;
  const Msg& win = X.peer[wr_];
  const int wrow = sel ? win.row : cg;                 // (while there is room the leaving pair takes the next free slot)
  if (warp < per && rank + warp * K < g) {
    // ---- Eq. 14 of the query rows this block finishes
    const int r = rank + warp * K;
    // lanes 0-7: the blocks' sums, 8-15: their lowest pairs, 16: the new pair, 17: the linear term (a score of 0)
    const bool sum = lane < K, pair = (lane & 24) == 8 && k8 < K && k8 != wr_ && khi != 0xffffffffu;
    const float zz = sum ? X.peer[k8].m[r] : pair ? X.peer[k8].z[r] : lane == 16 ? X.zn[r] : lane == 17 ? 0.f : -CUDART_INF_F;
    const float mx = warp_max_redux(zz), w = expf(zz - (mx > kStepLag ? mx : 0.f));
    const float4 p = *reinterpret_cast<const float4*>(&X.phiq[r][lane * 4]), f = *reinterpret_cast<const float4*>(&win.phi[lane * 4]);
    float dot = sel ? fmaf(p.x, f.x, fmaf(p.y, f.y, fmaf(p.z, f.z, p.w * f.w))) : 0.f;   // phi(q) . phi of the folded pair
    dot = warp_sum(dot);
    const float den = warp_sum(w * (sum ? X.peer[k8].l[r] : lane == 17 ? X.lden[r] + dot : 1.f));
    const float wn = __shfl_sync(0xffffffffu, w, 16), wl = __shfl_sync(0xffffffffu, w, 17);
    float y[4][NC];                                    // (four sums again)
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int col = NC * lane + i;
      y[0][i] = wl * (sel ? fmaf(dot, win.v[col], X.lin[r][col]) : X.lin[r][col]);
      y[1][i] = wn * X.kv_new[1][col];
      y[2][i] = y[3][i] = 0.f;
    }
#pragma unroll
    for (int q0 = 0; q0 < 8; q0 += 4)
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int q = q0 + x;
        const float ws = __shfl_sync(0xffffffffu, w, q), wp = __shfl_sync(0xffffffffu, w, 8 + q);
        if (q >= K) continue;
#pragma unroll
        for (int i = 0; i < NC; i += 2) {
          const float2 o = *reinterpret_cast<const float2*>(&X.peer_o[q * per + warp][NC * lane + i]), v = *reinterpret_cast<const float2*>(&X.peer[q].v[NC * lane + i]);
          y[x][i] = fmaf(ws, o.x, y[x][i]); y[x][i + 1] = fmaf(ws, o.y, y[x][i + 1]);
          if (wp != 0.f) { y[x][i] = fmaf(wp, v.x, y[x][i]); y[x][i + 1] = fmaf(wp, v.y, y[x][i + 1]); }
        }
      }
#pragma unroll
    for (int i = 0; i < NC; ++i) y[0][i] = ((y[0][i] + y[1][i]) + (y[2][i] + y[3][i])) / den;
    if (ok)
#pragma unroll
      for (int i = 0; i < NC; i += 2) *reinterpret_cast<float2*>((float*)c.out + qofs + (size_t)r * d + NC * lane + i) = make_float2(y[0][i], y[0][i + 1]);
  }
  // ---- Eq. 13: this block's rows of H, added where they lie
  if (sel && ok) {
    const int j0 = rank * 128 / K, j1 = (rank + 1) * 128 / K;
#pragma unroll 1
    for (int i = tid; i < (j1 - j0) * d4; i += kStepThreads) {
      const int j = j0 + i / d4, c4 = i % d4 * 4;
      const float p = win.phi[j];
      const float4 v = *reinterpret_cast<const float4*>(&win.v[c4]);
      tc::red_add_v4(L.H + ((size_t)unit * 128 + j) * d + c4, make_float4(p * v.x, p * v.y, p * v.z, p * v.w));
    }
    if (tid >= j0 && tid < j1) atomicAdd(L.s + (size_t)unit * 128 + tid, win.phi[tid]);
    if (rank == 0 && warp == 7) {                      // lowest kept / highest folded score of this update
      const unsigned kept = __reduce_min_sync(0xffffffffu, min(k8 < K ? X.peer[k8].second : 0xffffffffu, k8 == wr_ ? 0xffffffffu : khi));
      if (lane == 0) {
        L.thr[(size_t)unit * 2 + 0] = __uint_as_float(kept);
        L.thr[(size_t)unit * 2 + 1] = __uint_as_float(whi);
      }
    }
    if (tid == 192 && low != ~0ull && (rank != wr_ || wrow >= cg)) scu[low_row < cg ? low_row : lam] = __uint_as_float((unsigned)(low >> 32));
  }
  // ---- the leaving pair takes the folded member's slot (none if it is folded itself), the new pair its place in the ring
  if (rank == mover && ok) {
    const bool moves = sel ? wrow < cg : c.mode == UPD_APPEND;
    if (tid < 2 * d4) {
      const int c4 = tid % d4 * 4;
      if (moves) *reinterpret_cast<float4*>((float*)(tid < d4 ? L.gk : L.gv) + gofs + (size_t)wrow * d + c4) = lev;
      *reinterpret_cast<float4*>((float*)(tid < d4 ? L.wk : L.wv) + wofs + (size_t)s_ev * d + c4) = *reinterpret_cast<const float4*>(&X.kv_new[tid < d4 ? 0 : 1][c4]);
    }
    if (tid == 128 && moves) {
      L.gpos[(size_t)unit * lam + wrow] = c.r_pos0;
      scu[wrow] = sel ? X.lev_score : CUDART_NAN_F;    // never scored while the cache still has room
    }
  }
  if (*abw != 0) {                                     // (a block did not answer: what is on its way here arrives first)
    __nanosleep(200000);
    if (tid == 0) atomicOr(L.status, 8);
  }
}

}  // namespace lola
