// The whole step of an fp32 layer - a run of prefill chunks, or one generation step of the shapes that k_unit_step does not
// serve (F other than 64, no window or no sparse cache, query restrictions, more than 8 query heads) - as ONE kernel: a cluster of K
// thread blocks carries one (batch row, KV head) unit through the run, all arithmetic in fp32 on the CUDA cores.
//
// What bounds it: latency.  A chunk of the tiny fp32 layer (64 tokens, 256 keys, d = 64) is 6 MFMA per unit; as a
// chain of four kernels with a block per 16 or 32 rows it took 167 us, nearly all of it launches, round trips to
// memory between dependent phases and a quadratic selection.  Here a unit's H, s, W and positions stay in shared
// memory for the whole run and the phases of a chunk are separated by cluster barriers:
//   A  every block, two groups of 256 threads side by side:
//        group 0: its share of E = sparse cache + leaving pairs: feature map (kept), Eq. 10 score, sent to all blocks of the cluster
//        group 1 (d = 128: and group 0 when it has scored): (prefill) its share of the queries: Eq. 14 against the H, s of the chunk's start
//   -- barrier: all scores are everywhere, nobody reads the old H or ring any more
//   B  every block for itself: the selection (Eq. 12); the feature rows of the folded pairs come from the blocks that
//      computed them, each block folds its D / K rows of H and s (Eq. 13) and sends them to the others
//   -- barrier: the folded pairs have been read, their slots may be overwritten
//   C  moves into the sparse cache and window roll, a warp per token
//   -- barrier; (generation step) Eq. 14 on the updated memories
// One group after the other a chunk took 27.0 us, side by side 22.2 (4 units of 192 pairs, 64 tokens, d = 64; 16 units of 364 pairs, two
// heads, 93.7 and 74.4): the two share the SM's path to shared memory, which the products keep busy.
// K is the largest of 8, 4, 2, 1 that lets every block have an SM of its own: more blocks only shorten the phases.
// The body of the chunk loop has to stay in the instruction cache: with everything unrolled (226 KB of code) a chunk
// took 33 us, three quarters of it instruction fetch.  Hence short rolled loops, no integer division inside them and
// one copy of each phase (the generation step takes the loop twice).
// Sums are taken in a fixed order, so a run of chunks and single calls give the same bits.
#pragma once
#include <cooperative_groups.h>

#include "lola_generic.cuh"
#include "lola_select.cuh"
#include "lola_tc.cuh"

namespace lola {

constexpr int kUnThreads = 512;   // two groups of 256: scoring and attention side by side, then both
constexpr int kUnGroup = 256;
constexpr int kUnSmem = 227 * 1024;
constexpr int kUnRows = 32;    // members of E per scoring tile: thread = 2 rows x 4 columns of a 32 x 64 product
constexpr int kUnQ = 8;        // query rows per batch (one per warp in the softmax)
constexpr int kUnKeys = 256;   // keys per tile
constexpr int kUnFold = 64;    // folded pairs per pass
constexpr int kUnSrcFloats = 56;

struct UnitLayout {            // shared memory of k_unit_run, offsets in floats
  int fp, dp;                  // F and D rounded up to a multiple of 4 (zero padding)
  int jn, jsh;                 // rows of H a block folds, and the power of two that covers them
  int phi_ld;
  int both;                    // group 0 attends, too, once it has scored
  int att0;                    // from the attention scratch of group 1 to that of group 0
  int W, H, s, phi, xs, den, vf, pf, q, pq, z, p, vptr, red, row, key, pos, cand, mark, fold, dst, sel, src, part, total;
};

// Does one group of threads have all entries of a block's rows of H?  The groups then take half of the folded pairs each.
LOLA_HD inline bool unit_fold_halves(int jn, int d) { return jn * (d / 4) <= kUnGroup; }

LOLA_HD inline UnitLayout unit_layout_of(const Layer& L, int K, int both) {
  auto imax = [](int a, int b) { return a > b ? a : b; };
  UnitLayout Y{};
  Y.both = both;
  const int d = L.d, nE = L.lam + L.cmax, rp = (nE + K - 1) / K;
  Y.fp = (L.F + 3) & ~3;
  Y.dp = (L.D + 3) & ~3;
  Y.jn = (L.D + K - 1) / K;
  while ((1 << Y.jsh) < Y.jn) ++Y.jsh;
  Y.phi_ld = Y.dp + 4;
  int o = 0;
  auto take = [&o](int n) { const int at = o; o += (n + 3) & ~3; return at; };
  Y.W = take(d * Y.fp);
  Y.H = take(Y.dp * d);
  Y.s = take(Y.dp);
  Y.phi = take((rp + kUnRows - 1) / kUnRows * kUnRows * Y.phi_ld);
  // the phases of a chunk take turns in the same space: first group 1's query batch beside group 0's scoring tile and then (both)
  // query batch
  const int phase0 = o;
  Y.q = take(kUnQ * d);
  Y.pq = take(Y.dp * kUnQ);
  Y.z = take(kUnQ * kUnKeys);              // (first the queries' u, 128 floats a row)
  Y.p = take(kUnKeys * kUnQ);
  Y.vptr = take(kUnKeys * 2);
  Y.row = take(kUnQ * 3);
  Y.red = Y.z;                             // (after the last key tile: over z and p)
  static_assert(kUnGroup / 32 * kUnQ * 64 <= kUnQ * kUnKeys + kUnKeys * kUnQ, "the key groups' sums do not fit");
  Y.att0 = o - phase0;
  int end = both ? o + Y.att0 : o;
  Y.xs = take(kUnRows * (d + 4));
  Y.den = take(kUnRows);
  end = imax(end, o);
  o = phase0;
  Y.vf = take(kUnFold * d);
  Y.pf = take(kUnFold * Y.jn);
  if (unit_fold_halves(Y.jn, d)) Y.part = take(kUnGroup * 4);
  end = imax(end, o);
  // the selection is over when the folded pairs come in; only its first value row is there beside it (the fold of one pair)
  o = Y.vf + d;
  Y.sel = take((int)(sizeof(SelectScratch) + 3) / 4);
  Y.cand = take(nE);
  Y.mark = take((nE + 3) / 4);
  o = imax(end, o);
  Y.key = take(nE);
  Y.pos = take(nE);
  Y.fold = take(L.cmax);
  Y.dst = take(L.cmax);
  Y.src = take(kUnSrcFloats);
  Y.total = o;
  return Y;
}

// rows: query rows of a unit in one chunk.  Both groups attend where a block has two batches of them or more, d = 128: with 128 registers
// a thread one group is slower at them than 256 threads with 255 were (4 units, 200 slots, two heads, chunks of 200: one each 295 us, both
// 226, 256 threads 289; where a block has one batch the kernel for both is 3% slower).
LOLA_HD inline UnitLayout unit_layout(const Layer& L, int K, int rows) {
  const UnitLayout Y = unit_layout_of(L, K, L.d == 128 && rows > K * kUnQ);
  return Y.total * 4 <= kUnSmem ? Y : unit_layout_of(L, K, 0);
}

// Where the rows of a unit lie during one chunk (shared memory; every pointer is the unit's own first row).
struct UnitSrc {
  const float *gk, *gv, *wk, *wv, *k, *v;
  int cg, r_ring, ring0;         // sparse-cache members; leaving pairs that lie in the ring, and the slot of the first
  int eta, kstep;                // slots of the ring; floats between two incoming tokens
  int att_g, att_wn, att_w0;     // keys the queries see: sparse cache, window (slot of its first)
  int taken;                     // query batches of this block taken so far (both groups attend)
  int tok_of[2][kUnQ], out_row[2][kUnQ];   // a group's query batch: tokens, rows of q / out (-1: none)
};
static_assert(sizeof(UnitSrc) <= kUnSrcFloats * 4, "UnitSrc does not fit");
// member e of E = sparse cache ++ leaving pairs: element offset from (k ? gk : gv) etc. resolved to the row itself
__device__ __forceinline__ void unit_member(const UnitSrc& U, int e, int d, const float*& kp, const float*& vp) {
  const int i = e - U.cg;
  if (i < 0) { kp = U.gk + (size_t)e * d; vp = U.gv + (size_t)e * d; }
  else if (i < U.r_ring) {
    int slot = U.ring0 + i;
    if (slot >= U.eta) slot -= U.eta;
    kp = U.wk + (size_t)slot * d; vp = U.wv + (size_t)slot * d;
  } else { kp = U.k + (size_t)(i - U.r_ring) * U.kstep; vp = U.v + (size_t)(i - U.r_ring) * U.kstep; }
}
__device__ __forceinline__ void unit_key(const UnitSrc& U, int i, int d, const float*& kp, const float*& vp) {
  if (i < U.att_g) { kp = U.gk + (size_t)i * d; vp = U.gv + (size_t)i * d; return; }
  i -= U.att_g;
  if (i < U.att_wn) {
    int slot = U.att_w0 + i;
    if (slot >= U.eta) slot -= U.eta;
    kp = U.wk + (size_t)slot * d; vp = U.wv + (size_t)slot * d;
  } else { kp = U.k + (size_t)(i - U.att_wn) * U.kstep; vp = U.v + (size_t)(i - U.att_wn) * U.kstep; }
}

// The feature map of R rows by one warp, side by side (a row alone is a chain of reductions, exponentials and
// divisions), N features of each sign per lane (F <= 32 N): u[r * u_ld + f] -> out[r * o_row + j * o_col], j over the D features;
// ds[r] = phi . ss.
template <int R, int N>
__device__ __noinline__ void unit_phi(const float* u, int u_ld, float* out, int o_row, int o_col, int F, int kind, const float* ss, float* ds_out) {
  const int lane = threadIdx.x & 31;
  float mx[R], mn[R], s1[R], s2[R], ds[R];
  float a[R][N];
#pragma unroll
  for (int r = 0; r < R; ++r) { mx[r] = -CUDART_INF_F; mn[r] = CUDART_INF_F; s1[r] = s2[r] = 1.f; ds[r] = 0.f; }
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool in = lane + 32 * i < F;
      a[r][i] = in ? u[r * u_ld + lane + 32 * i] : 0.f;
      if (in) { mx[r] = fmaxf(mx[r], a[r][i]); mn[r] = fminf(mn[r], a[r][i]); }
    }
  __syncwarp();                                        // (out may lie over u)
  if (kind == 1) {
#pragma unroll
    for (int r = 0; r < R; ++r) mx[r] = mn[r] = 0.f;
  } else {
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], o));
        mn[r] = fminf(mn[r], __shfl_xor_sync(0xffffffffu, mn[r], o));
      }
  }
  float p[R][N], q[R][N];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float t1 = 0.f, t2 = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      p[r][i] = q[r][i] = 0.f;
      if (lane + 32 * i < F) { p[r][i] = expf(a[r][i] - mx[r]); q[r][i] = expf(mn[r] - a[r][i]); }
      t1 += p[r][i];
      t2 += q[r][i];
    }
    if (kind != 1) { s1[r] = t1; s2[r] = t2; }
  }
  if (kind != 1) {
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        s1[r] += __shfl_xor_sync(0xffffffffu, s1[r], o);
        s2[r] += __shfl_xor_sync(0xffffffffu, s2[r], o);
      }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int f = lane + 32 * i;
      if (f < F) {
        const float x = p[r][i] / s1[r], y = q[r][i] / s2[r];
        out[r * o_row + f * o_col] = x;
        out[r * o_row + (F + f) * o_col] = y;
        ds[r] = fmaf(x, ss[f], fmaf(y, ss[F + f], ds[r]));
      }
    }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < R; ++r) ds[r] += __shfl_xor_sync(0xffffffffu, ds[r], o);
  if (lane == 0)
#pragma unroll
    for (int r = 0; r < R; ++r) ds_out[r] = ds[r];
}

// Eq. 14 for the query rows of one block of the cluster, in batches of kUnQ rows, by group 1 or by both groups (which take the
// batches as they get to them).  Key tile: four lanes a key; the values (thread = 4 columns x every 16th key) are requested before the
// softmax.  The linear term is the accumulator's first summand, with the weight of a key whose score is 0.
template <int DPL, bool BOTH>
__device__ __forceinline__ void unit_attend(const Layer& L, const Call& c, const UnitLayout& Y, float* sm, UnitSrc& U, int b, int h, int rank, int K, int grp) {
  constexpr int d = DPL * 32, NC = d / 64, KG = kUnGroup / 16;     // NC: 64-column blocks, KG: key groups
  const int tid = threadIdx.x & (kUnGroup - 1), warp = tid >> 5, lane = tid & 31;
  if (!BOTH) grp = 1;
  auto sync = [grp] { tc::named_bar_sync(1 + grp, kUnGroup); };
  const int nrows = L.g * c.nq, NK = c.att_g + c.att_wn + c.att_chunk, chunk0 = c.att_g + c.att_wn;
  const float* Hs = sm + Y.H;
  float* own = sm + (grp == 0 ? Y.att0 : 0);
  float *qs = own + Y.q, *pq = own + Y.pq, *zs = own + Y.z, *ps = own + Y.p, *red = own + Y.red, *rw = own + Y.row;
  const float** vptr = reinterpret_cast<const float**>(own + Y.vptr);
  int *tok_of = U.tok_of[grp], *out_row = U.out_row[grp];
  const int c4 = (tid & 15) * 4, kg = tid >> 4;
#pragma unroll 1
  for (int row0 = rank * kUnQ; BOTH || row0 < nrows; row0 += K * kUnQ) {
    if (BOTH && warp == 0) row0 = (rank + __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(&U.taken, 1) : 0, 0) * K) * kUnQ;
    if (tid < kUnQ) {
      const int row = row0 + tid, hl = row / c.nq, tok = row - hl * c.nq;
      tok_of[tid] = tok;
      out_row[tid] = row < nrows ? (b * c.nq + tok) * L.Hq + h * L.g + hl : -1;
    }
    sync();
    if (BOTH && out_row[0] < 0) break;
    if (tid < kUnQ * (d / 4)) {
      const int rr = tid / (d / 4), row = out_row[rr];
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row >= 0) x = *reinterpret_cast<const float4*>((const float*)c.q + (size_t)row * d + tid % (d / 4) * 4);
      *reinterpret_cast<float4*>(qs + tid * 4) = x;
    }
    sync();
    // u = q W: warp = row, 4 features per lane and pass; then the row's feature map, transposed into pq
    const bool two = Y.fp <= 64;                       // (half a warp has all features: the other half takes half of the inner dimension)
#pragma unroll 1
    for (int f = (two ? lane & 15 : lane) * 4; f < Y.fp; f += 128) {
      const int jb = two && lane >= 16 ? d / 2 : 0, jn = two ? d / 2 : d;
      const float *x = qs + warp * d + jb, *w = sm + Y.W + jb * Y.fp + f;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int j = 0; j < jn; ++j) {
        const float4 wv = *reinterpret_cast<const float4*>(w + j * Y.fp);
        const float xj = x[j];
        a.x = fmaf(xj, wv.x, a.x); a.y = fmaf(xj, wv.y, a.y); a.z = fmaf(xj, wv.z, a.z); a.w = fmaf(xj, wv.w, a.w);
      }
      if (two) {
        const unsigned m16 = (1u << min(16, Y.fp / 4)) - 1u, both = m16 | m16 << 16;
        a.x += __shfl_xor_sync(both, a.x, 16); a.y += __shfl_xor_sync(both, a.y, 16);
        a.z += __shfl_xor_sync(both, a.z, 16); a.w += __shfl_xor_sync(both, a.w, 16);
      }
      if (!two || lane < 16) *reinterpret_cast<float4*>(zs + warp * 128 + f) = a;
    }
    sync();
    if (two) unit_phi<1, 2>(zs + warp * 128, 128, pq + warp, 1, kUnQ, L.F, L.phi_kind, sm + Y.s, rw + 2 * kUnQ + warp);
    else unit_phi<1, 4>(zs + warp * 128, 128, pq + warp, 1, kUnQ, L.F, L.phi_kind, sm + Y.s, rw + 2 * kUnQ + warp);
    sync();
    float m = 0.f, l = (c.att_flags & 1) ? 0.f : rw[2 * kUnQ + warp];   // this warp's row: stabiliser max(0, max z), sum of the weights
    float acc[NC][kUnQ][4];
#pragma unroll
    for (int nc = 0; nc < NC; ++nc)
#pragma unroll
      for (int r = 0; r < kUnQ; ++r) acc[nc][r][0] = acc[nc][r][1] = acc[nc][r][2] = acc[nc][r][3] = 0.f;
    auto add = [&](int nc, const float4& v, const float* w8) {
      const float4 pa = *reinterpret_cast<const float4*>(w8), pb = *reinterpret_cast<const float4*>(w8 + 4);
      const float w[kUnQ] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
      for (int r = 0; r < kUnQ; ++r) {
        acc[nc][r][0] = fmaf(w[r], v.x, acc[nc][r][0]);
        acc[nc][r][1] = fmaf(w[r], v.y, acc[nc][r][1]);
        acc[nc][r][2] = fmaf(w[r], v.z, acc[nc][r][2]);
        acc[nc][r][3] = fmaf(w[r], v.w, acc[nc][r][3]);
      }
    };
    if (!(c.att_flags & 1)) {                          // (1: the queries do not see H, s)
#pragma unroll 2
      for (int j = kg; j < L.D; j += KG)
#pragma unroll
        for (int nc = 0; nc < NC; ++nc) add(nc, *reinterpret_cast<const float4*>(Hs + j * d + nc * 64 + c4), pq + j * kUnQ);
    }
#pragma unroll 1
    for (int kt = 0; kt < NK; kt += kUnKeys) {
      const int nk = min(kUnKeys, NK - kt);
      // q.k: four lanes per key, four keys per thread (two at a time where a thread holds 128 columns).  A lane takes every fourth 16 bytes of a key (a whole row per thread touches a
      // line per lane and load); the queries' pieces serve all its keys; the lanes' sums meet in a reduce-scatter, two queries a lane
      constexpr int NP = DPL == 4 ? 2 : 4;
      const int sub = tid & 3;
#pragma unroll 1
      for (int k0 = tid >> 2; k0 < kUnKeys; k0 += NP * (kUnGroup / 4)) {
        float z[NP][kUnQ];
        const float* kp[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const int kb = k0 + p * (kUnGroup / 4);
          const float *kk = qs, *vp = qs;              // (beyond the last key: masked)
          if (kb < nk) unit_key(U, kt + kb, d, kk, vp);
          kp[p] = kk + sub * 4;
          if (sub == 0) vptr[kb] = vp;
#pragma unroll
          for (int r = 0; r < kUnQ; ++r) z[p][r] = 0.f;
        }
#pragma unroll 1
        for (int j0 = 0; j0 < d; j0 += 64) {
          float4 kv[NP][4];
#pragma unroll
          for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int j = 0; j < 4; ++j) kv[p][j] = *reinterpret_cast<const float4*>(kp[p] + j0 + j * 16);
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < kUnQ; ++r) {
              const float4 qv = *reinterpret_cast<const float4*>(qs + r * d + j0 + j * 16 + sub * 4);
#pragma unroll
              for (int p = 0; p < NP; ++p)
                z[p][r] = fmaf(qv.w, kv[p][j].w, fmaf(qv.z, kv[p][j].z, fmaf(qv.y, kv[p][j].y, fmaf(qv.x, kv[p][j].x, z[p][r]))));
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const int kb = k0 + p * (kUnGroup / 4), ci = kt + kb - chunk0;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float keep = sub & 2 ? z[p][r + 4] : z[p][r], give = sub & 2 ? z[p][r] : z[p][r + 4];
            z[p][r] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
          }
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float keep = sub & 1 ? z[p][r + 2] : z[p][r], give = sub & 1 ? z[p][r] : z[p][r + 2];
            const float zz = keep + __shfl_xor_sync(0xffffffffu, give, 1);
            const int row = (sub & 2) * 2 + (sub & 1) * 2 + r;
            zs[row * kUnKeys + kb] = kb < nk && (ci < 0 || ci <= tok_of[row]) ? zz * L.scale : -CUDART_INF_F;
          }
        }
      }
      sync();
      float4 vv[8];                                    // the first half of the first column block's values, ahead of the softmax
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int key = kg + i * KG;
        vv[i] = key < nk ? *reinterpret_cast<const float4*>(vptr[key] + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      {
        float v[kUnKeys / 32], mt = m;
#pragma unroll
        for (int i = 0; i < kUnKeys / 32; ++i) { v[i] = zs[warp * kUnKeys + lane + 32 * i]; mt = fmaxf(mt, v[i]); }
        mt = warp_max(mt);
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < kUnKeys / 32; ++i) {
          v[i] = expf(v[i] - mt);                      // (masked: exp(-inf) = 0)
          sum += v[i];
          ps[(lane + 32 * i) * kUnQ + warp] = v[i];
        }
        const float alpha = expf(m - mt);
        l = l * alpha + warp_sum(sum);
        m = mt;
        if (lane == 0) rw[warp] = alpha;
      }
      sync();
#pragma unroll
      for (int r = 0; r < kUnQ; ++r) {
        const float alpha = rw[r];
#pragma unroll
        for (int nc = 0; nc < NC; ++nc) { acc[nc][r][0] *= alpha; acc[nc][r][1] *= alpha; acc[nc][r][2] *= alpha; acc[nc][r][3] *= alpha; }
      }
#pragma unroll
      for (int nc = 0; nc < NC; ++nc)
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          const int k0 = kg + half * 8 * KG;
          if (nc + half > 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              vv[i] = k0 + i * KG < nk ? *reinterpret_cast<const float4*>(vptr[k0 + i * KG] + nc * 64 + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          // (keys beyond the tile: values 0, weights 0 or left from an earlier tile)
#pragma unroll
          for (int i = 0; i < 8; ++i) add(nc, vv[i], ps + (k0 + i * KG) * kUnQ);
        }
      sync();
    }
    if (lane == 0) rw[kUnQ + warp] = l;
    // the 16 key groups meet: two inside a warp, then eight warps through shared memory
#pragma unroll
    for (int nc = 0; nc < NC; ++nc) {
#pragma unroll
      for (int r = 0; r < kUnQ; ++r) {
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[nc][r][x] += __shfl_xor_sync(0xffffffffu, acc[nc][r][x], 16);
        if (lane < 16)
          *reinterpret_cast<float4*>(red + (warp * kUnQ + r) * 64 + c4) = make_float4(acc[nc][r][0], acc[nc][r][1], acc[nc][r][2], acc[nc][r][3]);
      }
      sync();
#pragma unroll 1
      for (int i = tid; i < kUnQ * 64; i += kUnGroup) {
        const int r = i >> 6, cc = i & 63;
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < kUnGroup / 32; ++w) a += red[(w * kUnQ + r) * 64 + cc];
        if (out_row[r] >= 0) ((float*)c.out)[(size_t)out_row[r] * d + nc * 64 + cc] = a / rw[kUnQ + r];
      }
      sync();
    }
  }
}

// BOTH: group 0 attends, too
template <int DPL, bool BOTH>
__global__ void __launch_bounds__(kUnThreads, 1) k_unit_run(Layer L, Call c, int n_chunks, int decode, UnitLayout Y) {
  namespace co = cooperative_groups;
  constexpr int d = DPL * 32, d4 = d / 4;
  extern __shared__ __align__(16) float sm[];
  co::cluster_group cl = co::this_cluster();
  const int K = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int unit = blockIdx.x / K, b = unit / L.Hkv, h = unit % L.Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = tid >> 8, gt = tid & (kUnGroup - 1), tx = gt & 15, ty = gt >> 4;
  auto gsync = [] { tc::named_bar_sync(1, kUnGroup); };   // the scoring group
  float *Ws = sm + Y.W, *Hs = sm + Y.H, *ss = sm + Y.s, *phi = sm + Y.phi, *xs = sm + Y.xs, *den = sm + Y.den, *vf = sm + Y.vf, *pf = sm + Y.pf;
  unsigned* key = reinterpret_cast<unsigned*>(sm + Y.key);
  int *pos = reinterpret_cast<int*>(sm + Y.pos), *cand = reinterpret_cast<int*>(sm + Y.cand), *fold = reinterpret_cast<int*>(sm + Y.fold),
      *dst = reinterpret_cast<int*>(sm + Y.dst);
  unsigned char* mark = reinterpret_cast<unsigned char*>(sm + Y.mark);
  SelectScratch& S = *reinterpret_cast<SelectScratch*>(sm + Y.sel);
  UnitSrc& U = *reinterpret_cast<UnitSrc*>(sm + Y.src);

  if (tid == 0) tc::grid_dep_launch_dependents();
#pragma unroll 1
  for (int j = warp; j < d; j += kUnThreads / 32)
    for (int f = lane; f < Y.fp; f += 32) Ws[j * Y.fp + f] = f < L.F ? ((const float*)L.W)[((size_t)h * d + j) * L.F + f] : 0.f;
  tc::grid_dep_wait();                                // everything before this kernel in the stream is complete
  if (state_failed(L)) return;                        // an earlier kernel failed: do nothing (the same for all blocks)
  const float* Hg = L.H + (size_t)unit * L.D * d;
#pragma unroll 4
  for (int i = tid; i < Y.dp * d4; i += kUnThreads)
    *reinterpret_cast<float4*>(Hs + i * 4) = i < L.D * d4 ? *reinterpret_cast<const float4*>(Hg + (size_t)i * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid < Y.dp) ss[tid] = tid < L.D ? L.s[(size_t)unit * L.D + tid] : 0.f;
  for (int i = tid; i < L.lam; i += kUnThreads) pos[i] = L.gpos[(size_t)unit * L.lam + i];
  const int j0 = min(L.D, rank * Y.jn), jn = min(Y.jn, L.D - j0);   // this block's rows of H
  float* scu = L.score + (size_t)unit * (L.lam + L.cmax);
  int n_seen = c.n_seen;
  const int n = c.n;
  const size_t qstep = (size_t)L.B * n * L.Hq * d, kstep = (size_t)L.B * n * L.Hkv * d;
  bool folded = false;

#pragma unroll 1
  for (int it = 0; it < (decode ? 2 : n_chunks); ++it) {
    // (the generation step: round 0 updates, round 1 attends)
    int nF = 0, rp = 1;
    bool scored = false;
    if (!decode || it == 0) {
      plan_call(L, c, n_seen, n, decode != 0);
      scored = c.mode == UPD_SELECT;
      nF = scored ? c.count_g + c.r - L.lam : c.mode == UPD_FOLD_ALL ? c.r : 0;
      rp = (c.count_g + c.r + K - 1) / K;
    }
    const int cg = c.count_g, nE = cg + c.r, e0 = rank * rp, ne = nF > 0 ? max(0, min(rp, nE - e0)) : 0;
    if (tid == 0) {
      U.gk = (const float*)L.gk + (size_t)unit * L.lam * d;
      U.gv = (const float*)L.gv + (size_t)unit * L.lam * d;
      U.wk = (const float*)L.wk + (size_t)unit * L.eta * d;
      U.wv = (const float*)L.wv + (size_t)unit * L.eta * d;
      U.k = (const float*)c.k + ((size_t)b * n * L.Hkv + h) * d;
      U.v = (const float*)c.v + ((size_t)b * n * L.Hkv + h) * d;
      U.cg = cg;
      U.r_ring = min(c.r, n_seen - c.r_pos0);
      U.ring0 = L.eta > 0 ? c.r_pos0 % L.eta : 0;
      U.eta = L.eta;
      U.kstep = L.Hkv * d;
      U.att_g = c.att_g;
      U.att_wn = c.att_wn;
      U.att_w0 = L.eta > 0 ? c.att_w0 % L.eta : 0;
      if (BOTH) U.taken = 0;
    }
    __syncthreads();
    // ---- A: feature rows and scores of this block's members of E
#pragma unroll 1
    for (int t0 = 0; t0 < (grp == 0 ? ne : 0); t0 += kUnRows) {
#pragma unroll 2
      for (int i = gt; i < kUnRows * d4; i += kUnGroup) {
        const int row = i / d4, c4 = i % d4;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t0 + row < ne) {
          const float *kp, *vp;
          unit_member(U, e0 + t0 + row, d, kp, vp);
          x = *reinterpret_cast<const float4*>(kp + c4 * 4);
        }
        *reinterpret_cast<float4*>(xs + row * (d + 4) + c4 * 4) = x;
      }
      gsync();
      float* prow = phi + (size_t)(t0 + 2 * ty) * Y.phi_ld;         // this thread's two feature rows
      // a 2 x 4 tile of x m per thread: x rows in shared memory (ldx floats apart), m [k][ldm]
      auto tile = [&](const float* x, int ldx, const float* m, int ldm, int kk, float (&a)[2][4]) {
#pragma unroll 4
        for (int k = 0; k < kk; k += 4) {
          const float4 x0 = *reinterpret_cast<const float4*>(x + k), x1 = *reinterpret_cast<const float4*>(x + ldx + k);
          const float xa[4] = {x0.x, x0.y, x0.z, x0.w}, xb[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 w = *reinterpret_cast<const float4*>(m + (k + q) * ldm);
            a[0][0] = fmaf(xa[q], w.x, a[0][0]); a[0][1] = fmaf(xa[q], w.y, a[0][1]); a[0][2] = fmaf(xa[q], w.z, a[0][2]); a[0][3] = fmaf(xa[q], w.w, a[0][3]);
            a[1][0] = fmaf(xb[q], w.x, a[1][0]); a[1][1] = fmaf(xb[q], w.y, a[1][1]); a[1][2] = fmaf(xb[q], w.z, a[1][2]); a[1][3] = fmaf(xb[q], w.w, a[1][3]);
          }
        }
      };
#pragma unroll 1
      for (int f = tx * 4; f < Y.fp; f += 64) {
        float a[2][4] = {};
        tile(xs + 2 * ty * (d + 4), d + 4, Ws + f, Y.fp, d, a);
        *reinterpret_cast<float4*>(prow + f) = make_float4(a[0][0], a[0][1], a[0][2], a[0][3]);
        *reinterpret_cast<float4*>(prow + Y.phi_ld + f) = make_float4(a[1][0], a[1][1], a[1][2], a[1][3]);
      }
      float4 val[2][d / 64];                           // the values of this thread's rows, on their way meanwhile
#pragma unroll
      for (int rr = 0; rr < 2; ++rr)
        if (scored && t0 + 2 * ty + rr < ne) {
          const float *kp, *vp;
          unit_member(U, e0 + t0 + 2 * ty + rr, d, kp, vp);
#pragma unroll
          for (int q = 0; q < d / 64; ++q) val[rr][q] = *reinterpret_cast<const float4*>(vp + q * 64 + tx * 4);
        }
      gsync();
      {
        float* f = phi + (size_t)(t0 + warp * 4) * Y.phi_ld;
        if (L.F <= 64) unit_phi<4, 2>(f, Y.phi_ld, f, Y.phi_ld, 1, L.F, L.phi_kind, ss, den + warp * 4);
        else unit_phi<4, 4>(f, Y.phi_ld, f, Y.phi_ld, 1, L.F, L.phi_kind, ss, den + warp * 4);
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (lane < Y.dp - L.D) f[r * Y.phi_ld + L.D + lane] = 0.f;
      }
      gsync();
      if (scored) {
        float err[2] = {0.f, 0.f};
#pragma unroll
        for (int cb = 0; cb < d / 64; ++cb) {
          float a[2][4] = {};
          tile(prow, Y.phi_ld, Hs + cb * 64 + tx * 4, d, Y.dp, a);
#pragma unroll
          for (int rr = 0; rr < 2; ++rr) {
            if (t0 + 2 * ty + rr >= ne) continue;
            const float4 v = val[rr][cb];
            const float dn = den[2 * ty + rr], inv = dn > 0.f ? 1.0f / dn : 0.f;
            const float x0 = fmaf(a[rr][0], inv, -v.x), x1 = fmaf(a[rr][1], inv, -v.y), x2 = fmaf(a[rr][2], inv, -v.z), x3 = fmaf(a[rr][3], inv, -v.w);
            err[rr] = fmaf(x0, x0, fmaf(x1, x1, fmaf(x2, x2, fmaf(x3, x3, err[rr]))));
          }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
          for (int rr = 0; rr < 2; ++rr) err[rr] += __shfl_xor_sync(0xffffffffu, err[rr], o);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          const int m = e0 + t0 + 2 * ty + rr;
          if (t0 + 2 * ty + rr < ne) {
            const float sc = sqrtf(err[rr]);
            if (tx < K) cl.map_shared_rank(key, tx)[m] = __float_as_uint(sc);
            if (tx == 8) scu[m < cg ? m : L.lam + (m - cg)] = sc;
          }
        }
      }
      gsync();
    }
    if ((BOTH || grp == 1) && c.out && (!decode || it == 1)) unit_attend<DPL, BOTH>(L, c, Y, sm, U, b, h, rank, K, grp);
    if (decode && it == 1) break;
    cl.sync();
    // ---- B: which pairs fold, which leaving pairs stay
    // One leaving pair, one fold (a generation step on full caches): the lowest score is all there is to find, and every
    // block folds that pair into its whole copy of H: no lists, and no exchange of rows of H (F = 32, 4 units: 23.6 us a step, with lists
    // 26.5; 80 units 47.5 and 50.6)
    const bool one = scored && nF == 1 && c.r == 1;
    if (one) {
      if (tid == 0) pos[cg] = c.r_pos0;
      __syncthreads();
      unsigned long long best = ~0ull;
      unsigned second = 0xffffffffu;                   // this thread's lowest score but that
      int be = 0;
      for (int e = tid; e < nE; e += kUnThreads) {
        const unsigned long long k = ((unsigned long long)key[e] << 32) | (unsigned)(0x7fffffff - pos[e]);   // (ties: the younger pair)
        second = min(second, (unsigned)(max(k, best) >> 32));
        if (k < best) { best = k; be = e; }
      }
      const unsigned hi = (unsigned)(best >> 32), whi = __reduce_min_sync(0xffffffffu, hi);
      const unsigned lo = hi == whi ? (unsigned)best : 0xffffffffu, wlo = __reduce_min_sync(0xffffffffu, lo);
      const bool mine = hi == whi && (unsigned)best == wlo;
      const unsigned w2 = __reduce_min_sync(0xffffffffu, mine ? second : hi);
      if (mine) { S.lo[warp] = whi; S.hi[warp] = wlo; S.scan[warp] = w2; S.hist[warp] = (unsigned)be; }
      __syncthreads();
      int bw = 0;
      unsigned keep = S.scan[0];
      for (int w = 1; w < kUnThreads / 32; ++w) {
        const bool less = S.lo[w] < S.lo[bw] || (S.lo[w] == S.lo[bw] && S.hi[w] < S.hi[bw]);
        keep = min(keep, min(S.scan[w], less ? S.lo[bw] : S.lo[w]));
        if (less) bw = w;
      }
      const int e = (int)S.hist[bw], owner = e / rp;
      const float* prow = cl.map_shared_rank(phi, owner) + (size_t)(e - owner * rp) * Y.phi_ld;
      for (int j = tid; j < L.D; j += kUnThreads) pf[j] = prow[j];
      if (tid < d4) {
        const float *kp, *vp;
        unit_member(U, e, d, kp, vp);
        *reinterpret_cast<float4*>(vf + tid * 4) = *reinterpret_cast<const float4*>(vp + tid * 4);
      }
      if (tid == 0) {
        dst[0] = e < cg ? e : -1;
        if (rank == 0) {
          L.thr[(size_t)unit * 2 + 0] = __uint_as_float(keep);
          L.thr[(size_t)unit * 2 + 1] = __uint_as_float(S.lo[bw]);
        }
      }
      __syncthreads();
      for (int i = tid; i < L.D * d4; i += kUnThreads) {
        const float p = pf[i / d4];
        const float4 v = *reinterpret_cast<const float4*>(vf + i % d4 * 4);
        float4* hp = reinterpret_cast<float4*>(Hs + i * 4);
        float4 hv = *hp;
        hv.x += __fmul_rn(p, v.x); hv.y += __fmul_rn(p, v.y); hv.z += __fmul_rn(p, v.z); hv.w += __fmul_rn(p, v.w);
        *hp = hv;
      }
      for (int j = tid; j < L.D; j += kUnThreads) ss[j] += pf[j];
      folded = true;
      __syncthreads();
    } else if (scored) {
      for (int i = tid; i < c.r; i += kUnThreads) pos[cg + i] = c.r_pos0 + i;
      __syncthreads();
      auto pos_of = [&](int e) { return pos[e]; };
      auto put = [&](int i, int to) { dst[i] = to; };
      if (nE > 32 * kUnGroup) select_lists<kUnThreads>(key, pos_of, cand, mark, nE, nF, cg, fold, S, tid, [] { __syncthreads(); }, put, [] {});
      else if (grp == 0) select_lists<kUnGroup>(key, pos_of, cand, mark, nE, nF, cg, fold, S, tid, gsync, put, [] {});
      if (rank == 0 && tid == 0) {                     // (what is gathered next lies over the selection's scratch)
        L.thr[(size_t)unit * 2 + 0] = __uint_as_float(S.min_keep);
        L.thr[(size_t)unit * 2 + 1] = __uint_as_float(S.max_fold);
      }
      __syncthreads();
    } else {
      for (int i = tid; i < c.r; i += kUnThreads) { dst[i] = c.mode == UPD_APPEND ? cg + i : -1; if (nF > 0) fold[i] = cg + i; }
      __syncthreads();
    }
#pragma unroll 1
    for (int f0 = 0; f0 < nF && !one; f0 += kUnFold) {
      // the folded pairs' values and this block's part of their feature rows, four requests of each kind in flight
      const int nb = min(kUnFold, nF - f0);
#pragma unroll 1
      for (int base = tid; base < nb * d4; base += 4 * kUnThreads) {
        float4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = base + q * kUnThreads;
          if (i < nb * d4) {
            const float *kp, *vp;
            unit_member(U, fold[f0 + i / d4], d, kp, vp);
            x[q] = *reinterpret_cast<const float4*>(vp + i % d4 * 4);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (base + q * kUnThreads < nb * d4) *reinterpret_cast<float4*>(vf + (base + q * kUnThreads) * 4) = x[q];
      }
      const int jj = tid & ((1 << Y.jsh) - 1), rstep = kUnThreads >> Y.jsh;
#pragma unroll 1
      for (int row = tid >> Y.jsh; row < nb; row += 4 * rstep) {
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (row + q * rstep < nb && jj < jn) {
            const int e = fold[f0 + row + q * rstep], owner = e / rp;
            x[q] = cl.map_shared_rank(phi, owner)[(size_t)(e - owner * rp) * Y.phi_ld + j0 + jj];
          }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (row + q * rstep < nb && jj < jn) pf[(row + q * rstep) * Y.jn + jj] = x[q];
      }
      __syncthreads();
      const bool halves = unit_fold_halves(Y.jn, d);   // (jn <= Y.jn)
      const int fb = halves && grp == 1 ? nb / 2 : 0, fe = halves && grp == 0 ? nb / 2 : nb;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
      for (int i = halves ? gt : tid; i < jn * d4; i += kUnThreads) {
        const int j = i / d4, c4 = i % d4;
        a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int f = fb; f < fe; ++f) {
          const float p = pf[f * Y.jn + j];
          const float4 v = *reinterpret_cast<const float4*>(vf + f * d + c4 * 4);
          a.x = fmaf(p, v.x, a.x); a.y = fmaf(p, v.y, a.y); a.z = fmaf(p, v.z, a.z); a.w = fmaf(p, v.w, a.w);
        }
        if (halves) break;
        float4* hp = reinterpret_cast<float4*>(Hs + (size_t)(j0 + j) * d + c4 * 4);
        float4 hv = *hp;
        hv.x += a.x; hv.y += a.y; hv.z += a.z; hv.w += a.w;
        *hp = hv;
      }
      if (halves && grp == 1) *reinterpret_cast<float4*>(sm + Y.part + gt * 4) = a;
      if (halves) __syncthreads();
      if (halves && grp == 0 && gt < jn * d4) {
        const float4 o = *reinterpret_cast<const float4*>(sm + Y.part + gt * 4);
        float4* hp = reinterpret_cast<float4*>(Hs + (size_t)j0 * d + gt * 4);
        float4 hv = *hp;
        hv.x += a.x + o.x; hv.y += a.y + o.y; hv.z += a.z + o.z; hv.w += a.w + o.w;
        *hp = hv;
      }
      if (tid < jn) {
        float a = 0.f;
#pragma unroll 4
        for (int f = 0; f < nb; ++f) a += pf[f * Y.jn + tid];
        ss[j0 + tid] += a;
      }
      __syncthreads();
    }
    if (nF > 0 && !one) {
      folded = true;
#pragma unroll 1
      for (int r = 1 + grp; r < K; r += 2) {                          // the folded rows of H, s to the other blocks
        const int to = (rank + r) & (K - 1);
        float* Hr = cl.map_shared_rank(Hs, to);
        for (int i = gt; i < jn * d4; i += kUnGroup)
          *reinterpret_cast<float4*>(Hr + (size_t)j0 * d + i * 4) = *reinterpret_cast<const float4*>(Hs + (size_t)j0 * d + i * 4);
        if (gt < jn) cl.map_shared_rank(ss, to)[j0 + gt] = ss[j0 + gt];
      }
      cl.sync();
    }
    // ---- C: a warp per incoming token: the pair whose ring slot it takes (or, without one, the token itself) first
    // moves into the sparse cache if it stays
    const int new0 = L.eta > 0 ? n_seen % L.eta : 0;
#pragma unroll 1
    for (int ci = rank * (kUnThreads / 32) + warp; ci < n; ci += K * (kUnThreads / 32)) {
      const int i = n_seen + ci - L.eta - c.r_pos0;
      const bool moves = i >= 0 && i < c.r && dst[i] >= 0, enters = ci >= n - L.eta;   // the window keeps the last eta positions
      const float *kp = nullptr, *vp = nullptr;
      if (moves) unit_member(U, cg + i, d, kp, vp);
      const size_t o = moves ? ((size_t)unit * L.lam + dst[i]) * d : 0;
      const size_t w = enters ? ((size_t)unit * L.eta + (L.eta == n ? (new0 + ci >= L.eta ? new0 + ci - L.eta : new0 + ci) : (n_seen + ci) % L.eta)) * d : 0;
      if (lane < d4) {
        float4 k0, v0, k1, v1;
        if (moves) { k0 = *reinterpret_cast<const float4*>(kp + lane * 4); v0 = *reinterpret_cast<const float4*>(vp + lane * 4); }
        if (enters) { k1 = *reinterpret_cast<const float4*>(U.k + (size_t)ci * U.kstep + lane * 4); v1 = *reinterpret_cast<const float4*>(U.v + (size_t)ci * U.kstep + lane * 4); }
        if (moves) { *reinterpret_cast<float4*>((float*)L.gk + o + lane * 4) = k0; *reinterpret_cast<float4*>((float*)L.gv + o + lane * 4) = v0; }
        if (enters) { *reinterpret_cast<float4*>((float*)L.wk + w + lane * 4) = k1; *reinterpret_cast<float4*>((float*)L.wv + w + lane * 4) = v1; }
      }
      if (moves && lane == 0) {
        L.gpos[(size_t)unit * L.lam + dst[i]] = c.r_pos0 + i;
        scu[dst[i]] = scored ? __uint_as_float(key[cg + i]) : CUDART_NAN_F;
      }
    }
    for (int i = tid; i < c.r; i += kUnThreads)
      if (dst[i] >= 0) pos[dst[i]] = c.r_pos0 + i;
    cl.sync();
    if (!decode) {
      n_seen += n;
      c.q = c.q ? (const float*)c.q + qstep : nullptr;
      c.out = c.out ? (float*)c.out + qstep : nullptr;
      c.k = (const float*)c.k + kstep;
      c.v = (const float*)c.v + kstep;
    }
  }
  if (folded) {
    for (int i = tid; i < jn * d4; i += kUnThreads)
      *reinterpret_cast<float4*>(L.H + ((size_t)unit * L.D + j0) * d + (size_t)i * 4) = *reinterpret_cast<const float4*>(Hs + (size_t)j0 * d + i * 4);
    for (int j = tid; j < jn; j += kUnThreads) L.s[(size_t)unit * L.D + j0 + j] = ss[j0 + j];
  }
}

}  // namespace lola
