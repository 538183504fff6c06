// Eq. 12: exact top-lambda of the eligible set E by (score descending, older pair first) and the work lists of the
// update, by one block of NT threads with everything in shared memory.
//
// What bounds it: barriers and shared-memory latency, not work (|E| is about a thousand), so the pairs to fold (the
// nF = |E| - lambda lowest) are found with as few block-wide steps as possible: minimum and maximum of the score
// bits (scores are norms >= 0, their bit patterns order like unsigned integers), ONE histogram over 256 equal ranges
// of the bits, which every warp scans for itself, and then the handful of pairs in the range that holds the nF-th
// lowest are ranked among themselves by (score, age).  The ranges span from the minimum to an upper bound of the nF-th
// lowest: the largest of at least nF group minima (with the maximum instead, outliers left over 100 pairs in that
// range, 3 us).  Positions only matter for equal scores and are looked up then (fetched ahead for everyone they made
// the step 1 us longer).
// Many equal scores (degenerate inputs) only make that last step longer: it is quadratic in the pairs of the range, with
// the positions in shared memory, 256 at a time.
#pragma once
#include <cuda_runtime.h>

namespace lola {

constexpr int kSelBins = 256;
constexpr int kSelFew = 64;        // candidates that every warp ranks for itself

struct SelectScratch {
  alignas(16) unsigned hist[kSelBins];
  unsigned lo[32], hi[32];         // per-warp minimum and maximum
  unsigned scan[32];               // per-warp counts of the compaction
  alignas(16) unsigned cand_key[kSelFew];
  int cand_e[kSelFew];
  unsigned min_keep, max_fold;
  int n_cand;
};

// key[nE]: score bits, 16-byte aligned and readable up to a multiple of four; pos_of(e): token position; cand[nE], mark[nE]:
// scratch.  fold_e (nF entries): the pairs to fold as indices into E, ascending (so the slots that become free come first).
// put_dst(i, slot): called once per leaving pair i (E index cg + i) with the sparse-cache slot it takes, or -1 if it folds: freed
// slots in ascending order, then the slots from cg on.  1 <= nF < nE <= 32 NT.  Called by NT threads (tid 0 .. NT - 1, whole warps)
// with a barrier over them.  listed(): called by every thread once fold_e is complete; what put_dst wrote is complete behind the
// caller's next barrier.
//
// A thread owns the same contiguous run of E (groups of four) in every step, and what it finds out about its pairs stays in a mask
// in its registers.  No step has a chain of data-dependent branches: places in lists come from ballots, and every warp ranks
// the candidates for itself.  832 of 896 pairs, 256 threads: 8950 cycles with marks in shared memory, a serial ranking by the
// candidates' owners and a pass over E per step; 5200 now (512 threads 8900 and 6250).  A run of chunks of 8 units with 512 slots
// (d = 64) went from 15.3 to 13.9 us a chunk with it.
template <int NT, class Idx, class Pos, class Sync, class Put, class Listed>
__device__ __forceinline__ void select_lists(const unsigned* key, Pos pos_of, Idx* cand, unsigned char* mark, int nE, int nF, int cg,
                                             Idx* fold_e, SelectScratch& S, int tid, Sync sync, Put put_dst, Listed listed) {
  const int warp = tid >> 5, lane = tid & 31;
  constexpr int NW = NT / 32;
  static_assert(NT >= kSelBins, "a window of positions is loaded by one thread each");
  const int run = (nE + 4 * NT - 1) / (4 * NT) * 4, e0 = tid * run;
  const unsigned below_me = (1u << lane) - 1u;
  auto each4 = [&](auto f) {                                       // f(i, keys of this thread's pairs e0 + i .. + 3, how many of them exist), i = 0, 4, ..
#pragma unroll 1
    for (int i = 0; i < run; i += 4) {
      const int n = max(0, min(4, nE - e0 - i));
      uint4 q = make_uint4(0u, 0u, 0u, 0u);
      if (n > 0) q = *reinterpret_cast<const uint4*>(key + e0 + i);
      const unsigned k[4] = {q.x, q.y, q.z, q.w};
      f(i, k, n);
    }
  };
  if (tid < kSelBins) S.hist[tid] = 0;
  if (tid < kSelFew) S.cand_key[tid] = 0xffffffffu;
  if (tid == 0) { S.min_keep = 0xffffffffu; S.n_cand = 0; }
  unsigned mn = 0xffffffffu, mx = 0u;
  each4([&](int, const unsigned (&k)[4], int n) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (x < n) { mn = min(mn, k[x]); mx = max(mx, k[x]); }
  });
  {
    // groups of o threads, at least nF of them with pairs: the largest of their minima is no smaller than the nF-th lowest
    const int nt = (nE + run - 1) / run;
    unsigned gm = mn;
    int o = 1;
    for (; o < 32 && nt / (2 * o) >= nF; o <<= 1) gm = min(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if (nt >= nF) mx = (tid & -o) < nt ? gm : 0u;
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) { S.lo[warp] = mn; S.hi[warp] = mx; }
  sync();
  mn = __reduce_min_sync(0xffffffffu, S.lo[lane & (NW - 1)]);
  mx = __reduce_max_sync(0xffffffffu, S.hi[lane & (NW - 1)]);
  // range of a score: the upper half of a product (monotonic, whatever it rounds).  A pair's place among those of its range is
  // kept: should it be the range that matters, that is its place in the list of candidates
  const unsigned scale = (unsigned)fminf(4294967040.f, 1099511627776.f / ((float)(mx - mn) + 1.0f));
  auto bin_of = [&](unsigned k) { return k <= mx ? min((int)__umulhi(k - mn, scale), kSelBins - 1) : kSelBins; };
  each4([&](int i, const unsigned (&k)[4], int n) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (x < n && k[x] <= mx) cand[e0 + i + x] = (Idx)atomicAdd(&S.hist[bin_of(k[x])], 1u);
  });
  sync();
  // the range that holds the nF-th lowest: every warp scans all of them, eight per lane, and counts those that end before it
  int tbin, below, nc;
  {
    constexpr int PL = kSelBins / 32;
    unsigned cnt[PL], tot = 0;
#pragma unroll
    for (int i = 0; i < PL; i += 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(&S.hist[lane * PL + i]);
      cnt[i] = q.x; cnt[i + 1] = q.y; cnt[i + 2] = q.z; cnt[i + 3] = q.w;
      tot += q.x + q.y + q.z + q.w;
    }
    unsigned incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const unsigned v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
    unsigned sum = incl - tot, bins = 0, low = 0, up = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < PL; ++i) {
      sum += cnt[i];
      if (sum < (unsigned)nF) { ++bins; low = sum; } else up = min(up, sum);
    }
    tbin = (int)__reduce_add_sync(0xffffffffu, bins);
    below = (int)__reduce_max_sync(0xffffffffu, low);
    nc = (int)__reduce_min_sync(0xffffffffu, up) - below;
  }
  unsigned fm = 0, cm = 0, lk = 0xffffffffu;                       // this thread's folded pairs, candidates; lowest score above the range
  each4([&](int i, const unsigned (&k)[4], int n) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (x < n) {
        const int bin = bin_of(k[x]);
        fm |= bin < tbin ? 1u << (i + x) : 0u;
        cm |= bin == tbin ? 1u << (i + x) : 0u;
        lk = bin > tbin ? min(lk, k[x]) : lk;
      }
  });
#pragma unroll 1
  for (unsigned m = nc <= kSelFew ? cm : 0u; m; m &= m - 1) {
    const int e = e0 + __ffs(m) - 1, at = cand[e];
    S.cand_key[at] = key[e];
    S.cand_e[at] = e;
  }
  lk = __reduce_min_sync(0xffffffffu, lk);
  if (lane == 0) atomicMin(&S.min_keep, lk);
  sync();
  const int need = nF - below;                                     // `need` of the nc candidates fold: the lowest, the younger first
  auto settle = [&](int rank, unsigned k) {                        // (every rank is taken once)
    if (rank == need - 1) S.max_fold = k;
    else if (rank == need) atomicMin(&S.min_keep, k);
  };
  if (nc <= kSelFew) {
    unsigned long long fold = 0;
#pragma unroll 1
    for (int j0 = 0; j0 < nc; j0 += 32) {                          // a lane per candidate
      const unsigned ke = S.cand_key[j0 + lane];
      int rank = 0, same = 0;
#pragma unroll 1
      for (int j = 0; j < nc; j += 16)                             // (places without a candidate hold the largest key)
#pragma unroll
        for (int x = 0; x < 16; x += 4) {
          const uint4 q = *reinterpret_cast<const uint4*>(&S.cand_key[j + x]);
          rank += (q.x < ke) + (q.y < ke) + (q.z < ke) + (q.w < ke);
          same += (q.x == ke) + (q.y == ke) + (q.z == ke) + (q.w == ke);
        }
      const bool in = j0 + lane < nc;
      // Equal scores: a lane per candidate fetches its position.  (Fetched where it is compared, one after the other, the selections of
      // a prompt that repeats itself took up to 9 us longer: 32 units, d = 64, 960 slots, chunks of 128 40.7 us a chunk, now 30.4)
      if (__any_sync(0xffffffffu, in && same > 1)) {
        const int p0 = pos_of(S.cand_e[min(lane, nc - 1)]), p1 = nc > 32 ? pos_of(S.cand_e[min(32 + lane, nc - 1)]) : 0, pe = j0 ? p1 : p0;
#pragma unroll 1
        for (int j = 0; j < nc; ++j) {
          const int pj = __shfl_sync(0xffffffffu, j < 32 ? p0 : p1, j & 31);
          rank += S.cand_key[j] == ke && pj > pe ? 1 : 0;
        }
      }
      if (warp == 0 && in) settle(rank, ke);
      fold |= (unsigned long long)__ballot_sync(0xffffffffu, in && rank < need) << j0;
    }
#pragma unroll 1
    for (unsigned m = cm; m; m &= m - 1) { const int i = __ffs(m) - 1; fm |= (unsigned)(fold >> cand[e0 + i] & 1u) << i; }
  } else {
    int* wpos = reinterpret_cast<int*>(S.hist);                    // (the histogram and the places have been read)
    for (unsigned m = cm; m; m &= m - 1) cand[atomicAdd(&S.n_cand, 1)] = (Idx)(e0 + __ffs(m) - 1);
    sync();
    for (int i0 = 0; i0 < nc; i0 += NT) {
      const int i = i0 + tid, e = i < nc ? (int)cand[i] : 0, pe = i < nc ? pos_of(e) : 0;
      const unsigned ke = key[e];
      int rank = 0;
      for (int w0 = 0; w0 < nc; w0 += kSelBins) {
        const int nw = min(kSelBins, nc - w0);
        sync();
        if (tid < nw) wpos[tid] = pos_of(cand[w0 + tid]);
        sync();
        for (int j = 0; j < nw; ++j) {
          const unsigned kf = key[cand[w0 + j]];
          rank += (kf < ke || (kf == ke && wpos[j] > pe)) ? 1 : 0;
        }
      }
      if (i < nc) { mark[e] = rank < need ? 1 : 0; settle(rank, ke); }
    }
    sync();
    for (unsigned m = cm; m; m &= m - 1) { const int i = __ffs(m) - 1; if (mark[e0 + i]) fm |= 1u << i; }
  }
  // ordered compaction
  const unsigned gm = cg - e0 >= 32 ? 0xffffffffu : cg <= e0 ? 0u : (1u << (cg - e0)) - 1u;   // this thread's members of the sparse cache
  int of = 0;
  unsigned all = 0;                                                // folded pairs of this warp; those of them in G, << 16
#pragma unroll 4
  for (int i = 0; i < run; ++i) {
    const unsigned b = __ballot_sync(0xffffffffu, fm >> i & 1u);
    of += __popc(b & below_me);
    all += (unsigned)__popc(b);
  }
  all |= __reduce_add_sync(0xffffffffu, (unsigned)__popc(fm & gm)) << 16;
  if (lane == 0) S.scan[warp] = all;
  sync();
  all = lane < NW ? S.scan[lane] : 0u;
  of += (int)__reduce_add_sync(0xffffffffu, lane < warp ? all & 0xffffu : 0u);
  const int tg = (int)__reduce_add_sync(0xffffffffu, all >> 16);
  int om = max(0, e0 - cg) - max(0, of - tg);                      // leaving pairs that stay before this thread's
#pragma unroll 4
  for (int i = 0; i < run; ++i)
    if (fm >> i & 1u) {
      fold_e[of++] = (Idx)(e0 + i);
      if (!(gm >> i & 1u)) put_dst(e0 + i - cg, -1);
    }
  sync();
  listed();
  const int left = min(run, nE - e0);
#pragma unroll 1
  for (unsigned m = left > 0 ? ~(fm | gm) & (0xffffffffu >> (32 - left)) : 0u; m; m &= m - 1, ++om)
    put_dst(e0 + __ffs(m) - 1 - cg, om < tg ? (int)fold_e[om] : cg + (om - tg));
}

}  // namespace lola
