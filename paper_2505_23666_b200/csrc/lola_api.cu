// Host side of the C ABI declared in include/lola.h: argument checks, the carve-up of the caller's
// state buffer, the per-call geometry (every count is a function of the tokens seen so far, so no
// device value is ever read back to decide a launch), and the launches themselves.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/lola.h"
#include "lola_generic.cuh"
#include "lola_host_groups.h"
#include "lola_params.h"
#include "lola_score_tc.cuh"
#include "lola_attend_tc.cuh"
#include "lola_decode2_tc.cuh"
#include "lola_score2_tc.cuh"
#include "lola_update2_tc.cuh"
#include "lola_attend2_tc.cuh"
#include "lola_run_tc.cuh"
#include "lola_team_tc.cuh"
#include "lola_unit_f32.cuh"
#include "lola_step_f32.cuh"

using namespace lola;

namespace {

constexpr size_t kAlign = 256;
constexpr size_t kPinnedState = 4u << 20;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct StateLayout {
  size_t status, H, s, gk, gv, gpos, score, wk, wv, fold_idx, move_src, move_dst, counts, thr, wt, total;
};

bool config_ok(const lola_config* c) {
  if (!c) return false;
  if (c->batch < 1 || c->n_kv_heads < 1 || c->n_q_heads < 1) return false;
  if (c->n_q_heads % c->n_kv_heads) return false;
  if (c->head_dim != 64 && c->head_dim != 128) return false;
  if (c->feat_half < 1 || c->feat_half > 128) return false;
  if (c->window < 0 || c->sparse < 0 || c->max_chunk < 1) return false;
  if ((int64_t)c->sparse + c->max_chunk > 16384) return false;
  if (c->dtype != LOLA_F32 && c->dtype != LOLA_BF16) return false;
  if (c->phi_kind != LOLA_PHI_SOFTMAX && c->phi_kind != LOLA_PHI_EXP) return false;
  if (!(c->softmax_scale >= 0.f) || (c->flags & ~(uint32_t)LOLA_FLAGS_ALL) != 0) return false;
  if ((int64_t)2 * c->feat_half * c->head_dim > (int64_t)kUpdThreads * kUpdEPT) return false;
  return true;
}

StateLayout make_layout(const lola_config& c) {
  const size_t U = (size_t)c.batch * c.n_kv_heads, d = c.head_dim, D = 2 * (size_t)c.feat_half;
  const size_t es = c.dtype == LOLA_BF16 ? 2 : 4;
  const size_t lam = c.sparse, eta = c.window, cm = c.max_chunk;
  StateLayout l{};
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes); return at; };
  l.status = take(256);
  l.H = take(U * D * d * 4);
  l.s = take(U * D * 4);
  l.gk = take(U * lam * d * es);
  l.gv = take(U * lam * d * es);
  l.gpos = take(U * lam * 4);
  l.score = take(U * (lam + cm) * 4);
  l.wk = take(U * eta * d * es);
  l.wv = take(U * eta * d * es);
  l.fold_idx = take(U * cm * 4);
  l.move_src = take(U * cm * 4);
  l.move_dst = take(U * cm * 4);
  l.counts = take(U * 4 * 4);
  l.thr = take(U * 2 * 4);
  // W^T of every KV head in tensor-core operand layout (bf16 layers with F = 64 only)
  l.wt = take(c.dtype == LOLA_BF16 && c.feat_half == 64 ? (size_t)c.n_kv_heads * d * 64 * 2 : 0);
  l.total = o;
  return l;
}

inline bool aligned(const void* p, size_t a) { return ((uintptr_t)p % a) == 0; }

// The state as it is before the first token: zeros, and all ones in three byte ranges of it.  One pass: as four fills by the driver a
// reset took 10 - 14 us (states of 1 - 17 MB; 52 at 273 MB), as one kernel 4 - 6 (46).
struct ResetRanges { size_t a0, a1, b0, b1, c0, c1; };
__global__ void __launch_bounds__(512) k_reset(uint4* base, size_t units, ResetRanges R) {
  auto word = [&](size_t x) { return (x >= R.a0 && x < R.a1) || (x >= R.b0 && x < R.b1) || (x >= R.c0 && x < R.c1) ? 0xffffffffu : 0u; };
  for (size_t t0 = (size_t)blockIdx.x * 1024; t0 < units; t0 += (size_t)gridDim.x * 1024) {   // 16 KB at a time
    const size_t lo = t0 * 16, hi = lo + 16384;
    const bool plain = (hi <= R.a0 || lo >= R.a1) && (hi <= R.b0 || lo >= R.b1) && (hi <= R.c0 || lo >= R.c1);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const size_t i = t0 + x * 512 + threadIdx.x;
      if (i >= units) break;
      base[i] = plain ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(word(i * 16), word(i * 16 + 4), word(i * 16 + 8), word(i * 16 + 12));
    }
  }
}

template <typename T, int DPL>
int set_smem_attrs(int D) {
  cudaError_t e;
  e = cudaFuncSetAttribute(k_attend<T, DPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(attend_smem_floats<DPL>(D) * 4));
  if (e != cudaSuccess) return LOLA_ERR_CUDA;
  e = cudaFuncSetAttribute(k_score<T, DPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(score_smem_floats<DPL>(D) * 4));
  if (e != cudaSuccess) return LOLA_ERR_CUDA;
  e = cudaFuncSetAttribute(k_update<T, DPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(update_smem_floats<DPL>(D) * 4));
  if (e != cudaSuccess) return LOLA_ERR_CUDA;
  return LOLA_OK;
}

// Shared-memory limits of the TMA-fed kernels, and one carve-out for all of them: they follow each other in a
// step, and a change of the carve-out between two launches costs idle time on every SM.
template <int DPL>
bool set_tc_attrs() {
  struct { const void* fn; size_t smem; } ks[] = {
      {(const void*)k_score2_tc<DPL>, Score2Smem<DPL>::bytes},      {(const void*)k_apply_tc<DPL, false>, Update2Smem<DPL>::bytes},
      {(const void*)k_apply_tc<DPL, true>, Update2Smem<DPL>::bytes},
      {(const void*)k_attend2_tc<DPL, false>, Attend2Smem<DPL>::bytes}, {(const void*)k_attend2_tc<DPL, true>, Attend2Smem<DPL>::bytes},
      {(const void*)k_decode2_tc<DPL, 4, true, false>, DecodeSmem<DPL>::bytes},  {(const void*)k_decode2_tc<DPL, 4, false, false>, DecodeSmem<DPL>::bytes},
      {(const void*)k_decode2_tc<DPL, 8, true, false>, DecodeSmem<DPL>::bytes},  {(const void*)k_decode2_tc<DPL, 8, false, false>, DecodeSmem<DPL>::bytes},
      {(const void*)k_decode2_tc<DPL, 4, true, true>, DecodeSmem<DPL>::bytes},   {(const void*)k_decode2_tc<DPL, 4, false, true>, DecodeSmem<DPL>::bytes},
      {(const void*)k_decode2_tc<DPL, 8, true, true>, DecodeSmem<DPL>::bytes},   {(const void*)k_decode2_tc<DPL, 8, false, true>, DecodeSmem<DPL>::bytes},
      {(const void*)k_prefill_run<DPL, 32, false>, RunSmem<DPL, 32>::bytes}, {(const void*)k_prefill_run<DPL, 32, true>, RunSmem<DPL, 32>::bytes},
      {(const void*)k_prefill_run<DPL, 64, false>, RunSmem<DPL, 64>::bytes}, {(const void*)k_prefill_run<DPL, 64, true>, RunSmem<DPL, 64>::bytes},
      {(const void*)k_prefill_team<DPL, false>, TeamSmem<DPL>::bytes},       {(const void*)k_prefill_team<DPL, true>, TeamSmem<DPL>::bytes}};
  for (auto& k : ks)
    if (cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem) != cudaSuccess) return false;
  for (auto& k : ks) cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  cudaGetLastError();                  // a refused preference is not an error
  return true;
}

// Clusters of K blocks of a kernel that are resident at once (a block takes an SM to itself; how many clusters fit depends
// on the SMs of each GPC).  cache: of that kernel, one entry per device and K, number + 1.
typedef std::atomic<int> FitCache[64][9];
int clusters_that_fit(const void* kernel, int threads, size_t smem, int K, int dev, FitCache& cache) {
  int fit = dev < 64 ? cache[dev][K].load(std::memory_order_relaxed) - 1 : -1;
  if (fit >= 0) return fit;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)K);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)K;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); fit = 0; }
  if (dev < 64) cache[dev][K].store(fit + 1, std::memory_order_relaxed);
  return fit;
}

// Blocks per unit of the one-kernel prefill run: the largest of 8, 4, 2 whose clusters are all resident at once, 0 if none.
template <int DPL>
int choose_run_blocks(int units, int dev) {
  static FitCache cache;
  for (int K = 8; K > 1; K >>= 1)
    if (units <= clusters_that_fit((const void*)k_prefill_run<DPL, 64, true>, kRunThreads, RunSmem<DPL, 64>::bytes, K, dev, cache)) return K;
  return 0;
}

// fit[K]: clusters of K blocks of the prefill kernel with attention and scoring blocks that are resident at once.
template <int DPL>
void team_fits(int (&fit)[9], int dev) {
  static FitCache cache;
  for (int K = 2; K <= 8; ++K) fit[K] = clusters_that_fit((const void*)k_prefill_team<DPL, true>, kTeamThreads, TeamSmem<DPL>::bytes, K, dev, cache);
}

// fit[K]: clusters of K blocks of the generation kernel that are resident at once.
template <int DPL>
void decode_fits(int (&fit)[9], int dev) {
  static FitCache cache;
  for (int K = 1; K <= 8; ++K) fit[K] = clusters_that_fit((const void*)k_decode2_tc<DPL, 8, false, true>, kDec2Threads, DecodeSmem<DPL>::bytes, K, dev, cache);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point lookup (no link against libcuda).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// bf16 tensor [units][rows][d] viewed as rank 3 (d innermost); boxes of 64 columns x box_rows rows of
// one unit, written to shared memory with the 128-byte swizzle the MMA descriptors expect.
bool make_rows_map(CUtensorMap* tm, void* base, size_t units, size_t rows, size_t d, unsigned box_rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn || rows == 0) return false;
  cuuint64_t dims[3] = {d, rows, units};
  cuuint64_t strides[2] = {d * 2, rows * d * 2};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The sparse cache [units][rows][d]: blocks as above and whole tiles.
bool make_slot_maps(tc::SlotMaps* m, void* base, size_t units, size_t rows, size_t d) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn || rows == 0) return false;
  cuuint64_t dims[4] = {64, rows, d / 64, units};
  cuuint64_t strides[3] = {d * 2, 128, rows * d * 2};
  cuuint32_t box[4] = {64, 128, (cuuint32_t)(d / 64), 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return make_rows_map(&m->block, base, units, rows, d, 64) &&
         fn(&m->tile, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 tensor [chunks][B][n][heads][d] of a run viewed as rank 5; boxes of 64 columns x 1 head x box_tokens tokens.
bool make_run_map(CUtensorMap* tm, const void* base, size_t chunks, size_t B, size_t n, size_t heads, size_t d, unsigned box_tokens) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t dims[5] = {d, heads, n, B, chunks};
  cuuint64_t strides[4] = {d * 2, heads * d * 2, n * heads * d * 2, B * n * heads * d * 2};
  cuuint32_t box[5] = {64, 1, box_tokens, 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 tensor [B][n][heads][d] of one call viewed as rank 4 (d, head, token, batch row); boxes of 64
// columns x 1 head x 64 tokens, 128-byte swizzle.  Tokens beyond n read as zeros.
bool make_tokens_map(CUtensorMap* tm, const void* base, size_t B, size_t n, size_t heads, size_t d) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {d, heads, n, B};
  cuuint64_t strides[3] = {d * 2, heads * d * 2, n * heads * d * 2};
  cuuint32_t box[4] = {64, 1, 64, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

struct ProfRecord { int kind; cudaEvent_t a, b; };

struct lola_state {
  lola_config cfg;
  Layer L;
  StateLayout lay;
  char* base;
  int64_t n_seen;
  int64_t launches;
  bool tensor_path = false;            // bf16, F = 64: tcgen05 kernels
  int dev = 0, sms = 0;                // the device, its SMs
  int dec_fit[9] = {};                 // generation kernel: clusters of 1 .. 8 blocks that are resident at once
  bool fused_decode = false;           // shapes the one-kernel generation step is built for
  bool have_maps = false;              // TMA descriptors of the sparse cache and the window ring exist
  // lola_prefill_host: two copy streams and the events that order them against the kernels (made at first use)
  cudaStream_t cp_in = nullptr, cp_out = nullptr;
  cudaEvent_t ev_start = nullptr, ev_in[2] = {nullptr, nullptr}, ev_done[2] = {nullptr, nullptr}, ev_out[2] = {nullptr, nullptr};
  mutable char* pin = nullptr;         // lola_read_state: pinned image of a small state (made at first use)
  mutable std::mutex pin_mutex;
  bool force_chain = false;            // set while lola_decode_step_static runs: kernel chain with work lists
  int team_fit[9] = {};                // prefill kernel with attention and scoring blocks: clusters of 2 .. 8 that are resident at once
  int run_blocks = 0;                  // bf16 layers: blocks per unit of the one-kernel prefill run (0: not used)
  int unit_blocks = 0;                 // fp32 layers: blocks per unit of the one-kernel step (0: its shape does not fit)
  int step_blocks = 0;                 // ... and of the generation step with F = 64 (0: not used)
  tc::SlotMaps tm_gk, tm_gv;
  CUtensorMap tm_wk, tm_wv;
  lola_call_info info = {};            // what the last prefill / decode call enqueued
  bool profiling = false;
  std::vector<ProfRecord> records;     // events in use since the last lola_profile_read
  std::vector<ProfRecord> pool;        // events ready for reuse
};

namespace {

// Brackets one launch with a pair of events when profiling is on (kind = LOLA_KERNEL_*).
struct LaunchScope {
  lola_state* st; cudaStream_t s; ProfRecord rec; bool on;
  LaunchScope(lola_state* st_, int kind, cudaStream_t s_, uint32_t path = 0, int ctas = 0) : st(st_), s(s_), on(st_->profiling) {
    st->launches++;
    st->info.paths |= path;
    st->info.launches++;
    if (kind >= 0 && kind < LOLA_N_KERNEL_KINDS) st->info.ctas[kind] += ctas;
    if (!on) return;
    if (!st->pool.empty()) { rec = st->pool.back(); st->pool.pop_back(); }
    else if (cudaEventCreate(&rec.a) != cudaSuccess || cudaEventCreate(&rec.b) != cudaSuccess) { on = false; return; }
    rec.kind = kind;
    cudaEventRecord(rec.a, s);
  }
  ~LaunchScope() {
    if (!on) return;
    cudaEventRecord(rec.b, s);
    st->records.push_back(rec);
  }
};

// Launch with programmatic stream serialization: the kernel may become resident while the kernel before it
// in the stream still runs, and waits inside (griddepcontrol.wait) before it touches memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  return launch_pdl_cluster(kernel, 1, grid, block, smem, s, args...);
}

// Thread blocks of the TMA-fed attention kernel per unit: four query heads x 64 tokens each.
inline int attend2_ctas(const Layer& L, const Call& c) { return ((L.g + 1) / 2 + 1) / 2 * ((c.nq + 63) / 64); }

// before_scoring: the kernel after this one in the stream is the scoring kernel of the same call, which only
// reads the memories and runs beside this one: it is let go once this kernel has seen everything before it
// complete, and it waits for this kernel at its end (so that whatever follows sees both complete).
template <typename T, int DPL>
int launch_attend(lola_state* st, const Call& c, cudaStream_t s, bool before_scoring = false) {
  const Layer& L = st->L;
  dim3 grid((L.g * c.nq + kAttRows - 1) / kAttRows, L.B * L.Hkv);
  if (st->have_maps && !st->force_chain && c.att_chunk == c.nq && c.n == c.nq) {
    // prefill chunk: TMA-fed, warp-specialised kernel; the call's q, k, v get their own descriptors
    CUtensorMap tq, tk, tv, tout;
    if (make_tokens_map(&tq, c.q, L.B, c.nq, L.Hq, L.d) && make_tokens_map(&tk, c.k, L.B, c.n, L.Hkv, L.d) &&
        make_tokens_map(&tv, c.v, L.B, c.n, L.Hkv, L.d) && make_tokens_map(&tout, c.out, L.B, c.nq, L.Hq, L.d)) {
      dim3 grid2(attend2_ctas(L, c), L.B * L.Hkv);
      LaunchScope scope(st, LOLA_KERNEL_ATTEND, s, LOLA_PATH_ATTEND_TMA, (int)(grid2.x * grid2.y));
      const cudaError_t le = launch_pdl(c.nq > kLagMaxN ? k_attend2_tc<DPL, true> : k_attend2_tc<DPL, false>, grid2, dim3(kAt2Threads), Attend2Smem<DPL>::bytes, s, L, c, st->tm_gk, st->tm_gv,
                                        st->tm_wk, st->tm_wv, tq, tk, tv, tout, (const uint4*)(st->base + st->lay.wt),
                                        before_scoring ? 1 : 0);
      return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
    }
  }
  if (st->tensor_path && L.g * c.nq >= 64) {
    dim3 tgrid((L.g * c.nq + kAtM - 1) / kAtM, L.B * L.Hkv);
    LaunchScope scope(st, LOLA_KERNEL_ATTEND, s, LOLA_PATH_ATTEND_MMA, (int)(tgrid.x * tgrid.y));
    k_attend_tc<DPL><<<tgrid, 128, AttendTcSmem<DPL>::bytes, s>>>(L, c);
  } else {
    LaunchScope scope(st, LOLA_KERNEL_ATTEND, s, LOLA_PATH_ATTEND_GENERIC, (int)(grid.x * grid.y));
    k_attend<T, DPL><<<grid, 256, attend_smem_floats<DPL>(L.D) * 4, s>>>(L, c);
  }
  return cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

inline bool fast_update_path(const lola_state* st, const Call& c) {
  return c.mode == UPD_SELECT && st->have_maps && !st->force_chain && c.r_pos0 + c.r <= c.n_seen && c.count_g + c.r <= kUp2MaxE && c.n <= kUp2MaxFold;
}

// Eq. 10 scoring and the top-lambda selection on TMA-fed tensor-core kernels.  Both only read the
// memories (scores, positions) and write scores / work lists, so they may run beside the attention
// kernel (busy_sms > 0: that kernel precedes this one in the stream and this one is its programmatic dependent).
template <int DPL>
int launch_score_select(lola_state* st, const Call& c, cudaStream_t ss, int busy_sms = 0) {
  const Layer& L = st->L;
  const int U = L.B * L.Hkv;
  const int NT = ScoreBlocks(c.count_g, c.r, c.r_pos0, L.eta).tiles();
  int tpc = (U * NT + st->sms - 1) / st->sms;
  tpc = std::max(2, tpc + (tpc & 1));
  // beside the attention kernel (one block per SM, busy_sms of them) the blocks of this kernel should fit
  // the SMs that are left in one round: a second round would end after the attention kernel does
  if (busy_sms > 0 && busy_sms < st->sms) {
    const int avail = st->sms - busy_sms;
    int t2 = tpc;
    while (t2 < NT && U * ((NT + t2 - 1) / t2) > avail) ++t2;
    if (U * ((NT + t2 - 1) / t2) <= avail) tpc = t2;
  }
  const uint4* img = (const uint4*)(st->base + st->lay.wt);
  // the selection (Eq. 12) runs in the scoring kernel: the last block of a unit to finish does it
  dim3 grid((NT + tpc - 1) / tpc, U);
  LaunchScope scope(st, LOLA_KERNEL_SCORE, ss, LOLA_PATH_SCORE_TMA, (int)(grid.x * grid.y));
  const cudaError_t le = launch_pdl(k_score2_tc<DPL>, grid, dim3(kSc2Threads), Score2Smem<DPL>::bytes, ss, L, c, st->tm_gk, st->tm_gv, st->tm_wk,
                                    st->tm_wv, img, tpc, busy_sms > 0 ? 1 : 0);
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// Eq. 13 fold (added to H in memory), moves into the sparse cache and window roll from the selection's work lists.
template <int DPL>
int launch_apply(lola_state* st, const Call& c, cudaStream_t s) {
  const Layer& L = st->L;
  LaunchScope scope(st, LOLA_KERNEL_UPDATE, s, LOLA_PATH_APPLY_TMA, L.B * L.Hkv);
  const cudaError_t le = launch_pdl(fold_in_three(c) ? k_apply_tc<DPL, true> : k_apply_tc<DPL, false>, dim3(L.B * L.Hkv), dim3(kUp2Threads), Update2Smem<DPL>::bytes, s, L, c,
                                    (const uint4*)(st->base + st->lay.wt));
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

template <typename T, int DPL>
int launch_update_chain(lola_state* st, const Call& c, cudaStream_t s) {
  const Layer& L = st->L;
  const int U = L.B * L.Hkv;
  // chunkwise update on TMA-fed tensor-core kernels: every leaving pair already sits in the ring
  if (fast_update_path(st, c)) {
    int rc = launch_score_select<DPL>(st, c, s);
    return rc == LOLA_OK ? launch_apply<DPL>(st, c, s) : rc;
  }
  if (st->have_maps && !st->force_chain && (c.mode == UPD_NONE || c.mode == UPD_APPEND) && c.n <= kUp2MaxFold)
    return launch_apply<DPL>(st, c, s);  // nothing folds: moves into free slots and the window roll
  if (c.mode == UPD_SELECT) {
    const int nE = c.count_g + c.r;
    dim3 grid((nE + kScoreRows - 1) / kScoreRows, U);
    if (st->tensor_path) {
      dim3 tgrid((nE + kScTile - 1) / kScTile, U);
      LaunchScope scope(st, LOLA_KERNEL_SCORE, s, LOLA_PATH_SCORE_MMA, (int)(tgrid.x * tgrid.y));
      k_score_tc<DPL><<<tgrid, 128, ScoreTcSmem<DPL>::bytes, s>>>(L, c);
    } else {
      LaunchScope scope(st, LOLA_KERNEL_SCORE, s, LOLA_PATH_SCORE_GENERIC, (int)(grid.x * grid.y));
      k_score<T, DPL><<<grid, 256, score_smem_floats<DPL>(L.D) * 4, s>>>(L, c);
    }
    if (cudaGetLastError() != cudaSuccess) return LOLA_ERR_CUDA;
  }
  if (c.mode != UPD_NONE) {
    const int nE = c.count_g + c.r;
    size_t sm = (c.mode == UPD_SELECT) ? ((size_t)nE * 8 + (size_t)L.cmax * 4 + (size_t)nE + 16) : 0;
    LaunchScope scope(st, LOLA_KERNEL_SELECT, s, LOLA_PATH_SELECT_KERNEL, U);
    k_select<<<U, 256, sm, s>>>(L, c);
    if (cudaGetLastError() != cudaSuccess) return LOLA_ERR_CUDA;
  }
  LaunchScope scope(st, LOLA_KERNEL_UPDATE, s, LOLA_PATH_UPDATE_GENERIC, U);
  k_update<T, DPL><<<U, kUpdThreads, update_smem_floats<DPL>(L.D) * 4, s>>>(L, c);
  return cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// fp32 layers with F = 64: a generation step, whatever the size.  1 to 512 units of 32 to 16000 slots, d = 64 and 128, 1 to 8 heads: it is
// everywhere faster than k_unit_run or, where a unit does not fit one block's shared memory, the kernel chain (us a step, d = 64: 8 units of 128
// slots 9.4 against 25.9, of 16000 522 against 17 ms; a block a unit, 80 units of 300 slots 87 against 179, 128 of 2000 524 against 1365, 512 of
// 600 650 against 1182; d = 128: 80 of 2000 785 against 1942, 512 of 128 250 against 755).
template <int DPL>
int launch_unit_step(lola_state* st, const Call& c, cudaStream_t s) {
  const Layer& L = st->L;
  const int K = st->step_blocks, grid = L.B * L.Hkv * K;
  LaunchScope scope(st, LOLA_KERNEL_DECODE, s, LOLA_PATH_UNIT_RUN | LOLA_PATH_UNIT_STEP, grid);
  const cudaError_t le = launch_pdl_cluster(k_unit_step<DPL>, K, dim3(grid), dim3(kStepThreads), sizeof(StepSmem<DPL>), s, L, c);
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// fp32 layers: a run of prefill chunks, or one generation step, as one kernel.
template <int DPL>
int launch_unit_run(lola_state* st, const Call& c, int n_chunks, bool decode, cudaStream_t s) {
  const Layer& L = st->L;
  const int K = st->unit_blocks, grid = L.B * L.Hkv * K;
  const UnitLayout Y = unit_layout(L, K, c.out ? L.g * c.nq : 0);
  auto kernel = k_unit_run<DPL, false>;
  if constexpr (DPL == 4) { if (Y.both) kernel = k_unit_run<DPL, true>; }
  LaunchScope scope(st, decode ? LOLA_KERNEL_DECODE : LOLA_KERNEL_RUN, s, LOLA_PATH_UNIT_RUN, grid);
  const cudaError_t le = launch_pdl_cluster(kernel, K, dim3(grid), dim3(kUnThreads), (size_t)Y.total * 4, s, L, c, n_chunks, decode ? 1 : 0, Y);
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// bf16 layers: shapes the one-kernel prefill run serves: up to 2 K query items.  Chunks of more than 64 tokens, whose stabiliser
// follows the maximum (kLag), and units of two blocks with two items each are left to the kernel with attention and scoring
// blocks (64 units, g = 2: 33 us a chunk here, 31 there; g = 1: 29 and 31.  With a lag chunks of 128 tokens of 8 units took 24.3
// here, g = 2, and 26.9, g = 4; 25.6 and 27.1 there without; of 100 tokens, d = 64, g = 1, 20.9 and 20.3; 256 tokens 33 and 26).
inline int run_nq(const lola_state* st, int n) { return st->L.g * ((n + 31) / 32) <= st->run_blocks ? 32 : 64; }
inline bool run_path(const lola_state* st, int n) {
  return st->run_blocks > 0 && st->L.g * ((n + 31) / 32) <= 2 * st->run_blocks && !st->force_chain && n <= std::min(st->L.eta, kRunMaxN) &&
         st->L.lam + n <= run_max_e(run_nq(st, n)) && (st->run_blocks > 2 || run_nq(st, n) == 32);
}

// Does a chunk of the run fold in three parts?  Once the sparse cache is full its count is no longer any chunk's own.
inline bool run_folds_in_three(const Layer& L, Call c, int n_chunks) {
  for (int n_seen = c.n_seen; n_chunks > 0; --n_chunks, n_seen += c.n) {
    plan_call(L, c, n_seen, c.n, false);
    if (c.mode == UPD_SELECT && fold_in_three(c)) return true;
    if (c.count_g == L.lam) return false;
  }
  return false;
}

template <int DPL>
int launch_prefill_run(lola_state* st, const Call& c, int n_chunks, cudaStream_t s) {
  const Layer& L = st->L;
  const int K = st->run_blocks, grid = L.B * L.Hkv * K;
  RunMaps M;
  M.gk = st->tm_gk; M.gv = st->tm_gv; M.wk = st->tm_wk; M.wv = st->tm_wv;
  if (!make_run_map(&M.k, c.k, n_chunks, L.B, c.n, L.Hkv, L.d, 64) || !make_run_map(&M.v, c.v, n_chunks, L.B, c.n, L.Hkv, L.d, 64) ||
      !make_run_map(&M.q, c.out ? c.q : c.k, n_chunks, L.B, c.n, c.out ? L.Hq : L.Hkv, L.d, 32))
    return LOLA_ERR_CUDA;
  const bool wide = run_nq(st, c.n) == 64;
  LaunchScope scope(st, LOLA_KERNEL_RUN, s, LOLA_PATH_PREFILL_RUN, grid);
  const bool three = run_folds_in_three(L, c, n_chunks);
  const cudaError_t le = launch_pdl_cluster(wide ? (three ? k_prefill_run<DPL, 64, true> : k_prefill_run<DPL, 64, false>)
                                                 : (three ? k_prefill_run<DPL, 32, true> : k_prefill_run<DPL, 32, false>), K, dim3(grid), dim3(kRunThreads),
                                            wide ? RunSmem<DPL, 64>::bytes : RunSmem<DPL, 32>::bytes, s, L, c, n_chunks, M,
                                            (const uint4*)(st->base + st->lay.wt));
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// Attention and scoring blocks per unit (A, N) of the prefill kernel that has both, for chunks of n tokens on full caches; A = 0
// where its clusters do not fit or the three-kernel chain is faster.  Microseconds of the parts at d = 128, from when the selection took
// 7 us (it takes 4 now, in both): an item (two query tiles) 6 + 2.1 per key tile, 8 around them; scoring 4.8 per pair of tiles and block,
// selection and fold 11 and 4 per further 64 pairs.  The chain: an attention block (an item) 7 + 2.1 per key tile, in rounds of
// the SMs; 2.6 per scored tile on the SMs it leaves; 10 and 11 per further 64 pairs for the fold.  The set-up of a run, 6, is shared by its
// chunks.  The choices, measured with what the kernels take now (a chunk of a run of 16, here and there; d = 128, then d = 64): 64 units
// of 832 slots, 4 heads 30 and 37, 27 and 31, 8 heads 53.4 and 53.2, 49 and 47; 48 of 500, 8 heads 42 and 33, 38 and 29; chunks of 256, 16 units of
// 512, 4 heads 35 and 61, 30 and 47, 64 units 121 and 102, 105 and 83; of 128, 32 units of 960, 4 heads 38 and 52, 34 and 42; of 96, 24 units of
// 500, 4 heads 28 and 41, 25 and 34.  Of 60 shapes it takes the slower one for four, all of 8 heads: by 4% (64 units of 832, d = 64, and 32 of
// 960, chunks of 128) to 8% (the latter with d = 64, and 16 of 512, chunks of 256); and for single chunks of 64 units with 8 heads (65 and 56).
struct TeamShape { int A, N; };
inline TeamShape team_shape(const lola_state* st, int n, int n_chunks) {
  const Layer& L = st->L;
  TeamShape best{0, 0};
  if (st->force_chain || n > L.eta || n > kTeamMaxN || L.lam + n > kTeamMaxE) return best;
  const int U = L.B * L.Hkv, ntb = (n + 63) / 64, items = ntb * (((L.g + 1) / 2 + 1) / 2), sms = st->sms;
  const int blocks = (L.lam + 63) / 64 + (L.eta + 63) / 64, scored = ((L.lam + 63) / 64 + ntb + 1) / 2;
  const double tiles = 2.1 * ((blocks + ntb + 1) / 2);
  double t_best = (U * items + sms - 1) / sms * (7 + tiles);         // the chain
  if (U * items < sms) t_best = std::max(t_best, 7 + 2.6 * U * scored / (sms - U * items));
  t_best += 10 + 11 * (ntb - 1);
  for (int N = 1; N <= 4; N *= 2)
    for (int A = 1; A <= std::min(items, 8 - N); ++A) {
      if (U > st->team_fit[A + N]) continue;
      const double att = (items + A - 1) / A * (6 + tiles) + 8, sc = 4.8 * ((scored + 2 * N - 1) / (2 * N)) + 11 + 4 * (ntb - 1);
      const double t = std::max(att, sc) + 0.1 * (A + N) + 6.0 / n_chunks;
      if (t < t_best) { t_best = t; best = {A, N}; }
    }
  return best;
}

template <int DPL>
int launch_prefill_team(lola_state* st, const Call& c, int n_chunks, TeamShape ts, cudaStream_t s) {
  const Layer& L = st->L;
  const int K = ts.A + ts.N, grid = L.B * L.Hkv * K;
  TeamMaps M;
  M.gk = st->tm_gk; M.gv = st->tm_gv; M.wk = st->tm_wk; M.wv = st->tm_wv;
  const int hq = c.out ? L.Hq : L.Hkv;
  if (!make_run_map(&M.k, c.k, n_chunks, L.B, c.n, L.Hkv, L.d, 64) || !make_run_map(&M.v, c.v, n_chunks, L.B, c.n, L.Hkv, L.d, 64) ||
      !make_run_map(&M.q, c.out ? c.q : c.k, n_chunks, L.B, c.n, hq, L.d, 64) || !make_run_map(&M.out, c.out ? c.out : c.k, n_chunks, L.B, c.n, hq, L.d, 64))
    return LOLA_ERR_CUDA;
  LaunchScope scope(st, LOLA_KERNEL_RUN, s, LOLA_PATH_PREFILL_RUN, grid);
  const cudaError_t le = launch_pdl_cluster(c.n > kLagMaxN || run_folds_in_three(L, c, n_chunks) ? k_prefill_team<DPL, true> : k_prefill_team<DPL, false>, K, dim3(grid), dim3(kTeamThreads), TeamSmem<DPL>::bytes, s, L, c, n_chunks, M,
                                            (const uint4*)(st->base + st->lay.wt), ts.A);
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

// n_chunks > 1 only where the whole run is one launch.
template <typename T, int DPL>
int run_prefill(lola_state* st, Call c, int n_chunks, cudaStream_t s) {
  if (st->unit_blocks > 0 && !st->force_chain) return launch_unit_run<DPL>(st, c, n_chunks, false, s);
  if (run_path(st, c.n)) return launch_prefill_run<DPL>(st, c, n_chunks, s);
  const TeamShape ts = team_shape(st, c.n, n_chunks);
  if (ts.A > 0) return launch_prefill_team<DPL>(st, c, n_chunks, ts, s);
  int rc = LOLA_OK;
  // Attention and scoring both only read the memories: with outputs wanted and the tensor-core update path
  // in use they run side by side, all on the caller's stream, chained by programmatic dependent launches:
  // the attention kernel waits for everything before it and then lets the scoring kernel (with the selection
  // in its last block per unit) start; the scoring kernel waits for the attention kernel only at its end; the
  // fold waits for the scoring kernel, hence for both.
  if (c.out && fast_update_path(st, c)) {
    rc = launch_attend<T, DPL>(st, c, s, true);
    if (rc != LOLA_OK) return rc;
    rc = launch_score_select<DPL>(st, c, s, attend2_ctas(st->L, c) * st->L.B * st->L.Hkv);
    if (rc != LOLA_OK) return rc;
    return launch_apply<DPL>(st, c, s);
  }
  if (c.out) rc = launch_attend<T, DPL>(st, c, s);
  if (rc != LOLA_OK) return rc;
  return launch_update_chain<T, DPL>(st, c, s);
}

// One block per unit, or, where there are fewer units than SMs, a cluster of as many as are resident at once and have a
// tile each (8 units of 7 tiles: one block each 24, seven 13.4 us a step; 40 units: 24 and 17.9; 72 units: 25 and 20).  Units
// left over by whole rounds of blocks as a second launch of clusters were no gain: 64 against 47 us for 216 units.
template <int DPL>
int launch_decode_fused(lola_state* st, const Call& c, cudaStream_t s) {
  const Layer& L = st->L;
  const int U = L.B * L.Hkv;
  const int tiles = std::max(1, ((c.count_g + 63) / 64 + (std::min(L.eta, c.n_seen) + 63) / 64 + 1) / 2);
  int K = std::min(8, tiles);
  while (K > 1 && U > st->dec_fit[K]) --K;
  const int per = (tiles + K - 1) / K;
  K = (tiles + per - 1) / per;                       // no more blocks than it takes
  // meeting costs as much as one to two tiles: 64 units, g = 4, two blocks for 3 tiles 16.2 against 14.3 us, for 5 tiles 18.2
  // against 17.9, for 7 tiles (g = 8) 21.9 against 26.0; three blocks for 3 tiles 12.7 against 13.7.  d = 64, 64 units, two
  // blocks against one: g = 4 2 tiles 13.3 and 11.5, 3 tiles 15.1 and 13.2, 5 tiles 16.8 and 16.3; g = 8 13.3 and 13.1, 15.3 and
  // 14.7, 17.1 and 18.2; 8 units within 0.3 of each other for 2 tiles, three blocks for 3 tiles 12.2 against 12.8.  While the
  // caches fill there is no pair to agree on: two blocks for 2 tiles 11.3 against 11.8
  if (c.mode == UPD_SELECT && tiles - per < (K == 2 && L.g <= 4 ? 3 : 2)) K = 1;
  // 16-bit weights, phi(q) and H in Eq. 14 and a 16-bit feature row of the folded pair: full caches of whole 64-slot blocks
  // within 16 tiles.  Steps of all other shapes have them in fp32 (WIDE), as the CUDA-core kernels that served these shapes
  // before had: an output is then off by no more than its own rounding to bf16 (up to 16 times that otherwise, where a few
  // pairs carry the softmax).  It costs 1 us of 15.5 (40 units of 500 slots), while the caches fill 0.3 us of 10.8
  const bool wide = c.mode != UPD_SELECT || L.lam % 64 != 0 || (L.lam / 64 + (L.eta + 63) / 64 + 1) / 2 > kDecNarrowTiles;
  auto kernel = K > 1 ? (L.g <= 4 ? (wide ? k_decode2_tc<DPL, 4, true, true> : k_decode2_tc<DPL, 4, false, true>)
                                  : (wide ? k_decode2_tc<DPL, 8, true, true> : k_decode2_tc<DPL, 8, false, true>))
                      : (L.g <= 4 ? (wide ? k_decode2_tc<DPL, 4, true, false> : k_decode2_tc<DPL, 4, false, false>)
                                  : (wide ? k_decode2_tc<DPL, 8, true, false> : k_decode2_tc<DPL, 8, false, false>));
  LaunchScope scope(st, LOLA_KERNEL_DECODE, s, LOLA_PATH_DECODE_FUSED, U * K);
  const cudaError_t le = launch_pdl_cluster(kernel, K, dim3(U * K), dim3(kDec2Threads), DecodeSmem<DPL>::bytes, s, L, c, st->tm_gk, st->tm_gv, st->tm_wk,
                                            st->tm_wv, (const uint4*)(st->base + st->lay.wt), std::max(1, st->dec_fit[1]));
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

template <typename T, int DPL>
int run_decode(lola_state* st, Call c, cudaStream_t s) {
  if (st->step_blocks > 0 && !st->force_chain) return launch_unit_step<DPL>(st, c, s);
  if (st->unit_blocks > 0 && !st->force_chain) return launch_unit_run<DPL>(st, c, 1, true, s);
  // the whole step is one kernel, with full caches (UPD_SELECT) and while they fill (UPD_NONE, UPD_APPEND)
  const bool ablation = (st->cfg.flags & (LOLA_FLAG_QUERY_NO_LINEAR | LOLA_FLAG_QUERY_NO_SPARSE)) != 0;
  if (st->fused_decode && !st->force_chain && !ablation) return launch_decode_fused<DPL>(st, c, s);
  int rc = launch_update_chain<T, DPL>(st, c, s);
  if (rc != LOLA_OK) return rc;
  return launch_attend<T, DPL>(st, c, s);
}

#define LOLA_DISPATCH(fn, st, ...)                                                            \
  ((st)->cfg.dtype == LOLA_BF16                                                               \
       ? ((st)->cfg.head_dim == 128 ? fn<__nv_bfloat16, 4>(st, __VA_ARGS__) : fn<__nv_bfloat16, 2>(st, __VA_ARGS__)) \
       : ((st)->cfg.head_dim == 128 ? fn<float, 4>(st, __VA_ARGS__) : fn<float, 2>(st, __VA_ARGS__)))

size_t elem_size(const lola_config& c) { return c.dtype == LOLA_BF16 ? 2 : 4; }

// One warp waits, with the same bounded wait every kernel uses, for an mbarrier phase that nothing
// completes; the wait gives up after `limit_ns` and the failure is recorded like any other.
__global__ void k_selftest_wait(int* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_word;
  const uint32_t b = tc::smem_u32(&bar);
  if (threadIdx.x == 0) {
    abort_word = 0;
    tc::mbar_init(b, 1);
    tc::mbar_init_fence();
  }
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) ok = tc::mbar_try_wait(b, 0) || tc::mbar_wait_slow(b, 0, &abort_word, limit_ns);
  if (!ok) atomicOr(status, LOLA_STATUS_SELFTEST);
}

}  // namespace

extern "C" {

size_t lola_state_bytes(const lola_config* cfg) {
  if (!config_ok(cfg)) return 0;
  return make_layout(*cfg).total;
}

int lola_init_state(const lola_config* cfg, const void* W_dev, void* state_dev, size_t state_bytes, void* stream,
                    lola_state** out) {
  if (!cfg || !W_dev || !state_dev || !out) return LOLA_ERR_ARG;
  if (!config_ok(cfg)) {
    if (cfg->head_dim != 64 && cfg->head_dim != 128 && cfg->head_dim > 0) return LOLA_ERR_UNSUPPORTED;
    return LOLA_ERR_SHAPE;
  }
  if (!aligned(W_dev, 16) || !aligned(state_dev, kAlign)) return LOLA_ERR_ALIGN;
  StateLayout lay = make_layout(*cfg);
  if (state_bytes < lay.total) return LOLA_ERR_SIZE;
  int dev = 0, major = 0, sms = 0;     // (single attributes: filling in cudaDeviceProp takes milliseconds)
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return LOLA_ERR_CUDA;
  if (major != 10) return LOLA_ERR_UNSUPPORTED;

  lola_state* st = new (std::nothrow) lola_state();
  if (!st) return LOLA_ERR_ARG;
  st->cfg = *cfg;
  st->lay = lay;
  st->base = (char*)state_dev;
  st->dev = dev;
  st->sms = sms;
  st->n_seen = 0;
  st->launches = 0;
  Layer& L = st->L;
  L.B = cfg->batch; L.Hq = cfg->n_q_heads; L.Hkv = cfg->n_kv_heads; L.g = cfg->n_q_heads / cfg->n_kv_heads;
  L.d = cfg->head_dim; L.F = cfg->feat_half; L.D = 2 * cfg->feat_half;
  L.eta = cfg->window; L.lam = cfg->sparse; L.cmax = cfg->max_chunk;
  L.flags = cfg->flags; L.phi_kind = cfg->phi_kind; L.bf16 = cfg->dtype == LOLA_BF16;
  L.scale = cfg->softmax_scale > 0.f ? cfg->softmax_scale : 1.0f / std::sqrt((float)cfg->head_dim);
  char* b = st->base;
  L.status = (int*)(b + lay.status);
  L.H = (float*)(b + lay.H); L.s = (float*)(b + lay.s);
  L.gk = b + lay.gk; L.gv = b + lay.gv; L.gpos = (int*)(b + lay.gpos); L.score = (float*)(b + lay.score);
  L.wk = b + lay.wk; L.wv = b + lay.wv;
  L.fold_idx = (int*)(b + lay.fold_idx); L.move_src = (int*)(b + lay.move_src); L.move_dst = (int*)(b + lay.move_dst);
  L.counts = (int*)(b + lay.counts); L.thr = (float*)(b + lay.thr);
  L.W = W_dev;

  int rc = LOLA_OK;
  if (cfg->dtype == LOLA_BF16) rc = cfg->head_dim == 128 ? set_smem_attrs<__nv_bfloat16, 4>(L.D) : set_smem_attrs<__nv_bfloat16, 2>(L.D);
  else rc = cfg->head_dim == 128 ? set_smem_attrs<float, 4>(L.D) : set_smem_attrs<float, 2>(L.D);
  if (rc == LOLA_OK && cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize, 9 * 16384 + 4 * 16384 + 64) != cudaSuccess)
    rc = LOLA_ERR_CUDA;
  st->tensor_path = cfg->dtype == LOLA_BF16 && cfg->feat_half == 64 && !(cfg->flags & LOLA_FLAG_GENERIC_KERNELS);
  if (rc == LOLA_OK && cfg->dtype == LOLA_F32 && !(cfg->flags & LOLA_FLAG_GENERIC_KERNELS)) {
    // fp32 step as one kernel: as many blocks per unit as have an SM each, if a block's shared memory suffices
    const int U = cfg->batch * cfg->n_kv_heads, smem_max = kUnSmem;
    int K = 8;
    while (K > 1 && U * K > sms) K >>= 1;
    if (unit_layout_of(L, K, 0).total * 4 <= smem_max &&
        (cfg->head_dim != 128 || cudaFuncSetAttribute(k_unit_run<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max) == cudaSuccess) &&
        (cfg->head_dim == 128 ? cudaFuncSetAttribute(k_unit_run<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max)
                              : cudaFuncSetAttribute(k_unit_run<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max)) == cudaSuccess)
      st->unit_blocks = K;
    const bool ablation = (cfg->flags & (LOLA_FLAG_QUERY_NO_LINEAR | LOLA_FLAG_QUERY_NO_SPARSE)) != 0;
    if (cfg->feat_half == 64 && cfg->sparse >= 1 && cfg->window >= 1 && L.g <= kStepQ && !ablation &&
        (cfg->head_dim == 128 ? cudaFuncSetAttribute(k_unit_step<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StepSmem<4>))
                              : cudaFuncSetAttribute(k_unit_step<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StepSmem<2>))) == cudaSuccess)
      st->step_blocks = K;
  }
  if (rc == LOLA_OK && st->tensor_path) {
    cudaError_t e = cfg->head_dim == 128
        ? cudaFuncSetAttribute(k_score_tc<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ScoreTcSmem<4>::bytes)
        : cudaFuncSetAttribute(k_score_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ScoreTcSmem<2>::bytes);
    if (e != cudaSuccess) rc = LOLA_ERR_CUDA;
    e = cfg->head_dim == 128
        ? cudaFuncSetAttribute(k_attend_tc<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AttendTcSmem<4>::bytes)
        : cudaFuncSetAttribute(k_attend_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AttendTcSmem<2>::bytes);
    if (e != cudaSuccess) rc = LOLA_ERR_CUDA;
  }
  if (rc == LOLA_OK && st->tensor_path && cfg->sparse >= 1 && cfg->window >= 1) {
    const size_t U = (size_t)cfg->batch * cfg->n_kv_heads;
    st->have_maps = make_slot_maps(&st->tm_gk, L.gk, U, cfg->sparse, cfg->head_dim) &&
                    make_slot_maps(&st->tm_gv, L.gv, U, cfg->sparse, cfg->head_dim) &&
                    make_rows_map(&st->tm_wk, L.wk, U, cfg->window, cfg->head_dim, 64) &&
                    make_rows_map(&st->tm_wv, L.wv, U, cfg->window, cfg->head_dim, 64);
    if (!(cfg->head_dim == 128 ? set_tc_attrs<4>() : set_tc_attrs<2>())) st->have_maps = false;   // the older kernel chain serves every shape
  }
  st->fused_decode = st->have_maps && L.g <= kDecQ;
  if (st->fused_decode) { if (cfg->head_dim == 128) decode_fits<4>(st->dec_fit, dev); else decode_fits<2>(st->dec_fit, dev); }
  if (rc == LOLA_OK && st->have_maps) {
    const int U = cfg->batch * cfg->n_kv_heads;
    if (cfg->head_dim == 128) team_fits<4>(st->team_fit, dev); else team_fits<2>(st->team_fit, dev);
    st->run_blocks = cfg->head_dim == 128 ? choose_run_blocks<4>(U, dev) : choose_run_blocks<2>(U, dev);
  }
  if (rc == LOLA_OK && st->tensor_path) {
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16* img = (__nv_bfloat16*)(st->base + lay.wt);
    if (cfg->head_dim == 128) k_prep_wt_image<4><<<cfg->n_kv_heads, 256, 0, s>>>((const __nv_bfloat16*)W_dev, img, cfg->n_kv_heads);
    else k_prep_wt_image<2><<<cfg->n_kv_heads, 256, 0, s>>>((const __nv_bfloat16*)W_dev, img, cfg->n_kv_heads);
    if (cudaGetLastError() != cudaSuccess) rc = LOLA_ERR_CUDA;
  }
  if (rc == LOLA_OK) rc = lola_reset_state(st, stream);
  if (rc != LOLA_OK) { lola_destroy_state(st); return rc; }
  *out = st;
  return LOLA_OK;
}

int lola_reset_state(lola_state* st, void* stream) {
  if (!st) return LOLA_ERR_ARG;
  const lola_config& c = st->cfg;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t U = (size_t)c.batch * c.n_kv_heads;
  // all but the W^T image: zeros, positions -1, scores and thresholds NaN (all-ones bit pattern)
  const StateLayout& y = st->lay;
  const ResetRanges R{y.gpos, y.gpos + U * c.sparse * 4, y.score, y.score + U * (c.sparse + c.max_chunk) * 4, y.thr, y.thr + U * 2 * 4};
  const size_t units = y.wt / 16;
  // (the caller's device need not be the state's: a fill would not mind, a kernel runs where it is launched)
  int cur = st->dev;
  if (cudaGetDevice(&cur) != cudaSuccess || (cur != st->dev && cudaSetDevice(st->dev) != cudaSuccess)) return LOLA_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min<size_t>((units + 1023) / 1024, (size_t)st->sms * 4));
  cfg.blockDim = dim3(512);
  cfg.stream = s;
  const bool ok = cudaLaunchKernelEx(&cfg, k_reset, (uint4*)st->base, units, R) == cudaSuccess;   // (its own status: not what an earlier call left)
  if ((cur != st->dev && cudaSetDevice(cur) != cudaSuccess) || !ok) return LOLA_ERR_CUDA;
  st->n_seen = 0;
  return LOLA_OK;
}

int lola_prefill_chunk(lola_state* st, const void* q, const void* k, const void* v, int32_t n_tokens, void* out,
                       void* stream) {
  return lola_prefill_chunks(st, q, k, v, 1, n_tokens, out, stream);
}

int lola_prefill_chunks(lola_state* st, const void* q, const void* k, const void* v, int32_t n_chunks, int32_t n_tokens,
                        void* out, void* stream) {
  if (!st || !k || !v) return LOLA_ERR_ARG;
  if (out && !q) return LOLA_ERR_ARG;
  if (n_chunks < 1 || n_tokens < 1 || n_tokens > st->cfg.max_chunk) return LOLA_ERR_SHAPE;
  if (!aligned(k, 16) || !aligned(v, 16) || (out && (!aligned(q, 16) || !aligned(out, 16)))) return LOLA_ERR_ALIGN;
  const lola_config& cfg = st->cfg;
  const size_t es = cfg.dtype == LOLA_BF16 ? 2 : 4;
  const size_t qbytes = (size_t)cfg.batch * n_tokens * cfg.n_q_heads * cfg.head_dim * es;
  const size_t kbytes = (size_t)cfg.batch * n_tokens * cfg.n_kv_heads * cfg.head_dim * es;
  // chunks of one launch: all of them where one kernel carries a unit through the run, else one (also near the end of the
  // positions, which are int32)
  const bool all = (0x7fffffffLL - st->n_seen) / n_tokens >= n_chunks && (st->unit_blocks > 0 || run_path(st, n_tokens) || team_shape(st, n_tokens, n_chunks).A > 0);
  const int per = all ? n_chunks : 1;
  for (int i = 0; i < n_chunks; i += per) {
    if (st->n_seen + n_tokens > 0x7fffffffLL) return LOLA_ERR_SHAPE;
    st->info = lola_call_info{};
    Call c{};
    c.q = out ? (const char*)q + (size_t)i * qbytes : nullptr;
    c.k = (const char*)k + (size_t)i * kbytes;
    c.v = (const char*)v + (size_t)i * kbytes;
    c.out = out ? (char*)out + (size_t)i * qbytes : nullptr;
    plan_call(st->L, c, (int)st->n_seen, n_tokens, false);
    const int rc = LOLA_DISPATCH(run_prefill, st, c, per, (cudaStream_t)stream);
    if (rc != LOLA_OK) return rc;
    st->n_seen += (int64_t)per * n_tokens;
  }
  return LOLA_OK;
}

int lola_decode_step(lola_state* st, const void* q, const void* k, const void* v, void* out, void* stream) {
  if (!st || !q || !k || !v || !out) return LOLA_ERR_ARG;
  if (st->n_seen + 1 > 0x7fffffffLL) return LOLA_ERR_SHAPE;
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(v, 16) || !aligned(out, 16)) return LOLA_ERR_ALIGN;
  st->info = lola_call_info{};
  Call c{};
  c.q = q; c.k = k; c.v = v; c.out = out;
  plan_call(st->L, c, (int)st->n_seen, 1, true);
  int rc = LOLA_DISPATCH(run_decode, st, c, (cudaStream_t)stream);
  if (rc == LOLA_OK) st->n_seen += 1;
  return rc;
}

size_t lola_staging_bytes(const lola_config* cfg, int32_t n_tokens) {
  if (!config_ok(cfg) || n_tokens < 1) return 0;
  const size_t es = elem_size(*cfg), d = cfg->head_dim, B = cfg->batch;
  const size_t qb = align_up(B * n_tokens * cfg->n_q_heads * d * es);
  const size_t kb = align_up(B * n_tokens * cfg->n_kv_heads * d * es);
  return 2 * qb + 2 * kb;
}

static int run_host(lola_state* st, const void* qh, const void* kh, const void* vh, int32_t n, void* oh, void* stg,
                    size_t stg_bytes, void* stream, bool decode) {
  if (!st || !kh || !vh || !stg) return LOLA_ERR_ARG;
  if ((decode || oh) && !qh) return LOLA_ERR_ARG;
  if (decode && !oh) return LOLA_ERR_ARG;
  if (n < 1 || n > st->cfg.max_chunk) return LOLA_ERR_SHAPE;
  if (!aligned(stg, kAlign)) return LOLA_ERR_ALIGN;
  if (stg_bytes < lola_staging_bytes(&st->cfg, n)) return LOLA_ERR_SIZE;
  const lola_config& c = st->cfg;
  const size_t es = elem_size(c), d = c.head_dim, B = c.batch;
  const size_t qbytes = B * n * c.n_q_heads * d * es, kbytes = B * n * c.n_kv_heads * d * es;
  const size_t qb = align_up(qbytes), kb = align_up(kbytes);
  char* p = (char*)stg;
  void *qd = p, *kd = p + qb, *vd = p + qb + kb, *od = p + qb + 2 * kb;
  cudaStream_t s = (cudaStream_t)stream;
  if (oh && cudaMemcpyAsync(qd, qh, qbytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return LOLA_ERR_CUDA;
  if (cudaMemcpyAsync(kd, kh, kbytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return LOLA_ERR_CUDA;
  if (cudaMemcpyAsync(vd, vh, kbytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return LOLA_ERR_CUDA;
  int rc = decode ? lola_decode_step(st, qd, kd, vd, od, stream)
                  : lola_prefill_chunk(st, oh ? qd : nullptr, kd, vd, n, oh ? od : nullptr, stream);
  if (rc != LOLA_OK) return rc;
  if (oh && cudaMemcpyAsync(oh, od, qbytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) return LOLA_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return LOLA_ERR_CUDA;
  return LOLA_OK;
}

int lola_prefill_chunk_host(lola_state* st, const void* q_host, const void* k_host, const void* v_host,
                            int32_t n_tokens, void* out_host, void* staging_dev, size_t staging_bytes, void* stream) {
  return run_host(st, q_host, k_host, v_host, n_tokens, out_host, staging_dev, staging_bytes, stream, false);
}

int lola_decode_step_host(lola_state* st, const void* q_host, const void* k_host, const void* v_host, void* out_host,
                          void* staging_dev, size_t staging_bytes, void* stream) {
  return run_host(st, q_host, k_host, v_host, 1, out_host, staging_dev, staging_bytes, stream, true);
}

static bool ensure_copy_streams(lola_state* st) {
  if (st->cp_in) return true;
  cudaEvent_t* evs[7] = {&st->ev_start, &st->ev_in[0], &st->ev_in[1], &st->ev_done[0], &st->ev_done[1], &st->ev_out[0], &st->ev_out[1]};
  bool ok = cudaStreamCreateWithFlags(&st->cp_in, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&st->cp_out, cudaStreamNonBlocking) == cudaSuccess;
  for (cudaEvent_t* e : evs) ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    for (cudaEvent_t* e : evs) if (*e) { cudaEventDestroy(*e); *e = nullptr; }
    if (st->cp_in) { cudaStreamDestroy(st->cp_in); st->cp_in = nullptr; }
    if (st->cp_out) { cudaStreamDestroy(st->cp_out); st->cp_out = nullptr; }
  }
  return ok;
}

int lola_prefill_host(lola_state* st, const void* q_host, const void* k_host, const void* v_host, int32_t n_chunks,
                      int32_t n_tokens, void* out_host, void* staging_dev, size_t staging_bytes, void* stream) {
  if (!st || !k_host || !v_host || !staging_dev) return LOLA_ERR_ARG;
  if (out_host && !q_host) return LOLA_ERR_ARG;
  if (n_chunks < 1 || n_tokens < 1 || n_tokens > st->cfg.max_chunk) return LOLA_ERR_SHAPE;
  if (!aligned(staging_dev, kAlign)) return LOLA_ERR_ALIGN;
  const size_t per = lola_staging_bytes(&st->cfg, n_tokens);
  if (staging_bytes < 2 * per) return LOLA_ERR_SIZE;
  if (!ensure_copy_streams(st)) return LOLA_ERR_CUDA;
  const lola_config& c = st->cfg;
  const size_t es = elem_size(c), d = c.head_dim, B = c.batch;
  const size_t qbytes = B * n_tokens * c.n_q_heads * d * es, kbytes = B * n_tokens * c.n_kv_heads * d * es;
  cudaStream_t s = (cudaStream_t)stream;
  bool ok = cudaEventRecord(st->ev_start, s) == cudaSuccess && cudaStreamWaitEvent(st->cp_in, st->ev_start, 0) == cudaSuccess;
  int rc = LOLA_OK;
  bool out_pending[2] = {false, false};
  const HostGroups G(n_chunks, qbytes, kbytes, per, staging_bytes);   // chunks travel in groups
  const HostGroups::At at = G.at();
  int m = 0;
  for (int i = 0, gr = 0; ok && rc == LOLA_OK && i < n_chunks; i += m, ++gr) {
    const int b = gr & 1;
    m = G.size(i);
    char* p = (char*)staging_dev + (size_t)b * G.half;
    const size_t qm = (size_t)m * qbytes, km = (size_t)m * kbytes;
    void *qd = p + at.q, *kd = p + at.k, *vd = p + at.v, *od = p + at.out;
    // copies in (copy stream): the inputs' part of this half is free once the kernels of the group before the last are done (its
    // outputs may still be on their way out)
    if (gr >= 2) ok = ok && cudaStreamWaitEvent(st->cp_in, st->ev_done[b], 0) == cudaSuccess;
    if (out_host) ok = ok && cudaMemcpyAsync(qd, (const char*)q_host + (size_t)i * qbytes, qm, cudaMemcpyHostToDevice, st->cp_in) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(kd, (const char*)k_host + (size_t)i * kbytes, km, cudaMemcpyHostToDevice, st->cp_in) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(vd, (const char*)v_host + (size_t)i * kbytes, km, cudaMemcpyHostToDevice, st->cp_in) == cudaSuccess;
    ok = ok && cudaEventRecord(st->ev_in[b], st->cp_in) == cudaSuccess;
    // kernels (caller's stream): after the copies in, and after the copy out of that group has read `od`
    ok = ok && cudaStreamWaitEvent(s, st->ev_in[b], 0) == cudaSuccess;
    if (out_pending[b]) ok = ok && cudaStreamWaitEvent(s, st->ev_out[b], 0) == cudaSuccess;
    if (!ok) break;
    rc = lola_prefill_chunks(st, out_host ? qd : nullptr, kd, vd, m, n_tokens, out_host ? od : nullptr, stream);
    if (rc != LOLA_OK) break;
    ok = ok && cudaEventRecord(st->ev_done[b], s) == cudaSuccess;
    // copy out (second copy stream)
    if (out_host) {
      ok = ok && cudaStreamWaitEvent(st->cp_out, st->ev_done[b], 0) == cudaSuccess;
      ok = ok && cudaMemcpyAsync((char*)out_host + (size_t)i * qbytes, od, qm, cudaMemcpyDeviceToHost, st->cp_out) == cudaSuccess;
      ok = ok && cudaEventRecord(st->ev_out[b], st->cp_out) == cudaSuccess;
      out_pending[b] = ok;
    }
  }
  // everything joins the caller's stream again
  for (int b = 0; b < 2; ++b)
    if (out_pending[b]) ok = cudaStreamWaitEvent(s, st->ev_out[b], 0) == cudaSuccess && ok;
  const bool synced = cudaStreamSynchronize(st->cp_in) == cudaSuccess && cudaStreamSynchronize(st->cp_out) == cudaSuccess &&
                      cudaStreamSynchronize(s) == cudaSuccess;
  if (rc != LOLA_OK) return rc;
  return ok && synced ? LOLA_OK : LOLA_ERR_CUDA;
}

int lola_read_state(const lola_state* st, const lola_state_view* view, void* stream) {
  if (!st || !view) return LOLA_ERR_ARG;
  const lola_config& c = st->cfg;
  const Layer& L = st->L;
  const size_t U = (size_t)c.batch * c.n_kv_heads, d = c.head_dim, D = L.D, es = elem_size(c);
  const size_t lam = c.sparse, eta = c.window, cm = c.max_chunk;
  cudaStream_t s = (cudaStream_t)stream;
  // The memories of a small layer come in one copy, through a pinned buffer the state keeps (the copies into the caller's
  // pageable arrays cost about 20 us each).  The buffer serves one call at a time
  std::unique_lock<std::mutex> lock(st->pin_mutex, std::defer_lock);
  const char* pin = nullptr;
  if (st->lay.wt <= kPinnedState) {
    lock.lock();
    if (!st->pin && cudaMallocHost((void**)&st->pin, st->lay.wt) != cudaSuccess) { cudaGetLastError(); st->pin = nullptr; }
    pin = st->pin;
    if (pin && (cudaMemcpyAsync(st->pin, st->base, st->lay.wt, cudaMemcpyDeviceToHost, s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)) return LOLA_ERR_CUDA;
  }
  auto d2h = [&](void* dst, const void* src, size_t bytes) {
    if (!dst || bytes == 0) return true;
    if (pin) { std::memcpy(dst, pin + ((const char*)src - st->base), bytes); return true; }
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s) == cudaSuccess;
  };
  bool ok = true;
  ok = ok && d2h(view->H, L.H, U * D * d * 4);
  ok = ok && d2h(view->s, L.s, U * D * 4);
  ok = ok && d2h(view->sparse_pos, L.gpos, U * lam * 4);
  ok = ok && d2h(view->sparse_k, L.gk, U * lam * d * es);
  ok = ok && d2h(view->sparse_v, L.gv, U * lam * d * es);
  ok = ok && d2h(view->window_k, L.wk, U * eta * d * es);
  ok = ok && d2h(view->window_v, L.wv, U * eta * d * es);
  ok = ok && d2h(view->threshold, L.thr, U * 2 * 4);
  int status = 0;
  ok = ok && d2h(&status, L.status, 4);
  if (view->sparse_score && lam > 0 && pin) {   // the first lambda entries of each unit's score row
    for (size_t u = 0; u < U; ++u) d2h(view->sparse_score + u * lam, L.score + u * (lam + cm), lam * 4);
  } else if (view->sparse_score && lam > 0) {
    ok = ok && cudaMemcpy2DAsync(view->sparse_score, lam * 4, L.score, (lam + cm) * 4, lam * 4, U,
                                 cudaMemcpyDeviceToHost, s) == cudaSuccess;
  }
  if (!ok || cudaStreamSynchronize(s) != cudaSuccess) return LOLA_ERR_CUDA;
  const int g_cw = (int)std::min<int64_t>(c.window, st->n_seen), g_count = (int)std::min<int64_t>(c.sparse, st->n_seen - g_cw);
  for (size_t u = 0; u < U; ++u) {
    if (view->sparse_count) view->sparse_count[u] = g_count;
    if (view->window_count) view->window_count[u] = g_cw;
    if (view->window_pos) {
      for (size_t j = 0; j < eta; ++j) view->window_pos[u * eta + j] = -1;
      for (int64_t p = st->n_seen - g_cw; p < st->n_seen; ++p) view->window_pos[u * eta + (size_t)(p % (int64_t)eta)] = (int32_t)p;
    }
  }
  if (view->n_seen) for (int b = 0; b < c.batch; ++b) view->n_seen[b] = st->n_seen;
  if (view->status) view->status[0] = status;
  return status == 0 ? LOLA_OK : LOLA_ERR_DEVICE;
}

int lola_write_state(lola_state* st, const lola_state_view* v, void* stream) {
  if (!st || !v) return LOLA_ERR_ARG;
  if (!v->H || !v->s || !v->sparse_count || !v->window_count || !v->n_seen) return LOLA_ERR_ARG;
  const lola_config& c = st->cfg;
  const Layer& L = st->L;
  const size_t U = (size_t)c.batch * c.n_kv_heads, d = c.head_dim, D = L.D, es = elem_size(c);
  const size_t lam = c.sparse, eta = c.window, cm = c.max_chunk;
  if (lam > 0 && (!v->sparse_pos || !v->sparse_k || !v->sparse_v)) return LOLA_ERR_ARG;
  if (eta > 0 && (!v->window_pos || !v->window_k || !v->window_v)) return LOLA_ERR_ARG;
  const int64_t n_seen = v->n_seen[0];
  if (n_seen < 0 || n_seen > 0x7fffffffLL) return LOLA_ERR_ARG;
  for (int b = 0; b < c.batch; ++b) if (v->n_seen[b] != n_seen) return LOLA_ERR_ARG;
  const int g_cw = (int)std::min<int64_t>(c.window, n_seen), g_count = (int)std::min<int64_t>(c.sparse, n_seen - g_cw);
  for (size_t u = 0; u < U; ++u) {
    if (v->sparse_count[u] != g_count || v->window_count[u] != g_cw) return LOLA_ERR_ARG;
  }
  // window rows to ring order
  std::vector<char> wk(U * eta * d * es, 0), wv(U * eta * d * es, 0);
  for (size_t u = 0; u < U && eta > 0; ++u) {
    std::vector<char> seen(eta, 0);
    for (int j = 0; j < g_cw; ++j) {
      int64_t p = v->window_pos[u * eta + j];
      if (p < n_seen - g_cw || p >= n_seen) return LOLA_ERR_ARG;
      size_t slot = (size_t)(p % (int64_t)eta);
      if (seen[slot]) return LOLA_ERR_ARG;
      seen[slot] = 1;
      std::memcpy(&wk[(u * eta + slot) * d * es], (const char*)v->window_k + (u * eta + j) * d * es, d * es);
      std::memcpy(&wv[(u * eta + slot) * d * es], (const char*)v->window_v + (u * eta + j) * d * es, d * es);
    }
  }
  std::vector<float> sc(U * (lam + cm));
  { uint32_t nanbits = 0xFFFFFFFFu; float nanv; std::memcpy(&nanv, &nanbits, 4); std::fill(sc.begin(), sc.end(), nanv); }
  if (v->sparse_score)
    for (size_t u = 0; u < U; ++u) std::memcpy(&sc[u * (lam + cm)], v->sparse_score + u * lam, lam * 4);
  cudaStream_t s = (cudaStream_t)stream;
  auto h2d = [&](void* dst, const void* src, size_t bytes) {
    if (bytes == 0) return true;
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s) == cudaSuccess;
  };
  bool ok = true;
  ok = ok && h2d(L.H, v->H, U * D * d * 4);
  ok = ok && h2d(L.s, v->s, U * D * 4);
  ok = ok && h2d(L.gpos, v->sparse_pos, U * lam * 4);
  ok = ok && h2d(L.gk, v->sparse_k, U * lam * d * es);
  ok = ok && h2d(L.gv, v->sparse_v, U * lam * d * es);
  ok = ok && h2d(L.score, sc.data(), sc.size() * 4);
  ok = ok && h2d(L.wk, wk.data(), wk.size());
  ok = ok && h2d(L.wv, wv.data(), wv.size());
  if (v->threshold) ok = ok && h2d(L.thr, v->threshold, U * 2 * 4);
  ok = ok && cudaMemsetAsync(L.status, 0, 4, s) == cudaSuccess;      // a replaced state starts healthy
  if (!ok || cudaStreamSynchronize(s) != cudaSuccess) return LOLA_ERR_CUDA;   // host staging dies here
  st->n_seen = n_seen;
  return LOLA_OK;
}

int lola_profile_enable(lola_state* st, int enable) {
  if (!st) return LOLA_ERR_ARG;
  st->profiling = enable != 0;
  return LOLA_OK;
}

int lola_profile_read(lola_state* st, double* ms_by_kind, int64_t* launches_by_kind, void* stream) {
  if (!st || !ms_by_kind || !launches_by_kind) return LOLA_ERR_ARG;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return LOLA_ERR_CUDA;
  for (int i = 0; i < LOLA_N_KERNEL_KINDS; ++i) { ms_by_kind[i] = 0.0; launches_by_kind[i] = 0; }
  int rc = LOLA_OK;
  for (ProfRecord& r : st->records) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.a, r.b) != cudaSuccess) rc = LOLA_ERR_CUDA;
    else if (r.kind >= 0 && r.kind < LOLA_N_KERNEL_KINDS) { ms_by_kind[r.kind] += ms; launches_by_kind[r.kind]++; }
    st->pool.push_back(r);
  }
  st->records.clear();
  return rc;
}

int64_t lola_launch_count(const lola_state* st) { return st ? st->launches : -1; }
int64_t lola_tokens_seen(const lola_state* st) { return st ? st->n_seen : -1; }

int lola_set_tokens_seen(lola_state* st, int64_t n_seen) {
  if (!st) return LOLA_ERR_ARG;
  if (n_seen < 0 || n_seen > 0x7fffffffLL) return LOLA_ERR_SHAPE;
  st->n_seen = n_seen;
  return LOLA_OK;
}

int lola_last_call_info(const lola_state* st, lola_call_info* out) {
  if (!st || !out) return LOLA_ERR_ARG;
  *out = st->info;
  return LOLA_OK;
}

int lola_selftest_wait_timeout(lola_state* st, int32_t limit_us, void* stream) {
  if (!st) return LOLA_ERR_ARG;
  if (limit_us < 1 || limit_us > 250000) return LOLA_ERR_ARG;
  st->launches++;
  k_selftest_wait<<<1, 32, 0, (cudaStream_t)stream>>>(st->L.status, (unsigned long long)limit_us * 1000ull);
  return cudaGetLastError() == cudaSuccess ? LOLA_OK : LOLA_ERR_CUDA;
}

int lola_destroy_state(lola_state* st) {
  if (!st) return LOLA_ERR_ARG;
  for (auto* v : {&st->records, &st->pool})
    for (ProfRecord& r : *v) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
  if (st->cp_in) { cudaStreamSynchronize(st->cp_in); cudaStreamDestroy(st->cp_in); }
  if (st->cp_out) { cudaStreamSynchronize(st->cp_out); cudaStreamDestroy(st->cp_out); }
  for (cudaEvent_t e : {st->ev_start, st->ev_in[0], st->ev_in[1], st->ev_done[0], st->ev_done[1], st->ev_out[0], st->ev_out[1]})
    if (e) cudaEventDestroy(e);
  if (st->pin) cudaFreeHost(st->pin);
  delete st;
  return LOLA_OK;
}

// ---------------------------------------------------------------------------------------------
// Generation step whose per-call work lists live in library-owned static device memory.
//
// g_static_lists is a host-side stand-in for the device array: its address means nothing to a
// kernel.  The device address is resolved once per device with cudaGetSymbolAddress and handed
// to the kernels through the Layer block.
// three work lists of LOLA_STATIC_MAX_LIST_ENTRIES ints, then 4 counters per unit
static __device__ __align__(256) int g_static_lists[3 * LOLA_STATIC_MAX_LIST_ENTRIES + 4 * LOLA_STATIC_MAX_UNITS];

static int* static_lists_for_current_device(int* rc_out) {
  static int* ptrs[64] = {nullptr};
  static std::mutex mu;                // first calls from several host threads look the address up one at a time
  std::lock_guard<std::mutex> lock(mu);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { *rc_out = LOLA_ERR_CUDA; return nullptr; }
  if (!ptrs[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_lists) != cudaSuccess || !p) { *rc_out = LOLA_ERR_CUDA; return nullptr; }
    ptrs[dev] = (int*)p;
  }
  *rc_out = LOLA_OK;
  return ptrs[dev];
}

int lola_decode_step_static(lola_state* st, const void* q, const void* k, const void* v, void* out, void* stream) {
  if (!st) return LOLA_ERR_ARG;
  const int64_t U = (int64_t)st->cfg.batch * st->cfg.n_kv_heads;
  if (U > LOLA_STATIC_MAX_UNITS || U * st->cfg.max_chunk > LOLA_STATIC_MAX_LIST_ENTRIES) return LOLA_ERR_SIZE;
  int rc = LOLA_OK;
  int* base = static_lists_for_current_device(&rc);
  if (!base) return rc;
  // Same kernels, same launches as lola_decode_step; only the four work-list pointers differ.
  // Every entry a kernel reads in a step is written earlier in the same step (the selection kernel
  // fills the lists and both counters before the update kernel reads them), so nothing has to be
  // cleared between calls even though the array keeps the previous call's contents.
  const Layer saved = st->L;
  st->L.fold_idx = base;
  st->L.move_src = base + LOLA_STATIC_MAX_LIST_ENTRIES;
  st->L.move_dst = base + 2 * LOLA_STATIC_MAX_LIST_ENTRIES;
  st->L.counts = base + 3 * LOLA_STATIC_MAX_LIST_ENTRIES;
  st->force_chain = true;              // the kernel chain is the path that passes work lists between kernels
  rc = lola_decode_step(st, q, k, v, out, stream);
  st->force_chain = false;
  st->L = saved;                       // kernel arguments were copied at launch
  return rc;
}

const char* lola_strerror(int code) {
  switch (code) {
    case LOLA_OK: return "ok";
    case LOLA_ERR_ARG: return "invalid argument (null pointer, bad enum or inconsistent state view)";
    case LOLA_ERR_SHAPE: return "size out of range";
    case LOLA_ERR_ALIGN: return "pointer not sufficiently aligned";
    case LOLA_ERR_SIZE: return "caller-provided buffer too small";
    case LOLA_ERR_UNSUPPORTED: return "shape or device not supported by this build (needs sm_100)";
    case LOLA_ERR_CUDA: return "CUDA runtime call or kernel launch failed";
    case LOLA_ERR_DEVICE: return "a kernel recorded an internal error in the state's status word";
    default: return "unknown error code";
  }
}

}  // extern "C"
