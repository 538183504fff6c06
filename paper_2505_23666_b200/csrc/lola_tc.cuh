// Building blocks for the sm_100a tensor-core kernels: tcgen05.mma with operands in shared memory
// (128-byte swizzled canonical layouts), accumulators in tensor memory, mbarrier completion with
// bounded waits.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace lola {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- operand tiles ---------------------------------------------------------------------------
// A tile is a stack of "blocks"; a block is R rows of 128 bytes (64 bf16), and inside every group
// of 8 rows the eight 16-byte chunks of a row are XOR-swizzled with (row & 7).  The same bytes serve
//   * a K-major operand  [R (M or N) x 64 (K)]: rows are M/N indices, SBO = 1024 (8 rows), and
//   * an MN-major operand [64 (M or N) x R (K)]: rows are K indices, SBO = 1024, LBO = block bytes,
// which is also what a TMA box of 64 x R elements with 128-byte swizzle writes.
__device__ __forceinline__ uint32_t sw128_off(int row, int chunk) { return (uint32_t)row * 128u + (uint32_t)((chunk ^ (row & 7)) << 4); }

__device__ __forceinline__ uint64_t make_desc_sw128(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for sm_100
  d |= (uint64_t)2 << 61;  // 128-byte swizzle
  return d;
}

// kind::f16 instruction descriptor: bf16 x bf16 -> fp32, M x N tile.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, bool a_mn_major, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One lane of a converged warp (always the same one).  Knowing that one thread is left, the compiler hands the operands of MMAs
// and TMA requests over without a loop over lanes: 8 MMAs take their thread 200 cycles, not 474 as with "lane == 0", a request 52
// and not 100 (idle SM).  Taken where it measured faster: the roles of k_prefill_run and what requests tiles in k_prefill_team;
// the issuing threads of the other kernels, whose products follow each other closely, were 1 - 4% slower with it.
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile(
      "{\n\t"
      ".reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}\n"
      : "=r"(one));
  return one != 0;
}
__device__ __forceinline__ void mma_bf16_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t"
      ".reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "}\n" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Same product with the A operand in tensor memory (M = 128 lanes, two bf16 per 32-bit column,
// lower K index in the low half): one instruction consumes 8 columns (K = 16).
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t"
      ".reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
      "}\n" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[M x N] (+)= A[M x K] * B[N x K]^T with both operands K-major, K a multiple of 16.
// a_base / b_base: shared addresses of the first 64-wide K block; *_blk_bytes: bytes per K block.
__device__ __forceinline__ void mma_kmajor(uint32_t d_tmem, uint32_t a_base, uint32_t a_blk_bytes, uint32_t b_base,
                                           uint32_t b_blk_bytes, int K, uint32_t idesc, bool accumulate_first) {
  for (int k = 0; k < K; k += 16) {
    uint32_t ao = (uint32_t)(k >> 6) * a_blk_bytes + (uint32_t)(k & 63) * 2u;
    uint32_t bo = (uint32_t)(k >> 6) * b_blk_bytes + (uint32_t)(k & 63) * 2u;
    mma_bf16_ss(d_tmem, make_desc_sw128(a_base + ao, 16, 1024), make_desc_sw128(b_base + bo, 16, 1024), idesc,
                (k > 0 || accumulate_first) ? 1u : 0u);
  }
}

// D[M x N] (+)= A[M x K] * B with A K-major and B MN-major (stored [K rows][N], 64-wide N blocks).
__device__ __forceinline__ void mma_a_kmajor_b_mnmajor(uint32_t d_tmem, uint32_t a_base, uint32_t a_blk_bytes,
                                                       uint32_t b_base, uint32_t b_blk_bytes, int K, uint32_t idesc,
                                                       bool accumulate_first) {
  for (int k = 0; k < K; k += 16) {
    uint32_t ao = (uint32_t)(k >> 6) * a_blk_bytes + (uint32_t)(k & 63) * 2u;
    uint32_t bo = (uint32_t)k * 128u;   // 16 K rows of 128 bytes
    mma_bf16_ss(d_tmem, make_desc_sw128(a_base + ao, 16, 1024), make_desc_sw128(b_base + bo, b_blk_bytes, 1024), idesc,
                (k > 0 || accumulate_first) ? 1u : 0u);
  }
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// makes shared-memory writes of this thread visible to the tensor-core / TMA (async) proxy
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- tensor memory ---------------------------------------------------------------------------
// One warp allocates `cols` (power of two >= 32) columns and publishes the base address in shared memory.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_smem)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

// 32 lanes x 32 consecutive fp32 columns: thread i of the warp receives row (lane base + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])),
      "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])),
      "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
      "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])), "r"(__float_as_uint(v[27])),
      "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---- mbarrier --------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");
  return t;
}

// Waits for the phase with the given parity to complete.  Gives up after about a quarter of a second
// and returns false; the caller records the failure and carries on to its cleanup.  With an abort
// word (shared memory) the first wait that gives up raises it and every other wait of the CTA that
// polls it returns false at once, so one lost signal cannot add up to many timeouts.
// The polling loop is a real function (one copy per kernel): the kernels wait in dozens of places and
// their instruction footprint matters.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t"
      ".reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
constexpr unsigned long long kWaitLimitNs = 250000000ull;
constexpr uint32_t kSuspendNs = 20000;
// The same with a suspend-time hint: the thread sleeps in the hardware until the phase completes or the time is over.
// A waiting warp that comes back every few hundred cycles to ask again takes issue slots from the warps that work: up to
// half of all instructions of the role pipelines were such loops.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t"
      ".reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return done != 0;
}
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_word,
                                            unsigned long long limit_ns = kWaitLimitNs) {
  unsigned long long deadline = 0;
  for (;;) {
    if (mbar_try_wait_suspend(bar, parity)) return true;
    if (abort_word && *abort_word) return false;
    const unsigned long long now = global_ns();
    if (deadline == 0) deadline = now + limit_ns;
    else if (now > deadline) {
      if (abort_word) *abort_word = 1;
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_word = nullptr) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort_word);
}

// ---- TMA (bulk tensor copies global -> shared, completion on an mbarrier) ------------------------
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One box of a rank-3 tensor map; c0 is the innermost (element) coordinate and must keep the source
// address 16-byte aligned (a multiple of 8 for 16-bit elements).  Out-of-range rows read as zero.
__device__ __forceinline__ void tma_load_3d(uint32_t dst_smem, const void* tmap, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst_smem), "l"((uint64_t)(uintptr_t)tmap), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst_smem, const void* tmap, int c0, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst_smem), "l"((uint64_t)(uintptr_t)tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst_smem, const void* tmap, int c0, int c1, int c2, int c3, int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
      ::"r"(dst_smem), "l"((uint64_t)(uintptr_t)tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
// Tensor maps of a sparse cache [units][slots][d].  A tile is 128 rows of all columns, [d / 64][128 rows][128 bytes] in shared
// memory.  A request takes its issuing thread 100 cycles on an idle SM and some 300 beside working warps, whatever its size,
// so a tile that lies in the cache as a whole is one request, not four of 64 rows x 64 columns: eight of those a tile (keys and
// values) held the tiles of a prefill run apart (a chunk of 8 units, d = 128: 19.6 us, with whole tiles and elect_one 18.6; 64
// units: 28.2 and 27.7).
struct SlotMaps {
  CUtensorMap block;             // rank 3, boxes of 64 rows x 64 columns
  CUtensorMap tile;              // rank 4 (column, row, block of 64 columns, unit), boxes of 128 rows x all columns
};
// Tile `tile` (all 128 of its rows are places of sparse-cache blocks)
__device__ __forceinline__ void tma_load_slots(uint32_t dst_smem, const SlotMaps* m, int tile, int unit, uint32_t bar) {
  tma_load_4d(dst_smem, &m->tile, 0, tile * 128, 0, unit, bar);
}
// One box of a rank-4 tensor map, shared -> global (bulk async-group completion).  Rows of the box that lie
// outside the tensor are not written.  c0 as for the loads (16-byte aligned start); no negative coordinates.
__device__ __forceinline__ void tma_store_4d(const void* tmap, uint32_t src_smem, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"((uint64_t)(uintptr_t)tmap),
               "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(src_smem)
               : "memory");
}
__device__ __forceinline__ void tma_store_5d(const void* tmap, uint32_t src_smem, int c0, int c1, int c2, int c3, int c4) {
  asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];" ::"l"((uint64_t)(uintptr_t)tmap),
               "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(src_smem)
               : "memory");
}

// Linear bulk copy global -> shared (addresses and size multiples of 16 bytes), completion on an mbarrier.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"((uint64_t)(uintptr_t)src), "r"(bytes), "r"(bar)
               : "memory");
}
// adds four floats to memory, where they are (16-byte aligned); complete by the end of the kernel
__device__ __forceinline__ void red_add_v4(float* dst, float4 v) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// (the copies have read their shared-memory source; their writes complete with the kernel at the latest)
__device__ __forceinline__ void bulk_wait_group_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Programmatic dependent launch: a kernel launched with programmatic stream serialization may start
// while the kernel before it in the stream still runs; it must pass grid_dep_wait() before it touches
// anything that kernel (or an earlier one) produces or still reads.  Both are no-ops in a normal launch.
__device__ __forceinline__ void grid_dep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// asks for bytes (a multiple of 16, 16-byte aligned) to be brought into the L2
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ---- thread-block clusters ---------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
// the address of the same shared-memory location in block `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
// a store into another block's shared memory that counts 4 bytes on an mbarrier of that block (addresses from map_rank):
// data and signal in one trip, no fence
__device__ __forceinline__ void st_async_u32(uint32_t addr, uint32_t v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
               : "memory");
}
// 16 bytes global -> shared memory without registers (through the L2; bytes = 0: zeros), and the wait for this thread's
__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src, uint32_t bytes = 16) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// bulk copy from this block's shared memory into another's (dst and bar: addresses from map_rank; 16-byte units)
__device__ __forceinline__ void bulk_copy_s2peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// loads from another block's shared memory (addresses from map_rank)
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) { uint32_t v; asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory"); return v; }
__device__ __forceinline__ uint4 ld_cluster_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
// every thread of every block of the cluster (whole warps, converged)
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Whether the first block of the cluster has found an earlier failure (word: an address in every block's shared memory, where
// it has left it).  Starts and ends with a cluster barrier: all blocks run, and nobody leaves before all have read it.
__device__ __noinline__ bool cluster_failed(uint32_t word) {
  cluster_arrive();
  cluster_wait();
  const bool f = ld_cluster_u32(map_rank(word, 0)) != 0u;
  cluster_arrive();
  cluster_wait();
  return f;
}
// makes this thread's generic-proxy writes (shared and global memory) visible to the async proxy and back
__device__ __forceinline__ void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

// ---- narrower tensor-memory accesses ------------------------------------------------------------
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(taddr),
               "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
               "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
               "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
               : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 lanes x 64 consecutive fp32 columns (two loads, one wait)
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
  uint32_t r[64];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr), "r"(taddr + 32u)
      : "memory");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
        "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float (&v)[2]) {
  uint32_t r0, r1;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n\ttcgen05.wait::ld.sync.aligned;\n"
               : "=r"(r0), "=r"(r1) : "r"(taddr) : "memory");
  v[0] = __uint_as_float(r0);
  v[1] = __uint_as_float(r1);
}

// raw 32-bit variants (packed bf16 pairs)
__device__ __forceinline__ void tmem_st32u(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n\ttcgen05.wait::st.sync.aligned;\n"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]) : "memory");
}
__device__ __forceinline__ void tmem_ld32u(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\ttcgen05.wait::ld.sync.aligned;\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]) : "r"(taddr) : "memory");
}

// raw 32-bit: 64 consecutive columns (two loads, one wait)
__device__ __forceinline__ void tmem_ld64u(uint32_t taddr, uint32_t (&r)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr), "r"(taddr + 32u)
      : "memory");
}
// 64 consecutive columns at taddr and 4 more at zaddr (raw 32-bit), three loads under one wait
__device__ __forceinline__ void tmem_ld64u_and4(uint32_t taddr, uint32_t (&r)[64], uint32_t zaddr, uint32_t (&z)[4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%64, %65, %66, %67}, [%70];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%68];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%69];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]), "=r"(z[0]), "=r"(z[1]), "=r"(z[2]), "=r"(z[3])
      : "r"(taddr), "r"(taddr + 32u), "r"(zaddr)
      : "memory");
}
// 64 consecutive columns at taddr and 2 more at zaddr (raw 32-bit), three loads under one wait
__device__ __forceinline__ void tmem_ld64u_and2(uint32_t taddr, uint32_t (&r)[64], uint32_t zaddr, uint32_t (&z)[2]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%64, %65}, [%68];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%66];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%67];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]), "=r"(z[0]), "=r"(z[1])
      : "r"(taddr), "r"(taddr + 32u), "r"(zaddr)
      : "memory");
}
// 32 consecutive columns at taddr and 2 more at zaddr (raw 32-bit), two loads under one wait
__device__ __forceinline__ void tmem_ld32u_and2(uint32_t taddr, uint32_t (&r)[32], uint32_t zaddr, uint32_t (&z)[2]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%32, %33}, [%35];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%34];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(z[0]), "=r"(z[1])
      : "r"(taddr), "r"(zaddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
  uint32_t r0, r1, r2, r3;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(taddr) : "memory");
  v[0] = __uint_as_float(r0); v[1] = __uint_as_float(r1); v[2] = __uint_as_float(r2); v[3] = __uint_as_float(r3);
}

// named barrier over `count` threads (ids 1..15; 0 is __syncthreads)
__device__ __forceinline__ void named_bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int count) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory"); }

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- packed fp32 pairs (one instruction works on two values) ------------------------------------
__device__ __forceinline__ uint64_t pack_f2(float a, float b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ uint64_t pack_u2(uint32_t a, uint32_t b) { uint64_t r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ void unpack_f2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) { uint64_t d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d; }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t d; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t d; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b)); return d; }
__device__ __forceinline__ float max3(float a, float b, float c) { float d; asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d; }

// One half of the feature map (Eq. 6) of one row: 64 pre-activations u (raw fp32 bits) -> 64 bf16
// values as 32 packed pairs.  neg = false: softmax(u), neg = true: softmax(-u); exp_kind: exp(+-u)
// without the normalisation.  Four running sums (elements 4k, 4k+1, 4k+2, 4k+3), added pairwise.
// One instruction stream serves both signs (the sign is data): the two threads of a row run the same
// code, which keeps the instruction footprint of the kernels small.  Packed f32x2 instructions: half
// the instructions of the plain forms (each thread's instruction stream, not the pipes, bounds this phase).
__device__ __forceinline__ uint64_t phi_half_f32(const uint32_t (&u)[64], bool neg, bool exp_kind, uint64_t (&x2)[32]) {
  const float kL = neg ? -1.4426950408889634f : 1.4426950408889634f;
  const uint64_t sc2 = pack_f2(kL, kL);
#pragma unroll
  for (int q = 0; q < 32; ++q) x2[q] = mul2(pack_u2(u[2 * q], u[2 * q + 1]), sc2);   // u * kL, in log2 units
  float mm = 0.f;
  if (!exp_kind) {
    float a, b;
    unpack_f2(x2[0], a, b);
#pragma unroll
    for (int q = 1; q < 31; q += 2) {
      float c0, c1, c2, c3;
      unpack_f2(x2[q], c0, c1);
      unpack_f2(x2[q + 1], c2, c3);
      a = max3(a, c0, c1);
      b = max3(b, c2, c3);
    }
    float c0, c1;
    unpack_f2(x2[31], c0, c1);
    mm = fmaxf(max3(a, c0, c1), b);
  }
  const uint64_t off2 = pack_f2(-mm, -mm);
  uint64_t acc0 = pack_f2(0.f, 0.f), acc1 = acc0;
#pragma unroll
  for (int q = 0; q < 32; q += 2) {
    float x0, x1, x2f, x3;
    unpack_f2(add2(x2[q], off2), x0, x1);
    unpack_f2(add2(x2[q + 1], off2), x2f, x3);
    x2[q] = pack_f2(fast_exp2(x0), fast_exp2(x1));
    x2[q + 1] = pack_f2(fast_exp2(x2f), fast_exp2(x3));
    acc0 = add2(acc0, x2[q]);
    acc1 = add2(acc1, x2[q + 1]);
  }
  float inv = 1.0f;
  if (!exp_kind) {
    float s0, s1, s2, s3;
    unpack_f2(acc0, s0, s1);
    unpack_f2(acc1, s2, s3);
    inv = 1.0f / ((s0 + s1) + (s2 + s3));
  }
  return pack_f2(inv, inv);
}
__device__ __forceinline__ void phi_half(const uint32_t (&u)[64], bool neg, bool exp_kind, uint32_t (&out)[32]) {
  uint64_t x2[32];
  const uint64_t inv2 = phi_half_f32(u, neg, exp_kind, x2);
#pragma unroll
  for (int q = 0; q < 32; ++q) {
    float lo, hi;
    unpack_f2(exp_kind ? x2[q] : mul2(x2[q], inv2), lo, hi);
    __nv_bfloat162 pr = __floats2bfloat162_rn(lo, hi);
    out[q] = *reinterpret_cast<uint32_t*>(&pr);
  }
}
// [dH | ds] = phi^T [V | 1] of up to 64 pairs (one thread), overwriting the accumulator.  phi: [2 feature blocks][128 rows][128B], first parts
// in rows 0-63, second ones in 64-127; v: [d / 64 + 1 column blocks][128 rows][128B], the pairs in rows 0-63, the third parts of
// phi (if taken) in rows 64-127 of the first two blocks.  A product adds to its accumulator with truncation, 2^-25 of it
// per K step and always towards zero: with all 24 bits of phi the small parts go first, so that 4 steps of 12 see the full sum,
// and batches are added up outside (error of H's norm after 5 chunks of 48 folds 2.3e-7, with the small parts last 3.9e-7; 5
// chunks of 256 folds 2.0e-7, in one accumulator 1.1e-6; by fp32 on the CUDA cores 1.9e-7 and 3.2e-7).
template <int DPL, bool THREE>
__device__ __forceinline__ void fold_product(uint32_t acc, uint32_t phi, uint32_t v, bool three) {
  constexpr int d = DPL * 32;
  const uint32_t id = make_idesc_bf16(128, d + 16, true, true);
  auto step = [&](uint32_t a, int ks, uint32_t add) {
    mma_bf16_ss(acc, make_desc_sw128(a + ks * 2048, 16384, 1024), make_desc_sw128(v + ks * 2048, 16384, 1024), id, add);
  };
  if (THREE && three) {
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) step(v + 8192u, ks, ks > 0);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) step(phi + 8192u, ks, 1u);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) step(phi, ks, 1u);
  } else {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
      mma_bf16_ss(acc, make_desc_sw128(phi + ks * 2048, 16384, 1024), make_desc_sw128(v + (ks & 3) * 2048, 16384, 1024), id, ks > 0);
  }
}
// 32 of the 64 pre-activations of a half: exp(+-u - m) against their own maximum m (log2 units; 0 for exp_kind) as packed
// pairs and their sum.
__device__ __forceinline__ void phi_quarter_f32(const uint32_t (&u)[32], bool neg, bool exp_kind, uint64_t (&x2)[16], float& m, float& sum) {
  const float kL = neg ? -1.4426950408889634f : 1.4426950408889634f;
  const uint64_t sc2 = pack_f2(kL, kL);
  float a = -CUDART_INF_F, b = -CUDART_INF_F;
#pragma unroll
  for (int q = 0; q < 16; q += 2) {
    x2[q] = mul2(pack_u2(u[2 * q], u[2 * q + 1]), sc2);
    x2[q + 1] = mul2(pack_u2(u[2 * q + 2], u[2 * q + 3]), sc2);
    float c0, c1, c2, c3;
    unpack_f2(x2[q], c0, c1);
    unpack_f2(x2[q + 1], c2, c3);
    a = max3(a, c0, c1);
    b = max3(b, c2, c3);
  }
  m = exp_kind ? 0.f : fmaxf(a, b);
  const uint64_t off2 = pack_f2(-m, -m);
  uint64_t acc0 = pack_f2(0.f, 0.f), acc1 = acc0;
#pragma unroll
  for (int q = 0; q < 16; q += 2) {
    float x0, x1, x2f, x3;
    unpack_f2(add2(x2[q], off2), x0, x1);
    unpack_f2(add2(x2[q + 1], off2), x2f, x3);
    x2[q] = pack_f2(fast_exp2(x0), fast_exp2(x1));
    x2[q + 1] = pack_f2(fast_exp2(x2f), fast_exp2(x3));
    acc0 = add2(acc0, x2[q]);
    acc1 = add2(acc1, x2[q + 1]);
  }
  float s0, s1, s2, s3;
  unpack_f2(acc0, s0, s1);
  unpack_f2(acc1, s2, s3);
  sum = (s0 + s1) + (s2 + s3);
}
// A pair of fp32 values in three bf16 parts whose sum has all of their 24 bits: what is left of (a, b) goes on to the next part.
__device__ __forceinline__ uint32_t next_part(float& a, float& b) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h2);
  a -= hf.x;
  b -= hf.y;
  return *reinterpret_cast<const uint32_t*>(&h2);
}
__device__ __forceinline__ uint32_t phi_part(uint64_t ab, bool second) {   // the first or the second part
  float a, b;
  unpack_f2(ab, a, b);
  uint32_t part = next_part(a, b);
  if (second) part = next_part(a, b);
  return part;
}
__device__ __forceinline__ uint32_t phi_third(uint64_t ab) {
  float a, b;
  unpack_f2(ab, a, b);
  next_part(a, b);
  next_part(a, b);
  return next_part(a, b);
}

// 8 fp32 -> 8 bf16 packed in a uint4 (element 0 in the low half of x)
__device__ __forceinline__ uint4 pack8_bf16(const float* f) {
  __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]);
  __nv_bfloat162 b = __floats2bfloat162_rn(f[2], f[3]);
  __nv_bfloat162 c = __floats2bfloat162_rn(f[4], f[5]);
  __nv_bfloat162 d = __floats2bfloat162_rn(f[6], f[7]);
  uint4 o;
  o.x = *reinterpret_cast<uint32_t*>(&a);
  o.y = *reinterpret_cast<uint32_t*>(&b);
  o.z = *reinterpret_cast<uint32_t*>(&c);
  o.w = *reinterpret_cast<uint32_t*>(&d);
  return o;
}

}  // namespace tc

// warp-wide maximum / minimum of fp32 values through the integer reduction instruction
__device__ __forceinline__ int f2ord(float x) { int i = __float_as_int(x); return i ^ ((i >> 31) & 0x7fffffff); }
__device__ __forceinline__ float ord2f(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }
__device__ __forceinline__ float warp_max_redux(float x) { return ord2f(__reduce_max_sync(0xffffffffu, f2ord(x))); }

// two fp32 -> packed bf16x2 (a in the low half), and the rounded values back as fp32 by bit moves
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&p);
}
__device__ __forceinline__ float bf16lo_f(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf16hi_f(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }

}  // namespace lola
