// tcgen05 BF16 GEMM (TMA -> shared memory -> tcgen05.mma -> TMEM -> registers) and the
// BF16 H_eff chain built on it (sm_103a).
//
//   D[m][n] = sum_k A[m][k] * B[n][k]      A: M x K, B: N x K, both K-major BF16,
//   FP32 accumulation in tensor memory, epilogue stores BF16 or FP32 (plain or atomic).
//
// A persistent kernel (one CTA of 192 threads per SM) walks the 128 x BN output tiles
// (and their K splits): warp 0 lane 0 issues TMA loads into a STAGES-deep ring of
// 128B-swizzled tiles, warp 1 lane 0 issues tcgen05.mma (M=128, N=BN, K=16 per
// instruction) into one of two TMEM accumulators, and warps 2..5 drain the other one.
// Every mbarrier wait is bounded; a timeout raises a device error flag, every role
// leaves its loop, the in-flight copies and MMAs are waited for, TMEM is freed.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "tc_gemm.cuh"

namespace a2 {

namespace tc {

constexpr int BM = 128;
constexpr int BK = 64;              // 64 bf16 = 128 bytes = one swizzle row
constexpr uint32_t kWaitLimit = 1u << 26;

__device__ int g_tc_error = 0;     // set to a nonzero code when a bounded wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: returns false (and records `code`) if the phase never completes.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int code,
                                          uint32_t limit = kWaitLimit) {
  for (uint32_t it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (it > 64) __nanosleep(64);
  }
  atomicCAS(&g_tc_error, 0, code);   // the first wait that gave up is reported
  return false;
}

__device__ __forceinline__ void tma_load_2d(const CUtensorMap* map, uint64_t* bar, void* dst,
                                            int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(const CUtensorMap* map, uint64_t* bar, void* dst,
                                            int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(const CUtensorMap* map, uint64_t* bar, void* dst,
                                            int x, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
  const uint64_t addr = smem_u32(p);
  uint64_t d = 0;
  d |= (addr >> 4) & 0x3FFFull;            // start address
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                  // descriptor version for tcgen05
  d |= (uint64_t)2 << 61;                  // SWIZZLE_128B
  return d;
}

// Instruction descriptor, kind::f16: BF16 x BF16 -> FP32, both operands K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4)                     // D format F32
         | (1u << 7)                   // A format BF16
         | (1u << 10)                  // B format BF16
         | ((uint32_t)(N >> 3) << 17)  // N / 8
         | ((uint32_t)(M >> 4) << 24); // M / 16
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// The same MMA in a run of MMAs on one A tile: the first keeps A in the tensor core's
// collector buffer (fill), the others take it from there (use, lastuse) instead of reading
// shared memory again.
template <bool FIRST, bool LAST>
__device__ __forceinline__ void mma_bf16_a(uint32_t tmem_d, uint64_t a, uint64_t b,
                                           uint32_t idesc, uint32_t accumulate) {
#define A2_MMA_A(op)                                                                          \
  asm volatile(                                                                               \
      "{\n\t.reg .pred p;\n\t"                                                              \
      "setp.ne.b32 p, %4, 0;\n\t"                                                             \
      "tcgen05.mma.cta_group::1.kind::f16.collector::a::" op " [%0], %1, %2, %3, p;\n\t}" ::"r"( \
          tmem_d),                                                                            \
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate))
  if constexpr (FIRST && LAST) A2_MMA_A("discard");
  else if constexpr (FIRST) A2_MMA_A("fill");
  else if constexpr (LAST) A2_MMA_A("lastuse");
  else A2_MMA_A("use");
#undef A2_MMA_A
}

// One lane of a converged warp (always the same one).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

enum OutKind { OUT_BF16 = 0, OUT_F32 = 1, OUT_F32_ATOMIC = 2 };

struct TcArgs {
  int M, N, K;
  int nk1, nk2;            // K blocks of the plain product and of the optional second segment
  int nbc2, n12;           // second segment: b' chunks per w1, (s1 s2) rows per a
  int kblocks_per_split;   // K blocks (of BK) in one work unit
  int splits;              // K splits (work units per output tile)
  void* C;
  long long ldc;
  int out_kind;
  int tma_store;           // 1: epilogue through shared memory + TMA bulk tensor store
  uint32_t wait_limit;     // iterations of every bounded wait (kWaitLimit)
  int no_loads;            // self-test only: the producer issues no copies, so the first
                           // wait of the MMA role runs out (see tc_selftest_timeout)
};

// a2 / b2: the optional second K segment, A as a 4D view [a][w1][s12][b'] (box
// 64 x n12 x 1 x 128/n12, i.e. 128 rows (a, s12) x 64 b') and B as a 3D view
// [b][w1][b'] (box 64 x 1 x BN); both land in shared memory exactly like the 2D boxes.
struct TcMaps {
  CUtensorMap a, b, a2, b2;
  CUtensorMap c;           // output (FP32 box 32 x 32 or BF16 box 64 x 32, 128B swizzle)
};

// Epilogue warps: one per TMEM lane quarter, each draining all BN columns.
constexpr int kEpi = 4;
constexpr int kTcThreads = 64 + 32 * kEpi;

template <int BN, int STAGES>
struct TcSmem {
  alignas(1024) __nv_bfloat16 a[STAGES][BM * BK];
  alignas(1024) __nv_bfloat16 b[STAGES][BN * BK];
  alignas(1024) unsigned char cbuf[kEpi][2][4096];        // epilogue staging buffers
  alignas(8) uint64_t full[STAGES];                // TMA -> MMA
  alignas(8) uint64_t empty[STAGES];               // MMA -> TMA
  alignas(8) uint64_t acc_full[2];                 // MMA -> epilogue (per TMEM buffer)
  alignas(8) uint64_t acc_empty[2];                // epilogue -> MMA
  alignas(8) uint64_t drain;                       // MMA completion on abort
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x,
                                             int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(x), "r"(y), "r"(smem_u32(src))
      : "memory");
}
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, const void* src, int x,
                                                  int y) {
  asm volatile(
      "cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%1, %2}], [%3];" ::
          "l"(reinterpret_cast<uint64_t>(map)),
      "r"(x), "r"(y), "r"(smem_u32(src))
      : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read1() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read0() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c,
                                             uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
               "r"(d)
               : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

static_assert(sizeof(TcSmem<256, 4>) + 1024 <= 227 * 1024, "BN=256 ring exceeds smem");
static_assert(sizeof(TcSmem<128, 6>) + 1024 <= 227 * 1024, "BN=128 ring exceeds smem");

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait that also gives up early once another role has raised the abort flag.
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t* bar, uint32_t parity, int code,
                                                   const int* abort_flag,
                                                   uint32_t limit = kWaitLimit) {
  for (uint32_t it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255) == 255 && *(volatile const int*)abort_flag) return false;
    if (it > 64) __nanosleep(64);
  }
  atomicCAS(&g_tc_error, 0, code);   // the first wait that gave up is reported
  return false;
}

// The same for a converged warp: every lane waits, and all get the same answer.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, int code,
                                               const int* abort_flag,
                                               uint32_t limit = kWaitLimit) {
  return __all_sync(0xffffffffu, mbar_wait_or_abort(bar, parity, code, abort_flag, limit));
}

// Persistent warp-specialised GEMM.  Work unit = (128 x BN output tile, K split); CTA c
// takes units c, c + gridDim.x, ...  Warp 0 lane 0 streams (A, B) K blocks through a
// STAGES-deep ring with TMA, warp 1 lane 0 issues tcgen05.mma into one of two TMEM
// accumulators (2 x BN columns), warps 2..5 drain the other accumulator (warp w reads
// TMEM lanes 32*(w%4)..+31) and store it, so the epilogue of one unit overlaps the MMAs
// of the next.  Every wait is bounded; a timeout raises the device error flag and all
// roles leave their loops, wait (bounded) for their copies / MMAs in flight and exit.
template <int BN, int STAGES>
__global__ void __launch_bounds__(kTcThreads, 1)
tc_gemm_kernel(const __grid_constant__ TcMaps maps, TcArgs args) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;
  auto& S = *reinterpret_cast<TcSmem<BN, STAGES>*>(smem_raw + pad);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = (args.M + BM - 1) / BM;
  const int tiles_n = (args.N + BN - 1) / BN;
  const int nk_total = args.nk1 + args.nk2;
  const int nunits = tiles_m * tiles_n * args.splits;
  constexpr uint32_t kStageBytes = (BM + BN) * BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.acc_full[i], 1);
      mbar_init(&S.acc_empty[i], kEpi);
    }
    mbar_init(&S.drain, 1);
    S.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {   // two accumulators of BN fp32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem_base)),
                 "r"((uint32_t)(2 * BN)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = S.tmem_base;

  auto unit_k = [&](int u, int& kb0, int& nkb) {
    const int sp = u / (tiles_m * tiles_n);
    kb0 = sp * args.kblocks_per_split;
    nkb = max(0, min(nk_total - kb0, args.kblocks_per_split));
  };

  if (warp == 0) {
    if (lane == 0 && !args.no_loads) {
      // ---------------- producer
      uint32_t g = 0, issued = 0;
      for (int u = blockIdx.x; u < nunits && !*(volatile int*)&S.abort_flag; u += gridDim.x) {
        const int m0 = (u % tiles_m) * BM;
        const int n0 = ((u / tiles_m) % tiles_n) * BN;
        int kb0, nkb;
        unit_k(u, kb0, nkb);
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          const int s = g % STAGES;
          const uint32_t round = g / STAGES;
          if (round > 0 &&
              !mbar_wait_or_abort(&S.empty[s], (round - 1) & 1, 1, &S.abort_flag, args.wait_limit)) {
            S.abort_flag = 1;
            break;
          }
          if (*(volatile int*)&S.abort_flag) break;
          mbar_expect_tx(&S.full[s], kStageBytes);
          const int kbg = kb0 + kb;
          if (kbg < args.nk1) {
            const int kx = kbg * BK;
            tma_load_2d(&maps.a, &S.full[s], S.a[s], kx, m0);
            tma_load_2d(&maps.b, &S.full[s], S.b[s], kx, n0);
          } else {   // second segment: K block = (w1, chunk of b')
            const int j = kbg - args.nk1;
            const int w1 = j / args.nbc2, bx = (j % args.nbc2) * BK;
            tma_load_4d(&maps.a2, &S.full[s], S.a[s], bx, 0, w1, m0 / args.n12);
            tma_load_3d(&maps.b2, &S.full[s], S.b[s], bx, w1, n0);
          }
          issued = g + 1;
        }
      }
      // on abort: wait (bounded) for the copies still in flight before leaving
      if (*(volatile int*)&S.abort_flag) {
        for (uint32_t j = issued > (uint32_t)STAGES ? issued - STAGES : 0; j < issued; ++j)
          mbar_wait(&S.full[j % STAGES], (j / STAGES) & 1, 2, args.wait_limit);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (warp-uniform loops, one lane issues)
    const bool leader = elect_one();
    constexpr uint32_t idesc = idesc_bf16(BM, BN);
    constexpr uint32_t kStepA = (BM * BK * 2) >> 4, kStepB = (BN * BK * 2) >> 4;
    const uint64_t ad = smem_desc(S.a[0]), bd = smem_desc(S.b[0]);
    uint32_t s = 0, par = 0, ch = 0;                // ring stage, its parity, accumulators
    bool issued_any = false, ok = true;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x, ++ch) {
      int kb0, nkb;
      unit_k(u, kb0, nkb);
      const uint32_t buf = ch & 1, use = ch >> 1;
      if (use > 0)
        ok = mbar_wait_warp(&S.acc_empty[buf], (use - 1) & 1, 5, &S.abort_flag,
                            args.wait_limit);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + buf * BN;
      for (int kb = 0; kb < nkb; ++kb) {
        ok = mbar_wait_warp(&S.full[s], par, 3, &S.abort_flag, args.wait_limit);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_bf16(d, ad + s * kStepA + kk * 2, bd + s * kStepB + kk * 2, idesc,
                     (kb > 0 || kk > 0) ? 1u : 0u);
          mma_commit(&S.empty[s]);   // frees the stage once these MMAs have read it
        }
        issued_any = true;
        if (++s == STAGES) {
          s = 0;
          par ^= 1;
        }
      }
      if (!ok) break;
      if (leader) mma_commit(&S.acc_full[buf]);
    }
    if (!ok) S.abort_flag = 1;
    if (*(volatile int*)&S.abort_flag && issued_any && leader) {
      mma_commit(&S.drain);      // wait (bounded) for the MMAs still in flight
      mbar_wait(&S.drain, 0, 6, args.wait_limit);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps
    const int q = warp & 3;                          // TMEM lane quarter of this warp
    const int ew = warp - 2;                         // epilogue warp index
    unsigned char* wbuf = S.cbuf[ew][0];             // 2 x 4 KB, 1024-byte aligned
    const bool bf16_out = args.out_kind == OUT_BF16;
    uint32_t ch = 0, chunk = 0;
    bool ok = true;
    // wait for accumulator `ch` and return its TMEM base
    auto acquire = [&](uint32_t& tl) -> bool {
      const uint32_t buf = ch & 1, use = ch >> 1;
      if (!mbar_wait_or_abort(&S.acc_full[buf], use & 1, 4, &S.abort_flag, 4 * args.wait_limit))
        return false;   // (four times the limit of the role it waits for)
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tl = tmem + buf * BN + ((uint32_t)(q * 32) << 16);
      return true;
    };
    auto release = [&]() {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.acc_empty[ch & 1]);
      ++ch;
    };
    // stage one row segment of 32 FP32 values (this lane's row) and store the 32-row slab
    auto store32 = [&](const float (&v)[32], int n0c, int row0) {
      unsigned char* sb = wbuf + (chunk & 1) * 4096;
      if (lane == 0) bulk_wait_read1();   // the store issued from sb two chunks ago
      __syncwarp();
      const uint32_t rowa = smem_u32(sb) + lane * 128;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        st_shared_v4(rowa + ((j ^ (lane & 7)) << 4), __float_as_uint(v[4 * j]),
                     __float_as_uint(v[4 * j + 1]), __float_as_uint(v[4 * j + 2]),
                     __float_as_uint(v[4 * j + 3]));
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      // every chunk that wrote a staging buffer commits exactly one bulk group, which is
      // what the wait_group.read accounting above relies on
      if (lane == 0) {
        if (args.out_kind == OUT_F32_ATOMIC) tma_reduce_add_2d(&maps.c, sb, n0c, row0);
        else tma_store_2d(&maps.c, sb, n0c, row0);
        bulk_commit();
      }
      ++chunk;
    };
    // plain stores of one 32 x 32 block through a 4 KB transpose buffer: row r, column c
    // lives at r * 32 + (c ^ r), so that both the row writes and the column reads below
    // touch 32 different banks
    auto plain32 = [&](const float (&v)[32], int n0c, int row0, void* Cb) {
      float* stage = reinterpret_cast<float*>(wbuf);     // (used only without TMA stores)
#pragma unroll
      for (int i = 0; i < 32; ++i) stage[lane * 32 + (i ^ lane)] = v[i];
      __syncwarp();
      const int col = n0c + lane;
      const int nrow = min(32, args.M - row0);
      if (col < args.N) {
        if (args.out_kind == OUT_BF16) {
          __nv_bfloat16* cp =
              reinterpret_cast<__nv_bfloat16*>(Cb) + (long long)row0 * args.ldc + col;
          for (int r = 0; r < nrow; ++r)
            cp[(long long)r * args.ldc] = __float2bfloat16_rn(stage[r * 32 + (lane ^ r)]);
        } else if (args.out_kind == OUT_F32_ATOMIC) {
          float* cp = reinterpret_cast<float*>(Cb) + (long long)row0 * args.ldc + col;
          for (int r = 0; r < nrow; ++r)
            atomicAdd(cp + (long long)r * args.ldc, stage[r * 32 + (lane ^ r)]);
        } else {
          float* cp = reinterpret_cast<float*>(Cb) + (long long)row0 * args.ldc + col;
          for (int r = 0; r < nrow; ++r) cp[(long long)r * args.ldc] = stage[r * 32 + (lane ^ r)];
        }
      }
      __syncwarp();
    };
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      const int m0 = (u % tiles_m) * BM;
      const int n0 = ((u / tiles_m) % tiles_n) * BN;
      const int row0 = m0 + q * 32;
      const bool rows_here = row0 < args.M;
      {
        uint32_t tl;
        if (!acquire(tl)) { ok = false; break; }
        if (args.tma_store && rows_here) {
          // Each lane owns one row of the 32-row slab: it writes its 128-byte row segment
          // into a 128B-swizzled staging buffer (16-byte chunk j of row r lands at chunk
          // j ^ (r % 8)), then lane 0 issues one TMA store (or reduce-add) of the 32-row
          // box; the box is clipped at the matrix edges by the tensor map.
          const int cw = bf16_out ? 64 : 32;
#pragma unroll 1
          for (int c0 = 0; c0 < BN; c0 += cw) {
            if (n0 + c0 >= args.N) break;
            if (bf16_out) {
              unsigned char* sb = wbuf + (chunk & 1) * 4096;
              if (lane == 0) bulk_wait_read1();
              __syncwarp();
              const uint32_t rowa = smem_u32(sb) + lane * 128;
              float v0[32], v1[32];
              tmem_ld32(tl + (uint32_t)c0, v0);
              tmem_ld32(tl + (uint32_t)(c0 + 32), v1);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float* v = j < 4 ? v0 + 8 * j : v1 + 8 * (j - 4);
                st_shared_v4(rowa + ((j ^ (lane & 7)) << 4), pack_bf16(v[0], v[1]),
                             pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
              }
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              __syncwarp();
              if (lane == 0) {
                tma_store_2d(&maps.c, sb, n0 + c0, row0);
                bulk_commit();
              }
              ++chunk;
            } else {
              float v[32];
              tmem_ld32(tl + (uint32_t)c0, v);
              store32(v, n0 + c0, row0);
            }
          }
        } else if (!args.tma_store) {
#pragma unroll 1
          for (int c0 = 0; c0 < BN; c0 += 32) {
            if (n0 + c0 >= args.N) break;
            float v[32];
            tmem_ld32(tl + (uint32_t)c0, v);
            plain32(v, n0 + c0, row0, args.C);
          }
        }
        release();
      }
    }
    if (!ok) S.abort_flag = 1;
    if (args.tma_store && lane == 0) bulk_wait_all();   // stores complete before exit
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)(2 * BN)));
  }
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  if (!fn) throw CudaError("cuTensorMapEncodeTiled unavailable");
  return fn;
}

// 2D K-major BF16 operand: rows x K (row stride ld elements), box BK x box_rows, 128B swizzle.
CUtensorMap make_map(const __nv_bfloat16* ptr, int rows, int K, long long ld, int box_rows) {
  A2_REQUIRE((reinterpret_cast<uintptr_t>(ptr) & 15) == 0, "TMA base must be 16-byte aligned");
  A2_REQUIRE((ld * 2) % 16 == 0, "TMA row stride must be a multiple of 16 bytes");
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)ptr, dims, strides,
                           box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw CudaError("cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

// Tiled BF16 map of rank 3 or 4 (dims innermost first, strides in bytes for dims 1..),
// 128B swizzle, zero fill outside the extents.
CUtensorMap make_map_nd(const __nv_bfloat16* ptr, int rank, const cuuint64_t* dims,
                        const cuuint64_t* strides, const cuuint32_t* box) {
  A2_REQUIRE((reinterpret_cast<uintptr_t>(ptr) & 15) == 0, "TMA base must be 16-byte aligned");
  for (int i = 0; i < rank - 1; ++i)
    A2_REQUIRE(strides[i] % 16 == 0, "TMA strides must be multiples of 16 bytes");
  CUtensorMap m;
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, (void*)ptr, dims, strides,
                           box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw CudaError("cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

template <int BN, int STAGES>
void launch(const __nv_bfloat16* A, long long lda, const __nv_bfloat16* B, long long ldb, int M,
            int N, int K, const TcSeg2* seg, void* C, long long ldc, int out_kind, int splitk,
            cudaStream_t s) {
  TcMaps maps;
  maps.a = make_map(A, M, K, lda, BM);
  maps.b = make_map(B, N, K, ldb, BN);
  int nk2 = 0, nbc2 = 1, n12 = 1;
  if (seg) {
    const long long Dr = seg->Dr, R1 = seg->R1;
    n12 = seg->n12;
    A2_REQUIRE(n12 >= 1 && BM % n12 == 0 && (long long)M == (long long)seg->Dl * n12,
               "tc GEMM segment: rows must be (a, s12) with s12 dividing 128");
    A2_REQUIRE(Dr % 8 == 0 && seg->Nb == N, "tc GEMM segment: Dr % 8 == 0, N == Dr");
    nbc2 = (int)((Dr + BK - 1) / BK);
    nk2 = (int)(R1 * nbc2);
    const cuuint64_t ad[4] = {(cuuint64_t)Dr, (cuuint64_t)n12, (cuuint64_t)R1,
                              (cuuint64_t)seg->Dl};
    const cuuint64_t as[3] = {(cuuint64_t)(Dr * 2), (cuuint64_t)(n12 * Dr * 2),
                              (cuuint64_t)(R1 * n12 * Dr * 2)};
    const cuuint32_t ab[4] = {(cuuint32_t)BK, (cuuint32_t)n12, 1u, (cuuint32_t)(BM / n12)};
    maps.a2 = make_map_nd(seg->A[0], 4, ad, as, ab);
    const cuuint64_t bd[3] = {(cuuint64_t)Dr, (cuuint64_t)R1, (cuuint64_t)N};
    const cuuint64_t bs[2] = {(cuuint64_t)(Dr * 2), (cuuint64_t)(R1 * Dr * 2)};
    const cuuint32_t bb[3] = {(cuuint32_t)BK, 1u, (cuuint32_t)BN};
    maps.b2 = make_map_nd(seg->B[0], 3, bd, bs, bb);
  } else {
    maps.a2 = maps.a;
    maps.b2 = maps.b;
  }
  const size_t smem = sizeof(TcSmem<BN, STAGES>) + 1024;
  static PerDevice<bool> set;
  set.at(current_device(), [smem] {
    A2_CUDA(cudaFuncSetAttribute(tc_gemm_kernel<BN, STAGES>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return true;
  });
  const int nk1 = (K + BK - 1) / BK;
  const int nk_total = nk1 + nk2;
  splitk = std::max(1, std::min(splitk, nk_total));
  TcArgs args;
  args.M = M; args.N = N; args.K = K;
  args.nk1 = nk1; args.nk2 = nk2; args.nbc2 = nbc2; args.n12 = n12;
  args.kblocks_per_split = (nk_total + splitk - 1) / splitk;
  splitk = (nk_total + args.kblocks_per_split - 1) / args.kblocks_per_split;
  args.C = C; args.ldc = ldc; args.out_kind = out_kind;
  args.splits = splitk;
  args.wait_limit = kWaitLimit;
  args.no_loads = 0;
  // TMA store epilogue when C's base and row stride allow it
  {
    const size_t es = out_kind == OUT_BF16 ? 2 : 4;
    args.tma_store = ((reinterpret_cast<uintptr_t>(C) & 15) == 0 && (ldc * es) % 16 == 0 &&
                      ldc >= N) ? 1 : 0;
    if (args.tma_store) {
      const cuuint64_t cd[2] = {(cuuint64_t)N, (cuuint64_t)M};
      const cuuint64_t cs[1] = {(cuuint64_t)(ldc * es)};
      const cuuint32_t cb[2] = {(cuuint32_t)(out_kind == OUT_BF16 ? 64 : 32), 32u};
      const cuuint32_t ce[2] = {1, 1};
      CUresult r = encode_fn()(&maps.c,
                               out_kind == OUT_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                    : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                               2, C, cd, cs, cb, ce, CU_TENSOR_MAP_INTERLEAVE_NONE,
                               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) args.tma_store = 0;
    }
  }
  const long long units = (long long)cdiv(M, BM) * cdiv(N, BN) * splitk;
  A2_REQUIRE(units < (1LL << 31), "tcgen05 GEMM too large");
  const int grid = (int)std::min<long long>(units, device_sms());
  tc_gemm_kernel<BN, STAGES><<<grid, kTcThreads, smem, s>>>(maps, args);
  A2_CHECK_LAUNCH();
}

// ------------------------------------------------------------------ Ozaki GEMM
// FP64-class product of two operands given as kOzSlices BF16 slices each (the slicing of the
// FP64 emulation below): the slice pairs (i, j) with i + j <= 8, 28 of them.
//
// Bound: operand delivery.  The MMAs alone take 64 cycles each (M = N = 128, K = 16, operands
// already in shared memory), but L2 and TMA deliver about 0.45 rows per clock to an SM,
// whether a row is 64 or 128 bytes: with one pair of 128-byte-row tiles per slice pair the
// kernel ran at half the tensor rate (1.10 PFLOP/s on every shape).  Three things raise the
// products per delivered row:
//  * a tile serves all the pairs it can while it is in shared memory: the K loop runs over
//    chunks of 256, and each chunk is walked three times, for the levels l = i + j of
//        2, 3 (slices 1..2, 3 pairs) | 4, 5 (slices 1..4, 7 pairs) | 6, 7 + 8 (18 pairs)
//    with two TMEM accumulators of 128 columns per phase, so that the epilogue drains one
//    phase's two while the next phase fills the other two (4 x 128 columns, all of TMEM);
//  * the slices are interleaved in memory, [K / 32][row][slice][32], so that a 128-byte row of
//    a tile holds two slices of a K block of 32 (the seventh slice has 64-byte rows): 7 tile
//    loads per 28 products instead of 56 half as wide ones (with the rows outermost, a tile's
//    rows lie 2.3 MB apart in S4 and its loads take 7.2 ms instead of 4.6);
//  * MMAs on the same A slice follow each other and take it from the collector buffer.
// Exactness: |digit| <= 128, so level l's sum over a chunk is an integer below
// 256 (l - 1) 2^14 units, at most 2^24 for l <= 5: exact in FP32.  Level 6 reaches 1.25 x
// 2^24 only if all digits are extreme; its last additions are then off by up to one unit each, 2^-46
// of the row and column scale.  Levels 7 and 8 share an accumulator, so that an addition is off by
// up to 2^-24 of the level 7 sum: up to 2^-53 of the scales where all digits are extreme, ~2^-60
// where their signs are random.  Measured over operands whose digits all lie in [112, 127], [96, 127],
// [64, 127], [126, 127], [0, 127] or [-128, 127], against exact integers: at most 2^-46.6, 2^-46.0, 2^-45.2 of sum |a| |b| at
// K = 256, 512, 1024, where 36 pairs with exact level sums were off by up to 2^-45.4, 2^-44.7, 2^-43.7.
// Both are the rounding of the pairs' low part, which has an error for every drained accumulator.
// The epilogue adds every accumulator into a double-float register pair (hi + lo, Knuth's
// error-free two-sum), so no per-level tile reaches memory.
//
// Work unit = (128 x 128 output tile, K split).  A ring slot holds one tile of both operands
// (32 KB): slices 1-2, 3-4, 5-6 or 7 of one K block.  A phase loads 1, 2 or 4 tiles per K
// block, the last phase in the order 3-4, 1-2, 5-6, 7: its first pairs need only the first two,
// slices 3 and 4 are done first, and their slot is refilled while the rest runs.  Warp 0
// lane 0: TMA producer; warp 1: MMA issuer (warp-uniform loops, one lane issues, the MMAs of a K
// block unrolled: computed slots and branches in the issue loop took longer than the MMAs);
// warps 2..9: epilogue (two per TMEM lane quarter, 64 columns each).  Every wait is bounded
// as in tc_gemm_kernel.
// Measured, D = 256, R = 342 -> 444 (28 products, before: 36 with one tile pair each; ms): left
// update's 87552 x 1024 x 256 0.77 (1.50), its 256 x 113664 x 1024 0.99 (1.93), S4's 4096 x
// 256 x 143872 4.6 (9.88).
constexpr int kOzBN = 128;
constexpr int kOzBK = 32;
constexpr int kOzSlots = 6;
constexpr int kOzChunk = 256 / kOzBK;           // K blocks between drains
constexpr int kOzPhases = 3;
constexpr int kOzEpi = 8;
constexpr int kOzThreads = 64 + 32 * kOzEpi;

struct OzSmem {
  alignas(1024) __nv_bfloat16 a[kOzSlots][BM * 64];
  alignas(1024) __nv_bfloat16 b[kOzSlots][kOzBN * 64];
  alignas(1024) float stage[kOzEpi][2][32 * 16];   // epilogue transpose buffers (hi, lo)
  alignas(8) uint64_t full[kOzSlots];
  alignas(8) uint64_t empty[kOzSlots];
  alignas(8) uint64_t acc_full[2];
  alignas(8) uint64_t acc_empty[2];
  alignas(8) uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(OzSmem) + 1024 <= 227 * 1024, "Ozaki ring exceeds shared memory");

struct OzMaps {              // views [K block][row][slice and k]
  CUtensorMap a, b;          // box 1 x 128 x 64 (two slices), 128-byte swizzle
  CUtensorMap a7, b7;        // box 1 x 128 x 32 (the last slice), 64-byte swizzle
};

enum OzOut { OZ_F64 = 0, OZ_PAIR = 1, OZ_SPLIT = 2 };

struct OzArgs {
  int M, N, nk;              // rows, columns, K blocks of kOzBK
  int kblocks_per_split, splits;
  int n_fast;                // 1: consecutive units walk the N tiles of one row of tiles
  int out_mode;              // OZ_F64: C[m*ldc + n] = hi + lo (FP64)
                             // OZ_PAIR: FP32 hi at C[m*ldc + n], lo at + df_plane
                             // OZ_SPLIT: FP32 tiles of split sp, hi at C + 2sp*MN and lo at
                             //           C + (2sp+1)*MN, row stride N
  void* C;
  long long ldc, df_plane, MN;
};

// End of the chunk that starts at block c0 of a split (blocks kb0 .. kb0 + nkb - 1): chunks end at
// multiples of kOzChunk of the whole K range, where the operands' scales change.
__device__ __forceinline__ int oz_chunk_end(int kb0, int c0, int nkb) {
  return min(nkb, ((kb0 + c0) / kOzChunk + 1) * kOzChunk - kb0);
}

// Tiles of a phase in load order: 0 = slices 1-2, 1 = 3-4, 2 = 5-6, 3 = 7.
__host__ __device__ constexpr int oz_tiles(int ph) { return ph == 2 ? 4 : ph + 1; }
__host__ __device__ constexpr int oz_tile(int ph, int t) {
  return ph == 2 && t < 2 ? 1 - t : t;
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart.
__device__ __forceinline__ uint64_t smem_desc64(const void* p) {
  const uint64_t addr = smem_u32(p);
  uint64_t d = 0;
  d |= (addr >> 4) & 0x3FFFull;            // start address
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;         // stride byte offset: 8 rows x 64 B
  d |= (uint64_t)1 << 46;                  // descriptor version for tcgen05
  d |= (uint64_t)4 << 61;                  // SWIZZLE_64B
  return d;
}

// A run of MMAs on A slice I with the B slices J... of one K block, into the accumulator of
// level l0 (d0) or of the levels above it (d0 + 128 columns).  off[t]: descriptor offset of the ring
// slot that holds tile t.
template <int L0, int I, int... J>
__device__ __forceinline__ void oz_run(uint32_t d0, uint64_t ad, uint64_t bd, uint64_t ad7,
                                       uint64_t bd7, const uint32_t (&off)[4], bool& f0,
                                       bool& f1) {
  constexpr uint32_t idesc = idesc_bf16(BM, kOzBN);
  constexpr int js[] = {J...};
  constexpr int n = sizeof...(J);
#pragma unroll
  for (int kk = 0; kk < kOzBK / 16; ++kk)
#pragma unroll
    for (int q = 0; q < n; ++q) {
      const int j = js[q];
      const bool lead = I + j == L0;
      const uint32_t d = d0 + (lead ? 0 : kOzBN), keep = (lead ? f0 : f1) ? 0u : 1u;
      const uint64_t a = (I == 7 ? ad7 : ad) + off[(I - 1) / 2] + ((I - 1) & 1) * 4 + kk * 2;
      const uint64_t b = (j == 7 ? bd7 : bd) + off[(j - 1) / 2] + ((j - 1) & 1) * 4 + kk * 2;
      if (n == 1) mma_bf16_a<true, true>(d, a, b, idesc, keep);
      else if (q == 0) mma_bf16_a<true, false>(d, a, b, idesc, keep);
      else if (q == n - 1) mma_bf16_a<false, true>(d, a, b, idesc, keep);
      else mma_bf16_a<false, false>(d, a, b, idesc, keep);
      if (lead) f0 = false;
      else f1 = false;
    }
}

// 10 warps: three of them share one SM sub-partition's 16K registers, hence at most 168
// registers per thread.
__global__ void __launch_bounds__(kOzThreads, 1)
tc_oz_kernel(const __grid_constant__ OzMaps maps, OzArgs args) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;
  auto& S = *reinterpret_cast<OzSmem*>(smem_raw + pad);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = (args.M + BM - 1) / BM;
  const int tiles_n = (args.N + kOzBN - 1) / kOzBN;
  const int nunits = tiles_m * tiles_n * args.splits;
  constexpr uint32_t kSlotBytes = (BM + kOzBN) * 64 * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kOzSlots; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.acc_full[i], 1);
      mbar_init(&S.acc_empty[i], kOzEpi);
    }
    mbar_init(&S.drain, 1);
    S.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {   // two pairs of accumulators of 128 fp32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem_base)),
                 "r"((uint32_t)(4 * kOzBN)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = S.tmem_base;

  auto unit = [&](int u, int& m0, int& n0, int& kb0, int& nkb) {
    const int t = u % (tiles_m * tiles_n), sp = u / (tiles_m * tiles_n);
    if (args.n_fast) {
      n0 = (t % tiles_n) * kOzBN;
      m0 = (t / tiles_n) * BM;
    } else {
      m0 = (t % tiles_m) * BM;
      n0 = (t / tiles_m) * kOzBN;
    }
    kb0 = sp * args.kblocks_per_split;
    nkb = max(0, min(args.nk - kb0, args.kblocks_per_split));
  };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- producer: chunk, phase, K block, tile
      uint32_t g = 0, issued = 0;
      bool stop = false;
      for (int u = blockIdx.x; !stop && u < nunits && !*(volatile int*)&S.abort_flag;
           u += gridDim.x) {
        int m0, n0, kb0, nkb;
        unit(u, m0, n0, kb0, nkb);
        for (int c0 = 0, c1; !stop && c0 < nkb; c0 = c1) {
          c1 = oz_chunk_end(kb0, c0, nkb);
          for (int ph = 0; !stop && ph < kOzPhases; ++ph) {
            const int nt = oz_tiles(ph);
            for (int kb = c0; !stop && kb < c1; ++kb) {
              for (int t = 0; t < nt; ++t, ++g) {
                const int s = g % kOzSlots;
                const uint32_t round = g / kOzSlots;
                if ((round > 0 &&
                     !mbar_wait_or_abort(&S.empty[s], (round - 1) & 1, 11, &S.abort_flag)) ||
                    *(volatile int*)&S.abort_flag) {
                  S.abort_flag = 1;
                  stop = true;
                  break;
                }
                const int tile = oz_tile(ph, t);
                mbar_expect_tx(&S.full[s], tile == 3 ? kSlotBytes / 2 : kSlotBytes);
                tma_load_3d(tile == 3 ? &maps.a7 : &maps.a, &S.full[s], S.a[s], tile * 64, m0,
                            kb0 + kb);
                tma_load_3d(tile == 3 ? &maps.b7 : &maps.b, &S.full[s], S.b[s], tile * 64, n0,
                            kb0 + kb);
                issued = g + 1;
              }
            }
          }
        }
      }
      if (*(volatile int*)&S.abort_flag) {   // wait (bounded) for the copies in flight
        for (uint32_t j = issued > (uint32_t)kOzSlots ? issued - kOzSlots : 0; j < issued; ++j)
          mbar_wait(&S.full[j % kOzSlots], (j / kOzSlots) & 1, 12);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: two TMEM accumulators per (chunk, phase)
    const bool leader = elect_one();
    const uint64_t ad = smem_desc(S.a[0]), bd = smem_desc(S.b[0]);
    const uint64_t ad7 = smem_desc64(S.a[0]), bd7 = smem_desc64(S.b[0]);
    uint32_t slot = 0, par = 0, pc = 0;     // next slot, parity of its round, phase counter
    bool issued_any = false, ok = true;
    constexpr uint32_t kSlotStep = (BM * 64 * 2) >> 4;          // descriptor units
    uint32_t off[4];                        // by tile
    auto slot_of = [&](int t) {             // ring slot of the t-th tile of this K block
      const uint32_t sl = slot + t;
      return sl >= kOzSlots ? sl - kOzSlots : sl;
    };
    auto wait_tile = [&](int ph, int t) {   // the t-th tile of this K block has arrived
      const uint32_t sl = slot_of(t);
      ok = ok && mbar_wait_warp(&S.full[sl], par ^ (slot + t >= kOzSlots ? 1u : 0u), 14,
                                &S.abort_flag);
      off[oz_tile(ph, t)] = sl * kSlotStep;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto advance = [&](int nt) {
      slot += nt;
      if (slot >= kOzSlots) {
        slot -= kOzSlots;
        par ^= 1;
      }
    };
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      int m0, n0, kb0, nkb;
      unit(u, m0, n0, kb0, nkb);
      for (int c0 = 0, c1; ok && c0 < nkb; c0 = c1) {
        c1 = oz_chunk_end(kb0, c0, nkb);
#pragma unroll
        for (int ph = 0; ph < kOzPhases; ++ph) {
          if (!ok) break;
          const uint32_t set = pc & 1, use = pc >> 1;
          if (use > 0) {
            ok = mbar_wait_warp(&S.acc_empty[set], (use - 1) & 1, 13, &S.abort_flag);
            if (!ok) break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d0 = tmem + set * (2 * kOzBN);
          for (int kb = c0; kb < c1; ++kb) {
            bool f0 = kb == c0, f1 = f0;
#define A2_RUN(...) oz_run<__VA_ARGS__>(d0, ad, bd, ad7, bd7, off, f0, f1)
            if (ph == 0) {
              wait_tile(0, 0);
              if (ok && leader) {
                A2_RUN(2, 1, 1, 2);
                A2_RUN(2, 2, 1);
                mma_commit(&S.empty[slot_of(0)]);
              }
            } else if (ph == 1) {
              wait_tile(1, 0);
              wait_tile(1, 1);
              if (ok && leader) {
                A2_RUN(4, 2, 2, 3);
                A2_RUN(4, 1, 3, 4);
                A2_RUN(4, 3, 1, 2);
                A2_RUN(4, 4, 1);
                mma_commit(&S.empty[slot_of(0)]);
                mma_commit(&S.empty[slot_of(1)]);
              }
            } else {
              wait_tile(2, 0);
              wait_tile(2, 1);
              if (ok && leader) {
                A2_RUN(6, 3, 3, 4);
                A2_RUN(6, 4, 2, 3, 4);
                A2_RUN(6, 2, 4);
              }
              wait_tile(2, 2);
              if (ok && leader) {
                A2_RUN(6, 3, 5);
                A2_RUN(6, 5, 3, 1, 2);
                mma_commit(&S.empty[slot_of(0)]);        // slices 3, 4 are done
                A2_RUN(6, 1, 5, 6);
                A2_RUN(6, 2, 5, 6);
                A2_RUN(6, 6, 1, 2);
              }
              wait_tile(2, 3);
              if (ok && leader) {
                A2_RUN(6, 1, 7);
                A2_RUN(6, 7, 1);
                mma_commit(&S.empty[slot_of(1)]);
                mma_commit(&S.empty[slot_of(2)]);
                mma_commit(&S.empty[slot_of(3)]);
              }
            }
#undef A2_RUN
            issued_any |= ok;
            advance(oz_tiles(ph));
            if (!ok) break;
          }
          if (!ok) break;
          if (leader) mma_commit(&S.acc_full[set]);
          ++pc;
        }
      }
    }
    if (!ok) S.abort_flag = 1;
    if (*(volatile int*)&S.abort_flag && issued_any && leader) {
      mma_commit(&S.drain);
      mbar_wait(&S.drain, 0, 15);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: double-float sums of the accumulators, then the output
    const int q = warp & 3;                 // TMEM lane quarter of this warp
    const int ew = warp - 2;
    const int colbase = (ew >> 2) * 64;     // this warp's 64 columns of the tile
    float* sh = S.stage[ew][0];
    float* sl = S.stage[ew][1];
    uint32_t pc = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      int m0, n0, kb0, nkb;
      unit(u, m0, n0, kb0, nkb);
      float hi[64], lo[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) hi[i] = lo[i] = 0.f;
      for (int c0 = 0; ok && c0 < nkb; c0 = oz_chunk_end(kb0, c0, nkb)) {
        for (int ph = 0; ph < kOzPhases; ++ph, ++pc) {
          const uint32_t set = pc & 1, use = pc >> 1;
          if (!mbar_wait_or_abort(&S.acc_full[set], use & 1, 16, &S.abort_flag)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t tl =
              tmem + set * (2 * kOzBN) + (uint32_t)colbase + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
          for (int acc = 0; acc < 2; ++acc) {
#pragma unroll
            for (int c = 0; c < 64; c += 8) {
              float v[8];
              tmem_ld8(tl + (uint32_t)(acc * kOzBN + c), v);
#pragma unroll
              for (int i = 0; i < 8; ++i) {   // (hi, lo) += v exactly up to lo's rounding
                const float sum = __fadd_rn(hi[c + i], v[i]);
                const float bp = __fsub_rn(sum, hi[c + i]);
                const float err =
                    __fadd_rn(__fsub_rn(hi[c + i], __fsub_rn(sum, bp)), __fsub_rn(v[i], bp));
                hi[c + i] = sum;
                lo[c + i] = __fadd_rn(lo[c + i], err);
              }
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&S.acc_empty[set]);
        }
      }
      if (!ok) break;
      // output: 32 x 16 blocks through the transpose buffers (lane = row on the way in; a
      // half warp writes one row's 16 columns on the way out)
      const int row0 = m0 + q * 32;
#pragma unroll
      for (int c = 0; c < 64; c += 16) {
        const int col0 = n0 + colbase + c;
        if (col0 >= args.N || row0 >= args.M) continue;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          sh[lane * 16 + (i ^ (lane & 15))] = hi[c + i];
          sl[lane * 16 + (i ^ (lane & 15))] = lo[c + i];
        }
        __syncwarp();
        const int cc = lane & 15, col = col0 + cc;
        const int nrow = min(32, args.M - row0);
        if (col < args.N) {
          if (args.out_mode == OZ_F64) {
            double* cp = reinterpret_cast<double*>(args.C) + (long long)row0 * args.ldc + col;
#pragma unroll 4
            for (int r = lane >> 4; r < nrow; r += 2)
              cp[(long long)r * args.ldc] = (double)sh[r * 16 + (cc ^ (r & 15))] +
                                            (double)sl[r * 16 + (cc ^ (r & 15))];
          } else if (args.out_mode == OZ_PAIR) {
            float* cp = reinterpret_cast<float*>(args.C) + (long long)row0 * args.ldc + col;
#pragma unroll 4
            for (int r = lane >> 4; r < nrow; r += 2) {
              const float h = sh[r * 16 + (cc ^ (r & 15))], e = sl[r * 16 + (cc ^ (r & 15))];
              const float sum = __fadd_rn(h, e);   // renormalised pair
              cp[(long long)r * args.ldc] = sum;
              cp[(long long)r * args.ldc + args.df_plane] = __fsub_rn(e, __fsub_rn(sum, h));
            }
          } else {
            const int sp = u / (tiles_m * tiles_n);
            float* cp = reinterpret_cast<float*>(args.C) + 2LL * sp * args.MN +
                        (long long)row0 * args.N + col;
#pragma unroll 4
            for (int r = lane >> 4; r < nrow; r += 2) {
              cp[(long long)r * args.N] = sh[r * 16 + (cc ^ (r & 15))];
              cp[(long long)r * args.N + args.MN] = sl[r * 16 + (cc ^ (r & 15))];
            }
          }
        }
        __syncwarp();
      }
    }
    if (!ok) S.abort_flag = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)(4 * kOzBN)));
  }
}

// Maps of a sliced operand ([nkb][rows][8][32] BF16, slice 8 unused): two slices per box row,
// or the last one.
CUtensorMap make_oz_map(const __nv_bfloat16* ptr, int rows, int nkb, bool last) {
  const cuuint64_t dims[3] = {(cuuint64_t)(kOzSlices * kOzBK), (cuuint64_t)rows, (cuuint64_t)nkb};
  const cuuint64_t strides[2] = {(cuuint64_t)(kOzRowBlock * 2), (cuuint64_t)rows * kOzRowBlock * 2};
  const cuuint32_t box[3] = {last ? 32u : 64u, (cuuint32_t)BM, 1u};
  A2_REQUIRE((reinterpret_cast<uintptr_t>(ptr) & 15) == 0, "TMA base must be 16-byte aligned");
  CUtensorMap m;
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)ptr, dims, strides,
                           box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           last ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw CudaError("cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

// Launches tc_oz_kernel over the slices of A (M x K) and B (N x K).
void launch_oz(const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K, int splits,
               int out_mode, void* C, long long ldc, long long df_plane, cudaStream_t s) {
  static_assert(kOzBN == BM, "one box shape for both operands");
  const int nkb = (K + kOzBK - 1) / kOzBK;
  OzMaps maps;
  maps.a = make_oz_map(A, M, nkb, false);
  maps.b = make_oz_map(B, N, nkb, false);
  maps.a7 = make_oz_map(A, M, nkb, true);
  maps.b7 = make_oz_map(B, N, nkb, true);
  const size_t smem = sizeof(OzSmem) + 1024;
  static PerDevice<bool> set;
  set.at(current_device(), [smem] {
    A2_CUDA(cudaFuncSetAttribute(tc_oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    return true;
  });
  OzArgs args;
  args.M = M; args.N = N;
  args.nk = (K + kOzBK - 1) / kOzBK;
  splits = std::max(1, std::min(splits, args.nk));
  args.kblocks_per_split = (args.nk + splits - 1) / splits;
  args.splits = (args.nk + args.kblocks_per_split - 1) / args.kblocks_per_split;
  A2_REQUIRE(args.splits == 1 || out_mode == OZ_SPLIT, "Ozaki GEMM: K splits need split tiles");
  args.n_fast = cdiv(N, kOzBN) <= 64 ? 1 : 0;
  args.out_mode = out_mode;
  args.C = C; args.ldc = ldc; args.df_plane = df_plane;
  args.MN = (long long)M * N;
  const long long units = (long long)cdiv(M, BM) * cdiv(N, kOzBN) * args.splits;
  A2_REQUIRE(units < (1LL << 31), "Ozaki GEMM too large");
  const int grid = (int)std::min<long long>(units, device_sms());
  tc_oz_kernel<<<grid, kOzThreads, smem, s>>>(maps, args);
  A2_CHECK_LAUNCH();
}

// ------------------------------------------------------------------ split products
// C = A B^T to FP32 accuracy for operands given as three BF16 planes each (a value as
// high + middle + low part): the six plane pairs (i, j) with i + j <= 2 accumulated together.
//
// Bound: shared-memory bandwidth, as for the Ozaki GEMM.  With one pair of tiles loaded per plane
// pair, TMA writes (94) and the MMAs read (96) 190 bytes per clock and SM of a possible
// 128 at the full tensor rate, and the kernel ran at 63 to 65 % of it.  Here a K block of 32
// is loaded once, plane by plane (a ring slot holds plane i of both operands, 64-byte
// swizzled rows), and all six pairs run from it: half the loads, 141 bytes per clock.
// The pairs run in the order of their later plane, so that the MMAs start before the last
// plane has arrived.
// The tensor cores' FP32 accumulator truncates, so every kS3Chunk K blocks are accumulated
// into a fresh TMEM buffer of BN columns (two in turn) and the eight epilogue warps add the
// partial sums into IEEE FP32 registers (round to nearest), BN / 2 columns of one row per
// thread.  BN = 128 serves outputs of at most 128 columns (S4 at D <= 128) without
// multiplying padding.
// Roles, waits and the optional second K segment as in tc_gemm_kernel.  Measured at D = 256,
// bond 7 (R = 444, 562, 444; ms): S1 113664 x 4096 x 256 0.99 (1.15), S4 with its second
// segment 4096 x 256 x (113664 + 143872) 2.30 (2.61).
constexpr int kS3BK = 32;
constexpr int kS3Chunk = 4;                 // K blocks per partial sum
constexpr int kS3Epi = 8;
constexpr int kS3Threads = 64 + 32 * kS3Epi;
__host__ __device__ constexpr int s3_slots(int bn) { return bn == 256 ? 8 : 12; }

template <int BN>
struct S3Smem {
  static constexpr int SLOTS = s3_slots(BN);
  alignas(1024) __nv_bfloat16 a[SLOTS][BM * kS3BK];
  alignas(1024) __nv_bfloat16 b[SLOTS][BN * kS3BK];
  alignas(1024) unsigned char cbuf[kS3Epi][4096];         // epilogue staging buffers
  alignas(8) uint64_t full[SLOTS];
  alignas(8) uint64_t empty[SLOTS];
  alignas(8) uint64_t acc_full[2];
  alignas(8) uint64_t acc_empty[2];
  alignas(8) uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(S3Smem<256>) + 1024 <= 227 * 1024, "split ring exceeds shared memory");
static_assert(sizeof(S3Smem<128>) + 1024 <= 227 * 1024, "split ring exceeds shared memory");

struct S3Maps {
  CUtensorMap a[3], b[3];
  CUtensorMap a2[3], b2[3];      // optional second K segment (4D / 3D views)
  CUtensorMap c;
};
struct S3Args {
  int M, N, nk1, nk2;            // K blocks of the plain product and of the second segment
  int nbc2, n12;                 // second segment: b' chunks per w1, (s1 s2) rows per a
  int kblocks_per_split, splits;
  void* C;
  long long ldc;
  int out_kind, tma_store;
};

template <int BN>
__global__ void __launch_bounds__(kS3Threads, 1)
tc_split3_kernel(const __grid_constant__ S3Maps maps, S3Args args) {
  constexpr int SLOTS = s3_slots(BN), WC = BN / 2;         // columns of one epilogue warp
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;
  auto& S = *reinterpret_cast<S3Smem<BN>*>(smem_raw + pad);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = (args.M + BM - 1) / BM;
  const int tiles_n = (args.N + BN - 1) / BN;
  const int nk_total = args.nk1 + args.nk2;
  const int nunits = tiles_m * tiles_n * args.splits;
  constexpr uint32_t kSlotBytes = (BM + BN) * kS3BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.acc_full[i], 1);
      mbar_init(&S.acc_empty[i], kS3Epi);
    }
    mbar_init(&S.drain, 1);
    S.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {   // two accumulators of BN fp32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem_base)),
                 "r"((uint32_t)(2 * BN)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = S.tmem_base;

  auto unit = [&](int u, int& m0, int& n0, int& kb0, int& nkb) {
    m0 = (u % tiles_m) * BM;
    n0 = ((u / tiles_m) % tiles_n) * BN;
    kb0 = (u / (tiles_m * tiles_n)) * args.kblocks_per_split;
    nkb = max(0, min(nk_total - kb0, args.kblocks_per_split));
  };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- producer: K block, plane
      uint32_t g = 0, issued = 0;
      bool stop = false;
      for (int u = blockIdx.x; !stop && u < nunits && !*(volatile int*)&S.abort_flag;
           u += gridDim.x) {
        int m0, n0, kb0, nkb;
        unit(u, m0, n0, kb0, nkb);
        for (int kb = 0; !stop && kb < nkb; ++kb) {
          const int kbg = kb0 + kb;
          for (int p = 0; p < 3; ++p, ++g) {
            const int s = g % SLOTS;
            const uint32_t round = g / SLOTS;
            if ((round > 0 &&
                 !mbar_wait_or_abort(&S.empty[s], (round - 1) & 1, 1, &S.abort_flag)) ||
                *(volatile int*)&S.abort_flag) {
              S.abort_flag = 1;
              stop = true;
              break;
            }
            mbar_expect_tx(&S.full[s], kSlotBytes);
            if (kbg < args.nk1) {
              tma_load_2d(&maps.a[p], &S.full[s], S.a[s], kbg * kS3BK, m0);
              tma_load_2d(&maps.b[p], &S.full[s], S.b[s], kbg * kS3BK, n0);
            } else {   // second segment: K block = (w1, chunk of b')
              const int j = kbg - args.nk1;
              const int w1 = j / args.nbc2, bx = (j % args.nbc2) * kS3BK;
              tma_load_4d(&maps.a2[p], &S.full[s], S.a[s], bx, 0, w1, m0 / args.n12);
              tma_load_3d(&maps.b2[p], &S.full[s], S.b[s], bx, w1, n0);
            }
            issued = g + 1;
          }
        }
      }
      if (*(volatile int*)&S.abort_flag) {   // wait (bounded) for the copies in flight
        for (uint32_t j = issued > (uint32_t)SLOTS ? issued - SLOTS : 0; j < issued; ++j)
          mbar_wait(&S.full[j % SLOTS], (j / SLOTS) & 1, 2);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one TMEM buffer per chunk (warp-uniform loops, one lane
    // issues, the MMAs of a K block unrolled)
    const bool leader = elect_one();
    constexpr uint32_t idesc = idesc_bf16(BM, BN);
    constexpr uint32_t kStepA = (BM * kS3BK * 2) >> 4, kStepB = (BN * kS3BK * 2) >> 4;
    const uint64_t ad = smem_desc64(S.a[0]), bd = smem_desc64(S.b[0]);
    uint32_t slot = 0, par = 0, ch = 0;
    bool issued_any = false, ok = true;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      int m0, n0, kb0, nkb;
      unit(u, m0, n0, kb0, nkb);
      for (int c0 = 0; ok && c0 < nkb; c0 += kS3Chunk, ++ch) {
        const int c1 = min(nkb, c0 + kS3Chunk);
        const uint32_t buf = ch & 1, use = ch >> 1;
        if (use > 0)
          ok = mbar_wait_warp(&S.acc_empty[buf], (use - 1) & 1, 5, &S.abort_flag);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + buf * BN;
        for (int kb = c0; kb < c1; ++kb) {
          uint32_t sl[3];
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            sl[m] = slot + m;
            uint32_t pr = par;
            if (sl[m] >= SLOTS) {
              sl[m] -= SLOTS;
              pr ^= 1;
            }
            ok = ok && mbar_wait_warp(&S.full[sl[m]], pr, 3, &S.abort_flag);
          }
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {
#pragma unroll
            for (int i = 0; i < 3; ++i)          // A plane i against B planes 0 .. 2 - i
#pragma unroll
              for (int kk = 0; kk < kS3BK / 16; ++kk)
#pragma unroll
                for (int j = 0; j <= 2 - i; ++j) {
                  const uint64_t a = ad + sl[i] * kStepA + kk * 2, b = bd + sl[j] * kStepB + kk * 2;
                  const uint32_t keep = (i > 0 || kk > 0 || j > 0 || kb > c0) ? 1u : 0u;
                  if (i == 2) mma_bf16_a<true, true>(d, a, b, idesc, keep);
                  else if (j == 0) mma_bf16_a<true, false>(d, a, b, idesc, keep);
                  else if (j == 2 - i) mma_bf16_a<false, true>(d, a, b, idesc, keep);
                  else mma_bf16_a<false, false>(d, a, b, idesc, keep);
                }
#pragma unroll
            for (int m = 0; m < 3; ++m) mma_commit(&S.empty[sl[m]]);
          }
          issued_any = true;
          slot += 3;
          if (slot >= SLOTS) {
            slot -= SLOTS;
            par ^= 1;
          }
        }
        if (!ok) break;
        if (leader) mma_commit(&S.acc_full[buf]);
      }
    }
    if (!ok) S.abort_flag = 1;
    if (*(volatile int*)&S.abort_flag && issued_any && leader) {
      mma_commit(&S.drain);
      mbar_wait(&S.drain, 0, 6);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps: FP32 sums of the partial tiles, then the output
    const int q = warp & 3;                          // TMEM lane quarter of this warp
    const int ew = warp - 2;
    const int colbase = (ew >> 2) * WC;
    unsigned char* wbuf = S.cbuf[ew];
    uint32_t ch = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      int m0, n0, kb0, nkb;
      unit(u, m0, n0, kb0, nkb);
      const int row0 = m0 + q * 32;
      float acc[WC];
#pragma unroll
      for (int i = 0; i < WC; ++i) acc[i] = 0.f;
      for (int c0 = 0; c0 < nkb; c0 += kS3Chunk, ++ch) {
        const uint32_t buf = ch & 1, use = ch >> 1;
        if (!mbar_wait_or_abort(&S.acc_full[buf], use & 1, 4, &S.abort_flag)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t tl = tmem + buf * BN + (uint32_t)colbase + ((uint32_t)(q * 32) << 16);
#pragma unroll
        for (int c = 0; c < WC; c += 32) {
          float v[32];
          tmem_ld32(tl + (uint32_t)c, v);
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[c + i] += v[i];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.acc_empty[buf]);
      }
      if (!ok) break;
#pragma unroll
      for (int c = 0; c < WC; c += 32) {
        const int col0 = n0 + colbase + c;
        if (col0 >= args.N || row0 >= args.M) continue;
        if (args.tma_store) {
          // this lane's 128-byte row segment into a 128B-swizzled staging buffer, one TMA
          // store (or reduce-add) of the 32-row box, clipped by the map
          if (lane == 0) bulk_wait_read0();
          __syncwarp();
          const uint32_t rowa = smem_u32(wbuf) + lane * 128;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            st_shared_v4(rowa + ((j ^ (lane & 7)) << 4), __float_as_uint(acc[c + 4 * j]),
                         __float_as_uint(acc[c + 4 * j + 1]), __float_as_uint(acc[c + 4 * j + 2]),
                         __float_as_uint(acc[c + 4 * j + 3]));
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (args.out_kind == OUT_F32_ATOMIC) tma_reduce_add_2d(&maps.c, wbuf, col0, row0);
            else tma_store_2d(&maps.c, wbuf, col0, row0);
            bulk_commit();
          }
        } else {
          float* stage = reinterpret_cast<float*>(wbuf);
#pragma unroll
          for (int i = 0; i < 32; ++i) stage[lane * 32 + (i ^ lane)] = acc[c + i];
          __syncwarp();
          const int col = col0 + lane, nrow = min(32, args.M - row0);
          if (col < args.N) {
            float* cp = reinterpret_cast<float*>(args.C) + (long long)row0 * args.ldc + col;
            if (args.out_kind == OUT_F32_ATOMIC)
              for (int r = 0; r < nrow; ++r)
                atomicAdd(cp + (long long)r * args.ldc, stage[r * 32 + (lane ^ r)]);
            else
              for (int r = 0; r < nrow; ++r)
                cp[(long long)r * args.ldc] = stage[r * 32 + (lane ^ r)];
          }
          __syncwarp();
        }
      }
    }
    if (!ok) S.abort_flag = 1;
    if (args.tma_store && lane == 0) bulk_wait_all();   // stores complete before exit
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)(2 * BN)));
  }
}

// Tiled BF16 map of rank 2 to 4 (dims innermost first, strides in bytes for dims 1..) with
// 64-byte swizzle, zero fill outside the extents.
CUtensorMap make_map64(const __nv_bfloat16* ptr, int rank, const cuuint64_t* dims,
                       const cuuint64_t* strides, const cuuint32_t* box) {
  A2_REQUIRE((reinterpret_cast<uintptr_t>(ptr) & 15) == 0, "TMA base must be 16-byte aligned");
  for (int i = 0; i < rank - 1; ++i)
    A2_REQUIRE(strides[i] % 16 == 0, "TMA strides must be multiples of 16 bytes");
  CUtensorMap m;
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, (void*)ptr, dims, strides,
                           box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw CudaError("cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return m;
}

// FP32 output map of the epilogue's 32 x 32 boxes; false if C's base or stride rules it out.
bool make_out_map(CUtensorMap* m, void* C, int M, int N, long long ldc) {
  if ((reinterpret_cast<uintptr_t>(C) & 15) != 0 || (ldc * 4) % 16 != 0 || ldc < N) return false;
  const cuuint64_t cd[2] = {(cuuint64_t)N, (cuuint64_t)M};
  const cuuint64_t cs[1] = {(cuuint64_t)(ldc * 4)};
  const cuuint32_t cb[2] = {32u, 32u};
  const cuuint32_t ce[2] = {1, 1};
  return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, C, cd, cs, cb, ce,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN>
void launch_split3(const __nv_bfloat16* const* A, long long lda, const __nv_bfloat16* const* B,
                   long long ldb, int M, int N, int K, const TcSeg2* seg, void* C, long long ldc,
                   int out_kind, int splitk, cudaStream_t s) {
  S3Maps maps;
  S3Args args;
  for (int i = 0; i < 3; ++i) {
    const cuuint64_t ad[2] = {(cuuint64_t)K, (cuuint64_t)M}, bd[2] = {(cuuint64_t)K, (cuuint64_t)N};
    const cuuint64_t as[1] = {(cuuint64_t)(lda * 2)}, bs[1] = {(cuuint64_t)(ldb * 2)};
    const cuuint32_t ab[2] = {(cuuint32_t)kS3BK, (cuuint32_t)BM};
    const cuuint32_t bb[2] = {(cuuint32_t)kS3BK, (cuuint32_t)BN};
    maps.a[i] = make_map64(A[i], 2, ad, as, ab);
    maps.b[i] = make_map64(B[i], 2, bd, bs, bb);
  }
  args.nk1 = (K + kS3BK - 1) / kS3BK;
  args.nk2 = 0;
  args.nbc2 = args.n12 = 1;
  if (seg) {
    const long long Dr = seg->Dr, R1 = seg->R1;
    args.n12 = seg->n12;
    A2_REQUIRE(args.n12 >= 1 && BM % args.n12 == 0 && (long long)M == (long long)seg->Dl * args.n12,
               "tc GEMM segment: rows must be (a, s12) with s12 dividing 128");
    A2_REQUIRE(Dr % 8 == 0 && seg->Nb == N, "tc GEMM segment: Dr % 8 == 0, N == Dr");
    args.nbc2 = (int)((Dr + kS3BK - 1) / kS3BK);
    args.nk2 = (int)(R1 * args.nbc2);
    for (int i = 0; i < 3; ++i) {
      const cuuint64_t ad[4] = {(cuuint64_t)Dr, (cuuint64_t)args.n12, (cuuint64_t)R1,
                                (cuuint64_t)seg->Dl};
      const cuuint64_t as[3] = {(cuuint64_t)(Dr * 2), (cuuint64_t)(args.n12 * Dr * 2),
                                (cuuint64_t)(R1 * args.n12 * Dr * 2)};
      const cuuint32_t ab[4] = {(cuuint32_t)kS3BK, (cuuint32_t)args.n12, 1u,
                                (cuuint32_t)(BM / args.n12)};
      maps.a2[i] = make_map64(seg->A[i], 4, ad, as, ab);
      const cuuint64_t bd[3] = {(cuuint64_t)Dr, (cuuint64_t)R1, (cuuint64_t)N};
      const cuuint64_t bs[2] = {(cuuint64_t)(Dr * 2), (cuuint64_t)(R1 * Dr * 2)};
      const cuuint32_t bb[3] = {(cuuint32_t)kS3BK, 1u, (cuuint32_t)BN};
      maps.b2[i] = make_map64(seg->B[i], 3, bd, bs, bb);
    }
  } else {
    for (int i = 0; i < 3; ++i) {
      maps.a2[i] = maps.a[i];
      maps.b2[i] = maps.b[i];
    }
  }
  const size_t smem = sizeof(S3Smem<BN>) + 1024;
  static PerDevice<bool> set;
  set.at(current_device(), [smem] {
    A2_CUDA(cudaFuncSetAttribute(tc_split3_kernel<BN>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return true;
  });
  const int nk_total = args.nk1 + args.nk2;
  splitk = std::max(1, std::min(splitk, nk_total));
  args.M = M; args.N = N;
  args.kblocks_per_split = (nk_total + splitk - 1) / splitk;
  args.splits = (nk_total + args.kblocks_per_split - 1) / args.kblocks_per_split;
  args.C = C; args.ldc = ldc; args.out_kind = out_kind;
  args.tma_store = make_out_map(&maps.c, C, M, N, ldc) ? 1 : 0;
  if (!args.tma_store) maps.c = maps.a[0];
  const long long units = (long long)cdiv(M, BM) * cdiv(N, BN) * args.splits;
  A2_REQUIRE(units < (1LL << 31), "tcgen05 GEMM too large");
  const int grid = (int)std::min<long long>(units, device_sms());
  tc_split3_kernel<BN><<<grid, kS3Threads, smem, s>>>(maps, args);
  A2_CHECK_LAUNCH();
}

}  // namespace tc

bool tc_available() { return true; }

int tc_error_flag(bool reset) {
  int v = 0;
  A2_CUDA(cudaMemcpyFromSymbol(&v, tc::g_tc_error, sizeof(int)));
  if (reset && v) {
    int z = 0;
    A2_CUDA(cudaMemcpyToSymbol(tc::g_tc_error, &z, sizeof(int)));
  }
  return v;
}

int tc_selftest_timeout(cudaStream_t s) {
  // One 128 x 128 x 128 unit of the BF16 GEMM kernel whose producer issues no copies: the
  // MMA role's first wait (stage 0 full) can never complete, gives up after 2^14
  // iterations, raises the error word and the abort flag; the epilogue roles see the flag
  // and leave; no copy or MMA is ever in flight and TMEM is freed as on any abort.
  constexpr int n = 128;
  DevBuf a, b, c;
  a.ensure(sizeof(__nv_bfloat16) * n * n, s);
  b.ensure(sizeof(__nv_bfloat16) * n * n, s);
  c.ensure(sizeof(float) * n * n, s);
  fill_zero(a.p, sizeof(__nv_bfloat16) * n * n, s);
  fill_zero(b.p, sizeof(__nv_bfloat16) * n * n, s);
  tc::TcMaps maps;
  maps.a = tc::make_map(a.as<__nv_bfloat16>(), n, n, n, tc::BM);
  maps.b = tc::make_map(b.as<__nv_bfloat16>(), n, n, n, 128);
  maps.a2 = maps.a;
  maps.b2 = maps.b;
  maps.c = maps.a;
  tc::TcArgs args{};
  args.M = args.N = args.K = n;
  args.nk1 = n / tc::BK;
  args.nk2 = 0;
  args.nbc2 = args.n12 = 1;
  args.kblocks_per_split = args.nk1;
  args.splits = 1;
  args.C = c.p;
  args.ldc = n;
  args.out_kind = tc::OUT_F32;
  args.tma_store = 0;
  args.wait_limit = 1u << 14;
  args.no_loads = 1;
  const size_t smem = sizeof(tc::TcSmem<128, 6>) + 1024;
  A2_CUDA(cudaFuncSetAttribute(tc::tc_gemm_kernel<128, 6>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  tc::tc_gemm_kernel<128, 6><<<1, tc::kTcThreads, smem, s>>>(maps, args);
  A2_CHECK_LAUNCH();
  A2_CUDA(cudaStreamSynchronize(s));
  return tc_error_flag(true);
}

namespace {

// One GEMM configuration: the tile width and the number of K splits.
struct TcConfig {
  int bn = 256, splitk = 1;
};

// Autotuner: the first call of a GEMM shape class (tile counts of M and N, K in steps of
// 512, plain or split products, output kind, second segment) times the candidate
// configurations with CUDA events on the caller's stream and keeps the fastest for every
// later call of that class.  Candidates: BN = 128 / 256 (split products take 128 only for
// N <= 128, where the wide tile would multiply padding) and, for accumulated outputs, the
// caller's K-split count, half and twice it.  Trials with an accumulated output re-zero C
// first; the winner then runs on a zeroed C.
struct TuneKey {
  int M, N, K, split3, out_kind, seg_rows;
  bool operator<(const TuneKey& o) const {
    return std::tie(M, N, K, split3, out_kind, seg_rows) <
           std::tie(o.M, o.N, o.K, o.split3, o.out_kind, o.seg_rows);
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, TcConfig> g_tune;
bool g_tune_on = true;

template <class Run>
void tuned_gemm(int M, int N, int K, bool split3, void* C, long long ldc, int out_kind, int splitk,
                cudaStream_t s, const TcSeg2* seg, Run&& run) {
  A2_REQUIRE(K >= 1, "tc GEMM: K >= 1");
  if (splitk > 1)
    A2_REQUIRE(out_kind == tc::OUT_F32_ATOMIC, "split-K needs atomic FP32 output");
  TcConfig def;
  def.bn = N <= 128 ? 128 : 256;
  def.splitk = splitk;
  // shapes with the same tile counts (and K within 512) share one decision
  const TuneKey key{(M + 127) / 128, (N + 127) / 128, (K + 511) / 512, split3 ? 1 : 0, out_kind,
                    seg ? (seg->R1 * seg->Dr + 511) / 512 : 0};
  bool tune = false;
  TcConfig best = def;
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    if (g_tune_on) {
      auto it = g_tune.find(key);
      if (it != g_tune.end()) best = it->second;
      else tune = true;
    }
  }
  if (!tune) {
    run(best);
    return;
  }
  std::vector<TcConfig> cand;
  std::vector<int> widths = split3 ? std::vector<int>{def.bn} : std::vector<int>{128, 256};
  std::vector<int> splits{splitk};
  if (out_kind == tc::OUT_F32_ATOMIC) {
    splits.push_back(splitk * 2);
    if (splitk > 1) splits.push_back(std::max(1, splitk / 2));
  }
  for (int v : widths)
    for (int k : splits) cand.push_back(TcConfig{v, k});
  const size_t cbytes = (size_t)M * ldc * (out_kind == tc::OUT_BF16 ? 2 : 4);
  cudaEvent_t e0, e1;
  A2_CUDA(cudaEventCreate(&e0));
  A2_CUDA(cudaEventCreate(&e1));
  float best_ms = 1e30f;
  for (const TcConfig& cf : cand) {
    if (out_kind == tc::OUT_F32_ATOMIC) fill_zero(C, cbytes, s);
    A2_CUDA(cudaEventRecord(e0, s));
    run(cf);
    A2_CUDA(cudaEventRecord(e1, s));
    A2_CUDA(cudaEventSynchronize(e1));
    float ms = 0.f;
    A2_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    if (ms < best_ms) {
      best_ms = ms;
      best = cf;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune[key] = best;
  }
  if (out_kind == tc::OUT_F32_ATOMIC) fill_zero(C, cbytes, s);
  run(best);
}

}  // namespace

void tc_autotune(bool on) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  g_tune_on = on;
  if (!on) g_tune.clear();
}

void tc_gemm_bf16(const __nv_bfloat16* A, long long lda, const __nv_bfloat16* B, long long ldb,
                  int M, int N, int K, void* C, long long ldc, int out_kind, int splitk,
                  cudaStream_t s, const TcSeg2* seg) {
  if (M <= 0 || N <= 0) return;
  tuned_gemm(M, N, K, false, C, ldc, out_kind, splitk, s, seg, [&](const TcConfig& cf) {
    if (cf.bn == 128)
      tc::launch<128, 6>(A, lda, B, ldb, M, N, K, seg, C, ldc, out_kind, cf.splitk, s);
    else
      tc::launch<256, 4>(A, lda, B, ldb, M, N, K, seg, C, ldc, out_kind, cf.splitk, s);
  });
}

void tc_gemm_split3(const __nv_bfloat16* const* A, long long lda, const __nv_bfloat16* const* B,
                    long long ldb, int M, int N, int K, float* C, long long ldc, bool add,
                    int splitk, cudaStream_t s, const TcSeg2* seg) {
  if (M <= 0 || N <= 0) return;
  const int out_kind = add ? tc::OUT_F32_ATOMIC : tc::OUT_F32;
  tuned_gemm(M, N, K, true, C, ldc, out_kind, splitk, s, seg, [&](const TcConfig& cf) {
    if (cf.bn == 128)
      tc::launch_split3<128>(A, lda, B, ldb, M, N, K, seg, C, ldc, out_kind, cf.splitk, s);
    else
      tc::launch_split3<256>(A, lda, B, ldb, M, N, K, seg, C, ldc, out_kind, cf.splitk, s);
  });
}

// -------------------------------------------------------------- BF16 H_eff chain
namespace {
int s4_splitk(long long M4, int Dr, long long kblocks) {
  const long long tiles = (long long)cdiv(M4, 128) * cdiv(Dr, Dr <= 128 ? 128 : 256);
  int splitk = (int)std::max<long long>(1, 2 * 152 / std::max<long long>(1, tiles));
  return std::min<int>(splitk, std::max<int>(1, (int)(kblocks / 8)));
}
}  // namespace

void tc_heff_bf16(cudaStream_t s, int n1, int n2, int Rl, int R1, int Rr, int Dl, int Dr,
                  const __nv_bfloat16* Lb, long long ldl, const __nv_bfloat16* Rb, long long ldr,
                  const double* x, float* y, const SparseRows<float>& W1,
                  const SparseRows<float>& W2, const HeffFold& F, DevBuf& t1, DevBuf& t2,
                  DevBuf& xa, DevBuf& tf) {
  (void)tf;
  const long long NX = (long long)n1 * n2 * Dr;          // columns of S1
  const long long ldx = pad8(Dl);
  const long long s1 = (long long)Dl * Rl * NX;
  const long long s2 = (long long)Dl * R1 * NX;
  const long long K4 = (long long)Rr * Dr;
  const long long ld3 = pad8(K4);
  const long long s3 = (long long)Dl * n1 * n2 * ld3;
  xa.ensure(sizeof(__nv_bfloat16) * (size_t)NX * ldx, s);
  t1.ensure(sizeof(__nv_bfloat16) * (size_t)std::max(s1, s3), s);
  t2.ensure(sizeof(__nv_bfloat16) * (size_t)s2, s);
  __nv_bfloat16* XT = xa.as<__nv_bfloat16>();
  __nv_bfloat16* T1 = t1.as<__nv_bfloat16>();
  __nv_bfloat16* T2 = t2.as<__nv_bfloat16>();
  __nv_bfloat16* T3 = t1.as<__nv_bfloat16>();
  // x [Dl][(t1 t2 b')] -> XT [(t1 t2 b')][a'] (row stride ldx)
  // (pad columns a' >= Dl are never read: the tensor map's K extent is Dl)
  transpose2d_ld<double, __nv_bfloat16>(x, XT, Dl, (int)NX, ldx, s);
  // S1: T1[(a w)][(t1 t2 b')] = sum_a' L[(a w)][a'] XT[(t1 t2 b')][a']
  {
    const double M = (double)Dl * Rl, N = (double)NX, K = Dl;
    ProfScope ps(PK_TC_S1, s, 2.0 * M * N * K, 2.0 * (M * K + N * K + M * N));
    tc_gemm_bf16(Lb, ldl, XT, ldx, Dl * Rl, (int)NX, Dl, T1, NX, tc::OUT_BF16, 1, s);
  }
  if (F.Lt) {   // folded G of A_k: T2[(a w1)][(s1 t2 b')] = sum_a' Lt[(a w1)][a'] XT
    const double M = (double)Dl * R1, N = (double)NX, K = Dl;
    ProfScope ps(PK_TC_S1, s, 2.0 * M * N * K, 2.0 * (M * K + N * K + M * N));
    tc_gemm_bf16(F.Lt, ldl, XT, ldx, Dl * R1, (int)NX, Dl, T2, NX, tc::OUT_BF16, 1, s);
  }
  {  // S2 (W_rest added to the folded part when A_k is folded)
    ProfScope ps(PK_SPARSE_S2, s, 2.0 * W1.nnz_total * (double)n2 * Dr * Dl,
                 2.0 * (double)(s1 + s2) * (F.Lt ? 1.5 : 1.0));
    SparseGeom gm;
    gm.veclen = n2 * Dr;
    gm.in_sw = NX; gm.in_st = (long long)n2 * Dr;
    gm.out_sw = NX; gm.out_ss = (long long)n2 * Dr;
    gm.B1 = Dl; gm.in_b1 = (long long)Rl * NX; gm.out_b1 = (long long)R1 * NX;
    gm.accumulate = F.Lt ? 1 : 0;
    sparse_rows_apply<__nv_bfloat16, __nv_bfloat16, float>(W1, gm, T1, T2, s);
  }
  {  // S3 -> T3[(a s1 s2)][(w2 b')] with row stride ld3
    ProfScope ps(PK_SPARSE_S3, s, 2.0 * W2.nnz_total * (double)Dr * Dl * n1,
                 2.0 * (double)s2 + 2.0 * (double)Dl * n1 * n2 * Rr * Dr);
    SparseGeom gm;
    gm.veclen = Dr;
    gm.in_sw = NX; gm.in_st = Dr;
    gm.out_sw = Dr; gm.out_ss = ld3;
    gm.B1 = Dl; gm.B2 = n1;
    gm.in_b1 = (long long)R1 * NX; gm.in_b2 = (long long)n2 * Dr;
    gm.out_b1 = (long long)n1 * n2 * ld3; gm.out_b2 = (long long)n2 * ld3;
    sparse_rows_apply<__nv_bfloat16, __nv_bfloat16, float>(W2, gm, T2, T3, s);
  }
  // S4: y[(a s1 s2)][b] = sum_{(w2 b')} T3 HR[b][(w2 b')]   (split K, atomic FP32)
  //     (+ sum_{(w1 b')} T2[a][w1][(s1 s2)][b'] Rt[b][w1][b'] when A_{k+1} is folded)
  const int M4 = Dl * n1 * n2;
  TcSeg2 seg;
  long long kb = (K4 + 63) / 64;
  if (F.Rt) {
    seg.A[0] = seg.A[1] = seg.A[2] = T2;
    seg.B[0] = seg.B[1] = seg.B[2] = F.Rt;
    seg.Dl = Dl; seg.n12 = n1 * n2; seg.R1 = R1; seg.Dr = Dr; seg.Nb = Dr;
    kb += (long long)R1 * ((Dr + 63) / 64);
  }
  {
    const double M = M4, N = Dr, K = (double)K4 + (F.Rt ? (double)R1 * Dr : 0.0);
    ProfScope ps(PK_TC_S4, s, 2.0 * M * N * K, 2.0 * (M * K + N * K) + 4.0 * M * N);
    fill_zero(y, sizeof(float) * (size_t)M4 * Dr, s);
    tc_gemm_bf16(T3, ld3, Rb, ldr, M4, Dr, (int)K4, y, Dr, tc::OUT_F32_ATOMIC,
                 s4_splitk(M4, Dr, kb), s, F.Rt ? &seg : nullptr);
  }
}

}  // namespace a2

namespace a2 {

// y = H_eff x with FP32-accurate tensor-core products: every BF16 GEMM operand is the
// three-plane split of an FP32/FP64 value and six plane pairs are accumulated in TMEM;
// the sparse MPO stages run in FP32.  L, R: three BF16 planes each (plane strides
// lplane / rplane elements, row strides ldl / ldr).  When A_{k+1} is folded, T2 is kept
// as three BF16 planes (the second K segment of S4 reads it through TMA).
void tc_heff_f32emu(cudaStream_t s, int n1, int n2, int Rl, int R1, int Rr, int Dl, int Dr,
                    const __nv_bfloat16* Lp, long long ldl, long long lplane,
                    const __nv_bfloat16* Rp, long long ldr, long long rplane, const double* x,
                    float* y, const SparseRows<float>& W1, const SparseRows<float>& W2,
                    const HeffFold& F, DevBuf& t1, DevBuf& t2, DevBuf& xa, DevBuf& tf) {
  const long long NX = (long long)n1 * n2 * Dr;
  const long long ldx = pad8(Dl);
  const long long xplane = NX * ldx;
  const long long s1 = (long long)Dl * Rl * NX;
  const long long s2 = (long long)Dl * R1 * NX;
  const long long p2 = (s2 + 63) / 64 * 64;          // T2 plane stride (split form)
  const long long K4 = (long long)Rr * Dr;
  const long long ld3 = pad8(K4);
  const long long M4 = (long long)Dl * n1 * n2;
  const long long plane3 = M4 * ld3;
  const bool t2split = F.Rt != nullptr;
  xa.ensure(sizeof(__nv_bfloat16) * (size_t)(3 * xplane), s);
  t1.ensure(std::max(sizeof(float) * (size_t)s1, sizeof(__nv_bfloat16) * (size_t)(3 * plane3)), s);
  t2.ensure(t2split ? sizeof(__nv_bfloat16) * (size_t)(3 * p2) : sizeof(float) * (size_t)s2, s);
  __nv_bfloat16* XT = xa.as<__nv_bfloat16>();
  float* T1 = t1.as<float>();
  float* T2 = t2.as<float>();
  __nv_bfloat16* T2p = t2.as<__nv_bfloat16>();
  __nv_bfloat16* T3 = t1.as<__nv_bfloat16>();
  // with both cores folded the S1-fold product needs its own FP32 buffer
  float* Tg = nullptr;
  if (F.Lt && t2split) {
    tf.ensure(sizeof(float) * (size_t)s2, s);
    Tg = tf.as<float>();
  }
  transpose_split3(x, Dl, (int)NX, XT, ldx, xplane, s);
  {  // S1
    const __nv_bfloat16* A[3] = {Lp, Lp + lplane, Lp + 2 * lplane};
    const __nv_bfloat16* B[3] = {XT, XT + xplane, XT + 2 * xplane};
    const double M = (double)Dl * Rl, N = (double)NX, K = Dl;
    ProfScope ps(PK_EMU_S1, s, 6.0 * 2.0 * M * N * K, 6.0 * (M * K + N * K) + 4.0 * M * N);
    tc_gemm_split3(A, ldl, B, ldx, Dl * Rl, (int)NX, Dl, T1, NX, false, 1, s);
  }
  if (F.Lt) {   // folded G of A_k: Lt x, FP32 (into T2, or into Tg when T2 is split)
    const __nv_bfloat16* A[3] = {F.Lt, F.Lt + F.ltplane, F.Lt + 2 * F.ltplane};
    const __nv_bfloat16* B[3] = {XT, XT + xplane, XT + 2 * xplane};
    const double M = (double)Dl * R1, N = (double)NX, K = Dl;
    ProfScope ps(PK_EMU_S1, s, 6.0 * 2.0 * M * N * K, 6.0 * (M * K + N * K) + 4.0 * M * N);
    tc_gemm_split3(A, ldl, B, ldx, Dl * R1, (int)NX, Dl, Tg ? Tg : T2, NX, false, 1, s);
  }
  {  // S2 (FP32; W_rest added to the folded part when A_k is folded)
    ProfScope ps(PK_EMU_S2, s, 2.0 * W1.nnz_total * (double)n2 * Dr * Dl,
                 4.0 * (double)(s1 + s2) * (F.Lt ? 1.5 : 1.0));
    SparseGeom gm;
    gm.veclen = n2 * Dr;
    gm.in_sw = NX; gm.in_st = (long long)n2 * Dr;
    gm.out_sw = NX; gm.out_ss = (long long)n2 * Dr;
    gm.B1 = Dl; gm.in_b1 = (long long)Rl * NX; gm.out_b1 = (long long)R1 * NX;
    if (t2split) {
      sparse_rows_apply_split3<float, float>(W1, gm, T1, 0, Tg, T2p, p2, s);
    } else {
      gm.accumulate = F.Lt ? 1 : 0;
      sparse_rows_apply<float, float, float>(W1, gm, T1, T2, s);
    }
  }
  {  // S3 (FP32 or split input, three BF16 planes out)
    ProfScope ps(PK_EMU_S3, s, 2.0 * W2.nnz_total * (double)Dr * Dl * n1,
                 (t2split ? 6.0 : 4.0) * (double)s2 + 6.0 * (double)M4 * K4);
    SparseGeom gm;
    gm.veclen = Dr;
    gm.in_sw = NX; gm.in_st = Dr;
    gm.out_sw = Dr; gm.out_ss = ld3;
    gm.B1 = Dl; gm.B2 = n1;
    gm.in_b1 = (long long)R1 * NX; gm.in_b2 = (long long)n2 * Dr;
    gm.out_b1 = (long long)n1 * n2 * ld3; gm.out_b2 = (long long)n2 * ld3;
    if (t2split)
      sparse_rows_apply_split3<__nv_bfloat16, float>(W2, gm, T2p, p2, nullptr, T3, plane3, s);
    else
      sparse_rows_apply_split3<float, float>(W2, gm, T2, 0, nullptr, T3, plane3, s);
  }
  {  // S4 (+ the folded G of A_{k+1} as a second K segment over T2)
    const __nv_bfloat16* A[3] = {T3, T3 + plane3, T3 + 2 * plane3};
    const __nv_bfloat16* B[3] = {Rp, Rp + rplane, Rp + 2 * rplane};
    TcSeg2 seg;
    long long kb = (K4 + 63) / 64;
    if (t2split) {
      for (int i = 0; i < 3; ++i) {
        seg.A[i] = T2p + i * p2;
        seg.B[i] = F.Rt + i * F.rtplane;
      }
      seg.Dl = Dl; seg.n12 = n1 * n2; seg.R1 = R1; seg.Dr = Dr; seg.Nb = Dr;
      kb += (long long)R1 * ((Dr + 63) / 64);
    }
    const double M = (double)M4, N = Dr, K = (double)K4 + (t2split ? (double)R1 * Dr : 0.0);
    ProfScope ps(PK_EMU_S4, s, 6.0 * 2.0 * M * N * K, 6.0 * (M * K + N * K) + 4.0 * M * N);
    fill_zero(y, sizeof(float) * (size_t)M4 * Dr, s);
    tc_gemm_split3(A, ld3, B, ldr, (int)M4, Dr, (int)K4, y, Dr, true, s4_splitk(M4, Dr, kb), s,
                   t2split ? &seg : nullptr);
  }
}


// One-site H_eff with FP32-accurate tensor-core products (the one-site case of Alg. 2):
// T1 = L x (as S1), T2 = the MPO core on the rows in FP32 with three BF16 output planes
// (as S3), y = T2 R^T (as S4).
void tc_heff1_f32emu(cudaStream_t s, int n, int Rl, int Rr, int Dl, int Dr,
                     const __nv_bfloat16* Lp, long long ldl, long long lplane,
                     const __nv_bfloat16* Rp, long long ldr, long long rplane, const double* x,
                     float* y, const SparseRows<float>& W, DevBuf& t1, DevBuf& t2, DevBuf& xa) {
  const long long NX = (long long)n * Dr;
  const long long ldx = pad8(Dl);
  const long long xplane = (NX * ldx + 63) / 64 * 64;
  const long long s1 = (long long)Dl * Rl * NX;
  const long long K4 = (long long)Rr * Dr;
  const long long ld3 = pad8(K4);
  const long long M4 = (long long)Dl * n;
  const long long plane3 = (M4 * ld3 + 63) / 64 * 64;
  xa.ensure(sizeof(__nv_bfloat16) * (size_t)(3 * xplane), s);
  t1.ensure(sizeof(float) * (size_t)s1, s);
  t2.ensure(sizeof(__nv_bfloat16) * (size_t)(3 * plane3), s);
  __nv_bfloat16* XT = xa.as<__nv_bfloat16>();
  float* T1 = t1.as<float>();
  __nv_bfloat16* T2 = t2.as<__nv_bfloat16>();
  transpose_split3(x, Dl, (int)NX, XT, ldx, xplane, s);
  {
    const __nv_bfloat16* A[3] = {Lp, Lp + lplane, Lp + 2 * lplane};
    const __nv_bfloat16* B[3] = {XT, XT + xplane, XT + 2 * xplane};
    const double M = (double)Dl * Rl, N = (double)NX, K = Dl;
    ProfScope ps(PK_EMU_S1, s, 6.0 * 2.0 * M * N * K, 6.0 * (M * K + N * K) + 4.0 * M * N);
    tc_gemm_split3(A, ldl, B, ldx, Dl * Rl, (int)NX, Dl, T1, NX, false, 1, s);
  }
  {
    ProfScope ps(PK_EMU_S3, s, 2.0 * W.nnz_total * (double)Dr * Dl,
                 4.0 * (double)s1 + 6.0 * (double)M4 * K4);
    SparseGeom gm;
    gm.veclen = Dr;
    gm.in_sw = NX; gm.in_st = Dr;
    gm.out_sw = Dr; gm.out_ss = ld3;
    gm.B1 = Dl; gm.in_b1 = (long long)Rl * NX; gm.out_b1 = (long long)n * ld3;
    sparse_rows_apply_split3<float, float>(W, gm, T1, 0, nullptr, T2, plane3, s);
  }
  {
    const __nv_bfloat16* A[3] = {T2, T2 + plane3, T2 + 2 * plane3};
    const __nv_bfloat16* B[3] = {Rp, Rp + rplane, Rp + 2 * rplane};
    const double M = (double)M4, N = Dr, K = (double)K4;
    ProfScope ps(PK_EMU_S4, s, 6.0 * 2.0 * M * N * K, 6.0 * (M * K + N * K) + 4.0 * M * N);
    fill_zero(y, sizeof(float) * (size_t)M4 * Dr, s);
    tc_gemm_split3(A, ld3, B, ldr, (int)M4, Dr, (int)K4, y, Dr, true,
                   s4_splitk(M4, Dr, (K4 + 63) / 64), s);
  }
}

// ============================================================================ FP64 emulation
// Ozaki scheme (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its applications",
// Numer. Algorithms 59, 2012) on the BF16 tensor cores.  Every 256-wide chunk of a row of an
// FP64 operand is brought to 55-bit fixed point at the scale of its largest entry, S = X[r][k]
// 2^(55 - e) rounded to an integer, e = ilogb(max_k |X[r][k]|) + 1 over the chunk, and S is written
// in balanced digits of radix 2^kOzBits: slice i holds q_i 2^(e + 1 - 8 i) with -128 <= q_i <= 127
// (the leading digit up to 128), exact in BF16.  Balanced digits use BF16's whole
// significand (7 slices for 55 bits; digits of one sign would need 8 slices and 36 pairs for
// the same products of 2^14).  A product of slice i of A with slice j of B is an integer
// multiple of the unit 2^(e_A + e_B + 2 - 8 (i + j)) of the chunk; the pairs with i + j <= 8 are
// kept (28).  Of those left out, level 9 counts: six pairs of at most 2^-56 of the scales each, in
// all at most 2^-53.4 a product (eight slices of 7 bits and 36 pairs left out as much).  See
// tc_oz_kernel for the accumulation chunk by chunk.
// Range: slices are BF16 values, so a chunk that holds a NaN, an infinity or an entry of 2^128 or
// more has no slices.  Its first slice is written as NaN, which reaches every product of
// the row.  At the other end, slices whose scale lies below 2^-126 are zero: chunks whose largest
// entry is below 2^-72 keep an absolute accuracy of about 2^-126 instead of their 55 bits.
namespace {

static_assert(kOzSlices == 7 && kOzBits == 8, "the digits cover 55 bits and a sign");

__device__ __forceinline__ float pow2f(int k) {
  return (k >= -126 && k <= 127) ? __int_as_float((k + 127) << 23) : 0.f;
}

// Scale of slice i (1 ... kOzSlices) of a chunk whose entries are below 2^e.
__device__ __forceinline__ float oz_scale(int e, int i) {
  return i == 1 && e > 128 ? __int_as_float(0x7fffffff) : pow2f(e + 1 - kOzBits * i);
}

// Slicing with integer operations only (the FP64 pipe is slow on this part): the signed
// 55-bit fixed-point value of v at the row's scale 2^e (|v| < 2^e), rounded to nearest.
__device__ __forceinline__ long long oz_fixed(double v, int e) {
  const long long bits = __double_as_longlong(v);
  int f = (int)((bits >> 52) & 0x7FF);
  long long m = bits & ((1ll << 52) - 1);
  if (f) m |= 1ll << 52;
  else f = 1;                                    // subnormal: no hidden bit
  const int sh = f - e - 1020;                   // <= 2 since |v| < 2^e
  if (sh >= 0) m <<= sh;
  else m = sh > -60 ? (m + (1ll << (-sh - 1))) >> -sh : 0ll;
  return bits < 0 ? -m : m;
}
// The last digit of S (slice kOzSlices - t for the t-th call) and S without it.
__device__ __forceinline__ int oz_digit(long long& S) {
  const int q = (int)(signed char)(S & 0xFF);
  S = (S - q) >> kOzBits;
  return q;
}
// The digits of S as floats, slice 1 first (the leading digit takes what is left).
__device__ __forceinline__ void oz_digits(long long S, int (&q)[kOzSlices]) {
#pragma unroll
  for (int i = kOzSlices - 1; i > 0; --i) q[i] = oz_digit(S);
  q[0] = (int)S;
}

// Four digits at the scale sc as BF16 (exact).
__device__ __forceinline__ uint2 oz_pack(int a, int b, int c, int d, float sc) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn((float)a * sc, (float)b * sc);
  const __nv_bfloat162 hi = __floats2bfloat162_rn((float)c * sc, (float)d * sc);
  uint2 pk;
  pk.x = *reinterpret_cast<const unsigned int*>(&lo);
  pk.y = *reinterpret_cast<const unsigned int*>(&hi);
  return pk;
}

// One warp per row and 256-wide K chunk, whose entries stay in registers (eight per lane): one
// read, the chunk's largest exponent by a warp reduction, then each slice of four
// consecutive entries as one 8-byte vector.  The last K block is filled with zeros.  Bound by
// HBM: 8 bytes read and 14 written per entry.  Rows whose entries lie far apart (sk > 1, sr = 1: x,
// ket, bra) take this kernel too: neighbouring warps read neighbouring rows, whose sectors meet in
// L1 and L2 (x at D = 256, 4096 x 256: 12 us, by ozaki_split_cols_kernel 23; D = 64 7, 9; D = 512
// 27, 44).  With one scale for a whole row (read twice, one
// warp for 143872 entries of T3) the slicing of S4's operand took 2.75 ms at D = 256 with the
// slicing of x, now 1.82.
constexpr int kOzGroup = 256;              // entries that share a scale (tc_oz_kernel's chunk)
static_assert(kOzGroup == tc::kOzChunk * tc::kOzBK, "a chunk of the GEMM has one scale");
__global__ void __launch_bounds__(256)
ozaki_split_kernel(const double* __restrict__ X, long long sr, long long sk, int rows, int K,
                   __nv_bfloat16* __restrict__ P, long long ntasks) {
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int Kp = (K + kOzKBlock - 1) / kOzKBlock * kOzKBlock;
  for (long long task = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; task < ntasks;
       task += nwarps) {
    const int ch = (int)(task / rows), r = (int)(task - (long long)ch * rows);
    const double* xr = X + (long long)r * sr;
    double v[8];
    int fm = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = ch * kOzGroup + (u >> 2) * 128 + 4 * lane + (u & 3);
      v[u] = k < K ? xr[(long long)k * sk] : 0.0;
      fm = max(fm, (__double2hiint(v[u]) >> 20) & 0x7FF);
    }
    fm = __reduce_max_sync(0xffffffffu, fm);
    const int e = max(fm, 1) - 1022;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k0 = ch * kOzGroup + h * 128 + 4 * lane;
      if (k0 >= Kp) continue;
      int q[4][kOzSlices];
#pragma unroll
      for (int u = 0; u < 4; ++u) oz_digits(oz_fixed(v[4 * h + u], e), q[u]);
      __nv_bfloat16* dst =
          P + ((long long)(k0 / kOzKBlock) * rows + r) * kOzRowBlock + k0 % kOzKBlock;
#pragma unroll
      for (int i = 0; i < kOzSlices; ++i)
        *reinterpret_cast<uint2*>(dst + i * kOzKBlock) =
            oz_pack(q[0][i], q[1][i], q[2][i], q[3][i], oz_scale(e, i + 1));
    }
  }
}

// Slices of the rows of X^T, X a (K x N) row-major matrix (row stride ldx): output row n
// holds X[k][n], k < K.  A block takes 32 consecutive output rows and one K chunk, held in
// registers (32 entries per thread, read row by row of X, coalesced); the digits of 64 k at a
// time go through shared memory and leave as 8-byte vectors along K.  Same slices as
// ozaki_split of the transposed matrix.  Environment update, T2 1024 x 113664: 0.75 ms with two
// reads (one scale per row), now 0.68.
constexpr int kOzColChunk = 64, kOzColPad = kOzColChunk + 4;   // row of 68 BF16 = 136 B
__global__ void __launch_bounds__(256)
ozaki_split_cols_kernel(const double* __restrict__ X, long long ldx, int N, int K,
                        __nv_bfloat16* __restrict__ P) {
  __shared__ int emax[8][32];
  __shared__ __align__(16) __nv_bfloat16 tile[kOzSlices][32][kOzColPad];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n0 = blockIdx.x * 32, n = n0 + lane, kc = blockIdx.y * kOzGroup;
  const int Kp = (K + kOzKBlock - 1) / kOzKBlock * kOzKBlock;
  double v[kOzGroup / 8];
  int fm = 0;
#pragma unroll
  for (int t = 0; t < kOzGroup / 8; ++t) {
    const int k = kc + warp + 8 * t;
    v[t] = n < N && k < K ? X[(long long)k * ldx + n] : 0.0;
    fm = max(fm, (__double2hiint(v[t]) >> 20) & 0x7FF);
  }
  emax[warp][lane] = fm;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) fm = max(fm, emax[w][lane]);
  const int e = max(fm, 1) - 1022;
#pragma unroll
  for (int c = 0; c < kOzGroup / kOzColChunk; ++c) {
    const int k0 = kc + c * kOzColChunk;
    if (k0 >= Kp) break;
#pragma unroll
    for (int t = 0; t < kOzColChunk / 8; ++t) {
      int q[kOzSlices];
      oz_digits(oz_fixed(v[c * (kOzColChunk / 8) + t], e), q);
#pragma unroll
      for (int i = 0; i < kOzSlices; ++i)
        tile[i][lane][warp + 8 * t] =
            __float2bfloat16_rn((float)q[i] * oz_scale(e, i + 1));
    }
    __syncthreads();
    // vectors of 4 values, the slices of one (row, K block) one after another in memory
    for (int w = threadIdx.x; w < kOzSlices * 32 * (kOzColChunk / 4); w += 256) {
      const int c4 = w % (kOzKBlock / 4), i = (w / (kOzKBlock / 4)) % kOzSlices;
      const int rk = w / (kOzKBlock / 4 * kOzSlices), r = rk % 32, k = k0 + rk / 32 * kOzKBlock;
      if (n0 + r >= N || k >= Kp) continue;
      *reinterpret_cast<uint2*>(P + ((long long)(k / kOzKBlock) * N + n0 + r) * kOzRowBlock +
                                i * kOzKBlock + 4 * c4) =
          *reinterpret_cast<const uint2*>(&tile[i][r][rk / 32 * kOzKBlock + 4 * c4]);
    }
    __syncthreads();
  }
}

// C[r][c] = sum of the K splits' FP32 pairs (tile t at T + t * MN, row-major with N columns),
// in double-float arithmetic: the two-sum keeps the running sum as an FP32 pair hi + lo
// (~2^-48), and the result is written as FP64 (hi + lo) or as the pair.
template <bool DF>
__global__ void ozaki_combine_kernel(const float* __restrict__ T, long long MN, int nt, int N,
                                     double* __restrict__ C, float* __restrict__ Cdf,
                                     long long df_plane, long long ldc) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < MN;
       e += (long long)gridDim.x * blockDim.x) {
    float hi = 0.f, lo = 0.f;
    for (int t = nt - 1; t >= 0; --t) {
      const float v = __ldg(T + (long long)t * MN + e);
      const float s = __fadd_rn(hi, v);
      const float bp = __fsub_rn(s, hi);
      const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(v, bp));
      hi = s;
      lo = __fadd_rn(lo, err);
    }
    const long long o = (e / N) * ldc + e % N;
    if constexpr (DF) {   // renormalised pair
      const float s = __fadd_rn(hi, lo);
      Cdf[o] = s;
      Cdf[df_plane + o] = __fsub_rn(lo, __fsub_rn(s, hi));
    } else {
      C[o] = (double)hi + (double)lo;
    }
  }
}

}  // namespace

void ozaki_split_cols(const double* X, long long ldx, int N, int K, __nv_bfloat16* P,
                      cudaStream_t s) {
  if (N <= 0 || K <= 0) return;
  constexpr int kMost = 65535 * kOzGroup;              // grid.y chunks of a launch
  for (long long k0 = 0; k0 < K; k0 += kMost) {
    const int kn = (int)std::min<long long>(K - k0, kMost);
    ozaki_split_cols_kernel<<<dim3((N + 31) / 32, cdiv(kn, kOzGroup)), 256, 0, s>>>(
        X + k0 * ldx, ldx, N, kn, P + k0 / kOzKBlock * N * kOzRowBlock);
    A2_CHECK_LAUNCH();
  }
}

void ozaki_split(const double* X, long long sr, long long sk, int rows, int K, __nv_bfloat16* P,
                 cudaStream_t s) {
  if (rows <= 0 || K <= 0) return;
  const long long ntasks = (long long)rows * cdiv(K, kOzGroup);
  const int grid = (int)std::min<long long>((ntasks + 7) / 8, 152 * 32);   // eight warps per block
  ozaki_split_kernel<<<grid, 256, 0, s>>>(X, sr, sk, rows, K, P, ntasks);
  A2_CHECK_LAUNCH();
}

void tc_gemm_f64emu(const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K, double* C,
                    long long ldc, DevBuf& slab, cudaStream_t s, float* Cdf, long long df_plane) {
  if (M <= 0 || N <= 0) return;
  const int num_sms = device_sms();
  // K splits: at most kOzSplitBlocks K blocks per split (bounds the number of sums per
  // accumulator, hence the rounding of its lo part), and enough work units to fill the GPU
  // when the output has few tiles
  static_assert(kOzKBlock == tc::kOzBK, "K block of the sliced layout");
  constexpr int kOzSplitBlocks = 4096 / tc::kOzBK;
  const int nk = (K + tc::kOzBK - 1) / tc::kOzBK;
  const long long tiles = (long long)cdiv(M, tc::BM) * cdiv(N, tc::kOzBN);
  int splits = cdiv(nk, kOzSplitBlocks);
  if (tiles < num_sms) splits = std::max<int>(splits, (int)cdiv(2LL * num_sms, tiles));
  splits = std::max(1, std::min(splits, cdiv(nk, 2)));
  splits = cdiv(nk, cdiv(nk, splits));   // the count launch_oz will use
  if (splits == 1) {
    if (Cdf) tc::launch_oz(A, B, M, N, K, 1, tc::OZ_PAIR, Cdf, ldc, df_plane, s);
    else tc::launch_oz(A, B, M, N, K, 1, tc::OZ_F64, C, ldc, 0, s);
    return;
  }
  const long long MN = (long long)M * N;
  slab.ensure(sizeof(float) * (size_t)(2LL * splits * MN), s);
  float* T = slab.as<float>();
  tc::launch_oz(A, B, M, N, K, splits, tc::OZ_SPLIT, T, N, 0, s);
  const int grid = (int)std::min<long long>((MN + 255) / 256, 152LL * 16);
  if (Cdf)
    ozaki_combine_kernel<true><<<grid, 256, 0, s>>>(T, MN, 2 * splits, N, nullptr, Cdf,
                                                    df_plane, ldc);
  else
    ozaki_combine_kernel<false><<<grid, 256, 0, s>>>(T, MN, 2 * splits, N, C, nullptr, 0, ldc);
  A2_CHECK_LAUNCH();
}

}  // namespace a2
