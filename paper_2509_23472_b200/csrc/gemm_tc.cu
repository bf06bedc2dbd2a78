// Tensor-core engine for the dense contractions of the path (the sketch and the projection of Algorithm 1, the Gram
// matrices of the orthonormalisation, the application of the triangular factors, Reconstruct).
//
// Written for sm_100a: up to four threads fill a shared-memory ring of three to twelve stages by TMA (cp.async.bulk.tensor,
// 128-byte swizzle, no multicast), one thread issues tcgen05.mma (kind::f16, bf16 operands, M = 128,
// N <= 256, K = 16 per instruction) into an fp32 accumulator in tensor memory, eight warps read the
// accumulator back with tcgen05.ld and write the result.  Operands may be K-major or MN-major, which
// covers X Omega^T (K/K), U^T X and Y^T Y (MN/MN) and U V (K/MN) without transposing anything in memory.
// A contraction can be the sum of up to three products over the same shapes (split-precision terms),
// and can be split over K into partial results that a later kernel adds in a fixed order.
//
// Every wait on an mbarrier is bounded by a wall-clock limit; on expiry the kernel records
// LORACT_DEV_WAIT_EXPIRED, stops issuing work, frees its tensor memory and returns.
#include <cuda.h>

#include <map>
#include <atomic>
#include <mutex>
#include <tuple>

#include "common.cuh"

namespace loract {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;          // bf16 elements = one 128-byte swizzle row
// Stages of the operand ring: as many as fit, up to kMaxStages and to the K blocks there are (a short product leaves shared
// memory to the kernel behind it).  A stage of a narrow product is small, and what hides the latency of HBM is the bytes in
// flight.
constexpr int kMaxStages = 12;
constexpr uint32_t kRingBytes = 208 * 1024;
constexpr int kThreads = 320;    // warps 0, 2, 3, 4: TMA (kProducers), warp 1: MMA + tensor memory, warps 2..9: epilogue
constexpr int kProducers = 4;    // warps that fill the ring, at most
constexpr int kEpiWarps = 8;     // two per quarter of the tensor-memory lanes: they take alternate column groups
constexpr uint32_t kABytes = kBM * kBK * 2;
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s

struct alignas(64) TmapPack {
  CUtensorMap a[3];
  CUtensorMap b[3];
  CUtensorMap c[2];   // outputs (C0, C1) for the staged epilogue: boxes of 128 bytes x 32 rows.  Fused epilogue: the
                      // output and the matrix it is combined with, both in boxes of 64 bytes x 32 rows
};

struct TcParams {
  int M, N;
  int bn;             // tile width, multiple of 16, <= 256
  int kb_total;       // 64-wide K blocks per term
  int kb_per_split;
  int n_terms;
  int out;
  void* C0;
  void* C1;
  int64_t ldc;
  int64_t split_stride;
  uint32_t b_bytes;   // bytes of one B stage
  uint32_t tmem_cols;
  int accumulate;     // OUT_F32, one split: C += result
  const float* ep_row_a;   // OUT_RMS_BWD
  const float* ep_row_b;
  const void* ep_col;
  uint32_t* dev_status;
  int tma_store;      // 1: the epilogue stages 32-row boxes in shared memory and writes them with TMA stores
  int st_m_tiles;     // streaming kernel: 256-row tiles along M
  int st_units;       // streaming kernel: tiles in all (column tile major, then M)
  int st_keep_a;      // streaming kernel: ask for A to stay in L2
  int st_stages;      // streaming kernel: stages of the A ring (<= kStreamStages)
  int store_bufs;     // staging boxes per epilogue warp (one-tile kernels 2 or 4, streaming 1 or 2, fused epilogue 2 or 3)
  int fuse_parts;     // fused epilogue: warps per quarter of the accumulator's rows
  int stages;         // one-tile kernels: stages of the ring
  int lower;          // wide forms: the operand with two tiles is lower triangular (see GemmDesc::lower)
  int a_rows;         // rows of an A tile that one load brings: 64 (one-CTA kernel, up to 64 rows in all), otherwise kBM
  int panels;         // MN-major operands whose map has three dimensions (one load for all panels): bit 0 A, bit 1 B
  int early;          // operands that may be loaded before griddepcontrol.wait: bit 0 A, bit 1 B (streaming kernel: all)
  int halve_at_term;  // the accumulator is multiplied by 1/2 before the first product of this term (0: never)
  int a_keep_from_kb; // two-CTA kernel: K block from which the loads of A carry an evict-last hint (kb_total: none)
  // one-tile kernels: when set and the word it points to is zero, the kernel loads, multiplies and stores nothing
  // (a step that an earlier kernel of the same stream found unnecessary)
  const uint32_t* gate;
  // one-tile kernels: block (0, 0, 0) stores zero into *dev_status right after griddepcontrol.wait (for the first
  // kernel of a call: no memset node in front of the chain).  A bounded wait of this kernel can set a bit two seconds
  // later at the earliest, long after that store.
  int clear_status;
  // one-tile kernels, OUT_SPLIT: when set and the word is zero, the low part (C1) is not written
  const uint32_t* lo_gate;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {   // does not wait
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// One lane of a converged warp, the same one every time.  The loops that issue TMA copies and MMAs are entered through this
// and not through a comparison of the lane number: the compiler then knows that a single lane is active, and hands the
// instructions their uniform operands directly.  Measured (148 CTAs, one thread issuing): four tcgen05.mma and a commit 341 ->
// 167 cycles at N = 16 and 256 at N = 128 (the tensor time), with a wait for a barrier in front 494 -> 321.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait.  Returns false if the limit expired (or another role already gave up).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                                  uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  // the wall clock is read only once in a while, and first after 1024 failed polls: a read of %globaltimer is
  // slow enough to matter on the hand-offs of the operand ring, which all pass through here
  uint64_t t0 = 0;
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 1023u) == 0u) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) { *abort_flag = 1; return false; }
    }
  }
}
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
// Panels of 64 columns side by side, 64 rows each (3-D map: column, row, panel).
__device__ __forceinline__ void tma_load_panels(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int row, int panel) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(0), "r"(row), "r"(panel)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same instruction with the accumulator read as D / 2 (scale-input-d = 1): D = A B + D * 2^-1.
__device__ __forceinline__ void tc_mma_bf16_halved(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, 1, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p, 1;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc)
      : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t v[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_ld64(uint32_t taddr, uint32_t v[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]), "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39]), "=r"(v[40]), "=r"(v[41]), "=r"(v[42]), "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]), "=r"(v[48]), "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]), "=r"(v[54]), "=r"(v[55]), "=r"(v[56]), "=r"(v[57]), "=r"(v[58]), "=r"(v[59]), "=r"(v[60]), "=r"(v[61]), "=r"(v[62]), "=r"(v[63])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle.  K-major: rows of 128 bytes, groups of 8 rows
// 1024 bytes apart (stride byte offset); the leading byte offset is not used.  MN-major: rows are K
// indices, each 128 bytes = 64 elements along M/N; groups of 8 K rows 1024 bytes apart (stride byte
// offset) and consecutive 64-element groups along M/N one TMA box (64 rows = 8192 bytes) apart
// (leading byte offset).
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr, bool mn_major) {
  const uint64_t lbo = mn_major ? (8192u >> 4) : 1u;
  const uint64_t sbo = 1024u >> 4;
  return (uint64_t)((smem_addr >> 4) & 0x3FFFu) | (lbo << 16) | (sbo << 32) | (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&t);
}

// f'(a) of the element-wise consumers (OUT_ACT_BWD), times the upstream gradient, rounded to bf16 afterwards.  The fused
// epilogue is bound by the instructions it issues, so both are written out: two special-function instructions each.
//   SiLU: s (1 + a (1 - s)), s = 1 / (1 + exp(-a)); an exponential that overflows gives s = 0.
//   GELU (exact form): Phi(a) + a phi(a).  With E = exp(-a^2 / 2), phi(a) = E / sqrt(2 pi) and the upper tail
//   Q(|a|) = E P(t), t = 1 / (1 + 0.38 |a|), the form of Abramowitz and Stegun 7.1.26; the coefficients of P (degree 6) are
//   a least-maximum fit of exp(z^2 / 2) Q(z) (absolute error of Q 7e-9, 1.5e-7 when evaluated in fp32; a result is rounded
//   to 2^-9 of its value).  Phi(a) = Q(-a) for a < 0 and 1 - Q(a) otherwise, so the negative tail has no cancellation.
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
template <int kKind>
__device__ __forceinline__ float act_derivative(float a) {
  constexpr float kLog2e = 1.4426950408889634f;
  if (kKind == 0) {
    const float s = rcp_approx(1.f + exp2_approx(-kLog2e * a));
    return fmaf(s, fmaf(-s, a, a), s);
  }
  const float e = exp2_approx(-0.5f * kLog2e * a * a);
  const float t = rcp_approx(fmaf(0.38f, fabsf(a), 1.f));
  float q = 0.05599787458777428f;
  q = fmaf(q, t, -0.28459465503692627f);
  q = fmaf(q, t, 0.45932143926620483f);
  q = fmaf(q, t, -0.09984032809734344f);
  q = fmaf(q, t, 0.2310720831155777f);
  q = fmaf(q, t, 0.13692614436149597f);
  q = fmaf(q, t, 0.0011174236424267292f) * e;
  return fmaf(0.39894228040f * a, e, a < 0.f ? q : 1.f - q);
}

// ---- staged epilogue.  A thread owns one accumulator row, so a direct store instruction of a warp touches 32
// different rows, 16 bytes each: every 128-byte line of the output is written in eight pieces by eight
// instructions.  Instead each epilogue warp puts its 32 rows x 128 bytes into shared memory in the layout of a
// 128-byte-swizzled TMA box (conflict free: the 16-byte chunk c of row i goes to chunk c ^ (i & 7)) and one
// lane sends the box with a TMA store, which writes whole lines and clips at the edges of the output.  Each
// warp cycles through one, two or four boxes of its own, so no barrier between warps is needed.  Two warps share each
// quarter of the accumulator rows (a warp may only read the tensor-memory lanes 32 * (warp % 4) .. + 31); they
// take alternate column groups.
constexpr int kStoreBufs = 2;
constexpr uint32_t kStoreBoxBytes = 4096;                    // 32 rows x 128 bytes

struct StoreStage {
  unsigned char* base;   // this warp's boxes (1024-byte aligned); nullptr: direct stores only
  uint32_t cnt;          // boxes sent so far
  uint32_t bufs;         // boxes this warp cycles through (1, 2 or 4)
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* smem_src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"((uint64_t)map), "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}
template <int kPending>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kPending) : "memory");
}
// Boxes cnt .. cnt + kNeed - 1 may be written once the stores that last used them have read shared memory.
template <int kNeed>
__device__ __forceinline__ void stage_acquire(const StoreStage& st, int lane) {
  if (st.cnt + kNeed > st.bufs) {
    if (elect_one()) {
      if (st.bufs == 4) bulk_wait_read<4 - kNeed>();
      else if (st.bufs > (uint32_t)kNeed) bulk_wait_read<2 - kNeed>();
      else bulk_wait_read<0>();
    }
    __syncwarp();
  }
}
__device__ __forceinline__ unsigned char* stage_box(const StoreStage& st, uint32_t k) {
  return st.base + ((st.cnt + k) & (st.bufs - 1u)) * kStoreBoxBytes;
}
__device__ __forceinline__ void stage_write16(unsigned char* box, int lane, int chunk, uint4 v) {
  *reinterpret_cast<uint4*>(box + lane * 128 + ((chunk ^ (lane & 7)) << 4)) = v;
}
// All lanes have written their rows of `box`: make them visible to the async proxy and send the box.
__device__ __forceinline__ void stage_send(const CUtensorMap* map, unsigned char* box, int lane, int x, int y) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (elect_one()) {
    tma_store_2d(map, box, x, y);
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}
// Before the shared memory goes away: every store of this warp has read it (the writes themselves are complete when the grid
// is, which is what the next kernel waits for).
__device__ __forceinline__ void stage_drain(const StoreStage& st, int lane) {
  if (st.base && elect_one()) bulk_wait_read<0>();
  __syncwarp();
}

__device__ __forceinline__ void tc_store_tile_staged(const TcParams& p, const TmapPack& maps, uint32_t tmem_base,
                                                     int quad, int half_id, int lane, int m0, int n0,
                                                     int split, StoreStage& st, bool lo_on = true) {
  const int row0 = m0 + quad * 32;
  const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16);
  const int y = split * p.M + row0;
  if (p.out == OUT_F32) {
    for (int c0 = 32 * half_id; c0 < p.bn && n0 + c0 < p.N; c0 += 64) {
      uint32_t v[32];
      tc_ld32(taddr + (uint32_t)c0, v);
      tc_wait_ld();
      stage_acquire<1>(st, lane);
      unsigned char* box = stage_box(st, 0);
#pragma unroll
      for (int q = 0; q < 8; ++q) stage_write16(box, lane, q, make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
      stage_send(&maps.c[0], box, lane, n0 + c0, y);
      st.cnt += 1;
    }
    return;
  }
  const bool split_out = p.out == OUT_SPLIT && lo_on;   // lo_on false: only the leading part is wanted
  for (int c0 = 64 * half_id; c0 < p.bn && n0 + c0 < p.N; c0 += 128) {
    if (split_out) stage_acquire<2>(st, lane); else stage_acquire<1>(st, lane);
    unsigned char* box_hi = stage_box(st, 0);
    unsigned char* box_lo = stage_box(st, 1);
    uint32_t v64[64];
    tc_ld64(taddr + (uint32_t)c0, v64);
    tc_wait_ld();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const uint32_t* v = v64 + 32 * half;
      if (!split_out) {
        // one conversion instruction per pair of columns: this loop runs on a single warp per scheduler, so
        // its length in instructions is its duration
#pragma unroll
        for (int q = 0; q < 4; ++q)
          stage_write16(box_hi, lane, 4 * half + q,
                        make_uint4(pack_bf16x2(__uint_as_float(v[8 * q]), __uint_as_float(v[8 * q + 1])),
                                   pack_bf16x2(__uint_as_float(v[8 * q + 2]), __uint_as_float(v[8 * q + 3])),
                                   pack_bf16x2(__uint_as_float(v[8 * q + 4]), __uint_as_float(v[8 * q + 5])),
                                   pack_bf16x2(__uint_as_float(v[8 * q + 6]), __uint_as_float(v[8 * q + 7]))));
      } else {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const float x0 = __uint_as_float(v[2 * q]), x1 = __uint_as_float(v[2 * q + 1]);
          hi[q] = pack_bf16x2(x0, x1);
          lo[q] = pack_bf16x2(x0 - __uint_as_float(hi[q] << 16), x1 - __uint_as_float(hi[q] & 0xffff0000u));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          stage_write16(box_hi, lane, 4 * half + q, make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]));
          stage_write16(box_lo, lane, 4 * half + q, make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]));
        }
      }
    }
    stage_send(&maps.c[0], box_hi, lane, n0 + c0, y);
    if (split_out) stage_send(&maps.c[1], box_lo, lane, n0 + c0, y);
    st.cnt += split_out ? 2 : 1;
  }
}

// Writes one finished accumulator tile (128 rows of this CTA x bn columns, starting at tensor-memory column
// tmem_base) in the output mode of p.  Warp w may touch the lanes 32 * (w % 4) .. + 31.
__device__ __forceinline__ void tc_store_tile(const TcParams& p, const TmapPack& maps, uint32_t tmem_base, int warp,
                                              int lane, int m0, int n0, int split, StoreStage& st, bool lo_on = true) {
  const int quad = warp & 3;
  const int half_id = (warp - 2) >> 2;                       // which of the two warps of this quarter
  const int row = quad * 32 + lane;
  const int m = m0 + row;
  if (m0 + quad * 32 >= p.M) return;                         // none of this warp's rows exists
  // staged unless the output needs read-modify-write, or (split-K partials stacked along the rows of one
  // tensor map) the warp's 32 rows are not all inside M
  if (st.base && p.tma_store && !p.accumulate && (p.split_stride == 0 || m0 + quad * 32 + 32 <= p.M)) {
    tc_store_tile_staged(p, maps, tmem_base, quad, half_id, lane, m0, n0, split, st, lo_on);
    return;
  }
  {
    for (int c0 = 32 * half_id; c0 < p.bn; c0 += 64) {
      uint32_t v[32];
      tc_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
      tc_wait_ld();
      const int n = n0 + c0;
      if (m >= p.M) continue;
      const int valid = min(32, min(p.bn - c0, p.N - n));
      if (valid <= 0) continue;
      if (p.out == OUT_F32) {
        float* dst = (float*)p.C0 + (int64_t)split * p.split_stride + (int64_t)m * p.ldc + n;
        if (p.accumulate) {
          for (int q = 0; q < valid; ++q) dst[q] += __uint_as_float(v[q]);
        } else if (valid == 32 && ((((uintptr_t)dst) & 15) == 0)) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            reinterpret_cast<uint4*>(dst)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        } else {
          for (int q = 0; q < valid; ++q) dst[q] = __uint_as_float(v[q]);
        }
      } else {
        __nv_bfloat16* dst_hi = (__nv_bfloat16*)p.C0 + (int64_t)m * p.ldc + n;
        __nv_bfloat16* dst_lo = (p.out == OUT_SPLIT && lo_on) ? (__nv_bfloat16*)p.C1 + (int64_t)m * p.ldc + n : nullptr;
        if (valid == 32 && ((((uintptr_t)dst_hi) & 15) == 0)) {
          uint32_t hi[16], lo[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float x0 = __uint_as_float(v[2 * q]), x1 = __uint_as_float(v[2 * q + 1]);
            const __nv_bfloat16 h0 = __float2bfloat16(x0), h1 = __float2bfloat16(x1);
            hi[q] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            lo[q] = pack_bf16x2(x0 - __bfloat162float(h0), x1 - __bfloat162float(h1));
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            reinterpret_cast<uint4*>(dst_hi)[q] = make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
          if (dst_lo) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              reinterpret_cast<uint4*>(dst_lo)[q] = make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
          }
        } else {
          for (int q = 0; q < valid; ++q) {
            const float x = __uint_as_float(v[q]);
            const __nv_bfloat16 h = __float2bfloat16(x);
            dst_hi[q] = h;
            if (dst_lo) dst_lo[q] = __float2bfloat16(x - __bfloat162float(h));
          }
        }
      }
    }
  }
}

// Epilogue of one CTA (eight warps) of the one-tile kernels: waits for the accumulator, then writes it.
// `ring` is the operand ring: once the accumulator is complete every load has landed and every MMA has read
// its stage, so the epilogue warps take the ring over as staging space (two or four boxes of 4 KB per warp).
// n_acc accumulators, 256 tensor-memory columns apart: accumulator w is the tile at (m0 + w dm, n0 + w dn).
__device__ __forceinline__ void tc_epilogue(const TcParams& p, const TmapPack& maps, uint32_t tmem_base,
                                          uint64_t* accum_bar, volatile int* abort_flag_ptr, int warp, int lane,
                                          int m0, int n0, int split, int n_iter, unsigned char* ring, int n_acc = 1,
                                          int dm = 0, int dn = 0) {
  // OUT_SPLIT with a gate on the low part: read the word while the contraction is still running
  const bool lo_on = !(p.lo_gate != nullptr && *(const volatile uint32_t*)p.lo_gate == 0u);
  bool ok = mbar_wait_bounded(accum_bar, 0, abort_flag_ptr);
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  if (ok && n_iter > 0) {
    StoreStage st;
    st.bufs = (uint32_t)p.store_bufs;
    st.base = ring + (uint32_t)(warp - 2) * st.bufs * kStoreBoxBytes;
    st.cnt = 0;
    for (int w = 0; w < n_acc; ++w)
      tc_store_tile(p, maps, tmem_base + 256u * (uint32_t)w, warp, lane, m0 + w * dm, n0 + w * dn, split, st, lo_on);
    stage_drain(st, lane);
  } else if (ok && n_iter == 0 && p.out == OUT_F32 && warp < 6) {
    // an empty K range still owns its partial: write zeros
    for (int w = 0; w < n_acc; ++w) {
      const int m = m0 + w * dm + (warp & 3) * 32 + lane, n = n0 + w * dn;
      if (m >= p.M) continue;
      float* dst = (float*)p.C0 + (int64_t)split * p.split_stride + (int64_t)m * p.ldc + n;
      for (int q = 0; q < min(p.bn, p.N - n); ++q) dst[q] = 0.f;
    }
  }
}

// kShareA: the terms have A in common; a stage brings it once, with the B tiles of all terms.  (A form of its own: a run-time
// number of B tiles per stage costs the others 1 to 2 us a step.)
template <bool A_MN, bool B_MN, bool kShareA>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_kernel(const __grid_constant__ TmapPack maps, const TcParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t accum_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = p.stages;
  // No more producers than stages: a producer that waits for a stage then knows that the use before the last one of it is over (its own
  // previous wait was for a later K block), and cannot take the parity of that use for the one it waits for.
  const int producers = stages < kProducers ? 2 : kProducers;
  const int producer = warp == 0 ? 0 : (warp >= 2 && warp <= producers ? warp - 1 : -1);
  const int n0 = blockIdx.x * p.bn, m0 = blockIdx.y * kBM, split = blockIdx.z;
  const int kb_begin = split * p.kb_per_split;
  const int kb_count = max(0, min(p.kb_total, kb_begin + p.kb_per_split) - kb_begin);
  const int b_tiles = kShareA ? p.n_terms : 1;
  int n_iter = kb_count * (kShareA ? 1 : p.n_terms);
  const uint32_t stage_bytes = kABytes + (uint32_t)b_tiles * p.b_bytes;
  // up to 64 rows the second half of the A tile is not loaded: its accumulator rows are never read.  (Whole steps, half / whole
  // tiles: 4096 x 5120, r = 64 80.9 / 81.3 us, 8192 x 4096, r = 48 87.6 / 88.4, 16384 x 2048, r = 16 79.5 / 80.4.)
  const uint32_t tx_bytes = stage_bytes - (uint32_t)(kBM - p.a_rows) * (kBK * 2);
  // dynamic shared memory is declared 1024-aligned; round up anyway (swizzle atoms need it)
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem + 1023) & ~(uintptr_t)1023);

  // A gated launch that is not needed leaves before any set-up, and releases its successor first of all (the rule at GemmDesc::gate
  // says why the word may be read this early and why the wait is still executed).  Steps, released behind the wait / ahead of it:
  // 999 x 4096, r = 256 117.5 / 114.0 us, 4096 x 5120, r = 64 71.1 / 70.7, 16384 x 4096, r = 256 178.0 / 177.5, 2048 x 1024, r = 288 133.3 /
  // 132.7; 8192 x 5120, r = 128 with a power iteration 193.9 / 194.1.
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) { pdl_launch_dependents(); pdl_wait(); return; }

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(&accum_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  auto load_a = [&](int s, int term, int k0) {
    unsigned char* dst = tiles + (size_t)s * stage_bytes;
    if (A_MN && (p.panels & 1)) {
      tma_load_panels(dst, &maps.a[term], &full_bar[s], k0, m0 >> 6);
    } else if (A_MN) {
      tma_load_2d(dst, &maps.a[term], &full_bar[s], m0, k0);
      if (p.a_rows > 64) tma_load_2d(dst + 8192, &maps.a[term], &full_bar[s], m0 + 64, k0);
    } else {
      tma_load_2d(dst, &maps.a[term], &full_bar[s], k0, m0);
    }
  };
  auto load_b = [&](int s, int term0, int k0) {
    unsigned char* dst = tiles + (size_t)s * stage_bytes + kABytes;
    for (int t = 0; t < b_tiles; ++t, dst += p.b_bytes) {
      const CUtensorMap* map = &maps.b[term0 + t];
      if (B_MN && (p.panels & 2)) {
        tma_load_panels(dst, map, &full_bar[s], k0, n0 >> 6);
      } else if (B_MN) {
        for (uint32_t q = 0; q * 8192u < p.b_bytes; ++q) tma_load_2d(dst + q * 8192u, map, &full_bar[s], n0 + (int)q * 64, k0);
      } else {
        tma_load_2d(dst, map, &full_bar[s], k0, n0);
      }
    }
  };
  // K block and term of the next iteration of a producer: warps 0 and 2 to 4 (which become epilogue warps) take turns (0 and 2
  // where the ring has three stages).  One producer alone, with up to six loads and a barrier to wait for per K block, takes 440 to
  // 900 cycles for it.  Steps, two producers / four: 12608 x 768, r = 96 88.5 / 87.2 us, 8192 x 5120, r = 128 with a power iteration
  // 194.8 / 194.1, 2048 x 1024, r = 288 133.3 / 132.7, 16384 x 4096, r = 256 178.0 / 177.5; 5003 x 1000, r = 336 166.7 / 167.3.
  auto next_block = [&](int& term, int& kb) {
    kb += producers;
    while (kb >= kb_count) { kb -= kb_count; ++term; }
  };
  // The ring is filled with what does not depend on the previous kernel (see GemmDesc::a_early).
  const int n_pre = p.early ? min(stages, n_iter) : 0;
  if (n_pre > 0 && producer >= 0) {
    if (elect_one()) {
      int term = 0, kb = producer - producers;
      next_block(term, kb);
      for (int it = producer; it < n_pre; it += producers) {
        mbar_arrive_expect_tx(&full_bar[it], tx_bytes);
        if (p.early & 1) load_a(it, term, (kb_begin + kb) * kBK);
        if (p.early & 2) load_b(it, term, (kb_begin + kb) * kBK);
        next_block(term, kb);
      }
    }
    __syncwarp();
  }
  // everything above overlaps the tail of the previous kernel; its results only from here on
  pdl_wait();
  pdl_launch_dependents();
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) n_iter = -1;   // every role idles, nothing is stored
  if (p.clear_status && p.dev_status && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
    *(volatile uint32_t*)p.dev_status = 0u;

  if (producer >= 0 && n_iter > 0) {
    if (elect_one()) {
      // stage, parity, term and K block are carried along (no division in the loop)
      int s = producer, term = 0, kb = producer - producers;
      next_block(term, kb);
      uint32_t parity = 1u;
      for (int it = producer; it < n_iter; it += producers) {
        const int k0 = (kb_begin + kb) * kBK;
        const bool pre = it < n_pre;
        if (!pre) {
          if (!mbar_wait_bounded(&empty_bar[s], parity, &abort_flag)) break;
          mbar_arrive_expect_tx(&full_bar[s], tx_bytes);
        }
        if (!(pre && (p.early & 1))) load_a(s, term, k0);
        if (!(pre && (p.early & 2))) load_b(s, term, k0);
        s += producers; if (s >= stages) { s -= stages; parity ^= 1u; }
        next_block(term, kb);
      }
    }
    __syncwarp();
  }
  if (warp == 0) {
  } else if (warp == 1) {
    if (elect_one()) {
      // instruction descriptor: fp32 accumulator, bf16 A and B, operand majors, N >> 3, M >> 4
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_MN ? 1u : 0u) << 15) |
                             ((B_MN ? 1u : 0u) << 16) | ((uint32_t)(p.bn >> 3) << 17) |
                             ((uint32_t)(kBM >> 4) << 24);
      bool ok = true, ready = false;
      int s = 0;
      uint32_t parity = 0u;
      // descriptors address shared memory in 16-byte units: one addition per stage instead of building them anew
      const uint64_t a_desc0 = make_smem_desc(smem_u32(tiles), A_MN);
      const uint64_t b_desc0 = make_smem_desc(smem_u32(tiles) + kABytes, B_MN);
      const uint32_t stage_units = stage_bytes >> 4;
      const int halve_it = p.halve_at_term > 0 ? p.halve_at_term * kb_count : -1;
      for (int it = 0; it < n_iter && ok; ++it) {
        if (!ready) ok = mbar_wait_bounded(&full_bar[s], parity, &abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t a_desc = a_desc0 + (uint64_t)((uint32_t)s * stage_units);
        const uint64_t b_desc = b_desc0 + (uint64_t)((uint32_t)s * stage_units);
        uint64_t* done = &empty_bar[s];
        // the next stage is asked for before these MMAs are issued: the answer is here when they are
        if (++s == stages) { s = 0; parity ^= 1u; }
        ready = mbar_test(&full_bar[s], parity);
        for (int t = b_tiles - 1; t >= 0; --t) {             // (the last term is the smallest)
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) {
            // 16 elements along K: 32 bytes inside the swizzled row (K-major) or 16 rows (MN-major)
            const uint64_t a_k = a_desc + (uint64_t)((A_MN ? 2048u : 32u) >> 4) * k;
            const uint64_t b_k = b_desc + (uint64_t)((uint32_t)t * (p.b_bytes >> 4)) + (uint64_t)((B_MN ? 2048u : 32u) >> 4) * k;
            if (!kShareA && k == 0 && it == halve_it) tc_mma_bf16_halved(tmem_base, a_k, b_k, idesc);
            else tc_mma_bf16(tmem_base, a_k, b_k, idesc, (it > 0 || t < b_tiles - 1 || k > 0) ? 1u : 0u);
          }
        }
        tc_commit(done);           // frees the stage once these MMAs have read it
      }
      tc_commit(&accum_bar);       // accumulator complete (or nothing was issued)
    }
  } else {
    tc_epilogue(p, maps, tmem_base, &accum_bar, &abort_flag, warp, lane, m0, n0, split, n_iter, tiles);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols)
                 : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && p.dev_status) atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED);
}

// ------------------------------------------------------------------ two CTAs on one tile
// The same contraction with a pair of CTAs (a cluster of two along M) on one 256 x bn tile
// (tcgen05 cta_group::2): each CTA loads its 128 rows of A and HALF of the B tile, the tensor cores of both
// SMs read both halves, and each CTA ends up with its 128 rows of the accumulator in its own tensor
// memory.  Per SM and K block this moves 16 KB + half a B tile instead of 16 KB + a whole one, which is
// what limits the one-CTA kernel when B is re-read from L2 by every CTA; the ring gets six stages or more.
//   * Both CTAs allocate tensor memory (cta_group::2) and run a TMA producer; the loads of both complete
//     on the full barrier of the even CTA (the leader), which alone issues the MMAs.
//   * tcgen05.commit (cta_group::2, multicast to both CTAs) frees a stage in both CTAs and, at the end,
//     tells both epilogues that the accumulator is complete.
//   * No load uses cluster multicast.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}
// TMA load whose bytes are counted on a barrier that may live in the peer CTA.
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* map, uint32_t bar_cluster_addr,
                                                 int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"((uint64_t)map), "r"(bar_cluster_addr), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_load_panels_pair(void* smem_dst, const CUtensorMap* map, uint32_t bar_cluster_addr,
                                                     int row, int panel) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"((uint64_t)map), "r"(bar_cluster_addr), "r"(0), "r"(row), "r"(panel)
      : "memory");
}
// The same load with an L2 eviction-priority hint (a policy made by createpolicy).
__device__ __forceinline__ void tma_load_2d_pair_hint(void* smem_dst, const CUtensorMap* map, uint32_t bar_cluster_addr,
                                                      int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(smem_u32(smem_dst)), "l"((uint64_t)map), "r"(bar_cluster_addr), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(smem_u32(bar)), "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair_halved(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                                        uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, 1, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p, 1;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc)
      : "memory");
}

//
// kWide: two accumulators (512 tensor-memory columns) per pair.  WIDE_N: two column tiles side by side that share the rows
// of A; WIDE_M: two row tiles that share the columns of B.  A K block then brings 48 KB per CTA for 1024 cycles of tensor
// work instead of 32 KB for 512 (an SM reads 64 bytes per clock from L2, so the narrow form runs at that limit), the shared
// operand is read once, and a product with 512 rows or columns on one side needs half as many tiles: 16384 x 512 are 64
// of them, one round of the 74 SM pairs instead of two.  The ring has four stages.
// Measured, r = 512: sketch of 16384 x 11008 151 -> 135 us (1.37 PFLOP/s; cuBLAS holds 1.42 for seconds, 1.67 in a burst),
// projection 161 -> 141 us, sketch of 32768 x 5120 154 -> 137 us, application of L^-T to 32768 rows 66 -> 55 us.
enum Wide : int { WIDE_NONE = 0, WIDE_N = 1, WIDE_M = 2 };

template <bool A_MN, bool B_MN, int kWide>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_pair_kernel(const __grid_constant__ TmapPack maps, const TcParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];     // used in the leader: both CTAs' loads of a stage
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];    // in each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t accum_bar;                // in each CTA: the accumulator is complete
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  uint32_t cta_rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta_rank));
  const bool leader = cta_rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half_n = p.bn / 2;                               // B rows (or columns) this CTA loads
  // grid: x = 128-row tiles (the two CTAs of a pair are neighbours in x), y = column tiles, z = K splits.  CTAs start
  // in the order x, then y; the tile a pair works on is taken from that order with the column tile running fastest,
  // so that the pairs that share a row tile of A (pass 1 at r = 512: the same 256 rows of X, two column tiles) run
  // side by side and the second one finds those rows in L2 instead of streaming X from HBM a second time.
  const int pair_lin = (int)(blockIdx.x >> 1) + (int)(gridDim.x >> 1) * (int)blockIdx.y;
  const int tile_m = pair_lin / (int)gridDim.y, tile_n = pair_lin - tile_m * (int)gridDim.y;
  constexpr int kNA = kWide == WIDE_M ? 2 : 1, kNB = kWide == WIDE_N ? 2 : 1;   // tiles of A and of B per stage
  const int n0 = tile_n * p.bn * kNB, m0 = (2 * kNA * tile_m + (int)cta_rank) * kBM, split = blockIdx.z;
  const int kb_begin = split * p.kb_per_split;
  const int kb_count = max(0, min(p.kb_total, kb_begin + p.kb_per_split) - kb_begin);
  int n_iter = kb_count * p.n_terms;
  const uint32_t stage_bytes = kNA * kABytes + kNB * p.b_bytes;   // per CTA (b_bytes: half a B tile)
  const int stages = p.stages;                               // (four or more)
  const int producers = kWide == WIDE_NONE && p.bn <= 128 ? kProducers : 2;
  const int producer = warp == 0 ? 0 : (warp >= 2 && warp <= producers ? warp - 1 : -1);
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem + 1023) & ~(uintptr_t)1023);

  // a gated launch that is not needed: both CTAs of the pair read the same word and leave before any set-up (see the one-CTA kernel)
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) { pdl_launch_dependents(); pdl_wait(); return; }

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(&accum_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers exist before either CTA signals the other
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  // loads of K block kb of a term into stage s; both CTAs' bytes are counted on the leader's barrier
  const int nb0 = n0 + (int)cta_rank * half_n;               // this CTA's half of the B tile
  const uint64_t keep_policy = l2_policy_evict_last();
  // A lower triangular operand with two tiles: from this K block on the first tile is zero, and neither loaded nor multiplied.
  const int zero_kb = kWide != WIDE_NONE && p.lower
                          ? (kWide == WIDE_M ? (4 * tile_m + 2) * kBM : (2 * tile_n + 1) * p.bn) / kBK - kb_begin : 1 << 30;
  auto tx_bytes = [&](int kb) {
    return kb >= zero_kb ? stage_bytes - (kWide == WIDE_M ? kABytes : p.b_bytes) : stage_bytes;
  };
  auto load_a = [&](int s, int term, int kb) {
    unsigned char* a_dst = tiles + (size_t)s * stage_bytes;
    const uint32_t bar = map_to_rank(smem_u32(&full_bar[s]), 0u);
    const int k0 = (kb_begin + kb) * kBK;
#pragma unroll
    for (int i = 0; i < kNA; ++i) {
      if (kWide == WIDE_M && i == 0 && kb >= zero_kb) continue;
      unsigned char* dst = a_dst + i * kABytes;
      const int m = m0 + i * 2 * kBM;
      if (A_MN && (p.panels & 1)) {
        tma_load_panels_pair(dst, &maps.a[term], bar, k0, m >> 6);
      } else if (A_MN) {
        tma_load_2d_pair(dst, &maps.a[term], bar, m, k0);
        tma_load_2d_pair(dst + 8192, &maps.a[term], bar, m + 64, k0);
      } else if (kb_begin + kb >= p.a_keep_from_kb) {
        tma_load_2d_pair_hint(dst, &maps.a[term], bar, k0, m, keep_policy);
      } else {
        tma_load_2d_pair(dst, &maps.a[term], bar, k0, m);
      }
    }
  };
  auto load_b = [&](int s, int term, int kb) {
    unsigned char* b_dst = tiles + (size_t)s * stage_bytes + kNA * kABytes;
    const uint32_t bar = map_to_rank(smem_u32(&full_bar[s]), 0u);
    const int k0 = (kb_begin + kb) * kBK;
#pragma unroll
    for (int i = 0; i < kNB; ++i) {
      if (kWide == WIDE_N && i == 0 && kb >= zero_kb) continue;
      unsigned char* dst = b_dst + i * p.b_bytes;
      const int n = nb0 + i * p.bn;
      if (B_MN && (p.panels & 2)) {
        tma_load_panels_pair(dst, &maps.b[term], bar, k0, n >> 6);
      } else if (B_MN) {
        for (uint32_t q = 0; q * 8192u < p.b_bytes; ++q)
          tma_load_2d_pair(dst + q * 8192u, &maps.b[term], bar, n + (int)q * 64, k0);
      } else {
        tma_load_2d_pair(dst, &maps.b[term], bar, k0, n);
      }
    }
  };
  // K block and term of the next iteration of a producer.  Two producers take turns (warps 0 and 2), or four (0, 2, 3 and 4) where
  // the tile of B is narrow and a K block short: up to 128 columns.  Steps, two / four: 4096 x 5120, r = 64 71.7 / 70.7 us, 8192 x 5120,
  // r = 128 with a power iteration 195.5 / 194.1, 4090 x 1000, r = 128 83.0 / 81.9, 12608 x 768, r = 96 87.9 / 87.2.  (On wider tiles, too,
  // 5003 x 1000, r = 336 took 0.7 more.)
  auto next_block = [&](int& term, int& kb) {
    kb += producers;
    while (kb >= kb_count) { kb -= kb_count; ++term; }
  };
  // The ring is filled with what does not depend on the previous kernel (see GemmDesc::a_early).
  const int n_pre = p.early ? min(stages, n_iter) : 0;
  if (n_pre > 0 && producer >= 0) {
    if (elect_one()) {
      int term = 0, kb = producer - producers;
      next_block(term, kb);
      for (int it = producer; it < n_pre; it += producers) {
        if (leader) mbar_arrive_expect_tx(&full_bar[it], 2u * tx_bytes(kb));
        if (p.early & 1) load_a(it, term, kb);
        if (p.early & 2) load_b(it, term, kb);
        next_block(term, kb);
      }
    }
    __syncwarp();
  }
  pdl_wait();
  pdl_launch_dependents();
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) n_iter = -1;   // every role idles, nothing is stored
  if (p.clear_status && p.dev_status && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)
    *(volatile uint32_t*)p.dev_status = 0u;

  if (producer >= 0 && n_iter > 0) {
    if (elect_one()) {
      // stage, parity, term and K block are carried along (no division in the loop)
      int s = producer;
      uint32_t parity = 1u;
      int term = 0, kb = producer - producers;
      next_block(term, kb);
      for (int it = producer; it < n_iter; it += producers) {
        const bool pre = it < n_pre;
        if (!pre) {
          if (!mbar_wait_bounded(&empty_bar[s], parity, &abort_flag)) break;
          // the leader expects the bytes of both CTAs on its barrier
          if (leader) mbar_arrive_expect_tx(&full_bar[s], 2u * tx_bytes(kb));
        }
        if (!(pre && (p.early & 1))) load_a(s, term, kb);
        if (!(pre && (p.early & 2))) load_b(s, term, kb);
        s += producers; if (s >= stages) { s -= stages; parity ^= 1u; }
        next_block(term, kb);
      }
    }
    __syncwarp();
  }
  if (warp == 0) {
  } else if (warp == 1) {
    if (leader && elect_one()) {
      // instruction descriptor: fp32 accumulator, bf16 A and B, operand majors, N >> 3, M = 256 >> 4
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_MN ? 1u : 0u) << 15) |
                             ((B_MN ? 1u : 0u) << 16) | ((uint32_t)(p.bn >> 3) << 17) |
                             ((uint32_t)((2 * kBM) >> 4) << 24);
      bool ok = true, ready = false;
      int s = 0;
      uint32_t parity = 0u;
      // descriptors address shared memory in 16-byte units: one addition per stage instead of building them anew
      const uint64_t a_desc0 = make_smem_desc(smem_u32(tiles), A_MN);
      const uint64_t b_desc0 = make_smem_desc(smem_u32(tiles) + kNA * kABytes, B_MN);
      const uint32_t stage_units = stage_bytes >> 4;
      const int halve_it = p.halve_at_term > 0 ? p.halve_at_term * kb_count : -1;
      int kb = 0;
      for (int it = 0; it < n_iter && ok; ++it) {
        if (!ready) ok = mbar_wait_bounded(&full_bar[s], parity, &abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t a_desc = a_desc0 + (uint64_t)((uint32_t)s * stage_units);
        const uint64_t b_desc = b_desc0 + (uint64_t)((uint32_t)s * stage_units);
        uint64_t* done = &empty_bar[s];
        // the next stage is asked for before these MMAs are issued: the answer is here when they are
        if (++s == stages) { s = 0; parity ^= 1u; }
        ready = mbar_test(&full_bar[s], parity);
        const bool zero = kWide != WIDE_NONE && kb >= zero_kb;
        if (++kb == kb_count) kb = 0;
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k) {
          const uint64_t a_k = a_desc + (uint64_t)((A_MN ? 2048u : 32u) >> 4) * k;
          const uint64_t b_k = b_desc + (uint64_t)((B_MN ? 2048u : 32u) >> 4) * k;
#pragma unroll
          for (int w = 0; w < kNA * kNB; ++w) {
            if (kWide != WIDE_NONE && w == 0 && zero) continue;
            const uint64_t a_w = a_k + (uint64_t)(kWide == WIDE_M ? w * (kABytes >> 4) : 0u);
            const uint64_t b_w = b_k + (uint64_t)(kWide == WIDE_N ? w * (p.b_bytes >> 4) : 0u);
            if (k == 0 && it == halve_it) tc_mma_bf16_pair_halved(tmem_base + 256u * w, a_w, b_w, idesc);
            else tc_mma_bf16_pair(tmem_base + 256u * w, a_w, b_w, idesc, (it > 0 || k > 0) ? 1u : 0u);
          }
        }
        tc_commit_pair(done);            // frees the stage in both CTAs once these MMAs have read it
      }
      tc_commit_pair(&accum_bar);        // accumulator complete in both CTAs (or nothing was issued)
    }
  } else {
    tc_epilogue(p, maps, tmem_base, &accum_bar, &abort_flag, warp, lane, m0, n0, split, n_iter, tiles,
                kNA * kNB, kWide == WIDE_M ? 2 * kBM : 0, kWide == WIDE_N ? p.bn : 0);
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA frees tensor memory or leaves while the other may still use its shared or tensor memory (relaxed: nothing
  // written is handed over)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols)
                 : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && p.dev_status) atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED);
}

// ------------------------------------------------------------------ many tiles per CTA pair, B resident
// C = A B for a short contraction (K <= 512) and a large output, the shape of Reconstruct (X~ = U V): the
// work per output tile is a handful of K blocks, so a kernel that lives for one tile spends its time on set-up,
// one load round trip and one store round trip, none of them overlapped.  Here a CTA pair is persistent:
//   * the tiles are numbered column tile first; pair p takes the contiguous range [p U / P, (p + 1) U / P), so
//     it stays on one column tile for many tiles (and changes it once or twice at most);
//   * its half of the B tile (all K blocks) stays in shared memory while the column tile does not change;
//     only A is streamed through a ring of 128 x 64 stages;
//   * the accumulator is double buffered in tensor memory (2 x bn columns): the tensor cores work on tile
//     i + 1 while the eight epilogue warps read and store tile i.
// Tiles are 256 columns wide whenever the output mode allows it: with 128 columns one instruction keeps the
// tensor pipe busy for 64 cycles, less than the issuing thread needs per instruction (about 100 cycles with
// the fence and the commit of a K block), and the kernel ran issue-bound at about 0.6 of the 256-wide rate.
// Beyond four K blocks the resident B (16 KB per K block and CTA) leaves room for a shorter A ring and one
// staging box per epilogue warp only; the epilogue has the slack (it is about half the tensor time there).
// Barriers.  a_full / a_empty: the ring, as in the pair kernel.  b_full (leader): both halves of B have
// landed; b_empty (each CTA, by commit): every MMA that reads the resident B is done, it may be replaced.
// acc_full[j] (each CTA, by commit): buffer j holds a finished tile; acc_empty[j] (leader, one arrival
// per CTA, sent by the first epilogue warp once all eight have arrived on the CTA's own epi_done[j]): buffer j has been read in both CTAs.  No load uses cluster multicast.
constexpr int kStreamStages = 6;
// Every column tile reads A again, while the output (and the matrix it is combined with) passes through L2 once: loads of A
// ask to stay.  16384 x 11008, K = 512 (A 17 MB): reconstruction 162 -> 152 us, SiLU backward 215 -> 205; 49152 x 3072 (A
// 50 MB) 174 -> 170 and 207 -> 203.  At 67 MB, more than half of L2, it makes no difference: not asked for there.
constexpr long long kStreamKeepBytes = 60ll << 20;
constexpr int kStreamSmemMax = 226 * 1024;                 // dynamic shared memory the streaming kernel may ask for

// An arrival on a barrier of the peer CTA.  Relaxed: it announces that tensor-memory reads have completed
// (tcgen05.wait::ld has returned), no memory written by this thread has to become visible with it, and a
// releasing arrival at cluster scope costs most of a microsecond.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive_local(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  uint64_t t0 = 0;
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((spin & 1023u) == 0u) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
}

// ---- fused epilogue: the finished tile is combined with another matrix E of the output's shape (read once) and only the
// result is written.  EP_RMS: row_a col E - row_b / col acc (OUT_RMS_BWD); EP_SILU, EP_GELU: E f'(acc) (OUT_ACT_BWD).
// A thread owns one accumulator row, so loading E from global memory here would touch 32 lines per instruction with
// nothing in flight behind it.  Instead E comes in boxes of 32 rows x 32 columns by TMA, requested store_bufs - 1
// boxes ahead by each epilogue warp for itself; the result overwrites E in the box and leaves by TMA from there.
// The epilogue is bound by the instructions it issues and their latency: up to sixteen warps, four per quarter of the
// accumulator's rows.  Measured, SiLU / GELU backward, calls back to back with three sets of inputs in turn, against direct
// loads: 16384 x 11008, K = 512: 689 / 672 -> 233 / 272 us; 16384 x 4096, K = 256: 258 / 250 -> 64 / 74 (floors 115 and 43).
// On the way there, with the same inputs again and again (L2 keeps part of E): 252 / 376 and 96 / 141 us with the boxes and
// eight warps, 227 / 251 and 67 / 80 with twelve and the derivatives written out, 207 / 234 and 60 / 73 with sixteen.  Of
// that 207, 187 are left without the derivatives, 152 without E as well: SiLU's two special-function instructions an element
// (16 lanes a cycle) and the shared-memory pipe, which the operands, E and the result share.  An L2 prefetch of E or plain
// stores of the result cost more than they save.
enum EpKind : int { EP_NONE = 0, EP_RMS = 1, EP_SILU = 2, EP_GELU = 3 };
constexpr int kFuseMaxBufs = 3;
constexpr int kFuseMaxWarps = 16;
constexpr uint32_t kFuseBoxBytes = 2048;                   // 32 rows x 64 bytes

// Boxes of 32 columns that one epilogue warp goes through: every fuse_parts-th box of its row group, running on from unit to
// unit (so that a number of warps that does not divide the boxes of a tile is balanced over several tiles).  Row and
// column are carried along: divisions, about three a box, were a tenth of the kernel (SiLU, 16384 x 4096, K = 256: 66 ->
// 60 us).
struct FuseCursor {
  int u, mt, c0;         // unit, its row tile, column inside the tile
  int row, n0;           // first row of the box, first column of the tile
  __device__ __forceinline__ void advance(const TcParams& p) {
    c0 += 32 * p.fuse_parts;
    while (c0 >= p.bn) {
      c0 -= p.bn;
      ++u;
      row += 2 * kBM;
      if (++mt == p.st_m_tiles) { mt = 0; row -= p.st_m_tiles * 2 * kBM; n0 += p.bn; }
    }
  }
};

template <int kEp>
__device__ __forceinline__ float fuse_value(float acc, float e, float ra, float rb, float col, float inv_col) {
  if (kEp == EP_RMS) return ra * col * e - rb * acc * inv_col;
  if (kEp == EP_SILU) return e * act_derivative<0>(acc);
  return e * act_derivative<1>(acc);
}

template <int kEp>
__device__ __forceinline__ void fused_epilogue(const TcParams& p, const TmapPack& maps, uint32_t tmem_base, int warp,
                                               int lane, int cta_rank, int u_begin, int u_end, unsigned char* boxes,
                                               uint64_t* e_full, float* col_inv, uint64_t* acc_full, uint64_t* acc_empty,
                                               uint64_t* epi_done, volatile int* abort_flag) {
  const int quad = warp & 3, part = (warp - 2) >> 2;
  const uint32_t bufs = (uint32_t)p.store_bufs;
  const int threads = 128 * p.fuse_parts;    // of all epilogue warps
  const __nv_bfloat16* gamma = (const __nv_bfloat16*)p.ep_col;
  // boxes outside the output are neither loaded nor stored
  auto live = [&](const FuseCursor& k) { return k.row < p.M && k.n0 + k.c0 < p.N; };
  const int nt_begin = u_begin / p.st_m_tiles, mt_begin = u_begin - nt_begin * p.st_m_tiles;
  FuseCursor ld{u_begin, mt_begin, 32 * part, (2 * mt_begin + cta_rank) * kBM + quad * 32, nt_begin * p.bn}, k = ld;
  uint32_t n_ld = 0, n_use = 0;              // live boxes requested / used so far
  uint32_t ld_slot = 0, use_slot = 0, use_phase = 0;
  auto request = [&]() {                      // the next live box, if any
    while (ld.u < u_end && !live(ld)) ld.advance(p);
    if (ld.u >= u_end) return;
    if (elect_one()) {
      mbar_arrive_expect_tx(&e_full[ld_slot], kFuseBoxBytes);
      tma_load_2d(boxes + ld_slot * kFuseBoxBytes, &maps.c[1], &e_full[ld_slot], ld.n0 + ld.c0, ld.row);
    }
    ++n_ld;
    if (++ld_slot == bufs) ld_slot = 0;
    ld.advance(p);
  };
  for (uint32_t b = 0; b + 1 < bufs; ++b) request();
  if (kEp == EP_RMS && p.early) {
    pdl_wait();
    pdl_launch_dependents();
  }
  bool ok = true;
  int mt = mt_begin, nt = nt_begin;
  for (int u = u_begin, ui = 0; u < u_end; ++u, ++ui, ++mt) {
    const int j = ui & 1;
    if (mt == p.st_m_tiles) { mt = 0; ++nt; }
    const int row0 = (2 * mt + cta_rank) * kBM + quad * 32, m = row0 + lane;
    if (kEp == EP_RMS && (ui == 0 || mt == 0)) {
      // 1 / gamma of this column tile, for all epilogue warps (which all come through here, even once a wait has expired)
      asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
      for (int c = (warp - 2) * 32 + lane; c < p.bn; c += threads) {
        const int n = nt * p.bn + c;
        col_inv[c] = n < p.N ? 1.f / __bfloat162float(gamma[n]) : 0.f;
      }
      asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
    }
    if (!ok) continue;
    float ra = 0.f, rb = 0.f;
    if (kEp == EP_RMS && m < p.M) { ra = p.ep_row_a[m]; rb = p.ep_row_b[m]; }
    ok = mbar_wait_bounded(&acc_full[j], (uint32_t)((ui >> 1) & 1), abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) continue;
    tc_fence_after();
    const uint32_t taddr = tmem_base + (uint32_t)(j * p.bn) + ((uint32_t)(quad * 32) << 16);
    for (; k.u == u && ok; k.advance(p)) {
      if (!live(k)) continue;
      uint32_t v[32];
      tc_ld32(taddr + (uint32_t)k.c0, v);
      unsigned char* box = boxes + use_slot * kFuseBoxBytes;
      ok = mbar_wait_bounded(&e_full[use_slot], use_phase, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      tc_wait_ld();
      if (!ok) break;
      const int n = k.n0 + k.c0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q == 2) {
          // the next request goes into the box that was sent before this one, which has had half a box's time to be read
          if (elect_one()) bulk_wait_read<0>();
          __syncwarp();
          request();
        }
        // 64-byte swizzle: chunk q of row i is at chunk q ^ ((i >> 1) & 3)
        uint4* at = reinterpret_cast<uint4*>(box + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4));
        const uint4 ev = *at;
        const uint32_t ew[4] = {ev.x, ev.y, ev.z, ev.w};
        uint4 gv = make_uint4(0u, 0u, 0u, 0u);             // N is a multiple of 8: a chunk is inside or outside
        if (kEp == EP_RMS && n + 8 * q < p.N) gv = __ldg(reinterpret_cast<const uint4*>(gamma + n) + q);
        const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
        uint32_t ow[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          float2 ci = make_float2(0.f, 0.f);
          if (kEp == EP_RMS) ci = *reinterpret_cast<const float2*>(col_inv + k.c0 + 8 * q + 2 * h);
          ow[h] = pack_bf16x2(fuse_value<kEp>(__uint_as_float(v[8 * q + 2 * h]), __uint_as_float(ew[h] << 16), ra, rb,
                                              __uint_as_float(gw[h] << 16), ci.x),
                              fuse_value<kEp>(__uint_as_float(v[8 * q + 2 * h + 1]), __uint_as_float(ew[h] & 0xffff0000u),
                                              ra, rb, __uint_as_float(gw[h] & 0xffff0000u), ci.y));
        }
        *at = make_uint4(ow[0], ow[1], ow[2], ow[3]);
      }
      stage_send(&maps.c[0], box, lane, n, row0);
      ++n_use;
      if (++use_slot == bufs) { use_slot = 0; use_phase ^= 1u; }
    }
    if (!ok) continue;
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive_local(&epi_done[j]);
      if (warp == 2) {
        // one signal per CTA and tile: the first epilogue warp collects them and tells the leader
        if (mbar_wait_bounded(&epi_done[j], (uint32_t)((ui >> 1) & 1), abort_flag)) {
          if (cta_rank == 0) mbar_arrive_local(&acc_empty[j]);
          else mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[j]), 0u));
        }
      }
    }
    __syncwarp();
  }
  // every box that was requested has landed before the shared memory goes away, and every store is complete
  for (; n_use < n_ld; ++n_use) {
    (void)mbar_wait_bounded(&e_full[use_slot], use_phase, abort_flag);
    if (++use_slot == bufs) { use_slot = 0; use_phase ^= 1u; }
  }
  if (elect_one()) bulk_wait_read<0>();
  __syncwarp();
}

template <int kEp>
__global__ void __launch_bounds__(kEp ? 64 + 32 * kFuseMaxWarps : kThreads, 1)
gemm_tc_stream_kernel(const __grid_constant__ TmapPack maps, const TcParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t a_full[kStreamStages];
  __shared__ __align__(8) uint64_t a_empty[kStreamStages];
  __shared__ __align__(8) uint64_t b_full, b_empty;
  __shared__ __align__(8) uint64_t acc_full[2];
  __shared__ __align__(8) uint64_t acc_empty[2];
  __shared__ __align__(8) uint64_t epi_done[2];
  __shared__ __align__(8) uint64_t e_full[kEp ? kFuseMaxWarps : 1][kFuseMaxBufs];
  __shared__ __align__(16) float col_inv[kEp == EP_RMS ? 256 : 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  uint32_t cta_rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta_rank));
  const bool leader = cta_rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_pairs = (int)(gridDim.x >> 1), pair = (int)(blockIdx.x >> 1);
  const int u_begin = (int)((long long)pair * p.st_units / n_pairs);
  const int u_end = (int)((long long)(pair + 1) * p.st_units / n_pairs);
  const int half_n = p.bn / 2;
  const uint32_t b_kb_bytes = p.b_bytes;                     // this CTA's half of B, one K block
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem + 1023) & ~(uintptr_t)1023);
  unsigned char* b_res = tiles;
  unsigned char* ring = tiles + (size_t)p.kb_total * b_kb_bytes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStreamStages; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_empty[s], 1); }
    mbar_init(&b_full, 1);
    mbar_init(&b_empty, 1);
    for (int j = 0; j < 2; ++j) {
      mbar_init(&acc_full[j], 1);
      mbar_init(&acc_empty[j], 2);
      mbar_init(&epi_done[j], kEp ? 4 * p.fuse_parts : kEpiWarps);
    }
    if (kEp)
      for (int w = 0; w < kFuseMaxWarps; ++w)
        for (int b = 0; b < kFuseMaxBufs; ++b) mbar_init(&e_full[kEp ? w : 0][b], 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  // EP_RMS, with all matrices older than the previous kernel (p.early): only the epilogue needs its results (the row
  // coefficients), and waits for itself
  const bool early = kEp == EP_RMS && p.early != 0;
  if (!early) {
    pdl_wait();
    pdl_launch_dependents();
  }

  if (warp == 0) {
    if (elect_one()) {
      const uint32_t bar_b = map_to_rank(smem_u32(&b_full), 0u);
      const uint64_t a_policy = p.st_keep_a ? l2_policy_evict_last() : l2_policy_evict_normal();
      int nb = 0, cur_nt = -1;
      int s = 0;                 // ring stage and its phase, carried along (no division in the loop)
      uint32_t ph = 0u;
      bool ok = true;
      for (int u = u_begin; u < u_end && ok; ++u) {
        const int nt = u / p.st_m_tiles, mt = u - nt * p.st_m_tiles;
        if (nt != cur_nt) {
          // the MMAs that read the previous column tile's B are done in both CTAs before it is replaced
          if (nb > 0) ok = mbar_wait_bounded(&b_empty, (uint32_t)((nb - 1) & 1), &abort_flag);
          if (!ok) break;
          if (leader) mbar_arrive_expect_tx(&b_full, 2u * (uint32_t)p.kb_total * b_kb_bytes);
          const int nb0 = nt * p.bn + (int)cta_rank * half_n;
          for (int kb = 0; kb < p.kb_total; ++kb)
            for (uint32_t q = 0; q * 8192u < b_kb_bytes; ++q)
              tma_load_2d_pair(b_res + (size_t)kb * b_kb_bytes + q * 8192u, &maps.b[0], bar_b, nb0 + (int)q * 64,
                               kb * kBK);
          ++nb;
          cur_nt = nt;
        }
        const int m0 = mt * 2 * kBM + (int)cta_rank * kBM;
        for (int kb = 0; kb < p.kb_total; ++kb) {
          ok = mbar_wait_bounded(&a_empty[s], ph ^ 1u, &abort_flag);
          if (!ok) break;
          if (leader) mbar_arrive_expect_tx(&a_full[s], 2u * kABytes);
          tma_load_2d_pair_hint(ring + (size_t)s * kABytes, &maps.a[0], map_to_rank(smem_u32(&a_full[s]), 0u), kb * kBK, m0,
                                a_policy);
          if (++s == p.st_stages) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (leader && elect_one()) {
      // instruction descriptor: fp32 accumulator, bf16 A (K-major) and B (MN-major), N >> 3, M = 256 >> 4
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(p.bn >> 3) << 17) |
                             ((uint32_t)((2 * kBM) >> 4) << 24);
      // descriptors address shared memory in 16-byte units: a ring stage is kABytes, a K block of B b_kb_bytes
      const uint64_t a_desc0 = make_smem_desc(smem_u32(ring), false);
      const uint64_t b_desc0 = make_smem_desc(smem_u32(b_res), true);
      int nb = 0, cur_nt = -1;
      int s = 0;                 // ring stage and its phase, carried along (a division here costs 9 % of the kernel)
      uint32_t ph = 0u;
      bool ok = true, ready = false;
      for (int u = u_begin, ui = 0; u < u_end && ok; ++u, ++ui) {
        const int j = ui & 1;
        const int nt = u / p.st_m_tiles;
        // buffer j was read by both epilogues (the first use of each buffer passes at once)
        ok = mbar_wait_cluster_bounded(&acc_empty[j], (uint32_t)(((ui >> 1) & 1) ^ 1), &abort_flag);
        if (!ok) break;
        if (nt != cur_nt) {
          ok = mbar_wait_bounded(&b_full, (uint32_t)(nb & 1), &abort_flag);
          if (!ok) break;
          ++nb;
          cur_nt = nt;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(j * p.bn);
        for (int kb = 0; kb < p.kb_total; ++kb) {
          if (!ready) ok = mbar_wait_bounded(&a_full[s], ph, &abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a_desc = a_desc0 + (uint64_t)((uint32_t)s * (kABytes >> 4));
          uint64_t* done = &a_empty[s];
          if (++s == p.st_stages) { s = 0; ph ^= 1u; }
          ready = mbar_test(&a_full[s], ph);       // asked for before the MMAs are issued
          const uint64_t b_desc = b_desc0 + (uint64_t)((uint32_t)kb * (b_kb_bytes >> 4));
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            tc_mma_bf16_pair(d_tmem, a_desc + (uint64_t)(32u >> 4) * k, b_desc + (uint64_t)(2048u >> 4) * k, idesc,
                             (kb > 0 || k > 0) ? 1u : 0u);
          tc_commit_pair(done);
        }
        if (!ok) break;
        tc_commit_pair(&acc_full[j]);
        if (u + 1 == u_end || (u + 1) / p.st_m_tiles != nt) tc_commit_pair(&b_empty);
      }
    }
  } else if (kEp) {
    fused_epilogue<kEp>(p, maps, tmem_base, warp, lane, (int)cta_rank, u_begin, u_end,
                        ring + (size_t)p.st_stages * kABytes + (uint32_t)(warp - 2) * p.store_bufs * kFuseBoxBytes,
                        e_full[kEp ? warp - 2 : 0], col_inv, acc_full, acc_empty, epi_done, &abort_flag);
  } else {
    bool ok = true;
    StoreStage st;
    st.bufs = (uint32_t)p.store_bufs;
    st.base = ring + (size_t)p.st_stages * kABytes + (uint32_t)(warp - 2) * st.bufs * kStoreBoxBytes;
    st.cnt = 0;
    for (int u = u_begin, ui = 0; u < u_end; ++u, ++ui) {
      const int j = ui & 1;
      const int nt = u / p.st_m_tiles, mt = u - nt * p.st_m_tiles;
      ok = mbar_wait_bounded(&acc_full[j], (uint32_t)((ui >> 1) & 1), &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      tc_store_tile(p, maps, tmem_base + (uint32_t)(j * p.bn), warp, lane, mt * 2 * kBM + (int)cta_rank * kBM,
                    nt * p.bn, 0, st);
      // the tile is in registers / shared memory now: hand the buffer back before the stores have drained
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_local(&epi_done[j]);
        if (warp == 2) {
          // one signal per CTA and tile: the first epilogue warp collects the eight and tells the leader
          if (mbar_wait_bounded(&epi_done[j], (uint32_t)((ui >> 1) & 1), &abort_flag)) {
            if (leader) mbar_arrive_local(&acc_empty[j]);
            else mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[j]), 0u));
          }
        }
      }
      __syncwarp();
    }
    stage_drain(st, lane);
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA frees tensor memory or leaves while the other may still use its shared or tensor memory (relaxed: nothing
  // written is handed over)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols)
                 : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && p.dev_status) atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED);
}

// ------------------------------------------------------------------ the tall Gram product above 256 columns
// W = (Yh + Yl)^T (Yh + Yl) for a bf16 pair of n x l, 256 < l <= 512, as partial sums over the rows.  What the general kernel
// would spend on it: three terms that each load their operands anew, both off-diagonal tiles of a symmetric matrix, and
// chains of some thirty K blocks, whose truncated additions cost accuracy and with it a second round.  Here a CTA pair takes a range
// of K blocks of one 256 x 256 tile on or below the diagonal:
//   * both parts of a K block are loaded once (on the diagonal A is B as well: 32 instead of 96 KB per CTA);
//   * on the diagonal D = (Yl^T Yl + Yh^T Yh) / 2 + Yh^T Yl, whose sum with its transpose is W (three products); below it all
//     four products, and the tile above is the transpose: 10 products instead of 12.  The small products come first,
//     while the accumulator is small;
//   * every K block has an accumulator of its own (two in turn): the epilogue warps add it to running sums in fp32 registers, with
//     rounding.  A chain of the tensor cores is 64 rows long whatever n is.  The reading costs nothing: 128 columns a thread and K block
//     take the eight warps 500 cycles, the products 1536 or 2048.
// The tiles below the diagonal get more ranges than the others, as their K blocks take longer.  Partial sums are whole tiles,
// 256 x 256 in fp32, unit after unit.  Measured with the sum over them (traced, an event behind either kernel): 32768 x 512 59 ->
// 47 us, 16384 x 512 45 -> 35 us.
constexpr int kGramStages = 3;
constexpr int kGramTile = 2 * kBM;
struct GramParams {
  int kb_total;          // 64-row K blocks
  int tiles;             // 256-column tiles of a row of W (2)
  int s_diag, s_off;     // ranges of K blocks per tile on, below the diagonal
  int panels;            // the maps have three dimensions (see TcParams)
  const uint32_t* gate;
  uint32_t* dev_status;
};
struct alignas(64) GramMaps {
  CUtensorMap hi, lo, out;
};

__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_gram_kernel(const __grid_constant__ GramMaps maps, const GramParams p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full_bar[kGramStages];    // in the leader: both CTAs' loads of a stage
  __shared__ __align__(8) uint64_t empty_bar[kGramStages];   // in each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t acc_full[2];              // in each CTA: the products of a K block are complete
  __shared__ __align__(8) uint64_t acc_empty[2];             // in the leader: all epilogue warps of both CTAs have read them
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  uint32_t cta_rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta_rank));
  const bool leader = cta_rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = (int)(blockIdx.x >> 1);
  // unit -> tile (row tm, column tn <= tm; diagonal tiles first) and range of K blocks
  int tm, tn, part, parts;
  if (unit < p.tiles * p.s_diag) {
    parts = p.s_diag; tm = tn = unit / parts; part = unit - tm * parts;
  } else {
    parts = p.s_off; part = unit - p.tiles * p.s_diag; tm = 1; tn = 0;
    while (part >= parts) { part -= parts; if (++tn == tm) { ++tm; tn = 0; } }
  }
  const bool diag = tm == tn;
  const int kb_begin = (int)((long long)part * p.kb_total / parts);
  const int n_kb = (int)((long long)(part + 1) * p.kb_total / parts) - kb_begin;
  const uint32_t stage_bytes = 4 * kABytes, tx_bytes = diag ? 2 * kABytes : 4 * kABytes;
  unsigned char* tiles = (unsigned char*)(((uintptr_t)smem + 1023) & ~(uintptr_t)1023);

  // (see the one-CTA kernel)
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) { pdl_launch_dependents(); pdl_wait(); return; }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGramStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int j = 0; j < 2; ++j) { mbar_init(&acc_full[j], 1); mbar_init(&acc_empty[j], 2 * kEpiWarps); }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  pdl_wait();
  pdl_launch_dependents();

  // stage: A high, A low, B high, B low (16 KB each: 128 columns of this CTA, 64 rows)
  const int a_col = tm * kGramTile + (int)cta_rank * kBM, b_col = tn * kGramTile + (int)cta_rank * kBM;
  if (warp == 0) {
    if (elect_one()) {
      int s = 0;
      uint32_t parity = 1u;
      for (int i = 0; i < n_kb; ++i) {
        if (!mbar_wait_bounded(&empty_bar[s], parity, &abort_flag)) break;
        if (leader) mbar_arrive_expect_tx(&full_bar[s], 2u * tx_bytes);
        const uint32_t bar = map_to_rank(smem_u32(&full_bar[s]), 0u);
        unsigned char* dst = tiles + (size_t)s * stage_bytes;
        const int row = (kb_begin + i) * kBK;
        for (int o = 0; o < (diag ? 2 : 4); ++o, dst += kABytes) {
          const CUtensorMap* map = (o & 1) ? &maps.lo : &maps.hi;
          const int col = o < 2 ? a_col : b_col;
          if (p.panels) {
            tma_load_panels_pair(dst, map, bar, row, col >> 6);
          } else {
            tma_load_2d_pair(dst, map, bar, col, row);
            tma_load_2d_pair(dst + 8192, map, bar, col + 64, row);
          }
        }
        if (++s == kGramStages) { s = 0; parity ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (leader && elect_one()) {
      // instruction descriptor: fp32 accumulator, bf16 A and B, both MN-major, N = 256, M = 256
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(kGramTile >> 3) << 17) |
                             ((uint32_t)(kGramTile >> 4) << 24);
      bool ok = true;
      int s = 0;
      uint32_t parity = 0u;
      const uint64_t desc0 = make_smem_desc(smem_u32(tiles), true);
      const uint32_t units = kABytes >> 4;                  // of one operand, in descriptor units
      for (int i = 0; i < n_kb && ok; ++i) {
        const int j = i & 1;
        ok = mbar_wait_cluster_bounded(&acc_empty[j], (uint32_t)(((i >> 1) & 1) ^ 1), &abort_flag) &&
             mbar_wait_bounded(&full_bar[s], parity, &abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ah = desc0 + (uint64_t)((uint32_t)s * (stage_bytes >> 4)), al = ah + units;
        const uint64_t bh = diag ? ah : ah + 2 * units, bl = diag ? al : ah + 3 * units;
        const uint32_t d = tmem_base + (uint32_t)(j * kGramTile);
        auto product = [&](uint64_t a, uint64_t b, bool first, bool halve) {
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) {
            const uint64_t step = (uint64_t)(2048u >> 4) * k;
            if (halve && k == 0) tc_mma_bf16_pair_halved(d, a + step, b + step, idesc);
            else tc_mma_bf16_pair(d, a + step, b + step, idesc, first && k == 0 ? 0u : 1u);
          }
        };
        product(al, bl, true, false);
        if (diag) {
          product(ah, bh, false, false);
          product(ah, bl, false, true);
        } else {
          product(ah, bl, false, false);
          product(al, bh, false, false);
          product(ah, bh, false, false);
        }
        tc_commit_pair(&empty_bar[s]);
        tc_commit_pair(&acc_full[j]);
        if (++s == kGramStages) { s = 0; parity ^= 1u; }
      }
    }
  } else {
    const int quad = warp & 3, half_id = (warp - 2) >> 2;
    const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half_id * kBM);
    float sum[kBM];                                         // this thread's row, 128 columns
#pragma unroll
    for (int q = 0; q < kBM; ++q) sum[q] = 0.f;
    bool ok = true;
    for (int i = 0; i < n_kb && ok; ++i) {
      const int j = i & 1;
      ok = mbar_wait_bounded(&acc_full[j], (uint32_t)((i >> 1) & 1), &abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < kBM / 32; ++c) {
        uint32_t v[32];
        tc_ld32(taddr + (uint32_t)(j * kGramTile + 32 * c), v);
        tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 32; ++q) sum[32 * c + q] += __uint_as_float(v[q]);
      }
      tc_fence_before();
      __syncwarp();
      if (elect_one()) mbar_arrive_cluster(map_to_rank(smem_u32(&acc_empty[j]), 0u));
    }
    if (ok) {
      // every load has landed and every MMA has read its stage: the ring becomes staging space, four boxes a warp
      const int y = unit * kGramTile + (int)cta_rank * kBM + quad * 32;
      unsigned char* box = tiles + (size_t)(warp - 2) * 4 * kStoreBoxBytes;
#pragma unroll
      for (int c = 0; c < kBM / 32; ++c, box += kStoreBoxBytes) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float* v = sum + 32 * c + 4 * q;
          stage_write16(box, lane, q, make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]),
                                                 __float_as_uint(v[3])));
        }
        stage_send(&maps.out, box, lane, half_id * kBM + 32 * c, y);
      }
      if (elect_one()) bulk_wait_read<0>();
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA frees tensor memory or leaves while the other may still use its shared or tensor memory
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && p.dev_status) atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED);
}

// W (l x l, row-major, both triangles) from the tiles of the kernel above.  A CTA takes 32 x 32 elements on or below the diagonal
// and their mirror image: of a diagonal tile D, D + D^T; below, the sum itself.  Four groups of 256 threads share the
// partial sums (on the diagonal two for either side), a thread four elements; fixed order.  Bound: 19 MB from L2.
__global__ void __launch_bounds__(1024) reduce_gram_kernel(const float* __restrict__ partials, int tiles, int s_diag, int s_off,
                                                           int l, float* __restrict__ W, int n_blocks, const uint32_t* gate) {
  __shared__ float t[4][32][33];
  const int tid = threadIdx.x, group = tid >> 8, a = (tid >> 3) & 31, c4 = (tid & 7) * 4;
  // (see the one-CTA kernel)
  if (gate != nullptr && *(const volatile uint32_t*)gate == 0u) { pdl_launch_dependents(); pdl_wait(); return; }
  pdl_wait();
  pdl_launch_dependents();
  for (int b = blockIdx.x; b < n_blocks; b += gridDim.x) {
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    const int J = b - I * (I + 1) / 2, tm = I >> 3, tn = J >> 3;
    const bool diag = tm == tn;
    const int parts = diag ? s_diag : s_off;
    const int first = diag ? tm * s_diag : tiles * s_diag + (tm * (tm - 1) / 2 + tn) * s_off;
    // groups 0 and 1 of a diagonal tile take the block itself, 2 and 3 its mirror image
    const bool mirror = diag && I != J && group >= 2;
    const int bi = (mirror ? J : I) & 7, bj = (mirror ? I : J) & 7;
    const int n_share = diag && I != J ? 2 : 4, share = group & (n_share - 1);
    const float* src = partials + (int64_t)first * (kGramTile * kGramTile) + (bi * 32 + a) * kGramTile + bj * 32 + c4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int q = share; q < parts; q += n_share) {
      const float4 x = *reinterpret_cast<const float4*>(src + (int64_t)q * (kGramTile * kGramTile));
      v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
    }
    t[group][a][c4] = v.x; t[group][a][c4 + 1] = v.y; t[group][a][c4 + 2] = v.z; t[group][a][c4 + 3] = v.w;
    __syncthreads();
    const int x = tid & 31, y = tid >> 5;                   // element (y, x) of the block, and of its mirror image
    auto element = [&](int i, int k) {
      const float s01 = t[0][i][k] + t[1][i][k];
      if (!diag) return s01 + (t[2][i][k] + t[3][i][k]);
      if (I == J) return (s01 + (t[2][i][k] + t[3][i][k])) + ((t[0][k][i] + t[1][k][i]) + (t[2][k][i] + t[3][k][i]));
      return s01 + (t[2][k][i] + t[3][k][i]);
    };
    if (I * 32 + y < l && J * 32 + x < l) W[(int64_t)(I * 32 + y) * l + J * 32 + x] = element(y, x);
    if (I != J && J * 32 + y < l && I * 32 + x < l) W[(int64_t)(J * 32 + y) * l + I * 32 + x] = element(x, y);
    __syncthreads();
  }
}

// ------------------------------------------------------------------ the abort path, exercised on purpose
// One thread waits, with the engine's own bounded wait, on a barrier that nothing ever arrives on.  The wait
// must give up after `limit_ns`, and the kernel then does what every role of the engine does: it records
// LORACT_DEV_WAIT_EXPIRED and returns.  Nothing else runs, so the context stays usable.
__global__ void wait_expiry_probe_kernel(uint32_t* dev_status, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait_bounded(&bar, 0, &abort_flag, limit_ns);
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || abort_flag) && dev_status) atomicOr(dev_status, LORACT_DEV_WAIT_EXPIRED);
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)sym;
  });
  return fn;
}

// Tensor maps depend only on (pointer, extents, stride, box); they are cached so that a repeated call
// on the same buffers encodes nothing.
typedef std::tuple<const void*, uint64_t, uint64_t, uint64_t, uint32_t, uint32_t, int, uint32_t> TmapKey;
std::mutex g_tmap_mutex;
std::map<TmapKey, CUtensorMap> g_tmap_cache;

// 2-D tensor of bf16 (es = 2) or fp32 (es = 4): `inner` contiguous elements, `outer` rows `ld` elements apart;
// box inner x outer, swizzled over its inner extent (128 bytes, or 64).  panels > 0 (bf16, inner a multiple of 64): the same
// matrix as panels of 64 columns, a box `panels` of them side by side.
cudaError_t get_tmap(const void* ptr, uint64_t inner, uint64_t outer, uint64_t ld, uint32_t box_inner,
                     uint32_t box_outer, CUtensorMap* out, int es = 2, uint32_t panels = 0) {
  const TmapKey key(ptr, inner, outer, ld, box_inner, box_outer, es, panels);
  {
    std::lock_guard<std::mutex> lock(g_tmap_mutex);
    auto it = g_tmap_cache.find(key);
    if (it != g_tmap_cache.end()) { *out = it->second; return cudaSuccess; }
  }
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {panels ? 64 : inner, outer, inner / 64};
  cuuint64_t strides[2] = {ld * (uint64_t)es, 128};
  cuuint32_t box[3] = {box_inner, box_outer, panels};
  cuuint32_t elem[3] = {1, 1, 1};
  CUtensorMap m;
  const CUresult r = fn(&m, es == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, panels ? 3 : 2,
                        const_cast<void*>(ptr), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        box_inner * (uint32_t)es == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  {
    std::lock_guard<std::mutex> lock(g_tmap_mutex);
    if (g_tmap_cache.size() > 4096) g_tmap_cache.clear();
    g_tmap_cache[key] = m;
  }
  *out = m;
  return cudaSuccess;
}

int g_pair_mode = 1;   // 0: never use the two-CTA kernels (test hook); 1: by shape; 2: as 1, but no streaming or wide kernel

// Tile width.  Up to 256 columns one tile of whole 16s; above, the multiple of 64 with the least padding, the widest of these:
// a tile of whole 64s leaves through staged stores (whole lines), and is one that a CTA pair can share.  (By padding alone, 336
// columns were two tiles of 176: direct stores and one CTA a tile, 9 thousand cycles for an epilogue instead of 4.)  It is the
// better rule where it pads most, too (steps in us, this rule / least padding in 16s): 4096 x 1024, r = 272 143 / 154, r = 288
// 144 / 159, r = 304 153 / 162; 16384 x 4096, r = 288 238 / 242, r = 304 250.0 / 249.6; 8192 rows, r = 128: 520 columns 88 / 95,
// 776 88 / 91, 1160 95 / 105, 1920 102 / 116.  (Tiles of whole 32s: the same as this rule within 1 us, but 147 to 162 at r = 272
// to 304 and 4096 rows.)
int pick_bn(int N) {
  if (N <= 256) return (N + 15) / 16 * 16;
  int best = 256;
  for (int bn = 192; bn >= 128; bn -= 64)
    if ((N + bn - 1) / bn * bn < (N + best - 1) / best * best) best = bn;
  return best;
}

template <bool A_MN, bool B_MN, bool kShareA = false>
cudaError_t launch_variant(const TmapPack& maps, const TcParams& p, dim3 grid, size_t smem, cudaStream_t stream) {
  static std::atomic<bool> configured[64];   // zero-initialised; set once the attribute is in place on a device
  int dev = 0;
  LORACT_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
    LORACT_CUDA_TRY(cudaFuncSetAttribute(gemm_tc_kernel<A_MN, B_MN, kShareA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kRingBytes + 1024));
    if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  }
  LORACT_CUDA_TRY(launch_pdl(gemm_tc_kernel<A_MN, B_MN, kShareA>, grid, dim3(kThreads), smem, stream, maps, p));
  count_launch(__func__, stream);
  return cudaGetLastError();
}

template <bool A_MN, bool B_MN, int kWide = WIDE_NONE>
cudaError_t launch_pair_variant(const TmapPack& maps, const TcParams& p, dim3 grid, size_t smem, cudaStream_t stream) {
  if (p.a_rows != kBM) return cudaErrorInvalidValue;   // the kernel waits for whole tiles of A
  static std::atomic<bool> configured[64];   // zero-initialised; set once the attribute is in place on a device
  int dev = 0;
  LORACT_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
    LORACT_CUDA_TRY(cudaFuncSetAttribute(gemm_tc_pair_kernel<A_MN, B_MN, kWide>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kRingBytes + 1024));
    if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;   // the two CTAs of a pair are neighbours along M
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LORACT_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_tc_pair_kernel<A_MN, B_MN, kWide>, maps, p));
  count_launch(__func__, stream);
  return cudaGetLastError();
}

// Pairs the streaming kernel is launched with: as many as can be resident at once (one CTA per SM).
template <int kEp>
cudaError_t launch_stream(const TmapPack& maps, TcParams p, size_t smem, cudaStream_t stream) {
  if (p.a_rows != kBM) return cudaErrorInvalidValue;   // the kernel waits for whole tiles of A
  static std::atomic<bool> configured[64];   // zero-initialised; set once the attribute is in place on a device
  static std::atomic<int> max_pairs[64];
  int dev = 0;
  LORACT_CUDA_TRY(cudaGetDevice(&dev));
  const bool cached = dev >= 0 && dev < 64 && configured[dev].load(std::memory_order_acquire);
  int pairs = cached ? max_pairs[dev].load(std::memory_order_relaxed) : 0;
  if (!cached) {
    const int smem_max = kStreamSmemMax - (kEp == EP_RMS ? 1024 : 0);   // (1 KB of static tables)
    LORACT_CUDA_TRY(cudaFuncSetAttribute(gemm_tc_stream_kernel<kEp>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    cudaLaunchConfig_t q = {};
    q.gridDim = dim3(2); q.blockDim = dim3(kEp ? 64 + 32 * kFuseMaxWarps : kThreads); q.dynamicSmemBytes = smem_max;
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = 2; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
    q.attrs = qa; q.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_stream_kernel<kEp>, &q) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      cudaDeviceProp prop;
      LORACT_CUDA_TRY(cudaGetDeviceProperties(&prop, dev));
      n = prop.multiProcessorCount / 2;
    }
    pairs = n < 1 ? 1 : n;
    if (dev >= 0 && dev < 64) {
      max_pairs[dev].store(pairs, std::memory_order_relaxed);
      configured[dev].store(true, std::memory_order_release);
    }
  }
  if (pairs > p.st_units) pairs = p.st_units;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kEp ? 64 + 128 * p.fuse_parts : kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LORACT_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_tc_stream_kernel<kEp>, maps, p));
  count_launch(__func__, stream);
  return cudaGetLastError();
}


}  // namespace

void gemm_tc_set_pair_mode(int on) { g_pair_mode = on; }

cudaError_t gemm_tc_wait_probe_launch(uint32_t* dev_status, uint64_t limit_ns, cudaStream_t stream) {
  wait_expiry_probe_kernel<<<1, 32, 0, stream>>>(dev_status, limit_ns);
  count_launch(__func__, stream);
  return cudaGetLastError();
}

bool gemm_tc_supported(const GemmDesc& g) {
  if (g.a_type != ELEM_BF16 || g.b_type != ELEM_BF16) return false;
  if (!(g.out == OUT_F32 || g.out == OUT_BF16 || g.out == OUT_SPLIT || g.out == OUT_RMS_BWD || g.out == OUT_ACT_BWD))
    return false;
  if (g.out == OUT_ACT_BWD || g.out == OUT_RMS_BWD) {
    // the operand layout, and 16-byte alignment of everything TMA touches
    if (g.a_mn || !g.b_mn || g.n_terms != 1 || g.splits > 1 || g.K > 8 * kBK || g.gate || g.clear_status) return false;
    if (!g.ep_E || ((uintptr_t)g.ep_E & 15) || g.ep_ld % 8 || ((uintptr_t)g.C0 & 15) || g.ldc % 8) return false;
    if (g.out == OUT_ACT_BWD && (g.ep_kind < 0 || g.ep_kind > 1)) return false;
    if (g.out == OUT_RMS_BWD && (!g.ep_row_a || !g.ep_row_b || !g.ep_col || ((uintptr_t)g.ep_col & 15) || g.N % 8)) return false;
  }
  if (g.M < 1 || g.N < 1 || g.K < 1 || g.n_terms < 1 || g.n_terms > 3) return false;
  if (g.halve_at_term >= g.n_terms) return false;
  if (g.lda % 8 || g.ldb % 8) return false;
  if (g.splits > 1 && g.out != OUT_F32) return false;
  if (g.alpha != 1.0f) return false;
  if (g.accumulate && (g.out != OUT_F32 || g.splits > 1)) return false;
  for (int t = 0; t < g.n_terms; ++t)
    if (((uintptr_t)g.terms[t].A & 15) || ((uintptr_t)g.terms[t].B & 15)) return false;
  return true;
}

// How a product is tiled on the two-CTA kernel (the wide forms exist for the majors the path uses), and an estimate of its
// time in us: rounds of the 74 SM pairs (148 SMs for the one-CTA kernel) times K blocks per split and term times the
// measured time per K block (0.44 us at 256 x 256, 0.57 wide, 0.36 one-CTA), and an epilogue per round.
struct TileShape {
  int wide, bn;
  double us;
};
// wide_ok: whether the wide forms may be chosen (a split count must not depend on the test hook, a launch does).
static TileShape pick_shape(int M, int N, bool a_mn, bool b_mn, long long k_iters, int splits, bool wide_ok,
                            bool whole_rows = false) {
  auto div = [](long long a, long long b) { return (a + b - 1) / b; };
  const int bn = pick_bn(N);
  const bool pair = M >= 2 * kBM && (b_mn ? bn % 128 == 0 : bn % 32 == 0);
  TileShape best = {WIDE_NONE, bn, 0.0};
  const long long narrow = (pair ? div(M, 2 * kBM) : div(M, kBM)) * div(N, bn) * splits;
  best.us = (double)div(narrow, pair ? 74 : 148) * ((double)k_iters * (pair ? 0.44 : 0.36) + 3.0);
  auto consider = [&](int wide, int wbn, long long tiles) {
    const double us = (double)div(tiles * splits, 74) * ((double)k_iters * 0.57 + 5.0);
    if (us < 0.95 * best.us) best = {wide, wbn, us};
  };
  if (!wide_ok || M < 2 * kBM) return best;
  if (!a_mn && !b_mn && N > 256 && N <= 512) {
    const int half = (int)div(div(N, 2), 64) * 64;
    if (whole_rows) return {WIDE_N, half, 0.0};
    consider(WIDE_N, half, div(M, 2 * kBM));
  }
  if (b_mn && M > 2 * kBM && bn % 128 == 0) consider(WIDE_M, bn, div(M, 4 * kBM) * div(N, bn));
  return best;
}

// What gemm_tc_launch does with a product.
static int k_blocks_per_split(const GemmDesc& g) {
  const int kb = (g.K + kBK - 1) / kBK, splits = g.splits < 1 ? 1 : g.splits;
  return (kb + splits - 1) / splits;
}
static TileShape launch_shape(const GemmDesc& g) {
  TileShape s = pick_shape(g.M, g.N, g.a_mn, g.b_mn, (long long)k_blocks_per_split(g) * g.n_terms, g.splits < 1 ? 1 : g.splits,
                           g_pair_mode == 1, g.whole_rows);
  // Few rows and many columns, not split (the test matrix L^-1 T, an unsplit U^T X, Reconstruct of few tiles): with tiles of 256 columns
  // most SMs are idle, and what the others load per K block and store at the end is the product's time.  The narrowest of 64 (one CTA a
  // tile) and 128 columns whose tiles still run in one round.  Steps (256 columns / this): 4096 x 5120, r = 64 70.9 / 70.7 us, 12608 x
  // 768, r = 96 88.7 / 87.2, 999 x 4096, r = 256 118.2 / 114.0, 8192 x 5120, r = 128 with a power iteration 196.1 / 194.1,
  // 5003 x 1000, r = 336 169.2 / 167.3.  Reconstruct of 64 to 4096 rows, r = 64 to 512, 146 sizes: 0.84 of the time in the geometric
  // mean, 1.03 at worst (256 x 9472, r = 64); U^T X of 64 to 2048 rows, 149 sizes: 0.72 and 0.91.
  // Rows of A of less than 128 bytes (rank 16 to 48): every tile reads the same short rows, and from 64 tiles of 64 columns side by side
  // on 128 are better, from 80 of those on 256.  U^T X of 512 rows, r = 16, 64 / 128 / 256 columns: d = 4096 5.0 / - / 6.0 us, d = 5120
  // 6.4 / 4.6 / 6.0, d = 9472 7.3 / 5.9 / 6.1; L^-1 T, r = 16: d = 5120 4.0 / 3.2 / 3.7, d = 11008 - / 4.2 / 3.9.
  // The split counts are picked for the tiles of pick_bn all the same: the K ranges, and with them the bits of a result, stay put.
  if (s.wide == WIDE_NONE && g.b_mn && g.N > 256 && g.splits <= 1) {
    const bool pair = g_pair_mode != 0 && g.M >= 2 * kBM;
    const bool short_rows = !pair && (g.a_mn ? g.M : g.K) < 64;
    const long long m_tiles = (g.M + (pair ? 2 * kBM : kBM) - 1) / (pair ? 2 * kBM : kBM);
    for (int bn = pair ? 128 : 64; bn <= 128 && bn < s.bn; bn *= 2) {
      const int n_tiles = (g.N + bn - 1) / bn;
      if (m_tiles * n_tiles <= (pair ? 74 : 148) && (!short_rows || n_tiles <= (bn == 64 ? 64 : 80))) { s.bn = bn; break; }
    }
  }
  // Small results in partial sums (Gram matrices, T = U^T G): the same with the widths that divide the columns, from
  // 32 (a staged box of fp32; 64 where B is MN-major, 128 where a pair shares it).  Steps, one tile / this: 999 x 4096, r = 256 118.0 /
  // 114.0 us, 8192 x 5120, r = 128 with a power iteration 197.3 / 194.1, 16384 x 4096, r = 256 179.5 / 177.5, RMS unit of 8192 x 4096,
  // r = 128 178.2 / 176.2, 4090 x 1000, r = 128 83.9 / 81.9, 12608 x 768, r = 96 88.2 / 87.2, 4096 x 5120, r = 64 the same.  Above 256
  // columns (the sampled rows', K-major: there the widths that pad no more than the tile they replace) 2048 x 1024, r = 288 133.7 / 132.7,
  // 5003 x 1000, r = 336 168.0 / 167.3, 4096 x 2048, r = 272 144.2 / 143.7.
  const int largest = g.a_mn || g.b_mn ? 256 : 512;
  if (s.wide == WIDE_NONE && g.N <= largest && g.M <= largest && g.out == OUT_F32 && !g.whole_rows && g.splits > 1) {
    const bool pair = g_pair_mode != 0 && g.M >= 2 * kBM && (g.b_mn ? s.bn % 128 == 0 : s.bn % 32 == 0);
    const long long units = (long long)((g.M + (pair ? 2 * kBM : kBM) - 1) / (pair ? 2 * kBM : kBM)) * g.splits;
    for (int bn = g.b_mn ? (pair ? 128 : 64) : 32; bn < s.bn; bn *= 2)
      if ((g.N + bn - 1) / bn * bn <= (g.N > 256 ? (g.N + s.bn - 1) / s.bn * s.bn : g.N) &&
          units * ((g.N + bn - 1) / bn) <= (pair ? 74 : 148)) { s.bn = bn; break; }
  }
  return s;
}
int gemm_tc_wide_form(const GemmDesc& g) { return launch_shape(g).wide; }

bool gemm_tc_can_own_rows(int M, int N) { return N <= 256 || (N <= 512 && M >= 2 * kBM && g_pair_mode == 1); }

int gemm_tc_tile_width(const GemmDesc& g) { return launch_shape(g).bn; }
int gemm_tc_pick_splits(int M, int N, int K, bool a_mn, bool b_mn, int max_splits, int free_sums) {
  const int bn = pick_bn(N);
  const int n_tiles = (N + bn - 1) / bn;
  const int tiles = ((M + kBM - 1) / kBM) * n_tiles;
  const int kb = (K + kBK - 1) / kBK;
  int base = 1;
  if (tiles < 96) {
    base = 148 / tiles;
    if (base > kb / 4) base = kb / 4;  // at least four K blocks per split
    if (base > max_splits) base = max_splits;
    if (base < 1) base = 1;
  }
  // Whole waves: with U units of work on S slots the launch takes ceil(U / S) rounds, so 86 tile pairs on 74 SM
  // pairs cost two full rounds.  Splitting the contraction s ways makes the rounds shorter and fills the last one;
  // it costs the partial sums (s * M * N * 4 bytes, read back by the reduction).  Time in units of one
  // K block (about 0.35 us for a 256 x 256 pair tile); the split count of the simple rule above is kept unless
  // another one is at least 15 % cheaper.
  const bool pair = M >= 2 * kBM && (b_mn ? bn % 128 == 0 : bn % 32 == 0);   // by shape (not by the test hook)
  const long long units = pair ? (long long)((M + 2 * kBM - 1) / (2 * kBM)) * n_tiles : tiles;
  const int slots = pair ? 74 : 148;
  // no empty split: with ceil(kb / sp) K blocks each, fewer splits may already cover the contraction (197 blocks
  // in 32 splits of 7 leave three splits with nothing to do but write zeros)
  auto without_empty = [&](int sp) {
    const int per = (kb + sp - 1) / sp;
    return (kb + per - 1) / per;
  };
  if (base > 1 && base <= free_sums) return without_empty(base);
  auto cost = [&](int sp) {
    const double rounds = (double)((units * sp + slots - 1) / slots);
    // the partial sums are read back once by the reduction (about 4 TB/s) behind one more launch
    const double reduce_us = sp > 1 ? (double)sp * (double)M * (double)N * 4.0 / 4.0e6 + 4.0 : 0.0;
    return rounds * (double)((kb + sp - 1) / sp) + reduce_us / 0.35;
  };
  int best = base;
  if (a_mn && b_mn && M > 2 * kBM && N > 2 * M) {
    // A projection at more than 256 columns: tile shape and split count together (the partial sums are written once and
    // read back once)
    double least = 1e30;
    for (int sp = 1; sp <= 8 && (sp == 1 || kb / sp >= 4); ++sp) {
      const double us = pick_shape(M, N, a_mn, b_mn, (kb + sp - 1) / sp, sp, true).us +
                        (sp > 1 ? 4.0 + (double)sp * M * N * 4.0 * (1.0 / 4.0e6 + 1.0 / 8.0e6) : 0.0);
      if (us < 0.98 * least) { least = us; best = sp; }
    }
    return without_empty(best);
  }
  double best_cost = cost(base);
  const int cap = max_splits < 8 ? max_splits : 8;
  for (int sp = 1; sp <= cap; ++sp) {
    if (sp > 1 && kb / sp < 4) break;
    const double c = cost(sp);
    if (c < best_cost && c < 0.85 * cost(base)) { best = sp; best_cost = c; }
  }
  return without_empty(best);
}

// A product with many rows streams one operand (X) once, and its tiles take about 0.36 us per 64-wide K block whatever
// their width up to 256 (the issue of the MMAs bounds narrow ones, the loads wide ones).  4096 rows are sixteen pair tiles
// on 74 SM pairs: split over K the same work uses the idle SMs, at the price of partial sums (written and read through L2
// at about 3 MB per us) and one more launch.  The split count with the least estimate, if that is at least 10 % below one.
// (Measured, whole steps: 4096 x 5120, r = 64: 112 -> 90 us with four splits; two passes over 8192 x 5120, r = 128:
// 269 -> 235 us with two.)
int gemm_tc_pick_tall_splits(int M, int N, int K) {
  const int bn = pick_bn(N);
  const bool pair = M >= 2 * kBM && bn % 32 == 0;
  const int rows = pair ? 2 * kBM : kBM, slots = pair ? 74 : 148;
  const long long tiles = (long long)((M + rows - 1) / rows) * ((N + bn - 1) / bn);
  const int kb = (K + kBK - 1) / kBK;
  auto cost = [&](int sp) {
    const double rounds = (double)((tiles * sp + slots - 1) / slots);
    return rounds * (double)((kb + sp - 1) / sp) * 0.36 + (sp > 1 ? 4.0 + (double)sp * M * N * 4.0 / 3.0e6 : 0.0);
  };
  int best = 1;
  for (int sp = 2; sp <= 8 && kb / sp >= 4; ++sp)
    if (cost(sp) < cost(best) && cost(sp) < 0.9 * cost(1)) best = sp;
  const int per = (kb + best - 1) / best;
  return (kb + per - 1) / per;                             // no empty split
}

GramPlan gemm_tc_gram_plan(int n, int l) {
  GramPlan p;
  if (l <= kGramTile || l > 2 * kGramTile || l % 8) return p;
  // Ranges per tile such that all pairs work and the longest takes least: a K block below the diagonal is four products, on it
  // three; no fewer than four K blocks each.
  const int kb = (n + kBK - 1) / kBK, pairs = 74;
  int best = 0;
  for (int off = 1; off + 2 <= pairs; ++off) {
    const int diag = (pairs - off) / 2;
    const int so = std::max(1, std::min(off, kb / 4)), sd = std::max(1, std::min(diag, kb / 4));
    const int t = std::max(((kb + so - 1) / so) * 4, ((kb + sd - 1) / sd) * 3);
    if (best == 0 || t < best) { best = t; p.s_diag = sd; p.s_off = so; }
  }
  p.tiles = 2;
  p.units = 2 * p.s_diag + p.s_off;
  return p;
}
size_t gemm_tc_gram_bytes(const GramPlan& p) { return (size_t)p.units * kGramTile * kGramTile * sizeof(float); }

cudaError_t gemm_tc_gram_launch(const void* Yh, const void* Yl, int n, int l, const GramPlan& plan, float* partials, float* W,
                                uint32_t* dev_status, const uint32_t* gate, cudaStream_t stream) {
  static std::atomic<bool> configured[64];
  constexpr size_t smem = (size_t)kGramStages * 4 * kABytes + 1024;
  int dev = 0;
  LORACT_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !configured[dev].load(std::memory_order_acquire)) {
    LORACT_CUDA_TRY(cudaFuncSetAttribute(gemm_tc_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  }
  GramParams p;
  p.kb_total = (n + kBK - 1) / kBK;
  p.tiles = plan.tiles; p.s_diag = plan.s_diag; p.s_off = plan.s_off;
  p.panels = l % 64 == 0;
  p.gate = gate; p.dev_status = dev_status;
  GramMaps maps;
  LORACT_CUDA_TRY(get_tmap(Yh, l, n, l, 64, 64, &maps.hi, 2, p.panels ? kBM / 64 : 0));
  LORACT_CUDA_TRY(get_tmap(Yl, l, n, l, 64, 64, &maps.lo, 2, p.panels ? kBM / 64 : 0));
  LORACT_CUDA_TRY(get_tmap(partials, kGramTile, (uint64_t)plan.units * kGramTile, kGramTile, 32, 32, &maps.out, 4));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * plan.units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LORACT_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_tc_gram_kernel, maps, p));
  count_launch("gemm_tc_gram", stream);
  const int nb = (l + 31) / 32, n_blocks = nb * (nb + 1) / 2;
  LORACT_CUDA_TRY(launch_pdl(reduce_gram_kernel, dim3(std::min(n_blocks, 148)), dim3(1024), 0, stream, (const float*)partials,
                             plan.tiles, plan.s_diag, plan.s_off, l, W, n_blocks, gate));
  count_launch("reduce_gram", stream);
  return cudaGetLastError();
}

cudaError_t gemm_tc_launch(const GemmDesc& g, uint32_t* dev_status, cudaStream_t stream) {
  if (!gemm_tc_supported(g)) return cudaErrorNotSupported;
  TcParams p;
  p.M = g.M; p.N = g.N;
  p.bn = pick_bn(g.N);
  p.kb_total = (g.K + kBK - 1) / kBK;
  const int splits = g.splits < 1 ? 1 : g.splits;
  p.kb_per_split = k_blocks_per_split(g);
  p.n_terms = g.n_terms;
  p.out = g.out; p.C0 = g.C0; p.C1 = g.C1; p.ldc = g.ldc; p.split_stride = g.split_stride;
  // Two CTAs per 256-row tile when there are at least 256 rows and the B tile splits into two legal halves; two
  // accumulators per pair where that is estimated to be faster.
  const TileShape shape = launch_shape(g);
  p.bn = shape.bn;
  const bool pair = shape.wide != WIDE_NONE ||
                    (g_pair_mode != 0 && g.M >= 2 * kBM && (g.b_mn ? p.bn % 128 == 0 : p.bn % 32 == 0));
  const int b_rows = pair ? p.bn / 2 : p.bn;   // rows (or columns) of B one CTA loads per K block
  p.b_bytes = g.b_mn ? (uint32_t)((b_rows + 63) / 64) * 8192u : (uint32_t)b_rows * 128u;
  p.tmem_cols = 32;
  // (the staged epilogue of a bf16 output reads 64 columns at a time)
  while ((int)p.tmem_cols < std::max(p.bn, g.out == OUT_F32 ? 32 : 64)) p.tmem_cols *= 2;
  p.accumulate = g.accumulate ? 1 : 0;
  p.ep_row_a = g.ep_row_a; p.ep_row_b = g.ep_row_b; p.ep_col = g.ep_col;
  p.dev_status = dev_status;
  p.st_m_tiles = 0; p.st_units = 0; p.st_keep_a = (long long)g.M * g.K * 2 <= kStreamKeepBytes; p.tma_store = 0; p.stages = 0; p.st_stages = kStreamStages; p.store_bufs = kStoreBufs; p.fuse_parts = 4;
  p.halve_at_term = g.halve_at_term > 0 ? g.halve_at_term : 0;
  p.a_keep_from_kb = g.a_keep_from_k >= 0 ? (int)(g.a_keep_from_k / kBK) : p.kb_total;
  p.gate = g.gate;
  p.clear_status = g.clear_status ? 1 : 0;
  p.lo_gate = g.lo_gate;
  p.lower = g.lower ? 1 : 0;
  p.early = g.gate ? 0 : (g.a_early ? 1 : 0) | (g.b_early ? 2 : 0);
  // A ring of at least four stages (three where a stage holds the B tiles of several terms); the epilogue takes it over as staging space, four boxes per warp where it holds them (a
  // pair of outputs fills two at a time: 16384 x 4096, r = 256, a step of 190.4 -> 189.8 us).
  auto take_ring = [&](uint32_t stage_bytes) -> size_t {
    const int fit = std::min(kMaxStages, (int)(kRingBytes / stage_bytes));
    p.stages = std::max(std::min(fit, 4), std::min(fit, p.kb_per_split * p.n_terms));
    p.store_bufs = p.stages * stage_bytes >= 4u * kEpiWarps * kStoreBoxBytes ? 4 : 2;
    return (size_t)p.stages * stage_bytes + 1024;
  };

  TmapPack maps;
  // The fused epilogues run on the persistent kernel however few rows there are, and that one, like the other two-CTA forms (from
  // 256 rows), expects whole tiles of A.
  const bool fused = g.out == OUT_RMS_BWD || g.out == OUT_ACT_BWD;
  p.a_rows = g.M <= 64 && !fused ? 64 : kBM;
  // MN-major operands whose extent and tiles are whole panels of 64: one load for all panels of a tile
  p.panels = (g.a_mn && g.M % 64 == 0 ? 1 : 0) | (g.b_mn && g.N % 64 == 0 && b_rows % 64 == 0 ? 2 : 0);
  for (int t = 0; t < g.n_terms; ++t) {
    if (p.panels & 1) LORACT_CUDA_TRY(get_tmap(g.terms[t].A, g.M, g.K, g.lda, 64, 64, &maps.a[t], 2, (uint32_t)p.a_rows / 64));
    else if (g.a_mn) LORACT_CUDA_TRY(get_tmap(g.terms[t].A, g.M, g.K, g.lda, 64, 64, &maps.a[t]));
    else LORACT_CUDA_TRY(get_tmap(g.terms[t].A, g.K, g.M, g.lda, 64, (uint32_t)p.a_rows, &maps.a[t]));
    if (p.panels & 2) LORACT_CUDA_TRY(get_tmap(g.terms[t].B, g.N, g.K, g.ldb, 64, 64, &maps.b[t], 2, (uint32_t)b_rows / 64));
    else if (g.b_mn) LORACT_CUDA_TRY(get_tmap(g.terms[t].B, g.N, g.K, g.ldb, 64, 64, &maps.b[t]));
    else LORACT_CUDA_TRY(get_tmap(g.terms[t].B, g.K, g.N, g.ldb, 64, (uint32_t)b_rows, &maps.b[t]));
  }
  for (int t = g.n_terms; t < 3; ++t) { maps.a[t] = maps.a[0]; maps.b[t] = maps.b[0]; }
  maps.c[0] = maps.a[0]; maps.c[1] = maps.a[0];
  if (splits == 1) p.split_stride = 0;
  // Output maps for the staged epilogue (boxes of 128 bytes x 32 rows).  Split-K partials are stacked along the
  // rows of one map, which needs them back to back in memory.
  auto staged_ok = [&](int bn) {
    const int es = g.out == OUT_F32 ? 4 : 2;
    // a box that reaches beyond its tile must reach beyond the matrix as well (and is clipped there)
    if (g.accumulate || (bn % (128 / es) && bn < g.N)) return false;
    if (((uintptr_t)g.C0 & 15) || (g.ldc * es) % 16) return false;
    if (g.out == OUT_SPLIT && ((uintptr_t)g.C1 & 15)) return false;
    if (splits > 1 && g.split_stride != (int64_t)g.M * g.ldc) return false;
    return true;
  };
  auto make_out_maps = [&]() -> cudaError_t {
    const int es = g.out == OUT_F32 ? 4 : 2;
    const uint32_t box = (uint32_t)(128 / es);
    LORACT_CUDA_TRY(get_tmap(g.C0, g.N, (uint64_t)splits * g.M, g.ldc, box, 32, &maps.c[0], es));
    if (g.out == OUT_SPLIT) LORACT_CUDA_TRY(get_tmap(g.C1, g.N, g.M, g.ldc, box, 32, &maps.c[1], es));
    return cudaSuccess;
  };

  // The fused epilogues (pre-norm and activation backward) exist in the persistent kernel only, which takes any number
  // of tiles: 256 columns wide where that gives every SM pair a tile, 128 otherwise.
  if (fused) {
    TcParams sp = p;
    sp.early = g.out == OUT_RMS_BWD && g.a_early && g.b_early ? 1 : 0;
    sp.st_m_tiles = (g.M + 2 * kBM - 1) / (2 * kBM);
    sp.bn = (long long)sp.st_m_tiles * ((g.N + 255) / 256) >= 74 ? 256 : 128;
    sp.b_bytes = (uint32_t)(sp.bn / 2 / 64) * 8192u;
    sp.tmem_cols = 2u * (uint32_t)sp.bn;
    const long long units = (long long)sp.st_m_tiles * ((g.N + sp.bn - 1) / sp.bn);
    if (units >= (1ll << 30)) return cudaErrorNotSupported;
    sp.st_units = (int)units;
    // sixteen epilogue warps with three boxes of E each, or two, or twelve warps with two: the first that leaves a ring
    // of three stages beside the resident B (a ring of two costs a quarter of the rate)
    const int room = kStreamSmemMax - 2048 - p.kb_total * (int)sp.b_bytes;
    int box_bytes = 0;
    static const int kChoice[3][2] = {{4, 3}, {4, 2}, {3, 2}};
    for (const auto& c : kChoice) {
      sp.fuse_parts = c[0];
      sp.store_bufs = c[1];
      box_bytes = 4 * c[0] * c[1] * (int)kFuseBoxBytes;
      sp.st_stages = std::min(kStreamStages, (room - box_bytes) / (int)kABytes);
      if (sp.st_stages >= 3) break;
    }
    LORACT_CUDA_TRY(get_tmap(g.terms[0].B, g.N, g.K, g.ldb, 64, 64, &maps.b[0]));
    LORACT_CUDA_TRY(get_tmap(g.C0, g.N, g.M, g.ldc, 32, 32, &maps.c[0]));
    LORACT_CUDA_TRY(get_tmap(g.ep_E, g.N, g.M, g.ep_ld, 32, 32, &maps.c[1]));
    const size_t ssmem = (size_t)sp.kb_total * sp.b_bytes + (size_t)sp.st_stages * kABytes + (size_t)box_bytes + 1024;
    if (g.out == OUT_RMS_BWD) return launch_stream<EP_RMS>(maps, sp, ssmem, stream);
    return g.ep_kind == 0 ? launch_stream<EP_SILU>(maps, sp, ssmem, stream) : launch_stream<EP_GELU>(maps, sp, ssmem, stream);
  }
  // Short contraction, large output, A K-major, B MN-major, one term (Reconstruct):
  // the persistent kernel with B resident, when there is more than one tile per resident pair.
  if (g_pair_mode == 1 && g.M >= 2 * kBM && !g.a_mn && g.b_mn && g.n_terms == 1 && splits == 1 && p.kb_total <= 8 &&
      g.N >= 256 && g.gate == nullptr && !g.clear_status && g.lo_gate == nullptr) {
    TcParams sp = p;
    // 256 columns per tile (the tensor pipe is issue-bound on narrower instructions).  The resident B takes
    // 16 KB per K block and CTA; beyond four K blocks the A ring and the staging boxes shrink to make room
    // (one box per warp cannot serve the two-box split output, which keeps 128 columns).
    sp.bn = (p.kb_total <= 4 || g.out != OUT_SPLIT) ? 256 : 128;
    sp.b_bytes = (uint32_t)(sp.bn / 2 / 64) * 8192u;
    sp.tmem_cols = 2u * (uint32_t)sp.bn;
    sp.st_stages = kStreamStages;
    sp.store_bufs = kStoreBufs;
    if (sp.bn == 256 && p.kb_total > 4) {
      sp.store_bufs = 1;
      const int room = kStreamSmemMax - 1024 - p.kb_total * (int)sp.b_bytes - kEpiWarps * (int)kStoreBoxBytes;
      sp.st_stages = std::min(kStreamStages, room / (int)kABytes);
    }
    sp.st_m_tiles = (g.M + 2 * kBM - 1) / (2 * kBM);
    const long long units = (long long)sp.st_m_tiles * ((g.N + sp.bn - 1) / sp.bn);
    if (units >= 148 && units < (1ll << 30)) {
      sp.st_units = (int)units;
      sp.tma_store = staged_ok(sp.bn) ? 1 : 0;
      if (sp.tma_store) LORACT_CUDA_TRY(make_out_maps());
      LORACT_CUDA_TRY(get_tmap(g.terms[0].B, g.N, g.K, g.ldb, 64, 64, &maps.b[0]));
      const size_t ssmem = (size_t)sp.kb_total * sp.b_bytes + (size_t)sp.st_stages * kABytes +
                           (size_t)kEpiWarps * sp.store_bufs * kStoreBoxBytes + 1024;
      return launch_stream<EP_NONE>(maps, sp, ssmem, stream);
    }
  }
  p.tma_store = staged_ok(p.bn) ? 1 : 0;
  if (p.tma_store) LORACT_CUDA_TRY(make_out_maps());
  if (shape.wide != WIDE_NONE) {
    const int na = shape.wide == WIDE_M ? 2 : 1, nb = shape.wide == WIDE_N ? 2 : 1;
    p.tmem_cols = 512;
    dim3 wgrid(2 * ((g.M + 2 * na * kBM - 1) / (2 * na * kBM)), (g.N + nb * p.bn - 1) / (nb * p.bn), splits);
    const size_t wsmem = take_ring(na * kABytes + nb * p.b_bytes);
    if (shape.wide == WIDE_N) return launch_pair_variant<false, false, WIDE_N>(maps, p, wgrid, wsmem, stream);
    return g.a_mn ? launch_pair_variant<true, true, WIDE_M>(maps, p, wgrid, wsmem, stream)
                  : launch_pair_variant<false, true, WIDE_M>(maps, p, wgrid, wsmem, stream);
  }
  if (pair) {
    dim3 pgrid(2 * ((g.M + 2 * kBM - 1) / (2 * kBM)), (g.N + p.bn - 1) / p.bn, splits);
    const size_t psmem = take_ring(kABytes + p.b_bytes);
    if (g.a_mn && g.b_mn) return launch_pair_variant<true, true>(maps, p, pgrid, psmem, stream);
    if (g.a_mn && !g.b_mn) return launch_pair_variant<true, false>(maps, p, pgrid, psmem, stream);
    if (!g.a_mn && g.b_mn) return launch_pair_variant<false, true>(maps, p, pgrid, psmem, stream);
    return launch_pair_variant<false, false>(maps, p, pgrid, psmem, stream);
  }
  dim3 grid((g.N + p.bn - 1) / p.bn, (g.M + kBM - 1) / kBM, splits);
  // Terms with one A (V^T (Th + Tm + Tl), the second product of a weight gradient) load it once where its tile takes two loads (M
  // not in whole panels) and there are four K blocks or more, and the B tiles of all terms leave room for three stages.  Measured,
  // whole weight gradients in us, shared / not: d = 1000, g = 23: r = 128 12.4 / 11.9, r = 256 13.4 / 14.0, r = 512 15.5 / 18.7;
  // g = 96: 10.9 / 10.8, 11.9 / 12.8, 14.6 / 17.2.  With A in panels the wait for the larger stage costs more than the loads
  // it saves (d = 1024, g = 96: 10.9 / 10.3, 11.8 / 11.5, 14.3 / 14.2; d = 4096, r = 128: 11.0 / 10.4), but for narrow
  // tiles of B over many K blocks: 16 columns from six on (r = 336: d = 1024 10.5 / 10.6, d = 11008 13.7 / 14.2; r = 512 11.3 /
  // 11.6, 14.9 / 15.7; r = 256 not: 9.6 / 9.5, 12.9 / 12.4), 32 from eight on (d = 11008, g = 23: r = 512 23.7 / 24.3, r = 336 21.4 / 20.2).
  const bool one_a_pays = p.kb_total >= 4 + (p.panels & 1 ? p.bn / 8 : 0);
  bool one_a = g.a_mn && g.b_mn && g.n_terms > 1 && p.halve_at_term == 0 && one_a_pays &&
               kABytes + (uint32_t)g.n_terms * p.b_bytes <= kRingBytes / 3;
  for (int t = 1; t < g.n_terms; ++t) one_a = one_a && g.terms[t].A == g.terms[0].A;
  const size_t smem = take_ring(kABytes + (one_a ? (uint32_t)g.n_terms : 1u) * p.b_bytes);
  if (one_a) return launch_variant<true, true, true>(maps, p, grid, smem, stream);
  if (g.a_mn && g.b_mn) return launch_variant<true, true>(maps, p, grid, smem, stream);
  if (g.a_mn && !g.b_mn) return launch_variant<true, false>(maps, p, grid, smem, stream);
  if (!g.a_mn && g.b_mn) return launch_variant<false, true>(maps, p, grid, smem, stream);
  return launch_variant<false, false>(maps, p, grid, smem, stream);
}

}  // namespace loract
