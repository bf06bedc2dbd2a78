// Small-block factorisation: Cholesky factor of an r x r Gram matrix and the inverse of that factor (the serial part of
// the orthonormalisation, the QR step of Algorithm 1 done through Gram matrices), as one thread-block-cluster kernel
// whose working set never leaves shared memory.  fp32 up to r = 512, fp64 up to r = 192.
//
// What bounds it is the chain of r pivots: nothing else is large (11 MFLOP at r = 256).  So the matrix is cut into
// 32 x 32 blocks, block ROW i and block COLUMN i of the inverse belong to CTA i of the cluster, and everything flows
// forward along the chain in groups of four columns -- no block ever makes a round trip:
//   * pivot warp: factors the diagonal block, four columns at a time.  Every lane holds the 4 x 4 pivot block of a group
//     and factors it for itself (one reciprocal square root, one product, one FMA per pivot on the chain), lane = matrix
//     row otherwise.  Published columns are read back once by the warp itself to bring the next 4 x 4 block up to date.
//   * follow-up warps (four, eight columns each): take every published group off the rest of the diagonal block and hand
//     the pivot warp its columns one group ahead.  Between diagonal blocks they do the same for the block that the chain
//     needs next: A(i, k+1) -= L(i, k) L(k+1, k)^T group by group while L(i, k) is being solved.
//   * solver warps (four, eight rows each): L(i, k) = A(i, k) L(k, k)^-T by forward substitution while block k is being
//     factored, and later the block column of the inverse, whose transpose solves the same system.  No inverse of a
//     diagonal block is formed.
//   * bulk warps (six or eight, two to a block): the updates nobody waits for, and the output.
//   * sender warps (three taking turns, one in fp64) copy finished groups and blocks to the CTAs that need them (bulk
//     distributed-shared-memory copies; one round of wait, proxy fence and up to fifteen copies takes longer than a group).
// A block is stored as eight groups of [32 rows][4 columns]: a group is one contiguous copy, a lane's row and a
// broadcast row are one 16-byte load each, without bank conflicts.  Loops are rolled: the kernel runs cold in every call, and
// fetching its code is part of its time (90 KB instead of 50 cost 2 to 4 us a launch).  The hand-offs of the
// pivot warp are named barriers (31 cycles against 110 for an mbarrier), all others are mbarriers that complete once.
//
// Shared-memory rates that fixed the shapes (measured on B200, cycles of the SM's pipe per warp instruction): a 16-byte
// load takes two cycles when each quarter of the warp reads one address, four otherwise; a store and a load of it behind
// a warp barrier take 30 cycles, a bulk copy to another CTA 280 (512 bytes) to 480 (4.6 KB) or 730 with seven receivers.
//
// Measured (one Gram matrix, back to back from a graph): fp32 r = 32 / 64 / 128 / 256: 4.3 / 6.8 / 11.4 / 24.1 us, r = 336 / 512 39.3 /
// 67.0, fp64 r = 64 / 128 / 192 10.2 / 18.3 / 27.2.  The figures beside the choices below were taken in turn with these; where
// they belong to an earlier form, they say so.
// Cycles per group of four columns: about 400 (pivots 120 of them); the step from one diagonal block to the next adds about 460.
// From the sixth block on the rows behind the chain lag and a block takes 6000 cycles instead of 3700; above eight blocks the early
// steps are bound by the bulk updates and by what an SM can send (up to 16000 cycles a block).
//
// Every wait on another CTA is bounded by a wall-clock limit; on expiry the CTA records LORACT_DEV_WAIT_EXPIRED, stops
// waiting and runs to its end (results are then invalid but every access stays in bounds), where it waits once more, with
// the same limit, for the copies that are still on their way to it.  The named barriers need no
// limit: both sides run through the same fixed sequence whatever the data and whether or not a wait has expired.
#include <atomic>

#include "common.cuh"

namespace loract {

namespace {

constexpr int kB = 32;                   // block edge
// fp32: three senders.  An SM issues a copy of one group every 56 cycles, so that a sender which waits, fences and copies to
// seven peers falls behind the groups (one sender: r = 128 / 256 / 336 / 512 11.6 / 25.9 / 48.3 / 87.3 us instead of 11.4 / 24.1 / 39.3 /
// 67.1; 0.1 less at r = 32 and 64).  fp64, at most six blocks and a slower chain: one (three: r = 64 / 128 / 192 10.8 / 19.2 / 28.0
// instead of 10.3 / 18.2 / 27.2).
template <typename T> __host__ __device__ constexpr int senders_of() { return sizeof(T) == 8 ? 1 : 3; }
// Six bulk warps; eight above eight block rows, where theirs is the work that lags (six: r = 336 / 400 / 512 39.3 / 53.7 / 75.2 us instead
// of 39.3 / 49.6 / 67.1).  Below, the registers and the issue slots of two fewer are worth more (eight: r = 64 / 128 / 256
// 7.2 / 12.3 / 25.6 us instead of 6.9 / 11.4 / 24.1, fp64 r = 64 / 192 11.0 / 28.1 instead of 10.3 / 27.2).
template <bool kBig> __host__ __device__ constexpr int bulk_of() { return kBig ? 8 : 6; }
template <typename T, bool kBig> __host__ __device__ constexpr int warps_of() { return 9 + bulk_of<kBig>() + senders_of<T>(); }
constexpr int kPan = 8;                  // groups of four columns in a block
constexpr uint64_t kClusterWaitNs = 50000000ull;  // 50 ms
// Warp -> role (plus the index inside the role).  The scheduler a warp shares is its number mod 4: the pivot warp's
// companions are senders and bulk warps, which are idle or waiting while it works.
enum Role : int { R_PIVOT = 0, R_FOLLOW = 1, R_SOLVE = 5, R_BULK = 9, R_SEND = 17 };
__constant__ unsigned char kRoleBig[20] = {R_PIVOT, R_FOLLOW + 0, R_FOLLOW + 1, R_FOLLOW + 2, R_SEND + 0, R_SOLVE + 0,
                                              R_FOLLOW + 3, R_SOLVE + 2, R_BULK + 0, R_SOLVE + 3, R_SOLVE + 1, R_BULK + 6,
                                              R_BULK + 1, R_BULK + 3, R_BULK + 5, R_BULK + 7, R_BULK + 2, R_BULK + 4,
                                              R_SEND + 1, R_SEND + 2};
__constant__ unsigned char kRoleSmall[18] = {R_PIVOT, R_FOLLOW + 0, R_FOLLOW + 1, R_FOLLOW + 2, R_SEND + 0, R_SOLVE + 0,
                                             R_FOLLOW + 3, R_SOLVE + 2, R_BULK + 0, R_SOLVE + 3, R_SOLVE + 1, R_BULK + 1,
                                             R_BULK + 2, R_BULK + 3, R_BULK + 5, R_BULK + 4, R_SEND + 1, R_SEND + 2};

constexpr int kGrp = kB * 4;             // elements of a group of four columns
constexpr int kBlk = kB * kB;            // elements of a block
template <typename T> struct Cfg;
template <> struct Cfg<float> { static constexpr int kMaxR = 256; };    // (kept whole; see kBig)
template <> struct Cfg<double> { static constexpr int kMaxR = 192; };

struct SCParams {
  int r;
  const void* partials;    // T
  int n_partials;
  int64_t partial_stride;
  float shift_rel;
  float shift_diag_rel;    // each diagonal entry is also multiplied by (1 + shift_diag_rel)
  const uint32_t* gate;    // optional device word: zero means every CTA leaves at once
  // optional: three words that receive the decision on a further orthonormalisation round
  // { est > gate_threshold or est not finite or *dev_status != 0, est as float bits, 1 or 2 },
  // est = sum_ij Linv_ij^2 W_jj (W_jj the diagonal as factored): trace of the inverse of the diagonally scaled matrix
  uint32_t* gate_out;
  float gate_threshold;
  uint32_t absent_share_bytes;   // test hook: bytes of the shares that CTA 0 waits for and nobody sends
  float* linv_f32;
  __nv_bfloat16* linv_hi;
  __nv_bfloat16* linv_lo;
  uint32_t* dev_status;
  int64_t in_ld, out_ld;   // row strides of the partial matrices and of the outputs
};

__device__ __forceinline__ int off_slot(int i, int k) { return i * (i - 1) / 2 + k; }   // block (i, k), i > k

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void bar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
// All lanes have written; one arrival announces it.  Predicated, like the stores of single lanes on the chain: a branch around
// them costs more than they do.
__device__ __forceinline__ void warp_arrive(uint64_t* bar, int lane) {
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.eq.s32 p, %1, 0;\n\t"
      "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
      ::"r"(smem_addr(bar)), "r"(lane)
      : "memory");
}
// kFromPeers: what warps of other CTAs did before they arrived has to be ordered as well (acquire at cluster scope).
template <bool kFromPeers>
__device__ __forceinline__ bool bar_try(uint64_t* bar) {
  uint32_t ok;
  if (kFromPeers)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar))
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar))
        : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Every barrier of this kernel completes exactly once (phase 0).  Called by all lanes of a warp.  Returns false once
// the CTA has given up.
template <bool kFromPeers = false>
__device__ __forceinline__ bool bar_wait(uint64_t* bar, volatile int* gave_up, uint64_t limit_ns = kClusterWaitNs) {
  if (bar_try<kFromPeers>(bar)) return true;
  uint64_t t0 = 0;
#pragma unroll 1
  for (uint32_t spin = 1;; ++spin) {
    if (bar_try<kFromPeers>(bar)) return true;
    if ((spin & 255u) == 0u) {
      if (*gave_up) return false;
      const uint64_t now = timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) { *gave_up = 1; return false; }
    }
  }
}
// The same for a CTA that has given up: until the bytes have landed, or for as long again.
__device__ __forceinline__ void bar_drain(uint64_t* bar) {
  const uint64_t t0 = timer_ns();
#pragma unroll 1
  while (!bar_try<false>(bar) && timer_ns() - t0 <= kClusterWaitNs) {}
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// Execution only: does not wait for this thread's stores (the output) to reach L2, which takes 0.6 us.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Named barriers between the pivot warp and the follow-up warps, each used once: group g of the diagonal block has been
// handed over (64 threads), group g has been published (the pivot warp and every follow-up warp that needs it).
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ int id_staged(int g) { return 1 + g; }
__device__ __forceinline__ int id_published(int g) { return 9 + g; }                 // g < 6: nobody needs the last two
__device__ __forceinline__ int readers_of(int g) { return 32 * (4 - (g >> 1)); }     // pivot warp + follow-up warps

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) from this CTA's shared memory
// into a peer's; on arrival `bytes` is taken off the transaction count of the peer's barrier `bar`.
__device__ __forceinline__ void bulk_to_peer(uint32_t dst_cluster_addr, uint32_t src_local_addr, uint32_t bytes,
                                             uint32_t bar_cluster_addr) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst_cluster_addr), "r"(src_local_addr), "r"(bytes), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ------------------------------------------------------------------ four consecutive elements
template <typename T> struct V4 { T v[4]; };
__device__ __forceinline__ V4<float> ld4(const float* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  return {{q.x, q.y, q.z, q.w}};
}
__device__ __forceinline__ V4<double> ld4(const double* p) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(float* p, const V4<float>& x) {
  *reinterpret_cast<float4*>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
}
__device__ __forceinline__ void st4(double* p, const V4<double>& x) {
  *reinterpret_cast<double2*>(p) = make_double2(x.v[0], x.v[1]);
  *reinterpret_cast<double2*>(p + 2) = make_double2(x.v[2], x.v[3]);
}
// The same for the lanes with `on` set, without a branch.
__device__ __forceinline__ void st4_if(bool on, float* p, const V4<float>& x) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.s32 p, %5, 0;\n\t"
      "@p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n\t}"
      ::"r"(smem_addr(p)), "f"(x.v[0]), "f"(x.v[1]), "f"(x.v[2]), "f"(x.v[3]), "r"((int)on)
      : "memory");
}
__device__ __forceinline__ void st4_if(bool on, double* p, const V4<double>& x) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.s32 p, %5, 0;\n\t"
      "@p st.shared.v2.f64 [%0], {%1, %2};\n\t"
      "@p st.shared.v2.f64 [%0 + 16], {%3, %4};\n\t}"
      ::"r"(smem_addr(p)), "d"(x.v[0]), "d"(x.v[1]), "d"(x.v[2]), "d"(x.v[3]), "r"((int)on)
      : "memory");
}
// acc - a . b over four elements
template <typename T>
__device__ __forceinline__ T sub4(T acc, const V4<T>& a, const V4<T>& b) {
#pragma unroll
  for (int u = 0; u < 4; ++u) acc = fma(-a.v[u], b.v[u], acc);
  return acc;
}

// Reciprocal square root of a pivot (positive and normal where the result is used).  fp32: one MUFU instruction (2 ulp).
// fp64: the hardware's starting value (about 20 bits) and two Newton steps y <- y + y (1 - x y^2) / 2.
__device__ __forceinline__ float pivot_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ double pivot_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int s = 0; s < 2; ++s) y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
  return y;
}

// One published group of four columns of a diagonal block's factor: L[0..31][4], then the four reciprocals of the
// diagonal with zero where a pivot was clamped (what a column of L is scaled with: entries below such a pivot are
// rounding noise and are dropped), then the four reciprocals themselves (for the inverse).
constexpr int kPanElems = kGrp + 8;

// ------------------------------------------------------------------ the pivots (one warp, lane = row of the block)
// `staged`: the diagonal block, whose group g has every earlier group but g - 1 taken off when id_staged(g) completes.
// Rows of a group above its own diagonal carry values nobody reads.  Returns true if a pivot was clamped.
template <typename T>
__device__ __forceinline__ bool factor_diagonal(const T* staged, T* panels, uint64_t* bars, T floor_, int lane) {
  bool clamped = false;
  const T rfloor = pivot_rsqrt(floor_);
  V4<T> x = {{(T)0, (T)0, (T)0, (T)0}};
  V4<T> b[4] = {x, x, x, x};
  T* pan = panels;
#pragma unroll 1
  for (int p = 0; p < kPan; ++p) {
    named_sync(id_staged(p), 64);
    V4<T> a = ld4(staged + lane * 4);
    V4<T> g[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = ld4(staged + (4 * p + i) * 4);
    if (p > 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) b[i] = ld4(pan - kPanElems + (4 * p + i) * 4);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int i = j; i < 4; ++i) g[i].v[j] = sub4(g[i].v[j], b[i], b[j]);
      a.v[j] = sub4(a.v[j], x, b[j]);
    }
    V4<T> rz, rd;
    auto pivot = [&](int c, T d) {
      const bool bad = !(d > floor_);
      clamped |= bad;
      const T y = pivot_rsqrt(d);
      rz.v[c] = bad ? (T)0 : y;
      rd.v[c] = bad ? rfloor : y;
    };
    // column 0
    pivot(0, g[0].v[0]);
    const T l10 = g[1].v[0] * rz.v[0], l20 = g[2].v[0] * rz.v[0], l30 = g[3].v[0] * rz.v[0];
    x.v[0] = a.v[0] * rz.v[0];
    const T d1 = fma(-l10, l10, g[1].v[1]);
    const T s21 = fma(-l20, l10, g[2].v[1]), s31 = fma(-l30, l10, g[3].v[1]), t1 = fma(-x.v[0], l10, a.v[1]);
    const T d2 = fma(-l20, l20, g[2].v[2]), s32 = fma(-l30, l20, g[3].v[2]), t2 = fma(-x.v[0], l20, a.v[2]);
    const T d3 = fma(-l30, l30, g[3].v[3]), t3 = fma(-x.v[0], l30, a.v[3]);
    // column 1
    pivot(1, d1);
    const T l21 = s21 * rz.v[1], l31 = s31 * rz.v[1];
    x.v[1] = t1 * rz.v[1];
    const T e2 = fma(-l21, l21, d2), u32 = fma(-l31, l21, s32), v2 = fma(-x.v[1], l21, t2);
    const T e3 = fma(-l31, l31, d3), v3 = fma(-x.v[1], l31, t3);
    // column 2
    pivot(2, e2);
    const T l32 = u32 * rz.v[2];
    x.v[2] = v2 * rz.v[2];
    const T f3 = fma(-l32, l32, e3), w3 = fma(-x.v[2], l32, v3);
    // column 3
    pivot(3, f3);
    x.v[3] = w3 * rz.v[3];
    st4(pan + lane * 4, x);
    st4(pan + kGrp, rz);                   // (the same values in every lane)
    st4(pan + kGrp + 4, rd);
    __syncwarp();
    if (p < kPan - 2) named_arrive(id_published(p), readers_of(p));
    warp_arrive(bars + p, lane);
    staged += kGrp;
    pan += kPanElems;
  }
  return clamped;
}

// fp32: the products that are taken off a block in one step are summed first, and the sum is taken off once (substitution,
// follow-up and bulk warps).  Taken off one by one, every product is rounded at the size of the block, and the error of the
// factor grows with the square root of r: relative error of L^-1 against fp64 at condition number 1e2 / 1e4, r = 256:
// 1.2e-6 / 4.5e-5 so, 5.0e-7 / 2.5e-5 in sums (products of 32 x 32 blocks, the form before: 4.8e-7 / 2.6e-5), r = 512: 1.7e-6 /
// 6.3e-5, 5.3e-7 / 2.6e-5 (6.1e-7 / 4.8e-5).  It costs no time (one by one, r = 256 / 336 / 512: 24.1 / 40.1 / 68.0 us
// instead of 24.1 / 39.3 / 67.1).  fp64 results are rounded to fp32 and have no need of it.
template <typename T> constexpr bool kBlockSums = sizeof(T) == 4;

// ------------------------------------------------------------------ forward substitution (four warps, eight rows each)
// Solves x L^T = t in place (blk: t, then x) for the triangular factor L of a diagonal block that is being published.
// A lane holds one row's columns of the groups cg and cg + 4 (cg = lane / 8): the lanes of the current group form x, the
// others get it by shuffle and take the group off their columns.  `inverse`: scale with the plain reciprocals.
template <typename T, int H>
__device__ __forceinline__ void solve_half(const V4<T> (&was)[2], V4<T> (&acc)[2], T* blk, const T* panels, uint64_t* pan_bars, uint64_t* sol_bars,
                                           bool inverse, int row, int lane, volatile int* gave_up) {
  const int cg = lane >> 3;
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    const int p = 4 * H + q;
    const T* pan = panels + p * kPanElems;
    const T* low = pan + 16 * p;                           // row 4 p
    bar_wait(pan_bars + p, gave_up);
    const V4<T> rr = ld4(pan + kGrp + (inverse ? 4 : 0));
    const V4<T> r1 = ld4(low + 4), r2 = ld4(low + 8), r3 = ld4(low + 12);
    // fp32: the rows that the group is taken off with are fetched before x is known (where they are used: r = 128 / 256 / 336 / 512
    // 11.9 / 24.8 / 41.1 / 68.4 us instead of 11.5 / 24.1 / 39.2 / 66.9); fp64 has no registers for them
    V4<T> b[2][4];
    if (sizeof(T) == 4) {
#pragma unroll
      for (int h = H; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) b[h][j] = ld4(pan + (4 * (cg + 4 * h) + j) * 4);
    }
    V4<T> t = acc[H], x;
    if (kBlockSums<T>) {
#pragma unroll
      for (int u = 0; u < 4; ++u) t.v[u] += was[H].v[u];
    }
    x.v[0] = t.v[0] * rr.v[0];
    x.v[1] = fma(-x.v[0], r1.v[0], t.v[1]) * rr.v[1];
    x.v[2] = fma(-x.v[1], r2.v[1], fma(-x.v[0], r2.v[0], t.v[2])) * rr.v[2];
    x.v[3] = fma(-x.v[2], r3.v[2], fma(-x.v[1], r3.v[1], fma(-x.v[0], r3.v[0], t.v[3]))) * rr.v[3];
    st4_if(cg == q, blk + p * kGrp + row * 4, x);
    warp_arrive(sol_bars + p, lane);
#pragma unroll
    for (int u = 0; u < 4; ++u) x.v[u] = __shfl_sync(0xffffffffu, x.v[u], (q << 3) | (lane & 7));
#pragma unroll
    for (int h = H; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        acc[h].v[j] = sub4(acc[h].v[j], x, sizeof(T) == 4 ? b[h][j] : ld4(pan + (4 * (cg + 4 * h) + j) * 4));
  }
}

// ------------------------------------------------------------------ block updates
// A follow-up warp w holds columns 8 w .. 8 w + 7 of a block, a lane two quads acc[h] of them: in fp32 rows lane % 16 and
// lane % 16 + 16 of group 2 w + lane / 16 (six loads a group; with one row and both groups, as in fp64, nine, and r = 64 /
// 256 / 512 takes 7.0 / 24.7 / 67.5 instead of 6.9 / 24.1 / 67.1 us; fp64 with two rows: r = 64 / 192 10.5 / 27.5 instead of 10.3 / 27.2).
template <typename T>
struct FollowLane {
  static constexpr bool kTwoRows = sizeof(T) == 4;
  int w, lane;
  __device__ __forceinline__ int group(int h) const { return kTwoRows ? 2 * w + (lane >> 4) : 2 * w + h; }
  __device__ __forceinline__ int at(int h) const { return group(h) * kGrp + (kTwoRows ? (lane & 15) + 16 * h : lane) * 4; }
};
// acc -= (rows of group A) . (rows of group B)
template <typename T>
__device__ __forceinline__ void take_off_group(V4<T> (&acc)[2], const T* A, const T* Bg, const FollowLane<T>& f) {
  if (FollowLane<T>::kTwoRows) {
    const V4<T> a0 = ld4(A + (f.lane & 15) * 4), a1 = ld4(A + (f.lane & 15) * 4 + 64);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const V4<T> b = ld4(Bg + (4 * f.group(0) + j) * 4);
      acc[0].v[j] = sub4(acc[0].v[j], a0, b);
      acc[1].v[j] = sub4(acc[1].v[j], a1, b);
    }
  } else {
    const V4<T> a = ld4(A + f.lane * 4);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[h].v[j] = sub4(acc[h].v[j], a, ld4(Bg + (4 * f.group(h) + j) * 4));
  }
}
// C (or zero) -= A B^T for columns 16 half .. 16 half + 15 of a block, 4 x 4 outputs per lane: rows row0 + 8 i, columns
// col0 + 4 j.  With eight warps at it the shared-memory pipe is the bound: per group four loads of A at four cycles, four of
// B at two (two addresses per quarter warp), and C in single elements without conflicts (a warp access covers eight rows of a
// group); one warp alone waits for its loads, hence the unrolled loop (by eight in the kernels for
// many blocks and for fp64; in the small fp32 kernel the code of that costs 2 us a launch).
// Against rows 16 half .., with conflicts on C, unrolled by two: 2340 -> 2200 cycles for eight halves with eight warps, 1350
// -> 1100 with one.  A whole block per warp (a third fewer loads) or two halves at a time (a quarter fewer) leave too few warps at work:
// r = 512 75 and 73 us in a form that took 71.
template <typename T, int kUnroll>
__device__ __forceinline__ void take_off_half(T* C, const T* A, const T* Bm, bool from_zero, int half, int lane) {
  const int row0 = (lane & 3) + 4 * (lane >> 4), col0 = (lane >> 2) & 3;
  C += 4 * half * kGrp + row0 * 4 + col0;
  A += row0 * 4;
  Bm += (16 * half + col0) * 4;
  T acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][j] = from_zero || kBlockSums<T> ? (T)0 : C[j * kGrp + 32 * i];
#pragma unroll kUnroll
  for (int q = 0; q < kPan; ++q) {
    V4<T> a[4], b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = ld4(Bm + q * kGrp + 16 * j);
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = ld4(A + q * kGrp + 32 * i);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(-a[i].v[u], b[j].v[u], acc[i][j]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      C[j * kGrp + 32 * i] = kBlockSums<T> && !from_zero ? C[j * kGrp + 32 * i] + acc[i][j] : acc[i][j];
}

__device__ __forceinline__ void load_quad(const float* src, V4<float>& s) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(src));
  s.v[0] += v.x; s.v[1] += v.y; s.v[2] += v.z; s.v[3] += v.w;
}
__device__ __forceinline__ void load_quad(const double* src, V4<double>& s) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(src)), b = __ldg(reinterpret_cast<const double2*>(src) + 1);
  s.v[0] += a.x; s.v[1] += a.y; s.v[2] += b.x; s.v[3] += b.y;
}

// Shared memory of every CTA (the same layout in all of them, so a local address maps to any peer), in elements of T.
// Up to eight blocks: off-diagonal blocks (own row: A, then L; other rows: L as it arrives), the blocks of the own column of
// the inverse (transposed), and the published diagonal blocks.  The own diagonal block borrows a slot of the inverse that is
// not in use yet (the last one, first written after the block has been factored) or never used by this CTA.
// kBig, nine to sixteen blocks (a cluster of sixteen CTAs): what a CTA holds for good is its own row up to the diagonal
// and its own column of the inverse from there on, sixteen slots together, and the diagonal block.  Received blocks are
// needed during one step only: two sets of fifteen, used in turn, and a ring of six published diagonal blocks.  A set may
// be overwritten once every CTA that reads it has said so (free_bar, two steps back).
__host__ __device__ constexpr int x_slots(int nblk) { return nblk < 3 ? 3 : nblk; }
constexpr int kBigBlk = 16, kBigPans = 6;
constexpr int kReaders = 16;             // warps of a CTA that read received blocks or panels: follow-up, solver, bulk
template <typename T, bool kBig>
__host__ __device__ constexpr size_t smem_elems(int nblk) {
  return kBig ? (size_t)kBlk * (kBigBlk + 1 + 2 * (kBigBlk - 1)) + (size_t)kBigPans * kPan * kPanElems
              : (size_t)kBlk * (nblk * (nblk - 1) / 2 + x_slots(nblk)) + (size_t)nblk * kPan * kPanElems;
}

template <typename T, bool kBig>
__global__ void __launch_bounds__(32 * warps_of<T, kBig>(), 1) small_block_cluster_kernel(SCParams p) {
  constexpr int kWarps = warps_of<T, kBig>(), kCThreads = 32 * kWarps, kSendWarps = senders_of<T>();
  constexpr int kBulkWarps = bulk_of<kBig>();
  constexpr int kMaxBlk = kBig ? kBigBlk : 8;              // block rows, and CTAs of the cluster
  constexpr int kMaxOff = kMaxBlk * (kMaxBlk - 1) / 2;
  constexpr uint32_t kBlkBytes = (uint32_t)(kBlk * sizeof(T)), kGrpBytes = (uint32_t)(kGrp * sizeof(T));
  constexpr uint32_t kPanBytes = (uint32_t)(kPanElems * sizeof(T));
  extern __shared__ __align__(16) unsigned char sc_smem[];
  __shared__ __align__(8) uint64_t pan_bar[kMaxBlk][kPan];   // group g of diagonal block k is here
  __shared__ __align__(8) uint64_t next_bar[kMaxBlk][kPan];  // group g of L(k + 1, k), another CTA's, is here
  __shared__ __align__(8) uint64_t off_bar[kMaxOff];         // L(i, k), i >= k + 2, another CTA's, is here
  __shared__ __align__(8) uint64_t sol_bar[kMaxBlk][kPan];   // group g of L(own, k), k < own, or X(k, own) is solved
  __shared__ __align__(8) uint64_t rdy_bar[kMaxBlk];         // the block to solve at step k has every update
  __shared__ __align__(8) uint64_t bulk_bar[kMaxBlk];        // block j has every update but that of step j - 1
  __shared__ __align__(8) uint64_t free_bar[kBig ? kMaxBlk : 1];   // every peer is done with what step k received
  __shared__ __align__(8) uint64_t est_bar;                  // CTA 0: every share of the estimate is here
  __shared__ uint32_t s_done[kBig ? kMaxBlk : 1];            // warps of this CTA that are done with what step k received
  __shared__ T s_red[kWarps];
  __shared__ T s_shift, s_floor;
  __shared__ int s_gave_up;
  __shared__ float s_est[kBulkWarps * kMaxBlk];   // CTA 0: the shares of the estimate

  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int me = (int)rank;              // block row and block column of the inverse of this CTA
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // (fetched this early, from constant memory that nobody has touched: at its use it costs 600 cycles of the first pivots)
  const int role = kBig ? kRoleBig[warp] : kRoleSmall[warp];
  const int r = p.r;
  const int nblk = (r + kB - 1) / kB;
  const int noff = nblk * (nblk - 1) / 2;
  const bool active = me < nblk;
  T* off = reinterpret_cast<T*>(sc_smem);
  T* xt = off + (size_t)noff * kBlk;                     // (small) block (k, own) of the inverse at slot k
  T* pans = kBig ? off + (size_t)kBlk * (kBigBlk + 1 + 2 * (kBigBlk - 1)) : xt + (size_t)x_slots(nblk) * kBlk;
  T* own = kBig ? off + (size_t)kBigBlk * kBlk : xt + (size_t)(me + 2 <= nblk - 1 ? nblk - 1 : (me >= 1 ? 0 : 2)) * kBlk;
  // L(i, k) of another CTA's row (and, as an address in a peer, where this CTA's own L(me, k) is sent)
  auto slot = [&](int i, int k) {
    return kBig ? off + (size_t)(kBigBlk + 1 + (k & 1) * (kBigBlk - 1) + i - 1) * kBlk : off + (size_t)off_slot(i, k) * kBlk;
  };
  auto panel = [&](int k) { return pans + (size_t)(kBig ? k % kBigPans : k) * kPan * kPanElems; };
  // the block this CTA solves at step k, and where an update of block j (row: j < me, diagonal: j = me) goes
  auto solved = [&](int k) {
    return kBig ? off + (size_t)k * kBlk : (k < me ? off + (size_t)off_slot(me, k) * kBlk : xt + (size_t)k * kBlk);
  };
  auto target = [&](int j) { return j == me ? own : solved(j); };

  // A gated launch that is not needed leaves before any set-up: the same word in every CTA of the cluster.  Its predecessor is a gated
  // launch itself, so this grid may start before that one has waited: the rule at GemmDesc::gate says why the word may be read
  // this early and why the wait is still executed.
  if (p.gate != nullptr && *(const volatile uint32_t*)p.gate == 0u) { pdl_launch_dependents(); pdl_wait(); return; }

  // ---- set-up: barriers, with the byte counts they will receive
  auto panel_comes = [&](int k) { return active && k < nblk && k != me; };
  auto next_comes = [&](int k) { return active && k + 1 < nblk && k + 1 != me; };
  auto block_comes = [&](int i, int k) { return active && i < nblk && i != me && i >= k + 2 && (me <= k || me > i); };
  auto row_of_slot = [&](int b) { int i = 1; while (off_slot(i + 1, 0) <= b) ++i; return i; };
  if (tid < kMaxBlk * kPan) {
    const int k = tid / kPan, q = tid % kPan;
    bar_init(&pan_bar[k][q], 1);
    bar_init(&next_bar[k][q], 1);
    bar_init(&sol_bar[k][q], 4);
    if (q == 0) { bar_init(&rdy_bar[k], 4); bar_init(&bulk_bar[k], 2); }
    if (kBig && q == 1) { bar_init(&free_bar[k], (uint32_t)(nblk - 1)); s_done[k] = 0u; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (panel_comes(k)) bar_expect(&pan_bar[k][q], kPanBytes);
    if (next_comes(k)) bar_expect(&next_bar[k][q], kGrpBytes);
  } else if (tid >= kMaxBlk * kPan && tid < kMaxBlk * kPan + kMaxOff) {
    const int b = tid - kMaxBlk * kPan, i = row_of_slot(b);
    bar_init(&off_bar[b], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (block_comes(i, b - off_slot(i, 0))) bar_expect(&off_bar[b], kBlkBytes);
  } else if (tid == kMaxBlk * kPan + kMaxOff) {
    s_gave_up = 0;
    bar_init(&est_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!kBig && p.gate_out && me == 0) bar_expect(&est_bar, (uint32_t)(kBulkWarps * nblk * sizeof(float)) + p.absent_share_bytes);
  }
  __syncthreads();
  cluster_arrive();                       // waited for under the load: nobody sends before every CTA's barriers exist
  // everything above overlaps the tail of the previous kernel; global memory only from here on
  pdl_wait();
  pdl_launch_dependents();

  // ---- load: this CTA's block row, summed over the partials, raw into its place.  One matrix, the usual case, is copied with
  // cp.async: every copy is in flight before anything waits.  (Through registers, a CTA with sixteen block rows waited for seven loads in
  // turn and started 4.3 us after the first; now 1.6.  Steps, before / after: fp32 512 x 768, r = 64 102.1 / 100.2 us, 5003 x 1000,
  // r = 336 172.6 / 169.2, 8192 x 5120, r = 128 with a power iteration 210.7 / 208.8, 4096 x 5120, r = 64 76.7 / 75.6; 16384 x 4096, r = 256 and
  // 16384 x 11008, r = 512 the same within their noise.)  Meanwhile the trace of W (the same order of additions in every CTA
  // and warp) gives the diagonal shift and the pivot floor.  The thread that wrote a quad of the diagonal adds the shift to it.
  {
    const T* parts = (const T*)p.partials;
    constexpr int kQuads = kB * kB / 4;
    const int n_quads = active ? (me + 1) * kQuads : 0;
    auto quad_at = [&](int e) { return target(e / kQuads) + (e & 7) * kGrp + ((e & (kQuads - 1)) >> 3) * 4; };
#pragma unroll 1
    for (int e = tid; e < n_quads; e += kCThreads) {
      const int row = me * kB + ((e & (kQuads - 1)) >> 3), col = (e / kQuads) * kB + 4 * (e & 7);
      const bool in = row < r && col < r;
      const T* src = parts + (in ? (int64_t)row * p.in_ld + col : 0);
      T* dst = quad_at(e);
      if (p.n_partials == 1) {
#pragma unroll
        for (int h = 0; h < (int)sizeof(T) / 4; ++h)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                       ::"r"(smem_addr(dst) + 16 * h), "l"((const unsigned char*)src + 16 * h), "r"(in ? 16 : 0) : "memory");
      } else {
        V4<T> acc = {{(T)0, (T)0, (T)0, (T)0}};
        if (in) {
#pragma unroll 4
          for (int q = 0; q < p.n_partials; ++q) load_quad(src + (int64_t)q * p.partial_stride, acc);
        }
        st4(dst, acc);
      }
    }
    // (0.4 us however long ago the others arrived: under the copies; kBig: 0.5 us slower so)
    if (!kBig) {
      __syncwarp();
      cluster_wait();
    }
    T t = (T)0;
#pragma unroll 1
    for (int i = tid; i < r; i += kCThreads) {
      T d = (T)0;
#pragma unroll 4
      for (int q = 0; q < p.n_partials; ++q)
        d += __ldg(parts + (int64_t)q * p.partial_stride + (int64_t)i * p.in_ld + i);
      t += d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s_red[warp] = t;
    __syncthreads();
    t = lane < kWarps ? s_red[lane] : (T)0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    T mean_diag = t / (T)r;
    if (!(mean_diag == mean_diag) || mean_diag > (T)3.0e38 || mean_diag < (T)0) {
      if (p.dev_status && me == 0 && tid == 0) { atomicOr(p.dev_status, LORACT_DEV_NONFINITE); __threadfence(); }
      mean_diag = (T)1;
    }
    if (mean_diag == (T)0) mean_diag = (T)1;
    const T shift = (T)p.shift_rel * mean_diag;
    if (tid == 0) {
      s_shift = shift;
      s_floor = mean_diag * (sizeof(T) == 8 ? (T)1e-15 : (T)1e-7);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // this thread's quad of the diagonal block, if any (a block has fewer quads than the CTA threads)
    const int a0 = me * kQuads, e = a0 + (tid + kCThreads - a0 % kCThreads) % kCThreads;
    const int a = (e & (kQuads - 1)) >> 3, dcol = a - 4 * (e & 7);
    if (active && e < a0 + kQuads && dcol >= 0 && dcol < 4) {
      const bool in_range = me * kB + a < r;              // padding rows of a ragged last block: identity
      T* at = quad_at(e) + dcol;
      *at = in_range ? *at + (*at * (T)p.shift_diag_rel + shift) : (T)1;
    }
  }
  __syncthreads();
  if (kBig) cluster_wait();

  volatile int* gave_up = &s_gave_up;
  const T floor_ = s_floor;
  // the CTA this lane signals and copies to: the next one of the chain first
  const int to = lane < nblk ? (me + 1 + lane) % nblk : 0;
  const bool peer = lane + 1 < nblk;
  // Each lane copies something this CTA has finished to its CTA `to`, if `wanted` there.  Whoever wrote it arrived on a barrier
  // this warp has waited for (or is this warp); the proxy fence makes those stores visible to the copy.
  auto send = [&](const T* what, const T* where, uint32_t bytes, uint64_t* bar, bool wanted) {
    fence_async_proxy();
    __syncwarp();
    if (wanted) bulk_to_peer(map_to_cta(smem_addr(where), to), smem_addr(what), bytes, map_to_cta(smem_addr(bar), to));
  };
  // kBig: this warp has read all it will of what step k brought here; the last of the CTA's warps to say so tells the peers.
  // Their next copies into the same slots must stay behind these reads, some of which may still be on their way: the count
  // is a release and an acquire, the arrival a release at cluster scope, and the waits for it acquire there.  (A releasing
  // arrival by every warp waits for that warp's output as well: in an earlier form r = 336 / 512 took 42.8 / 71.9 us, 42.0 / 69.6 so.)
  auto done_with = [&](int k) {
    if (!kBig || k + 2 >= nblk) return;
    __syncwarp();
    uint32_t before = 0;
    if (lane == 0)
      asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(before) : "r"(smem_addr(&s_done[k])) : "memory");
    before = __shfl_sync(0xffffffffu, before, 0);
    __syncwarp();
    if (before == kReaders - 1 && peer)
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];"
                   ::"r"(map_to_cta(smem_addr(&free_bar[k]), to)) : "memory");
  };
  // kBig: before the first copy of step k leaves: its set of slots was last used two steps ago
  auto may_send = [&](int k) { if (kBig && k >= 2) bar_wait<true>(&free_bar[k - 2], gave_up); };
  if (!active) {
    // a CTA without a block row (the cluster size is a power of two)
  } else if (role == R_PIVOT) {
    const bool clamped = factor_diagonal<T>(own, panel(me), pan_bar[me], floor_, lane);
    if (kBig && me >= kBigPans) bar_wait<true>(&free_bar[me - kBigPans], gave_up);   // the ring slot is free in every peer
    send(panel(me) + (kPan - 1) * kPanElems, panel(me) + (kPan - 1) * kPanElems, kPanBytes, &pan_bar[me][kPan - 1], peer);
    if (clamped && lane == 0 && p.dev_status) { atomicOr(p.dev_status, LORACT_DEV_PIVOT_CLAMPED); __threadfence(); }
  } else if (role < R_SOLVE) {
    // ---- follow-up warps
    const int w = role - R_FOLLOW;
    const FollowLane<T> f{w, lane};
#pragma unroll 1
    for (int k = -1; k + 1 < nblk; ++k) {
      // step k: the block that step k + 1 works on takes L(own, k) or X(k, own) off, group by group
      const int j = k + 1;
      T* tgt = target(j);
      const bool fresh = j > me && k == me;                 // the first update of an inverse block
      if (j == 0 && me != 0) continue;                      // (the first block of a row needs no update)
      if (k >= 0 && (j <= me ? k >= 1 : k > me)) bar_wait(&bulk_bar[j], gave_up);
      V4<T> acc[2], was[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        acc[h] = was[h] = {{(T)0, (T)0, (T)0, (T)0}};
        if (!fresh) (kBlockSums<T> ? was : acc)[h] = ld4(tgt + f.at(h));
      }
      if (k >= 0) {
        const T* A = solved(k);
        const T* Bm = j == me ? A : slot(j, k);
#pragma unroll 1
        for (int q = 0; q < kPan; ++q) {
          bar_wait(&sol_bar[k][q], gave_up);
          if (j != me) bar_wait(&next_bar[k][q], gave_up);
          take_off_group<T>(acc, A + q * kGrp, Bm + q * kGrp, f);
        }
        done_with(k);
      }
      if (kBlockSums<T>) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[h].v[u] += was[h].v[u];
      }
      if (j != me) {
#pragma unroll
        for (int h = 0; h < 2; ++h) st4(tgt + f.at(h), acc[h]);
        warp_arrive(&rdy_bar[j], lane);
        continue;
      }
      // the diagonal block itself: groups 2 w and 2 w + 1 go to the pivot warp, each when every group but the one before
      // it has been taken off
      if (w == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) st4(own + f.at(h), acc[h]);
        named_arrive(id_staged(0), 64);
        named_arrive(id_staged(1), 64);
      }
      const T* pan = panel(me);
#pragma unroll 1
      for (int g = 0; g < 2 * w; ++g) {
        named_sync(id_published(g), readers_of(g));
        take_off_group<T>(acc, pan, pan, f);
        pan += kPanElems;
        if (g + 2 >= 2 * w) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (f.group(h) == g + 2) st4(own + f.at(h), acc[h]);
          named_arrive(id_staged(g + 2), 64);
        }
      }
    }
  } else if (role < R_BULK) {
    // ---- solver warps: eight rows each
    const int row = 8 * (role - R_SOLVE) + (lane & 7), cg = lane >> 3;
#pragma unroll 1
    for (int k = 0; k < nblk; ++k) {
      T* blk = solved(k);
      V4<T> acc[2], was[2];
      if (k != me) {
        if (k > 0) bar_wait(&rdy_bar[k], gave_up);
#pragma unroll
        for (int h = 0; h < 2; ++h) was[h] = ld4(blk + (cg + 4 * h) * kGrp + row * 4);
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < 4; ++j) was[h].v[j] = 4 * (cg + 4 * h) + j == row ? (T)1 : (T)0;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[h].v[j] = kBlockSums<T> ? (T)0 : was[h].v[j];
      solve_half<T, 0>(was, acc, blk, panel(k), pan_bar[k], sol_bar[k], k >= me, row, lane, gave_up);
      solve_half<T, 1>(was, acc, blk, panel(k), pan_bar[k], sol_bar[k], k >= me, row, lane, gave_up);
      done_with(k);
    }
  } else if (role < R_SEND) {
    // ---- bulk warps: the updates of step k to blocks beyond k + 1, and the output
    const int m = role - R_BULK;
    const int col = me * kB + lane;
    float wdiag = 0.f, est = 0.f;
    if (p.gate_out && col < r) {
      // for the estimate: the diagonal entry of this lane's column, as factored
      const T* parts = (const T*)p.partials;
      T d = (T)0;
#pragma unroll 4
      for (int q = 0; q < p.n_partials; ++q)
        d += __ldg(parts + (int64_t)q * p.partial_stride + (int64_t)col * p.in_ld + col);
      wdiag = (float)(d + d * (T)p.shift_diag_rel + s_shift);
    }
    // zeros above the diagonal block
#pragma unroll 1
    for (int row = m; row < me * kB; row += kBulkWarps) {
      if (col >= r) continue;
      const int64_t o = (int64_t)row * p.out_ld + col;
      if (p.linv_f32) p.linv_f32[o] = 0.f;
      if (p.linv_hi) p.linv_hi[o] = __float2bfloat16(0.f);
      if (p.linv_lo) p.linv_lo[o] = __float2bfloat16(0.f);
    }
#pragma unroll 1
    for (int k = 0; k < nblk; ++k) {
      const T* blk = solved(k);
      const int j_end = k < me ? me + 1 : nblk;
      if (kBig || k + 2 < j_end) bar_wait(&sol_bar[k][kPan - 1], gave_up);
#pragma unroll 1
      for (int j = k + 2; j < j_end; ++j) {
        if (j % (kBulkWarps / 2) != (m >> 1)) continue;        // the same pair of warps for a block in every step
        if (j != me) bar_wait(&off_bar[off_slot(j, k)], gave_up);
        take_off_half<T, (kBig || sizeof(T) == 8) ? 8 : 4>(target(j), blk, j == me ? blk : slot(j, k), k == me, m & 1, lane);
        if (j == k + 2) warp_arrive(&bulk_bar[j], lane);
      }
      done_with(k);
      if (k < me) continue;
#pragma unroll 1
      for (int q = m; q < kPan; q += kBulkWarps) {
        // without updates in front, as in the last step, group by group (kBig: a warp waits for the whole block in any case, as
        // the repeated look at a barrier costs 1 us at r = 512)
        if (!kBig) bar_wait(&sol_bar[k][q], gave_up);
        // rows 32 k + 4 q .. + 3 of the result: element (32 k + 4 q + u, col) = X[group q][lane][u]
        const V4<T> v4 = ld4(blk + q * kGrp + lane * 4);
        const int row = k * kB + 4 * q;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (row + a >= r || col >= r) continue;
          const float v = (float)v4.v[a];
          est = fmaf(v * v, wdiag, est);
          const int64_t o = (int64_t)(row + a) * p.out_ld + col;
          if (p.linv_f32) p.linv_f32[o] = v;
          if (p.linv_hi) {
            const __nv_bfloat16 hi = __float2bfloat16(v);
            p.linv_hi[o] = hi;
            if (p.linv_lo) p.linv_lo[o] = __float2bfloat16(v - __bfloat162float(hi));
          }
        }
        if (kBulkWarps >= kPan) break;
      }
    }
    if (p.gate_out) {
      // this warp's share of the estimate, summed in a fixed order and handed to CTA 0
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) est += __shfl_xor_sync(0xffffffffu, est, o);
      if (kBig && lane == 0)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_to_cta(smem_addr(&s_est[kBulkWarps * me + m]), 0)), "f"(est)
                     : "memory");
      if (!kBig && lane == 0)
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                     ::"r"(map_to_cta(smem_addr(&s_est[kBulkWarps * me + m]), 0)), "r"(__float_as_uint(est)),
                       "r"(map_to_cta(smem_addr(&est_bar), 0))
                     : "memory");
    }
  } else {
    // ---- senders
    const int w = role - R_SEND;
#pragma unroll 1
    for (int k = w; k + 1 < me; k += kSendWarps) {
      bar_wait(&sol_bar[k][kPan - 1], gave_up);
      may_send(k);
      send(solved(k), slot(me, k), kBlkBytes, &off_bar[off_slot(me, k)], peer && (to <= k || to > me));
    }
    if (me > 0) {
#pragma unroll 1
      for (int q = w; q < kPan; q += kSendWarps) {
        bar_wait(&sol_bar[me - 1][q], gave_up);
        may_send(me - 1);
        send(solved(me - 1) + q * kGrp, slot(me, me - 1) + q * kGrp, kGrpBytes, &next_bar[me - 1][q], peer);
      }
    }
    // (every peer is done with what the ring slot of this panel held: a later step has been waited for above)
#pragma unroll 1
    for (int q = w; q + 1 < kPan; q += kSendWarps) {   // (the pivot warp sends the last one itself)
      bar_wait(&pan_bar[me][q], gave_up);
      send(panel(me) + q * kPanElems, panel(me) + q * kPanElems, kPanBytes, &pan_bar[me][q], peer);
    }
  }
  __syncthreads();
  if (s_gave_up) {
    if (tid == 0 && p.dev_status) { atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED); __threadfence(); }
    // what nobody waited for to the end must land before the shared memory goes away
    if (tid < kMaxBlk * kPan) {
      const int k = tid / kPan, q = tid % kPan;
      if (panel_comes(k)) bar_drain(&pan_bar[k][q]);
      if (next_comes(k)) bar_drain(&next_bar[k][q]);
    } else if (tid < kMaxBlk * kPan + kMaxOff) {
      const int b = tid - kMaxBlk * kPan, i = row_of_slot(b);
      if (block_comes(i, b - off_slot(i, 0))) bar_drain(&off_bar[b]);
    }
    __syncthreads();
  }
  // No CTA leaves while another may still write into its shared memory or read its own through a copy.  kBig: the arrivals on
  // other CTAs' free_bar must have been performed as well, hence the releasing form there; elsewhere everything that is written into
  // another CTA is waited for there.
  if (kBig) cluster_arrive(); else cluster_arrive_relaxed();
  cluster_wait();
  if (p.gate_out && me == 0 && warp == 0) {
    // after the cluster barrier every status bit of this call is set (who sets one fences); the shares of the estimate are here (kBig)
    // or counted.  Where that count does not complete, the wait is reported here (the block above is past) and the second round runs.
    const bool here = kBig || __all_sync(0xffffffffu, bar_wait<true>(&est_bar, gave_up));
    if (!here) {
      bar_drain(&est_bar);
      __syncwarp();
      if (lane == 0 && p.dev_status) atomicOr(p.dev_status, LORACT_DEV_WAIT_EXPIRED);
    }
    const uint32_t st = p.dev_status ? *(const volatile uint32_t*)p.dev_status : 0u;
    float est = 0.f;
#pragma unroll 1
    for (int c = lane; c < kBulkWarps * nblk; c += 32) est += s_est[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) est += __shfl_xor_sync(0xffffffffu, est, o);
    if (!here) est = __uint_as_float(0x7fc00000u);          // (not a number: what is in s_est is not the sum)
    const bool again = !(est <= p.gate_threshold) || st != 0u;
    if (lane == 0) {
      p.gate_out[0] = again ? 1u : 0u;
      p.gate_out[1] = __float_as_uint(est);
      p.gate_out[2] = again ? 2u : 1u;
    }
  }
}

// The give-up path of this file's waits, exercised on purpose: a two-CTA cluster in which CTA 1 waits, with
// bar_wait, for bytes that CTA 0 never sends.  After `limit_ns` it records LORACT_DEV_WAIT_EXPIRED and both
// CTAs run to the closing cluster barrier, as the factorisation kernel does.
__global__ void __cluster_dims__(2, 1, 1) cluster_wait_probe_kernel(uint32_t* dev_status, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int gave_up;
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  if (threadIdx.x == 0) {
    bar_init(&bar, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bar_expect(&bar, 16);   // sixteen bytes that never arrive
  }
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  if (rank == 1 && threadIdx.x == 0) bar_wait(&bar, &gave_up, limit_ns);
  __syncthreads();
  if (threadIdx.x == 0 && gave_up && dev_status) atomicOr(dev_status, LORACT_DEV_WAIT_EXPIRED);
  cluster_arrive();
  cluster_wait();
}

// Kernel attributes, once per device.
template <typename T, bool kBig>
cudaError_t configure_cluster(int dev) {
  static std::atomic<bool> configured[64];
  if (dev >= 0 && dev < 64 && configured[dev].load(std::memory_order_acquire)) return cudaSuccess;
  LORACT_CUDA_TRY(cudaFuncSetAttribute(small_block_cluster_kernel<T, kBig>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(smem_elems<T, kBig>(Cfg<T>::kMaxR / kB) * sizeof(T))));
  if (kBig)   // a cluster of sixteen CTAs
    LORACT_CUDA_TRY(cudaFuncSetAttribute(small_block_cluster_kernel<T, kBig>,
                                         cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  if (dev >= 0 && dev < 64) configured[dev].store(true, std::memory_order_release);
  return cudaSuccess;
}

// Whether the device can hold a cluster of sixteen CTAs of the form for many blocks: sixteen SMs of one GPC, one CTA each.
// More than eight CTAs is a size that a device need not provide (a partition of a GPU has fewer SMs to a GPC).
bool big_cluster_resident(int dev) {
  static std::atomic<int> known[64];      // 0: not asked yet, 1: yes, 2: no
  const bool cached = dev >= 0 && dev < 64;
  if (cached && known[dev].load(std::memory_order_acquire)) return known[dev].load(std::memory_order_acquire) == 1;
  int n = 0;
  if (configure_cluster<float, true>(dev) == cudaSuccess) {
    cudaLaunchConfig_t q = {};
    q.gridDim = dim3(kBigBlk, 1, 1);
    q.blockDim = dim3(32 * warps_of<float, true>(), 1, 1);
    q.dynamicSmemBytes = smem_elems<float, true>(kBigBlk) * sizeof(float);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kBigBlk;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    q.attrs = attr;
    q.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, small_block_cluster_kernel<float, true>, &q) != cudaSuccess) n = 0;
  }
  if (n < 1) (void)cudaGetLastError();
  if (cached) known[dev].store(n >= 1 ? 1 : 2, std::memory_order_release);
  return n >= 1;
}

std::atomic<int> g_big_clusters{1};

template <typename T, bool kBig>
cudaError_t launch_cluster(const SCParams& p, cudaStream_t stream) {
  const int nblk = (p.r + kB - 1) / kB;
  int ctas = 1;                           // cluster sizes are powers of two
  while (ctas < nblk) ctas *= 2;
  int dev = 0;
  LORACT_CUDA_TRY(cudaGetDevice(&dev));
  LORACT_CUDA_TRY((configure_cluster<T, kBig>(dev)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, 1, 1);
  cfg.blockDim = dim3(32 * warps_of<T, kBig>(), 1, 1);
  cfg.dynamicSmemBytes = smem_elems<T, kBig>(nblk) * sizeof(T);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LORACT_CUDA_TRY(cudaLaunchKernelEx(&cfg, small_block_cluster_kernel<T, kBig>, p));
  count_launch(__func__, stream);
  return cudaGetLastError();
}

}  // namespace

cudaError_t small_block_cluster_wait_probe_launch(uint32_t* dev_status, uint64_t limit_ns, cudaStream_t stream) {
  cluster_wait_probe_kernel<<<2, 32, 0, stream>>>(dev_status, limit_ns);
  count_launch(__func__, stream);
  return cudaGetLastError();
}

bool small_block_cluster_supported(const SmallBlockArgs& a) {
  if (a.linv_full != nullptr || ((uintptr_t)a.partials & 15) || a.partial_stride % 4 || a.in_ld % 4 || a.r % 4) return false;
  if (a.use_f64) return a.partial_type == ELEM_F64 && a.r <= Cfg<double>::kMaxR;
  return a.partial_type == ELEM_F32 && a.r <= kBigBlk * kB;
}

void small_block_set_big_clusters(int on) { g_big_clusters.store(on); }

bool small_block_cluster_resident(const SmallBlockArgs& a) {
  if (a.use_f64 || a.r <= Cfg<float>::kMaxR) return true;   // up to eight CTAs: a size every device provides
  int dev = 0;
  return g_big_clusters.load() != 0 && cudaGetDevice(&dev) == cudaSuccess && big_cluster_resident(dev);
}

cudaError_t small_block_cluster_launch(const SmallBlockArgs& a, cudaStream_t stream) {
  SCParams p;
  p.r = a.r;
  p.partials = a.partials;
  p.in_ld = a.in_ld ? a.in_ld : a.r;
  p.out_ld = a.out_ld ? a.out_ld : a.r;
  p.n_partials = a.n_partials;
  p.partial_stride = a.partial_stride;
  p.shift_rel = a.shift_rel;
  p.shift_diag_rel = a.shift_diag_rel;
  p.gate = a.gate;
  p.gate_out = a.gate_out;
  p.gate_threshold = a.gate_threshold;
  p.absent_share_bytes = a.absent_share_bytes;
  p.linv_f32 = a.linv_f32;
  p.linv_hi = a.linv_hi;
  p.linv_lo = a.linv_lo;
  p.dev_status = a.dev_status;
  if (a.use_f64) return launch_cluster<double, false>(p, stream);
  return a.r <= Cfg<float>::kMaxR ? launch_cluster<float, false>(p, stream) : launch_cluster<float, true>(p, stream);
}

}  // namespace loract
