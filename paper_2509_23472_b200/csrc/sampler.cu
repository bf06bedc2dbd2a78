// Row sampling (the first step of Algorithm 1), the row gather, and the Gaussian test matrix of the RSVD
// comparator.  The generator is Philox4x32-10 (Salmon et al., SC'11), written out here from the
// published round function; it shares no code with the CPU oracle.
#include "common.cuh"

namespace loract {

namespace {

__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1, uint32_t out[4]) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0;
    const uint32_t n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

constexpr int kSamplerThreads = 256;
constexpr int kSamplerMaxRounds = 16384;  // 4M candidates; a permutation of 512 rows needs ~3500
constexpr int kMaxRank = 512;

// Every round draws 256 candidates in stream order; a candidate survives if no equal value
// stands earlier in the stream (in this round or among those accepted before); survivors are appended
// in stream order until `rank` are found.  This is exactly "the first rank distinct values of the
// stream".  "Stands earlier" is decided with a hash table in shared memory that keeps, for every value
// seen, the smallest stream position it occurred at (atomicMin), so the outcome does not depend on the
// order in which threads run.  The table holds every value seen before the last round (fewer than 512) and one
// round of candidates (at most 256), so 2048 slots never fill.
constexpr int kTableSlots = 2048;

struct SamplerShared {
  uint32_t accepted[kMaxRank];
  uint32_t tab_key[kTableSlots];   // value + 1, 0 = empty
  uint32_t tab_pos[kTableSlots];   // smallest stream position of that value
  int warp_alive[kSamplerThreads / 32];
  int count;
};

// The stream's key and counter words, and what is drawn from it.
struct SamplerArgs {
  uint32_t seed_lo, seed_hi, call_lo, call_hi;
  uint32_t n_rows;
  int rank;
};

// Returns how many values were found (`rank`, unless the stream ran out); they are in sh.accepted.
__device__ __forceinline__ int sample_rows(const SamplerArgs& a, SamplerShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < kTableSlots; e += kSamplerThreads) { sh.tab_key[e] = 0u; sh.tab_pos[e] = 0xFFFFFFFFu; }
  if (tid == 0) sh.count = 0;
  __syncthreads();
  for (int round = 0; round < kSamplerMaxRounds; ++round) {
    const int count = sh.count;
    if (count >= a.rank) break;
    const uint32_t i = (uint32_t)round * kSamplerThreads + tid;
    uint32_t w[4];
    philox4x32_10(i >> 2, 0u, a.call_lo, a.call_hi, a.seed_lo, a.seed_hi, w);
    const uint32_t c = __umulhi(w[i & 3u], a.n_rows);
    uint32_t h = (c * 2654435761u) >> 21;   // 11 bits
    bool placed = false;
    for (int probe = 0; probe < kTableSlots; ++probe) {
      const uint32_t prev = atomicCAS(&sh.tab_key[h], 0u, c + 1u);
      if (prev == 0u || prev == c + 1u) { placed = true; break; }
      h = (h + 1u) & (kTableSlots - 1);
    }
    if (placed) atomicMin(&sh.tab_pos[h], i);
    __syncthreads();
    const bool alive = placed && sh.tab_pos[h] == i;
    const uint32_t ballot = __ballot_sync(0xffffffffu, alive);
    if (lane == 0) sh.warp_alive[warp] = __popc(ballot);
    __syncthreads();
    int before = 0, total = 0;
    for (int q = 0; q < kSamplerThreads / 32; ++q) {
      const int v = sh.warp_alive[q];
      before += (q < warp) ? v : 0;
      total += v;
    }
    const int pos = count + before + __popc(ballot & ((1u << lane) - 1u));
    if (alive && pos < a.rank) sh.accepted[pos] = c;
    __syncthreads();
    if (tid == 0) sh.count = min(a.rank, count + total);
    __syncthreads();
  }
  return sh.count;
}

__device__ __forceinline__ int32_t sampled(const SamplerShared& sh, int j, int found) {
  return j < found ? (int32_t)sh.accepted[j] : 0;
}

__global__ void __launch_bounds__(kSamplerThreads)
sample_indices_kernel(SamplerArgs a, int32_t* __restrict__ idx_out, uint32_t* __restrict__ dev_status) {
  __shared__ SamplerShared sh;
  pdl_launch_dependents();
  const int found = sample_rows(a, sh);
  pdl_wait();   // the index array may still be read by the previous call's kernels
  for (int j = threadIdx.x; j < a.rank; j += kSamplerThreads) idx_out[j] = sampled(sh, j, found);
  if (threadIdx.x == 0 && dev_status && found < a.rank) atomicOr(dev_status, LORACT_DEV_SAMPLER_SHORT);
}

// Sampling and gather in one kernel: dst[j, :] = src[idx[j] - row0, :], 16 bytes per thread per step.  `src` holds the rows
// [row0, row0 + n_local) of the whole matrix (one shard of a token-sharded matrix, or all of it); a sampled row that lives
// elsewhere is written as zeros, so that the sum of all shards' results is the gathered matrix.
// Bound by latency (the copy is 0.5 to 11 MB): every CTA draws the same indices for itself, mostly under the tail of the
// previous kernel, instead of waiting for one that does.  The CTAs are small so that they fit beside those of that kernel:
// with 1024 threads, as many candidates a round, the step on 16384 x 4096 at rank 256 took 2 us more; four candidates a
// thread cost up to 5 us (the probes of a warp's slowest lane, four times over).  Against a sampling and a gather kernel, us:
// fp32 512 x 768 at rank 64 112.9 -> 111.4, bf16 4096 x 5120 at rank 64 89.8 -> 88.9, 16384 x 4096 at rank 256 201.6 -> 200.9.
__global__ void __launch_bounds__(kSamplerThreads)
sample_gather_kernel(SamplerArgs a, int32_t* __restrict__ idx_out, uint32_t* __restrict__ dev_status,
                     const uint4* __restrict__ src, int64_t ld_vec, int64_t d_vec, int64_t row0, int64_t n_local,
                     uint4* __restrict__ dst) {
  __shared__ SamplerShared sh;
  const int found = sample_rows(a, sh);
  pdl_wait();
  pdl_launch_dependents();   // (ahead of the sampling, the next kernel's CTAs crowd this one's out: fp32 step 1.5 us)
  if (blockIdx.x == 0) {
    if (idx_out)
      for (int j = threadIdx.x; j < a.rank; j += kSamplerThreads) idx_out[j] = sampled(sh, j, found);
    // first kernel of a call: it also sets the status word (no memset node in front of it)
    if (threadIdx.x == 0) *dev_status = found < a.rank ? LORACT_DEV_SAMPLER_SHORT : 0u;
  }
  const int64_t total = (int64_t)a.rank * d_vec, step = (int64_t)gridDim.x * kSamplerThreads;
  const bool narrow = total < (int64_t)1 << 32;
  constexpr int kAhead = 4;
  for (int64_t e0 = (int64_t)blockIdx.x * kSamplerThreads + threadIdx.x; e0 < total; e0 += kAhead * step) {
    uint4 v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int64_t e = e0 + u * step;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (e >= total) continue;
      const int64_t j = narrow ? (int64_t)((uint32_t)e / (uint32_t)d_vec) : e / d_vec;
      const int64_t row = (int64_t)sampled(sh, (int)j, found) - row0;
      if (row >= 0 && row < n_local) v[u] = __ldg(src + row * ld_vec + (e - j * d_vec));
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (e0 + u * step < total) dst[e0 + u * step] = v[u];
  }
}

// dst[c][j] = z(j * l + c): element e of the normal stream is z_(e mod 4) of Philox block e div 4,
// u = (w0 + 1) / 2^32, v = w1 / 2^32, z0 = sqrt(-2 ln u) cos(2 pi v), z1 = ... sin(2 pi v).
__global__ void gaussian_rows_kernel(uint32_t seed_lo, uint32_t seed_hi, uint32_t call_lo,
                                     uint32_t call_hi, int l, int64_t d, __nv_bfloat16* __restrict__ dst) {
  const int64_t total = (int64_t)l * d;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q * 4 < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    uint32_t w[4];
    philox4x32_10((uint32_t)q, 1u, call_lo, call_hi, seed_lo, seed_hi, w);
    float z[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float u = ((float)w[2 * h] + 1.0f) * 2.3283064365386963e-10f;
      const float v = (float)w[2 * h + 1] * 2.3283064365386963e-10f;
      const float rad = sqrtf(-2.0f * logf(fminf(u, 1.0f)));
      float s, c;
      sincospif(2.0f * v, &s, &c);
      z[2 * h] = rad * c;
      z[2 * h + 1] = rad * s;
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int64_t e = q * 4 + t;
      if (e < total) {
        const int64_t j = e / l;
        const int c = (int)(e - j * l);
        dst[(int64_t)c * d + j] = __float2bfloat16(z[t]);
      }
    }
  }
}

}  // namespace

static SamplerArgs sampler_args(uint64_t seed, uint64_t call_id, uint32_t n_rows, int rank) {
  return {(uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)call_id, (uint32_t)(call_id >> 32), n_rows, rank};
}

cudaError_t sample_indices_launch(uint64_t seed, uint64_t call_id, uint32_t n_rows, int rank, int32_t* idx_dev,
                                  uint32_t* dev_status, cudaStream_t stream) {
  LORACT_CUDA_TRY(launch_pdl(sample_indices_kernel, dim3(1), dim3(kSamplerThreads), 0, stream,
                             sampler_args(seed, call_id, n_rows, rank), idx_dev, dev_status));
  count_launch(__func__, stream);
  return cudaGetLastError();
}

cudaError_t sample_gather_launch(uint64_t seed, uint64_t call_id, uint32_t n_rows, int rank, int32_t* idx_out,
                                 uint32_t* dev_status, const void* src, int64_t ld, int64_t d, int elem_bytes, int64_t row0,
                                 int64_t n_local, void* dst, cudaStream_t stream) {
  const int64_t per_vec = 16 / elem_bytes, d_vec = d / per_vec;
  const int64_t ctas = ((int64_t)rank * d_vec + kSamplerThreads - 1) / kSamplerThreads;
  const int grid = ctas > 4 * 148 ? 4 * 148 : (int)ctas;
  LORACT_CUDA_TRY(launch_pdl(sample_gather_kernel, dim3(grid), dim3(kSamplerThreads), 0, stream,
                             sampler_args(seed, call_id, n_rows, rank), idx_out, dev_status, (const uint4*)src, ld / per_vec,
                             d_vec, row0, n_local, (uint4*)dst));
  count_launch(__func__, stream);
  return cudaGetLastError();
}

cudaError_t gaussian_rows_launch(uint64_t seed, uint64_t call_id, int l, int64_t d,
                                 __nv_bfloat16* dst, cudaStream_t stream) {
  const int64_t blocks4 = ((int64_t)l * d + 3) / 4;
  int grid = (int)((blocks4 + 255) / 256);
  if (grid > 148 * 8) grid = 148 * 8;
  gaussian_rows_kernel<<<grid, 256, 0, stream>>>((uint32_t)seed, (uint32_t)(seed >> 32),
                                                 (uint32_t)call_id, (uint32_t)(call_id >> 32), l, d,
                                                 dst);
  count_launch(__func__, stream);
  return cudaGetLastError();
}

}  // namespace loract
