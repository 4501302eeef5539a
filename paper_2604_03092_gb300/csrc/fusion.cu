// Accumulation gate of map fusion (Sec. 4.3, "Map Fusion": new primitives
// are added only where the global map does not yet reconstruct the frame,
// found by rendering its accumulation map and comparing with a threshold).
//
// The accumulation map is the forward's alpha output A = 1 - T_final at the
// new keyframe's pose; the frame's new primitives are per pixel, so the gate
// is an ordered stream compaction: keep_idx lists, in ascending order, the
// pixels with A < tau.  Two chained launches: per-block counts, and a scatter
// in which each block adds up the counts before its own and ranks its kept
// pixels with warp ballots.  (Far too many blocks for that take a scan of the
// counts in between.)
#include <cuda_runtime.h>

#include "splat2d_internal.cuh"

namespace s2d {

constexpr int GATE_THREADS = 256;
constexpr int GATE_PER_THREAD = 4;
constexpr int GATE_TILE = GATE_THREADS * GATE_PER_THREAD;  // pixels per block

__device__ __forceinline__ bool gate_keep(const float* alpha, int64_t i, int64_t n, float tau) {
  return i < n && alpha[i] < tau;  // false for NaN
}

// Up to this many blocks, each adds up the counts before its own (at most 16
// loads a thread, under the scatter's own loads); a scan of them by one block
// in a launch of its own is 2.9 us for 200 or 300 blocks.
constexpr int64_t SUM_BLOCKS = 4096;

// The counts before this block's: its thread's part of them, or all of them
// (thread 0) where they have been scanned.
template <int THREADS>
__device__ __forceinline__ uint32_t counts_before(const uint32_t* __restrict__ count, bool scanned) {
  if (scanned) return threadIdx.x == 0 ? count[blockIdx.x] : 0u;
  uint32_t c = 0;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += THREADS) c += count[i];
  return c;
}

__global__ void __launch_bounds__(GATE_THREADS) k_gate_count(const float* __restrict__ alpha, int64_t n, float tau,
                                                             uint32_t* __restrict__ block_count) {
  chain_release();
  chain_wait();
  __shared__ uint32_t s_w[GATE_THREADS / 32];
  const int64_t base = (int64_t)blockIdx.x * GATE_TILE;
  uint32_t c = 0;
#pragma unroll
  for (int k = 0; k < GATE_PER_THREAD; k++) c += gate_keep(alpha, base + k * GATE_THREADS + threadIdx.x, n, tau);
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < GATE_THREADS / 32; w++) t += s_w[w];
    block_count[blockIdx.x] = t;
  }
}

// One block: exclusive scan of the block counts in place; the total goes to *n_keep.
__global__ void __launch_bounds__(1024) k_gate_scan(uint32_t* __restrict__ block_count, int64_t nb,
                                                    int64_t* __restrict__ n_keep) {
  chain_release();
  chain_wait();
  __shared__ unsigned long long s_w[32];
  __shared__ unsigned long long s_carry;
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t b0 = 0; b0 < nb; b0 += 1024) {
    const int64_t i = b0 + threadIdx.x;
    const unsigned long long v = i < nb ? block_count[i] : 0ull;
    unsigned long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    if (wid == 0) {
      unsigned long long w = s_w[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      s_w[lane] = w;
    }
    __syncthreads();
    const unsigned long long incl = x + (wid > 0 ? s_w[wid - 1] : 0ull) + s_carry;
    if (i < nb) block_count[i] = (uint32_t)(incl - v);
    __syncthreads();
    if (threadIdx.x == 1023) s_carry = incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) *n_keep = (int64_t)s_carry;
}

__global__ void __launch_bounds__(GATE_THREADS) k_gate_scatter(const float* __restrict__ alpha, int64_t n, float tau,
                                                               const uint32_t* __restrict__ count, bool scanned,
                                                               uint32_t* __restrict__ keep_idx,
                                                               int64_t* __restrict__ n_keep) {
  constexpr int NW = GATE_THREADS / 32;
  static_assert(GATE_PER_THREAD * NW == 32, "a lane per (round, warp)");
  __shared__ uint32_t s_kept[32], s_before[NW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const int64_t base = (int64_t)blockIdx.x * GATE_TILE;
  chain_release();
  chain_wait();
  // rounds of GATE_THREADS consecutive pixels keep the output in ascending order
  uint32_t m[GATE_PER_THREAD];
#pragma unroll
  for (int k = 0; k < GATE_PER_THREAD; k++)
    m[k] = gate_keep(alpha, base + k * GATE_THREADS + threadIdx.x, n, tau) ? 1u : 0u;
  const uint32_t part = __reduce_add_sync(0xffffffffu, counts_before<GATE_THREADS>(count, scanned));
  if (lane == 0) s_before[wid] = part;
#pragma unroll
  for (int k = 0; k < GATE_PER_THREAD; k++) {
    m[k] = __ballot_sync(0xffffffffu, m[k]);
    if (lane == 0) s_kept[k * NW + wid] = __popc(m[k]);
  }
  __syncthreads();
  uint32_t start = 0;
#pragma unroll
  for (int w = 0; w < NW; w++) start += s_before[w];
  const uint32_t c = s_kept[lane];
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (!scanned && blockIdx.x == gridDim.x - 1 && threadIdx.x == GATE_THREADS - 1) *n_keep = (int64_t)start + x;
#pragma unroll
  for (int k = 0; k < GATE_PER_THREAD; k++) {
    const uint32_t before = start + __shfl_sync(0xffffffffu, x - c, k * NW + wid);
    if ((m[k] >> lane) & 1u)
      keep_idx[before + __popc(m[k] & lt)] = (uint32_t)(base + k * GATE_THREADS + threadIdx.x);
  }
}

size_t accum_gate_tmp_size(int64_t n) {
  const int64_t nb = (n + GATE_TILE - 1) / GATE_TILE;
  return sizeof(uint32_t) * (size_t)(nb > 0 ? nb : 1);
}

cudaError_t launch_accum_gate(const float* alpha, int64_t n, float tau, uint32_t* keep_idx, int64_t* n_keep,
                              void* tmp, cudaStream_t st) {
  const int64_t nb = (n + GATE_TILE - 1) / GATE_TILE;
  if (nb == 0) return cudaMemsetAsync(n_keep, 0, sizeof(int64_t), st);
  uint32_t* counts = static_cast<uint32_t*>(tmp);
  cudaError_t e = launch_chained(k_gate_count, (int)nb, GATE_THREADS, 0, st, alpha, n, tau, counts);
  if (e != cudaSuccess) return e;
  const bool scanned = nb > SUM_BLOCKS;
  if (scanned && (e = launch_chained(k_gate_scan, 1, 1024, 0, st, counts, nb, n_keep)) != cudaSuccess) return e;
  return launch_chained(k_gate_scatter, (int)nb, GATE_THREADS, 0, st, alpha, n, tau, counts, scanned, keep_idx,
                        n_keep);
}

// ---------------------------------------------------------------------------
// Adaptive voxelization (Sec. 4.3, "Adaptive Voxelization"): a keyframe's
// per-pixel map (primitive y * W + x) is cut into 2x2 blocks; each block
// becomes one primitive whose center, opacity, colour and scales are the
// block means and whose rotation is the normalised sum of its quaternions,
// each first turned to the hemisphere of the block's first one, unless the
// block's depth variation (largest minus smallest camera-frame depth of its
// primitives) exceeds tau_d, in which case its primitives are kept.  Output
// is ordered: blocks in row-major order, a kept block's primitives in
// row-major order.  One thread per block; the same count and scatter scheme
// as the gate.
// ---------------------------------------------------------------------------
constexpr int VOX_THREADS = 256;

struct VoxIn {
  const float *means, *scales, *quats, *opacity, *rgb;
  int32_t W, H, bw;
  int64_t nb;
  float tau_d;
};

struct VoxOut {
  float *means, *scales, *quats, *opacity, *rgb;
  int32_t* block;
};

// The four places of block b (row-major): their indices, which of them lie in
// the image (the others' index is the first one's), and whether the block
// merges.
struct VoxBlock {
  int64_t idx[4];
  bool in[4];
  int n;
  __device__ __forceinline__ VoxBlock(const VoxIn& I, int64_t b) {
    const int x = 2 * (int)(b % I.bw), y = 2 * (int)(b / I.bw);
    const int64_t first = (int64_t)y * I.W + x;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      in[k] = x + (k & 1) < I.W && y + (k >> 1) < I.H;
      idx[k] = in[k] ? first + (k & 1) + (int64_t)(k >> 1) * I.W : first;
    }
    n = 1 + in[1] + in[2] + in[3];
  }
  __device__ __forceinline__ bool merges(const float (&z)[4], float tau_d) const {
    float zmin = z[0], zmax = z[0];
#pragma unroll
    for (int k = 1; k < 4; k++)
      if (in[k]) {
        zmin = fminf(zmin, z[k]);
        zmax = fmaxf(zmax, z[k]);
      }
    return !(zmax - zmin > tau_d);
  }
};

__global__ void __launch_bounds__(VOX_THREADS) k_vox_count(const VoxIn I, uint32_t* __restrict__ block_count) {
  __shared__ uint32_t s_w[VOX_THREADS / 32];
  const int64_t b = (int64_t)blockIdx.x * VOX_THREADS + threadIdx.x;
  chain_release();
  chain_wait();
  uint32_t c = 0;
  if (b < I.nb) {
    const VoxBlock B(I, b);
    float z[4];
#pragma unroll
    for (int k = 0; k < 4; k++) z[k] = I.means[3 * B.idx[k] + 2];
    c = B.merges(z, I.tau_d) ? 1u : (uint32_t)B.n;
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < VOX_THREADS / 32; w++) t += s_w[w];
    block_count[blockIdx.x] = t;
  }
}

// Latency-bound (some 320 blocks per SM for a 512x384 keyframe): all 52 floats
// of a block's primitives are read at once, before its place is known.  With a
// loop over the members behind the scan, and the scan of the counts in a launch
// of its own, such a keyframe took 4.1 + 2.8 + 13.6 us (count, scan, scatter);
// now 3.4 + 8.4 us.
__global__ void __launch_bounds__(VOX_THREADS) k_vox_scatter(const VoxIn I, const uint32_t* __restrict__ count,
                                                             bool scanned, const VoxOut O,
                                                             int64_t* __restrict__ n_out) {
  constexpr int NW = VOX_THREADS / 32;
  __shared__ uint32_t s_w[NW], s_before[NW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t b = (int64_t)blockIdx.x * VOX_THREADS + threadIdx.x;
  chain_release();
  chain_wait();
  const VoxBlock B(I, b < I.nb ? b : 0);
  float mu[4][3], sc[4][2], q[4][4], op[4], rgb[4][3];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int64_t i = B.idx[k];
#pragma unroll
    for (int j = 0; j < 3; j++) mu[k][j] = I.means[3 * i + j];
#pragma unroll
    for (int j = 0; j < 2; j++) sc[k][j] = I.scales[2 * i + j];
#pragma unroll
    for (int j = 0; j < 4; j++) q[k][j] = I.quats[4 * i + j];
    op[k] = I.opacity[i];
#pragma unroll
    for (int j = 0; j < 3; j++) rgb[k][j] = I.rgb[3 * i + j];
  }
  const uint32_t part = __reduce_add_sync(0xffffffffu, counts_before<VOX_THREADS>(count, scanned));
  const float z[4] = {mu[0][2], mu[1][2], mu[2][2], mu[3][2]};
  const bool merge = B.merges(z, I.tau_d);
  const uint32_t c = b < I.nb ? (merge ? 1u : (uint32_t)B.n) : 0u;
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) {
    s_w[wid] = x;
    s_before[wid] = part;
  }
  __syncthreads();
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < NW; w++) before += s_before[w] + (w < wid ? s_w[w] : 0u);
  if (!scanned && blockIdx.x == gridDim.x - 1 && threadIdx.x == VOX_THREADS - 1) *n_out = (int64_t)before + x;
  if (b >= I.nb) return;
  int64_t o = (int64_t)before + (x - c);
  auto put = [&](const float (&m)[3], const float (&s2)[2], const float (&r)[4], float a, const float (&col)[3]) {
#pragma unroll
    for (int j = 0; j < 3; j++) O.means[3 * o + j] = m[j];
#pragma unroll
    for (int j = 0; j < 2; j++) O.scales[2 * o + j] = s2[j];
#pragma unroll
    for (int j = 0; j < 4; j++) O.quats[4 * o + j] = r[j];
    O.opacity[o] = a;
#pragma unroll
    for (int j = 0; j < 3; j++) O.rgb[3 * o + j] = col[j];
    if (O.block) O.block[o] = (int32_t)b;
    o++;
  };
  if (!merge) {
#pragma unroll
    for (int k = 0; k < 4; k++)
      if (B.in[k]) put(mu[k], sc[k], q[k], op[k], rgb[k]);
    return;
  }
  const float inv = 1.0f / (float)B.n;
  float m[3] = {0.f, 0.f, 0.f}, s2[2] = {0.f, 0.f}, r[4] = {0.f, 0.f, 0.f, 0.f}, a = 0.f, col[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    if (!B.in[k]) continue;
#pragma unroll
    for (int j = 0; j < 3; j++) m[j] += mu[k][j];
#pragma unroll
    for (int j = 0; j < 2; j++) s2[j] += sc[k][j];
    const float d = q[k][0] * q[0][0] + q[k][1] * q[0][1] + q[k][2] * q[0][2] + q[k][3] * q[0][3];
    const float sg = d >= 0.f ? 1.f : -1.f;  // align to the block's first quaternion
#pragma unroll
    for (int j = 0; j < 4; j++) r[j] += sg * q[k][j];
    a += op[k];
#pragma unroll
    for (int j = 0; j < 3; j++) col[j] += rgb[k][j];
  }
  const float qn = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + r[3] * r[3]);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    m[j] *= inv;
    col[j] *= inv;
  }
#pragma unroll
  for (int j = 0; j < 2; j++) s2[j] *= inv;
#pragma unroll
  for (int j = 0; j < 4; j++) r[j] /= qn;
  put(m, s2, r, a * inv, col);
}

size_t voxelize_tmp_size(int32_t W, int32_t H) {
  const int64_t nb = (int64_t)((W + 1) / 2) * ((H + 1) / 2);
  const int64_t g = (nb + VOX_THREADS - 1) / VOX_THREADS;
  return sizeof(uint32_t) * (size_t)(g > 0 ? g : 1);
}

cudaError_t launch_voxelize(const splat2d_surfels& in, int32_t W, int32_t H, float tau_d,
                            const splat2d_surfel_buffers& out, int32_t* out_block, int64_t* n_out, void* tmp,
                            cudaStream_t st) {
  VoxIn I;
  I.means = in.means; I.scales = in.scales; I.quats = in.quats; I.opacity = in.opacity; I.rgb = in.rgb;
  I.W = W; I.H = H; I.bw = (W + 1) / 2;
  I.nb = (int64_t)I.bw * ((H + 1) / 2);
  I.tau_d = tau_d;
  VoxOut O;
  O.means = out.means; O.scales = out.scales; O.quats = out.quats; O.opacity = out.opacity; O.rgb = out.rgb;
  O.block = out_block;
  if (I.nb == 0) return cudaMemsetAsync(n_out, 0, sizeof(int64_t), st);
  const int64_t g = (I.nb + VOX_THREADS - 1) / VOX_THREADS;
  uint32_t* counts = static_cast<uint32_t*>(tmp);
  cudaError_t e = launch_chained(k_vox_count, (int)g, VOX_THREADS, 0, st, I, counts);
  if (e != cudaSuccess) return e;
  const bool scanned = g > SUM_BLOCKS;
  if (scanned && (e = launch_chained(k_gate_scan, 1, 1024, 0, st, counts, g, n_out)) != cudaSuccess) return e;
  return launch_chained(k_vox_scatter, (int)g, VOX_THREADS, 0, st, I, counts, scanned, O, n_out);
}

// ---------------------------------------------------------------------------
// Sim(3) transforms of primitives ("Map Fusion": camera-to-world insertion,
// mu' = s R mu + t, r' = q r; "Loop Correction of Gaussian Map": a keyframe's
// Delta T = T_new T_old^-1 applied rigidly to its primitives).  Tangent
// scales are multiplied by s (a similarity scales the disks with the map).
// One thread per primitive, in place; transform rows are (qw, qx, qy, qz,
// tx, ty, tz, s), chosen per primitive by `index` (or row 0).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_sim3(int64_t n, float* __restrict__ means, float* __restrict__ quats,
                                              float* __restrict__ scales, const float* __restrict__ sim3,
                                              const int32_t* __restrict__ index) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float* T = sim3 + 8 * (index ? (int64_t)index[i] : 0);
  float qw = T[0], qx = T[1], qy = T[2], qz = T[3];
  const float qn = sqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
  qw /= qn; qx /= qn; qy /= qn; qz /= qn;
  const float s = T[7];
  // rotation matrix of the unit quaternion
  const float R00 = 1.f - 2.f * (qy * qy + qz * qz), R01 = 2.f * (qx * qy - qw * qz), R02 = 2.f * (qx * qz + qw * qy);
  const float R10 = 2.f * (qx * qy + qw * qz), R11 = 1.f - 2.f * (qx * qx + qz * qz), R12 = 2.f * (qy * qz - qw * qx);
  const float R20 = 2.f * (qx * qz - qw * qy), R21 = 2.f * (qy * qz + qw * qx), R22 = 1.f - 2.f * (qx * qx + qy * qy);
  if (means) {
    const float x = means[3 * i], y = means[3 * i + 1], z = means[3 * i + 2];
    means[3 * i + 0] = s * (R00 * x + R01 * y + R02 * z) + T[4];
    means[3 * i + 1] = s * (R10 * x + R11 * y + R12 * z) + T[5];
    means[3 * i + 2] = s * (R20 * x + R21 * y + R22 * z) + T[6];
  }
  if (quats) {
    const float rw = quats[4 * i], rx = quats[4 * i + 1], ry = quats[4 * i + 2], rz = quats[4 * i + 3];
    quats[4 * i + 0] = qw * rw - qx * rx - qy * ry - qz * rz;
    quats[4 * i + 1] = qw * rx + qx * rw + qy * rz - qz * ry;
    quats[4 * i + 2] = qw * ry - qx * rz + qy * rw + qz * rx;
    quats[4 * i + 3] = qw * rz + qx * ry - qy * rx + qz * rw;
  }
  if (scales) {
    scales[2 * i] *= s;
    scales[2 * i + 1] *= s;
  }
}

cudaError_t launch_sim3(int64_t n, float* means, float* quats, float* scales, const float* sim3, const int32_t* index,
                        cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_sim3<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, means, quats, scales, sim3, index);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace s2d
