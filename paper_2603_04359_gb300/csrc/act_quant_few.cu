// Block transform + per-row absmax + INT4 quantization of a few rows (decode, n <= 32; Sec. 3 Eq. 5, Sec. 6).
//
// A handful of tokens is a chain of latencies on the tensor-core kernel (act_quant_tc.cu): the planes of T, a
// 128-row tile's MMAs, row maxima by global atomics, a fence, a count, a poll, the maxima back, the codes --
// ~9 us whatever the rows.  Here a cluster of up to 16 CTAs takes up to four rows through the whole of T: a CTA has
// d / 16 outputs, every warp streams rows of the float32 T from L2 straight into registers and multiplies them
// with its slice of the token rows, and the row maxima cross the cluster through distributed shared memory, so
// there is no global scratch and one cluster barrier.  The clusters that are resident at once (7 of 16 CTAs, 15
// of 8 on this device) share the rows; every one reads all of T from L2, and that stream bounds the kernel.
// Sums are float32: four products in order per lane, then a tree over the lanes.
// Measured (cat_transform_quantize_act_split, k = 128): 1 x 4096 8.3 -> 5.6 us, 16 x 4096 8.9 -> 5.9.
#include <cstring>

#include "common.cuh"
#include "gemm_pair.cuh"
#include "per_device.h"

namespace cat {
namespace {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kRows = 4;                      // rows per cluster
constexpr int kMaxCluster = 16;
constexpr int kBatch = 8;                     // loads of T in flight per lane

__device__ __forceinline__ void st_cluster_u32(uint32_t* p, uint32_t rank, uint32_t v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(v) : "memory");
}

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xFFFF0000u));
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}

constexpr int64_t kMaxT16 = 1200 * 1024, kMaxT8 = 700 * 1024;   // elements of T for clusters of 16, of 8 and fewer
constexpr size_t kMaxSmem = 40 * 1024;

cudaLaunchAttribute cluster_of(int ctas) {
  cudaLaunchAttribute a;
  memset(&a, 0, sizeof(a));
  a.id = cudaLaunchAttributeClusterDimension;
  a.val.clusterDim.x = (unsigned)ctas;
  a.val.clusterDim.y = a.val.clusterDim.z = 1;
  return a;
}

// Shared memory: V [kRows][outputs of the CTA + 8] floats.
__host__ __device__ constexpr size_t few_smem(int64_t d, int cluster) {
  return (size_t)kRows * ((d / 32 + cluster - 1) / cluster * 32 + 8) * sizeof(float);
}

template <typename Tin, int K>
__global__ void __launch_bounds__(kThreads, 1)
    transform_quant_few_kernel(const Tin* __restrict__ x, int n, int d, const float* __restrict__ T, int rows,
                               uint8_t* __restrict__ codes, int e8, float* __restrict__ scale,
                               uint32_t* __restrict__ status, int cluster) {
  constexpr int LPR = K < 128 ? K / 4 : 32;   // lanes that share an output's inputs
  constexpr int OPL = 32 / LPR;               // outputs per load of T (512 B of it per warp)
  constexpr int OB = kBatch * OPL;            // outputs per batch
  constexpr int H = K > 128 ? K / 128 : 1;    // float4 per lane and output
  constexpr int FV = 32 / LPR;                // sums a lane ends with
  static_assert(kBatch * kRows == 32 && OB <= 32, "a batch's sums: one per lane and load of 32 / LPR");
  extern __shared__ __align__(16) float V[];
  __shared__ uint32_t red[kRows], inbox[kMaxCluster][kRows], fin[kRows];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)(blockIdx.x % cluster);
  const int t0 = (int)(blockIdx.x / cluster) * rows, nr = min(rows, n - t0);
  const int units = d / 32, u0 = rank * units / cluster, u1 = (rank + 1) * units / cluster;
  const int o0 = u0 * 32, no = (u1 - u0) * 32, ld = no + 8;
  if (tid < kRows) red[tid] = 0u;
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // waited for before the first remote store
  pdl_wait_then_release();                    // no global access before this
  __syncthreads();

  uint32_t mx[FV];
#pragma unroll
  for (int i = 0; i < FV; ++i) mx[i] = 0u;
  // float32 rows, as on the SIMT kernels: a NaN has code 0 and no part in the maximum; bf16 rows, as on the
  // tensor-core kernel: it makes all of its row's codes and the step 0
  [[maybe_unused]] bool nan = false;
  const int batches = no / OB;
  const int b0 = warp * batches / kWarps, b1 = (warp + 1) * batches / kWarps;
  int cur = -1;
  float4 xr[kRows][H];
  for (int bt = b0; bt < b1; ++bt) {
    const int ob = o0 + bt * OB;              // the batch's outputs lie in one block
    const float* src = T + (size_t)ob * K + 4 * lane;
    float4 tv[kBatch][H];
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
#pragma unroll
      for (int h = 0; h < H; ++h) tv[q][h] = load4(src + q * (128 * H) + 128 * h);
    if (ob / K != cur) {
      cur = ob / K;
#pragma unroll
      for (int r = 0; r < kRows; ++r)
#pragma unroll
        for (int h = 0; h < H; ++h)
          xr[r][h] = r < nr ? load4(x + (size_t)(t0 + r) * d + cur * K + 4 * (lane % LPR) + 128 * h)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float v[32];                              // index q * kRows + r
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        float s = 0.f;
#pragma unroll
        for (int h = 0; h < H; ++h) s = dot4(tv[q][h], xr[r][h], s);
        v[q * kRows + r] = s;
      }
    // halving butterfly over the LPR lanes: every step adds the other lane's half and keeps half of the sums, the
    // upper half of the index where the lane's bit is set
#pragma unroll
    for (int m = LPR / 2, cnt = 32; m > 0; m >>= 1, cnt >>= 1)
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (i < cnt / 2) {
          const bool up = lane & m;
          const float keep = up ? v[i + cnt / 2] : v[i], send = up ? v[i] : v[i + cnt / 2];
          v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, m);
        }
#pragma unroll
    for (int i = 0; i < FV; ++i) {
      const int idx = (lane % LPR) * FV + i, q = idx / kRows, r = idx % kRows;
      V[r * ld + bt * OB + q * OPL + lane / LPR] = v[i];
      uint32_t u = __float_as_uint(v[i]) & 0x7FFFFFFFu;           // a NaN lies above the infinity
      if (sizeof(Tin) == 4 && u > 0x7F800000u) {
        nan = true;
        u = 0u;
      }
      mx[i] = max(mx[i], u);
    }
  }
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    uint32_t m = 0u;
#pragma unroll
    for (int i = 0; i < FV; ++i)
      if (((lane % LPR) * FV + i) % kRows == r) m = max(m, mx[i]);
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0) atomicMax(&red[r], m);
  }
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // the peers run
  if (tid < cluster * kRows) st_cluster_u32(&inbox[rank][tid % kRows], (uint32_t)(tid / kRows), red[tid % kRows]);
  __syncwarp();
  cluster_sync();
  if (tid < kRows) {
    uint32_t m = 0u;
    for (int c = 0; c < cluster; ++c) m = max(m, inbox[c][tid]);
    // a maximum that is not finite becomes a NaN: the row's codes and step are 0
    fin[tid] = m < 0x7F800000u ? m : 0x7FFFFFFFu;
  }
  __syncthreads();
  const int words = no / 8;
  for (int w = tid; w < nr * words; w += kThreads) {
    const int r = w / words, i = w % words;
    const QRow qr = qrow_setup(__uint_as_float(fin[r]), 7.0f);
    const float4 a = load4(V + r * ld + 8 * i), b = load4(V + r * ld + 8 * i + 4);
    const float e[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    int q[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) q[j] = qcode_exact(e[j], qr, 7.0f);
    const size_t at = (size_t)(t0 + r) * d + o0 + 8 * i;
    if (e8) {
      uint2 o;
      o.x = e4m3_code_byte(q[0]) | e4m3_code_byte(q[1]) << 8 | e4m3_code_byte(q[2]) << 16 | e4m3_code_byte(q[3]) << 24;
      o.y = e4m3_code_byte(q[4]) | e4m3_code_byte(q[5]) << 8 | e4m3_code_byte(q[6]) << 16 | e4m3_code_byte(q[7]) << 24;
      *reinterpret_cast<uint2*>(codes + at) = o;
    } else {
      *reinterpret_cast<uint32_t*>(codes + at / 2) = sm4_pack(q);
    }
  }
  if (nan) report(status, kStatusNonFinite);
  if (rank == 0 && tid < nr) {
    const float a = __uint_as_float(fin[tid]);
    float s = 0.f;
    if (isfinite(a))
      s = __fdiv_rn(a, 7.0f);
    else
      report(status, kStatusNonFinite);
    scale[t0 + tid] = s;
  }
}

// Clusters of 1, 2, 4, 8 and 16 CTAs that are resident at once (asked once per device and kernel; 16 is opt-in).
struct Resident {
  int of[5];
};
template <typename Tin, int K>
Resident resident() {
  static PerDevice<Resident> asked;
  return asked.get([] {
    Resident r = {{0, 0, 0, 0, 0}};
    auto kernel = transform_quant_few_kernel<Tin, K>;
    const bool wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int i = 0; i < (wide ? 5 : 4); ++i) {
      cudaLaunchConfig_t cfg;
      memset(&cfg, 0, sizeof(cfg));
      cfg.gridDim = dim3(1u << i, 1, 1);
      cfg.blockDim = dim3(kThreads, 1, 1);
      cfg.dynamicSmemBytes = kMaxSmem;
      cudaLaunchAttribute attr = cluster_of(1 << i);
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&r.of[i], kernel, &cfg) != cudaSuccess) r.of[i] = 0;
    }
    cudaGetLastError();
    return r;
  });
}

// The largest cluster that leaves each CTA 128 outputs and takes the rows in one wave, while streaming T through it
// is faster than the tensor-core kernel's ~9 us: with 16 CTAs 3.7 us + 4.0 per 2^20 elements of T (measured at
// 4096 and 14336 channels, k = 128), with 8 4.1 + 7.2.
template <typename Tin, int K>
cudaError_t launch_k(const Tin* x, int64_t n, int64_t d, const float* T, uint8_t* codes, int e8, float* scale,
                     uint32_t* status, cudaStream_t stream) {
  auto kernel = transform_quant_few_kernel<Tin, K>;
  const Resident res = resident<Tin, K>();
  int i = 4;
  while (i > 0 && d < 128 << i) --i;
  const int64_t most[5] = {kMaxT8, kMaxT8, kMaxT8, kMaxT8, kMaxT16};
  for (;; --i) {
    if (i < 0 || d * K > most[i]) return cudaErrorNotSupported;
    if (n <= (int64_t)kRows * res.of[i]) break;
  }
  const int cluster = 1 << i;
  const size_t smem = few_smem(d, cluster);
  if (smem > kMaxSmem) return cudaErrorNotSupported;
  const int rows = (int)((n + res.of[i] - 1) / res.of[i]);
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)((n + rows - 1) / rows * cluster), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr = cluster_of(cluster);
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kernel, x, (int)n, (int)d, T, rows, codes, e8, scale, status, cluster);
}

template <typename Tin>
cudaError_t launch_t(const Tin* x, int64_t n, int64_t d, int k, const float* T, uint8_t* codes, int e8, float* scale,
                     uint32_t* status, cudaStream_t stream) {
  switch (k) {
    case 32: return launch_k<Tin, 32>(x, n, d, T, codes, e8, scale, status, stream);
    case 64: return launch_k<Tin, 64>(x, n, d, T, codes, e8, scale, status, stream);
    case 128: return launch_k<Tin, 128>(x, n, d, T, codes, e8, scale, status, stream);
    case 256: return launch_k<Tin, 256>(x, n, d, T, codes, e8, scale, status, stream);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace

// A few rows (n <= 32), k in 32..256, T as launch_k's rule bounds it; cudaErrorNotSupported (nothing launched)
// otherwise.  e8: one code per byte, else SM4x8 words.
cudaError_t launch_transform_quantize_few(const void* x, int dtype, int64_t n, int64_t d, int k, const float* T,
                                          uint8_t* codes, int e8, float* scale, uint32_t* status, cudaStream_t stream) {
  if (n < 1 || n > 32 || d % 32 != 0) return cudaErrorNotSupported;
  if (dtype == 0) return launch_t(static_cast<const float*>(x), n, d, k, T, codes, e8, scale, status, stream);
  return launch_t(static_cast<const __nv_bfloat16*>(x), n, d, k, T, codes, e8, scale, status, stream);
}

}  // namespace cat
