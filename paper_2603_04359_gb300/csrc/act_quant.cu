// Block transform + per-row absmax + symmetric INT4 quantization + SM4x8 packing.
//
//   v'_{t,b} = A_b v_{t,b}             for every row t and k x k block b
//   s_t      = max_i |v'_{t,i}| / 7    (Lemma 2 symmetric range r = 2 max|v|; grid step r / 14)
//   q_{t,i}  = clamp(rint(v'_{t,i} * 7 / max|v'_t|), -7, 7)       (round half to even)
//
// Activations (Sec. 3, Eq. 5: x' = T x, quantized per token, Sec. 6) use A_b = T_b; weight rows
// (W' = W T^{-1}, quantized per output channel) use A_b = (T_b^{-1})^T.
//
// The row maximum spans every block of the row while a CTA holds one block, so the work runs in
// two passes over the same tiles: pass 0 folds per-row maxima into the scale buffer with integer
// atomicMax on the (non-negative) float bits; pass 1 recomputes the tile, quantizes and packs;
// a last pass turns the maxima into steps.  No scratch memory is used.
//
// Tile: 64 rows x OC output channels of one block (OC = min(k, 128)), the block slab A_b[c0:c0+OC, :]
// and the 64 input rows are staged transposed in shared memory; each thread owns 4 rows x 8
// consecutive channels (32 fp32 accumulators), which is exactly one packed word per row.
//
// Small transforms (transform_quant_rows_kernel): where T has few blocks, a CTA takes 16 whole rows through every
// block, so the row maximum never leaves it: one launch and one pass instead of a memset, two passes and a
// finalize launch, with the same sums in the same order.  512 float32 rows of 256 channels at k = 32: 19 us
// and four launches before, 8.6 us now.
#include "common.cuh"

namespace cat {
namespace {

constexpr int kRows = 64;

template <int K>
struct ActCfg {
  static constexpr int OC = K < 128 ? K : 128;         // output channels per CTA
  static constexpr int THREADS = 2 * OC;               // 16 row groups x OC/8 channel groups
  static constexpr int AS_LD = OC + 4;                 // padded row of the transposed slab
  static constexpr int XS_LD = kRows + 4;              // padded row of the transposed inputs
  static constexpr size_t SMEM = (size_t)(K * AS_LD + K * XS_LD) * sizeof(float);
};

// Eight codes as bytes.
__device__ __forceinline__ uint2 code_bytes(const int (&q)[8]) {
  return make_uint2(
      e4m3_code_byte(q[0]) | e4m3_code_byte(q[1]) << 8 | e4m3_code_byte(q[2]) << 16 | e4m3_code_byte(q[3]) << 24,
      e4m3_code_byte(q[4]) | e4m3_code_byte(q[5]) << 8 | e4m3_code_byte(q[6]) << 16 | e4m3_code_byte(q[7]) << 24);
}

// PASS 0: the maxima; 1: the codes as SM4x8 words; 2: as bytes.
template <typename Tin, int K, int PASS>
__global__ void __launch_bounds__(ActCfg<K>::THREADS) transform_quant_kernel(
    const Tin* __restrict__ x, int64_t n, int64_t d, const float* __restrict__ A, uint32_t* __restrict__ amax_bits,
    uint32_t* __restrict__ codes, uint32_t* __restrict__ status) {
  using C = ActCfg<K>;
  extern __shared__ __align__(16) float smem[];
  float* As = smem;                    // [K][AS_LD]: As[j][i] = A_b[c0 + i][j]
  float* xs = smem + K * C::AS_LD;     // [K][XS_LD]: xs[j][r] = x[t0 + r][b*K + j]
  __shared__ uint32_t red[kRows];

  const int slabs = K / C::OC;
  const int b = blockIdx.y / slabs;
  const int c0 = (blockIdx.y % slabs) * C::OC;
  const int64_t t0 = (int64_t)blockIdx.x * kRows;
  const int tid = threadIdx.x;
  const int tg = tid & 15;   // rows 4*tg .. 4*tg+3
  const int cg = tid >> 4;   // channels c0 + 8*cg .. +7

  // Stage the slab transposed.
  const float* Ab = A + (size_t)b * K * K;
  for (int e = tid; e < C::OC * K; e += C::THREADS) {
    const int i = e / K, j = e % K;
    As[j * C::AS_LD + i] = Ab[(size_t)(c0 + i) * K + j];
  }
  // Stage the input rows transposed (rows past n read as zero).
  for (int e = tid; e < kRows * K; e += C::THREADS) {
    const int r = e / K, j = e % K;
    const int64_t t = t0 + r;
    xs[j * C::XS_LD + r] = (t < n) ? to_f32(x[t * d + (int64_t)b * K + j]) : 0.f;
  }
  if (PASS == 0)
    for (int r = tid; r < kRows; r += C::THREADS) red[r] = 0u;
  __syncthreads();

  float acc[4][8];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;

#pragma unroll 4
  for (int j = 0; j < K; ++j) {
    const float4 xv = *reinterpret_cast<const float4*>(&xs[j * C::XS_LD + 4 * tg]);
    const float4 a0 = *reinterpret_cast<const float4*>(&As[j * C::AS_LD + 8 * cg]);
    const float4 a1 = *reinterpret_cast<const float4*>(&As[j * C::AS_LD + 8 * cg + 4]);
    const float xr[4] = {xv.x, xv.y, xv.z, xv.w};
    const float ac[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(ac[c], xr[r], acc[r][c]);
  }

  if (PASS == 0) {
    bool finite = true;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float m = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        finite &= isfinite(acc[r][c]);
        m = fmaxf(m, fabsf(acc[r][c]));
      }
      atomicMax(&red[4 * tg + r], __float_as_uint(m));
    }
    if (!finite) report(status, kStatusNonFinite);
    __syncthreads();
    for (int r = tid; r < kRows; r += C::THREADS)
      if (t0 + r < n) atomicMax(&amax_bits[t0 + r], red[r]);
  } else {
    const int64_t words_per_row = d / 8;               // eight codes: one word, or two of bytes
    const int64_t word = ((int64_t)b * K + c0 + 8 * cg) / 8;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t t = t0 + 4 * tg + r;
      if (t >= n) continue;
      const QRow qr = qrow_setup(__uint_as_float(amax_bits[t]), 7.0f);
      int q[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) q[c] = qcode_exact(acc[r][c], qr, 7.0f);
      if constexpr (PASS == 1)
        codes[t * words_per_row + word] = sm4_pack(q);
      else
        reinterpret_cast<uint2*>(codes)[t * words_per_row + word] = code_bytes(q);
    }
  }
}

// ---- small transforms: 16 whole rows per CTA -------------------------------------------------
// Thread: output channel c of a slab, RPT rows.  The rows lie in shared memory, all loaded at the start, and a
// block's x' replaces its x there; the transposed slabs of A arrive by cp.async one ahead (two buffers), so a
// block costs its sums and two barriers, not a trip to L2.
// Every CTA reads all of A (from L2) and goes through it one block after the other: small A only (rows_pay).
constexpr int kWholeRows = 16;
constexpr int kRowsThreads = 256;
constexpr size_t kRowsMaxSmem = 220 * 1024;

template <int K>
struct RowsCfg {
  static constexpr int OC = K < 128 ? K : 128, SLABS = K / OC;
  static constexpr int AS_LD = OC + 1;
  static constexpr int BUFS = K <= 128 ? 2 : 1;                   // two slabs of 256 inputs would not fit
  static constexpr int RPT = kWholeRows * OC / kRowsThreads;      // rows per thread
  static constexpr size_t smem(int64_t d) {
    return (size_t)kWholeRows * (d + 4) * sizeof(float) + (size_t)BUFS * K * AS_LD * sizeof(float);
  }
};

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

template <typename Tin, int K>
__global__ void __launch_bounds__(kRowsThreads) transform_quant_rows_kernel(
    const Tin* __restrict__ x, int64_t n, int d, const float* __restrict__ A, uint8_t* __restrict__ codes, int e8,
    float* __restrict__ scale, uint32_t* __restrict__ status) {
  using C = RowsCfg<K>;
  extern __shared__ __align__(16) float smem[];
  float* V = smem;                                   // [16][d + 4]: x, then x'
  float* As = V + kWholeRows * (d + 4);              // BUFS x [K][AS_LD], transposed slabs
  __shared__ uint32_t red[kWholeRows];
  const int tid = threadIdx.x, c = tid % C::OC, r0 = tid / C::OC * C::RPT, ld = d + 4;
  const int64_t t0 = (int64_t)blockIdx.x * kWholeRows;
  const int slabs = d / K * C::SLABS;
  auto load_slab = [&](int s) {                      // slab s: rows s OC .. of the stacked blocks
    float* dst = As + (s % C::BUFS) * K * C::AS_LD;
    const float* src = A + (size_t)s * C::OC * K;
    for (int e = tid; e < C::OC * K; e += kRowsThreads) cp_async4(dst + e % K * C::AS_LD + e / K, src + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  load_slab(0);
  if (tid < kWholeRows) red[tid] = 0u;
  for (int e = tid; e < kWholeRows * d; e += kRowsThreads) {
    const int r = e / d, j = e % d;
    V[r * ld + j] = (t0 + r < n) ? to_f32(x[t0 * d + e]) : 0.f;   // rows past n read as zero
  }
  bool finite = true;
  float m[C::RPT];
#pragma unroll
  for (int r = 0; r < C::RPT; ++r) m[r] = 0.f;
  for (int b = 0; b < d / K; ++b) {
    float acc[C::SLABS][C::RPT];
#pragma unroll
    for (int h = 0; h < C::SLABS; ++h) {
      const int s = b * C::SLABS + h;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();                               // slab s (and at first the rows) are in; the slab before is done with
      if (C::BUFS == 2 && s + 1 < slabs) load_slab(s + 1);
      const float* a = As + (s % C::BUFS) * K * C::AS_LD + c;
      const float* v = V + r0 * ld + b * K;
#pragma unroll
      for (int r = 0; r < C::RPT; ++r) acc[h][r] = 0.f;
#pragma unroll 4
      for (int j = 0; j < K; j += 4) {
        const float a0 = a[j * C::AS_LD], a1 = a[(j + 1) * C::AS_LD], a2 = a[(j + 2) * C::AS_LD], a3 = a[(j + 3) * C::AS_LD];
#pragma unroll
        for (int r = 0; r < C::RPT; ++r) {           // inputs in ascending order, as the tiled kernels add them
          const float4 xv = *reinterpret_cast<const float4*>(v + r * ld + j);
          acc[h][r] = fmaf(a3, xv.w, fmaf(a2, xv.z, fmaf(a1, xv.y, fmaf(a0, xv.x, acc[h][r]))));
        }
      }
      if (C::BUFS == 1) {
        __syncthreads();
        if (s + 1 < slabs) load_slab(s + 1);
      }
    }
    __syncthreads();                                 // the block's x has been read
#pragma unroll
    for (int h = 0; h < C::SLABS; ++h)
#pragma unroll
      for (int r = 0; r < C::RPT; ++r) {
        finite &= isfinite(acc[h][r]);
        m[r] = fmaxf(m[r], fabsf(acc[h][r]));
        V[(r0 + r) * ld + b * K + h * C::OC + c] = acc[h][r];
      }
  }
#pragma unroll
  for (int r = 0; r < C::RPT; ++r) atomicMax(&red[r0 + r], __float_as_uint(m[r]));
  if (!finite) report(status, kStatusNonFinite);
  __syncthreads();
  for (int w = tid; w < kWholeRows * (d / 8); w += kRowsThreads) {
    const int r = w / (d / 8), i = w % (d / 8);
    if (t0 + r >= n) break;                          // rows ascend with w
    const QRow qr = qrow_setup(__uint_as_float(red[r]), 7.0f);
    const float4 v0 = *reinterpret_cast<const float4*>(V + r * ld + 8 * i);
    const float4 v1 = *reinterpret_cast<const float4*>(V + r * ld + 8 * i + 4);
    const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    int q[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) q[e] = qcode_exact(v[e], qr, 7.0f);
    if (e8) {
      *reinterpret_cast<uint2*>(codes + (t0 + r) * d + 8 * i) = code_bytes(q);
    } else {
      *reinterpret_cast<uint32_t*>(codes + (t0 + r) * (d / 2) + 4 * i) = sm4_pack(q);
    }
  }
  if (tid < kWholeRows && t0 + tid < n) {
    const float a = __uint_as_float(red[tid]);
    float s = 0.f;
    if (isfinite(a))
      s = __fdiv_rn(a, 7.0f);
    else
      report(status, kStatusNonFinite);
    scale[t0 + tid] = s;
  }
}

// Where whole rows are faster than the tiled kernels (a memset, two passes and a launch for the steps).  A CTA takes
// ~7 us and per block 0.66, 1.0, 2.2, 6.3 us at k = 16, 32, 64, 128 (whatever the other CTAs do, while each has an SM);
// the tiled kernels take 24, 30, 28, 40 us up to ~150 tiles of 64 rows and one block, then as their sums.  us, whole
// rows against tiled, 304 / 2432 / 16384 rows of float32:
//   k = 16:  384 channels 23/26 23/28 42/50,  512 28/25 28/28 54/56, 3072 132/28 137/52 669/276
//   k = 32:  512 channels 24/34 24/36 64/73,  640 29/33 28/36 80/91,  768 33/33 33/37 103/99, 1760 65/34 66/45 411/214
//   k = 64:  512 channels 25/30 26/34 89/98,  640 30/30 30/36 110/107, 768 34/30 35/36 149/129
//   k = 128: every block costs a wave of CTAs (140 KB and more of shared memory, one per SM): 128 channels 14/42 15/42
//            60/54 (7 waves), 512 33/43 34/44 185/167;  at 4864 rows (two waves) 256 channels 35/46, 512 58/54
//   k = 256: 256 channels 30/70 30/69 162/212
bool rows_pay(int k, int64_t blocks, int64_t ctas, int64_t sms) {
  switch (k) {
    case 16: return blocks <= 24;
    case 32: return blocks <= 18 || (blocks <= 24 && ctas <= sms);
    case 64: return blocks <= 8 || (blocks <= 10 && ctas <= sms);
    case 128: return (ctas + sms - 1) / sms * blocks <= 6 && blocks <= 4;
    default: return blocks == 1;
  }
}

int num_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
  return sms;
}

template <typename Tin, int K>
cudaError_t launch_rows_k(const Tin* x, int64_t n, int64_t d, const float* A, uint8_t* codes, int e8, float* scale,
                          uint32_t* status, cudaStream_t stream) {
  const size_t smem = RowsCfg<K>::smem(d);
  const int64_t ctas = (n + kWholeRows - 1) / kWholeRows;
  if (!rows_pay(K, d / K, ctas, num_sms()) || smem > kRowsMaxSmem || ctas > 0x7FFFFFFF) return cudaErrorNotSupported;
  // always the same limit: calls from other threads may set it in between
  cudaError_t e = cudaFuncSetAttribute(transform_quant_rows_kernel<Tin, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kRowsMaxSmem);
  if (e != cudaSuccess) return e;
  note_launch();
  transform_quant_rows_kernel<Tin, K><<<(unsigned)ctas, kRowsThreads, smem, stream>>>(x, n, (int)d, A, codes, e8, scale,
                                                                                    status);
  return cudaGetLastError();
}

// cudaErrorNotSupported (nothing launched): T or the rows are too large, the tiled kernels take the call.
template <typename Tin>
cudaError_t launch_rows(const Tin* x, int64_t n, int64_t d, int k, const float* A, uint8_t* codes, int e8, float* scale,
                        uint32_t* status, cudaStream_t stream) {
  switch (k) {
    case 16: return launch_rows_k<Tin, 16>(x, n, d, A, codes, e8, scale, status, stream);
    case 32: return launch_rows_k<Tin, 32>(x, n, d, A, codes, e8, scale, status, stream);
    case 64: return launch_rows_k<Tin, 64>(x, n, d, A, codes, e8, scale, status, stream);
    case 128: return launch_rows_k<Tin, 128>(x, n, d, A, codes, e8, scale, status, stream);
    case 256: return launch_rows_k<Tin, 256>(x, n, d, A, codes, e8, scale, status, stream);
    default: return cudaErrorInvalidValue;
  }
}

// scale[t] = max|v'_t| / 7 (in place).  Non-finite maxima become 0 and raise the status bit.
__global__ void finalize_scale_kernel(uint32_t* __restrict__ amax_bits, int64_t n, uint32_t* __restrict__ status) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float a = __uint_as_float(amax_bits[t]);
  float s = 0.f;
  if (isfinite(a))
    s = __fdiv_rn(a, 7.0f);
  else
    report(status, kStatusNonFinite);
  reinterpret_cast<float*>(amax_bits)[t] = s;
}

template <typename Tin, int K>
cudaError_t launch_k(const Tin* x, int64_t n, int64_t d, const float* A, uint8_t* codes, int e8, float* scale,
                     uint32_t* status, cudaStream_t stream) {
  using C = ActCfg<K>;
  cudaError_t e = cudaMemsetAsync(scale, 0, (size_t)n * sizeof(float), stream);
  if (e != cudaSuccess) return e;
  auto k0 = transform_quant_kernel<Tin, K, 0>;
  auto k1 = e8 ? transform_quant_kernel<Tin, K, 2> : transform_quant_kernel<Tin, K, 1>;
  if ((e = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM)) != cudaSuccess) return e;
  const int64_t row_tiles = (n + kRows - 1) / kRows;
  if (row_tiles > 0x7FFFFFFF) return cudaErrorInvalidValue;
  const int64_t ny = (d / K) * (K / C::OC);
  if (ny > 65535) return cudaErrorInvalidValue;
  dim3 grid((unsigned)row_tiles, (unsigned)ny);
  uint32_t* amax = reinterpret_cast<uint32_t*>(scale);
  uint32_t* words = reinterpret_cast<uint32_t*>(codes);
  note_launch();
  k0<<<grid, C::THREADS, C::SMEM, stream>>>(x, n, d, A, amax, words, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  note_launch();
  k1<<<grid, C::THREADS, C::SMEM, stream>>>(x, n, d, A, amax, words, status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  note_launch();
  finalize_scale_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(amax, n, status);
  return cudaGetLastError();
}

template <typename Tin>
cudaError_t launch_t(const Tin* x, int64_t n, int64_t d, int k, const float* A, uint8_t* codes, int e8, float* scale,
                     uint32_t* status, cudaStream_t stream) {
  switch (k) {
    case 16: return launch_k<Tin, 16>(x, n, d, A, codes, e8, scale, status, stream);
    case 32: return launch_k<Tin, 32>(x, n, d, A, codes, e8, scale, status, stream);
    case 64: return launch_k<Tin, 64>(x, n, d, A, codes, e8, scale, status, stream);
    case 128: return launch_k<Tin, 128>(x, n, d, A, codes, e8, scale, status, stream);
    case 256: return launch_k<Tin, 256>(x, n, d, A, codes, e8, scale, status, stream);
    default: return cudaErrorInvalidValue;
  }
}

// Float32 units: whole rows where they pay, else the tiled kernels.
template <typename Tin>
cudaError_t launch_simt(const Tin* x, int64_t n, int64_t d, int k, const float* A, uint8_t* codes, int e8, float* scale,
                        uint32_t* status, cudaStream_t stream) {
  const cudaError_t e = launch_rows(x, n, d, k, A, codes, e8, scale, status, stream);
  return e != cudaErrorNotSupported ? e : launch_t(x, n, d, k, A, codes, e8, scale, status, stream);
}

}  // namespace

bool transform_quantize_tc_supported(int dtype, int k, int64_t n, int64_t d);
cudaError_t launch_transform_quantize_tc(const void* x, int64_t n, int64_t d, int k, const float* A,
                                         const uint8_t* planes, uint32_t* amax, uint32_t* words, float* scale,
                                         uint32_t* status, cudaStream_t stream);

cudaError_t launch_transform_quantize_tc_fused(const void* x, int64_t n, int64_t d, int k, const float* A,
                                               const uint8_t* planes, uint32_t* amax, uint32_t* words, int e8,
                                               uint32_t* status, cudaStream_t stream);

cudaError_t launch_transform_quantize_few(const void* x, int dtype, int64_t n, int64_t d, int k, const float* T,
                                          uint8_t* codes, int e8, float* scale, uint32_t* status, cudaStream_t stream);

// planes (optional): T's pre-split bf16 planes (cat_split_transform), used by the tensor-core path.
cudaError_t launch_transform_quantize(const void* x, int dtype, int64_t n, int64_t d, int k, const float* A,
                                      uint8_t* codes, float* scale, uint32_t* status, cudaStream_t stream,
                                      const uint8_t* planes) {
  if (n == 0) return cudaSuccess;
  const cudaError_t e1 = launch_transform_quantize_few(x, dtype, n, d, k, A, codes, 0, scale, status, stream);
  if (e1 != cudaErrorNotSupported) return e1;             // a few rows
  if (transform_quantize_tc_supported(dtype, k, n, d)) {  // bf16 rows: tensor-core path
    uint32_t* amax = reinterpret_cast<uint32_t*>(scale);
    const cudaError_t ef = launch_transform_quantize_tc_fused(x, n, d, k, A, planes, amax,
                                                              reinterpret_cast<uint32_t*>(codes), 0, status, stream);
    if (ef != cudaErrorNotSupported) return ef;  // done (or failed) in one launch
    if (k != 256) {                               // k = 256 has the fused kernel only
      // two passes with the maxima in device scratch: pass 1 writes the steps
      const cudaError_t es = launch_transform_quantize_tc(x, n, d, k, A, planes, nullptr,
                                                          reinterpret_cast<uint32_t*>(codes), scale, status, stream);
      if (es != cudaErrorNotSupported) return es;
      // more rows than the scratch holds: the maxima in the scale buffer, then a finalize launch
      cudaError_t e = cudaMemsetAsync(scale, 0, (size_t)n * sizeof(float), stream);
      if (e == cudaSuccess) e = launch_transform_quantize_tc(x, n, d, k, A, planes, amax,
                                                             reinterpret_cast<uint32_t*>(codes), nullptr, status, stream);
      if (e != cudaSuccess) return e;
      note_launch();
      finalize_scale_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(amax, n, status);
      return cudaGetLastError();
    }
    // k = 256 beyond the fused kernel (more 64-output groups than SMs, more rows than its scratch):
    // the SIMT kernel below
  }
  if (dtype == 0) return launch_simt(static_cast<const float*>(x), n, d, k, A, codes, 0, scale, status, stream);
  return launch_simt(static_cast<const __nv_bfloat16*>(x), n, d, k, A, codes, 0, scale, status, stream);
}

// The same codes as byte codes ([n][d], one E4M3 byte per code); cudaErrorNotSupported (nothing launched) where packed
// ones come from the two-pass tensor-core kernel, which has no byte form.
cudaError_t launch_transform_quantize_e8(const void* x, int dtype, int64_t n, int64_t d, int k, const float* A,
                                         uint8_t* codes8, float* scale, uint32_t* status, cudaStream_t stream,
                                         const uint8_t* planes) {
  if (n == 0) return cudaSuccess;
  const cudaError_t e1 = launch_transform_quantize_few(x, dtype, n, d, k, A, codes8, 1, scale, status, stream);
  if (e1 != cudaErrorNotSupported) return e1;
  if (transform_quantize_tc_supported(dtype, k, n, d)) {
    const cudaError_t ef = launch_transform_quantize_tc_fused(x, n, d, k, A, planes, reinterpret_cast<uint32_t*>(scale),
                                                              reinterpret_cast<uint32_t*>(codes8), 1, status, stream);
    if (ef != cudaErrorNotSupported || transform_tc_group(k, d) != 256) return ef;
    // k = 256 beyond the fused kernel: the SIMT kernels, as for packed codes
  }
  if (dtype == 0) return launch_simt(static_cast<const float*>(x), n, d, k, A, codes8, 1, scale, status, stream);
  return launch_simt(static_cast<const __nv_bfloat16*>(x), n, d, k, A, codes8, 1, scale, status, stream);
}

}  // namespace cat
