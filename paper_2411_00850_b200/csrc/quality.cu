// The two objectives the method states for a quantized layer (Section 3.1), evaluated on the device:
//   squared error        ||W - W_Q||_2^2          (Eq. "Q")
//   first-order change   g^T (W - W_Q)            (Eq. "Taylor": L(W_Q) ~ L(W) - g^T (W - W_Q); Eq. "final_OPO")
// with W_Q = s (q - z) + S, the outliers S being the kept FP16 weights.  Every term is formed and
// summed in FP64 (fp16 / fp32 inputs convert exactly, s (q - z) is exact in FP64), rows are reduced in a
// fixed order, so the two numbers do not depend on scheduling.
#include "common.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kAhead = 2;   // stretches of a lane whose loads are in flight

// The packed words that hold columns 8 j .. 8 j + 7 of a run of 32 (j = 0 .. 3), and the codes out of them.
template <int BITS>
struct Eight {
  static constexpr int kWords = BITS == 3 ? 3 : (BITS == 8 ? 2 : 1);
  unsigned w[kWords];
  __device__ __forceinline__ void fetch(const uint32_t* __restrict__ run, const int j) {
    const uint32_t* p = run + (BITS == 3 ? 0 : (BITS == 8 ? 2 * j : (BITS == 4 ? j : j / 2)));
#pragma unroll
    for (int i = 0; i < kWords; ++i) w[i] = __ldg(p + i);
  }
  // magic | code as the bits of a float (2^23 + code)
  __device__ __forceinline__ void codes(const int j, unsigned (&code)[8]) const {
    constexpr unsigned M = (1u << BITS) - 1u, kMagic = 0x4B000000u;
    unsigned even, odd;   // the codes of columns 8 j, 8 j + 2, .. and 8 j + 1, 8 j + 3, .., BITS apart
    if (BITS == 3) {   // 15 bits of each half-word one after the other, then the top bits: codes of columns 30 and 31
      auto half = [&](const int sh) {
        const unsigned long long all =
            (unsigned long long)(w[0] >> sh & 0x7FFFu) | (unsigned long long)(w[1 % kWords] >> sh & 0x7FFFu) << 15 |
            (unsigned long long)(w[2 % kWords] >> sh & 0x7FFFu) << 30 |
            (unsigned long long)((w[0] >> (sh + 15) & 1u) | (w[1 % kWords] >> (sh + 15) & 1u) << 1 |
                                 (w[2 % kWords] >> (sh + 15) & 1u) << 2) << 45;
        return (unsigned)(all >> (12 * j));
      };
      even = half(0);
      odd = half(16);
    } else if (BITS == 8) {
      even = (w[0] & 0xFFFFu) | w[1 % kWords] << 16;
      odd = w[0] >> 16 | (w[1 % kWords] & 0xFFFF0000u);
    } else {
      even = BITS == 2 ? w[0] >> (8 * (j & 1)) : w[0];
      odd = even >> 16;
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      code[2 * h] = (even >> (BITS * h) & M) | kMagic;
      code[2 * h + 1] = (odd >> (BITS * h) & M) | kMagic;
    }
  }
};

// One warp per row: lane l takes the stretches of 8 columns l, l + 32, ... (16 bytes of W, 32 of G, so that a warp's
// loads are whole lines), all loads kAhead stretches ahead of the arithmetic; outlier positions are marked in a bit map
// and handled from the CSR entries instead.  s (q - z) has at most 20 bits: the FP32 product is exact.
// Bound by memory latency and the FP64 conversions (a third of the conversion unit).  11008 x 4096: one thread per run
// of 32 columns with 2- and 4-byte loads 291 us, one CTA per row with these loads 103 (waiting at its
// barriers), this 73.  WIDE: W and G start on 16 bytes (a view of a larger buffer need not: element loads then).
template <int BITS, bool WIDE>
__global__ void __launch_bounds__(kThreads, 5)
quality_row_kernel(const uint16_t* __restrict__ W, const float* __restrict__ G, const uint32_t* __restrict__ codes,
                   const uint16_t* __restrict__ scales, const uint8_t* __restrict__ zeros,
                   const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
                   const uint16_t* __restrict__ val, int N, int K, int group, double* __restrict__ rows) {
  extern __shared__ unsigned masks[];   // [kThreads / 32][K / 32]
  const int lane = threadIdx.x & 31, n = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
  if (n >= N) return;
  const int nruns = K / 32, ngroups = K / group, n8 = K / 8;
  unsigned* mask = masks + (threadIdx.x >> 5) * nruns;
  const uint16_t* wrow = W + (size_t)n * K;
  const float* grow = G + (size_t)n * K;
  const uint32_t* crow = codes + (size_t)n * nruns * BITS;
  const uint16_t* srow = scales + (size_t)n * ngroups;
  const uint8_t* zrow = zeros + (size_t)n * ngroups;
  uint4 w[kAhead];
  float4 ga[kAhead], gb[kAhead];
  Eight<BITS> packed[kAhead];
  unsigned scale[kAhead];   // fp16 scale | zero-point << 16
  const int shift = 31 - __clz(group);
  auto fetch = [&](const int u, const int i) {
    if (i < n8) {
      if constexpr (WIDE) {
        w[u] = __ldcs(reinterpret_cast<const uint4*>(wrow) + i);
        ga[u] = __ldcs(reinterpret_cast<const float4*>(grow) + 2 * i);
        gb[u] = __ldcs(reinterpret_cast<const float4*>(grow) + 2 * i + 1);
      } else {
        auto pair = [&](const int e) { return (unsigned)wrow[8 * i + e] | (unsigned)wrow[8 * i + e + 1] << 16; };
        const float* g = grow + 8 * i;
        w[u] = make_uint4(pair(0), pair(2), pair(4), pair(6));
        ga[u] = make_float4(g[0], g[1], g[2], g[3]);
        gb[u] = make_float4(g[4], g[5], g[6], g[7]);
      }
      packed[u].fetch(crow + (i >> 2) * BITS, i & 3);
      scale[u] = __ldg(srow + ((i * 8) >> shift)) | (unsigned)__ldg(zrow + ((i * 8) >> shift)) << 16;
    }
  };
#pragma unroll
  for (int u = 0; u < kAhead; ++u) fetch(u, lane + u * 32);
  for (int r = lane; r < nruns; r += 32) mask[r] = 0u;
  __syncwarp();
  const int jb = row_ptr[n], je = row_ptr[n + 1];
  double sq = 0.0, fo = 0.0;
  for (int j = jb + lane; j < je; j += 32) {
    const int c = col_idx[j];
    atomicOr(&mask[c >> 5], 1u << (c & 31));
    const double d = (double)__half2float(__ushort_as_half(wrow[c])) - (double)__half2float(__ushort_as_half(val[j]));
    sq += d * d;
    fo += (double)grow[c] * d;
  }
  __syncwarp();
  for (int base = lane; base < n8; base += kAhead * 32) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int i = base + u * 32;
      if (i >= n8) break;
      const unsigned h[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
      const float g[8] = {ga[u].x, ga[u].y, ga[u].z, ga[u].w, gb[u].x, gb[u].y, gb[u].z, gb[u].w};
      unsigned code[8];
      packed[u].codes(i & 3, code);
      const float s = __half2float(__ushort_as_half((unsigned short)scale[u]));
      const float z = __uint_as_float(0x4B000000u | scale[u] >> 16);
      fetch(u, i + kAhead * 32);
      const unsigned m = mask[i >> 2] >> (8 * (i & 3));
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        // an outlier's place holds the zero-point: its dense term is zero as it stands, its weight is left out
        const float x = (m >> e) & 1u ? 0.f : __half2float(__ushort_as_half((unsigned short)(h[e / 2] >> (16 * (e & 1)))));
        const double d = (double)x - (double)(s * (__uint_as_float(code[e]) - z));
        sq += d * d;
        fo += (double)g[e] * d;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
    fo += __shfl_xor_sync(0xFFFFFFFFu, fo, o);
  }
  if (lane == 0) {
    rows[2 * (size_t)n] = sq;
    rows[2 * (size_t)n + 1] = fo;
  }
}

// Sum of the per-row pairs in a fixed order: thread t adds rows t, t + 1024, ..., then a tree over the threads.
__global__ void __launch_bounds__(1024) quality_sum_kernel(const double* __restrict__ rows, int N, double* __restrict__ out) {
  __shared__ double sa[1024], sb[1024];
  double a = 0.0, b = 0.0;
  for (int n = threadIdx.x; n < N; n += 1024) {
    a += rows[2 * (size_t)n];
    b += rows[2 * (size_t)n + 1];
  }
  sa[threadIdx.x] = a;
  sb[threadIdx.x] = b;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sa[threadIdx.x] += sa[threadIdx.x + o];
      sb[threadIdx.x] += sb[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = sa[0];
    out[1] = sb[0];
  }
}

}  // namespace

extern "C" gwq_status gwq_quality(const uint16_t* W, const float* G, const gwq_packed* P, double* sq_err,
                                  double* first_order, void* stream_) {
  if (!W || !G || !P || P->tag != GWQ_TAG_PACKED || !P->S || !sq_err || !first_order) return GWQ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(W) & 1u) != 0 || (reinterpret_cast<uintptr_t>(G) & 3u) != 0) return GWQ_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  gwq_status st = GWQ_OK;
  void* scratch = nullptr;
  double* rows = nullptr;
  double* host = static_cast<double*>(gwq_pinned_slot());
  const size_t smem = (size_t)(P->K / 32) * sizeof(unsigned) * (kThreads / 32);
  if (!host) return GWQ_ERR_ALLOC;
  GWQ_CUDA_TRY(gwq_dev_alloc(&scratch, (size_t)P->N * 2 * sizeof(double), stream));
  rows = static_cast<double*>(scratch);
#define GWQ_QUALITY_LAUNCH(BITS, WIDE)                                                                               \
  do {                                                                                                               \
    GWQ_CUDA_TRY(cudaFuncSetAttribute(quality_row_kernel<BITS, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                      (int)smem));                                                                   \
    quality_row_kernel<BITS, WIDE><<<(P->N + kThreads / 32 - 1) / (kThreads / 32), kThreads, smem, stream>>>(        \
        W, G, P->codes, P->scales, P->zeros, P->S->row_ptr, P->S->col_idx, P->S->val, P->N, P->K, P->group, rows);   \
  } while (0)
  if (gwq_aligned16(W) && gwq_aligned16(G)) {
    if (P->bits == 4) GWQ_QUALITY_LAUNCH(4, true);
    else if (P->bits == 3) GWQ_QUALITY_LAUNCH(3, true);
    else if (P->bits == 8) GWQ_QUALITY_LAUNCH(8, true);
    else GWQ_QUALITY_LAUNCH(2, true);
  } else {
    if (P->bits == 4) GWQ_QUALITY_LAUNCH(4, false);
    else if (P->bits == 3) GWQ_QUALITY_LAUNCH(3, false);
    else if (P->bits == 8) GWQ_QUALITY_LAUNCH(8, false);
    else GWQ_QUALITY_LAUNCH(2, false);
  }
#undef GWQ_QUALITY_LAUNCH
  GWQ_CUDA_TRY(cudaGetLastError());
  quality_sum_kernel<<<1, 1024, 0, stream>>>(rows, P->N, host);
  GWQ_CUDA_TRY(cudaGetLastError());
  GWQ_CUDA_TRY(cudaStreamSynchronize(stream));
  *sq_err = host[0];
  *first_order = host[1];
fail:
  gwq_dev_free_async(scratch, stream);
  gwq_pinned_slot_return(host);
  return st;
}
