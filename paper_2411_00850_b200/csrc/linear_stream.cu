// Host side of the streaming decode kernel (stream_kernel.cuh): which calls it takes, the variant, the pre-pass that
// transposes the activations, and the launch.
#include "stream_kernel.cuh"

namespace gwq_stream {

size_t smem_bytes(const Variant& v, int bits, int K) {
  const int ngroups = K / 128, kw = v.kw, rw = v.warps / kw;
  const size_t act = v.tp == 1 ? ((size_t)ngroups * 260 + 15) / 16 * 16 : (size_t)kw * kRing * block_bytes(bits, v.tp, v.gs);
  const size_t codes = (size_t)v.warps * steps_ahead(bits, v.tp, v.rt) * v.rt * slot_bytes(bits, v.tp, v.gs);
  const size_t sums = (size_t)kw * rw * v.rt * (v.tp == 1 ? 16 : v.tp * 16) * 4;
  return act + codes + sums;
}

}  // namespace gwq_stream

namespace {
using namespace gwq_stream;

// One CTA per step of 128 columns and block of 8 mma columns, thread = column of x: the step's part of the transposed
// activations (columns at place()) and, behind it, per token the sums of x by group (FP32) and the power of two that bf16
// activations were divided by (see stream_kernel.cuh).  Tokens from M on are zeros.  Every product of several tokens waits for
// this kernel, which is one trip to memory long: with the blocks of a step one after the other in one CTA it took 8.7 us at
// 16 tokens (4096 x 4096 with its product 10.7 -> 9.6 us, 28672 x 8192 at 32 tokens 95.6 -> 89.4 us).
// `groups` (1 or 2): groups split by accumulators; `log_cols` (0 to 3): columns of a token, one per group of the step.
template <bool BF16>
__global__ void __launch_bounds__(128) transpose_kernel(const uint16_t* __restrict__ x, unsigned char* __restrict__ xt, int groups,
                                                        int log_cols, int M, int K) {
  __shared__ float red[8][8];      // sums over 16 columns
  __shared__ unsigned most[4][8];
  // launched with programmatic stream serialization: the product that follows may start fetching its weights now;
  // x may still be being written by the kernel before this one
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int c = threadIdx.x, lane = c & 31, warp = c >> 5, nb = blockIdx.y, tp = gridDim.y * 8;
  const int tok = 8 >> log_cols, first = (c >> (7 - log_cols)) * tok;   // tokens of a block; the column of its first one that c belongs to
  const uint16_t* src = x + (size_t)blockIdx.x * 128 + c;
  unsigned char* block = xt + (size_t)blockIdx.x * (tp / 8 * 2048 + (groups + 1) * tp * 4);
  float* const stats = reinterpret_cast<float*>(block + tp / 8 * 2048) + nb * 8;
  unsigned v[8];   // column i of the block
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = nb * tok + i - first;
    v[i] = i >= first && i < first + tok && m < M ? (unsigned)__ldg(src + (size_t)m * K) : 0u;
  }
  if (BF16) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned w = __reduce_max_sync(0xFFFFFFFFu, v[i] & 0x7FFFu);
      if (lane == 0) most[warp][i] = w;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float power = power_for(max(max(most[0][i], most[1][i]), max(most[2][i], most[3][i])));
      if (c == 0) stats[groups * tp + i] = power;
      v[i] = scaled_pair(v[i], inverse_power(power)) & 0xFFFFu;
    }
  } else if (c < 8) {
    stats[groups * tp + c] = 1.f;
  }
  *reinterpret_cast<uint4*>(block + nb * 2048 + place(c, groups) * 16) =
      make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
  float f[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) f[i] = __half2float(__ushort_as_half((unsigned short)v[i]));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] += __shfl_xor_sync(0xFFFFFFFFu, f[i], o);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if ((lane & 15) == 0) red[c >> 4][i] = f[i];
  __syncthreads();
  if (c < 8) {   // (columns outside a group hold zeros there)
    const float lo = (red[0][c] + red[1][c]) + (red[2][c] + red[3][c]), hi = (red[4][c] + red[5][c]) + (red[6][c] + red[7][c]);
    stats[c] = groups == 2 ? lo : lo + hi;
    if (groups == 2) stats[tp + c] = hi;
  }
}

constexpr size_t kSmemMost = 227 * 1024;

bool plan(const gwq_packed* const* P, int count, int M, Variant* v, int* first_cta, int* grid) {
  if (count < 1 || count > kMaxLayers || M < 1 || M > 32) return false;
  const int K = P[0]->K, group = P[0]->group, bits = P[0]->bits;
  if (K % 128 != 0) return false;
  for (int i = 0; i < count; ++i) {
    const gwq_priv* pv = static_cast<const gwq_priv*>(P[i]->priv);
    if (P[i]->K != K || P[i]->group != group || P[i]->bits != bits || !pv->cv || !pv->szp) return false;
  }
  const gwq_priv* pv = static_cast<const gwq_priv*>(P[0]->priv);
  v->gs = 128 / group;
  const bool cols = M > 1 && by_columns(bits, v->gs);
  const int columns = cols ? M * v->gs : M;
  if (columns > 32) return false;
  v->tp = M == 1 ? 1 : (columns <= 8 ? 8 : (columns <= 16 ? 16 : 32));
  // How K is split decides the order of the sums, so it has to be the same in every call that a layer may be part of: by
  // the number of tokens and, up to 8 columns, the layer's own tiles (eight slices where a CTA gets one tile, whose second
  // row of warps would idle: 4096 x 11008 at 4 tokens 18.6 -> 14.1 us).
  const int sms = pv->sm_count > 0 ? pv->sm_count : 148;
  v->kw = v->tp >= 16 ? 4 : 8;
  if (M > 1) {
    if (!pv->xt) return false;
    for (int i = 0; i < count && v->tp == 8; ++i) {
      const int kw = (P[i]->N + 15) / 16 <= ctas_per_sm(8) * sms ? 8 : 4;
      if (i > 0 && kw != v->kw) return false;
      v->kw = kw;
    }
  }
  // CTAs of each layer: its share of the wave by tiles, one tile each at least
  const int slots = ctas_per_sm(v->tp) * sms;
  long long tiles = 0, before = 0;
  for (int i = 0; i < count; ++i) tiles += (P[i]->N + 15) / 16;
  // 17 to 32 columns: eight warps with registers to spare, or sixteen where there are rows of tiles for them (us at 32
  // tokens: 13.9 / 19.5 on 4096 x 4096, 34.7 / 37.5 on 8192 x 8192, 30.3 / 30.8 on 11008 x 4096, 55.9 / 54.9 on 20480 x
  // 5120, 105 / 94 on 28672 x 8192; two accumulators per position and the three positions of
  // 3-bit codes do not fit the sixteen's registers: 0.62 of the speed on 20480 x 5120).
  v->warps = v->tp == 32 && split_groups(bits, 32, v->gs) == 1 && bits != 3 && tiles > 5LL * sms ? 16 : 8;
  int most = 1, cta = 0;
  for (int i = 0; i < count; ++i) {
    const int lt = (P[i]->N + 15) / 16;
    first_cta[i] = cta;
    int share = (int)(slots * (before + lt) / tiles - slots * before / tiles);
    share = share < 1 ? 1 : (share > lt ? lt : share);
    before += lt;
    cta += share;
    if ((lt + share - 1) / share > most) most = (lt + share - 1) / share;
  }
  *grid = cta;
  // tiles that share a step's activations: no more than a warp gets
  const int rw = v->warps / v->kw;
  const int per_warp = (most + rw - 1) / rw, limit = most_tiles(v->tp, bits);
  v->rt = per_warp >= 3 && limit >= 4 ? 4 : (per_warp >= 2 && limit >= 2 ? 2 : 1);
  if (v->rt == 2 && smem_bytes(*v, bits, K) > kSmemMost) v->rt = 1;   // 8-bit codes beyond 16 columns
  return smem_bytes(*v, bits, K) <= kSmemMost;
}

}  // namespace

size_t gwq_stream_scratch_bytes(int K) { return (size_t)(K / 128) * block_bytes(4, 32, 2); }

bool gwq_stream_takes(const gwq_packed* P, int M) {
  Variant v;
  int first_cta[kMaxLayers], grid;
  return plan(&P, 1, M, &v, first_cta, &grid);
}

// `count` layers that read the same x, in one launch.  GWQ_ERR_UNSUPPORTED where the kernel has no variant (nothing has
// been launched then).  The transposed activations of several tokens go to `scratch`.
gwq_status gwq_launch_stream(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y,
                             gwq_dtype yd, void* scratch, cudaStream_t stream) {
  Variant v;
  int first_cta[kMaxLayers], grid;
  if (!plan(P, count, M, &v, first_cta, &grid)) return GWQ_ERR_UNSUPPORTED;
  Args a = {};
  for (int i = 0; i < count; ++i) {
    const gwq_priv* pv = static_cast<const gwq_priv*>(P[i]->priv);
    a.layer[i].codes = P[i]->codes; a.layer[i].szp = pv->szp;
    a.layer[i].row_ptr = P[i]->S->row_ptr; a.layer[i].cv = pv->cv;
    a.layer[i].tb = pv->tb; a.layer[i].tb_ptr = pv->tb_ptr;
    a.layer[i].y = y[i]; a.layer[i].N = P[i]->N;
    a.layer[i].first_cta = first_cta[i];
  }
  a.count = count;
  a.x = static_cast<const uint16_t*>(x);
  a.yd = yd; a.K = P[0]->K; a.M = M;
  const bool bf = xd == GWQ_BF16;
  cudaError_t e = cudaSuccess;
  if (v.tp > 1) {
    unsigned char* xt = static_cast<unsigned char*>(scratch);
    if (!xt) return GWQ_ERR_WORKSPACE;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.K / 128), (unsigned)(v.tp / 8));
    cfg.blockDim = dim3(128);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int groups = split_groups(P[0]->bits, v.tp, v.gs), cols = by_columns(P[0]->bits, v.gs) ? v.gs : 1, log_cols = cols == 8 ? 3 : cols >> 1;
    e = bf ? cudaLaunchKernelEx(&cfg, transpose_kernel<true>, a.x, xt, groups, log_cols, M, a.K)
           : cudaLaunchKernelEx(&cfg, transpose_kernel<false>, a.x, xt, groups, log_cols, M, a.K);
    a.xt = xt;
  }
  if (e == cudaSuccess) {
    switch (P[0]->bits) {
      case 4: e = bf ? launch_w4_bf16(v, a, grid, stream) : launch_w4_f16(v, a, grid, stream); break;
      case 3: e = bf ? launch_w3_bf16(v, a, grid, stream) : launch_w3_f16(v, a, grid, stream); break;
      case 8: e = bf ? launch_w8_bf16(v, a, grid, stream) : launch_w8_f16(v, a, grid, stream); break;
      default: e = bf ? launch_w2_bf16(v, a, grid, stream) : launch_w2_f16(v, a, grid, stream); break;
    }
  }
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return GWQ_ERR_CUDA;
  }
  return GWQ_OK;
}
