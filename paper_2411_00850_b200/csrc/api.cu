// Entry points that are not kernels of their own: dispatch of the forward product,
// the host-buffer variant, object release and status names.
#include "common.cuh"

#ifndef GWQ_DECODE_MAX_M
#define GWQ_DECODE_MAX_M 32   // up to here the decode kernels; above, the kernels of prompts
#endif

static size_t dtype_bytes(gwq_dtype d) { return d == GWQ_F32 ? 4 : 2; }

// 2 to 32 tokens with a workspace: the tcgen05 decode kernel where it is the fastest.
static bool wants_skinny(const gwq_packed* P, gwq_dtype xd, int M) {
  return M > 1 && M <= GWQ_DECODE_MAX_M && gwq_skinny_ahead(P, xd, M);
}
static bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

static bool takes_few(const gwq_packed* P, gwq_dtype xd, int M) { return gwq_decode_ahead(P, xd, M) || gwq_stream_takes(P, M); }
bool gwq_takes_decode(const gwq_packed* P, gwq_dtype xd, int M) {
  return M <= GWQ_DECODE_MAX_M && !gwq_skinny_before(P, xd, M) && takes_few(P, xd, M);
}
static bool one_kernel(const gwq_packed* const* P, int count, gwq_dtype xd, int M) {
  for (int i = 1; i < count; ++i)
    if (gwq_decode_ahead(P[i], xd, M) != gwq_decode_ahead(P[0], xd, M)) return false;
  return true;
}
// Layers that read the same x, up to 32 tokens, in one launch: the kernel that each layer takes by itself.  `scratch`: for
// the copy of the activations that most kernels of several tokens make first, few_scratch bytes.
static gwq_status launch_few(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y,
                             gwq_dtype yd, void* scratch, cudaStream_t stream) {
  if (!one_kernel(P, count, xd, M)) return GWQ_ERR_UNSUPPORTED;
  return gwq_decode_ahead(P[0], xd, M) ? gwq_launch_decode_multi(P, count, x, xd, M, y, yd, scratch, stream)
                                       : gwq_launch_stream(P, count, x, xd, M, y, yd, scratch, stream);
}
static size_t few_scratch(const gwq_packed* const* P, int count, gwq_dtype xd, int M) {
  if (M > GWQ_DECODE_MAX_M || !one_kernel(P, count, xd, M)) return 0;
  if (gwq_decode_ahead(P[0], xd, M) ? gwq_decode_stages(P, count, M) : M == 1 || !gwq_stream_takes(P[0], M)) return 0;
  return gwq_stream_scratch_bytes(P[0]->K);
}
// the caller's workspace as that scratch
static void* scratch_in(void* ws, size_t ws_bytes, size_t need) {
  return need > 0 && ws && ws_bytes >= need && aligned256(ws) ? ws : nullptr;
}
static void* own_scratch(const gwq_packed* P) { return static_cast<const gwq_priv*>(P->priv)->xt; }

// Calls without a workspace.  From nine tokens on they take the scratch inside the layer, so that calls on one layer have to
// be ordered; with fewer they share nothing: where the kernel would need scratch, the tokens are taken a few at
// a time, as many as the kernel with a CTA per tile stages in shared memory, or one by one.
static const int kMostTokensAlone = 8;
static gwq_status launch_alone(const gwq_packed* P, const void* x, gwq_dtype xd, int M, void* y, gwq_dtype yd, cudaStream_t stream) {
  if (!takes_few(P, xd, M)) return GWQ_ERR_UNSUPPORTED;
  if (few_scratch(&P, 1, xd, M) == 0) return launch_few(&P, 1, x, xd, M, &y, yd, nullptr, stream);
  if (M > kMostTokensAlone) return launch_few(&P, 1, x, xd, M, &y, yd, own_scratch(P), stream);
  for (int m = 0; m < M;) {
    int n = M - m;
    while (n > 1 && !gwq_decode_stages(&P, 1, n)) --n;
    const char* const xm = static_cast<const char*>(x) + (size_t)m * P->K * dtype_bytes(xd);
    void* const ym = static_cast<char*>(y) + (size_t)m * P->N * dtype_bytes(yd);
    const gwq_status st = n > 1 ? gwq_launch_decode_multi(&P, 1, xm, xd, n, &ym, yd, nullptr, stream)
                                : launch_few(&P, 1, xm, xd, 1, &ym, yd, nullptr, stream);
    if (st != GWQ_OK) return st;
    m += n;
  }
  return GWQ_OK;
}

extern "C" size_t gwq_linear_workspace_bytes(const gwq_packed* P, gwq_dtype xd, int32_t M) {
  if (!P || P->tag != GWQ_TAG_PACKED || !P->priv || M <= 0) return 0;
  if (wants_skinny(P, xd, M)) return gwq_skinny_workspace_bytes(&P, 1, xd, M);
  if (M <= GWQ_DECODE_MAX_M && takes_few(P, xd, M)) return few_scratch(&P, 1, xd, M);
  return gwq_prefill_workspace_bytes(P, xd, M);
}

extern "C" gwq_status gwq_linear_ws(const gwq_packed* P, const void* x, gwq_dtype xd, int32_t M, void* y,
                                    gwq_dtype yd, void* ws, size_t ws_bytes, void* stream_) {
  if (!P || P->tag != GWQ_TAG_PACKED || !P->S || !P->priv || !x || !y || M <= 0) return GWQ_ERR_INVALID_ARG;
  if (xd != GWQ_F16 && xd != GWQ_BF16) return GWQ_ERR_UNSUPPORTED;
  if (yd != GWQ_F16 && yd != GWQ_BF16 && yd != GWQ_F32) return GWQ_ERR_INVALID_ARG;
  if (!gwq_aligned16(x) || !gwq_aligned16(y)) return GWQ_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  // without a workspace (and with one that is too small or not aligned, where that has not always been an error) the other kernels
  // serve what the tcgen05 decode kernel would take
  if (wants_skinny(P, xd, M) && ws && ws_bytes >= gwq_skinny_workspace_bytes(&P, 1, xd, M)) {
    if (aligned256(ws)) return gwq_launch_skinny(&P, 1, x, xd, M, &y, yd, ws, stream);
    if (gwq_skinny_before(P, xd, M)) return GWQ_ERR_WORKSPACE;
  }
  if (M <= GWQ_DECODE_MAX_M) {
    void* const scratch = scratch_in(ws, ws_bytes, few_scratch(&P, 1, xd, M));
    const gwq_status st = scratch ? launch_few(&P, 1, x, xd, M, &y, yd, scratch, stream) : launch_alone(P, x, xd, M, y, yd, stream);
    if (st != GWQ_ERR_UNSUPPORTED) return st;   // shapes they do not take: the tensor-core kernel
  }
  return gwq_launch_prefill(P, x, xd, M, y, yd, ws, ws_bytes, stream);
}

extern "C" gwq_status gwq_linear(const gwq_packed* P, const void* x, gwq_dtype xd, int32_t M, void* y,
                                 gwq_dtype yd, void* stream_) {
  return gwq_linear_ws(P, x, xd, M, y, yd, nullptr, 0, stream_);
}

// The layers of a call of up to 32 tokens that the tcgen05 decode kernel takes by themselves, or the others: each kind goes as one
// launch (one by one about 64 us, so 53 on 8192 + 4096 + 4096 rows x 8192 in groups of 64 at 16 tokens, where the first is of the one kind;
// 51 and 36 on 4096 + 1024 + 1024 rows x 4096 at 32).
struct Kind {
  const gwq_packed* P[GWQ_MULTI_MAX];
  void* y[GWQ_MULTI_MAX];
  int count;
  bool alike;   // one width and one group size
};
static Kind layers_of_kind(bool skinny, const gwq_packed* const* P, void* const* y, int count, gwq_dtype xd, int M) {
  Kind k = {};
  k.alike = true;
  for (int i = 0; i < count; ++i) {
    if (wants_skinny(P[i], xd, M) != skinny) continue;
    k.P[k.count] = P[i];
    k.y[k.count++] = y ? y[i] : nullptr;
    k.alike = k.alike && P[i]->bits == k.P[0]->bits && P[i]->group == k.P[0]->group;
  }
  return k;
}

static bool valid_layers(const gwq_packed* const* P, int32_t count, int32_t M) {
  if (!P || count < 1 || count > GWQ_MULTI_MAX || M <= 0) return false;
  for (int i = 0; i < count; ++i)
    if (!P[i] || P[i]->tag != GWQ_TAG_PACKED || !P[i]->S || !P[i]->priv || P[i]->K != P[0]->K) return false;
  return true;
}

extern "C" size_t gwq_linear_multi_workspace_bytes(const gwq_packed* const* P, int32_t count, gwq_dtype xd, int32_t M) {
  if (!valid_layers(P, count, M) || (xd != GWQ_F16 && xd != GWQ_BF16)) return 0;
  size_t need = 0;
  if (M <= GWQ_DECODE_MAX_M) {
    const Kind few = layers_of_kind(false, P, nullptr, count, xd, M), skinny = layers_of_kind(true, P, nullptr, count, xd, M);
    if (few.count > 0) need = few_scratch(few.P, few.count, xd, M);
    const size_t wide = skinny.count > 0 && skinny.alike ? gwq_skinny_workspace_bytes(skinny.P, skinny.count, xd, M) : 0;
    need = wide > need ? wide : need;
  }
  for (int i = 0; i < count; ++i) {
    const size_t own = gwq_linear_workspace_bytes(P[i], xd, M);
    need = own > need ? own : need;
  }
  return need;
}

static gwq_status one_by_one(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y, gwq_dtype yd,
                             void* ws, size_t ws_bytes, cudaStream_t stream) {
  for (int i = 0; i < count; ++i) {
    const gwq_status st = gwq_linear_ws(P[i], x, xd, M, y[i], yd, ws, ws_bytes, stream);
    if (st != GWQ_OK) return st;
  }
  return GWQ_OK;
}
// Layers that are not the tcgen05 kernel's (or a call without a workspace): one launch where they share a kernel.
static gwq_status few_together(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y, gwq_dtype yd,
                                void* ws, size_t ws_bytes, cudaStream_t stream) {
  const size_t need = few_scratch(P, count, xd, M);
  void* scratch = scratch_in(ws, ws_bytes, need);
  if (!scratch && M > kMostTokensAlone) scratch = own_scratch(P[0]);
  if (scratch || need == 0) {
    const gwq_status st = launch_few(P, count, x, xd, M, y, yd, scratch, stream);
    if (st != GWQ_ERR_UNSUPPORTED) return st;
  }
  return one_by_one(P, count, x, xd, M, y, yd, ws, ws_bytes, stream);
}

extern "C" gwq_status gwq_linear_multi_ws(const gwq_packed* const* P, int32_t count, const void* x, gwq_dtype xd, int32_t M,
                                          void* const* y, gwq_dtype yd, void* ws, size_t ws_bytes, void* stream_) {
  if (!P || !y || !x || count < 1 || count > GWQ_MULTI_MAX || M <= 0) return GWQ_ERR_INVALID_ARG;
  if (xd != GWQ_F16 && xd != GWQ_BF16) return GWQ_ERR_UNSUPPORTED;
  if (yd != GWQ_F16 && yd != GWQ_BF16 && yd != GWQ_F32) return GWQ_ERR_INVALID_ARG;
  if (!gwq_aligned16(x) || !valid_layers(P, count, M)) return GWQ_ERR_INVALID_ARG;
  for (int i = 0; i < count; ++i)
    if (!y[i] || !gwq_aligned16(y[i])) return GWQ_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  if (M <= GWQ_DECODE_MAX_M && !ws) return few_together(P, count, x, xd, M, y, yd, nullptr, 0, stream);
  if (M <= GWQ_DECODE_MAX_M) {
    const Kind few = layers_of_kind(false, P, y, count, xd, M), skinny = layers_of_kind(true, P, y, count, xd, M);
    if (few.count > 0) {
      const gwq_status st = few_together(few.P, few.count, x, xd, M, few.y, yd, ws, ws_bytes, stream);
      if (st != GWQ_OK) return st;
    }
    if (skinny.count > 0 && skinny.alike && aligned256(ws) && ws_bytes >= gwq_skinny_workspace_bytes(skinny.P, skinny.count, xd, M))
      return gwq_launch_skinny(skinny.P, skinny.count, x, xd, M, skinny.y, yd, ws, stream);
    return one_by_one(skinny.P, skinny.count, x, xd, M, skinny.y, yd, ws, ws_bytes, stream);
  }
  return one_by_one(P, count, x, xd, M, y, yd, ws, ws_bytes, stream);
}

extern "C" gwq_status gwq_linear_multi(const gwq_packed* const* P, int32_t count, const void* x, gwq_dtype xd,
                                       int32_t M, void* const* y, gwq_dtype yd, void* stream_) {
  return gwq_linear_multi_ws(P, count, x, xd, M, y, yd, nullptr, 0, stream_);
}

// A staging buffer of at least `need` bytes; its last use was on whatever stream the caller had then.
static cudaError_t grow(void** buf, size_t* have, size_t need, cudaStream_t stream) {
  if (*have >= need) return cudaSuccess;
  gwq_dev_free(*buf);
  *have = 0;
  const cudaError_t e = gwq_dev_alloc(buf, need, stream);
  if (e != cudaSuccess) return e;
  *have = need;
  return cudaStreamSynchronize(stream);   // from here on usable on every stream
}

// The address at which kernels see `bytes` of host memory, NULL unless all of it is pinned.
static void* device_view(const void* p, size_t bytes) {
  cudaPointerAttributes first = {}, last = {};
  if (cudaPointerGetAttributes(&first, p) != cudaSuccess ||
      cudaPointerGetAttributes(&last, static_cast<const char*>(p) + bytes - 1) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  if (first.type != cudaMemoryTypeHost || last.type != cudaMemoryTypeHost || !first.devicePointer ||
      static_cast<char*>(last.devicePointer) != static_cast<char*>(first.devicePointer) + bytes - 1)
    return nullptr;
  return first.devicePointer;
}

// results that kernels write to host memory themselves: beyond, the copy engine's longer bursts win
static const size_t kDirectMostBytes = 256 * 1024;

static gwq_status linear_host(gwq_packed* P, const void* x_host, gwq_dtype xd, int32_t M, void* y_host, gwq_dtype yd,
                              void* stream_, bool synchronise) {
  if (!P || P->tag != GWQ_TAG_PACKED || !P->priv || !x_host || !y_host || M <= 0) return GWQ_ERR_INVALID_ARG;
  if (xd != GWQ_F16 && xd != GWQ_BF16) return GWQ_ERR_UNSUPPORTED;
  if (yd != GWQ_F16 && yd != GWQ_BF16 && yd != GWQ_F32) return GWQ_ERR_INVALID_ARG;
  gwq_priv* pv = static_cast<gwq_priv*>(P->priv);
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  const size_t xb = (size_t)M * P->K * dtype_bytes(xd), yb = (size_t)M * P->N * dtype_bytes(yd);
  gwq_status st = GWQ_OK;
  // Few tokens: what is pinned is read and written by the kernels themselves.  The activations are read once (by the
  // transposing pre-pass, or, where every CTA reads them, by a kernel that copies them first) and y is
  // written once, so that nothing is gained by the copy engine, whose two copies take longer than the product
  // (4096 x 11008 at 4 tokens: 47 -> 34 us).
  const bool skinny = wants_skinny(P, xd, M), direct = skinny || gwq_takes_decode(P, xd, M);
  const bool copied = M == 1 || (direct && !skinny && gwq_decode_ahead(P, xd, M));
  const void* x = direct && gwq_aligned16(x_host) ? device_view(x_host, xb) : nullptr;
  // (the kernels store element by element; the copy engine takes any address)
  const bool whole = (reinterpret_cast<uintptr_t>(y_host) & (dtype_bytes(yd) - 1)) == 0;
  void* y = direct && whole && yb <= kDirectMostBytes ? device_view(y_host, yb) : nullptr;
  if (!x || copied) GWQ_CUDA_TRY(grow(&pv->x_stage, &pv->x_stage_bytes, xb, stream));
  if (!y) GWQ_CUDA_TRY(grow(&pv->y_stage, &pv->y_stage_bytes, yb, stream));
  if (!direct || skinny) GWQ_CUDA_TRY(grow(&pv->ws_stage, &pv->ws_stage_bytes, gwq_linear_workspace_bytes(P, xd, M), stream));
  if (!x) {
    GWQ_CUDA_TRY(cudaMemcpyAsync(pv->x_stage, x_host, xb, cudaMemcpyHostToDevice, stream));
  } else if (copied) {
    GWQ_CUDA_TRY(gwq_copy_arrays(1, &x, &pv->x_stage, &xb, stream));
  }
  if (!x || copied) x = pv->x_stage;
  if (direct) {
    void* const out = y ? y : pv->y_stage;
    st = skinny ? gwq_launch_skinny(&P, 1, x, xd, M, &out, yd, pv->ws_stage, stream)
                : launch_few(&P, 1, x, xd, M, &out, yd, own_scratch(P), stream);
  } else {
    st = gwq_linear_ws(P, x, xd, M, pv->y_stage, yd, pv->ws_stage, pv->ws_stage_bytes, stream);
  }
  if (st != GWQ_OK) return st;
  if (!y) GWQ_CUDA_TRY(cudaMemcpyAsync(y_host, pv->y_stage, yb, cudaMemcpyDeviceToHost, stream));
  if (synchronise) GWQ_CUDA_TRY(cudaStreamSynchronize(stream));
  return GWQ_OK;
fail:
  return st;
}

extern "C" gwq_status gwq_linear_host(gwq_packed* P, const void* x_host, gwq_dtype xd, int32_t M,
                                      void* y_host, gwq_dtype yd, void* stream_) {
  return linear_host(P, x_host, xd, M, y_host, yd, stream_, true);
}

extern "C" gwq_status gwq_linear_host_async(gwq_packed* P, const void* x_host, gwq_dtype xd, int32_t M,
                                            void* y_host, gwq_dtype yd, void* stream_) {
  return linear_host(P, x_host, xd, M, y_host, yd, stream_, false);
}

extern "C" gwq_status gwq_device_status(const gwq_packed* P, void* stream_) {
  if (!P || P->tag != GWQ_TAG_PACKED || !P->priv) return GWQ_ERR_INVALID_ARG;
  const gwq_priv* pv = static_cast<const gwq_priv*>(P->priv);
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  int32_t h = 0;
  if (cudaMemcpyAsync(&h, pv->dev_status, sizeof(h), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    (void)cudaGetLastError();
    return GWQ_ERR_CUDA;
  }
  if (h != 0) (void)cudaMemsetAsync(pv->dev_status, 0, sizeof(int32_t), stream);
  return (gwq_status)h;
}

extern "C" gwq_status gwq_set_wait_limit(gwq_packed* P, int64_t cycles) {
  if (!P || P->tag != GWQ_TAG_PACKED || !P->priv) return GWQ_ERR_INVALID_ARG;
  static_cast<gwq_priv*>(P->priv)->wait_cycles = cycles < 0 ? GWQ_DEFAULT_WAIT_CYCLES : (long long)cycles;
  return GWQ_OK;
}

extern "C" void gwq_free(void* obj) {
  if (!obj) return;
  const uint32_t tag = *static_cast<const uint32_t*>(obj);
  if (tag == GWQ_TAG_OUTLIERS) {
    gwq_delete_outliers(static_cast<gwq_outliers*>(obj));
  } else if (tag == GWQ_TAG_PACKED) {
    gwq_packed* P = static_cast<gwq_packed*>(obj);
    gwq_priv* pv = static_cast<gwq_priv*>(P->priv);
    gwq_dev_free(P->codes);   // the start of the one allocation with all arrays of the layer
    gwq_delete_outliers(P->S);
    if (pv) {
      gwq_dev_free(pv->x_stage);
      gwq_dev_free(pv->y_stage);
      gwq_dev_free(pv->ws_stage);
      delete pv;
    }
    P->tag = 0;
    delete P;
  }
}

extern "C" const char* gwq_status_string(gwq_status s) {
  switch (s) {
    case GWQ_OK: return "GWQ_OK";
    case GWQ_ERR_INVALID_ARG: return "GWQ_ERR_INVALID_ARG";
    case GWQ_ERR_UNSUPPORTED: return "GWQ_ERR_UNSUPPORTED";
    case GWQ_ERR_ALLOC: return "GWQ_ERR_ALLOC";
    case GWQ_ERR_NONFINITE: return "GWQ_ERR_NONFINITE";
    case GWQ_ERR_TIMEOUT: return "GWQ_ERR_TIMEOUT";
    case GWQ_ERR_CUDA: return "GWQ_ERR_CUDA";
    case GWQ_ERR_WORKSPACE: return "GWQ_ERR_WORKSPACE";
  }
  return "GWQ_ERR_UNKNOWN";
}
