// Shared host/device helpers of the GWQ library (internal; not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gwq.h"

#define GWQ_TAG_OUTLIERS 0x4F515747u /* "GWQO" */
#define GWQ_TAG_PACKED 0x50515747u   /* "GWQP" */

// Needs a local `gwq_status st` and a label `fail`.
#define GWQ_CUDA_TRY(expr)                                                    \
  do {                                                                        \
    cudaError_t e__ = (expr);                                                 \
    if (e__ != cudaSuccess) {                                                 \
      (void)cudaGetLastError();                                               \
      st = (e__ == cudaErrorMemoryAllocation) ? GWQ_ERR_ALLOC : GWQ_ERR_CUDA; \
      goto fail;                                                              \
    }                                                                         \
  } while (0)

// Kernel-private part of a packed layer.
struct gwq_priv {
  uint32_t* cv;          // per outlier: fp16 value << 16 | column (NULL when K > 65536)
  void* x_stage;         // staging for gwq_linear_host
  void* y_stage;
  size_t x_stage_bytes;
  size_t y_stage_bytes;
  uint32_t* sz_t;        // [K/group][N]: scale fp16 bits | zero-point << 16 (tensor-core path)
  uint32_t* szp;         // the same words for the streaming kernel: [tile of 16 rows][step of 128 columns][row & 7]
                         // [group of the step][row >> 3], rows past the last one zero (NULL where it takes no call)
  void* ws_stage;        // scratch for gwq_linear_host where the product needs some
  size_t ws_stage_bytes;
  void* xt;              // scratch of the decode kernels (transposed activations) for calls without a workspace
  uint32_t* tb;          // outliers ordered by tile of 16 rows and step of 128 columns: fp16 value << 16 | column << 4 | row
  int32_t* tb_ptr;       // [tiles * steps + 1] extents of the blocks in tb (K a multiple of 128)
  int32_t* dev_status;   // device status word written by bounded waits
  int sm_count;
  long long wait_cycles; // SM cycles a bounded device-side wait may spin (gwq_set_wait_limit)
};

#define GWQ_DEFAULT_WAIT_CYCLES (1000LL * 1000LL * 1000LL)

static inline bool gwq_aligned16(const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

// Device memory of library objects, from a bounded pool (alloc.cu).  gwq_dev_free waits for the device as cudaFree does.
cudaError_t gwq_dev_alloc(void** p, size_t bytes, cudaStream_t stream);
void gwq_dev_free_async(void* p, cudaStream_t stream);
void gwq_dev_free(void* p);
// Pinned host words that a kernel or a copy writes its result to; NULL when there is no memory.
#define GWQ_PINNED_SLOT_BYTES 64
void* gwq_pinned_slot();
void gwq_pinned_slot_return(void* slot);

// Up to eight arrays copied by one kernel; starts are multiples of 16 bytes.
cudaError_t gwq_copy_arrays(int count, const void* const* from, void* const* to, const size_t* bytes, cudaStream_t stream);

// Cuts one allocation into arrays whose starts are multiples of 256 bytes: first pass with base NULL for the size.
struct gwq_carver {
  char* base;
  size_t used;
  template <typename T>
  T* take(size_t count) {
    T* p = base ? reinterpret_cast<T*>(base + used) : nullptr;
    used += (count * sizeof(T) + 255) / 256 * 256;
    return p;
  }
};

// An outlier object with its three arrays in one allocation (row_ptr holds its start), made on `stream`.
gwq_status gwq_new_outliers(int32_t N, int32_t K, int64_t nnz, cudaStream_t stream, gwq_outliers** out);
void gwq_delete_outliers(gwq_outliers* S);

// Kernel launchers implemented in the other translation units.
gwq_status gwq_launch_simt(const gwq_packed* P, const void* x, gwq_dtype xd, int M, void* y,
                           gwq_dtype yd, cudaStream_t stream);
// scratch: gwq_stream_scratch_bytes, not read where every layer's activations are staged (and with one token)
gwq_status gwq_launch_decode_multi(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M,
                                   void* const* y, gwq_dtype yd, void* scratch, cudaStream_t stream);
bool gwq_decode_stages(const gwq_packed* const* P, int count, int M);   // it serves the call without scratch
bool gwq_decode_ahead(const gwq_packed* P, gwq_dtype xd, int M);   // the kernel with a CTA per tile is the faster one for (P, xd, M)
gwq_status gwq_launch_prefill(const gwq_packed* P, const void* x, gwq_dtype xd, int M, void* y,
                              gwq_dtype yd, void* ws, size_t ws_bytes, cudaStream_t stream);
size_t gwq_prefill_workspace_bytes(const gwq_packed* P, gwq_dtype xd, int M);
bool gwq_skinny_takes(const gwq_packed* P, gwq_dtype xd, int M);   // the tcgen05 decode kernel has a variant for (P, xd, M)
bool gwq_skinny_ahead(const gwq_packed* P, gwq_dtype xd, int M);   // ... and is the fastest one
bool gwq_skinny_before(const gwq_packed* P, gwq_dtype xd, int M);  // ... and has always served the call
size_t gwq_skinny_workspace_bytes(const gwq_packed* const* P, int count, gwq_dtype xd, int M);
gwq_status gwq_launch_skinny(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y,
                             gwq_dtype yd, void* ws, cudaStream_t stream);
bool gwq_takes_decode(const gwq_packed* P, gwq_dtype xd, int M);   // one of the two mma.sync decode kernels serves (P, xd, M) without a workspace
bool gwq_stream_takes(const gwq_packed* P, int M);   // the streaming kernel has a variant for (P, M)
size_t gwq_stream_scratch_bytes(int K);              // scratch of a call of several tokens, for either decode kernel
gwq_status gwq_launch_stream(const gwq_packed* const* P, int count, const void* x, gwq_dtype xd, int M, void* const* y,
                             gwq_dtype yd, void* scratch, cudaStream_t stream);
