// Outlier location for small fractions in one read of G (Section 3.2, Eq. "o"): same result as the radix select of
// select.cu, entry for entry.
//
// The radix select reads G five times (three digits, row counts, emission).  Here a sample of 128-byte lines, spread
// evenly over the columns and at random over the rows, gives a key below the k-th largest one with a margin of a
// quarter; ONE pass over G then keeps the entries from that key on (about 1.3 k of them) and everything after it works
// on those, which fit the L2 cache.  Whether enough and not too many entries were kept is known afterwards on the
// device: if not (an unlucky sample, masses of equal magnitudes), the host is told and runs the radix select instead.
//
// The pass is bound by the read of G.  11008 x 4096, 1 %: 1000 -> 115 us a call with the object's allocation,
// 4096 x 4096: 520 -> 70 us.
#include "common.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kSampleBins = 4096;     // of the sampled keys: exponent and four bits of the fraction
constexpr int kSampleShift = 19;
constexpr int kSampleLines = 8192;    // lines of 32 entries
constexpr int kCoarseBins = 2048;     // of the kept keys, from the lowest kept one on
constexpr int kCoarseShift = 14;
constexpr int kFineBins = 1 << kCoarseShift;   // one key each, inside the coarse bin of the threshold
constexpr int kChunk = 1024;          // consecutive entries (flat index) of one warp
constexpr int kCounterPitch = 64;     // words between counters: atomics on one line of the L2 queue up (44000 of them: 60 us)
constexpr int kKeepCtas = 4;          // of the pass over G on an SM
constexpr int kRegions = 16;          // of the list of kept entries, each with a counter of its own
constexpr int kFineCtas = 24;         // CTAs per region of the fine histogram
constexpr int kGroupChunks = 256;     // chunks of one CTA of the counting kernel
constexpr int kEmitSplit = 16;        // CTAs of the emitting kernel that share such a group: two chunks per warp, whose
                                      // chains of dependent reads (about 2 us each) are what that kernel's time is

struct State {
  unsigned int lo;            // lowest kept key
  unsigned int coarse;        // coarse bin that holds the k-th largest key
  unsigned int k_rem;         // entries still to take in it, then among those equal to the threshold
  unsigned int thr;           // the k-th largest key
  unsigned int failed;        // the kept entries do not decide the selection
  unsigned int done[3];       // CTAs that have finished, per kernel with a last step
  unsigned int count[kRegions * kCounterPitch];   // kept entries of region r at r * kCounterPitch
};

struct Work {   // device scratch; `state`, `sample`, `coarse`, `fine` are cleared first
  State* state;
  unsigned int *sample, *coarse, *fine;
  unsigned int *key, *at;             // kept entries: key and flat index
  uint2* chunk;                       // per chunk: where its kept entries start, how many there are
  uint2* part;                        // per chunk: selected entries before it in its group: above / equal
  uint2* total;                       // per group of chunks: above / equal
  unsigned int region;                // capacity of a region
};

__device__ __forceinline__ unsigned int abs_key(unsigned int bits) { return bits & 0x7FFFFFFFu; }

// True in every thread of the CTA that finishes last; its reads then see what the other CTAs wrote.
__device__ bool last_cta(unsigned int* done) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// The highest bin b with at least k entries in bins >= b, and the entries above b; false if there are fewer than k in
// all.  Every thread takes BINS / kThreads neighbouring bins.
template <int BINS>
__device__ bool find_bin(const unsigned int* hist, unsigned int k, unsigned int* bin, unsigned int* above) {
  constexpr int PER = BINS / kThreads;
  __shared__ unsigned int warp_sum[kWarps], found[2];
  const int t = kThreads - 1 - threadIdx.x;   // thread 0 has the highest bins
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned int h[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; i += 4) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(hist + t * PER + i));
    h[i] = v.x; h[i + 1] = v.y; h[i + 2] = v.z; h[i + 3] = v.w;
    sum += v.x + v.y + v.z + v.w;
  }
  unsigned int inc = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int u = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) warp_sum[warp] = inc;
  if (threadIdx.x == 0) found[0] = 0xFFFFFFFFu;
  __syncthreads();
  unsigned int before = inc - sum;
  for (int w = 0; w < warp; ++w) before += warp_sum[w];
  if (before < k && before + sum >= k) {   // one thread at most
#pragma unroll
    for (int i = PER - 1; i >= 0; --i) {
      if (before < k && before + h[i] >= k) {
        found[0] = t * PER + i;
        found[1] = before;
      }
      before += h[i];
    }
  }
  __syncthreads();
  *bin = found[0];
  *above = found[1];
  return found[0] != 0xFFFFFFFFu;
}

// Spreads the sampled rows: the 32-bit integer hash "lowbias32" of C. Wellons' hash-prospector (published, public domain).
__device__ __forceinline__ unsigned int mix(unsigned int x) {
  x ^= x >> 16; x *= 0x7FEB352Du;
  x ^= x >> 15; x *= 0x846CA68Bu;
  return x ^ (x >> 16);
}

// Histogram of the sampled lines: for each of the K / 32 column blocks `rows` rows, one at random out of each of as
// many equal stretches (all rows when there are no more).  The last CTA sets the lowest key to keep, so that about
// `want` of the sampled entries lie above.
__global__ void __launch_bounds__(kThreads) sample_kernel(const uint4* __restrict__ G4, int N, int K, int rows,
                                                          unsigned int want, const Work w) {
  __shared__ unsigned int sh[kSampleBins];
  for (int i = threadIdx.x; i < kSampleBins; i += kThreads) sh[i] = 0;
  __syncthreads();
  const int blocks = K / 32;
  const int n = blocks * rows * 8;   // 16-byte pieces
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
    const int line = i >> 3, j = line / blocks, cb = line - j * blocks;
    const int r0 = (int)((long long)N * j / rows), r1 = (int)((long long)N * (j + 1) / rows);
    const int row = r0 + (int)(mix(line) % (unsigned)(r1 - r0));
    const uint4 v = __ldg(G4 + (long long)row * (K / 4) + cb * 8 + (i & 7));
    atomicAdd(&sh[abs_key(v.x) >> kSampleShift], 1u);
    atomicAdd(&sh[abs_key(v.y) >> kSampleShift], 1u);
    atomicAdd(&sh[abs_key(v.z) >> kSampleShift], 1u);
    atomicAdd(&sh[abs_key(v.w) >> kSampleShift], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kSampleBins; i += kThreads)
    if (sh[i]) atomicAdd(&w.sample[i], sh[i]);
  if (!last_cta(&w.state->done[0])) return;
  unsigned int bin, above;
  const bool ok = find_bin<kSampleBins>(w.sample, want, &bin, &above);
  if (threadIdx.x == 0) w.state->lo = ok ? bin << kSampleShift : 0u;
}

// The pass over G: a warp takes a chunk of 1024 consecutive entries (eight 16-byte loads per lane), appends the kept
// ones to the chunk's region and counts them by coarse bin.  The next chunk is requested before the current one's
// chain (region counter, the kept entries once more from the cache) begins: without that the SMs waited for memory
// with two fifths of the copy rate reached (11008 x 4096: 65 us; now 41).  The last CTA finds the coarse bin of the threshold.
__global__ void __launch_bounds__(kThreads, kKeepCtas) keep_kernel(const uint4* __restrict__ G4, unsigned int numel,
                                                                   unsigned int chunks, unsigned int k, const Work w) {
  __shared__ unsigned int sh[kCoarseBins];
  const int lane = threadIdx.x & 31;
  const unsigned int n4 = numel / 4, stride = gridDim.x * kWarps;
  uint4 v[8];
  auto fetch = [&](const unsigned int c) {
    const unsigned int base4 = c * (kChunk / 4) + lane;
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = base4 + u * 32 < n4 ? __ldg(G4 + base4 + u * 32) : make_uint4(0u, 0u, 0u, 0u);
  };
  unsigned int c = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (c < chunks) fetch(c);
  for (int i = threadIdx.x; i < kCoarseBins; i += kThreads) sh[i] = 0;
  __syncthreads();
  const unsigned int lo = w.state->lo;
  const float lo_f = __uint_as_float(lo);
  for (; c < chunks; c += stride) {
    const unsigned int base4 = c * (kChunk / 4) + lane;
    // bit 4u + e: entry e of load u is kept.  |g| and the lowest key compare as floats as they do as keys, infinities
    // and (the comparison being unordered) NaN included.
    unsigned int m = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      m |= (fabsf(__uint_as_float(v[u].x)) < lo_f ? 0u : 1u) << (4 * u);
      m |= (fabsf(__uint_as_float(v[u].y)) < lo_f ? 0u : 2u) << (4 * u);
      m |= (fabsf(__uint_as_float(v[u].z)) < lo_f ? 0u : 4u) << (4 * u);
      m |= (fabsf(__uint_as_float(v[u].w)) < lo_f ? 0u : 8u) << (4 * u);
    }
    if (c == chunks - 1) {   // the last chunk may be short
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (base4 + u * 32 >= n4) m &= ~(15u << (4 * u));
    }
    if (c + stride < chunks) fetch(c + stride);
    const unsigned int mine = __popc(m);
    unsigned int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int up = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += up;
    }
    const unsigned int total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    const unsigned int region = c % kRegions;
    unsigned int start = 0;
    if (lane == 0 && total) start = atomicAdd(&w.state->count[region * kCounterPitch], total);
    start = __shfl_sync(0xFFFFFFFFu, start, 0);
    const bool fits = start + total <= w.region;
    if (lane == 0) {
      w.chunk[c] = make_uint2(region * w.region + start, fits ? total : 0u);
      if (!fits) w.state->failed = 1u;
    }
    if (!fits) continue;
    // few are kept (one lane in three has one): walking the set bits and reading those entries again, from the cache,
    // is cheaper than 32 predicated steps
    unsigned int pos = region * w.region + start + inc - mine;
    for (; m; m &= m - 1) {
      const int b = __ffs(m) - 1;
      const unsigned int flat = (base4 + (b >> 2) * 32) * 4 + (b & 3);
      const unsigned int key = abs_key(__ldg(reinterpret_cast<const unsigned int*>(G4) + flat));
      w.key[pos] = key;
      w.at[pos] = flat;
      ++pos;
      atomicAdd(&sh[min((key - lo) >> kCoarseShift, (unsigned)kCoarseBins - 1)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kCoarseBins; i += kThreads)
    if (sh[i]) atomicAdd(&w.coarse[i], sh[i]);
  if (!last_cta(&w.state->done[1])) return;
  unsigned int bin, above;
  const bool ok = find_bin<kCoarseBins>(w.coarse, k, &bin, &above);
  if (threadIdx.x == 0) {
    if (!ok || bin == kCoarseBins - 1) w.state->failed = 1u;   // the last bin has no upper end
    w.state->coarse = bin;
    w.state->k_rem = k - above;
  }
}

// Histogram by key of the kept entries of the threshold's coarse bin; lanes of a warp with equal keys add together, so
// that masses of equal magnitudes do not queue at one word.  The last CTA finds the threshold key.
__global__ void __launch_bounds__(kThreads) fine_kernel(const Work w) {
  const State* s = w.state;
  if (__ldcg(&s->failed)) return;
  const unsigned int first = s->lo + (s->coarse << kCoarseShift);
  const int r = blockIdx.x % kRegions;
  const unsigned int n = s->count[r * kCounterPitch];
  const unsigned int* key = w.key + (size_t)r * w.region;
  for (unsigned int i = blockIdx.x / kRegions * kThreads + threadIdx.x; i < n; i += gridDim.x / kRegions * kThreads) {
    const unsigned int d = __ldcg(key + i) - first;
    if (d < (unsigned)kFineBins) {
      const unsigned int same = __match_any_sync(__activemask(), d);
      if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&w.fine[d], (unsigned)__popc(same));
    }
  }
  if (!last_cta(&w.state->done[2])) return;
  unsigned int bin, above;
  const unsigned int k_rem = s->k_rem;
  const bool ok = find_bin<kFineBins>(w.fine, k_rem, &bin, &above);
  if (threadIdx.x == 0) {
    if (!ok) w.state->failed = 1u;
    w.state->thr = first + bin;
    w.state->k_rem = k_rem - above;   // of the entries equal to the threshold, the first k_rem are taken
  }
}

// Exclusive scan of pairs over a CTA of kGroupChunks threads.
__device__ uint2 scan_pairs(uint2 v, uint2* total) {
  __shared__ uint2 sums[kGroupChunks / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint2 inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int x = __shfl_up_sync(0xFFFFFFFFu, inc.x, o), y = __shfl_up_sync(0xFFFFFFFFu, inc.y, o);
    if (lane >= o) {
      inc.x += x;
      inc.y += y;
    }
  }
  if (lane == 31) sums[warp] = inc;
  __syncthreads();
  uint2 before = make_uint2(inc.x - v.x, inc.y - v.y), all = make_uint2(0u, 0u);
  for (int i = 0; i < kGroupChunks / 32; ++i) {
    const uint2 s = sums[i];
    if (i < warp) before = make_uint2(before.x + s.x, before.y + s.y);
    all = make_uint2(all.x + s.x, all.y + s.y);
  }
  *total = all;
  __syncthreads();
  return before;
}

// Per chunk (one thread): kept entries above the threshold and equal to it, as prefixes inside the group of chunks.
__global__ void __launch_bounds__(kGroupChunks) count_kernel(unsigned int chunks, const Work w) {
  if (__ldcg(&w.state->failed)) return;
  const unsigned int thr = w.state->thr;
  const unsigned int c = blockIdx.x * kGroupChunks + threadIdx.x;
  uint2 n = make_uint2(0u, 0u);
  if (c < chunks) {
    const uint2 where = w.chunk[c];
    for (unsigned int i = 0; i < where.y; ++i) {
      const unsigned int key = w.key[where.x + i];
      n.x += key > thr;
      n.y += key == thr;
    }
  }
  uint2 total;
  const uint2 before = scan_pairs(n, &total);
  if (c < chunks) w.part[c] = before;
  if (threadIdx.x == 0) w.total[blockIdx.x] = total;
}

// Writes the CSR arrays, one warp per chunk: the chunk's selected entries are marked in a bit map of its 1024 places,
// whose prefix counts are the positions in flat-index order; a row that starts inside the chunk gets its pointer from
// the same counts.
__global__ void __launch_bounds__(kGroupChunks) emit_kernel(const uint16_t* __restrict__ W, unsigned int numel,
                                                            unsigned int K, unsigned int chunks, const Work w,
                                                            int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                                                            uint16_t* __restrict__ val, unsigned int* host_failed) {
  __shared__ unsigned int gt_map[kWarps][32], tie_map[kWarps][32];
  const unsigned int failed = __ldcg(&w.state->failed);
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *host_failed = failed;
  if (failed) return;
  // selected entries before this group of chunks
  uint2 base = make_uint2(0u, 0u);
  for (unsigned int g = threadIdx.x; g < blockIdx.x; g += kGroupChunks) {
    const uint2 t = w.total[g];
    base = make_uint2(base.x + t.x, base.y + t.y);
  }
  uint2 all;
  scan_pairs(base, &all);
  const unsigned int thr = w.state->thr, ties = w.state->k_rem;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < kGroupChunks / kEmitSplit; i += kWarps) {
    const unsigned int c = blockIdx.x * kGroupChunks + blockIdx.y * (kGroupChunks / kEmitSplit) + i;
    if (c >= chunks) return;
    const uint2 where = w.chunk[c], part = w.part[c];
    const unsigned int gt0 = all.x + part.x, tie0 = all.y + part.y, flat0 = c * kChunk;
    // a chunk touches two rows at most where K >= kChunk: one division then serves all its entries
    const unsigned int row0 = flat0 / K, col0 = flat0 - row0 * K;
    const bool wide = K >= (unsigned)kChunk;
    gt_map[warp][lane] = 0u;
    tie_map[warp][lane] = 0u;
    __syncwarp();
    for (unsigned int j = lane; j < where.y; j += 32) {
      const unsigned int key = w.key[where.x + j], p = w.at[where.x + j] - flat0;
      if (key > thr) atomicOr(&gt_map[warp][p >> 5], 1u << (p & 31));
      else if (key == thr) atomicOr(&tie_map[warp][p >> 5], 1u << (p & 31));
    }
    __syncwarp();
    const unsigned int gt = gt_map[warp][lane], tie = tie_map[warp][lane];   // places 32 lane .. 32 lane + 31
    unsigned int gt_before = __popc(gt), tie_before = __popc(tie);
    const unsigned int own_gt = gt_before, own_tie = tie_before;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int x = __shfl_up_sync(0xFFFFFFFFu, gt_before, o), y = __shfl_up_sync(0xFFFFFFFFu, tie_before, o);
      if (lane >= o) {
        gt_before += x;
        tie_before += y;
      }
    }
    gt_before += gt0 - own_gt;
    tie_before += tie0 - own_tie;
    for (unsigned int left = gt | tie; left; left &= left - 1) {
      const int b = __ffs(left) - 1;
      const unsigned int below = (1u << b) - 1u;
      const unsigned int t = tie_before + __popc(tie & below);
      if (((tie >> b) & 1u) && t >= ties) continue;   // enough entries equal to the threshold came before
      const unsigned int pos = gt_before + __popc(gt & below) + min(t, ties);
      const unsigned int flat = flat0 + lane * 32 + b;
      const unsigned int col = col0 + lane * 32 + b;
      col_idx[pos] = (int32_t)(wide ? (col >= K ? col - K : col) : flat % K);
      val[pos] = __ldg(W + flat);
    }
    // K is a multiple of 32: a row can only start at the first place of a lane
    const unsigned int flat = flat0 + lane * 32;
    const bool starts = wide ? col0 + lane * 32 == K || (col0 | lane) == 0u : flat % K == 0;
    if (flat < numel && starts) row_ptr[wide ? row0 + (col0 ? 1 : 0) : flat / K] = (int32_t)(gt_before + min(tie_before, ties));
    if (flat + 32 == numel)
      row_ptr[numel / K] = (int32_t)(gt_before + __popc(gt) + min(tie_before + (unsigned)__popc(tie), ties));
    __syncwarp();
  }
}

struct Plan {
  int rows;               // sampled rows per column block
  unsigned int want;      // sampled entries above the lowest kept key
  unsigned int chunks, groups, region;
};

Plan plan(int N, int K, unsigned int k) {
  Plan p;
  const long long blocks = K / 32, lines = blocks * N;
  long long rows = kSampleLines / blocks;
  if (rows < 1) rows = 1;
  if (rows > N) rows = N;
  p.rows = (int)rows;
  const double part = (double)(blocks * rows) / (double)lines;   // of the matrix that is sampled
  const double in_sample = (double)k * part;
  double root = 1.0;
  while (root * root < in_sample) root *= 1.25;   // within a quarter above the square root
  p.want = (unsigned)(1.25 * in_sample + 4.0 * root + 16.0);
  const long long numel = (long long)N * K;
  p.chunks = (unsigned)((numel + kChunk - 1) / kChunk);
  p.groups = (p.chunks + kGroupChunks - 1) / kGroupChunks;
  // three times the entries expected (keys of one sample bin are kept together), evenly over the regions
  const double most = 3.0 * (double)p.want / part + 65536.0;
  const double cap = most < (double)numel ? most : (double)numel;
  p.region = (unsigned)(cap / kRegions) + kChunk;
  return p;
}

Work carve(gwq_carver& c, const Plan& p) {
  Work w;
  w.state = c.take<State>(1);
  w.sample = c.take<unsigned int>(kSampleBins);
  w.coarse = c.take<unsigned int>(kCoarseBins);
  w.fine = c.take<unsigned int>(kFineBins);
  w.key = c.take<unsigned int>((size_t)p.region * kRegions);
  w.at = c.take<unsigned int>((size_t)p.region * kRegions);
  w.chunk = c.take<uint2>(p.chunks);
  w.part = c.take<uint2>(p.chunks);
  w.total = c.take<uint2>(p.groups);
  w.region = p.region;
  return w;
}

}  // namespace

// Up to one entry in eight: beyond, the kept entries stop being few.  Below 2^18 entries the whole selection is
// launches, of which the radix select has no more that matter.
bool gwq_select_fast_takes(int N, int K, unsigned int k) {
  const long long numel = (long long)N * K;
  return numel >= (1 << 18) && k >= 1 && (long long)k <= numel / 8;
}

size_t gwq_select_fast_bytes(int N, int K, unsigned int k) {
  gwq_carver c = {nullptr, 0};
  carve(c, plan(N, K, k));
  return c.used;
}

// Queues the selection; after the stream has been synchronised *host_failed (pinned) says whether the outputs stand.
cudaError_t gwq_select_fast_run(const uint16_t* W, const float* G, int N, int K, unsigned int k, int32_t* row_ptr,
                                int32_t* col_idx, uint16_t* val, void* scratch, unsigned int* host_failed, int sm_count,
                                cudaStream_t stream) {
  const Plan p = plan(N, K, k);
  gwq_carver c = {static_cast<char*>(scratch), 0};
  const Work w = carve(c, p);
  const uint4* G4 = reinterpret_cast<const uint4*>(G);
  const unsigned int numel = (unsigned)((long long)N * K);
  const size_t cleared = (size_t)(reinterpret_cast<char*>(w.key) - static_cast<char*>(scratch));
  cudaError_t e = cudaMemsetAsync(scratch, 0, cleared, stream);
  if (e != cudaSuccess) return e;
  const int pieces = K / 32 * p.rows * 8;
  int sample_grid = (pieces + kThreads * 2 - 1) / (kThreads * 2);
  if (sample_grid > sm_count) sample_grid = sm_count;
  sample_kernel<<<sample_grid, kThreads, 0, stream>>>(G4, N, K, p.rows, p.want, w);
  const unsigned int want_ctas = (p.chunks + kWarps - 1) / kWarps, most_ctas = (unsigned)sm_count * kKeepCtas;
  keep_kernel<<<want_ctas < most_ctas ? want_ctas : most_ctas, kThreads, 0, stream>>>(G4, numel, p.chunks, k, w);
  fine_kernel<<<kRegions * kFineCtas, kThreads, 0, stream>>>(w);
  count_kernel<<<p.groups, kGroupChunks, 0, stream>>>(p.chunks, w);
  emit_kernel<<<dim3(p.groups, kEmitSplit), kGroupChunks, 0, stream>>>(W, numel, (unsigned)K, p.chunks, w, row_ptr, col_idx, val,
                                                     host_failed);
  return cudaGetLastError();
}
