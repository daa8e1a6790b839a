// Stage A1: load + bin.  Hits of a batch are counting-sorted by (event, layer, phi bin)
// into a (x, y, z, r) float4 array so that the doublet search reads each outer-layer
// azimuthal window as one contiguous range (Sec. 2.2.1, Fig. 2: hits per layer are
// paired with hits of the adjacent layer).  r = sqrt(x*x + y*y) in correctly rounded
// float32; the azimuth is used for binning only, never inside a cut.
#include "ptca_internal.cuh"

namespace ptca {

namespace {

constexpr float kPi = 3.14159265358979323846f;

// The four input arrays in one launch, four hits per thread in flight.  It lengthens the whole
// chain by 7 us on 64 pileup-200 events (34 MB) and by 10 on 64 pileup-50 events (8.5 MB), a
// copy per array by 33 and 30.
constexpr int kTake = 4;
__global__ void k_take_inputs(Buffers b, const float* __restrict__ x, const float* __restrict__ y,
                              const float* __restrict__ z, const uint8_t* __restrict__ layer,
                              int64_t n) {
  pdl_sync();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kTake * stride) {
    float v[kTake][3];
    uint8_t u[kTake];
#pragma unroll
    for (int k = 0; k < kTake; ++k) {
      const int64_t i = i0 + k * stride;
      if (i >= n) break;
      v[k][0] = x[i], v[k][1] = y[i], v[k][2] = z[i], u[k] = layer[i];
    }
#pragma unroll
    for (int k = 0; k < kTake; ++k) {
      const int64_t i = i0 + k * stride;
      if (i >= n) break;
      b.in_x[i] = v[k][0], b.in_y[i] = v[k][1], b.in_z[i] = v[k][2], b.in_layer[i] = u[k];
    }
  }
}

// Reset per-batch counters and the histogram / flag arrays, sized from the header.
__global__ void k_clear(Buffers b, int32_t phi_bins) {
  pdl_sync();
  const int E = b.hdr->n_events, N = b.hdr->n_hits;
  const int nb = E * kLayers * phi_bins;
  const int stride = gridDim.x * blockDim.x;
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = t0; i <= nb; i += stride) b.bin_cnt[i] = 0;
  for (int i = t0; i < kScanBlocks; i += stride) b.scan_part[i] = 0;
  for (int i = t0; i < E * kLayers; i += stride) {
    b.layer_rmax[i] = 0u;
    b.layer_rmin[i] = 0x7f800000u;  // +inf
    b.layer_zmin[i] = 0xffffffffu;
    b.layer_zmax[i] = 0u;
  }
  if (b.nt_head) {  // a caller that stops at the doublets has no ntuplet arrays
    for (int i = t0; i < N; i += stride) {
      b.nt_head[i] = kHole;
      b.used[i] = 0;
    }
    for (int i = t0; i <= N; i += stride) b.sv_cnt[i] = 0;
  }
  if (t0 == 0) {
    b.cnt[CNT_CELLS] = 0;
    b.cnt[CNT_LINKS] = 0;
    b.cnt[CNT_NT] = 0;
    b.cnt[CNT_STATUS] = 0;
    b.cnt[CNT_DEBUG_SITE] = 0;
    b.cnt[CNT_GATE_KEPT] = 0;
    b.cnt[CNT_SCAN_NT] = 0;
    b.cnt[CNT_SV] = 0;
    b.cnt[CNT_NT_BEST] = 0;
    b.cnt[CNT_NT_TIES] = 0;
    b.cnt[CNT_CELLS_USED] = 0;
    b.cnt[CNT_LINKS_USED] = 0;
    b.cnt[CNT_DBL_WORK] = 0;
    b.cnt[CNT_LNK_WORK] = 0;
    if (!b.hdr->raw) b.cnt[CNT_RAW_STATUS] = 0;
    b.cnt[CNT_SCAN_BINS] = (unsigned long long)nb;
    b.cnt[CNT_SCAN_HITS] = (unsigned long long)N;
  }
}

__device__ __forceinline__ float hit_radius(float x, float y) {
  return fsqrt(fadd(fmul(x, x), fmul(y, y)));
}

// r and z range of a layer of one event in one block, as the global arrays hold them.
struct LayerRange {
  uint32_t rmax, rmin, zmin, zmax;
};

// Histogram: global bin of every input hit and its rank inside the bin; the r and z ranges
// per (event, layer).  Inputs that the caller has on the device (or that came up with the
// header) are read where they are and copied to the context's arrays here, instead of by
// four copies of their own.
//
// A block takes consecutive hits, so that it meets one event, seldom two or three: the
// ranges are gathered in shared memory and go to the global arrays once per event and block
// (a warp's hits lie on some ten layers, and four global atomics for each of them were most
// of the kernel: 64 pileup-200 events 93 us, now 38), and the event of a tile is
// looked up once where all its hits share it.  The sums that the scan of the counts starts
// from, one per share of the bins, come from here as well, counted in shared memory, which
// saves the scan its first pass and launch.
constexpr int kCountThreads = 256;
__global__ void __launch_bounds__(kCountThreads) k_bin_count(Buffers b, int32_t B) {
  pdl_sync();
  __shared__ LayerRange s_range[kLayers];
  __shared__ uint32_t s_share[kScanBlocks];
  const int E = b.hdr->n_events, N = b.hdr->n_hits;
  const uint32_t share = (uint32_t)scan_share((uint64_t)E * kLayers * B);
  for (int i = threadIdx.x; i < kScanBlocks; i += kCountThreads) s_share[i] = 0;
  const float scale = (float)B / (2.0f * kPi);
  const bool copy = b.hdr->x != nullptr;
  const float* X = copy ? b.hdr->x : b.in_x;
  const float* Y = copy ? b.hdr->y : b.in_y;
  const float* Z = copy ? b.hdr->z : b.in_z;
  const uint8_t* LAY = copy ? b.hdr->layer : b.in_layer;
  auto reset = [&]() {
    if (threadIdx.x < kLayers) s_range[threadIdx.x] = {0u, 0x7f800000u, 0xffffffffu, 0u};
  };
  auto flush = [&](int e) {  // all threads; the ranges gathered for event e
    __syncthreads();
    if (threadIdx.x < kLayers && e >= 0) {
      const LayerRange v = s_range[threadIdx.x];
      const int i = e * kLayers + threadIdx.x;
      if (v.zmax || v.zmin != 0xffffffffu) {
        atomicMax(&b.layer_rmax[i], v.rmax);
        atomicMin(&b.layer_rmin[i], v.rmin);
        atomicMax(&b.layer_zmax[i], v.zmax);
        atomicMin(&b.layer_zmin[i], v.zmin);
      }
    }
    reset();
    __syncthreads();
  };
  reset();
  __syncthreads();
  const int tiles = (N + kCountThreads - 1) / kCountThreads;
  const int per = (tiles + (int)gridDim.x - 1) / (int)gridDim.x;
  const int t0 = min(tiles, per * (int)blockIdx.x), t1 = min(tiles, t0 + per);
  int e_now = -1;  // the event that s_range belongs to (-1: none)
  for (int tile = t0; tile < t1; ++tile) {
    const int first = tile * kCountThreads, last = min(N, first + kCountThreads) - 1;
    if (e_now < 0 || first >= b.hit_off[e_now + 1]) {
      if (e_now >= 0) flush(e_now);
      e_now = find_event(b.hit_off, E, first);
    }
    const bool whole = last < b.hit_off[e_now + 1];  // all of the tile lies in e_now
    const int g = first + threadIdx.x;
    if (g > last) continue;
    const int L = LAY[g];
    const float x = X[g], y = Y[g], z = Z[g];
    if (copy) {
      b.in_x[g] = x;
      b.in_y[g] = y;
      b.in_z[g] = z;
      b.in_layer[g] = (uint8_t)L;
    }
    if (L >= kLayers) {
      atomicOr(&b.cnt[CNT_STATUS], ST_LAYER);
      b.in_bin[g] = 0xffffffffu;
      continue;
    }
    const int e = whole || g < b.hit_off[e_now + 1] ? e_now : find_event(b.hit_off, E, g);
    const float r = hit_radius(x, y);
    const uint32_t zk = float_order_key(z);
    int bin = (int)floorf((atan2f(y, x) + kPi) * scale);
    bin = bin < 0 ? 0 : (bin >= B ? B - 1 : bin);
    const uint32_t key = (uint32_t)(e * kLayers + L);
    const uint32_t gb = key * (uint32_t)B + (uint32_t)bin;
    b.in_bin[g] = gb;
    b.in_rank[g] = atomicAdd(&b.bin_cnt[gb], 1u);
    atomicAdd(&s_share[gb / share], 1u);
    // r >= 0, so the integer order of the bit patterns is the float order
    if (e == e_now) {
      // most hits lie inside the range gathered so far
      LayerRange& v = s_range[L];
      const uint32_t rb = __float_as_uint(r);
      if (rb > v.rmax) atomicMax(&v.rmax, rb);
      if (rb < v.rmin) atomicMin(&v.rmin, rb);
      if (zk > v.zmax) atomicMax(&v.zmax, zk);
      if (zk < v.zmin) atomicMin(&v.zmin, zk);
    } else {
      atomicMax(&b.layer_rmax[key], __float_as_uint(r));
      atomicMin(&b.layer_rmin[key], __float_as_uint(r));
      atomicMax(&b.layer_zmax[key], zk);
      atomicMin(&b.layer_zmin[key], zk);
    }
  }
  flush(e_now);
  for (int i = threadIdx.x; i < kScanBlocks; i += kCountThreads)
    if (s_share[i]) atomicAdd(&b.scan_part[i], s_share[i]);
}

__global__ void k_bin_scatter(Buffers b, float kmax) {
  pdl_sync();
  const int N = b.hdr->n_hits;
  const int stride = gridDim.x * blockDim.x;
  // per event layer: the outer- and inner-radius terms of the azimuthal windows of the
  // doublet search (inner term 0, the widest window, where the bound does not apply)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < b.hdr->n_events * kLayers; i += stride) {
    const float a = 0.5f * kmax * __uint_as_float(b.layer_rmax[i]);
    b.layer_asin[i] = a >= 0.7f ? __int_as_float(0x7f800000) : asinf(a);
    const float c = 0.5f * kmax * __uint_as_float(b.layer_rmin[i]);
    b.layer_asin_lo[i] = c < 0.7f ? asinf(c) : 0.0f;
  }
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < N; g += stride) {
    const uint32_t gb = b.in_bin[g];
    if (gb == 0xffffffffu) continue;
    const uint32_t s = b.bin_start[gb] + b.in_rank[g];
    if (!PT_CHECK(b.cnt, s < (uint32_t)N, DBG_BIN_SCATTER)) continue;
    const float x = b.in_x[g], y = b.in_y[g], z = b.in_z[g];
    b.hit4[s] = make_float4(x, y, z, hit_radius(x, y));
    b.perm[s] = (uint32_t)g;
    b.hbin[s] = gb;
  }
}

// ---------------------------------------------------------------- device scan
constexpr int kScanThreads = 512;

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* warp_sums,
                                                    uint32_t* total) {
  const int lane = lane_id(), w = threadIdx.x >> 5;
  const uint32_t inc = warp_incl_scan(v);
  if (lane == 31) warp_sums[w] = inc;
  __syncthreads();
  if (w == 0) {
    const uint32_t ws = lane < (kScanThreads / 32) ? warp_sums[lane] : 0u;
    const uint32_t wi = warp_incl_scan(ws);
    if (lane < (kScanThreads / 32)) warp_sums[lane] = wi - ws;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  const uint32_t r = warp_sums[w] + inc - v;
  __syncthreads();
  return r;
}

__device__ __forceinline__ void chunk_of(uint64_t n, uint64_t* lo, uint64_t* hi) {
  const uint64_t per = scan_share(n);
  *lo = min(n, per * blockIdx.x);
  *hi = min(n, *lo + per);
}

__device__ __forceinline__ uint4 scan_load(const uint32_t* in, uint64_t i, uint64_t hi, bool vec) {
  if (vec && i + 4 <= hi) return *(const uint4*)(in + i);
  return make_uint4(i < hi ? in[i] : 0u, i + 1 < hi ? in[i + 1] : 0u, i + 2 < hi ? in[i + 2] : 0u,
                    i + 3 < hi ? in[i + 3] : 0u);
}

// Sum of each block's share.
__global__ void __launch_bounds__(kScanThreads) k_scan_partial(const uint32_t* in, uint32_t* part,
                                                               const unsigned long long* n_dev) {
  pdl_sync();
  __shared__ uint32_t ws[kScanThreads / 32];
  __shared__ uint32_t tot;
  uint64_t lo, hi;
  chunk_of(*n_dev, &lo, &hi);
  const bool vec = ((uintptr_t)in & 15u) == 0;
  uint32_t acc = 0;
#pragma unroll 4
  for (uint64_t i = lo + 4 * threadIdx.x; i < hi; i += 4 * kScanThreads) {
    const uint4 v = scan_load(in, i, hi, vec);
    acc += v.x + v.y + v.z + v.w;
  }
  block_excl_scan(acc, ws, &tot);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// Each block adds up the shares before its own (no third launch for them) and scans its
// share, four entries per thread at a time.
__global__ void __launch_bounds__(kScanThreads) k_scan_final(const uint32_t* in, uint32_t* out,
                                                             const uint32_t* part,
                                                             const unsigned long long* n_dev) {
  pdl_sync();
  __shared__ uint32_t ws[kScanThreads / 32];
  __shared__ uint32_t tot;
  static_assert(kScanBlocks <= kScanThreads, "one partial sum per thread");
  const uint64_t n = *n_dev;
  uint64_t lo, hi;
  chunk_of(n, &lo, &hi);
  block_excl_scan(threadIdx.x < blockIdx.x ? part[threadIdx.x] : 0u, ws, &tot);
  uint32_t carry = tot;
  const bool vec_in = ((uintptr_t)in & 15u) == 0, vec_out = ((uintptr_t)out & 15u) == 0;
  for (uint64_t base = lo; base < hi; base += 4 * kScanThreads) {
    __syncthreads();  // tot has been read
    const uint64_t i = base + 4 * threadIdx.x;
    const uint4 v = scan_load(in, i, hi, vec_in);
    uint4 r;
    r.x = carry + block_excl_scan(v.x + v.y + v.z + v.w, ws, &tot);
    r.y = r.x + v.x;
    r.z = r.y + v.y;
    r.w = r.z + v.z;
    if (vec_out && i + 4 <= hi) {
      *(uint4*)(out + i) = r;
    } else {
      if (i < hi) out[i] = r.x;
      if (i + 1 < hi) out[i + 1] = r.y;
      if (i + 2 < hi) out[i + 2] = r.z;
      if (i + 3 < hi) out[i + 3] = r.w;
    }
    carry += tot;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = carry;
}

}  // namespace

void launch_scan(const uint32_t* in, uint32_t* out, const unsigned long long* n_dev,
                 uint32_t* part, cudaStream_t s) {
  launch_pdl(k_scan_partial, kScanBlocks, kScanThreads, 0, s, in, part, n_dev);
  launch_scan_counted(in, out, n_dev, part, s);
}

void launch_scan_counted(const uint32_t* in, uint32_t* out, const unsigned long long* n_dev,
                         const uint32_t* part, cudaStream_t s) {
  launch_pdl(k_scan_final, kScanBlocks, kScanThreads, 0, s, in, out, part, n_dev);
}

void launch_take_inputs(const Buffers& b, const float* x, const float* y, const float* z,
                        const uint8_t* layer, int64_t n, const Launch& l, cudaStream_t s) {
  launch_pdl(k_take_inputs, l.sms * 8, 256, 0, s, b, x, y, z, layer, n);
}

void launch_clear(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s) {
  PT_TRACE(l, s, "k_clear", launch_pdl(k_clear, l.grid, 256, 0, s, b, p.phi_bins));
}

void launch_bin_hits(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s) {
  PT_TRACE(l, s, "k_bin_count", launch_pdl(k_bin_count, l.grid, kCountThreads, 0, s, b, p.phi_bins));
  PT_TRACE(l, s, "scan", launch_scan_counted(b.bin_cnt, b.bin_start, &b.cnt[CNT_SCAN_BINS],
                                           b.scan_part, s));
  PT_TRACE(l, s, "k_bin_scatter", launch_pdl(k_bin_scatter, l.grid, 256, 0, s, b, p.cuts.kmax));
}

namespace {
__global__ void k_debug_inject(Buffers b, unsigned site) {
#ifdef PT_DEBUG
  debug_fail(b.cnt, site);
#endif
}
}  // namespace

cudaError_t launch_debug_inject(const Buffers& b, unsigned site, cudaStream_t s) {
  k_debug_inject<<<1, 1, 0, s>>>(b, site);
  return cudaGetLastError();
}

}  // namespace ptca
