// Primary vertices of the fitted tracks (Sec. 2.2.1: vertex reconstruction is the last
// of Patatrack's sub-algorithms, and the chain returns the reconstructed tracks and
// vertices, Fig. 2).  The paper gives no algorithm; the library's reading:
//   [V1] an event's tracks with at least min_hits hits and a finite z0 take part;
//   [V2] they are ordered by z0 (ties: position in the event's canonical track order)
//        and the ordered list is cut where the float32 step to the next z0 exceeds dz
//        (single-linkage clustering in z0);
//   [V3] every group of at least two tracks is a vertex: z = mean z0, sum of pT^2,
//        number of tracks; vertices in order of z; every used track records its vertex.
//
// One block of 1024 threads per event.  The selected tracks' (z0, position) keys are
// sorted in shared memory (up to 16384 per event): a counting sort into 16384 buckets of
// equal z width, each track held in registers while the array is rewritten in place, then
// every track's rank among the few of its bucket.  The buckets span the event's z0 range
// inside +-1.25 z0max (the outer ones take what lies beyond); an event that puts more than
// 512 tracks into one bucket is sorted bitonically instead, which any keys suit but which
// takes 91 passes over 8192 tracks.  A block scan numbers the groups of two or more, and
// a warp sums each vertex (float32, the lanes' sums added pairwise).  The vertices of
// event e go to a staging area at floor(t0 / 2) (an event with T tracks has at most T / 2
// vertices); a second kernel places them in one batch-wide list (each block adds up the
// events before its own) and turns each track's vertex into a batch-wide index.
//
// Bound by the latency of the passes of one block.  12 pileup-200 events (9.8k
// tracks each): 52 + 7 us, against 328 us for the bitonic sort with one thread per vertex
// and 31 us for a scan and a placing kernel of one block per event.
#include <algorithm>

#include "ptca_internal.cuh"

namespace ptca {

namespace {

constexpr int kVtxThreads = 1024;
constexpr int kVtxMax = 16384;                    // selected tracks per event
constexpr int kVtxPer = kVtxMax / kVtxThreads;    // scan elements per thread
constexpr int kVtxBucketMax = 512;                // tracks of one bucket that are ranked directly
// keys (8 bytes), buckets / scan array (4 bytes), first track of each vertex (2 bytes)
constexpr size_t kVtxSmem = (size_t)kVtxMax * 12 + (size_t)kVtxMax / 2 * 2;

// In-place exclusive scan of a[0, per * kVtxThreads), `per` <= kVtxPer consecutive entries per
// thread (FULL: kVtxPer of them, read four at a time); returns the total.  All threads of the
// block take part.
template <bool FULL>
__device__ uint32_t vtx_block_scan_of(uint32_t* a, int per, uint32_t* warp_tot) {
  if (FULL) per = kVtxPer;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint32_t loc[kVtxPer];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kVtxPer; ++i) {
    if (i >= per) break;
    loc[i] = a[t * per + i];
    s += loc[i];
  }
  const uint32_t inc = warp_incl_scan(s);
  if (lane == 31) warp_tot[w] = inc;
  __syncthreads();
  if (w == 0) {
    const uint32_t x = warp_tot[lane];
    const uint32_t xi = warp_incl_scan(x);
    warp_tot[lane] = xi - x;
    if (lane == 31) warp_tot[32] = xi;
  }
  __syncthreads();
  uint32_t run = warp_tot[w] + inc - s;
#pragma unroll
  for (int i = 0; i < kVtxPer; ++i) {
    if (i >= per) break;
    a[t * per + i] = run;
    run += loc[i];
  }
  const uint32_t total = warp_tot[32];
  __syncthreads();
  return total;
}

__device__ __forceinline__ uint32_t vtx_block_scan(uint32_t* a, int per, uint32_t* warp_tot) {
  return per == kVtxPer ? vtx_block_scan_of<true>(a, per, warp_tot)
                        : vtx_block_scan_of<false>(a, per, warp_tot);
}

// Sorts key[0, n) bitonically, padded to a power of two.
__device__ __noinline__ void vtx_bitonic(unsigned long long* key, uint32_t n) {
  uint32_t P = 1;
  while (P < n) P <<= 1;
  for (uint32_t i = n + threadIdx.x; i < P; i += kVtxThreads) key[i] = ~0ull;
  __syncthreads();
  for (uint32_t k = 2; k <= P; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t i = threadIdx.x; i < P; i += kVtxThreads) {
        const uint32_t l = i ^ j;
        if (l > i) {
          const unsigned long long a = key[i], c = key[l];
          if ((a > c) == ((i & k) == 0)) {
            key[i] = c;
            key[l] = a;
          }
        }
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kVtxThreads) k_vertex_event(Buffers b, int32_t min_hits,
                                                              float dz, float z_range,
                                                              uint64_t cap_nt) {
  pdl_sync();
  extern __shared__ unsigned char vsm[];
  unsigned long long* key = reinterpret_cast<unsigned long long*>(vsm);  // [kVtxMax]
  uint32_t* vf = reinterpret_cast<uint32_t*>(vsm + (size_t)kVtxMax * 8);  // [kVtxMax]
  uint16_t* vstart = reinterpret_cast<uint16_t*>(vsm + (size_t)kVtxMax * 12);  // [kVtxMax / 2]
  __shared__ uint32_t warp_tot[33];
  __shared__ uint32_t s_n, s_lo, s_hi, s_full;
  const int e = blockIdx.x, tid = threadIdx.x;
  if (e == 0 && tid == 0) b.cnt[CNT_SCAN_EV] = (unsigned long long)gridDim.x;
  // the event's tracks, clamped to the cleaned ntuplets of the batch
  const int64_t S = (int64_t)min(b.cnt[CNT_SV], (unsigned long long)cap_nt);
  const int64_t t0 = min(max(b.ev_nt_off[e], (int64_t)0), S);
  const int64_t nt = min(max(b.ev_nt_off[e + 1], t0), S) - t0;
  // Buckets, and so the length of the scans, follow the event's size, up to four per track:
  // 1000 events of 200 hits take 33 us, 77 with 16384 buckets for every event.
  const int per = (int)min((int64_t)kVtxPer, max((int64_t)1, (nt + 255) / 256));
  const int nb = per * kVtxThreads;  // >= nt, or kVtxMax
  if (tid == 0) {
    s_n = 0;
    s_lo = ~0u;
    s_hi = 0;
    s_full = 0;
  }
#pragma unroll
  for (int j = 0; j < kVtxPer; ++j) {
    if (j >= per) break;
    vf[tid + j * kVtxThreads] = 0;
  }
  __syncthreads();
  // [V1] the tracks that take part, keyed by (z0, position)
  uint32_t zlo = ~0u, zhi = 0;
#pragma unroll 4
  for (int64_t i = tid; i < nt; i += kVtxThreads) {
    const pt_track& tr = b.tracks[t0 + i];
    const float z0 = tr.z0;
    b.trk_vtx[t0 + i] = -1;
    if ((int)tr.nhits >= min_hits && isfinite(z0)) {
      const uint32_t k = atomicAdd(&s_n, 1u);
      const uint32_t o = float_order_key(z0);
      zlo = min(zlo, o);
      zhi = max(zhi, o);
      if (k < (uint32_t)kVtxMax) key[k] = ((unsigned long long)o << 32) | (uint32_t)i;
    }
  }
  zlo = __reduce_min_sync(kFull, zlo);
  zhi = __reduce_max_sync(kFull, zhi);
  if ((tid & 31) == 0) {
    atomicMin(&s_lo, zlo);
    atomicMax(&s_hi, zhi);
  }
  __syncthreads();
  const uint32_t n = s_n;
  if (n > (uint32_t)kVtxMax) {
    if (tid == 0) {
      atomicOr(&b.cnt[CNT_STATUS], ST_VTX);
      b.ev_nv[e] = 0;
    }
    return;
  }
  // [V2] sort
  auto zk = [&](uint32_t k) { return float_from_order_key((uint32_t)(key[k] >> 32)); };
  const float lo = fmaxf(float_from_order_key(s_lo), -z_range);
  const float hi = fminf(float_from_order_key(s_hi), z_range);
  // buckets per cm (0: all tracks in one bucket); a track's bucket does not fall as z0 grows
  const float scale = hi > lo ? __fdividef((float)nb, hi - lo) : 0.0f;
  auto bucket = [&](unsigned long long v) {
    const float x = __fmul_rn(__fsub_rn(float_from_order_key((uint32_t)(v >> 32)), lo), scale);
    return (uint32_t)min(nb - 1, max(0, __float2int_rz(x)));
  };
  {
    unsigned long long v[kVtxPer];
    uint32_t br[kVtxPer];  // bucket << 16 | rank
    bool full = false;
#pragma unroll
    for (int j = 0; j < kVtxPer; ++j) {
      const uint32_t k = tid + j * kVtxThreads;
      if (k >= n) break;
      v[j] = key[k];
      const uint32_t bk = bucket(v[j]);
      const uint32_t rank = atomicAdd(&vf[bk], 1u);
      full |= rank >= (uint32_t)kVtxBucketMax;
      br[j] = bk << 16 | rank;
    }
    if (full) s_full = 1;
    __syncthreads();
    if (s_full) {
      vtx_bitonic(key, n);
    } else {
      vtx_block_scan(vf, per, warp_tot);
#pragma unroll
      for (int j = 0; j < kVtxPer; ++j) {
        if ((uint32_t)tid + j * kVtxThreads >= n) break;
        key[vf[br[j] >> 16] + (br[j] & 0xffffu)] = v[j];
      }
      __syncthreads();
      // rank among the bucket's tracks
#pragma unroll
      for (int j = 0; j < kVtxPer; ++j) {
        const uint32_t k = tid + j * kVtxThreads;
        if (k >= n) break;
        v[j] = key[k];
        const uint32_t bk = bucket(v[j]);
        const uint32_t first = vf[bk], last = bk + 1 < (uint32_t)nb ? vf[bk + 1] : n;
        br[j] = first;
        for (uint32_t q = first; q < last; ++q) br[j] += key[q] < v[j] ? 1u : 0u;
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kVtxPer; ++j) {
        if ((uint32_t)tid + j * kVtxThreads >= n) break;
        key[br[j]] = v[j];
      }
      __syncthreads();
    }
  }
  auto starts = [&](uint32_t k) { return k == 0 || fsub(zk(k), zk(k - 1)) > dz; };
  // a group start whose group holds at least two tracks marks a vertex
  for (uint32_t k = tid; k < (uint32_t)nb; k += kVtxThreads) {
    uint32_t f = 0;
    if (k + 1 < n && starts(k)) f = !starts(k + 1);
    vf[k] = f;
  }
  __syncthreads();
  const uint32_t nv = vtx_block_scan(vf, per, warp_tot);
  for (uint32_t k = tid; k < n; k += kVtxThreads)
    if ((k + 1 < n ? vf[k + 1] : nv) > vf[k]) vstart[vf[k]] = (uint16_t)k;
  __syncthreads();
  // [V3] one warp per vertex; its tracks record it
  const int64_t vbase = t0 / 2;
  const uint32_t lane = lane_id();
  for (uint32_t v = tid >> 5; v < nv; v += kVtxThreads / 32) {
    const uint32_t k = vstart[v];
    float zs = 0.0f, p2 = 0.0f;
    uint32_t size = 0;
    for (uint32_t m0 = k;; m0 += 32) {
      const uint32_t m = m0 + lane;
      const unsigned in = __ballot_sync(kFull, m < n && (m == k || !starts(m)));
      const uint32_t take = __ffs(~in) ? __ffs(~in) - 1 : 32;  // the group goes on so far
      if (lane < take) {
        const uint32_t i = (uint32_t)key[m];
        const float pt = b.tracks[t0 + i].pt;
        zs = fadd(zs, zk(m));
        p2 = fadd(p2, fmul(pt, pt));
        b.trk_vtx[t0 + i] = (int32_t)v;
      }
      size += take;
      if (take < 32) break;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      zs = fadd(zs, __shfl_xor_sync(kFull, zs, o));
      p2 = fadd(p2, __shfl_xor_sync(kFull, p2, o));
    }
    if (lane == 0) {
      pt_vertex out;
      out.z = fdiv(zs, (float)size);
      out.sum_pt2 = p2;
      out.n_tracks = (int32_t)size;
      out.event = e;
      b.vtx_stage[vbase + v] = out;
    }
  }
  if (tid == 0) b.ev_nv[e] = nv;
}

// Event e's vertices to the batch-wide list after those of the events before it; its
// tracks' vertices become batch-wide indices; per-event offsets as int64 and the total
// count.  blockIdx.y shares an event's tracks among blocks.  A block of up to kPlaceSum events
// adds up the counts before its own itself; more events have them scanned first (SCANNED,
// ev_nv[e] = vertices before event e), since those sums grow with the square of the events.
constexpr int kPlaceThreads = 256;
constexpr int kPlaceBlocks = 8;
constexpr int kPlaceSum = 2048;
template <bool SCANNED>
__global__ void __launch_bounds__(kPlaceThreads) k_vertex_compact(Buffers b, uint64_t cap_nt) {
  pdl_sync();
  __shared__ uint32_t s_sum[kPlaceThreads / 32];
  const int e = blockIdx.x, E = gridDim.x;
  const int64_t S = (int64_t)min(b.cnt[CNT_SV], (unsigned long long)cap_nt);
  const int64_t t0 = min(max(b.ev_nt_off[e], (int64_t)0), S);
  const int64_t t1 = min(max(b.ev_nt_off[e + 1], t0), S);
  uint32_t v0 = 0, nv;
  if (SCANNED) {
    v0 = b.ev_nv[e];
    nv = b.ev_nv[e + 1] - v0;
  } else {
    uint32_t sum = 0;
    for (int i = threadIdx.x; i < e; i += kPlaceThreads) sum += b.ev_nv[i];
    sum = __reduce_add_sync(kFull, sum);
    if (lane_id() == 0) s_sum[threadIdx.x >> 5] = sum;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPlaceThreads / 32; ++i) v0 += s_sum[i];
    nv = b.ev_nv[e];
  }
  const uint32_t first = blockIdx.y * kPlaceThreads + threadIdx.x;
  const uint32_t step = kPlaceThreads * gridDim.y;
  for (uint32_t v = first; v < nv; v += step) b.vtx[v0 + v] = b.vtx_stage[t0 / 2 + v];
#pragma unroll 4
  for (int64_t t = t0 + first; t < t1; t += step) {
    const int32_t v = b.trk_vtx[t];
    if (v >= 0) b.trk_vtx[t] = v + (int32_t)v0;
  }
  if (first == 0) {
    b.ev_vtx_off[e] = (int64_t)v0;
    if (e == E - 1) {
      b.ev_vtx_off[E] = (int64_t)(v0 + nv);
      b.cnt[CNT_VTX] = v0 + nv;
    }
  }
}

}  // namespace

cudaError_t launch_vertices(const Buffers& b, const Params& p, int n_events, int32_t min_hits,
                            float dz, const Launch& l, cudaStream_t s) {
  if (n_events < 1) return cudaSuccess;
  const uint64_t cap_nt = (uint64_t)p.max_ntuplets;
  cudaError_t err = cudaFuncSetAttribute(k_vertex_event,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVtxSmem);
  if (err != cudaSuccess) return err;
  PT_TRACE(l, s, "k_vertex_event",
           launch_pdl(k_vertex_event, n_events, kVtxThreads, kVtxSmem, s, b, min_hits, dz,
                      1.25f * p.cuts.z0max, cap_nt));
  // blocks for an event's tracks: enough to fill the GPU where the events do not
  const dim3 grid(n_events, std::max(1, std::min(kPlaceBlocks, kPlaceBlocks * l.sms / n_events)));
  if (n_events <= kPlaceSum) {
    PT_TRACE(l, s, "k_vertex_compact",
             launch_pdl(k_vertex_compact<false>, grid, kPlaceThreads, 0, s, b, cap_nt));
  } else {
    PT_TRACE(l, s, "scan",
             launch_scan(b.ev_nv, b.ev_nv, &b.cnt[CNT_SCAN_EV], b.scan_part, s));
    PT_TRACE(l, s, "k_vertex_compact",
             launch_pdl(k_vertex_compact<true>, grid, kPlaceThreads, 0, s, b, cap_nt));
  }
  return cudaGetLastError();
}

}  // namespace ptca
