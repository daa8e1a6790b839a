// Stage A2: doublets ("cells").  Every hit is paired with the hits of each adjacent
// layer that pass the cuts D0..D4 (Sec. 2.2.1, Fig. 2: the chain's first combinatorial
// step joins hits of neighbouring layers two by two).
//
// The search runs from the outer hit of each pair towards its inner layers, so that
// the cells ending on one hit come out contiguous: for each outer hit and inner-layer
// slot, one segment of cells ordered by inner hit.  The link stage then finds the cells
// arriving at a middle hit in its own segments, with no scatter by outer hit and no
// returning atomic per cell.
//
// Candidates are the inner-layer hits of an azimuthal window that can pass D1 and D2:
// a circle through the beam spot with curvature <= kmax turns by at most
// asin(kmax*ro/2) - asin(kmax*ri/2) between radii ri < ro (and every radius of this
// detector lies on the first half of such a circle, which D1 keeps), so with ri bounded
// below by the smallest radius seen on the inner layer in this event the window is
// asin(kmax*ro/2) - asin(kmax*ri_min/2), plus a safety margin, either side of the hit.
// It is one contiguous range of the sorted hits, or two when it wraps, taken in
// increasing index order.  Lanes stride over it, test the exact float32 cuts and stage
// the passing inner hits in shared memory; the segment is then appended with one
// reservation per (hit, inner slot).  Slots are reserved through a per-warp chunk
// allocator; a slot that no segment covers is a hole.  A cell is written as its inner hit
// alone (4 bytes): the segment names its outer hit, and its link state starts with its
// first link.
#include "ptca_internal.cuh"

namespace ptca {

namespace {

constexpr float kTwoPi = 6.28318530717958647692f;
constexpr float kHalfPi = 1.57079632679489661923f;
constexpr int kWarpsPerBlock = 8;

// Azimuthal window of outer hit `ho` (global bin gb, azimuth phi, asin_o = asin(kmax*ro/2),
// +inf where kmax*ro/2 >= 0.7) towards inner slot k of its layer: the range [x, y) of the
// sorted hits, or, with kWindowWraps in x, from x to the inner layer's end and from its start
// to y; y may carry kWindowExact (window_flag).  Empty where the inner layer has no hit inside
// the outer hit's radius, or none of its r-z extent can pass D2 and D3 with the outer hit.
__device__ __forceinline__ uint2 reverse_window(const Buffers& b, const pt_cuts& cuts,
                                                const PairTable& pt, int32_t B,
                                                float bins_per_rad, uint32_t gb, float4 ho,
                                                float asin_o, float phi, int k) {
  const int el = gb / B;  // event*10 + layer
  const int e = el / kLayers, L = el - e * kLayers;
  uint2 r = make_uint2(0u, 0u);
  const int Li = pt.inner[L][k];
  const float ri_min = __uint_as_float(b.layer_rmin[e * kLayers + Li]);
  const float ri_max = __uint_as_float(b.layer_rmax[e * kLayers + Li]);
  if (!(ho.w > ri_min)) return r;  // D0 fails for every hit of the inner layer
  if (!rz_box_reachable(cuts, ho.w, ho.z, ri_min, ri_max,
                        float_from_order_key(b.layer_zmin[e * kLayers + Li]),
                        float_from_order_key(b.layer_zmax[e * kLayers + Li]), false))
    return r;
  float win = kHalfPi + 1e-3f;     // where the curvature bound is void, D1's
  if (asin_o != __int_as_float(0x7f800000))
    win = fminf(asin_o - b.layer_asin_lo[e * kLayers + Li] + 1e-4f, win);
  const uint32_t base = (uint32_t)(e * kLayers + Li) * (uint32_t)B;
  const int2 w = window_bins(phi, win, bins_per_rad, B);
  const uint32_t wraps = w.x < 0 || w.y > B ? kWindowWraps : 0u;
  r.x = b.bin_start[base + (w.x < 0 ? w.x + B : w.x)] | wraps;
  r.y = b.bin_start[base + (w.y > B ? w.y - B : w.y)] |
        window_flag(cuts, win, bins_per_rad, ho.w, ri_min, ri_max);
  return r;
}

// The windows of sorted hit s on a layer with nin inner layers (global bin gb), given to
// put(k, window).
template <class Put>
__device__ __forceinline__ void reverse_windows(const Buffers& b, const pt_cuts& cuts,
                                                const PairTable& pt, int32_t B, uint32_t gb,
                                                float4 ho, int nin, uint32_t n_sorted, Put put) {
  const float bins_per_rad = (float)B / kTwoPi;
  const float a = 0.5f * cuts.kmax * ho.w;
  const float asin_o = a >= 0.7f ? __int_as_float(0x7f800000) : asinf(a);
  const float phi = azimuth(ho);
  for (int k = 0; k < nin; ++k) {
    uint2 rg = reverse_window(b, cuts, pt, B, bins_per_rad, gb, ho, asin_o, phi, k);
    const uint32_t rx = rg.x & ~kWindowWraps, ry = rg.y & ~kWindowExact;
    if (!PT_CHECK(b.cnt, (rx <= ry || (rg.x & kWindowWraps)) && rx <= n_sorted && ry <= n_sorted,
                  DBG_DBL_WINDOW))
      rg = make_uint2(0u, 0u);
    put(k, rg);
  }
}

// The windows of every sorted hit, one thread per hit, into the slots that the search then
// overwrites with the hit's segments; the slots that the hit's layer does not use are written
// empty.  In the search a chunk's windows take the instructions of searching one or two hits,
// on as few lanes as the chunk has hits.  The whole call in us with the windows found here
// (in the search): 64 pileup-200 events 5439 (5516), 7 gap-pair events 1109 (1133), one
// pileup-200 event 320 (326); but one pileup-50 event 188 (185), where the launch costs more,
// so contexts of fewer than kWindowsMinHits hits have no such launch.  A small batch in a
// larger context does: an event of 200 hits 88 us with it and 90 without, of 10139 hits 132 to
// 137 and 128.
constexpr int64_t kWindowsMinHits = 32768;
__global__ void k_windows(Buffers b, pt_cuts cuts, PairTable pt, int32_t B) {
  pdl_sync();
  const uint32_t n_sorted = b.bin_start[b.hdr->n_events * kLayers * B];
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n_sorted;
       s += gridDim.x * blockDim.x) {
    const uint32_t gb = b.hbin[s];
    const int nin = pt.n_inner[(gb / (uint32_t)B) % kLayers];
    uint2* seg = b.seg + (uint64_t)s * pt.max_inner;
    reverse_windows(b, cuts, pt, B, gb, b.hit4[s], nin, n_sorted,
                    [&](int k, uint2 rg) { seg[k] = rg; });
    for (int k = nin; k < pt.max_inner; ++k) seg[k] = make_uint2(0u, 0u);
  }
}

// Warps take chunks of a few consecutive sorted (outer) hits (search_chunk), every one from a
// work counter.  The chunk's windows are read (WINDOWS: k_windows has run) or found
// lane-parallel, one hit per lane, and kept in shared memory; the warp then searches them hit
// by hit.
template <bool WINDOWS>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, 5)
    k_doublets(Buffers b, pt_cuts cuts, PairTable pt, int32_t B, uint64_t cap_cells) {
  pdl_wait();
  __shared__ uint32_t st_val[kWarpsPerBlock][kStage];
  __shared__ uint2 st_rng[kWarpsPerBlock][32][kMaxInner];
  __shared__ float4 st_hit[kWarpsPerBlock][32];
  __shared__ uint8_t st_nin[kWarpsPerBlock][32];  // inner layers of each hit's layer
  const int lane = lane_id(), wib = threadIdx.x >> 5;
  uint32_t* sval = st_val[wib];
  const unsigned lt_mask = (1u << lane) - 1u;

  const int E = b.hdr->n_events;
  const uint32_t n_sorted = b.bin_start[E * kLayers * B];
  WarpChunk ch;

  const uint32_t n_warps = gridDim.x * kWarpsPerBlock;
  for (uint32_t s0 = 0;;) {
    const uint32_t per = search_chunk(n_sorted - s0, n_warps);
    if (lane == 0) s0 = (uint32_t)atomicAdd(&b.cnt[CNT_DBL_WORK], (unsigned long long)per);
    s0 = __shfl_sync(kFull, s0, 0);
    if (s0 >= n_sorted) break;
    const uint32_t nh = min(per, n_sorted - s0);
    __syncwarp();
    if ((uint32_t)lane < nh) {
      const uint32_t s = s0 + lane;
      const uint32_t gb = b.hbin[s];
      const float4 ho = b.hit4[s];
      const int nin = pt.n_inner[(gb / (uint32_t)B) % kLayers];
      st_hit[wib][lane] = ho;
      st_nin[wib][lane] = (uint8_t)nin;
      if (WINDOWS) {
        for (int k = 0; k < nin; ++k)
          st_rng[wib][lane][k] = b.seg[(uint64_t)s * pt.max_inner + k];
      } else {
        reverse_windows(b, cuts, pt, B, gb, ho, nin, n_sorted,
                        [&](int k, uint2 rg) { st_rng[wib][lane][k] = rg; });
      }
    }
    __syncwarp();

    for (uint32_t j = 0; j < nh; ++j) {
      const uint32_t s = s0 + j;
      const float4 ho = st_hit[wib][j];
      const int nin = st_nin[wib][j];
      const float half_k = 0.5f * cuts.kmax * ho.w;
      // the slots the hit's layer does not use are written empty, so readers need not
      // know the hit's layer
      if (!WINDOWS && lane >= nin && lane < pt.max_inner)
        b.seg[(uint64_t)s * pt.max_inner + lane] = make_uint2(0u, 0u);
      for (int k = 0; k < nin; ++k) {
        const uint2 win = st_rng[wib][j][k];
        const float tiny = window_tiny(win.y);
        uint4 rg = make_uint4(win.x & ~kWindowWraps, win.y & ~kWindowExact, 0u, 0u);
        if (win.x & kWindowWraps) {
          // the inner layer's bins: its start up to y, and x up to its end
          const uint32_t el = b.hbin[s] / (uint32_t)B;
          const uint32_t first = (el - el % kLayers + pt.inner[el % kLayers][k]) * (uint32_t)B;
          rg = make_uint4(b.bin_start[first], rg.y, rg.x, b.bin_start[first + B]);
        }
        uint32_t cnt = 0;
        // pass 1: test, stage up to kStage passing hits, count all; two candidates per
        // lane in flight (both loads issued before either test)
        for (int part = 0; part < 2; ++part) {
          const uint32_t beg = part ? rg.z : rg.x, end = part ? rg.w : rg.y;
          for (uint32_t i0 = beg; i0 < end; i0 += 64) {
            float4 hv[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const uint32_t i = i0 + 32 * u + lane;
              hv[u] = i < end ? b.hit4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const uint32_t i = i0 + 32 * u + lane;
              const bool pass =
                  doublet_quick(cuts, i < end, hv[u], ho, half_k, hv[u].w, tiny);
              const unsigned bal = __ballot_sync(kFull, pass);
              if (pass) {
                const uint32_t pos = cnt + __popc(bal & lt_mask);
                if (pos < kStage) sval[pos] = i;
              }
              cnt += __popc(bal);
            }
          }
        }

        uint32_t seg_off = 0, seg_cnt = 0;
        if (cnt > 0) {
          const unsigned long long base =
              chunk_take(ch, &b.cnt[CNT_CELLS], cnt, search_ahead(n_sorted, s + 1));
          if (base + cnt > cap_cells) {
            if (lane == 0) atomicOr(&b.cnt[CNT_STATUS], ST_CELLS);
          } else if (cnt <= (uint32_t)kStage) {
            __syncwarp();
            for (uint32_t i = lane; i < cnt; i += 32)
              if (PT_CHECK(b.cnt, base + i < cap_cells, DBG_DBL_CELL))
                b.cell_in[base + i] = sval[i];
            seg_off = (uint32_t)base;
            seg_cnt = cnt;
          } else {
            // too many for the stage: recompute and write in test order
            uint32_t pos0 = 0;
            for (int part = 0; part < 2; ++part) {
              const uint32_t beg = part ? rg.z : rg.x, end = part ? rg.w : rg.y;
              for (uint32_t i0 = beg; i0 < end; i0 += 32) {
                const uint32_t i = i0 + lane;
                const bool pass = i < end && doublet_pass(cuts, b.hit4[i], ho);
                const unsigned bal = __ballot_sync(kFull, pass);
                if (pass && PT_CHECK(b.cnt, base + pos0 + __popc(bal & lt_mask) < cap_cells,
                                     DBG_DBL_CELL))
                  b.cell_in[base + pos0 + __popc(bal & lt_mask)] = i;
                pos0 += __popc(bal);
              }
            }
            seg_off = (uint32_t)base;
            seg_cnt = cnt;
          }
        }
        if (lane == 0) b.seg[(uint64_t)s * pt.max_inner + k] = make_uint2(seg_off, seg_cnt);
        __syncwarp();
      }
    }
  }
  if (lane == 0 && ch.total) atomicAdd(&b.cnt[CNT_CELLS_USED], (unsigned long long)ch.total);
}

}  // namespace

void launch_doublets(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s) {
  constexpr unsigned block = kWarpsPerBlock * 32;
  if (p.max_hits >= kWindowsMinHits)
    PT_TRACE(l, s, "k_doublets",
             launch_pdl(k_windows, l.grid, 256, 0, s, b, p.cuts, p.pairs, p.phi_bins),
             launch_pdl(k_doublets<true>, l.sgrid, block, 0, s, b, p.cuts, p.pairs, p.phi_bins,
                        (uint64_t)p.max_cells));
  else
    PT_TRACE(l, s, "k_doublets",
             launch_pdl(k_doublets<false>, l.sgrid, block, 0, s, b, p.cuts, p.pairs, p.phi_bins,
                        (uint64_t)p.max_cells));
}

}  // namespace ptca
