// Stage A3: cellular-automaton links.  Cell a = (h0, h1) is linked to cell
// b = (h1, h2) when the three hits pass the r-z alignment cut C1, the curvature cut C2
// and the beam-spot distance cut C3 (Sec. 2.2.1, Fig. 2: doublets are paired into
// triplets by the cellular automaton).
//
// One warp per middle hit h1.  The cells arriving at h1 are its incoming segments
// (written contiguously by the doublet stage).  The cells leaving h1 are found again
// here by the doublet search towards its outer layers (the same window and exact cuts,
// so exactly the cells the doublet stage made), staged in shared memory with their
// outer hit and r-z slope, and ordered by slope with a counting sort into 128 buckets
// spanning the staged slopes.  With d1 = r1-r0, d2 = r2-r1 and t_a, t_b the slopes of
// a and b, C1 reads
//   d1 d2 |t_a - t_b| <= rz0 (d1 + d2) + rz1 |t_a d1 + t_b d2|,
// so |t_a - t_b| <= rz0 (1/d1 + 1/d2) + rz1 (|t_a|/d2 + |t_b|/d1).  Bounding |t_b| by
// cotmax (D4), or by |t_a| + |t_a - t_b| and solving for |t_a - t_b|, and d2 by the
// smallest r2-r1 of the staged cells, m, gives the window
//   |t_a - t_b| <= min((rz0 + rz1 cotmax)/d1 + (rz0 + rz1 |t_a|)/m,
//                      (rz0 + rz1 |t_a|)(1/d1 + 1/m) / (1 - rz1/d1)),
// the second term only where d1 > rz1.  It is widened by 1 % + 1e-3, far beyond the
// float32 rounding of C1 (about 4e-7 |t_a| d1/m + 1e-6) and of the approximate
// quotients used for the slopes and the window (a few 1e-7 relative).  Each lane takes
// one incoming cell and visits only the buckets its window overlaps (the bucket of a
// slope is a monotone function of it, evaluated the same way for the staged slopes and
// for the window's ends, which are moved out by a further 0.1 % + 1e-5 so that rounding
// of t_a -+ w cannot exclude a bucket); the staged cells there that fall inside the
// window are queued as (source cell, target) pairs.  A queued pair names its three hits,
// so the queue runs on across incoming groups and middle hits, and C1, C2 and C3 are
// tested only once 32 pairs are waiting, all lanes busy (about six pairs fall in the
// windows of a group of 32 incoming cells).  A link takes the next slot of the warp's
// reservation and is pushed onto its source's out-link list (CellState::head, Link::next),
// the list the ntuplet search walks; a cell's state is set up by the lane that holds the
// cell before any of its pairs is queued, and only then: three of four cells have no pair.
//
// The target cell (h1, h2) of a link is found afterwards, one thread per link, in h2's
// incoming segment from h1's layer (ordered by inner hit): in the warp's own path those
// dependent loads would hold up the search.  A middle hit with more outgoing cells than the
// stage holds is handled piece by piece, every piece staged once and visited by all of the
// incoming groups (staged again for each group, the search of 7 gap-pair events, with some
// 150 outgoing cells a hit, took 693 instead of 492 us).
#include "ptca_internal.cuh"

namespace ptca {

namespace {

constexpr float kTwoPi = 6.28318530717958647692f;
constexpr float kHalfPi = 1.57079632679489661923f;
constexpr int kConnWarps = 8;
constexpr int kConnBlocksPerSm = 4;  // up to 64 registers per thread
constexpr int kOut = 128;            // staged outgoing cells of one piece
constexpr int kNb = 128;             // slope buckets of a piece (a multiple of 32)
static_assert(kNb % 32 == 0, "buckets are scanned kNb / 32 per lane");
constexpr int kGroup = 8;            // middle hits whose windows are found at once
constexpr int kQueue = 64;           // window pairs waiting for C1-C3 (power of two)
static_assert(kOut % 32 == 0, "staged cells are sorted 32 at a time");
static_assert(kQueue >= 63 && (kQueue & (kQueue - 1)) == 0, "queue holds 31 + 32 entries");

// Azimuthal window of inner hit `hi` (global bin gb, azimuth phi) towards outer slot k, the doublet
// search's window from the inner side: the outer layer's asin(kmax*ro_max/2) less
// asin(kmax*ri/2) (+1e-4 rad).  It is the range [x, y) of the sorted hits, or, with
// kWindowWraps in x, from x to the outer layer's end and from its start to y; y may carry
// kWindowExact (window_flag).  Empty where the slot is unused, the outer layer ends inside
// the inner hit's radius, or none of its r-z extent can pass D2 and D3 with the inner hit.
__device__ __forceinline__ uint2 forward_window(const Buffers& b, const pt_cuts& cuts,
                                                const PairTable& pt, int32_t B,
                                                float bins_per_rad, uint32_t gb, float4 hi,
                                                float phi, int k) {
  const int el = gb / B;  // event*10 + layer
  const int e = el / kLayers, L = el - e * kLayers;
  uint2 r = make_uint2(0u, 0u);
  const int Lo = pt.outer[L][k];
  const float ro_max = __uint_as_float(b.layer_rmax[e * kLayers + Lo]);
  const float ro_min = __uint_as_float(b.layer_rmin[e * kLayers + Lo]);
  if (!(ro_max > hi.w)) return r;
  if (!rz_box_reachable(cuts, hi.w, hi.z, ro_min, ro_max,
                        float_from_order_key(b.layer_zmin[e * kLayers + Lo]),
                        float_from_order_key(b.layer_zmax[e * kLayers + Lo]), true))
    return r;
  const float asin_o = b.layer_asin[e * kLayers + Lo];
  float win = kHalfPi + 1e-3f;
  if (asin_o != __int_as_float(0x7f800000))
    win = fminf(asin_o - asinf(0.5f * cuts.kmax * hi.w) + 1e-4f, win);
  const uint32_t base = (uint32_t)(e * kLayers + Lo) * (uint32_t)B;
  const int2 w = window_bins(phi, win, bins_per_rad, B);
  const uint32_t wraps = w.x < 0 || w.y > B ? kWindowWraps : 0u;
  r.x = b.bin_start[base + (w.x < 0 ? w.x + B : w.x)] | wraps;
  r.y = b.bin_start[base + (w.y > B ? w.y - B : w.y)] |
        window_flag(cuts, win, bins_per_rad, hi.w, ro_min, ro_max);
  return r;
}

constexpr uint32_t kOnLayer0 = 0x80000000u;

// Per-warp shared state.
struct ConnWarp {
  float t[kOut];             // staged outgoing cells: r-z slope
  uint32_t code[kOut];       //   outer hit (sorted index) | slot of the middle hit's layer
                             //   among the outer hit's inner layers << 29
  float ts[kOut];            // slopes in bucket order
  uint32_t cs[kOut];         //   and codes
  uint32_t bstart[kNb + 1];  // first bucket-ordered position of each slope bucket
  uint4 q[kQueue];           // window pairs: source cell, target (outer hit | slot << 29),
                             //   middle hit, inner hit (with kOnLayer0 or without)
  uint2 rg[kGroup][kMaxOuter];  // forward windows of a group of middle hits, by outer slot
  uint32_t so[kMaxInner];    // middle hit: its incoming segments: first cell
  uint32_t sb[kMaxInner + 1];  //   incoming cells before each segment (the last: all)
  float tmin, scale, m;      // the staged piece: slope origin and scale of the buckets,
                             //   smallest r2 - r1
  unsigned long long chunk_next, chunk_end;  // link slots
  uint32_t used;             //   handed out
  uint32_t s0, per, dyn0;    // its chunk of sorted hits: first, size; the counter's first one
  float ahead;               //   search_ahead of the warp's hits
};

// Bucket of a slope (monotone non-decreasing in x): the same correctly rounded
// operations for the staged slopes and the window ends.
__device__ __forceinline__ int slope_bucket(float x, float tmin, float scale) {
  const int k = __float2int_rz(__fmul_rn(__fsub_rn(x, tmin), scale));
  return min(kNb - 1, max(0, k));
}

// Largest chunk of link slots a warp takes at once: a warp's last chunk is mostly
// unused (a hole), and link slots are scanned by the later stages.
constexpr uint32_t kLinkChunkMax = 256;

// Warp chunk reservation (as chunk_take) with the chunk state in shared memory, lane 0 acting.
__device__ __forceinline__ unsigned long long chunk_take_shared(
    ConnWarp& W, unsigned long long* counter, uint32_t n, unsigned long long* hlo,
    unsigned long long* hhi) {
  unsigned long long r = 0, lo = 0, hi = 0;
  if ((threadIdx.x & 31) == 0) {
    unsigned long long next = W.chunk_next, end = W.chunk_end;
    if (next + n > end) {
      lo = next;
      hi = end;
      const uint32_t want = chunk_size(n, W.used, W.ahead, kLinkChunkMax);
      next = atomicAdd(counter, (unsigned long long)want);
      end = next + want;
    }
    r = next;
    W.chunk_next = next + n;
    W.chunk_end = end;
    W.used += n;
  }
  r = __shfl_sync(kFull, r, 0);
  *hlo = __shfl_sync(kFull, lo, 0);
  *hhi = __shfl_sync(kFull, hi, 0);
  return r;
}

__global__ void __launch_bounds__(kConnWarps * 32, kConnBlocksPerSm)
    k_connect(Buffers b, pt_cuts cuts, PairTable pt, int32_t B, uint64_t cap_links) {
  pdl_wait();
  __shared__ ConnWarp s_w[kConnWarps];
  const int lane = lane_id();
  ConnWarp& W = s_w[threadIdx.x >> 5];
  const unsigned lt_mask = (1u << lane) - 1u;
  const int E = b.hdr->n_events;
  const uint32_t n_sorted = b.bin_start[E * kLayers * B];
  const float bins_per_rad = (float)B / kTwoPi;
  if (lane == 0) {
    W.chunk_next = W.chunk_end = 0;
    W.used = 0;
    W.ahead = 0.0f;
  }
  __syncwarp();
  auto mark_link_hole = [&](unsigned long long lo, unsigned long long hi) {
    hi = min(hi, (unsigned long long)cap_links);
    for (unsigned long long i = lo + lane; i < hi; i += 32) b.link[i].src = kHole;
  };
  // C1, C2 and C3 on nt queued pairs, one per lane, each with its hits, its source cell and
  // its target's slot, so that pairs of different incoming groups and middle hits share one
  // pass; a link is appended to its source's out-link list.
  uint32_t qhead = 0, qtail = 0;  // warp-uniform queue positions
  auto process = [&](uint32_t nt) {
    __syncwarp();
    const bool v = (uint32_t)lane < nt;
    const uint32_t qi = (qhead + lane) & (kQueue - 1);
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (v) e = W.q[qi];
    qhead += nt;
    __syncwarp();
    bool ok = false;
    float q = 0.0f;
    const uint32_t src = e.x;
    if (v) {
      const float4 q0 = b.hit4[e.w & ~kOnLayer0], q1 = b.hit4[e.z], q2 = b.hit4[e.y & 0x1fffffffu];
      ok = link_c1(cuts, q0, q1, q2) && link_c23(cuts, q0, e.w >> 31, q1, q2, q);
    }
    const unsigned pm = __ballot_sync(kFull, ok);
    const uint32_t n = __popc(pm);
    if (n) {
      unsigned long long hlo, hhi;
      const unsigned long long base = chunk_take_shared(W, &b.cnt[CNT_LINKS], n, &hlo, &hhi);
      mark_link_hole(hlo, hhi);
      if (base + n > cap_links) {
        if (lane == 0) atomicOr(&b.cnt[CNT_STATUS], ST_LINKS);
        mark_link_hole(base, base + n);  // slots below the capacity stay readable
      } else if (ok) {
        const uint64_t slot = base + __popc(pm & lt_mask);
        if (PT_CHECK(b.cnt, slot < cap_links, DBG_CON_LINK)) {
          *link_hi(&b.link[slot]) = make_uint4(src, e.y, e.z, __float_as_uint(q));
          b.link[slot].next = atomicExch(&b.cell[src].head, (uint32_t)slot);
        }
      }
    }
    __syncwarp();
  };

  const uint32_t n_warps = gridDim.x * kConnWarps;
  // chunks of sorted middle hits, the first by the warp's number, the others from a work
  // counter (the chunk in shared memory: the kernel has no registers left)
  if (lane == 0) {
    W.per = search_chunk(n_sorted, n_warps);
    W.dyn0 = W.per * n_warps;
    W.s0 = (blockIdx.x * kConnWarps + (threadIdx.x >> 5)) * W.per;
  }
  __syncwarp();
  for (;;) {
    const uint32_t s0 = W.s0, per = W.per;
    if (s0 >= n_sorted) break;
    // one round of loads finds the hits with incoming cells and outer layers
    uint32_t my_gb = 0;
    bool work = false;
    {
      const uint32_t s = s0 + lane;
      if ((uint32_t)lane < per && s < n_sorted) {
        my_gb = b.hbin[s];
        const int L = (my_gb / (uint32_t)B) % kLayers;
        if (pt.n_outer[L] > 0) {
          uint32_t any = 0;
          // slots past the layer's own inner layers are written empty
          for (int k = 0; k < pt.n_inner[L]; ++k) any |= b.seg[(uint64_t)s * pt.max_inner + k].y;
          work = any != 0;
        }
      }
    }
    unsigned todo = __ballot_sync(kFull, work);
    uint32_t group = 0xffffffffu;
    while (todo) {
      const int src = __ffs(todo) - 1;
      const uint32_t h1 = W.s0 + src;
      const uint32_t gb = __shfl_sync(kFull, my_gb, src);
      const int L1 = (gb / (uint32_t)B) % kLayers;
      const float4 p1 = b.hit4[h1];
      // h1's incoming segments, one slot per lane, and the cells before each
      const uint2 sgl = lane < pt.n_inner[L1] ? b.seg[(uint64_t)h1 * pt.max_inner + lane]
                                              : make_uint2(0u, 0u);
      if (h1 / kGroup != group) {
        // the windows of the group's hits that are in the chunk and have work, lanes over
        // hits and outer slots (hit by hit, a few lanes busy, they made the call on 64
        // pileup-200 events 170 us longer; groups of 16 or 32 gain nothing more)
        group = h1 / kGroup;
        const uint32_t h = group * kGroup + lane % kGroup;
        const uint32_t j = h - W.s0;
        const uint32_t hgb = __shfl_sync(kFull, my_gb, j & 31);
        __syncwarp();
        if (j < 32u && (todo >> j & 1u)) {
          const float4 p = b.hit4[h];
          const float phi = azimuth(p);
          const int n = pt.n_outer[(hgb / (uint32_t)B) % kLayers];
          for (int k = lane / kGroup; k < n; k += 32 / kGroup) {
            uint2 rg = forward_window(b, cuts, pt, B, bins_per_rad, hgb, p, phi, k);
            const uint32_t rx = rg.x & ~kWindowWraps, ry = rg.y & ~kWindowExact;
            if (!PT_CHECK(b.cnt, (rx <= ry || (rg.x & kWindowWraps)) && rx <= n_sorted &&
                                     ry <= n_sorted, DBG_CON_WINDOW))
              rg = make_uint2(0u, 0u);
            W.rg[lane % kGroup][k] = rg;
          }
        }
      }
      todo &= todo - 1;
      __syncwarp();
      {
        const uint32_t inc = warp_incl_scan(sgl.y);
        if (lane < kMaxInner) {
          W.so[lane] = sgl.x - (inc - sgl.y);
          W.sb[lane] = inc - sgl.y;
        }
        if (lane == kMaxInner) W.sb[kMaxInner] = inc;
      }
      if (lane == 0) W.ahead = search_ahead(n_sorted, h1 + 1);
      __syncwarp();
      const uint32_t nin = W.sb[kMaxInner];

      uint32_t h0a = 0, h0b = 0;
      float4 p0n = make_float4(0.f, 0.f, 0.f, 0.f);
      // Stages piece `piece` (the passing outgoing cells of ordinal [piece*kOut,
      // (piece+1)*kOut) in search order) and orders it by slope; returns the number of
      // outgoing cells of h1.
      auto stage_piece = [&](int piece) -> uint32_t {
        const uint32_t lo_ord = (uint32_t)piece * kOut;
        uint32_t cnt = 0;
        float m = __int_as_float(0x7f800000), tlo = m, thi = -m;
        const float half_k = 0.5f * cuts.kmax * p1.w;
        for (int k = 0; k < pt.n_outer[L1]; ++k) {
          const uint8_t j2 = (uint8_t)pt.slot[pt.outer[L1][k]][L1];
          const uint2 rk = W.rg[h1 % kGroup][k];
          const float tiny = window_tiny(rk.y);
          uint32_t beg = rk.x & ~kWindowWraps, end = rk.y & ~kWindowExact;
          uint32_t first = 0;  // the outer layer's bins, where the window wraps
          bool wraps = rk.x & kWindowWraps;
          if (wraps) {
            first = (b.hbin[h1] / (kLayers * B) * kLayers + pt.outer[L1][k]) * B;
            end = b.bin_start[first + B];
          }
          for (;;) {
            // two candidates per lane in flight: both loads are issued before either test
            for (uint32_t o0 = beg; o0 < end; o0 += 64) {
              float4 hv[2];
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const uint32_t o = o0 + 32 * u + lane;
                hv[u] = o < end ? b.hit4[o] : make_float4(0.f, 0.f, 0.f, 0.f);
              }
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const uint32_t o = o0 + 32 * u + lane;
                const float4 ho = hv[u];
                const bool pass = doublet_quick(cuts, o < end, p1, ho, half_k, ho.w, tiny);
                const unsigned bal = __ballot_sync(kFull, pass);
                if (pass) {
                  const uint32_t pos = cnt + __popc(bal & lt_mask);
                  if (pos >= lo_ord && pos < lo_ord + kOut) {
                    const uint32_t st = pos - lo_ord;
                    const float t = __fdividef(ho.z - p1.z, ho.w - p1.w);
                    W.t[st] = t;
                    W.code[st] = o | ((uint32_t)j2 << 29);
                    m = fminf(m, fsub(ho.w, p1.w));
                    tlo = fminf(tlo, t);
                    thi = fmaxf(thi, t);
                  }
                }
                cnt += __popc(bal);
              }
            }
            if (!wraps) break;
            wraps = false;
            beg = b.bin_start[first];
            end = rk.y & ~kWindowExact;
          }
        }
        if ((uint32_t)lane < nin) p0n = b.hit4[h0a];
        asm volatile("redux.sync.min.f32 %0, %0, 0xffffffff;" : "+f"(m));
        asm volatile("redux.sync.min.f32 %0, %0, 0xffffffff;" : "+f"(tlo));
        asm volatile("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(thi));
        const uint32_t n = cnt > lo_ord ? min(cnt - lo_ord, (uint32_t)kOut) : 0u;
        const float scale = thi - tlo > 1e-6f ? __fdiv_rn((float)kNb, thi - tlo) : 0.0f;
        // counting sort of the staged cells by slope bucket
        __syncwarp();
        for (int i = lane; i <= kNb; i += 32) W.bstart[i] = 0;
        __syncwarp();
        int key[kOut / 32];
        uint32_t rank[kOut / 32];
#pragma unroll
        for (int u = 0; u < kOut / 32; ++u) {
          const uint32_t st = lane + 32 * u;
          key[u] = 0;
          rank[u] = 0;
          if (st < n) {
            key[u] = slope_bucket(W.t[st], tlo, scale);
            rank[u] = atomicAdd(&W.bstart[key[u] + 1], 1u);
          }
        }
        __syncwarp();
        {
          // bucket starts: kNb / 32 consecutive buckets per lane
          uint32_t cb[kNb / 32], sum = 0;
#pragma unroll
          for (int u = 0; u < kNb / 32; ++u) {
            cb[u] = W.bstart[(kNb / 32) * lane + u + 1];
            sum += cb[u];
          }
          uint32_t run = warp_incl_scan(sum) - sum;
          __syncwarp();
#pragma unroll
          for (int u = 0; u < kNb / 32; ++u) {
            run += cb[u];
            W.bstart[(kNb / 32) * lane + u + 1] = run;
          }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kOut / 32; ++u) {
          const uint32_t st = lane + 32 * u;
          if (st < n) {
            const uint32_t sp = W.bstart[key[u]] + rank[u];
            W.cs[sp] = W.code[st];
            W.ts[sp] = W.t[st];
          }
        }
        if (lane == 0) {
          W.tmin = tlo;
          W.scale = scale;
          W.m = m;
        }
        __syncwarp();
        return cnt;
      };

      // incoming cell i of h1: its cell id and inner-layer slot
      auto incoming = [&](uint32_t i, int& kin) -> uint32_t {
        kin = 0;
        while (i >= W.sb[kin + 1]) ++kin;  // i < W.sb[max_inner] bounds the walk
        return W.so[kin] + i;
      };
      auto inner_hit = [&](uint32_t i) -> uint32_t {
        int kin;
        if (i >= nin) return 0u;
        const uint32_t c = incoming(i, kin);
        return PT_CHECK(b.cnt, c < b.cnt[CNT_CELLS], DBG_CON_INCOMING) ? b.cell_in[c] : 0u;
      };
      // Every piece of the outgoing cells is staged once and visited by all incoming groups.
      // With more than one piece a cell's pairs come up again after some were tested, so
      // all incoming cells have their state set up first.
      uint32_t nout = 0;
#pragma unroll 1
      for (int piece = 0; piece == 0 || (uint32_t)piece * kOut < nout; ++piece) {
        // Inner hits of the lane's cells: the first two groups' indices are fetched while the
        // outgoing cells are searched, the first group's coordinates while they are sorted;
        // each group then fetches the next one's coordinates and the indices of the one
        // after that, and a queued pair names its inner hit instead of carrying it.  With
        // the first group's two dependent loads ahead of the search, and the pairs' inner
        // hits in shared memory, 64 pileup-200 events took 5700 instead of 5490 us.
        h0a = inner_hit(lane);
        h0b = inner_hit(lane + 32);
        nout = stage_piece(piece);
        if (nout == 0) break;
        if (piece == 0 && nout > (uint32_t)kOut) {
          for (uint32_t i = lane; i < nin; i += 32) {
            int kin;
            const uint32_t c = incoming(i, kin);
            if (PT_CHECK(b.cnt, c < b.cnt[CNT_CELLS], DBG_CON_INCOMING))
              *(uint2*)&b.cell[c] = make_uint2(kHole, 0u);
          }
        }
#pragma unroll 1
        for (uint32_t g0 = 0; g0 < nin; g0 += 32) {
          // the lane's incoming cell
          const uint32_t i = g0 + lane;
          bool valid = i < nin;
          uint32_t c = 0;
          int kin = 0;
          if (valid) {
            c = incoming(i, kin);
            valid = PT_CHECK(b.cnt, c < b.cnt[CNT_CELLS], DBG_CON_INCOMING);
          }
          const float4 p0 = p0n;
          const uint32_t h0 = h0a | (valid && pt.inner[L1][kin] == 0 ? kOnLayer0 : 0u);
          h0a = h0b;
          if (i + 32 < nin) p0n = b.hit4[h0a];
          h0b = inner_hit(i + 64);
          const float ta = __fdividef(p1.z - p0.z, p1.w - p0.w);  // the cell's slope dz/dr
          const float id1 = __fdividef(1.0f, p1.w - p0.w);
          const float wa = (cuts.rz0 + cuts.rz1 * cuts.cotmax) * id1;
          const float ua = cuts.rz0 + cuts.rz1 * fabsf(ta);
          const float shrink = 1.0f - cuts.rz1 * id1;

          bool inited = nout > (uint32_t)kOut;  // the lane's cell had its state set up
          const float m = W.m, tmin = W.tmin, scale = W.scale;
          float w = 0.0f;
          uint32_t pos = 0, pend = 0;
          if (valid) {
            const float im = __fdividef(1.0f, m);
            float wk = fmaf(ua, im, wa);
            if (shrink > 0.0f) wk = fminf(wk, __fdividef(ua * (id1 + im), shrink));
            w = wk * 1.01f + 1e-3f;
            const float w2 = w * 1.001f + 1e-5f;
            pos = W.bstart[slope_bucket(__fsub_rn(ta, w2), tmin, scale)];
            pend = W.bstart[slope_bucket(__fadd_rn(ta, w2), tmin, scale) + 1];
            if (!PT_CHECK(b.cnt, pos <= pend && pend <= (uint32_t)kOut, DBG_CON_BUCKET))
              pend = pos;
          }
          // each lane walks its own bucket range; the staged cells inside its window are
          // queued with their target and tested with C1-C3 once 32 are waiting
          while (__any_sync(kFull, pos < pend)) {
            bool pass = false;
            uint32_t code = 0;
            if (pos < pend) {
              pass = fabsf(W.ts[pos] - ta) <= w;
              if (pass) {
                // the target cell, named by its outer hit and the slot of h1's layer
                // among that hit's inner layers until k_link_targets finds it
                code = W.cs[pos];
                if (!inited) {
                  // before any of its pairs is tested: no links, no flags
                  *(uint2*)&b.cell[c] = make_uint2(kHole, 0u);
                  inited = true;
                }
              }
              ++pos;
            }
            const unsigned bal = __ballot_sync(kFull, pass);
            (void)PT_CHECK(b.cnt, qtail + __popc(bal) - qhead <= (uint32_t)kQueue, DBG_CON_QUEUE);
            if (pass) {
              const uint32_t qi = (qtail + __popc(bal & lt_mask)) & (kQueue - 1);
              W.q[qi] = make_uint4(c, code, h1, h0);
            }
            qtail += __popc(bal);
            if (qtail - qhead >= 32u) process(32u);
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      const uint32_t next = search_chunk(n_sorted - W.s0, n_warps);
      W.per = next;
      W.s0 = W.dyn0 + (uint32_t)atomicAdd(&b.cnt[CNT_LNK_WORK], (unsigned long long)next);
    }
    __syncwarp();
  }
  while (qtail != qhead) process(min(32u, qtail - qhead));
  __syncwarp();
  mark_link_hole(W.chunk_next, W.chunk_end);
  if (lane == 0 && W.used) atomicAdd(&b.cnt[CNT_LINKS_USED], (unsigned long long)W.used);
}

// Position of inner hit h in the cells [lo, hi) of one segment (ordered by inner hit, each
// inner hit once): the first cell whose inner hit is >= h (hi if none), `found` telling
// whether it is h.  The segment's inner hits spread over the outer hit's window in the
// inner layer, so h's position is guessed from the first and last of them and the eight
// cells around the guess are read at once; a guess that misses leaves a bisection of the
// side beyond it.  Segments of up to eight cells are read whole.  Dependent loads: two or
// three levels for most links, against about seven for a bisection of the whole segment.
__device__ __forceinline__ uint32_t find_inner(const Buffers& b, uint32_t lo, uint32_t hi,
                                               uint32_t h, bool& found) {
  const uint32_t end = hi;
  uint32_t w0 = lo;
  if (hi - lo > 8) {
    const uint32_t f = b.cell_in[lo], la = b.cell_in[hi - 1];
    if (h <= f) {
      found = h == f;
      return lo;
    }
    if (h > la) {
      found = false;
      return hi;
    }
    // f < h <= la
    const uint32_t g =
        lo + (uint32_t)((uint64_t)(h - f) * (uint64_t)(hi - 1 - lo) / (uint64_t)(la - f));
    w0 = min(max(g, lo + 3u) - 3u, hi - 8u);
  }
  // the (up to) eight cells from w0
  uint32_t less = 0;
  bool eq = false;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t v = w0 + k < hi ? b.cell_in[w0 + k] : 0xffffffffu;
    less += v < h ? 1u : 0u;
    eq |= v == h;
  }
  if (hi - lo <= 8 || (less > 0 && less < 8)) {
    found = eq;
    return w0 + less;
  }
  // the guess missed: the position lies before w0 (less == 0) or after w0 + 7
  if (less == 0) hi = w0; else lo = w0 + 8;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (b.cell_in[mid] < h) lo = mid + 1; else hi = mid;
  }
  found = lo < end && b.cell_in[lo] == h;
  return lo;
}

// The target cell (h1, h2) of every link: h1 in h2's incoming segment from h1's layer,
// which is ordered by inner hit (find_inner); one thread per link slot.  The link is
// completed for the ntuplet walk.  The target has links of its own when the list head in
// its state names a link that starts from it: a cell without links may hold anything
// there, but no link then names it as its source.  Such a leaf gets its state here, named
// by whichever of its in-links writes last.  Plain form: the flag of the target's incoming link is set (a leaf needs
// none: only cells with links can be roots).  Gated form: the link's bf16 feature row for
// the gate's MLP is computed, one thread per link with every lane busy, from the three
// hits (mostly still in L2).  A target can be missing only when the doublet stage ran out
// of cell slots (its status bit is set then); the link then points back to its source, a
// valid cell, so that the later stages stay within their arrays.
//
// Bound by its random sectors.  64 pileup-200 events (5.3M links): 0.34 ms, against 0.27
// when it left the walk's other fields to the search, which now reads a link in one sector
// (A4 to A6 0.73 against 1.62 ms).
template <bool GATE>
__global__ void k_link_targets(Buffers b, pt_cuts cuts, int32_t B, int max_inner,
                               uint64_t cap_links) {
  pdl_wait();
  const uint64_t nl = min(b.cnt[CNT_LINKS], (unsigned long long)cap_links);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t l = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; l < nl; l += stride) {
    const uint4 hi = *link_hi(&b.link[l]);
    const uint32_t a = hi.x, t = hi.y, h1 = hi.z;
    if (a == kHole) continue;
    const uint32_t next = b.link[l].next;
    uint2 sg = b.seg[(uint64_t)(t & 0x1fffffffu) * max_inner + (t >> 29)];
    if (!PT_CHECK(b.cnt, (uint64_t)sg.x + sg.y <= b.cnt[CNT_CELLS], DBG_TGT_SEGMENT))
      sg = make_uint2(0u, 0u);
    bool found;
    const uint32_t pos = find_inner(b, sg.x, sg.x + sg.y, h1, found);
    const uint32_t c = found ? pos : a;
    uint32_t head = b.cell[c].head;
    if (head >= nl || b.link[head].src != c) {
      head = kHole;
      *(uint2*)&b.cell[c] = make_uint2((uint32_t)l, 0u);
    } else if (!GATE && found) {
      b.cell[c].has_in = 1;
    }
    *link_lo(&b.link[l]) = make_uint4(next, c, head, found ? (t & 0x1fffffffu) : h1);
    if (GATE) {
      const uint32_t h0 = b.cell_in[a], h2 = t & 0x1fffffffu;
      float f[kGateFeat];
      gate_link_features(cuts, b.hit4[h0], b.hit4[h1], b.hit4[h2], (b.hbin[h0] / B) % kLayers,
                         (b.hbin[h1] / B) % kLayers, (b.hbin[h2] / B) % kLayers, f);
      store_gate_row(b.gate_x + l * kGateK1, f);
    }
  }
}

}  // namespace

void launch_connect(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                    bool gated) {
  PT_TRACE(l, s, "k_connect",
           launch_pdl(k_connect, l.sms * kConnBlocksPerSm, kConnWarps * 32, 0, s, b, p.cuts,
                      p.pairs, p.phi_bins, (uint64_t)p.max_links));
  if (gated)
    PT_TRACE(l, s, "k_link_targets",
             launch_pdl(k_link_targets<true>, l.grid, 256, 0, s, b, p.cuts, p.phi_bins,
                        p.pairs.max_inner, (uint64_t)p.max_links));
  else
    PT_TRACE(l, s, "k_link_targets",
             launch_pdl(k_link_targets<false>, l.grid, 256, 0, s, b, p.cuts, p.phi_bins,
                        p.pairs.max_inner, (uint64_t)p.max_links));
}

}  // namespace ptca
