// Stages A4-A6: ntuplet extraction, duplicate cleaning and canonical order (Sec.
// 2.2.1, Fig. 2: starting from the seeds, the chain selects the sets of hits that are
// candidate tracks).
//
// A4  every path of linked cells from a root (a cell with no incoming link) to a leaf
//     (a cell with no outgoing link) with 3..6 hits.  Roots are taken among the sources
//     of the link lists (a root without an outgoing link would give a 2-hit path,
//     which is dropped).  One thread per root walks its out-links depth first with an
//     explicit stack (the layer graph bounds the depth at 5 cells), writing the paths to
//     its warp's shared buffer, which one atomic per 32 roots reserves and the warp
//     copies out (a batch of roots with more paths than the buffer holds is walked a
//     second time and written directly).  The path quality q is the float32 sum of its link qualities,
//     added from the innermost link outwards.
// A5  duplicate cleaning: ntuplets are ranked by (more hits, smaller q, smaller hit tuple)
//     (batch input indices, -1 padded, signed); one survives when it is the best of every
//     one of its cells, and a triplet then dies if it shares a hit with a surviving ntuplet
//     of >= 4 hits.  The key (6 - nhits, q bits, ntuplet) packed in 64 bits orders ntuplets
//     that way except where two have the same hit count and q, and it needs no sorted
//     position.  One pass reduces the keys into the cells (atomicMin).  An ntuplet that finds another one with its own hit count and q in a cell
//     compares the tuples and takes the cell if its own is smaller.
// A6  canonical order: events in order, hit tuples ascending.  Only the survivors are
//     ordered (0.67M of 4.6M ntuplets on 64 pileup-200 events): they are counted and listed
//     per first hit, a scan over the hits gives each first hit its place, and each survivor
//     finds its rank among those that start at the same hit by walking that hit's list.
//
// The whole-batch graph runs A5 and A6 that way.  The stage call runs them as the separate
// steps that a trace of the stage path lists: all ntuplets are put in canonical order (a
// counting sort on the first hit, then each bucket's few entries by insertion), the sorted
// position stands in the key for the first hit (so that keys never tie), and the survivors
// are compacted in that order.  Both give the same ntuplets in the same order.  A4 to A6
// on 64 pileup-200 events: 0.73 ms, against 1.62 ms when the graph ran the separate steps.
#include "ptca_internal.cuh"

namespace ptca {

namespace {

// Ntuplets buffered per warp in shared memory before one global reservation, and the
// search's blocks per SM (more walks in flight hide more of their load latency; the
// build may set both for tuning sweeps).
#ifndef PT_NT_BUF
#define PT_NT_BUF 64
#endif
#ifndef PT_NT_BLOCKS_PER_SM
#define PT_NT_BLOCKS_PER_SM 6
#endif
constexpr int kNtBuf = PT_NT_BUF;
constexpr int kNtWarps = 8;  // warps per block of the ntuplet search
constexpr int kNtBlocksPerSm = PT_NT_BLOCKS_PER_SM;
struct NtWarp {
  uint32_t roots[64];                        // queued roots (< 32 + 32)
  int32_t hits[kNtBuf][kMaxHits];            // buffered ntuplets (sorted hit indices)
  uint32_t cells[kNtBuf][kMaxCellsPerNt];
  float q[kNtBuf];
  uint32_t n[kNtBuf];
  uint32_t cnt;                              // ntuplets found by the batch (may exceed kNtBuf)
};

enum WalkMode { kEmit = 1, kBuffer = 2 };

// The cleaning key of an ntuplet; `id` (below 2^29) separates equal hit counts and q.
__device__ __forceinline__ unsigned long long dedup_key(uint32_t n, float q, uint32_t id) {
  return ((unsigned long long)(kMaxHits - n) << 61) |
         ((unsigned long long)__float_as_uint(q) << kRankBits) | (unsigned long long)id;
}

// The cleaning key's place for the k-th of an ntuplet's n - 1 cells, named by link slot c.
__device__ __forceinline__ unsigned long long* best_of(const Buffers& b, uint32_t c, uint32_t k,
                                                       uint32_t n, bool last_is_source) {
  LinkBest* p = &b.link_best[c];
  return k + 2 == n && !last_is_source ? &p->leaf : &p->src;
}

// Writes ntuplet t (hits g[0..5], batch indices, -1 padded; cells c[0..4], link slots,
// kHole padded) and resets its cells' keys for the cleaning.
__device__ __forceinline__ void write_ntuplet(const Buffers& b, uint64_t t, uint32_t n, float q,
                                              bool last_is_source, const int32_t (&g)[kMaxHits],
                                              const uint32_t (&c)[kMaxCellsPerNt]) {
  int2* hp = (int2*)(b.nt_hits + t * kMaxHits);
#pragma unroll
  for (int k = 0; k < kMaxHits / 2; ++k) hp[k] = make_int2(g[2 * k], g[2 * k + 1]);
#pragma unroll
  for (int k = 0; k < kMaxCellsPerNt; ++k) b.nt_cells[t * kMaxCellsPerNt + k] = c[k];
  b.nt_n[t] = (uint8_t)n;
  b.nt_q[t] = last_is_source ? -q : q;
#pragma unroll
  for (int k = 0; k < kMaxCellsPerNt; ++k) {
    if ((uint32_t)k + 1 >= n) break;
    *best_of(b, c[k], k, n, last_is_source) = ~0ull;
  }
}

// Depth-first walk from the root whose out-link list is headed by slot l0; returns the
// number of ntuplets.  kEmit: writes them at slots t0, t0 + 1, ... (slots >= cap_nt are
// dropped); kBuffer: to the warp's shared buffer (entries >= kNtBuf are dropped; the
// caller then walks again with kEmit).  A cell's links are a list (its head, then each
// link's next slot); a step reads the link's one sector and, in the masked forms, its keep
// flag and whether the target cell kept a link.  The walk names a cell by its list's head,
// a leaf by its cell, and keeps sorted hit indices; the leaf's link slot and the batch
// indices (perm) are looked up when a path is written (kEmit) or when the warp copies its
// buffer out (kBuffer).
constexpr uint32_t kLastIsSource = 1u << 8;  // beside an entry's hit count in the buffer
template <int MODE, bool GATED>
__device__ uint32_t walk(const Buffers& b, uint32_t l0, unsigned long long t0, uint64_t cap_nt,
                         NtWarp* W) {
  uint32_t path[kMaxCellsPerNt];  // list head of each cell
  uint32_t it[kMaxCellsPerNt];    // next out-link slot of path[k] (kHole: none left)
  float qs[kMaxCellsPerNt];
  uint32_t gh[kMaxCellsPerNt];    // sorted index of the outer hit of path[k]
  // a link slot read from the lists (debug build: kHole unless inside the link slots)
  auto slot = [&](uint32_t x) -> uint32_t {
    return (x == kHole || PT_CHECK(b.cnt, x < b.cnt[CNT_LINKS], DBG_NT_LINKS)) ? x : kHole;
  };
  path[0] = l0;
  it[0] = slot(l0);
  qs[0] = 0.0f;
  const uint4 first = *link_hi(&b.link[l0]);
  const uint32_t g0 = b.cell_in[first.x];
  gh[0] = first.z;
  uint32_t found = 0;
  int depth = 1;
  while (depth > 0) {
    const int d = depth - 1;
    if (it[d] == kHole) {
      --depth;
      continue;
    }
    const uint32_t l = it[d];
    const uint4 lo = *link_lo(&b.link[l]);  // next, target, its list's head, its outer hit
    const float lq = b.link[l].q;
    bool leaf = lo.z == kHole;
    const bool last_is_source = GATED && !leaf && !b.cell[lo.y].has_out;
    if (last_is_source) leaf = true;  // its list holds removed links only
    const bool keep = !GATED || b.gate_keep[l];
    it[d] = slot(lo.x);
    if (depth == kMaxCellsPerNt || !keep) continue;  // deeper than the layer graph, or removed
    if (!PT_CHECK(b.cnt, lo.y < b.cnt[CNT_CELLS], DBG_NT_CELL)) continue;
    const float q = fadd(qs[d], lq);
    if (leaf) {
      // leaf: path[0..d] + target, i.e. depth + 1 cells, depth + 2 hits
      const uint32_t last = last_is_source ? lo.z : lo.y;
      if (MODE == kEmit) {
        const unsigned long long t = t0 + found;
        if (t < cap_nt) {
          int32_t g[kMaxHits];
          uint32_t c[kMaxCellsPerNt];
          g[0] = (int32_t)b.perm[g0];
#pragma unroll
          for (int k = 0; k < kMaxCellsPerNt; ++k) {
            c[k] = k > depth ? kHole : k < depth ? path[k]
                   : last_is_source ? last : b.cell[last].head;
            g[k + 1] = k > depth ? -1 : (int32_t)b.perm[k < depth ? gh[k] : lo.w];
          }
          write_ntuplet(b, t, (uint32_t)(depth + 2), q, last_is_source, g, c);
        }
      } else {
        const uint32_t e = atomicAdd(&W->cnt, 1u);
        if (e < (uint32_t)kNtBuf) {
          W->n[e] = (uint32_t)(depth + 2) | (last_is_source ? kLastIsSource : 0u);
          W->q[e] = q;
          W->hits[e][0] = (int32_t)g0;
          for (int k = 0; k <= depth; ++k) {
            W->hits[e][k + 1] = (int32_t)(k < depth ? gh[k] : lo.w);
            W->cells[e][k] = k < depth ? path[k] : last;
          }
          for (int k = depth + 2; k < kMaxHits; ++k) W->hits[e][k] = -1;
          for (int k = depth + 1; k < kMaxCellsPerNt; ++k) W->cells[e][k] = kHole;
        }
      }
      ++found;
      continue;
    }
    path[depth] = lo.z;
    it[depth] = slot(lo.z);
    qs[depth] = q;
    gh[depth] = lo.w;
    ++depth;
  }
  return found;
}

// The slot that heads a source cell's out-link list names a candidate root, which is a
// root when the cell has no incoming link (masked forms: a kept outgoing link and no kept
// incoming one).  Each warp queues the roots of its link slots in shared memory and walks
// them 32 at a time, one per lane, writing the ntuplets to its shared buffer; one atomic
// then reserves them and the warp copies them out.  If a batch finds more than the buffer
// holds, it is walked again and written directly.
//
// Bound by the latency of its random reads.  64 pileup-200 events (4.6M ntuplets): 0.40 ms,
// against 0.68 when a step read four arrays.  Reducing the cleaning keys here as well holds
// up the walks behind the atomics: 0.75 ms with the keys in link space (0.07 for them in a
// pass of their own), 1.07 with the keys among all cells, 1.11 if their results are waited
// for.
template <bool GATED>
__global__ void __launch_bounds__(kNtWarps * 32, kNtBlocksPerSm)
    k_find_ntuplets(Buffers b, uint64_t cap_links, uint64_t cap_nt) {
  pdl_wait();
  __shared__ NtWarp s_w[kNtWarps];
  NtWarp& W = s_w[threadIdx.x >> 5];
  const uint64_t nl = min(b.cnt[CNT_LINKS], (unsigned long long)cap_links);
  const int lane = lane_id();
  const unsigned lt_mask = (1u << lane) - 1u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint32_t nq = 0;  // queued roots (warp-uniform), each named by its list's head slot
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < nl;
       i0 += stride) {
    const uint64_t i = i0 + lane;
    uint32_t a = kHole;
    if (i < nl) a = b.link[i].src;
    bool root = false;
    if (a != kHole) {
      const uint2 st = *(const uint2*)&b.cell[a];  // head; has_in, has_out, kill
      root = st.x == (uint32_t)i && !(st.y & 0xffu) && (!GATED || (st.y & 0xff00u));
    }
    const unsigned rm = __ballot_sync(kFull, root);
    if (root) W.roots[nq + __popc(rm & lt_mask)] = (uint32_t)i;
    nq += __popc(rm);
    const bool final = i0 + stride >= nl;
    while (nq >= 32u || (final && nq > 0u)) {
      const uint32_t take = min(nq, 32u);
      __syncwarp();
      const uint32_t r = (uint32_t)lane < take ? W.roots[lane] : kHole;
      if (lane == 0) W.cnt = 0;
      __syncwarp();
      const uint32_t n = r != kHole ? walk<kBuffer, GATED>(b, r, 0, cap_nt, &W) : 0u;
      __syncwarp();
      const uint32_t tot = W.cnt;
      // the roots not taken move to the front of the queue
      const uint32_t rest = nq - take;
      const uint32_t moved = (uint32_t)lane < rest ? W.roots[take + lane] : 0u;
      __syncwarp();
      if ((uint32_t)lane < rest) W.roots[lane] = moved;
      nq = rest;
      if (tot == 0) continue;
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(&b.cnt[CNT_NT], (unsigned long long)tot);
      base = __shfl_sync(kFull, base, 0);
      if (base + tot > cap_nt && lane == 0) atomicOr(&b.cnt[CNT_STATUS], ST_NT);
      if (tot <= (uint32_t)kNtBuf) {
        for (uint32_t e = lane; e < tot; e += 32) {
          const unsigned long long t = base + e;
          if (t < cap_nt) {
            int32_t g[kMaxHits];
            uint32_t c[kMaxCellsPerNt];
#pragma unroll
            for (int k = 0; k < kMaxHits; ++k) {
              const int32_t sh = W.hits[e][k];  // sorted index, -1 pad
              g[k] = sh >= 0 ? (int32_t)b.perm[sh] : -1;
            }
#pragma unroll
            for (int k = 0; k < kMaxCellsPerNt; ++k) c[k] = W.cells[e][k];
            const uint32_t n = W.n[e] & (kLastIsSource - 1u);
            const bool last_is_source = (W.n[e] & kLastIsSource) != 0;
            if (!last_is_source) {  // a leaf is named by its cell until here
#pragma unroll
              for (int k = 1; k < kMaxCellsPerNt; ++k)
                if ((uint32_t)k + 2 == n) c[k] = b.cell[c[k]].head;
            }
            write_ntuplet(b, t, n, W.q[e], last_is_source, g, c);
          }
        }
      } else {
        const uint32_t inc = warp_incl_scan(n);
        if (n) walk<kEmit, GATED>(b, r, base + inc - n, cap_nt, &W);
      }
    }
  }
}

__device__ __forceinline__ bool tuple_less(const int32_t* a, const int32_t* c) {
#pragma unroll
  for (int k = 0; k < kMaxHits; ++k) {
    if (a[k] != c[k]) return a[k] < c[k];
  }
  return false;
}

constexpr unsigned long long kIdMask = (1ull << kRankBits) - 1;

// Ntuplet t (key) has met another one of the same hit count and q in a cell: it takes the
// cell if its tuple is the smaller one.  Once every such ntuplet has tried, the cell holds
// the smallest tuple.
__device__ __noinline__ void take_tied_cell(const Buffers& b, uint32_t t, unsigned long long key,
                                            unsigned long long* best) {
  unsigned long long cur = *best;
  while ((cur >> kRankBits) == (key >> kRankBits) && cur != key &&
         tuple_less(b.nt_hits + (uint64_t)t * kMaxHits,
                    b.nt_hits + (cur & kIdMask) * kMaxHits)) {
    const unsigned long long old = atomicCAS(best, cur, key);
    if (old == cur) break;
    cur = old;
  }
  b.cnt[CNT_NT_TIES] = 1;
}

// Reduces every ntuplet's key into its cells; `rank` NULL: the key's id is the ntuplet.
__global__ void k_dedup_min(Buffers b, const uint32_t* rank, uint64_t cap_nt) {
  pdl_wait();
  const uint64_t T = min(b.cnt[CNT_NT], (unsigned long long)cap_nt);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride) {
    const float sq = b.nt_q[t];
    const bool last_is_source = (__float_as_uint(sq) >> 31) != 0;
    uint32_t c[kMaxCellsPerNt], n = 1;
#pragma unroll
    for (int k = 0; k < kMaxCellsPerNt; ++k) {
      c[k] = b.nt_cells[t * kMaxCellsPerNt + k];
      n += c[k] != kHole;
    }
    const unsigned long long key = dedup_key(n, fabsf(sq), rank ? rank[t] : (uint32_t)t);
#pragma unroll
    for (int k = 0; k < kMaxCellsPerNt; ++k)
      if (c[k] != kHole) atomicMin(best_of(b, c[k], k, n, last_is_source), key);
  }
}

// Ntuplets that no cell ranks behind another hit count or q go to best_list (one
// reservation per warp); cells where two of the same meet are decided on the way.
__global__ void k_dedup_best(Buffers b, uint64_t cap_nt) {
  pdl_wait();
  const uint64_t T = min(b.cnt[CNT_NT], (unsigned long long)cap_nt);
  if (blockIdx.x == 0 && threadIdx.x == 0) b.cnt[CNT_SCAN_NT] = T;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const int lane = lane_id();
  for (uint64_t t0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < T;
       t0 += stride) {
    const uint64_t t = t0 + lane;
    bool ok = t < T;
    if (ok) {
      uint32_t c[kMaxCellsPerNt];
      unsigned long long v[kMaxCellsPerNt];
      const float sq = b.nt_q[t];
      const bool last_is_source = (__float_as_uint(sq) >> 31) != 0;
      uint32_t n = 1;
#pragma unroll
      for (int k = 0; k < kMaxCellsPerNt; ++k) {
        c[k] = b.nt_cells[t * kMaxCellsPerNt + k];
        n += c[k] != kHole;
      }
#pragma unroll
      for (int k = 0; k < kMaxCellsPerNt; ++k)
        v[k] = c[k] != kHole ? *best_of(b, c[k], k, n, last_is_source) : 0ull;
      const unsigned long long key = dedup_key(n, fabsf(sq), (uint32_t)t);
#pragma unroll
      for (int k = 0; k < kMaxCellsPerNt; ++k) {
        if (c[k] == kHole) continue;
        const bool same = (v[k] >> kRankBits) == (key >> kRankBits);
        ok = ok && same;
        if (same && v[k] != key)
          take_tied_cell(b, (uint32_t)t, key, best_of(b, c[k], k, n, last_is_source));
      }
    }
    const unsigned m = __ballot_sync(kFull, ok);
    if (!m) continue;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&b.cnt[CNT_NT_BEST], (unsigned long long)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (ok) b.best_list[base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)t;
  }
}

// Whether ntuplet t (n hits) holds the best key of all its cells.
__device__ __forceinline__ bool holds_all(const Buffers& b, uint64_t t, uint32_t n, uint32_t id) {
  const float sq = b.nt_q[t];
  const bool last_is_source = (__float_as_uint(sq) >> 31) != 0;
  const unsigned long long key = dedup_key(n, fabsf(sq), id);
  bool ok = true;
  for (uint32_t k = 0; k + 1 < n; ++k)
    ok = ok && *best_of(b, b.nt_cells[t * kMaxCellsPerNt + k], k, n, last_is_source) == key;
  return ok;
}

// The listed ntuplets that hold all their cells (where cells were tied, that is looked up
// again) and have four or more hits mark their hits used.
__global__ void k_used_hits(Buffers b) {
  pdl_sync();
  const uint64_t N = b.cnt[CNT_NT_BEST];
  const bool ties = b.cnt[CNT_NT_TIES] != 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
    const uint32_t t = b.best_list[i];
    const int n = b.nt_n[t];
    if (ties && !holds_all(b, t, (uint32_t)n, t)) {
      b.best_list[i] = kHole;
      continue;
    }
    if (n >= 4)
      for (int k = 0; k < n; ++k) b.used[b.nt_hits[(uint64_t)t * kMaxHits + k]] = 1;
  }
}

// Survivors: the listed ntuplets of four or more hits, and the triplets that share no hit
// with them; each goes on its first hit's list and is counted there.
__global__ void k_survivors(Buffers b) {
  pdl_sync();
  const uint64_t N = b.cnt[CNT_NT_BEST];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
    const uint32_t t = b.best_list[i];
    if (t == kHole) continue;
    const int32_t* h = b.nt_hits + (uint64_t)t * kMaxHits;
    if (b.nt_n[t] == 3 && (b.used[h[0]] || b.used[h[1]] || b.used[h[2]])) {
      b.best_list[i] = kHole;
      continue;
    }
    b.nt_next[t] = atomicExch(&b.nt_head[h[0]], t);
    atomicAdd(&b.sv_cnt[h[0]], 1u);
  }
}

// Place of every survivor: its first hit's, plus the survivors with a smaller tuple on that
// hit's list.  Per-event offsets and the total come from the places of the events' first
// hits.  The ntuplet also goes out, with event-local indices: to the caller's arrays or, if
// they do not hold the batch, to the export staging.
__global__ void k_order(Buffers b) {
  pdl_sync();
  const uint64_t N = b.cnt[CNT_NT_BEST];
  const int E = b.hdr->n_events;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t S = b.sv_start[b.hdr->n_hits];
  if (tid == 0) b.cnt[CNT_SV] = S;
  const bool direct = results_go_out(b, S);
  int32_t* out_hits = direct ? b.hdr->out_hits : b.exp_hits;
  uint8_t* out_n = direct ? b.hdr->out_n : b.exp_n;
  int64_t* out_off = direct ? b.hdr->out_off : nullptr;
  for (uint64_t e = tid; e <= (uint64_t)E; e += stride) {
    const int64_t first = (int64_t)b.sv_start[b.hit_off[e]];
    b.ev_nt_off[e] = first;
    if (out_off) out_off[e] = first;
  }
  for (uint64_t i = tid; i < N; i += stride) {
    const uint32_t t = b.best_list[i];
    if (t == kHole) continue;
    int32_t h[kMaxHits];
    const int2* hp = (const int2*)(b.nt_hits + (uint64_t)t * kMaxHits);
#pragma unroll
    for (int k = 0; k < kMaxHits / 2; ++k) {
      const int2 v = hp[k];
      h[2 * k] = v.x;
      h[2 * k + 1] = v.y;
    }
    uint32_t pos = b.sv_start[h[0]];
    if (b.sv_start[h[0] + 1] - pos > 1)
      for (uint32_t o = b.nt_head[h[0]]; o != kHole; o = b.nt_next[o])
        if (tuple_less(b.nt_hits + (uint64_t)o * kMaxHits, h)) ++pos;
    b.sv[pos] = t;
    if (out_hits) {
      const int32_t off = b.hit_off[find_event(b.hit_off, E, h[0])];
      int32_t* ep = out_hits + (uint64_t)pos * kMaxHits;  // a caller's array: any 4-byte place
#pragma unroll
      for (int k = 0; k < kMaxHits; ++k) ep[k] = h[k] >= 0 ? h[k] - off : -1;
    }
    if (out_n) out_n[pos] = b.nt_n[t];
  }
}

// ------------------------------------------------------------ the stage call's steps
// Its scratch lies in memory that these steps leave free: the sorted positions in nt_next,
// the order in best_list, the flags and their scan in the export staging.
struct StageSort {
  uint32_t *cnt, *start, *rank, *ord, *alive, *alive_scan;
};
__host__ __device__ inline StageSort stage_sort(const Buffers& b, uint64_t cap_nt) {
  uint32_t* e = (uint32_t*)b.exp_hits;  // 6 x cap_nt words
  return {b.sv_cnt, b.sv_start, b.nt_next, b.best_list, e, e + cap_nt};
}

__global__ void k_bucket_count(Buffers b, StageSort w, uint64_t cap_nt) {
  const uint64_t T = min(b.cnt[CNT_NT], (unsigned long long)cap_nt);
  if (blockIdx.x == 0 && threadIdx.x == 0) b.cnt[CNT_SCAN_NT] = T;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride)
    w.rank[t] = atomicAdd(&w.cnt[b.nt_hits[t * kMaxHits]], 1u);
}

__global__ void k_bucket_scatter(Buffers b, StageSort w) {
  const uint64_t T = b.cnt[CNT_SCAN_NT];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride)
    w.ord[w.start[b.nt_hits[t * kMaxHits]] + w.rank[t]] = (uint32_t)t;
}

__global__ void k_bucket_sort(Buffers b, StageSort w) {
  const int N = b.hdr->n_hits;
  const int stride = gridDim.x * blockDim.x;
  for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < N; h += stride) {
    const uint32_t lo = w.start[h], hi = w.start[h + 1];
    for (uint32_t i = lo + 1; i < hi; ++i) {
      const uint32_t v = w.ord[i];
      const int32_t* hv = b.nt_hits + (uint64_t)v * kMaxHits;
      uint32_t j = i;
      while (j > lo && tuple_less(hv, b.nt_hits + (uint64_t)w.ord[j - 1] * kMaxHits)) {
        w.ord[j] = w.ord[j - 1];
        --j;
      }
      w.ord[j] = v;
    }
    for (uint32_t i = lo; i < hi; ++i) w.rank[w.ord[i]] = i;  // sorted position
  }
}

__global__ void k_dedup_alive(Buffers b, StageSort w) {
  const uint64_t T = b.cnt[CNT_SCAN_NT];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride) {
    const int n = b.nt_n[t];
    const uint32_t i = w.rank[t];
    const bool ok = holds_all(b, t, (uint32_t)n, i);
    w.alive[i] = ok ? 1u : 0u;
    if (ok && n >= 4)
      for (int k = 0; k < n; ++k) b.used[b.nt_hits[t * kMaxHits + k]] = 1;
  }
}

__global__ void k_dedup_triplets(Buffers b, StageSort w) {
  const uint64_t T = b.cnt[CNT_SCAN_NT];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < T; i += stride) {
    if (!w.alive[i]) continue;
    const uint32_t t = w.ord[i];
    if (b.nt_n[t] != 3) continue;
    const int32_t* h = b.nt_hits + (uint64_t)t * kMaxHits;
    if (b.used[h[0]] || b.used[h[1]] || b.used[h[2]]) w.alive[i] = 0u;
  }
}

__global__ void k_compact(Buffers b, StageSort w) {
  const uint64_t T = b.cnt[CNT_SCAN_NT];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  if (blockIdx.x == 0 && threadIdx.x == 0) b.cnt[CNT_SV] = w.alive_scan[T];
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < T; i += stride)
    if (w.alive[i]) b.sv[w.alive_scan[i]] = w.ord[i];
}

// ev_nt_off[e] = first survivor of event >= e; survivors are ordered by event because
// batch input indices are.
__global__ void k_event_offsets(Buffers b) {
  const uint64_t S = b.cnt[CNT_SV];
  const int E = b.hdr->n_events;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= S; j += stride) {
    const int e_cur =
        j < S ? find_event(b.hit_off, E, b.nt_hits[(uint64_t)b.sv[j] * kMaxHits]) : E;
    const int e_prev =
        j > 0 ? find_event(b.hit_off, E, b.nt_hits[(uint64_t)b.sv[j - 1] * kMaxHits]) : -1;
    for (int e = e_prev + 1; e <= e_cur; ++e) b.ev_nt_off[e] = (int64_t)j;
  }
}

}  // namespace

static void launch_search(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                          bool gated) {
  const uint64_t cap_links = (uint64_t)p.max_links, cap_nt = (uint64_t)p.max_ntuplets;
  const int grid = l.sms * kNtBlocksPerSm, block = kNtWarps * 32;
  if (gated)
    PT_TRACE(l, s, "k_find_ntuplets",
             launch_pdl(k_find_ntuplets<true>, grid, block, 0, s, b, cap_links, cap_nt));
  else
    PT_TRACE(l, s, "k_find_ntuplets",
             launch_pdl(k_find_ntuplets<false>, grid, block, 0, s, b, cap_links, cap_nt));
}

void launch_ntuplets(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                     bool gated) {
  const uint64_t cap_nt = (uint64_t)p.max_ntuplets;
  launch_search(b, p, l, s, gated);
  launch_pdl(k_dedup_min, l.grid, 256, 0, s, b, nullptr, cap_nt);
  launch_pdl(k_dedup_best, l.grid, 256, 0, s, b, cap_nt);
  launch_pdl(k_used_hits, l.grid, 256, 0, s, b);
  launch_pdl(k_survivors, l.grid, 256, 0, s, b);
  launch_scan(b.sv_cnt, b.sv_start, &b.cnt[CNT_SCAN_HITS], b.scan_part, s);
  launch_pdl(k_order, l.grid, 256, 0, s, b);
}

void launch_ntuplet_steps(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                          bool gated) {
  const uint64_t cap_nt = (uint64_t)p.max_ntuplets;
  const StageSort w = stage_sort(b, cap_nt);
  launch_search(b, p, l, s, gated);
  PT_TRACE(l, s, "k_bucket_count", k_bucket_count<<<l.grid, 256, 0, s>>>(b, w, cap_nt));
  PT_TRACE(l, s, "scan", launch_scan(w.cnt, w.start, &b.cnt[CNT_SCAN_HITS], b.scan_part, s));
  PT_TRACE(l, s, "k_bucket_scatter", k_bucket_scatter<<<l.grid, 256, 0, s>>>(b, w));
  PT_TRACE(l, s, "k_bucket_sort", k_bucket_sort<<<l.grid, 256, 0, s>>>(b, w));
  PT_TRACE(l, s, "k_dedup_min", k_dedup_min<<<l.grid, 256, 0, s>>>(b, w.rank, cap_nt));
  PT_TRACE(l, s, "k_dedup_alive", k_dedup_alive<<<l.grid, 256, 0, s>>>(b, w));
  PT_TRACE(l, s, "k_dedup_triplets", k_dedup_triplets<<<l.grid, 256, 0, s>>>(b, w));
  PT_TRACE(l, s, "scan", launch_scan(w.alive, w.alive_scan, &b.cnt[CNT_SCAN_NT], b.scan_part, s));
  PT_TRACE(l, s, "k_compact", k_compact<<<l.grid, 256, 0, s>>>(b, w));
  PT_TRACE(l, s, "k_event_offsets", k_event_offsets<<<l.grid, 256, 0, s>>>(b));
}

}  // namespace ptca
