// Export of results and intermediates with event-local input indices (the batch
// stores batch-wide input indices internally).
#include "ptca_internal.cuh"

namespace ptca {

namespace {

__device__ __forceinline__ void to_local(const Buffers& b, int E, const int32_t* src, int32_t* dst,
                                         int32_t* ev) {
  const int e = find_event(b.hit_off, E, src[0]);
  const int32_t off = b.hit_off[e];
#pragma unroll
  for (int k = 0; k < kMaxHits; ++k) dst[k] = src[k] >= 0 ? src[k] - off : -1;
  *ev = e;
}

// Cleaned ntuplets (the stage path; the whole-batch graph's cleaning writes them itself).
__global__ void k_export_ntuplets(Buffers b) {
  const uint64_t S = b.cnt[CNT_SV];
  const int E = b.hdr->n_events;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < S; j += stride) {
    const uint32_t t = b.sv[j];
    int32_t ev;
    to_local(b, E, b.nt_hits + (uint64_t)t * kMaxHits, b.exp_hits + j * kMaxHits, &ev);
    b.exp_n[j] = b.nt_n[t];
  }
}

__global__ void k_export_candidates(Buffers b) {
  const uint64_t T = b.cnt[CNT_SCAN_NT];
  const int E = b.hdr->n_events;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += stride) {
    int32_t ev;
    to_local(b, E, b.nt_hits + t * kMaxHits, b.exp_hits + t * kMaxHits, &ev);
    b.exp_n[t] = b.nt_n[t];
    b.exp_q[t] = fabsf(b.nt_q[t]);
    b.exp_ev[t] = ev;
  }
}

// A warp takes 32 sorted hits, one per lane, and slot by slot writes the cells of their
// incoming segments, one per lane, at the cells' own slots (the caller has marked every slot a
// hole): an event of few hits has one or two cells in a segment, a large one a hundred.
// pt_get_cells on 20000 events of 4 hits 119 us, 150 with a warp per hit.
__global__ void k_export_cells(Buffers b, int32_t B, int max_inner, uint64_t cap_cells,
                               int32_t* out3) {
  const uint64_t nc = min(b.cnt[CNT_CELLS], (unsigned long long)cap_cells);
  const int E = b.hdr->n_events;
  const uint32_t n_sorted = b.bin_start[E * kLayers * B];
  const uint32_t stride = gridDim.x * blockDim.x, lane = lane_id();
  for (uint32_t s0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); s0 < n_sorted; s0 += stride) {
    const uint32_t s = s0 + lane;
    const bool valid = s < n_sorted;
    const int32_t go = valid ? (int32_t)b.perm[s] : 0;
    const int e = find_event(b.hit_off, E, go);
    const int32_t off = b.hit_off[e];
    for (int k = 0; k < max_inner; ++k) {
      const uint2 sg = valid ? b.seg[(uint64_t)s * max_inner + k] : make_uint2(0u, 0u);
      const uint32_t end = warp_incl_scan(sg.y), total = __shfl_sync(kFull, end, 31);
      for (uint32_t i0 = 0; i0 < total; i0 += 32) {
        const uint32_t i = i0 + lane;
        uint32_t h = 0;  // the lane whose segment holds the i-th cell
#pragma unroll
        for (uint32_t o = 16; o > 0; o >>= 1)
          if (i >= __shfl_sync(kFull, end, h + o - 1)) h += o;
        const uint32_t first = __shfl_sync(kFull, sg.x, h);
        const uint32_t before = __shfl_sync(kFull, end, h) - __shfl_sync(kFull, sg.y, h);
        const int32_t h_go = __shfl_sync(kFull, go, h), h_off = __shfl_sync(kFull, off, h);
        const int32_t h_e = __shfl_sync(kFull, e, h);
        const uint64_t c = (uint64_t)first + (i - before);
        if (i >= total || c >= nc) continue;
        out3[c * 3 + 0] = (int32_t)b.perm[b.cell_in[c]] - h_off;
        out3[c * 3 + 1] = h_go - h_off;
        out3[c * 3 + 2] = h_e;
      }
    }
  }
}

__global__ void k_export_links(Buffers b, uint64_t cap_links, int32_t* out4, float* outq,
                               bool gated) {
  const uint64_t nl = min(b.cnt[CNT_LINKS], (unsigned long long)cap_links);
  const int E = b.hdr->n_events;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t l = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; l < nl; l += stride) {
    const Link k = b.link[l];
    if (k.src == kHole || (gated && !b.gate_keep[l])) continue;  // hole or removed link
    const int32_t g0 = (int32_t)b.perm[b.cell_in[k.src]], g1 = (int32_t)b.perm[k.h1];
    const int32_t g2 = (int32_t)b.perm[k.h2];
    const int e = find_event(b.hit_off, E, g0);
    const int32_t off = b.hit_off[e];
    out4[l * 4 + 0] = g0 - off;
    out4[l * 4 + 1] = g1 - off;
    out4[l * 4 + 2] = g2 - off;
    out4[l * 4 + 3] = e;
    outq[l] = k.q;
  }
}

}  // namespace

void launch_export_ntuplets(const Buffers& b, const Launch& l, cudaStream_t s) {
  PT_TRACE(l, s, "k_export_ntuplets", k_export_ntuplets<<<l.grid, 256, 0, s>>>(b));
}
void launch_export_candidates(const Buffers& b, const Launch& l, cudaStream_t s) {
  k_export_candidates<<<l.grid, 256, 0, s>>>(b);
}
void launch_export_cells(const Buffers& b, const Params& p, const Launch& l, int32_t* out3,
                         cudaStream_t s) {
  k_export_cells<<<l.grid, 256, 0, s>>>(b, p.phi_bins, p.pairs.max_inner, (uint64_t)p.max_cells,
                                        out3);
}
void launch_export_links(const Buffers& b, const Params& p, const Launch& l, int32_t* out4,
                         float* outq, cudaStream_t s, bool gated) {
  k_export_links<<<l.grid, 256, 0, s>>>(b, (uint64_t)p.max_links, out4, outq, gated);
}

}  // namespace ptca
