// Internal declarations of the GB300 pixel-track CA library: device buffer layout,
// exact float32 cut predicates and the host-side launchers of every kernel.
//
// Every kernel is a fixed-grid, grid-stride kernel that reads its work size from
// device memory (batch header or a device counter).  No stage needs a host round
// trip, so the whole chain of a batch can be replayed from one captured CUDA graph
// whatever the batch's hit, cell or link counts are.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pt_ca.h"

namespace ptca {

constexpr int kLayers = 10;
constexpr int kMaxHits = 6;                // longest chain of the layer graph
constexpr int kMaxCellsPerNt = kMaxHits - 1;
constexpr int kMaxOuter = 6;               // outer layers paired with one inner layer
constexpr int kMaxInner = 6;               // inner layers paired with one outer layer
constexpr int kMaxPairs = 64;              // layer pairs of one table
constexpr int kStage = 256;                // staged doublets per (hit, outer layer)
constexpr int kLocalLinks = 8;             // links of one cell kept in registers
constexpr int kRankBits = 29;              // duplicate-cleaning key: rank field width

// device counters (unsigned long long)
enum : int {
  CNT_CELLS = 0,
  CNT_LINKS = 1,
  CNT_NT = 2,
  CNT_STATUS = 3,
  CNT_SCAN_BINS = 4,  // sizes for the device-wide scans
  CNT_SCAN_HITS = 5,
  CNT_SCAN_NT = 6,    // ntuplets before cleaning that were stored
  CNT_GATE_KEPT = 7,
  CNT_SV = 8,         // cleaned ntuplets
  CNT_SCORE_STATUS = 9,  // status bits of the standalone gate scoring (pt_gate_score)
  CNT_CELLS_USED = 10,  // cells written (CNT_CELLS counts reserved slots incl. holes)
  CNT_LINKS_USED = 11,  // links written (CNT_LINKS counts reserved slots incl. holes)
  CNT_SCAN_EV = 13,     // events (size of the scan over per-event vertex counts)
  CNT_VTX = 14,         // vertices of the batch
  CNT_RAW_STATUS = 15,  // raw input: status bits (RAW_*), not reset by the chain
  CNT_RAW_DIGIS = 16,   // raw input: digis of the batch (size of the run-flag scan)
  CNT_RAW_RUNS = 17,    // raw input: module runs (size of the hit-count scan)
  CNT_RAW_HITS = 18,    // raw input: hits made from the digis
  CNT_RAW_BIG = 19,     // raw input: long module runs listed for the block-per-run launch
  CNT_NT_BEST = 21,     // ntuplets on best_list
  CNT_DEBUG_SITE = 22,  // debug build: the first failing bounds check (DebugSite)
  CNT_NT_TIES = 23,     // nonzero: ntuplets of the same hit count and q met in a cell
  // The searches' work counters, each in a 128-byte line of its own: a warp adds to one for
  // nearly every hit of a single event, and to CNT_CELLS or CNT_LINKS meanwhile (one gated
  // pileup-200 event 345 us with all of them in one line, 330 so).
  CNT_DBL_WORK = 32,    // doublet search: next chunk of sorted hits
  CNT_LNK_WORK = 48,    // link search: next chunk of sorted middle hits
  CNT_N = 64
};
// raw-input status bits (cnt[CNT_RAW_STATUS])
enum : unsigned long long {
  RAW_INVALID = 1ull,           // bad module, pixel, adc or pixel order
  RAW_RUN_CAPACITY = 2ull,      // more than 1024 digis of one module in one event
  RAW_CLUSTER_CAPACITY = 4ull,  // a cluster of more than 128 pixels
  RAW_HIT_CAPACITY = 8ull,      // more hits than max_hits
};
// status bits
enum : unsigned long long {
  ST_CELLS = 1ull,
  ST_LINKS = 2ull,
  ST_NT = 4ull,
  ST_LAYER = 8ull,
  ST_GATE_TIMEOUT = 16ull,  // a bounded wait in the gate kernel expired
  ST_VTX = 32ull,           // an event has more tracks for vertexing than a block sorts
  ST_DEBUG = 64ull,         // a bounds check of the debug build failed (cnt[CNT_DEBUG_SITE])
};

// Sites of the debug build's bounds checks (the first one that fails is recorded).
enum DebugSite : unsigned {
  DBG_BIN_SCATTER = 1,   // sorted position of a hit < hits
  DBG_DBL_WINDOW = 2,    // a doublet window inside the sorted hits
  DBG_DBL_CELL = 3,      // a cell slot < max_cells
  DBG_CON_WINDOW = 4,    // a forward window inside the sorted hits
  DBG_CON_INCOMING = 5,  // an incoming cell id < cell slots
  DBG_CON_BUCKET = 6,    // a bucket range inside the staged piece
  DBG_CON_QUEUE = 7,     // queued pairs <= queue size
  DBG_CON_LINK = 8,      // a link slot < max_links
  DBG_TGT_SEGMENT = 9,   // a target's incoming segment inside the cell slots
  DBG_NT_LINKS = 10,     // a cell's link run inside the link slots
  DBG_NT_CELL = 11,      // a link target < cell slots
  DBG_FIT_HITS = 12,     // 3..6 hits per fitted ntuplet
  DBG_FB_RECORD = 13,    // a fishbone record position < max_links
};

// Gate parameters on the device: W1 and W2 as bf16 in the tensor-core operand layout,
// biases and the last layer in float32.
constexpr int kGateFeat = 12;
constexpr int kGateK1 = 16;   // layer-1 K padded to the MMA K
constexpr int kGateHidden = 64;
constexpr int kGateParams = 5057;
struct GateWeights {
  uint16_t w1[kGateHidden * kGateK1];      // core-matrix layout, see gate.cu
  uint16_t w2[kGateHidden * kGateHidden];  // core-matrix layout
  float b1[kGateHidden];
  float b2[kGateHidden];
  float w3[kGateHidden];
  float b3;
  float tau;
};

// Link state of a cell, one record because the later stages reach the cells at random (161M
// cells on 64 pileup-200 events, one of 16 on a link).  Written for the cells that take part
// in links only: the link stage sets up its sources, the target pass the targets without
// links of their own (leaves).
struct alignas(8) CellState {
  uint32_t head;    // a source's latest out-link slot, the head of its out-link list (kHole:
                    //   no link passed); a leaf: one of the links that end on it
  uint8_t has_in;   // a link ends on the cell (masked forms: a kept link; sources only)
  uint8_t has_out;  // masked forms: a kept link starts from the cell
  uint8_t kill;     // removed by the fishbone step
  uint8_t pad;
};
static_assert(sizeof(CellState) == 8, "one 8-byte record");

// A link in one memory sector, all that a step of the ntuplet walk needs.  The link stage
// writes `next` and the second half, the target pass the rest.
struct alignas(32) Link {
  uint32_t next;  // the source's next out-link slot (kHole: last)
  uint32_t dst;   // target cell
  uint32_t head;  // the target's out-link list head (kHole: a leaf)
  uint32_t h2;    // the target's outer hit (sorted index)
  uint32_t src;   // source cell (kHole: an unused slot)
  uint32_t code;  // the target before the target pass: outer hit | slot << 29
  uint32_t h1;    // middle hit (sorted index)
  float q;        // link quality
};
static_assert(sizeof(Link) == 32, "one memory sector");
__device__ __forceinline__ uint4* link_lo(Link* l) { return (uint4*)l; }
__device__ __forceinline__ uint4* link_hi(Link* l) { return (uint4*)l + 1; }

// Duplicate-cleaning keys.  A cell of an ntuplet is named by a link slot, a source by its
// list's head and a leaf by the in-link in its state, so the keys lie in 16 bytes per link
// (85 MB on 64 pileup-200 events, which stays in L2) instead of among all cells (2.6 GB).
// Reading them back (k_dedup_best) takes 0.13 instead of 0.38 ms.
struct alignas(16) LinkBest {
  unsigned long long src, leaf;  // of the source headed by the slot, of the leaf named by it
};

// What a call says about its batch; the kernels read it, so that one captured graph serves
// any batch, its inputs wherever they lie and its outputs wherever they go.
struct BatchHeader {
  int32_t n_events;
  int32_t n_hits;
  int32_t raw;  // the hits were made from raw digis
  int32_t pad;
  // where the binning pass takes the hits from, copying them to in_x, ...  (x NULL: they
  // are there)
  const float *x, *y, *z;
  const uint8_t* layer;
  // where the whole-batch graph writes the cleaned ntuplets and tracks (each may be NULL)
  // when there are at most out_cap of them and nothing went wrong; otherwise the ntuplets
  // go to the export staging
  int32_t* out_hits;
  uint8_t* out_n;
  pt_track* out_tracks;
  int64_t* out_off;
  int64_t out_cap;
};
constexpr size_t kHeaderBytes = 256;  // hit_off follows, and small host inputs follow that
static_assert(sizeof(BatchHeader) <= kHeaderBytes, "header fits its place");
// Host inputs of up to kSmallHits hits go up in one copy, packed behind the header: an event
// of 205 hits 94 us for the whole call instead of 103 with a copy per array, of 3666 hits 120
// instead of 124, of 7314 no less.  Results of up to kSmallTracks tracks come back in a pinned
// block instead of in a copy per array: 42 tracks 94 instead of 129 us into ordinary memory
// and 89 instead of 99 into pinned memory, 3107 tracks 180 instead of 192, but 166 instead of
// 160 into pinned memory.
constexpr int64_t kSmallHits = 4096;
constexpr int64_t kSmallTracks = 4096;

// The layer-pair table of a context, as the kernels read it (a kernel argument):
// outer[L][k], k < n_outer[L], are the outer layers paired with inner layer L, inner[L][k],
// k < n_inner[L], the inner layers paired with outer layer L (a hit's incoming segments
// are numbered by these slots), slot[L][Li] = k with inner[L][k] == Li (-1 if none), and
// max_inner = the largest n_inner (the number of incoming segments stored per hit).
struct PairTable {
  int8_t outer[kLayers][kMaxOuter];
  int8_t n_outer[kLayers];
  int8_t inner[kLayers][kMaxInner];
  int8_t n_inner[kLayers];
  int8_t slot[kLayers][kLayers];
  int8_t max_inner;
};

// Builds the table of n (inner, outer) pairs, in the given order; false if a pair is out
// of range, repeated or pairs a layer with itself, if a layer gets more than kMaxOuter
// outer or kMaxInner inner layers, or if the layer graph has a cycle or a path of more
// than kMaxHits - 1 pairs.
bool make_pair_table(int n, const int32_t* inner, const int32_t* outer, PairTable* t);
// The chain's 13 pairs: barrel 0-1, 1-2, 2-3, and per side the three inner barrel
// layers and the disk chain into the first disk (0/1/2-4, 4-5, 5-6; 0/1/2-7, 7-8, 8-9).
PairTable default_pair_table();

struct Params {
  pt_cuts cuts;
  PairTable pairs;
  long long wait_cycles;  // limit of the bounded device-side waits (SM clock cycles)
  float bfield;
  int32_t phi_bins;
  int64_t max_events, max_hits, max_cells, max_links, max_ntuplets;
};

// Device buffers carved out of one workspace block (see layout() in runtime.cu).
struct Buffers {
  BatchHeader* hdr;
  unsigned long long* cnt;   // [CNT_N]
  // inputs, batch order
  float* in_x;
  float* in_y;
  float* in_z;
  uint8_t* in_layer;
  int32_t* hit_off;          // [max_events + 1], directly after the header; a small
                             //   batch's inputs follow, into hit4, until it is written
  uint32_t* in_bin;          // [max_hits] global bin of input hit (or ~0)
  uint32_t* in_rank;         // [max_hits] rank within the bin
  // hits sorted by (event, layer, phi bin)
  float4* hit4;              // [max_hits] (x, y, z, r)
  uint32_t* perm;            // [max_hits] sorted -> input (batch) index
  uint32_t* hbin;            // [max_hits] global bin of sorted hit
  uint32_t* bin_cnt;         // [max_events*10*B + 1]
  uint32_t* bin_start;       // [max_events*10*B + 1]
  uint32_t* layer_rmax;      // [max_events*10] float bits of max r per event layer
  float* layer_asin;         // [max_events*10] asin(kmax r_max / 2) per event layer,
                             //   +inf when kmax r_max / 2 >= 0.7
  uint32_t* layer_rmin;      // [max_events*10] float bits of min r per event layer (+inf
                             //   for an empty layer)
  float* layer_asin_lo;      // [max_events*10] asin(kmax r_min / 2) (0 where that is >= 0.7
                             //   or the layer is empty)
  uint32_t* layer_zmin;      // [max_events*10] order keys (float_order_key) of min and max
  uint32_t* layer_zmax;      //   z per event layer (~0 and 0 for an empty layer)
  // incoming segments: per sorted (outer) hit and inner-layer slot, the cells ending on
  // the hit from that layer, cells [x, x + y), ordered by inner hit; the table's
  // max_inner slots per hit, all written; before the doublet search the hit's windows
  uint2* seg;                // [max_hits*kMaxInner]
  // cells
  uint32_t* cell_in;         // [max_cells] inner hit (sorted index); the outer hit is the
                             //   one whose segment holds the cell
  CellState* cell;           // [max_cells] cells that take part in links
  uint32_t* fb_cnt;          // [max_hits + 1] fishbone: active cells per outer hit (all zero
                             //   again after the step)
  uint32_t* fb_start;        // [max_hits + 1]   and their first position in fb_rec
  float4* fb_rec;            // [max_links * 2] active cells grouped by outer hit: vector to
                             //   the hit and |.|^2; list head, inner hit's input index,
                             //   layer, sensor (the memory of gate_x, free by then)
  Link* link;                // [max_links]
  LinkBest* link_best;       // [max_links]
  // ntuplets before cleaning
  int32_t* nt_hits;          // [max_ntuplets*6] batch input index, -1 pad
  uint32_t* nt_cells;        // [max_ntuplets*5] link slots naming the cells (LinkBest), kHole
                             //   padded; the last one names a leaf, or a source where nt_q
                             //   is negative (masked forms: none of its links was kept)
  uint8_t* nt_n;             // [max_ntuplets]
  float* nt_q;               // [max_ntuplets] quality q >= 0, or -q (see nt_cells)
  uint32_t* nt_next;         // [max_ntuplets] next survivor with the same first hit (kHole:
                             //   none)
  // duplicate cleaning and canonical order (hits are batch input indices here)
  uint32_t* nt_head;         // [max_hits] list of the survivors that start at the hit (kHole:
                             //   none)
  uint32_t* sv_cnt;          // [max_hits + 1] surviving ntuplets that start at the hit (the
                             //   memory of fb_cnt)
  uint32_t* sv_start;        // [max_hits + 1]   and the first one's place (that of fb_start)
  uint32_t* best_list;       // [max_ntuplets] ntuplets that may survive (kHole: it did not)
  uint8_t* used;             // [max_hits] on a surviving ntuplet of four or more hits
  uint32_t* sv;              // [max_ntuplets] cleaned ntuplets in canonical order
  int64_t* ev_nt_off;        // [max_events + 1]
  pt_track* tracks;          // [max_ntuplets]
  // primary vertices (pt_find_vertices)
  pt_vertex* vtx_stage;      // [max_ntuplets / 2 + 1] event e's vertices from floor(t0 / 2)
  pt_vertex* vtx;            // [max_ntuplets / 2 + 1] the batch's vertices, events in order
  int32_t* trk_vtx;          // [max_ntuplets] vertex of each track, -1 for none
  uint32_t* ev_nv;           // [max_events + 1] vertices per event (large batches: scanned in
                             //   place, vertices before each event)
  int64_t* ev_vtx_off;       // [max_events + 1] vertices before each event
  // learned gate (valid when enabled)
  uint16_t* gate_x;          // [max_links*16] bf16 features per link slot (12 used)
  float* gate_score;         // [max_links] logit per link slot
  uint8_t* gate_keep;        // [max_links] 1 where the link passes the gate
  int32_t* exp_hits;         // [max_ntuplets*6] export staging (event-local indices)
  uint8_t* exp_n;            // [max_ntuplets]
  float* exp_q;              // [max_ntuplets]
  int32_t* exp_ev;           // [max_ntuplets]
  uint32_t* scan_part;       // [kScanBlocks + 1]
};

constexpr int kScanBlocks = 256;

// Raw-input scratch (allocated on the first pt_load_raw): the digis and the per-digi /
// per-run arrays of the clustering; max_digis entries (+1 for the scans).
struct RawBuffers {
  int n_events = 0;
  int64_t* digi_off = nullptr;   // [max_events + 1] event e owns digis [off[e], off[e+1])
  uint64_t* words = nullptr;     // [max_digis] packed digis
  uint32_t* flag = nullptr;      // [max_digis + 1] 1 where a module run starts
  uint32_t* run_scan = nullptr;  // [max_digis + 1] runs starting before each digi
  uint32_t* run_first = nullptr; // [max_digis + 1] first digi of each run (+ end)
  uint32_t* run_nh = nullptr;    // [max_digis + 1] hits of each run
  uint32_t* run_hoff = nullptr;  // [max_digis + 1] first hit of each run (+ total)
  float4* stage = nullptr;       // [max_digis] hits (x, y, z, layer bits) at digi positions
  uint32_t* big_runs = nullptr;  // aliases flag (free once the runs are numbered): long runs
  uint32_t* scan_part = nullptr; // the context's scan partials
  unsigned long long* cnt = nullptr;  // the context's counters
};

// Optional per-kernel timing of the stage calls (pt_set_tracing): CUDA events on the
// launching stream around every kernel; never active while the whole-batch graph is
// captured.  Defined in runtime.cu.
struct Tracer;
size_t trace_begin(Tracer* t, cudaStream_t s);
void trace_end(Tracer* t, const char* name, size_t i0, cudaStream_t s);
#define PT_TRACE(l, s, name, ...)                                  \
  do {                                                             \
    const size_t pt_t0_ = (l).tr ? trace_begin((l).tr, (s)) : 0;   \
    __VA_ARGS__;                                                   \
    if ((l).tr) trace_end((l).tr, (name), pt_t0_, (s));            \
  } while (0)

struct Launch {
  int sms;                // multiprocessors
  int grid;               // generic persistent grid (blocks of 256 threads)
  int sgrid;              // grid of the doublet search (warp per hit)
  Tracer* tr = nullptr;   // per-kernel timing, when enabled
};

#ifdef __CUDACC__
// Launches a kernel that may be scheduled while the kernel before it on the stream drains
// (programmatic dependent launch, also inside a captured graph): a chain of some 20 kernels
// on one small event spends more time between them than in them.  The kernel must begin
// with pdl_sync() (directly, or before it touches anything an earlier kernel wrote).
template <class... P, class... A>
inline void launch_pdl(void (*k)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s,
                       A... a) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k, static_cast<P>(a)...);
}
// Waits until the kernels before this one have completed and their writes are visible; every
// thread of a kernel calls it before it can return, so that a kernel's completion implies
// that of all before it.  pdl_sync also lets the next kernel be scheduled at once; the
// kernels that fill the GPU for long use pdl_wait alone: blocks of the next kernel that sit
// waiting on the multiprocessors cost them more than the launch that is hidden (64
// pileup-200 events 6724 instead of 6564 us).
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_sync() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

// Sets the calling thread's pt_last_error() message.
void set_last_error(const char* msg);

// Requests a server has completed since it was created (for the router's balancing).
int64_t server_finished(pt_server* s);

// Asynchronous pieces of a batch for the request server (runtime.cu): read-back of the
// counters, status check of that copy, and copies of the cleaned ntuplets, tracks and
// per-event offsets into host memory, each completion recorded on `done`.
cudaStream_t ctx_stream(pt_ctx* c);
// pt_enqueue_batch that returns at once; the caller keeps the inputs until the batch is done.
pt_status ctx_enqueue_async(pt_ctx* c, int n_events, const int64_t* hit_offsets, const float* x,
                            const float* y, const float* z, const uint8_t* layer, int on_device);
pt_status ctx_counters_async(pt_ctx* c, cudaEvent_t done);
pt_status ctx_read_counters(pt_ctx* c, int64_t* n_ntuplets);
pt_status ctx_results_async(pt_ctx* c, int64_t S, int32_t* hits, uint8_t* nhits,
                            pt_track* tracks, int64_t* event_offsets, cudaEvent_t done);

// ------------------------------------------------------------------ launchers
// device arrays of n hits to the context's input arrays
void launch_take_inputs(const Buffers& b, const float* x, const float* y, const float* z,
                        const uint8_t* layer, int64_t n, const Launch& l, cudaStream_t s);
void launch_clear(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s);
void launch_bin_hits(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s);
void launch_doublets(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s);
// gated = true: the link search also writes each link's gate features and source cell,
// and leaves the in/out flags to the gate (launch_gate)
void launch_connect(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                    bool gated = false);
// Fishbone step and the link filter after it (keep mask and link flags of the ntuplet
// search); gated: the gate's keep mask is the starting point.
void launch_fishbone(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                     bool gated);
// Debug build: records a failure of bounds check `site` as a failing check does.
cudaError_t launch_debug_inject(const Buffers& b, unsigned site, cudaStream_t s);
// Ntuplet search, cleaning and order; gated: the search follows the keep mask.  The first
// form is the whole-batch graph's (the survivors' lists must be as launch_clear leaves
// them; the ntuplets also go out), the second the stage call's, which may run again on the
// same links.
void launch_ntuplets(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                     bool gated);
void launch_ntuplet_steps(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                          bool gated);
// results: the tracks also go where the batch header says
void launch_fit(const Buffers& b, const Params& p, const Launch& l, cudaStream_t s,
                bool results = false);
// raw digis -> hits in the chain's input arrays, per-event offsets and header
cudaError_t launch_raw(const RawBuffers& r, const Buffers& b, const pt_module* mods, int n_mod,
                       int64_t cap_hits, const Launch& l, cudaStream_t s);
// primary vertices of the fitted tracks of n_events events (tracks with >= min_hits
// hits, groups cut at z0 steps > dz)
cudaError_t launch_vertices(const Buffers& b, const Params& p, int n_events, int32_t min_hits,
                            float dz, const Launch& l, cudaStream_t s);
// scan of n+1 entries: out[i] = sum(in[0..i)), n = *n_dev
void launch_scan(const uint32_t* in, uint32_t* out, const unsigned long long* n_dev,
                 uint32_t* part, cudaStream_t s);
// the same where part[] holds the sums of the blocks' shares (scan_share) already
void launch_scan_counted(const uint32_t* in, uint32_t* out, const unsigned long long* n_dev,
                         const uint32_t* part, cudaStream_t s);
// learned gate: features, tensor-core MLP and link pruning (enabled contexts only);
// gate_prepare() sets the MLP kernel's shared-memory attribute (call before capture)
cudaError_t gate_prepare();
void launch_gate(const Buffers& b, const Params& p, const Launch& l, const GateWeights* w,
                 cudaStream_t s);
// scores of n feature rows (float32 [n][12], device) with the gate's MLP -> out [n]
void launch_gate_score(const GateWeights* w, const float* feat, int64_t n, float* out,
                       unsigned long long* status, int sms, long long wait_cycles,
                       cudaStream_t s);
// float32 features of the current links (gated: kept only) -> out [slots][12]
void launch_export_link_features(const Buffers& b, const Params& p, const Launch& l, bool gated,
                                 float* out, cudaStream_t s);
// gate training: mean BCE loss and its gradient (zeroed first); Adam step
cudaError_t launch_gate_grad(const float* w, const float* X, const float* y, int64_t n,
                             float* grad, float* loss, int sms, cudaStream_t s);
cudaError_t launch_gate_adam(float* w, float* m, float* v, const float* g, int64_t n, float lr,
                             float b1, float b2, float eps, int step, cudaStream_t s);
// exports with event-local input indices
void launch_export_ntuplets(const Buffers& b, const Launch& l, cudaStream_t s);
void launch_export_candidates(const Buffers& b, const Launch& l, cudaStream_t s);
// cells -> out3 [n][3] (inner, outer, event); links -> out4 [n][4] (h0, h1, h2, event), q
void launch_export_cells(const Buffers& b, const Params& p, const Launch& l, int32_t* out3,
                         cudaStream_t s);
void launch_export_links(const Buffers& b, const Params& p, const Launch& l, int32_t* out4,
                         float* outq, cudaStream_t s, bool gated = false);

// ------------------------------------------------------------ device helpers
#ifdef __CUDACC__
constexpr unsigned kFull = 0xffffffffu;

// Entries of one scan block's share of n, a multiple of four so that aligned arrays are read
// four at a time.
__device__ __forceinline__ uint64_t scan_share(uint64_t n) {
  return ((n + kScanBlocks - 1) / kScanBlocks + 3) & ~3ull;
}

// Correctly rounded float32 operations that the compiler never contracts into FMA.
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fsqrt(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }

// Order-preserving map of a float to an unsigned key (for atomicMin / atomicMax), and
// back.
__device__ __forceinline__ uint32_t float_order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float float_from_order_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Whether a layer whose hits lie in the r-z box [rlo, rhi] x [zlo, zhi] can hold a
// partner of the hit (r, z), outward (larger r) or inward, that passes D2 and D3.  Both
// cuts bound the r-z slope s of the cell: |s| <= cotmax, and the line's z at r = 0,
// which is z - r s from either hit, within +-z0max.  Seen from the hit, the slopes of
// the box's points with a positive radial step fill the interval between its corners'
// slopes; the layer is ruled out only when that interval lies wholly beyond the allowed
// one, compared in multiplied form with margins (1e-3 on slopes, 1e-3 cm on z) far above
// float32 rounding.  Boxes reaching to the hit's radius or inside it are kept (D0
// decides them).
__device__ __forceinline__ bool rz_box_reachable(const pt_cuts& c, float r, float z, float rlo,
                                                 float rhi, float zlo, float zhi, bool outward) {
  float d0, d1, e0, e1;  // radial steps and z steps (towards the partner) over the box
  if (outward) {
    d0 = fmaxf(rlo - r, 0.0f), d1 = rhi - r, e0 = zlo - z, e1 = zhi - z;
  } else {
    d0 = fmaxf(r - rhi, 0.0f), d1 = r - rlo, e0 = z - zhi, e1 = z - zlo;
  }
  if (!(d1 > 0.0f) || !(r > 0.0f)) return true;
  const float lo = fmaxf((z - c.z0max) / r, -c.cotmax);
  const float hi = fminf((z + c.z0max) / r, c.cotmax);
  const float slo = lo - 1e-3f * (1.0f + fabsf(lo)), shi = hi + 1e-3f * (1.0f + fabsf(hi));
  e0 -= 1e-3f;
  e1 += 1e-3f;
  // largest slope of the box below slo, or its smallest above shi
  const bool below = e1 >= 0.0f ? e1 < slo * d0 : e1 < slo * d1;
  const bool above = e0 <= 0.0f ? e0 > shi * d0 : e0 > shi * d1;
  return !(below || above);
}

// Doublet cuts D0..D4 on (x, y, z, r) of the inner and outer hit, in the library's
// fixed evaluation order (see pt_cuts in pt_ca.h).
// The four cheap cuts are all evaluated before one branch skips the square root: leaving at
// each of them took 1463 instead of 1432 us in the doublet search of 64 pileup-200 events,
// no branch at all 3 % longer than that in the link search.
__device__ __forceinline__ bool doublet_pass(const pt_cuts& c, float4 hi, float4 ho) {
  const float dx = fsub(ho.x, hi.x), dy = fsub(ho.y, hi.y);
  const float dr = fsub(ho.w, hi.w), dz = fsub(ho.z, hi.z);
  const bool d0 = dr > 0.0f;
  const bool d1 = fadd(fmul(hi.x, ho.x), fmul(hi.y, ho.y)) > 0.0f;
  const bool d3 = fabsf(fsub(fmul(hi.z, dr), fmul(hi.w, dz))) <= fmul(c.z0max, dr);
  const bool d4 = fabsf(dz) <= fmul(c.cotmax, dr);
  const float l2 = fmul(fabsf(fsub(fmul(hi.x, ho.y), fmul(hi.y, ho.x))), 2.0f);
  if (!(d0 & d1 & d3 & d4)) return false;
  const float r2 = fmul(c.kmax, fmul(fmul(hi.w, ho.w), fsqrt(fadd(fmul(dx, dx), fmul(dy, dy)))));
  return l2 <= r2;
}

// The same decision as doublet_pass with fewer operations, for the searches.  The curvature
// cut is decided from its squared form c^2 <= t, t = (kmax ri ro / 2)^2 (dx^2 + dy^2), with c
// the exact form's cross product: both sides' rounding is below 1.5e-6 t, so where c^2 and t
// differ by more than 4e-6 t + tiny the squared form decides, and elsewhere (or where either
// is not finite) doublet_pass itself.  `half_k` is kmax/2 times one hit's radius, `r` the
// other's radius.  The half-plane cut x.x + y.y > 0 is not looked at: a window_tiny() of
// infinity, which sends every pair to doublet_pass, stands wherever the window does not
// imply it.  The searches are bound by the instructions they issue; without the square root
// and the half-plane cut the doublet search of 64 pileup-200 events takes 1331 instead of
// 1434 us, the whole call with it in the link search as well 5735 instead of 5790.
constexpr float kHalfPlane = 1.569f;  // pi/2, less the azimuth's rounding and that of the cut
constexpr uint32_t kWindowExact = 0x80000000u;  // a window's flags, in its last word
constexpr uint32_t kWindowWraps = 0x80000000u;  //   and in its first
__device__ __forceinline__ float window_tiny(uint32_t flagged) {
  return flagged & kWindowExact ? __int_as_float(0x7f800000) : 1e-20f;
}
// The flag of a window of +-win (and the bins that it cuts) between a hit of radius r and hits
// of radii [rlo, rhi].
__device__ __forceinline__ uint32_t window_flag(const pt_cuts& c, float win, float bins_per_rad,
                                                float r, float rlo, float rhi) {
  const bool implied = (win - kHalfPlane) * bins_per_rad < -1.0f && fminf(r, rlo) > 1e-9f &&
                       r < 1e9f && rhi < 1e9f && c.kmax >= 0.0f;
  return implied ? 0u : kWindowExact;
}

// Azimuth of a hit from 0, and the bins [lo, hi) that the range phi -+ win touches: lo < 0 or
// hi > B where it wraps, 0 and B where it covers them all.  win has room (1e-4 rad) for the
// rounding of the azimuths and of their bins.  Around the hit's bin instead of its azimuth the
// range had to have two bins more at either end, half of them beyond need: a hit of a pileup-200
// event has 151 doublet and 170 link candidates with 256 bins (237 and 244 then), 138 and 158
// with 512 (181 and 197), 128 and 150 with 2048 (139 and 160).
__device__ __forceinline__ float azimuth(float4 h) {  // from 0
  return atan2f(h.y, h.x) + 3.14159265358979323846f;
}
__device__ __forceinline__ int2 window_bins(float phi, float win, float bins_per_rad, int32_t B) {
  win = fmaxf(win, 0.0f);
  int lo = min((int)floorf((phi - win) * bins_per_rad), B - 1);
  int hi = (int)floorf((phi + win) * bins_per_rad) + 1;
  if (hi - lo >= B) {
    lo = 0;
    hi = B;
  }
  return make_int2(lo, hi);
}
__device__ __forceinline__ bool doublet_quick(const pt_cuts& c, bool in, float4 hi, float4 ho,
                                              float half_k, float r, float tiny) {
  const float dx = ho.x - hi.x, dy = ho.y - hi.y;
  const float dr = fsub(ho.w, hi.w), dz = fsub(ho.z, hi.z);
  const bool d0 = dr > 0.0f;
  const bool d3 = fabsf(fsub(fmul(hi.z, dr), fmul(hi.w, dz))) <= fmul(c.z0max, dr);
  const bool d4 = fabsf(dz) <= fmul(c.cotmax, dr);
  const float cross = fsub(fmul(hi.x, ho.y), fmul(hi.y, ho.x));
  const float a = half_k * r;
  const float t = a * a * fmaf(dx, dx, dy * dy);
  const float diff = fmaf(cross, cross, -t);
  bool pass = in & d0 & d3 & d4;
  if (pass & !(fabsf(diff) > fmaf(4e-6f, t, tiny)))
    pass = doublet_pass(c, hi, ho);
  else
    pass &= diff < 0.0f;
  return pass;
}

// r-z alignment C1 only (cheap first test of a link).
__device__ __forceinline__ bool link_c1(const pt_cuts& c, float4 p0, float4 p1, float4 p2) {
  const float lc1 = fabsf(fsub(fmul(fsub(p1.z, p0.z), fsub(p2.w, p0.w)),
                               fmul(fsub(p2.z, p0.z), fsub(p1.w, p0.w))));
  const float rc1 = fadd(fmul(c.rz0, fsub(p2.w, p0.w)), fmul(c.rz1, fabsf(fsub(p2.z, p0.z))));
  return lc1 <= rc1;
}

// Curvature C2 and beam-spot distance C3 of the circle through three hits; q gets the
// distance (link quality) when both pass.
__device__ __forceinline__ bool link_c23(const pt_cuts& c, float4 p0, bool first_on_b0, float4 p1,
                                         float4 p2, float& q) {
  const float ax = fsub(p1.x, p0.x), ay = fsub(p1.y, p0.y);
  const float bx = fsub(p2.x, p0.x), by = fsub(p2.y, p0.y);
  const float cx = fsub(p2.x, p1.x), cy = fsub(p2.y, p1.y);
  const float a2 = fadd(fmul(ax, ax), fmul(ay, ay));
  const float b2 = fadd(fmul(bx, bx), fmul(by, by));
  const float cr = fsub(fmul(ax, by), fmul(ay, bx));
  const float lc2 = fmul(fabsf(cr), 2.0f);
  const float rc2 =
      fmul(c.kmax, fmul(fmul(fsqrt(a2), fsqrt(b2)), fsqrt(fadd(fmul(cx, cx), fmul(cy, cy)))));
  if (!(lc2 <= rc2)) return false;
  const float D = fmul(cr, 2.0f);
  const float ux = fsub(fmul(by, a2), fmul(ay, b2));
  const float uy = fsub(fmul(ax, b2), fmul(bx, a2));
  const float num = fadd(fmul(fadd(fmul(p0.x, p0.x), fmul(p0.y, p0.y)), D),
                         fmul(fadd(fmul(p0.x, ux), fmul(p0.y, uy)), 2.0f));
  const float px = fadd(fmul(p0.x, D), ux);
  const float py = fadd(fmul(p0.y, D), uy);
  const float den =
      fadd(fsqrt(fadd(fmul(px, px), fmul(py, py))), fsqrt(fadd(fmul(ux, ux), fmul(uy, uy))));
  const float dcamax = first_on_b0 ? c.dca_b0 : c.dca_other;
  const float l3 = fabsf(num);
  if (!(l3 <= fmul(dcamax, den))) return false;
  q = fdiv(l3, den);
  return true;
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// Bounds checks of the debug build (compiled with -DPT_DEBUG, libptca_debug.so): a
// failing check sets the status bit ST_DEBUG and records the first failing site, and the
// access it guards is skipped, so that the kernel reports the fault instead of making
// it.  In the normal build every check is the constant true and costs nothing.
#ifdef PT_DEBUG
__device__ __noinline__ inline void debug_fail(unsigned long long* cnt, unsigned site) {
  atomicOr(&cnt[CNT_STATUS], ST_DEBUG);
  atomicCAS(&cnt[CNT_DEBUG_SITE], 0ull, (unsigned long long)site);
}
#define PT_CHECK(cnt, cond, site) ((cond) ? true : (::ptca::debug_fail((cnt), (site)), false))
#else
#define PT_CHECK(cnt, cond, site) true
#endif

// Learned-gate features of link (h0 -> h1 -> h2) from the hit coordinates (x, y, z, r)
// and layers: C1, C2, C3 cut ratios, t_a/cotmax, 10 (t_b - t_a), r0/16, r1/16, r2/16,
// (z0 - r0 t_a)/z0max, layer0/9, layer1/9, layer2/9.
__device__ __forceinline__ void gate_link_features(const pt_cuts& c, float4 p0, float4 p1,
                                                   float4 p2, int L0, int L1, int L2,
                                                   float (&f)[12]) {
  const float lc1 = fabsf((p1.z - p0.z) * (p2.w - p0.w) - (p2.z - p0.z) * (p1.w - p0.w));
  const float rc1 = c.rz0 * (p2.w - p0.w) + c.rz1 * fabsf(p2.z - p0.z);
  const float ax = p1.x - p0.x, ay = p1.y - p0.y, bx = p2.x - p0.x, by = p2.y - p0.y;
  const float cx = p2.x - p1.x, cy = p2.y - p1.y;
  const float a2 = ax * ax + ay * ay, b2 = bx * bx + by * by;
  const float cr = ax * by - ay * bx;
  const float kap = 2.0f * fabsf(cr) / (sqrtf(a2) * sqrtf(b2) * sqrtf(cx * cx + cy * cy));
  const float D = 2.0f * cr;
  const float ux = by * a2 - ay * b2, uy = ax * b2 - bx * a2;
  const float num = (p0.x * p0.x + p0.y * p0.y) * D + 2.0f * (p0.x * ux + p0.y * uy);
  const float px = p0.x * D + ux, py = p0.y * D + uy;
  const float den = sqrtf(px * px + py * py) + sqrtf(ux * ux + uy * uy);
  const float dmax = L0 == 0 ? c.dca_b0 : c.dca_other;
  const float ta = (p1.z - p0.z) / (p1.w - p0.w);
  const float tb = (p2.z - p1.z) / (p2.w - p1.w);
  f[0] = lc1 / rc1;
  f[1] = kap / c.kmax;
  f[2] = fabsf(num) / den / dmax;
  f[3] = ta / c.cotmax;
  f[4] = 10.0f * (tb - ta);
  f[5] = p0.w * (1.0f / 16.0f);
  f[6] = p1.w * (1.0f / 16.0f);
  f[7] = p2.w * (1.0f / 16.0f);
  f[8] = (p0.z - p0.w * ta) / c.z0max;
  f[9] = L0 * (1.0f / 9.0f);
  f[10] = L1 * (1.0f / 9.0f);
  f[11] = L2 * (1.0f / 9.0f);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(a));
  const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(b));
  return lo | (hi << 16);
}

// The 12 features as one bf16 row of 16 (4 zeros) = 32 bytes.
__device__ __forceinline__ void gate_row(const float (&f)[12], uint4& lo, uint4& hi) {
  lo.x = pack_bf16x2(f[0], f[1]);
  lo.y = pack_bf16x2(f[2], f[3]);
  lo.z = pack_bf16x2(f[4], f[5]);
  lo.w = pack_bf16x2(f[6], f[7]);
  hi.x = pack_bf16x2(f[8], f[9]);
  hi.y = pack_bf16x2(f[10], f[11]);
  hi.z = 0;
  hi.w = 0;
}
__device__ __forceinline__ void store_gate_row(uint16_t* row, const float (&f)[12]) {
  uint4 lo, hi;
  gate_row(f, lo, hi);
  ((uint4*)row)[0] = lo;
  ((uint4*)row)[1] = hi;
}

__device__ __forceinline__ unsigned warp_incl_scan(unsigned v) {
  const int lane = lane_id();
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

constexpr uint32_t kHole = 0xffffffffu;  // marks a reserved but unused slot

// Sorted hits that a warp of the two searches takes next, of `left` not yet taken, with
// `warps` warps.  A search warp handles its hits one after the other, so large chunks leave
// most of the GPU idle on a single event (41k hits in chunks of 32 keep 1281 of 6080 warps
// busy), and uneven hits leave the last warps of a batch running alone; small ones pay the
// chunk's set-up, which is lane-parallel over its hits, more often.  So a chunk is an eighth
// of an even share of what is left, 1 to 32 hits.  The whole call in us, with an eighth (a
// quarter, a sixth, a twelfth; an eighth of at most 16 hits): 64 pileup-200 events 5499 (5645,
// 5545, 5614; 5514), 7 gap-pair events 1125 (1199, 1104, 1171; 1129), one pileup-200 event 327
// (328, 333, 333; 333).  With 32 hits always the two searches of that one event alone took 782.
__device__ __forceinline__ uint32_t search_chunk(uint32_t left, uint32_t warps) {
  return min(32u, max(1u, left / (8u * warps)));
}

// How much a search warp still has to do, as half of the hits after `done` over the hits
// up to it: times what the warp has handed out so far, half of what it may still need.
__device__ __forceinline__ float search_ahead(uint32_t n_sorted, uint32_t done) {
  return done < n_sorted ? __fdividef(0.5f * (float)(n_sorted - done), (float)done) : 0.0f;
}

// Size of the chunk of slots that a warp takes for a request of n, having handed out
// `total`: as much again up to `most`, but no more than it may still need.
__device__ __forceinline__ uint32_t chunk_size(uint32_t n, uint32_t total, float ahead,
                                               uint32_t most) {
  return max(n, min(min(total, most), (uint32_t)fminf((float)total * ahead, (float)most)));
}

// Per-warp bump allocator over a global counter.  A warp that makes one request wastes
// nothing; a busy warp takes a global atomic about once per kChunkMax slots instead of
// once per request.  The unused tail of a chunk becomes a hole.  All members are
// warp-uniform.
struct WarpChunk {
  unsigned long long next = 0, end = 0;
  uint32_t total = 0;  // slots handed out
};
constexpr uint32_t kChunkMax = 2048;

// Reserves n contiguous slots; returns the first.
__device__ __forceinline__ unsigned long long chunk_take(WarpChunk& ch, unsigned long long* counter,
                                                         uint32_t n, float ahead) {
  if (ch.next + n > ch.end) {
    const uint32_t want = chunk_size(n, ch.total, ahead, kChunkMax);
    unsigned long long base = 0;
    if ((threadIdx.x & 31) == 0) base = atomicAdd(counter, (unsigned long long)want);
    base = __shfl_sync(0xffffffffu, base, 0);
    ch.next = base;
    ch.end = base + want;
  }
  const unsigned long long r = ch.next;
  ch.next += n;
  ch.total += n;
  return r;
}

// Whether the batch's S results are written to the arrays in the header.
__device__ __forceinline__ bool results_go_out(const Buffers& b, unsigned long long S) {
  return (int64_t)S <= b.hdr->out_cap && b.cnt[CNT_STATUS] == 0;
}

// Event owning batch hit g: largest e with off[e] <= g (empty events are skipped).
__device__ __forceinline__ int find_event(const int32_t* off, int n_events, int g) {
  int lo = 0, hi = n_events - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

#endif

}  // namespace ptca
