// Host side of the PSA library: argument validation, geometry, per-device workspace,
// TMA descriptors and the extern "C" entry points declared in psa.h.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "psa_common.cuh"

namespace psa {
bool mask_build_small(const Geom& g);
cudaError_t launch_mask_build(const HeadParamsArray& hp, const AxisSet* sets, const int* head_bases, const Geom& g, int n_heads_here,
                              uint8_t* block_mask, int* row_ptr, int* col_idx, int total_nnz_through_chunk,
                              int n_sms, cudaStream_t stream, int* launches);
cudaError_t attn_init(int clusters[3]);
size_t plan_smem_bytes(const Geom& g);
cudaError_t launch_plan(const PlanParams& hp, const Geom& g, int n_heads_here, int* ws_header, psa_head_params* hp_dev,
                        WorkItem* items, cudaStream_t stream);
cudaError_t launch_attn(const TensorMapsCut& tm, const HeadParamsArray& heads, const AttnParamsCut& prm, int n_sms, int cluster,
                        Grid grid, bool direct, bool short_items, bool empty_slabs, cudaStream_t stream, Mode* mode);
size_t search_partial_bytes(int n_cand);
cudaError_t launch_search_losses(const void* outs, const void* ref, long long elems_per_cand, int n_cand, double* partial,
                                 float* losses, cudaStream_t stream, int* launches);
cudaError_t launch_wait_probe(int* ws_header, int call_id, unsigned long long limit_ns, cudaStream_t stream);
}  // namespace psa

namespace {

using namespace psa;

std::atomic<long long> g_launches{0};
std::mutex g_mu;

constexpr int kMaxDevices = 64;
struct Workspace {
  void* base = nullptr;
  size_t bytes = 0;
  int n_sms = 0;
  int cc_major = 0;
  int last_call = 0;             // id of the last API call whose kernels report to the status words
  bool attn_ready = false;
  int clusters[3] = {0, 0, 0};   // clusters of 2, 4 and 8 attention CTAs that run at a time
};
Workspace g_ws[kMaxDevices];

// The last attention launch of any entry point (g_mu held).
struct {
  Mode mode = kTicket;
  int items = 0, cluster = 1;
  Grid grid = kWhole;
  int slabs = 0, last_keys = 0, edge_axes = 0;
  uint8_t query_slabs[8] = {}, together[8] = {};
  uint16_t keys[8] = {};   // of every `together` attended blocks
} g_last_attn;

// Id of a new API call on `stream` (g_mu held).  Never 0, which is what untouched status words hold.  A call that is
// being captured has kCapturedCall set: its kernels run again whenever the graph is replayed.
constexpr int kCapturedCall = 1 << 30;
int g_calls = 0;
int next_call_id(cudaStream_t stream) {
  g_calls = g_calls + 1 == kCapturedCall ? 1 : g_calls + 1;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(stream, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive ? g_calls | kCapturedCall : g_calls;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
cudaEvent_t g_ev_start = nullptr, g_ev_stop = nullptr;

int load_driver_entry() {
  if (g_encode) return PSA_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || fn == nullptr) {
    return PSA_ERR_CUDA;
  }
  g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  return PSA_OK;
}

// What call `call_id`, or a replay of a captured call, reported in the status words at `header` (its work has finished);
// what a replay reported is cleared.
int read_status(void* header, int call_id, int32_t* detail) {
  int hdr[4] = {0, 0, 0, 0};
  if (cudaMemcpy(hdr, header, sizeof(hdr), cudaMemcpyDeviceToHost) != cudaSuccess) return PSA_ERR_CUDA;
  const int from = hdr[kWsCallId];
  const bool mine = from != 0 && (from == call_id || (from & kCapturedCall));
  if (detail) *detail = mine ? hdr[kWsDetail] : 0;
  if (!mine) return PSA_OK;
  const int zero = 0;
  if ((from & kCapturedCall) && cudaMemcpy(static_cast<int*>(header) + kWsCallId, &zero, sizeof(zero), cudaMemcpyHostToDevice) != cudaSuccess)
    return PSA_ERR_CUDA;
  return hdr[kWsStatus];
}

bool valid_params(const psa_head_params& p) {
  const int lim = 1 << 30;
  return p.Tw >= 1 && p.Sw >= 1 && p.Ts >= 0 && p.Ss >= 0 && p.To > -lim && p.To < lim && p.So > -lim && p.So < lim;
}

// Chunks of a host-tensor call: 20 from a measured sweep at the 75,600-token, 40-head shape
// (4: 54.3 ms, 8: 50.3, 10: 48.9, 20: 47.6, 40: 49.7); PSA_HOST_CHUNKS overrides it for measurements.
int host_chunks() {
  static int v = 0;
  if (v == 0) {
    const char* e = std::getenv("PSA_HOST_CHUNKS");
    const int n = e ? std::atoi(e) : 0;
    v = n >= 1 ? n : 20;
  }
  return v;
}

// Geometry with what only grids with edge blocks need: their classes, and the box shapes of maps 3 on.
struct BoxShape {
  int w, h, t;
};
struct HostGeom : Geom {
  EdgeClass cls[8];
  Grid grid;
  int planned, n_classes;
  bool empty_slabs;   // some blocks have, uncut, slabs without any token
  uint8_t order[8];
  int n_shapes;
  BoxShape shape[kMaxMaps - 3];
};

// Blocks of the grid of class c.
int class_blocks(const Geom& g, int c) {
  if (c & ~g.edge_axes) return 0;
  auto along = [&](int n, int bit) -> int { return c & bit ? 1 : (g.edge_axes & bit ? n - 1 : n); };
  return along(g.Tp, 1) * along(g.Hp, 2) * along(g.Wp, 4);
}

int round_up(int n, int to) { return (n + to - 1) / to * to; }
int log2_up(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// Map of a box shape, or -1 if there are too many.
int map_of(HostGeom* g, int w, int h, int t) {
  if (w == g->cw && h == g->ch && t == g->ct) return 0;
  for (int i = 0; i < g->n_shapes; ++i)
    if (g->shape[i].w == w && g->shape[i].h == h && g->shape[i].t == t) return 3 + i;
  if (g->n_shapes == kMaxMaps - 3) return -1;
  g->shape[g->n_shapes] = BoxShape{w, h, t};
  return 3 + g->n_shapes++;
}

bool add_box(EdgeClass* e, int* rows, int map, int t, int h, int w, int n) {
  if (map < 0 || e->n_boxes == kMaxEdgeBoxes) return false;
  e->box[e->n_boxes++] = EdgeBox{(uint8_t)map, (uint8_t)(*rows / 8), (uint16_t)t, (uint16_t)h, (uint16_t)w};
  *rows += n;
  return true;
}

// Zeros up to `to` rows behind the `rows` that the class's boxes fill of its last slab so far: lines behind the grid's last one in the
// same box, where the slab ends with them, or a box of their own from beyond the last frame.
bool fill_slab(HostGeom* g, EdgeClass* e, bool at_bottom, int rows, int to) {
  if (rows >= to) return true;
  const EdgeBox last = e->box[e->n_boxes - 1];
  const int w = 1 << e->lw, need = to - rows;
  const BoxShape s = last.map >= 3 ? g->shape[last.map - 3] : BoxShape{g->cw, g->ch, g->ct};
  if (at_bottom && e->together == 1 && last.map != 1 && s.t == 1 && s.w == w && (last.h + s.h) * w == e->frame && need % w == 0) {
    int users = 0;   // of the box's map in finished classes: if it is this box alone, the map changes with it
    for (const EdgeClass& x : g->cls)
      for (int b = 0; b < x.n_boxes; ++b) users += x.box[b].map == last.map;
    if (users == 1 && last.map >= 3 && e >= g->cls && e < g->cls + 8) {
      g->shape[last.map - 3].h += need / w;
      return true;
    }
    const int map = map_of(g, w, s.h + need / w, 1);
    if (map < 0) return false;
    e->box[e->n_boxes - 1].map = (uint8_t)map;
    return true;
  }
  return add_box(e, &rows, map_of(g, 8, need / 8, 1), kZeros, 0, 0, need);
}

// A block of nt x nh x nw tokens as an ordinary one, without the slabs that have no token.
void whole_slabs(const HostGeom& g, EdgeClass* e, int nt, int nh, int nw) {
  const int tokens = g.sub_axis == 0 ? nt : (g.sub_axis == 1 ? nh : nw), slab = g.sub_axis == 0 ? g.ct : (g.sub_axis == 1 ? g.ch : g.cw),
            block = g.sub_axis == 0 ? g.bt : (g.sub_axis == 1 ? g.bh : g.bw), along = round_up(tokens, slab) < block ? round_up(tokens, slab) : block;
  std::memset(e, 0, sizeof(*e));
  const int t = g.sub_axis == 0 ? along : g.bt, h = g.sub_axis == 1 ? along : g.bh, w = g.sub_axis == 2 ? along : g.bw;
  e->rows = (uint16_t)(t * h * w);
  e->frame = (uint16_t)(h * w);
  e->lw = (uint8_t)log2_up(w);
  e->step = kSlabTokens;
  e->together = 1;
  for (int at = 0; at < along; at += slab) {
    int rows = 0;
    e->first_box[e->n_slabs++] = e->n_boxes;
    add_box(e, &rows, along - at < slab ? 1 : 0, g.sub_axis == 0 ? at : 0, g.sub_axis == 1 ? at : 0, g.sub_axis == 2 ? at : 0, 0);
  }
}

// Keys that a slab of so many rows is multiplied as, at the end of a block: the widths of the softmax.
int key_width(int rows) { return rows <= 64 ? 64 : (rows <= 96 ? 96 : (rows <= 112 ? 112 : 128)); }
int last_rows(const EdgeClass& e) { return e.rows - (e.n_slabs - 1) * e.step; }

// The same cut to its tokens, if that can be done and makes fewer slabs of keys (or a narrower last one that makes or follows the
// pattern).  Lines have
// a power of two of tokens, and a frame is a multiple of 8 rows (the unit of the 128-byte swizzle, so that boxes can be put
// behind one another).  What that adds lies beyond the grid, where it is loaded as zeros -- never in the next block, whose values a
// probability of 0 would not keep out if they are infinite -- so lines shorter than 8 tokens need a whole number of groups of
// 8 rows in every block's height.
bool cut_to_tokens(HostGeom* g, EdgeClass* e, int c, bool for_pattern, int nt, int nh, int nw) {
  const int shapes_before = g->n_shapes;
  EdgeClass x = {};
  auto lines = [](int width) -> int { return width < 8 ? 8 / width : 1; };   // that make whole groups of 8 rows
  int w = g->bw;
  if (c & 4) {
    w = 1 << log2_up(nw);
    while (w < g->bw && !(c & 2) && g->bh % lines(w) != 0) w *= 2;
  }
  const int h = c & 2 ? round_up(nh, lines(w)) : nh, frame = h * w, rows = nt * frame;
  // slabs of whole frames, or of lines with up to four boxes a slab where that makes fewer of them (or a narrower last one)
  auto slabs = [&](int step) -> int { return (rows + step - 1) / step; };
  auto last_of = [&](int step) -> int { return rows - (slabs(step) - 1) * step; };
  auto cost = [&](int step) -> int { return 128 * slabs(step) + (for_pattern || g->main_last < kSlabTokens ? key_width(last_of(step)) : 0); };
  const int per = kSlabTokens / frame, step = rows <= kSlabTokens ? rows : (per > 0 && cost(per * frame) <= cost(kSlabTokens) ? per * frame : kSlabTokens);
  x.rows = (uint16_t)rows;
  x.frame = (uint16_t)frame;
  x.lw = (uint8_t)log2_up(w);
  x.step = (uint16_t)step;
  x.together = (uint8_t)(rows <= kSlabTokens / 2 ? kSlabTokens / rows : 1);
  bool ok = slabs(step) < e->n_slabs || x.together > 1 ||
            (slabs(step) == e->n_slabs && key_width(last_of(step)) < key_width(last_rows(*e)) &&
             (for_pattern || (e->n_slabs == g->main_slabs && last_rows(*e) > g->main_last && last_of(step) <= g->main_last)));
  for (int r = 0; ok && r < rows; r += step) {
    int end = 0;
    x.first_box[x.n_slabs++] = x.n_boxes;
    for (int y = r, to = r + step < rows ? r + step : rows; ok && y < to;) {
      const int left = to - y, in_frame = y % frame;
      if (in_frame == 0 && left >= frame) {   // whole frames
        const int n = left / frame;
        ok = add_box(&x, &end, map_of(g, w, h, n), y / frame, 0, 0, n * frame);
        y += n * frame;
      } else {
        const int n = left < frame - in_frame ? left : frame - in_frame;
        ok = add_box(&x, &end, map_of(g, w, n / w, 1), y / frame, in_frame / w, 0, n);
        y += n;
      }
    }
    if (r + step < rows) ok = ok && fill_slab(g, &x, (c & 2) || g->Hp == 1, end, kSlabTokens);
  }
  int classes = 0;   // set_edges has a map and a box left for each of them
  for (int k = 1; k < 8; ++k) classes += class_blocks(*g, k) > 0;
  if (!ok || g->n_shapes + classes > kMaxMaps - 3 || x.n_boxes == kMaxEdgeBoxes) {
    g->n_shapes = shapes_before;
    return false;
  }
  *e = x;
  return true;
}

// EdgeClass::valid of a class whose blocks hold nt x nh x nw tokens, by lines (a slab holds whole ones); `to`: keys of the last slab,
// beyond which there are none to mask.
void set_valid(EdgeClass* e, int nt, int nh, int nw, int to) {
  using u128 = unsigned __int128;
  auto low = [](int n) -> u128 { return n >= 128 ? ~(u128)0 : ((u128)1 << n) - 1; };
  const u128 line = low(nw);
  const int w = 1 << e->lw, lines = e->frame >> e->lw;   // of a frame
  int t = 0, h = 0;
  for (int s = 0; s < e->n_slabs; ++s) {
    const bool last = s + 1 == e->n_slabs;
    const int have = last ? last_rows(*e) : e->step;
    u128 one = 0, all = last ? ~low(to) : 0;
    for (int r = 0; r < have; r += w) {
      if (t < nt && h < nh) one |= line << r;
      if (++h == lines) { h = 0; ++t; }
    }
    for (int b = 0; b < e->together; ++b) all |= one << b * have;
    for (int i = 0; i < 4; ++i) e->valid[s][i] = (uint32_t)(all >> 32 * i);
  }
}

// Work items of a head.
void count_items(HostGeom* g) {
  g->items_per_block = (g->n_sub + 1) / 2;
  g->items_per_head = g->NB * g->items_per_block + g->n_titems;
  if (g->n_sub == 3)   // (only blocks of three slabs have a second item)
    for (int c = 0; c < 8; ++c)
      if (g->slabs_of[c] < 3) g->items_per_head -= class_blocks(*g, c);
}

// Makes a padded grid a cut one (EdgeClass); false, if no class is cut, and then *g is of no use.
//
// Why: 3D-padding is issued work, along the keys and along the queries.  The last of the seven 30x8 blocks across 52 columns
// holds 120 of its 240 tokens (12 heads of 21x30x52: 2.60 -> 2.39 ms), the last 3x8x16 block down 45 rows 240 of 384 (40 heads of
// 21x45x80: 28.7 -> 26.3 ms).  Cut like this an edge block is mostly one box a slab, as an ordinary one: the load warp, which has
// some 10 clocks for an instruction next to the softmax, fell behind with rows packed tightly across blocks, by boxes of 8 to
// 128 rows (5,000 clocks a slab) as well as by 16-byte copies (8,000).
bool cut_edges(HostGeom* g) {
  const int rt = g->T - (g->Tp - 1) * g->bt, rh = g->H - (g->Hp - 1) * g->bh, rw = g->W - (g->Wp - 1) * g->bw;   // of the last block
  const int axes = (rt < g->bt ? 1 : 0) | (rh < g->bh ? 2 : 0) | (rw < g->bw ? 4 : 0);
  if (g->sub_axis == 2 || g->bh * g->bw < 8) return false;
  if ((axes & 6) == 6 && g->Sp > kMaxSp / 2) return false;   // (the kernel keeps four sets of spatial coordinates of such a grid)
  // Blocks of one slab run in split-KV mode, where a slab takes 1,900 clocks and the load warp has no time for lists of boxes: 7
  // heads of 7x19x25 with 2x8x8 blocks 93 us padded and 135 cut, 18 of 3x25x73 with 1x8x16 165 and 177.
  if (g->n_sub == 1) return false;
  std::memset(g->cls, 0, sizeof(g->cls));
  g->edge_axes = axes;
  g->n_shapes = g->n_classes = 0;
  int pattern = 0;   // its class
  for (int c = 0; c < 8; ++c)
    if (class_blocks(*g, 0) == 0 && class_blocks(*g, c) > class_blocks(*g, pattern)) pattern = c;
  bool cut = false;
  auto make = [&](int c) {
    const int nt = c & 1 ? rt : g->bt, nh = c & 2 ? rh : g->bh, nw = c & 4 ? rw : g->bw;   // tokens along the axes
    whole_slabs(*g, &g->cls[c], nt, nh, nw);
    if (c != 0 && cut_to_tokens(g, &g->cls[c], c, c == pattern, nt, nh, nw)) cut = true;
  };
  make(pattern);
  const EdgeClass& m = g->cls[pattern];
  g->main_slabs = m.together > 1 ? 1 : m.n_slabs;
  g->main_last = m.together > 1 ? kSlabTokens : key_width(last_rows(m));
  for (int c = 0; c < 8; ++c)
    if (c != pattern && class_blocks(*g, c)) make(c);
  if (!cut) return false;
  g->planned = 1;
  for (int c = 0; c < 8; ++c) {
    if (!class_blocks(*g, c)) continue;
    EdgeClass& e = g->cls[c];
    e.in_pattern = e.together == 1 && e.n_slabs == g->main_slabs && last_rows(e) <= g->main_last;
    g->planned &= e.in_pattern;
    const int to = e.in_pattern ? g->main_last : kSlabTokens;
    fill_slab(g, &e, (c & 2) || g->Hp == 1, e.together * last_rows(e), to);   // (see cut_to_tokens)
    set_valid(&e, c & 1 ? rt : g->bt, c & 2 ? rh : g->bh, c & 4 ? rw : g->bw, to);
    e.first_box[e.n_slabs] = e.n_boxes;
    g->slabs_of[c] = e.n_slabs;
  }
  for (int in = 1; in >= 0; --in)
    for (int c = 0; c < 8; ++c)
      if (class_blocks(*g, c) && g->cls[c].in_pattern == in) g->order[g->n_classes++] = (uint8_t)c;
  g->grid = kCut;
  count_items(g);
  return true;
}

// Classes of a padded grid, which has no boxes: blocks with fewer slabs than the others, the last ones along the axis on which slabs
// stack, are the only ones told apart.  Where there are none the grid has one class and its items are what the planning kernel
// counted.  (With a class for every combination of ragged axes, as in a cut grid, 3 heads of 6x15x23 with 2x8x8 blocks took 26.3 us
// and take 21.0, 2 of 13x13x14 34.2 and 26.3: their tables, two dozen constants, and the tests in the loop over the key blocks.)
void pad_edges(HostGeom* g, int edge_slabs) {
  const int blocks = g->sub_axis == 0 ? g->Tp : (g->sub_axis == 1 ? g->Hp : g->Wp);
  const bool two = edge_slabs < g->n_sub && blocks > 1;
  g->edge_axes = two ? 1 << g->sub_axis : 0;
  g->n_shapes = 0;
  g->main_slabs = two ? g->n_sub : edge_slabs;
  g->main_last = g->main_slabs == g->n_sub ? g->n_last : kSlabTokens;
  g->slabs_of[0] = (uint8_t)g->main_slabs;
  if (two) g->slabs_of[g->edge_axes] = (uint8_t)edge_slabs;
}

// Whether the grid is whole or padded, and its edge blocks.  T, H, W, the block and its slabs are set.
void set_edges(HostGeom* g) {
  const int rt = g->T - (g->Tp - 1) * g->bt, rh = g->H - (g->Hp - 1) * g->bh, rw = g->W - (g->Wp - 1) * g->bw;   // of the last block
  const int along = g->sub_axis == 0 ? rt : (g->sub_axis == 1 ? rh : rw), slab = g->sub_axis == 0 ? g->ct : (g->sub_axis == 1 ? g->ch : g->cw);
  const int edge_slabs = (along + slab - 1) / slab;   // of the last block along the axis on which slabs stack, with any token
  g->empty_slabs = edge_slabs < g->n_sub;
  g->s_edge = g->Sp - g->Wp;
  g->grid = rt == g->bt && rh == g->bh && rw == g->bw ? kWhole : kPadded;
  pad_edges(g, edge_slabs);   // (a whole grid has one class of blocks)
}

// Geometry of the block grid; `for_attn` additionally derives the 128-token slab.
int make_geom(const psa_problem* prob, int T, int H, int W, bool for_attn, HostGeom* g) {
  if (!prob || T < 1 || H < 1 || W < 1 || prob->n_heads < 1) return PSA_ERR_INVALID_ARG;
  const psa_tile t = prob->tile;
  if (t.bt < 1 || t.bh < 1 || t.bw < 1) return PSA_ERR_INVALID_ARG;
  const long long L = (long long)T * H * W;
  if (L >= (1ll << 31)) return PSA_ERR_INVALID_ARG;
  std::memset(static_cast<Geom*>(g), 0, sizeof(Geom));
  g->T = T; g->H = H; g->W = W;
  g->bt = t.bt; g->bh = t.bh; g->bw = t.bw;
  g->Tp = (T + t.bt - 1) / t.bt;
  g->Hp = (H + t.bh - 1) / t.bh;
  g->Wp = (W + t.bw - 1) / t.bw;
  g->Sp = g->Hp * g->Wp;
  const long long nb = (long long)g->Tp * g->Sp;
  if (nb > (1 << 20)) return PSA_ERR_UNSUPPORTED;
  g->NB = (int)nb;
  g->n_heads = prob->n_heads;
  g->L = L;
  g->ct = t.bt; g->ch = t.bh; g->cw = t.bw;
  g->n_sub = 1;
  g->sub_axis = 0;
  g->items_per_block = 1;
  if (for_attn) {
    g->c_last = 1;
    g->n_last = kSlabTokens;
    if (prob->head_dim != kHeadDim) return PSA_ERR_UNSUPPORTED;
    if (!(prob->scale > 0.f) || !std::isfinite(prob->scale)) return PSA_ERR_INVALID_ARG;
    // Split the block into slabs along its outermost axis of extent > 1: full slabs of 128
    // tokens, and a last slab that may be shorter (112, 96 or 64 tokens) so that blocks such
    // as 1x15x16 tile a 45-row grid without padding.
    const long long tokens = (long long)t.bt * t.bh * t.bw;
    if (tokens < 128 || tokens > 384) return PSA_ERR_UNSUPPORTED;
    int axis, extent;
    long long other;
    if (t.bt > 1 || (t.bh == 1 && t.bw == 1)) { axis = 0; extent = t.bt; other = (long long)t.bh * t.bw; }
    else if (t.bh > 1) { axis = 1; extent = t.bh; other = (long long)t.bt * t.bw; }
    else { axis = 2; extent = t.bw; other = (long long)t.bt * t.bh; }
    if (other > kSlabTokens || (kSlabTokens % other) != 0) return PSA_ERR_UNSUPPORTED;
    const int c0 = (int)(kSlabTokens / other);
    const int n_sub = (extent + c0 - 1) / c0;
    const int c_last = extent - (n_sub - 1) * c0;
    const int n_last = (int)(c_last * other);
    if (n_sub > 3 || !(n_last == 128 || n_last == 112 || n_last == 96 || n_last == 64)) return PSA_ERR_UNSUPPORTED;
    if (axis == 0) g->ct = c0; else if (axis == 1) g->ch = c0; else g->cw = c0;
    g->sub_axis = axis;
    g->c_last = c_last;
    g->n_last = n_last;
    if (g->ct > 128 || g->ch > 128 || g->cw > 128) return PSA_ERR_UNSUPPORTED;
    // (the extents of a full slab are powers of two: they multiply to 128; a block's last slab is only shorter along its
    // slowest axis, so positions in it are the same)
    while ((1 << g->pos_ws) < g->cw) ++g->pos_ws;
    g->pos_ts = g->pos_ws;
    while ((1 << g->pos_ts) < g->cw * g->ch) ++g->pos_ts;
    if (g->Tp > kMaxTp || g->Sp > kMaxSp || plan_smem_bytes(*g) > kMaxSmemBytes) return PSA_ERR_UNSUPPORTED;
    g->n_sub = n_sub;
    set_edges(g);
    g->scale_log2 = prob->scale * 1.4426950408889634f;
  }
  count_items(g);
  g->Lt = L;
  return PSA_OK;
}

// Adds n_text text tokens per head to an attention geometry.
int set_text(Geom* g, long long n_text) {
  if (n_text < 0 || g->L + n_text >= (1ll << 31)) return PSA_ERR_INVALID_ARG;
  g->n_text = (int)n_text;
  g->n_ts = (int)((n_text + kSlabTokens - 1) / kSlabTokens);
  if (g->n_ts > 0xffff) return PSA_ERR_UNSUPPORTED;
  g->n_titems = (g->n_ts + 1) / 2;
  g->items_per_head += g->n_titems;
  g->Lt = g->L + n_text;
  return PSA_OK;
}

// Attended block pairs of one head: product of the two axis pair counts.
long long head_nnz(const psa_head_params& p, const Geom& g) {
  auto pairs = [](int n, int w, int o, int s) -> long long {
    if (n <= 64) return axis_set(n, w, o, s).pairs;
    long long c = 0;
    for_attended(n, w, o, s, [&](int, int d) { c += n - (d < 0 ? -d : d); });
    return c;
  };
  return pairs(g.Tp, p.Tw, p.To, p.Ts) * pairs(g.Sp, p.Sw, p.So, p.Ss);
}

int device_info(int* dev, Workspace** ws) {
  if (cudaGetDevice(dev) != cudaSuccess) return PSA_ERR_CUDA;
  if (*dev < 0 || *dev >= kMaxDevices) return PSA_ERR_UNSUPPORTED;
  Workspace& w = g_ws[*dev];
  if (w.n_sms == 0) {
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, *dev) != cudaSuccess) return PSA_ERR_CUDA;
    w.n_sms = prop.multiProcessorCount;
    w.cc_major = prop.major;
  }
  *ws = &w;
  return PSA_OK;
}

// First attention call on a device: driver entry point, kernel attributes.
int init_attn(Workspace* w) {
  if (w->attn_ready) return PSA_OK;
  if (w->cc_major != 10) return PSA_ERR_UNSUPPORTED;
  const int rc = load_driver_entry();
  if (rc != PSA_OK) return rc;
  if (attn_init(w->clusters) != cudaSuccess) return PSA_ERR_CUDA;
  w->attn_ready = true;
  return PSA_OK;
}

int ensure_workspace(Workspace* w, size_t bytes) {
  if (w->bytes >= bytes) return PSA_OK;
  if (w->base) {
    if (cudaDeviceSynchronize() != cudaSuccess) return PSA_ERR_CUDA;
    cudaFree(w->base);
    w->base = nullptr;
    w->bytes = 0;
  }
  const size_t want = bytes + bytes / 4 + 4096;
  if (cudaMalloc(&w->base, want) != cudaSuccess) return PSA_ERR_CUDA;
  if (cudaMemset(w->base, 0, want) != cudaSuccess) return PSA_ERR_CUDA;
  w->bytes = want;
  return PSA_OK;
}

// Map of [heads][T][H][W][128] with a box of 64 columns of box.w x box.h x box.t tokens.
int encode_map(CUtensorMap* tm, const void* base, const Geom& g, long long stride_head, long long stride_token,
               int n_heads_here, const BoxShape& shape) {
  const cuuint64_t dims[5] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.T,
                              (cuuint64_t)n_heads_here};
  const cuuint64_t st = (cuuint64_t)stride_token * 2;
  const cuuint64_t strides[4] = {st, st * g.W, st * g.W * g.H,
                                 n_heads_here > 1 ? (cuuint64_t)stride_head * 2 : st * g.W * g.H * g.T};
  const cuuint32_t box[5] = {64, (cuuint32_t)shape.w, (cuuint32_t)shape.h, (cuuint32_t)shape.t, 1};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? PSA_OK : PSA_ERR_INVALID_ARG;
}

// Map of the text tokens of every head: a [heads][n_text][128] view starting L tokens into each head,
// box = 128 tokens x 64 columns (same shared-memory image as a full video slab).
int encode_text_map(CUtensorMap* tm, const void* base, const Geom& g, long long stride_head, long long stride_token,
                    int n_heads_here) {
  const cuuint64_t st = (cuuint64_t)stride_token * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.n_text, 1, 1, (cuuint64_t)n_heads_here};
  const cuuint64_t strides[4] = {st, st * g.n_text, st * g.n_text,
                                 n_heads_here > 1 ? (cuuint64_t)stride_head * 2 : st * g.n_text};
  const cuuint32_t box[5] = {64, (cuuint32_t)kSlabTokens, 1, 1, 1};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const void* text0 = static_cast<const uint16_t*>(base) + g.L * stride_token;
  const CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(text0), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? PSA_OK : PSA_ERR_INVALID_ARG;
}

// Strides (in elements) of the inputs and of the output of one attention launch.
struct Layout {
  long long in_head, in_token;    // q, k, v
  long long out_head, out_token;  // out
  bool shared_qkv;                // every head reads head 0 of q, k, v
};

// The four tensors with every box shape (TensorMaps).
int encode_maps(TensorMapsCut* tm, const void* q, const void* k, const void* v, void* out, const HostGeom& g,
                const Layout& lay, int n_heads_here) {
  int rc;
  const int n_in = lay.shared_qkv ? 1 : n_heads_here;
  auto encode = [&](int i, const BoxShape& box) -> int {
    if ((rc = encode_map(&tm->q[i], q, g, lay.in_head, lay.in_token, n_in, box)) != PSA_OK) return rc;
    if ((rc = encode_map(&tm->k[i], k, g, lay.in_head, lay.in_token, n_in, box)) != PSA_OK) return rc;
    if ((rc = encode_map(&tm->v[i], v, g, lay.in_head, lay.in_token, n_in, box)) != PSA_OK) return rc;
    return encode_map(&tm->o[i], out, g, lay.out_head, lay.out_token, n_heads_here, box);
  };
  if ((rc = encode(0, BoxShape{g.cw, g.ch, g.ct})) != PSA_OK) return rc;
  if (g.n_last == kSlabTokens) {   // a block's last slab is a full one
    tm->q[1] = tm->q[0]; tm->k[1] = tm->k[0]; tm->v[1] = tm->v[0]; tm->o[1] = tm->o[0];
  } else if ((rc = encode(1, BoxShape{g.sub_axis == 2 ? g.c_last : g.cw, g.sub_axis == 1 ? g.c_last : g.ch, g.sub_axis == 0 ? g.c_last : g.ct})) != PSA_OK) {
    return rc;
  }
  for (int i = 0; i < g.n_shapes; ++i)
    if ((rc = encode(3 + i, g.shape[i])) != PSA_OK) return rc;
  if (g.n_text > 0) {
    if ((rc = encode_text_map(&tm->q[2], q, g, lay.in_head, lay.in_token, n_in)) != PSA_OK) return rc;
    if ((rc = encode_text_map(&tm->k[2], k, g, lay.in_head, lay.in_token, n_in)) != PSA_OK) return rc;
    if ((rc = encode_text_map(&tm->v[2], v, g, lay.in_head, lay.in_token, n_in)) != PSA_OK) return rc;
    if ((rc = encode_text_map(&tm->o[2], out, g, lay.out_head, lay.out_token, n_heads_here)) != PSA_OK) return rc;
  } else {  // never used; keep the descriptors valid
    tm->q[2] = tm->q[0]; tm->k[2] = tm->k[0]; tm->v[2] = tm->v[0]; tm->o[2] = tm->o[0];
  }
  return PSA_OK;
}

// Attended block pairs of every head.
void head_weights(const psa_head_params* params, int n, const Geom& g, long long* w) {
  for (int h = 0; h < n; ++h) {
    // (the samples of a batch or the heads of a group often repeat the parameters of the head before)
    w[h] = h > 0 && std::memcmp(&params[h], &params[h - 1], sizeof(psa_head_params)) == 0 ? w[h - 1] : head_nnz(params[h], g);
  }
}

// Planning arguments of one launch: the heads' parameters and their places in the work order, heavier heads first.
void plan_params(PlanParams* pp, const psa_head_params* params, const long long* w, int n) {
  for (int h = 0; h < n; ++h) {
    pp->p[h] = params[h];
    int place = 0;
    for (int j = 0; j < n; ++j) place += w[j] > w[h] || (w[j] == w[h] && j < h);
    pp->place[h] = (uint8_t)place;
  }
}

// Key slabs of the average block.
double slabs_per_block(const HostGeom& g) {
  double n = 0;
  for (int c = 0; c < 8; ++c)
    if (class_blocks(g, c)) n += (double)class_blocks(g, c) * g.slabs_of[c] / (g.grid == kCut ? g.cls[c].together : 1);
  return n / g.NB;
}

// What share_items needs to know of a cut grid, in clocks.  A slab takes the load warp 1,200 for each of its boxes (of K and of V),
// which is more than it takes the others where it has more than one or two; an item, 1,750 for each class of blocks, and a quarter of a
// slab for blocks that share one, as there are not always enough of them.  (Least squares over 230 drawn problems of 8 to 6,000
// items, cut and padded.)
void cut_clocks(const HostGeom& g, double per_slab, double* block, double* rest, double* setup) {
  *block = *rest = 0;
  *setup = 1750.0 * g.n_classes;
  auto width = [](int keys) -> double { return 0.5 + 0.5 * keys / kSlabTokens; };   // a narrower slab's time
  for (int i = 0; i < g.n_classes; ++i) {
    const EdgeClass& e = g.cls[g.order[i]];
    const double boxes = e.together > 1 ? e.together + e.n_boxes - 1 : (double)e.n_boxes / e.n_slabs;
    auto slab = [&](double clocks) -> double { return 1200.0 * boxes > clocks ? 1200.0 * boxes : clocks; };
    const double last = e.in_pattern ? per_slab * width(g.main_last) / width(g.main_slabs == g.n_sub ? g.n_last : kSlabTokens) : per_slab;
    *block += (slab(per_slab) * (e.n_slabs - 1) + slab(last)) * class_blocks(g, g.order[i]) / e.together / g.NB;
    if (e.together > 1) *rest += 0.25 * slab(per_slab);
  }
}

// CTAs that share a work item: 1 (persistent CTAs that draw whole items), 2, 4 or 8.  A launch takes about as many
// rounds as its items need on the SMs, and at least as long as its longest item, so a problem of few items, of a few more
// than a whole number of rounds, or of a few very long ones (text queries attend every key) leaves SMs idle; sharing
// items makes the rounds shorter.  Clocks, from time stamps in the kernel: a key slab takes 3,300 for two query slabs and
// 1,900 for one (split-KV mode); start-up, epilogue and exit take 15,000 in a persistent CTA and 20,000 in a cluster
// (which also merges).  Over 56 drawn problems of 12 to 700 items the choice was within 9 % of the best of the four,
// except one at 18 % (12 items); without text, whole items were best in all 24 problems of more than two rounds.
// weights: attended block pairs of every head.
struct Sharing {
  int cluster;
  double clocks;   // the launch's estimated time with them
};
Sharing share_items(const Workspace& ws, const HostGeom& g, const long long* weights, int n_heads) {
  const int heads = n_heads < kMaxHeads ? n_heads : kMaxHeads;   // of one launch
  const int n_items = heads * g.items_per_head, n_text = heads * g.n_titems;
  long long total = 0, most = 0;
  for (int h = 0; h < n_heads; ++h) {
    total += weights[h];
    if (weights[h] > most) most = weights[h];
  }
  // blocks attended by the average query block, of all heads and of the heaviest
  const double avg = (double)total / ((double)n_heads * g.NB), heavy = (double)most / g.NB;
  const int of_block = g.main_slabs, singles = of_block & 1, doubles = of_block >> 1;
  const double per_slab = (3300.0 * doubles + 1900.0 * singles) / (doubles + singles), slabs = slabs_per_block(g);
  const double text = n_text ? (g.NB * slabs + g.n_ts) * (g.n_ts > 1 ? 3300.0 : 1900.0) : 0.0;
  // (a block: clocks of an attended one; rest: clocks of an item besides)
  auto time = [&](int at_a_time, int c, double fixed, double block, double rest) -> double {
    const double item = avg * block + rest + g.n_ts * per_slab, heavy_item = heavy * block + rest + g.n_ts * per_slab;
    const double one = (heavy_item > text ? heavy_item : text) / c + fixed;
    if (n_items <= at_a_time) return one;
    const double all = (double)((n_items + at_a_time - 1) / at_a_time) * (((n_items - n_text) * item + n_text * text) / n_items / c + fixed);
    return all > one ? all : one;
  };
  const double block = slabs * per_slab, heavy_item = heavy * block + g.n_ts * per_slab, longest = heavy_item > text ? heavy_item : text;
  int cluster = 1, at_a_time = ws.n_sms;
  double best = time(at_a_time, 1, 15000.0, block, 0);
  // beyond two rounds at most a third is to be gained, unless text queries make long items
  for (int i = 0; i < 3 && n_items <= (n_text ? 8 : 2) * ws.n_sms; ++i) {
    const int c = 2 << i;
    if (ws.clusters[i] < 1 || longest < c * block) break;   // a share of a long item holds at least one block
    const double t = time(ws.clusters[i], c, 20000.0, block, 0);
    // (rounds of whole items overlap more than the estimate knows: the longer ones go first)
    if (t < (n_items <= ws.clusters[i] ? 0.97 : 0.88) * best) { best = t; cluster = c; at_a_time = ws.clusters[i]; }
  }
  if (g.grid == kCut) {
    double cut_block, rest, setup;
    cut_clocks(g, per_slab, &cut_block, &rest, &setup);
    best = time(at_a_time, cluster, (cluster > 1 ? 20000.0 : 15000.0) + setup, cut_block, rest);
  }
  return Sharing{cluster, cluster > 1 && n_items > at_a_time ? best / 0.88 : best};   // (as above)
}

// Cuts a padded grid if the launch is estimated to take less time then; the CTAs that share an item.  Decided for a call as a whole,
// so that the chunks of a host-tensor call compute what the device call computes, bit for bit.
//
// What a cut grid saves is in proportion to the launch's slabs, what it costs is not: over 230 drawn problems of 8 to 6,000 items
// that can be cut it was from 0.47 to 3.0 times as fast as padded.  By this rule 168 of them are cut, 15 of these lose more than 2 %
// by it (0.79 times as fast the worst, 51 us) and 8 of the others would have gained more (15 % at most).  Below an estimate of 30,000
// clocks (about 20 us) none gains, and the call would wait for the host's tables.
int choose_edges(const Workspace& ws, HostGeom* g, const long long* weights, int n_heads) {
  const Sharing padded = share_items(ws, *g, weights, n_heads);
  if (g->grid != kPadded || padded.clocks < 30000.0) return padded.cluster;
  HostGeom cut = *g;
  if (!cut_edges(&cut)) return padded.cluster;
  const Sharing s = share_items(ws, cut, weights, n_heads);
  if (s.clocks >= padded.clocks) return padded.cluster;
  *g = cut;
  return s.cluster;
}

// Whether every item of a launch runs at the same time.  Then their order does not matter and no planning is needed:
// one kernel instead of two (a 2,048-token call is bound by such latencies).
bool runs_at_once(const Workspace& ws, int n_items, int cluster) {
  const int at_once = cluster == 1 ? ws.n_sms : ws.clusters[cluster == 2 ? 0 : (cluster == 4 ? 1 : 2)];
  return n_items <= at_once;
}

// Whether a planned launch uses the kernel that overlaps the ends of its items with the next ones: blocks of one slab, whose
// items are the shortest, attending fewer than 64 key slabs on average.  1x8x16 blocks of an 8x32x48 grid, 12 heads, us
// without and with: 15.6 key blocks 193 / 178, 19.5 221 / 198, 33.7 312 / 301, 65 532 / 532.  Items of two query slabs have
// two warpgroups' rows to write and lose by it: 1x16x16 blocks attending 9.2 blocks 174 / 169 but 26.6 of a 16x48x80 grid
// 1,308 / 1,353, 1x15x16 30.1 974 / 1,015; so do blocks of three slabs (3x8x16, 6.6 blocks 204 / 225).
bool short_items(const HostGeom& g, const long long* weights, int n_heads) {
  long long total = 0;
  for (int h = 0; h < n_heads; ++h) total += weights[h];
  return g.n_sub == 1 && (double)total * slabs_per_block(g) < (64.0 - g.n_ts) * n_heads * g.NB;
}

// Planning (unless the launch is direct) and attention.
cudaError_t launch_call(const TensorMapsCut& tm, const AttnParams& prm, const HostGeom& hg, const psa_head_params* params, const long long* weights,
                        const Workspace& ws, int cluster, bool record, cudaStream_t st) {
  HeadParamsArray heads;   // entries beyond the launch's heads are never read, nor any of a planned launch
  const int n = prm.g.n_heads;
  const bool direct = runs_at_once(ws, prm.n_items, cluster);
  if (direct) {
    std::memcpy(heads.p, params, sizeof(psa_head_params) * (size_t)n);
  } else {
    PlanParams pp;
    plan_params(&pp, params, weights, n);
    const cudaError_t e = launch_plan(pp, prm.g, n, prm.ws_header, const_cast<psa_head_params*>(prm.hp_dev),
                                      const_cast<WorkItem*>(prm.items), st);
    if (e != cudaSuccess) return e;
    ++g_launches;
  }
  if (record && g_ev_start && g_ev_stop) cudaEventRecord(g_ev_start, st);
  AttnParamsCut pe;
  static_cast<AttnParams&>(pe) = prm;
  if (hg.grid == kCut) {
    std::memcpy(pe.cls, hg.cls, sizeof(pe.cls));
    pe.planned = hg.planned;
    pe.n_classes = hg.n_classes;
    std::memcpy(pe.order, hg.order, sizeof(pe.order));
  }
  const cudaError_t e = launch_attn(tm, heads, pe, ws.n_sms, cluster, hg.grid, direct, short_items(hg, weights, n), hg.empty_slabs, st,
                                    &g_last_attn.mode);
  if (e == cudaSuccess) {
    ++g_launches;
    g_last_attn.items = prm.n_items;
    g_last_attn.cluster = cluster;
    g_last_attn.grid = hg.grid;
    g_last_attn.slabs = hg.main_slabs;
    g_last_attn.last_keys = hg.main_last;
    g_last_attn.edge_axes = hg.edge_axes;
    for (int c = 0; c < 8; ++c) {
      const int slabs = class_blocks(hg, c) ? hg.slabs_of[c] : 0;
      const bool follows = hg.grid == kCut ? hg.cls[c].in_pattern != 0 : slabs == hg.main_slabs;
      g_last_attn.query_slabs[c] = (uint8_t)slabs;
      g_last_attn.together[c] = hg.grid == kCut && slabs ? hg.cls[c].together : 1;
      g_last_attn.keys[c] = (uint16_t)(slabs == 0 ? 0 : (slabs - 1) * kSlabTokens + (follows ? hg.main_last : kSlabTokens));
    }
  }
  return e;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- helper streams of psa_attn_fwd_host (one set per device, created on first use) ----------
constexpr int kHostChunks = 64;   // upper bound on the chunks of one host-tensor call
struct HostPipe {
  bool ready = false;
  cudaStream_t h2d = nullptr, d2h = nullptr;
  cudaEvent_t ev_start = nullptr, ev_end = nullptr, ev_mid[kHostChunks] = {}, ev_in[kHostChunks] = {}, ev_done[kHostChunks] = {};
};
HostPipe g_pipe[kMaxDevices];

HostPipe* host_pipe(int dev) {   // caller holds g_mu; returns nullptr if the streams cannot be created
  HostPipe& p = g_pipe[dev];
  if (p.ready) return &p;
  if (cudaStreamCreateWithFlags(&p.h2d, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (cudaStreamCreateWithFlags(&p.d2h, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (cudaEventCreateWithFlags(&p.ev_start, cudaEventDisableTiming) != cudaSuccess) return nullptr;
  if (cudaEventCreateWithFlags(&p.ev_end, cudaEventDisableTiming) != cudaSuccess) return nullptr;
  for (int i = 0; i < kHostChunks; ++i) {
    if (cudaEventCreateWithFlags(&p.ev_mid[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&p.ev_in[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&p.ev_done[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
  }
  p.ready = true;
  return &p;
}

// ---- scratch of psa_attn_fwd_noalloc ------------------------------------------------------
// Layout: 16 int32 header words (status, detail, scheduler ticket, reporting call), kMaxHeads head parameter
// records, then up to kNoAllocMaxItems work items.  It lives in every GPU that loads the
// library, from load to exit.
constexpr int kNoAllocMaxItems = 16384;
constexpr size_t kNoAllocParamsOff = sizeof(int) * kWsHeaderWords;
constexpr size_t kNoAllocItemsOff = (kNoAllocParamsOff + sizeof(psa_head_params) * kMaxHeads + 255) & ~size_t(255);
constexpr size_t kNoAllocBytes = kNoAllocItemsOff + sizeof(WorkItem) * (size_t)kNoAllocMaxItems;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device address of the array, looked up once per device with that device current.  In host
// code the array's name is only a handle for the runtime, never an address a kernel may use.
void* g_noalloc_ptr[kMaxDevices] = {};

int noalloc_scratch(int dev, void** ptr) {
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) return PSA_ERR_CUDA;
    g_noalloc_ptr[dev] = p;
  }
  *ptr = g_noalloc_ptr[dev];
  return PSA_OK;
}

}  // namespace

extern "C" {

const char* psa_status_string(int status) {
  switch (status) {
    case PSA_OK: return "ok";
    case PSA_ERR_INVALID_ARG: return "invalid argument";
    case PSA_ERR_UNSUPPORTED: return "unsupported configuration";
    case PSA_ERR_CAPACITY: return "capacity exceeded (col_idx too small, or problem beyond the fixed scratch)";
    case PSA_ERR_CUDA: return "CUDA call failed";
    case PSA_ERR_TIMEOUT: return "device-side wait timed out";
    case PSA_ERR_INTERNAL: return "kernel-side consistency check failed (checked build)";
    default: return "unknown status";
  }
}

int64_t psa_launch_count(void) { return g_launches.load(); }

int psa_last_attn_launch(int32_t* mode, int32_t* ctas_per_item) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (mode) *mode = g_last_attn.mode;
  if (ctas_per_item) *ctas_per_item = g_last_attn.cluster;
  return g_last_attn.items;
}

int psa_last_attn_grid(int32_t* slabs, int32_t* last_keys) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (slabs) *slabs = g_last_attn.slabs;
  if (last_keys) *last_keys = g_last_attn.last_keys;
  return g_last_attn.grid;
}

int psa_last_attn_class(int c, int32_t* query_slabs, int32_t* keys, int32_t* together) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (c < 0 || c > 7) return PSA_ERR_INVALID_ARG;
  if (query_slabs) *query_slabs = g_last_attn.query_slabs[c];
  if (keys) *keys = g_last_attn.keys[c];
  if (together) *together = g_last_attn.together[c];
  return g_last_attn.edge_axes;
}

int psa_profile_events(void* start_event, void* stop_event) {
  std::lock_guard<std::mutex> lock(g_mu);
  if ((start_event == nullptr) != (stop_event == nullptr)) return PSA_ERR_INVALID_ARG;
  g_ev_start = static_cast<cudaEvent_t>(start_event);
  g_ev_stop = static_cast<cudaEvent_t>(stop_event);
  return PSA_OK;
}

int psa_mask_sizes(const psa_head_params* params, const psa_problem* prob, int T, int H, int W, int64_t* nb,
                   int64_t* nnz) {
  HostGeom g;
  const int rc = make_geom(prob, T, H, W, false, &g);
  if (rc != PSA_OK) return rc;
  if (nb) *nb = g.NB;
  if (nnz) {
    if (!params) return PSA_ERR_INVALID_ARG;
    long long tot = 0;
    for (int h = 0; h < prob->n_heads; ++h) {
      if (!valid_params(params[h])) return PSA_ERR_INVALID_ARG;
      tot += head_nnz(params[h], g);
    }
    *nnz = tot;
  }
  return PSA_OK;
}

int psa_mask_build(const psa_head_params* params, const psa_problem* prob, int T, int H, int W, uint8_t* block_mask,
                   int32_t* row_ptr, int32_t* col_idx, int64_t col_capacity, void* stream) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, false, &g);
  if (rc != PSA_OK) return rc;
  if (!params) return PSA_ERR_INVALID_ARG;
  if (col_idx && !row_ptr) return PSA_ERR_INVALID_ARG;
  if (block_mask && !aligned16(block_mask)) return PSA_ERR_INVALID_ARG;
  if ((row_ptr && (reinterpret_cast<uintptr_t>(row_ptr) & 3u)) || (col_idx && (reinterpret_cast<uintptr_t>(col_idx) & 3u)))
    return PSA_ERR_INVALID_ARG;
  // exclusive prefix of the per-head pair counts, and each head's axis sets where the kernel takes them (one walk over
  // the differences gives both)
  const bool small = mask_build_small(g);
  std::vector<long long> base(prob->n_heads + 1, 0);
  std::vector<AxisSet> sets(small ? 2 * (size_t)prob->n_heads : 0);
  for (int h = 0; h < prob->n_heads; ++h) {
    const psa_head_params& p = params[h];
    if (!valid_params(p)) return PSA_ERR_INVALID_ARG;
    if (small) {
      sets[2 * h] = axis_set(g.Tp, p.Tw, p.To, p.Ts);
      sets[2 * h + 1] = axis_set(g.Sp, p.Sw, p.So, p.Ss);
      base[h + 1] = base[h] + (long long)sets[2 * h].pairs * sets[2 * h + 1].pairs;
    } else {
      base[h + 1] = base[h] + head_nnz(p, g);
    }
  }
  const long long nnz = base[prob->n_heads];
  if (nnz >= (1ll << 31) || (long long)prob->n_heads * g.NB >= (1ll << 31) - 1) return PSA_ERR_UNSUPPORTED;
  if (col_idx && col_capacity < nnz) return PSA_ERR_CAPACITY;
  int dev;
  Workspace* ws;
  std::lock_guard<std::mutex> lock(g_mu);
  rc = device_info(&dev, &ws);
  if (rc != PSA_OK) return rc;
  for (int head0 = 0; head0 < prob->n_heads; head0 += kMaxHeads) {
    const int n_here = prob->n_heads - head0 < kMaxHeads ? prob->n_heads - head0 : kMaxHeads;
    HeadParamsArray hp;
    int bases[kMaxHeads];
    for (int h = 0; h < n_here; ++h) {
      hp.p[h] = params[head0 + h];
      bases[h] = (int)base[head0 + h];
    }
    int launches = 0;
    const cudaError_t e = launch_mask_build(hp, small ? &sets[2 * (size_t)head0] : nullptr, bases, g, n_here, block_mask ? block_mask + (long long)head0 * g.NB * g.NB : nullptr,
                                            row_ptr ? row_ptr + (long long)head0 * g.NB : nullptr, col_idx,
                                            (int)base[head0 + n_here], ws->n_sms, static_cast<cudaStream_t>(stream), &launches);
    g_launches += launches;
    if (e != cudaSuccess) return PSA_ERR_CUDA;
  }
  return PSA_OK;
}

// Planning + attention launches for n_heads heads (in launches of at most kMaxHeads) on the cached
// per-device workspace.  Arguments are already validated; g_mu is held by the caller.
// new_call: this is the first launch sequence of an API call (later ones report under the same id, so that an error of
// an earlier one -- more than 128 heads, chunks of a host-tensor call, samples of a batched call -- is not lost).
// cluster: CTAs per work item, and the grid as it is; 0: both by choose_edges for these heads; -1: one CTA, the grid by choose_edges.
static int run_attn(const void* q, const void* k, const void* v, void* out, float* lse, const psa_head_params* head_params,
                    int n_heads, HostGeom g, const Layout& lay, cudaStream_t st, bool new_call = true, int cluster = 0) {
  int dev;
  Workspace* ws;
  int rc = device_info(&dev, &ws);
  if (rc != PSA_OK) return rc;
  rc = init_attn(ws);
  if (rc != PSA_OK) return rc;
  const int chunk = n_heads < kMaxHeads ? n_heads : kMaxHeads;
  const size_t items_bytes = sizeof(WorkItem) * (size_t)chunk * g.items_per_head;
  const size_t hp_off = sizeof(int) * kWsHeaderWords;
  const size_t items_off = (hp_off + sizeof(psa_head_params) * kMaxHeads + 255) & ~size_t(255);
  rc = ensure_workspace(ws, items_off + items_bytes);
  if (rc != PSA_OK) return rc;
  int* ws_header = static_cast<int*>(ws->base);
  psa_head_params* hp_dev = reinterpret_cast<psa_head_params*>(static_cast<char*>(ws->base) + hp_off);
  WorkItem* items = reinterpret_cast<WorkItem*>(static_cast<char*>(ws->base) + items_off);
  std::vector<long long> weights((size_t)n_heads);
  head_weights(head_params, n_heads, g, weights.data());
  if (cluster <= 0) {
    const int chosen = choose_edges(*ws, &g, weights.data(), n_heads);
    cluster = cluster < 0 ? 1 : chosen;
  }
  if (new_call) ws->last_call = next_call_id(st);
  for (int head0 = 0; head0 < n_heads; head0 += kMaxHeads) {
    const int n_here = n_heads - head0 < kMaxHeads ? n_heads - head0 : kMaxHeads;
    const long long in_off = lay.shared_qkv ? 0 : (long long)head0 * lay.in_head;
    const long long out_off = (long long)head0 * lay.out_head;
    TensorMapsCut tm;
    if ((rc = encode_maps(&tm, static_cast<const uint16_t*>(q) + in_off, static_cast<const uint16_t*>(k) + in_off,
                          static_cast<const uint16_t*>(v) + in_off, static_cast<uint16_t*>(out) + out_off, g, lay, n_here)) != PSA_OK)
      return rc;
    Geom gh = g;
    gh.n_heads = n_here;
    const int n_items = n_here * g.items_per_head;
    const AttnParams prm = {gh, items, hp_dev, ws_header, lse + (long long)head0 * g.Lt, n_items,
                            ws->last_call, lay.shared_qkv ? 1 : 0, static_cast<uint16_t*>(out) + out_off, lay.out_head, lay.out_token};
    if (launch_call(tm, prm, g, head_params + head0, weights.data() + head0, *ws, cluster, true, st) != cudaSuccess) return PSA_ERR_CUDA;
    if (g_ev_start && g_ev_stop) cudaEventRecord(g_ev_stop, st);
  }
  return PSA_OK;
}

// psa_attn_fwd with the choice of continuing an API call, of the CTAs per item and of the grid's edges (chunks of one host-tensor call).
static int attn_fwd_checked(const void* q, const void* k, const void* v, void* out, float* lse,
                            const psa_head_params* head_params, const psa_problem* prob, int T, int H, int W, void* stream,
                            bool new_call, int cluster = 0, const HostGeom* chosen = nullptr) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  if (!q || !k || !v || !out || !lse || !head_params) return PSA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || (reinterpret_cast<uintptr_t>(lse) & 3u))
    return PSA_ERR_INVALID_ARG;
  if (out == q || out == k || out == v) return PSA_ERR_INVALID_ARG;
  if (prob->stride_token < kHeadDim || (prob->stride_token % 8) != 0) return PSA_ERR_INVALID_ARG;
  if (prob->n_heads > 1 && (prob->stride_head < kHeadDim || (prob->stride_head % 8) != 0)) return PSA_ERR_INVALID_ARG;
  for (int h = 0; h < prob->n_heads; ++h)
    if (!valid_params(head_params[h])) return PSA_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  const Layout lay = {prob->stride_head, prob->stride_token, prob->stride_head, prob->stride_token, false};
  return run_attn(q, k, v, out, lse, head_params, prob->n_heads, chosen ? *chosen : g, lay, static_cast<cudaStream_t>(stream), new_call,
                  cluster);
}

int psa_attn_fwd(const void* q, const void* k, const void* v, void* out, float* lse, const psa_head_params* head_params,
                 const psa_problem* prob, int T, int H, int W, void* stream) {
  return attn_fwd_checked(q, k, v, out, lse, head_params, prob, T, H, W, stream, true);
}

int psa_search_select_at_sparsity(const float* losses, const float* sparsity, int n, float target) {
  if (!losses || !sparsity || n < 1) return PSA_ERR_INVALID_ARG;
  int best = -1;
  for (int i = 0; i < n; ++i)
    if (sparsity[i] >= target && (best < 0 || losses[i] < losses[best])) best = i;
  return best < 0 ? PSA_ERR_CAPACITY : best;
}

int psa_attn_fwd_batched(const void* q, const void* k, const void* v, void* out, float* lse,
                         const psa_head_params* head_params, const psa_problem* prob, int n_batch, int64_t stride_batch,
                         int T, int H, int W, void* stream) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  if (!q || !k || !v || !out || !lse || !head_params || n_batch < 1) return PSA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || (reinterpret_cast<uintptr_t>(lse) & 3u))
    return PSA_ERR_INVALID_ARG;
  if (out == q || out == k || out == v) return PSA_ERR_INVALID_ARG;
  if (prob->stride_token < kHeadDim || (prob->stride_token % 8) != 0) return PSA_ERR_INVALID_ARG;
  if (prob->n_heads > 1 && (prob->stride_head < kHeadDim || (prob->stride_head % 8) != 0)) return PSA_ERR_INVALID_ARG;
  if (n_batch > 1 && (stride_batch < kHeadDim || (stride_batch % 8) != 0)) return PSA_ERR_INVALID_ARG;
  for (int h = 0; h < prob->n_heads; ++h)
    if (!valid_params(head_params[h])) return PSA_ERR_INVALID_ARG;
  const int nh = prob->n_heads;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(g_mu);
  const bool fold = n_batch == 1 || (nh == 1 ? true : stride_batch == (int64_t)nh * prob->stride_head);
  if (fold) {
    // samples are evenly spaced heads: one launch sequence over n_batch * n_heads heads
    if ((long long)n_batch * nh >= (1ll << 24)) return PSA_ERR_UNSUPPORTED;
    std::vector<psa_head_params> params((size_t)n_batch * nh);
    for (int b = 0; b < n_batch; ++b)
      for (int h = 0; h < nh; ++h) params[(size_t)b * nh + h] = head_params[h];
    const long long hs = nh == 1 ? (n_batch > 1 ? stride_batch : prob->stride_head) : prob->stride_head;
    const Layout lay = {hs, prob->stride_token, hs, prob->stride_token, false};
    return run_attn(q, k, v, out, lse, params.data(), n_batch * nh, g, lay, st);
  }
  const Layout lay = {prob->stride_head, prob->stride_token, prob->stride_head, prob->stride_token, false};
  for (int b = 0; b < n_batch; ++b) {
    const long long off = (long long)b * stride_batch;
    rc = run_attn(static_cast<const uint16_t*>(q) + off, static_cast<const uint16_t*>(k) + off,
                  static_cast<const uint16_t*>(v) + off, static_cast<uint16_t*>(out) + off,
                  lse + (long long)b * nh * g.L, head_params, nh, g, lay, st, b == 0);
    if (rc != PSA_OK) return rc;
  }
  return PSA_OK;
}

int psa_attn_fwd_joint(const void* q, const void* k, const void* v, void* out, float* lse,
                       const psa_head_params* head_params, const psa_problem* prob, int64_t n_text, int T, int H, int W,
                       void* stream) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  if ((rc = set_text(&g, n_text)) != PSA_OK) return rc;
  if (!q || !k || !v || !out || !lse || !head_params) return PSA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || (reinterpret_cast<uintptr_t>(lse) & 3u))
    return PSA_ERR_INVALID_ARG;
  if (out == q || out == k || out == v) return PSA_ERR_INVALID_ARG;
  if (prob->stride_token < kHeadDim || (prob->stride_token % 8) != 0) return PSA_ERR_INVALID_ARG;
  if (prob->n_heads > 1 && (prob->stride_head < kHeadDim || (prob->stride_head % 8) != 0)) return PSA_ERR_INVALID_ARG;
  for (int h = 0; h < prob->n_heads; ++h)
    if (!valid_params(head_params[h])) return PSA_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  const Layout lay = {prob->stride_head, prob->stride_token, prob->stride_head, prob->stride_token, false};
  return run_attn(q, k, v, out, lse, head_params, prob->n_heads, g, lay, static_cast<cudaStream_t>(stream));
}

// ---- PSA-Search for one head (Algorithm 3) ------------------------------------------------------
// scratch layout: outputs of the n_cand candidates and of full attention ((n_cand + 1) x L x 128 bf16),
// their lse ((n_cand + 1) x L fp32), the partial sums of the loss reduction.
static size_t search_out_bytes(int n_cand, long long L) { return ((size_t)(n_cand + 1) * L * kHeadDim * 2 + 255) & ~size_t(255); }
static size_t search_lse_bytes(int n_cand, long long L) { return ((size_t)(n_cand + 1) * L * 4 + 255) & ~size_t(255); }

int64_t psa_search_scratch_bytes(int n_cand, int T, int H, int W) {
  if (n_cand < 1 || T < 1 || H < 1 || W < 1) return PSA_ERR_INVALID_ARG;
  const long long L = (long long)T * H * W;
  return (int64_t)(search_out_bytes(n_cand, L) + search_lse_bytes(n_cand, L) + search_partial_bytes(n_cand));
}

int psa_search_losses(const void* q, const void* k, const void* v, const psa_head_params* candidates, int n_cand,
                      const psa_problem* prob, int T, int H, int W, void* scratch, float* losses, void* stream) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  if (!q || !k || !v || !candidates || !scratch || !losses || n_cand < 1) return PSA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || (reinterpret_cast<uintptr_t>(scratch) & 255u) ||
      (reinterpret_cast<uintptr_t>(losses) & 3u))
    return PSA_ERR_INVALID_ARG;
  if (prob->stride_token < kHeadDim || (prob->stride_token % 8) != 0) return PSA_ERR_INVALID_ARG;
  // candidate masks, then one all-covering mask: full attention with the same kernel
  std::vector<psa_head_params> params(candidates, candidates + n_cand);
  for (int c = 0; c < n_cand; ++c)
    if (!valid_params(params[c])) return PSA_ERR_INVALID_ARG;
  const psa_head_params full = {g.Tp, 0, 0, g.Sp, 0, 0};
  params.push_back(full);
  char* base = static_cast<char*>(scratch);
  uint16_t* outs = reinterpret_cast<uint16_t*>(base);
  float* lse = reinterpret_cast<float*>(base + search_out_bytes(n_cand, g.L));
  double* partial = reinterpret_cast<double*>(base + search_out_bytes(n_cand, g.L) + search_lse_bytes(n_cand, g.L));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(g_mu);
  const Layout lay = {0, prob->stride_token, g.L * kHeadDim, kHeadDim, true};
  // whole items: with n_cand + 1 of them per block they are rarely few, and every candidate's output is then rounded as
  // a plain call's is (the losses are differences of outputs)
  rc = run_attn(q, k, v, outs, lse, params.data(), n_cand + 1, g, lay, st, true, -1);
  if (rc != PSA_OK) return rc;
  int launches = 0;
  const cudaError_t e = launch_search_losses(outs, outs + (long long)n_cand * g.L * kHeadDim, g.L * kHeadDim, n_cand, partial,
                                             losses, st, &launches);
  g_launches += launches;
  return e == cudaSuccess ? PSA_OK : PSA_ERR_CUDA;
}

int psa_search_select(const float* losses, const float* sparsity, int n, float alpha) {
  if (!losses || !sparsity || n < 1) return PSA_ERR_INVALID_ARG;
  // Algorithm 3 walks the candidates in order of (loss, index), starts at the first and moves to
  // any strictly sparser one whose loss is within alpha.  Its result, stated directly: if no loss
  // is within alpha, the candidate of minimal (loss, index); otherwise the sparsest candidate
  // among those within alpha, ties by minimal (loss, index).
  int lowest = -1, best = -1;
  for (int i = 0; i < n; ++i) {
    if (!std::isfinite(losses[i]) || std::isnan(sparsity[i])) return PSA_ERR_INVALID_ARG;
    if (lowest < 0 || losses[i] < losses[lowest]) lowest = i;
    if (losses[i] <= alpha &&
        (best < 0 || sparsity[i] > sparsity[best] || (sparsity[i] == sparsity[best] && losses[i] < losses[best])))
      best = i;
  }
  return best >= 0 ? best : lowest;
}

int psa_attn_fwd_noalloc(const void* q, const void* k, const void* v, void* out, float* lse,
                         const psa_head_params* head_params, const psa_problem* prob, int T, int H, int W, void* stream,
                         int32_t* status_detail) {
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  if (!q || !k || !v || !out || !lse || !head_params) return PSA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || (reinterpret_cast<uintptr_t>(lse) & 3u))
    return PSA_ERR_INVALID_ARG;
  if (out == q || out == k || out == v) return PSA_ERR_INVALID_ARG;
  if (prob->stride_token < kHeadDim || (prob->stride_token % 8) != 0) return PSA_ERR_INVALID_ARG;
  if (prob->n_heads > 1 && (prob->stride_head < kHeadDim || (prob->stride_head % 8) != 0)) return PSA_ERR_INVALID_ARG;
  for (int h = 0; h < prob->n_heads; ++h)
    if (!valid_params(head_params[h])) return PSA_ERR_INVALID_ARG;
  // the fixed scratch bounds the problem: one launch worth of heads and kNoAllocMaxItems items
  // (edge blocks counted like the others, whatever items they save: the limit that the header states)
  if (prob->n_heads > kMaxHeads || (long long)prob->n_heads * g.NB * g.items_per_block > kNoAllocMaxItems) return PSA_ERR_CAPACITY;

  std::lock_guard<std::mutex> lock(g_mu);
  int dev;
  Workspace* ws;
  rc = device_info(&dev, &ws);
  if (rc != PSA_OK) return rc;
  rc = init_attn(ws);
  if (rc != PSA_OK) return rc;
  void* base = nullptr;
  rc = noalloc_scratch(dev, &base);
  if (rc != PSA_OK) return rc;
  int* header = static_cast<int*>(base);
  psa_head_params* hp_dev = reinterpret_cast<psa_head_params*>(static_cast<char*>(base) + kNoAllocParamsOff);
  WorkItem* items = reinterpret_cast<WorkItem*>(static_cast<char*>(base) + kNoAllocItemsOff);
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  // What the kernels read of the scratch is written by this call's planning kernel; nothing of the previous call is read.
  long long weights[kMaxHeads];
  head_weights(head_params, prob->n_heads, g, weights);
  const int cluster = choose_edges(*ws, &g, weights, prob->n_heads);
  TensorMapsCut tm;
  const Layout lay = {prob->stride_head, prob->stride_token, prob->stride_head, prob->stride_token, false};
  if ((rc = encode_maps(&tm, q, k, v, out, g, lay, prob->n_heads)) != PSA_OK) return rc;
  const int n_items = prob->n_heads * g.items_per_head, call_id = next_call_id(st);
  const AttnParams prm = {g, items, hp_dev, header, lse, n_items, call_id, 0,
                          out, lay.out_head, lay.out_token};
  if (launch_call(tm, prm, g, head_params, weights, *ws, cluster, false, st) != cudaSuccess) return PSA_ERR_CUDA;
  if (status_detail) {
    if (cudaStreamSynchronize(st) != cudaSuccess) return PSA_ERR_CUDA;
    return read_status(header, call_id, status_detail);
  }
  return PSA_OK;
}

int psa_attn_fwd_host(const void* q, const void* k, const void* v, void* out, float* lse, void* d_q, void* d_k, void* d_v,
                      void* d_out, float* d_lse, const psa_head_params* head_params, const psa_problem* prob, int T, int H,
                      int W, void* stream) {
  if (!prob || !q || !k || !v || !out || !lse || !d_q || !d_k || !d_v || !d_out || !d_lse || !head_params)
    return PSA_ERR_INVALID_ARG;
  if (T < 1 || H < 1 || W < 1 || prob->n_heads < 1) return PSA_ERR_INVALID_ARG;
  const long long L = (long long)T * H * W;
  const size_t head_span = (size_t)(L - 1) * prob->stride_token + prob->head_dim;  // elements one head touches
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  // Heads are independent problems: when they are the outermost dimension of the layout the
  // call is pipelined over chunks of heads -- chunk c+1 is copied in and chunk c-1 copied out
  // while chunk c computes (two helper streams per device, created on first use).
  const bool head_major = prob->n_heads == 1 || (size_t)prob->stride_head >= head_span;
  int dev = 0;
  HostPipe* pipe = nullptr;
  if (head_major && prob->n_heads >= 2 && cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_mu);
    pipe = host_pipe(dev);
  }
  if (!pipe) {
    const size_t bytes = ((size_t)(prob->n_heads - 1) * prob->stride_head + head_span) * 2;
    if (cudaMemcpyAsync(d_q, q, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaMemcpyAsync(d_k, k, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaMemcpyAsync(d_v, v, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return PSA_ERR_CUDA;
    const int rc = psa_attn_fwd(d_q, d_k, d_v, d_out, d_lse, head_params, prob, T, H, W, stream);
    if (rc != PSA_OK) return rc;
    if (cudaMemcpyAsync(out, d_out, bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaMemcpyAsync(lse, d_lse, sizeof(float) * (size_t)prob->n_heads * L, cudaMemcpyDeviceToHost, st) != cudaSuccess)
      return PSA_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PSA_ERR_CUDA;
    return PSA_OK;
  }

  // Chunk size: the call is bound by the host-to-device copies, so what is exposed is the first
  // chunk's copy-in and the last chunk's compute and copy-out -- both shrink with the chunk.
  int want = host_chunks();
  if (want > kHostChunks - 8) want = kHostChunks - 8;   // single-head edge chunks and broken runs add a few
  const int n_chunks = prob->n_heads < want ? prob->n_heads : want;
  const int per = (prob->n_heads + n_chunks - 1) / n_chunks;
  // everything enqueued on `stream` before this call precedes the first copy
  if (cudaEventRecord(pipe->ev_start, st) != cudaSuccess) return PSA_ERR_CUDA;
  if (cudaStreamWaitEvent(pipe->h2d, pipe->ev_start, 0) != cudaSuccess) return PSA_ERR_CUDA;
  if (cudaStreamWaitEvent(pipe->d2h, pipe->ev_start, 0) != cudaSuccess) return PSA_ERR_CUDA;
  // The first and the last chunks are the exposed ones, so the call starts and ends with
  // single-head chunks (two at each end, when the regular chunk is larger than that), and the two
  // heads with the fewest attended block pairs (the shortest kernels) are kept for the end: what
  // remains after the last byte has arrived is the lightest head's kernel and its copy-out.
  // (With one head per chunk, too: 12 heads of 32,760 tokens 6.53 -> 6.42 ms.)
  const int n_edge = (per >= 2 && prob->n_heads >= 4 * per) ? 2 : 0;
  struct Chunk { int h0, nh; };
  Chunk chunks[kHostChunks];
  int n_list = 0;
  int last1 = -1, last2 = -1;   // lightest and second-lightest head
  HostGeom g;
  int rc = make_geom(prob, T, H, W, true, &g);
  if (rc != PSA_OK) return rc;
  for (int h = 0; h < prob->n_heads; ++h)
    if (!valid_params(head_params[h])) return PSA_ERR_INVALID_ARG;
  std::vector<long long> weights((size_t)prob->n_heads);
  head_weights(head_params, prob->n_heads, g, weights.data());
  int cluster;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    Workspace* ws;
    if ((rc = device_info(&dev, &ws)) != PSA_OK || (rc = init_attn(ws)) != PSA_OK) return rc;
    cluster = choose_edges(*ws, &g, weights.data(), prob->n_heads);
  }
  if (n_edge || (per == 1 && prob->n_heads >= 3)) {
    for (int h = 0; h < prob->n_heads; ++h) {
      const long long w = weights[h];
      if (last1 < 0 || w < weights[last1]) { last2 = last1; last1 = h; }
      else if (last2 < 0 || w < weights[last2]) last2 = h;
    }
  }
  {
    int singles = n_edge;   // single-head chunks still to open the call with
    int h = 0;
    while (h < prob->n_heads) {
      if (h == last1 || h == last2) { ++h; continue; }
      int nh = 1;
      if (singles > 0) --singles;
      else
        while (nh < per && h + nh < prob->n_heads && h + nh != last1 && h + nh != last2) ++nh;
      if (n_list >= kHostChunks - 2) return PSA_ERR_UNSUPPORTED;
      chunks[n_list++] = Chunk{h, nh};
      h += nh;
    }
    if (last2 >= 0) chunks[n_list++] = Chunk{last2, 1};
    if (last1 >= 0) chunks[n_list++] = Chunk{last1, 1};
  }
  auto offset = [&](int c) -> size_t { return (size_t)chunks[c].h0 * prob->stride_head; };   // elements
  auto span = [&](int c) -> size_t { return ((size_t)(chunks[c].nh - 1) * prob->stride_head + head_span) * 2; };
  // Copies chunk c out when it is computed -- and, while copies in follow, not before the next chunk's second one has ended, so
  // that it starts together with the third.  A copy out that starts in the middle of a copy in leaves a gap of 45 us in front of
  // the next copy in, where one that starts at the boundary leaves 15: 12 heads of 32,760 tokens, whose kernels take 130 to 290 us
  // and a tensor of a chunk 155, 6.52 ms without this and 6.21 with it (6.14 for the copies alone); 28 heads of 2,560 tokens 1.51
  // and 1.45; no difference where two tensors take longer or shorter than the kernels by much.  Behind the first copy instead: 6.52.
  auto copy_out = [&](int c) -> bool {
    const size_t first = (size_t)chunks[c].h0 * L;
    return cudaStreamWaitEvent(pipe->d2h, pipe->ev_done[c], 0) == cudaSuccess &&
           (c + 1 == n_list || cudaStreamWaitEvent(pipe->d2h, pipe->ev_mid[c + 1], 0) == cudaSuccess) &&
           cudaMemcpyAsync(static_cast<uint16_t*>(out) + offset(c), static_cast<uint16_t*>(d_out) + offset(c), span(c), cudaMemcpyDeviceToHost,
                           pipe->d2h) == cudaSuccess &&
           cudaMemcpyAsync(lse + first, d_lse + first, sizeof(float) * (size_t)chunks[c].nh * L, cudaMemcpyDeviceToHost, pipe->d2h) == cudaSuccess;
  };
  for (int c = 0; c < n_list; ++c) {
    const int h0 = chunks[c].h0, nh = chunks[c].nh;
    const size_t off = offset(c), bytes = span(c);
    const uint16_t *hq = static_cast<const uint16_t*>(q) + off, *hk = static_cast<const uint16_t*>(k) + off,
                   *hv = static_cast<const uint16_t*>(v) + off;
    uint16_t *dq = static_cast<uint16_t*>(d_q) + off, *dk = static_cast<uint16_t*>(d_k) + off,
             *dv = static_cast<uint16_t*>(d_v) + off, *dout = static_cast<uint16_t*>(d_out) + off;
    if (cudaMemcpyAsync(dq, hq, bytes, cudaMemcpyHostToDevice, pipe->h2d) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaMemcpyAsync(dk, hk, bytes, cudaMemcpyHostToDevice, pipe->h2d) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaEventRecord(pipe->ev_mid[c], pipe->h2d) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaMemcpyAsync(dv, hv, bytes, cudaMemcpyHostToDevice, pipe->h2d) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaEventRecord(pipe->ev_in[c], pipe->h2d) != cudaSuccess) return PSA_ERR_CUDA;
    if (cudaStreamWaitEvent(st, pipe->ev_in[c], 0) != cudaSuccess) return PSA_ERR_CUDA;
    psa_problem sub = *prob;
    sub.n_heads = nh;
    rc = attn_fwd_checked(dq, dk, dv, dout, d_lse + (size_t)h0 * L, head_params + h0, &sub, T, H, W, stream, c == 0, cluster, &g);
    if (rc != PSA_OK) return rc;
    if (cudaEventRecord(pipe->ev_done[c], st) != cudaSuccess) return PSA_ERR_CUDA;
    if (c > 0 && !copy_out(c - 1)) return PSA_ERR_CUDA;
  }
  if (!copy_out(n_list - 1)) return PSA_ERR_CUDA;
  if (cudaEventRecord(pipe->ev_end, pipe->d2h) != cudaSuccess) return PSA_ERR_CUDA;
  if (cudaStreamWaitEvent(st, pipe->ev_end, 0) != cudaSuccess) return PSA_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return PSA_ERR_CUDA;
  return PSA_OK;
}

int psa_selftest_wait_timeout(int limit_ms, void* stream) {
  if (limit_ms < 1 || limit_ms > 1000) return PSA_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  int dev;
  Workspace* ws;
  int rc = device_info(&dev, &ws);
  if (rc != PSA_OK) return rc;
  rc = ensure_workspace(ws, 4096);
  if (rc != PSA_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ws->last_call = next_call_id(st);
  if (launch_wait_probe(static_cast<int*>(ws->base), ws->last_call, 1000000ull * (unsigned long long)limit_ms, st) != cudaSuccess)
    return PSA_ERR_CUDA;
  ++g_launches;
  return PSA_OK;
}

int psa_last_device_status(int32_t* detail) {
  std::lock_guard<std::mutex> lock(g_mu);
  int dev;
  Workspace* ws;
  int rc = device_info(&dev, &ws);
  if (rc != PSA_OK) return rc;
  if (cudaDeviceSynchronize() != cudaSuccess) return PSA_ERR_CUDA;
  if (detail) *detail = 0;
  if (!ws->base) return PSA_OK;
  return read_status(ws->base, ws->last_call, detail);
}

int psa_shutdown(void) {
  std::lock_guard<std::mutex> lock(g_mu);
  int cur = 0;
  if (cudaGetDevice(&cur) != cudaSuccess) return PSA_OK;  // no usable device: nothing was allocated
  for (int d = 0; d < kMaxDevices; ++d) {
    if (g_ws[d].base) {
      cudaSetDevice(d);
      cudaDeviceSynchronize();
      cudaFree(g_ws[d].base);
      g_ws[d].base = nullptr;
      g_ws[d].bytes = 0;
    }
  }
  cudaSetDevice(cur);
  return PSA_OK;
}

}  // extern "C"
