// Shared host/device definitions of the PSA library (not part of the public ABI).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "psa.h"

namespace psa {

constexpr int kHeadDim = 128;     // head dimension the attention kernel is built for
constexpr int kSlabTokens = 128;  // tokens per compute slab (one MMA tile of rows / keys)
constexpr int kMaxHeads = 128;    // heads per launch (parameters travel by value)
constexpr int kMaxTp = 256;       // limits of the in-kernel key-block bitmasks
constexpr int kMaxSp = 2048;
constexpr size_t kMaxSmemBytes = 232448;   // 227 KB of shared memory that a CTA may use

// How a launch treats blocks that reach beyond the grid (3D-padding).
//   kWhole    the block divides the grid: there are none
//   kPadded   they are loaded like the others, with masks, less the slabs that hold no token
//   kCut      some are cut to their tokens
// (the values are those of psa_grid_kind)
enum Grid { kWhole, kPadded, kCut };
// They are edge blocks, the last ones along an axis.  A class has a bit for each axis on which they are the last (1: t, 2: h, 4: w);
// class 0 is an ordinary block.  A padded grid tells only blocks of fewer slabs apart, the last ones along the axis on which slabs stack.
// Key slabs follow a pattern, that of the ordinary blocks or, where there are none, of the most frequent class: main_slabs slabs
// per block, of 128 keys and the last one of main_last.  The slabs of blocks that do not follow it come behind, 128 keys each.
// In a cut grid an edge block is the part that holds its tokens: `rows` of them, in the order t, h, w of frames of lines of 1 << lw,
// padded as far as loading by TMA boxes asks for.  What tokens do not fill is zeros, with validity bits of 0.
struct alignas(8) EdgeBox {   // a box of a slab: its map, first row, and first token relative to the block's
  uint8_t map, row8;        // (row / 8)
  uint16_t t, h, w;         // t == kZeros: a box of zeros
};
constexpr int kMaxEdgeBoxes = 8;
constexpr uint16_t kZeros = 0xffff;
struct EdgeClass {
  uint16_t rows, frame;     // of a block; of a frame
  uint16_t step;            // rows of a slab that is not the last one
  uint8_t lw;               // log2 of the line length
  uint8_t n_slabs;          // slabs of a block
  alignas(4) uint8_t first_box[4];   // boxes of slab s: first_box[s] .. first_box[s + 1] - 1
  uint8_t together;         // blocks that share one slab of keys (1 unless they have at most 64 rows): of box[0] each, then box[1]
  uint8_t n_boxes;
  uint8_t in_pattern;
  EdgeBox box[kMaxEdgeBoxes];
  uint32_t valid[3][4];     // the slabs' rows with tokens, bit r % 32 of word r / 32; of `together` blocks
};

// Problem geometry handed to every kernel by value.
struct Geom {
  int T, H, W;             // real token grid
  int bt, bh, bw;          // mask block (PSABlock) extents in tokens
  int Tp, Hp, Wp, Sp, NB;  // block grid after 3D-padding; Sp = Hp*Wp, NB = Tp*Sp
  int ct, ch, cw;          // 128-token slab = one TMA box (ct*ch*cw == 128)
  int pos_ws, pos_ts;      // log2(cw) and log2(cw * ch): position c of a slab is w = c % cw, h = (c >> pos_ws) % ch, t = c >> pos_ts
  int n_sub;               // slabs per mask block (1..3)
  int sub_axis;            // axis along which the slabs of a block stack: 0 = t, 1 = h, 2 = w
  int c_last;              // extent of a block's LAST slab along sub_axis (<= the full slab's)
  int n_last;              // tokens of that last slab: 128, 112, 96 or 64
  int edge_axes;           // axes on which the grid has edge blocks (EdgeClass)
  int s_edge;              // spatial block coordinates from here on are the last ones along h
  uint8_t slabs_of[8];     // query slabs of a block by class
  int main_slabs, main_last;   // the pattern of key slabs
  int n_heads;
  int items_per_block;     // work items per query block = ceil(n_sub / 2); of an edge block by its n_slabs
  float scale_log2;        // softmax scale times log2(e)
  long long L;             // T*H*W
  // joint video + text sequences: n_text text tokens follow the L video tokens of every head
  int n_text;              // 0: video only
  int n_ts;                // text slabs of 128 tokens = ceil(n_text / 128)
  int n_titems;            // work items of the text queries per head = ceil(n_ts / 2)
  int items_per_head;      // of all blocks, and n_titems
  long long Lt;            // L + n_text: tokens per head, row length of lse
};

struct HeadParamsArray {
  psa_head_params p[kMaxHeads];
};

// Arguments of the planning kernel: the heads' parameters and each head's place in the work order.
struct PlanParams {
  psa_head_params p[kMaxHeads];
  uint8_t place[kMaxHeads];
};

// One unit of work of the attention kernel: up to two query slabs of one query block.
// x = head, y = query block id, z = number of attended key blocks,
// w = first slab index | (number of slabs << 16) | (split-KV mode << 24) | (text-query item << 25)
// (inside a CTA of a cluster that shares one item: its share of the blocks, bit 26 of w = no text keys; inside a CTA, for grids
// with edge blocks: z = attended blocks that follow the pattern, x = head | (slabs of the others' keys << 8)).
// Key slabs come in this order: those of the blocks that follow the pattern, of the other edge blocks by class, of the text.
typedef int4 WorkItem;

// [0]: box of a full 128-token slab, [1]: of a block's last slab, [2]: of a text slab, [3] on: those of edge blocks
constexpr int kMaxMaps = 20;
struct TensorMaps {
  CUtensorMap q[3], k[3], v[3], o[3];
};
struct TensorMapsCut {
  CUtensorMap q[kMaxMaps], k[kMaxMaps], v[kMaxMaps], o[kMaxMaps];
};
// How an attention launch hands out its work items (see attn_fwd_kernel); the values are those of psa_launch_mode.  (kTicketEdge
// is only reported; the kernel is that of kTicket.)
enum Mode { kTicket, kDirect, kShared, kSharedDirect, kTicketEdge, kTicketShort };

// Arguments of one attention launch; lse and out start at the launch's first head.
struct AttnParams {
  Geom g;
  const WorkItem* items;
  const psa_head_params* hp_dev;
  int* ws_header;
  float* lse;
  int n_items;
  int call_id;      // id of the API call, for the status words
  int shared_qkv;   // 1: every head reads head 0 of q, k, v (candidate masks of one head, PSA-Search)
  void* out;        // for rows that are stored without TMA; strides in elements
  long long out_head, out_token;
};

// The same of a launch on a cut grid.
struct AttnParamsCut : AttnParams {
  EdgeClass cls[8];
  int planned;                 // 1: every class follows the pattern, so that an item's number of key blocks is the planned one
  int n_classes;               // classes that the grid has, those of the pattern first
  uint8_t order[8];
};

// Layout of the per-device workspace (all int32 words).
constexpr int kWsStatus = 0;     // first device-side error of call kWsCallId
constexpr int kWsDetail = 1;     // diagnostic of that error
constexpr int kWsCallId = 3;     // API call that reported an error last (0 = none yet)
constexpr int kWsCounter = 2;    // dynamic scheduler ticket
constexpr int kWsHeaderWords = 16;

// One axis condition of the stripe mask (Algorithm 1): delta is key minus query
// coordinate in blocks; stride 0 encodes an infinite stride.
__host__ __device__ __forceinline__ bool axis_attends(int delta, int width, int offset, int stride) {
  int x = delta - offset;
  x = x < 0 ? -x : x;
  if (stride != 0) x = x % stride;
  return x <= width - 1;
}

// Walks one axis' differences -(n - 1) .. n - 1 in order with the distance's remainder carried along (one division
// per axis instead of one per difference: the host evaluates some 70 differences per head, at 6 ns a division) and
// calls f(index, difference) for every attended one.
template <class F>
inline void for_attended(int n, int width, int offset, int stride, F f) {
  int d = -(n - 1);
  long long x = (long long)d - offset;            // key minus query minus offset
  const long long dist = x < 0 ? -x : x;
  long long r = stride ? dist % stride : dist;    // remainder of the distance
  for (int i = 0; i < 2 * n - 1; ++i, ++d, ++x) {
    if (r <= width - 1) f(i, d);
    if (x < 0) {                                  // the distance falls by one
      if (stride && r == 0) r = stride;
      --r;
    } else {
      ++r;
      if (stride && r == stride) r = 0;
    }
  }
}

// One axis' attended differences as a bit set, bit d + n - 1 for difference d, with the number of attended
// coordinate pairs (n <= 64).
struct AxisSet {
  unsigned long long lo, hi;
  int pairs;
};
inline unsigned long long reverse_bits(unsigned long long x) {
  x = (x >> 1 & 0x5555555555555555ull) | (x & 0x5555555555555555ull) << 1;
  x = (x >> 2 & 0x3333333333333333ull) | (x & 0x3333333333333333ull) << 2;
  x = (x >> 4 & 0x0f0f0f0f0f0f0f0full) | (x & 0x0f0f0f0f0f0f0f0full) << 4;
  return __builtin_bswap64(x);
}
// Sum of (i + 1) over the set bits i of x.
inline int weighted_bits(unsigned long long x) {
  struct Table {
    uint8_t weight[256], count[256];
    Table() {
      for (int v = 0; v < 256; ++v) {
        weight[v] = count[v] = 0;
        for (int i = 0; i < 8; ++i)
          if (v >> i & 1) { weight[v] = (uint8_t)(weight[v] + i + 1); ++count[v]; }
      }
    }
  };
  static const Table t;
  int sum = 0;
  for (int base = 0; x; base += 8, x >>= 8) sum += t.weight[x & 255] + base * t.count[x & 255];
  return sum;
}
// (About 25 ns an axis up to 32 coordinates and 35 up to 64, where the walk takes 80 and 160: psa_mask_build evaluates 80
// axes for a 40-head layer in front of a 5.7 us kernel, and a call of 40 heads of 8 x 60 blocks took the host 14.8 us
// instead of 9.8 with the walk beyond 32.)
inline AxisSet axis_set(int n, int width, int offset, int stride) {
  AxisSet s = {0, 0, 0};
  const long long center = (long long)(n - 1) + offset;   // index of the difference at distance 0 from the offset
  if (n <= 32 && center >= 0 && center <= 63) {
    // attended distances 0 .. 63: `width` ones at every multiple of the stride, by doubling; to the right of the
    // center, and mirrored to its left
    unsigned long long dist = width >= 64 || (stride > 0 && width >= stride) ? ~0ull : ((1ull << width) - 1);
    if (stride > 0)
      for (long long w = stride; w < 64; w <<= 1) dist |= dist << w;
    s.lo = (dist << center | reverse_bits(dist) >> (63 - center)) & (~0ull >> (65 - 2 * n));
  } else if (n <= 64 && center >= 0 && center <= 127) {   // the same in 128 bits
    using u128 = unsigned __int128;
    u128 dist = width >= 128 || (stride > 0 && width >= stride) ? ~(u128)0 : (((u128)1 << width) - 1);
    if (stride > 0)
      for (long long w = stride; w < 128; w <<= 1) dist |= dist << w;
    const u128 mirrored = (u128)reverse_bits((unsigned long long)dist) << 64 | reverse_bits((unsigned long long)(dist >> 64));
    const u128 set = (dist << center | mirrored >> (127 - center)) & (~(u128)0 >> (129 - 2 * n));
    s.lo = (unsigned long long)set;
    s.hi = (unsigned long long)(set >> 64);
  } else {
    for_attended(n, width, offset, stride, [&](int i, int) { (i < 64 ? s.lo : s.hi) |= 1ull << (i & 63); });
  }
  // difference d occurs n - |d| times: weights 1 .. n up to the middle bit n - 1, mirrored beyond it
  const unsigned long long low = n == 64 ? s.lo : s.lo & ((1ull << n) - 1);
  const unsigned long long high = n == 64 ? s.hi : s.lo >> n | (n > 0 && s.hi ? s.hi << (64 - n) : 0ull);   // n - 1 bits
  s.pairs = weighted_bits(low) + (n > 1 ? weighted_bits(reverse_bits(high) >> (65 - n)) : 0);
  return s;
}

}  // namespace psa
