// psa_mask_build: block mask and GetKVBlocks index lists from the stripe parameters
// (Algorithm 1 evaluated on block coordinates; Algorithm 2, producer side).
// Integer work only.  Two kernels: one for block grids of at most 64 temporal x 32 spatial
// coordinates (mask_build_small_kernel, further down: one thread block per head and temporal
// query coordinate), and the general one described here.
//
// The two conditions of Algorithm 1 depend only on coordinate differences, so each block of threads first tabulates, for
// its head, "does difference d attend" for every temporal and every spatial difference: bit d + n - 1 of a bit array per
// axis, and the sorted list of the attended bits' positions.  The key coordinates that a query coordinate x attends are a
// window of n bits and a contiguous piece of the list.  The block mask of a head is the Kronecker product of its two axis
// masks, so the count of row (t', s') is cntT(t') * cntS(s') and its offset in the column list has a closed form.
#include "psa_common.cuh"

namespace psa {

struct HeadBases {
  int base[kMaxHeads];  // number of attended block pairs of all earlier heads
};

// Shared-memory tables of one axis with n coordinates: bits (a word of zeros behind them, so that a window may be read from
// any bit), the number of bits set before each word, the positions of the set bits, and pre[x] = attended pairs of the
// query coordinates before x.  At most 8.5 bytes a coordinate.
struct Axis {
  int n, words;
  uint32_t* bits;
  int* before;
  int* pre;
  uint16_t* list;

  // attended differences below bit i
  __device__ __forceinline__ int rank(int i) const { return before[i >> 5] + __popc(bits[i >> 5] & ((1u << (i & 31)) - 1u)); }
  __device__ __forceinline__ int first(int x) const { return rank(n - 1 - x); }   // of x's piece of the list
  __device__ __forceinline__ int count(int x) const { return rank(2 * n - 1 - x) - rank(n - 1 - x); }
  __device__ __forceinline__ int pairs() const { return pre[n - 1] + count(n - 1); }
  // 32 bits from bit i on
  __device__ __forceinline__ uint32_t window(int i) const { return __funnelshift_r(bits[i >> 5], bits[(i >> 5) + 1], i & 31); }
};

// (one more than the sets themselves take: see bits)
__host__ __device__ inline int table_words(int n) { return (2 * n - 1 + 31) / 32 + 1; }
__host__ __device__ inline size_t axis_bytes(int n) {
  return (8 * (size_t)table_words(n) + 4 * (size_t)n + 2 * (size_t)(2 * n - 1) + 3) & ~size_t(3);
}
__device__ __forceinline__ Axis carve_axis(uint8_t* smem, int n) {
  Axis a;
  a.n = n;
  a.words = table_words(n);
  a.bits = reinterpret_cast<uint32_t*>(smem);
  a.before = reinterpret_cast<int*>(a.bits + a.words);
  a.pre = a.before + a.words;
  a.list = reinterpret_cast<uint16_t*>(a.pre + n);
  return a;
}

__device__ __forceinline__ void axis_bits(const Axis& a, int warp, int nwarps, int lane, int width, int offset, int stride) {
  for (int w = warp; w < a.words; w += nwarps) {
    const int i = w * 32 + lane;
    const unsigned m = __ballot_sync(0xffffffffu, i < 2 * a.n - 1 && axis_attends(i - (a.n - 1), width, offset, stride));
    if (lane == 0) a.bits[w] = m;
  }
}
// Exclusive prefix sums of value(0 .. n - 1) by one warp.
template <class F>
__device__ __forceinline__ void warp_prefix(int* out, int n, int lane, F value) {
  int carry = 0;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane, v = i < n ? value(i) : 0;
    int s = v;
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, s, off);
      if (lane >= off) s += o;
    }
    if (i < n) out[i] = carry + s - v;
    carry += __shfl_sync(0xffffffffu, s, 31);
  }
}
__device__ __forceinline__ void axis_list(const Axis& a, int first, int step) {
  for (int i = first; i < 2 * a.n - 1; i += step)
    if (a.bits[i >> 5] >> (i & 31) & 1u) a.list[a.rank(i)] = (uint16_t)i;
}

// y / n and the remainder, for quotients below 2^20 (the product is then off by less than one)
__device__ __forceinline__ int div_near(int y, int n, float inv, int& rem) {
  int q = (int)((float)y * inv);
  rem = y - q * n;
  if (rem < 0) { --q; rem += n; }
  else if (rem >= n) { ++q; rem -= n; }
  return q;
}

// One block per (group of consecutive rows, head); a row is a query block.  The rows' mask bytes are one region, written in
// aligned 32-byte pieces (the region's ends bytewise): a piece is built as 32 bits, a window of the spatial bits for every
// attended temporal coordinate it touches.  A warp then writes the list of a row, entry e of it being the (e / cntS)-th
// attended temporal and the (e mod cntS)-th attended spatial coordinate.
// Bound by latencies (the tables' barriers, then few independent stores per warp) on small problems and by the list's 4-byte
// stores on large ones.  Microseconds, calls back to back, against one row per warp with a byte and a ballot per key block:
// 6 heads of 32 x 36 blocks 22.2 -> 12.4, 20 such heads 57.5 -> 28.6, 6 of 21 x 60 26.8 -> 12.4, 40 of 8 x 60 28.8 -> 16.5,
// 10 of 11 x 56 16.5 -> 9.2.
__global__ void __launch_bounds__(256)
mask_build_kernel(const HeadParamsArray hp, const HeadBases hb, const Geom g, int n_heads_here, int rows_per_block,
                  uint8_t* __restrict__ block_mask, int* __restrict__ row_ptr, int* __restrict__ col_idx,
                  int total_nnz) {
  extern __shared__ __align__(16) uint8_t smem_tab[];
  const int h = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int Tp = g.Tp, Sp = g.Sp, NB = g.NB;
  const Axis aS = carve_axis(smem_tab, Sp), aT = carve_axis(smem_tab + axis_bytes(Sp), Tp);
  const psa_head_params& p = hp.p[h];
  axis_bits(aS, warp, nwarps, lane, p.Sw, p.So, p.Ss);
  axis_bits(aT, nwarps - 1 - warp, nwarps, lane, p.Tw, p.To, p.Ts);
  __syncthreads();
  if (warp == 0) warp_prefix(aS.before, aS.words, lane, [&](int w) { return __popc(aS.bits[w]); });
  if (warp == 1) warp_prefix(aT.before, aT.words, lane, [&](int w) { return __popc(aT.bits[w]); });
  __syncthreads();
  if (warp == 0) warp_prefix(aS.pre, Sp, lane, [&](int x) { return aS.count(x); });
  else if (warp == 1) warp_prefix(aT.pre, Tp, lane, [&](int x) { return aT.count(x); });
  else {
    axis_list(aS, threadIdx.x - 64, blockDim.x - 64);
    axis_list(aT, threadIdx.x - 64, blockDim.x - 64);
  }
  __syncthreads();
  const float inv_nb = 1.f / (float)NB, inv_sp = 1.f / (float)Sp;
  const int q0 = blockIdx.x * rows_per_block;
  const int q1 = min(NB, q0 + rows_per_block);

  if (block_mask) {
    const long long x0 = ((long long)h * NB + q0) * NB, x1 = ((long long)h * NB + q1) * NB;
    for (long long x = (x0 & ~31ll) + threadIdx.x * 32ll; x < x1; x += blockDim.x * 32ll) {
      const int from = x < x0 ? (int)(x0 - x) : 0, to = x1 - x < 32 ? (int)(x1 - x) : 32;
      int sk, sq;
      int tk, tq, rem;
      const int row = q0 + div_near((int)(x + from - x0), NB, inv_nb, rem);
      tk = div_near(rem, Sp, inv_sp, sk);
      tq = div_near(row, Sp, inv_sp, sq);
      uint32_t m = 0;
      for (int n = from; n < to;) {
        const int len = min(to - n, Sp - sk), dt = tk - tq + Tp - 1;
        if (aT.bits[dt >> 5] >> (dt & 31) & 1u) m |= (aS.window(Sp - 1 - sq + sk) & (0xffffffffu >> (32 - len))) << n;
        n += len;
        sk += len;
        if (sk == Sp) {
          sk = 0;
          if (++tk == Tp) {
            tk = 0;
            if (++sq == Sp) { sq = 0; ++tq; }
          }
        }
      }
      uint8_t* dst = block_mask + x;
      if (to - from == 32) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = (m >> (4 * i) & 15u) * 0x00204081u & 0x01010101u;
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
      } else {
        for (int n = from; n < to; ++n) dst[n] = (uint8_t)(m >> n & 1u);
      }
    }
  }
  if (row_ptr == nullptr) return;   // (no lists without it)
  const int pairsS = aS.pairs();
  for (int qb = q0 + warp; qb < q1; qb += nwarps) {
    int sq;
    const int tq = div_near(qb, Sp, inv_sp, sq);
    const int cT = aT.count(tq), cS = aS.count(sq);
    const int pos = hb.base[h] + aT.pre[tq] * pairsS + cT * aS.pre[sq];
    if (lane == 0) row_ptr[(long long)h * NB + qb] = pos;
    if (col_idx == nullptr || cT * cS == 0) continue;
    const uint16_t* lT = aT.list + aT.first(tq);
    const uint16_t* lS = aS.list + aS.first(sq);
    const int shift = (tq - (Tp - 1)) * Sp + sq - (Sp - 1);
    int s, t = div_near(lane, cS, 1.f / (float)cS, s);
    int ds, dt = div_near(32, cS, 1.f / (float)cS, ds);
#pragma unroll 4
    for (int e = lane; e < cT * cS; e += 32) {
      col_idx[pos + e] = (int)lT[t] * Sp + (int)lS[s] + shift;
      t += dt;
      s += ds;
      if (s >= cS) { s -= cS; ++t; }
    }
  }
  if (blockIdx.x == 0 && h == n_heads_here - 1 && threadIdx.x == 0) row_ptr[(long long)n_heads_here * NB] = total_nnz;
}

// Fast path for block grids with at most 64 temporal and 32 spatial block coordinates (all the
// paper's shapes): no block-wide table building.  The host evaluates the two axis conditions of
// Algorithm 1 once per head for every coordinate difference and hands the kernel two bit sets
// per head (127 and 63 bits; bit d + n - 1 of an axis' set = "difference d attends"), so the key
// coordinates a query coordinate x attends are one shift away: (set >> (n - 1 - x)) & ((1 << n) - 1).
//
// One thread block per (head, temporal query coordinate tq): its S' rows are consecutive, so
// their mask bytes are one contiguous region and their column lists one contiguous range.
//   * Warp 0 derives the row counts (popcounts), their prefix sums (one warp scan), the block's
//     first list offset, "the r-th attended temporal coordinate" of tq, and writes the S' row
//     offsets.
//   * Meanwhile all threads write the mask region 32 bytes at a time: a thread assembles 32
//     consecutive mask bits (the row of the Kronecker product is the spatial bit pattern repeated
//     under the temporal bits), spreads them to bytes with four multiplies per 16 and stores two
//     16-byte words.
//   * After one barrier the rows of the block are taken by sub-groups of 8, 16 or 32 lanes: entry e
//     of a row's list is (the (e / cS)-th attended temporal coordinate, the (e % cS)-th attended
//     spatial one); the division is a multiply and a shift (e < 2048, cS <= 32).
struct HeadSets {
  unsigned long long setT[kMaxHeads], setT_hi[kMaxHeads], setS[kMaxHeads];   // temporal set: 127 bits
  int base[kMaxHeads];  // number of attended block pairs of all earlier heads
};

// Constants of the closed-form 32-bit mask window (see the kernel).  groups = temporal groups a
// window can touch; mul / keep spread `groups` consecutive temporal bits to a spacing of S' bits
// (bit i lands on i * S'; all partial products fall on distinct bits while groups <= S' - 1).
struct WindowConsts {
  unsigned long long mul, keep;
  int groups, enabled;
};

// n / d for n < 2^16, d <= 2^11 with m = ceil(2^40 / d): exact (n * (m * d - 2^40) < 2^40)
__device__ __forceinline__ int div_magic(int n, unsigned long long m) { return (int)(((unsigned long long)(unsigned)n * m) >> 40); }

// (Six resident blocks per SM -- 40 registers -- let the 840 blocks of the Wan 14B shape start in one wave.)
__global__ void __launch_bounds__(256, 6)
mask_build_small_kernel(const HeadSets hs, const Geom g, int n_heads_here, unsigned long long magic_nb,
                        unsigned long long magic_sp, const WindowConsts wc, uint8_t* __restrict__ block_mask, int* __restrict__ row_ptr,
                        int* __restrict__ col_idx, int total_nnz) {
  const int h = blockIdx.y, tq = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int Tp = g.Tp, Sp = g.Sp, NB = g.NB;
  __shared__ int s_preS[32], s_cS[32], s_tsel[64], s_hdr[2];
  __shared__ int s_strip[8 * 4 * 32];      // per warp and sub-group: the r-th attended spatial coordinate of its row
  __shared__ unsigned s_inv[33];           // ceil(2^20 / c): e / c = (e * inv) >> 20 for e < 2048, c <= 32
  const unsigned long long setT = hs.setT[h], setT_hi = hs.setT_hi[h], setS = hs.setS[h];
  const unsigned long long maskT = Tp == 64 ? ~0ull : ((1ull << Tp) - 1ull);
  const unsigned maskS = Sp == 32 ? 0xffffffffu : ((1u << Sp) - 1u);
  // temporal key coordinates attended by query coordinate x (up to 64 of them: a 64-bit mask)
  auto rowT = [&](int x) -> unsigned long long {
    const int sh = Tp - 1 - x;   // 0 .. 63
    const unsigned long long lo = setT >> sh, hi = sh ? (setT_hi << (64 - sh)) : 0ull;
    return (lo | hi) & maskT;
  };
  auto rowS = [&](int x) -> unsigned { return (unsigned)(setS >> (Sp - 1 - x)) & maskS; };
  const unsigned long long mT = rowT(tq);
  const unsigned lane_lt = (1u << lane) - 1u;

  if (threadIdx.x >= 64 && threadIdx.x <= 96) {
    const unsigned c = threadIdx.x - 64;
    s_inv[c] = c ? ((1u << 20) + c - 1u) / c : 0u;
  }
  if (warp == 0) {
    // lane x holds the counts of coordinates x (and x + 32 on the temporal axis) and the exclusive
    // prefixes of the counts before them
    const int cntT0 = lane < Tp ? __popcll(rowT(lane)) : 0, cntT1 = lane + 32 < Tp ? __popcll(rowT(lane + 32)) : 0;
    const int cntS = lane < Sp ? __popc(rowS(lane)) : 0;
    int incT0 = cntT0, incT1 = cntT1, incS = cntS;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, incT0, off), c = __shfl_up_sync(0xffffffffu, incT1, off);
      const int b = __shfl_up_sync(0xffffffffu, incS, off);
      if (lane >= off) { incT0 += a; incT1 += c; incS += b; }
    }
    const int sumT0 = __shfl_sync(0xffffffffu, incT0, 31);
    const int preT0 = incT0 - cntT0, preT1 = sumT0 + incT1 - cntT1, preS = incS - cntS;
    const int sumS = __shfl_sync(0xffffffffu, incS, 31);
    const int cT = __popcll(mT);
    const int pT = __shfl_sync(0xffffffffu, tq < 32 ? preT0 : preT1, tq & 31);
    const int pos0 = hs.base[h] + pT * sumS;
    s_preS[lane] = preS;
    s_cS[lane] = cntS;
    if ((mT >> lane) & 1ull) s_tsel[__popcll(mT & (unsigned long long)lane_lt)] = lane;
    if ((mT >> (lane + 32)) & 1ull) s_tsel[__popcll(mT & ((1ull << (lane + 32)) - 1ull))] = lane + 32;
    if (lane == 0) { s_hdr[0] = cT; s_hdr[1] = pos0; }
    if (row_ptr) {
      if (lane < Sp) row_ptr[(long long)h * NB + tq * Sp + lane] = pos0 + cT * preS;
      if (tq == 0 && h == n_heads_here - 1 && lane == 0) row_ptr[(long long)n_heads_here * NB] = total_nnz;
    }
  }

  if (block_mask) {
    // The block writes the 32-byte aligned chunks that START inside its rows' region; its last chunk
    // runs on into the next region (next tq, or the next head), whose own first chunk starts at the
    // next aligned address.  Only the very first bytes of the whole mask (when its base is not
    // aligned) and a clipped chunk at its very end are written bytewise.
    const int len = Sp * NB;                                 // bytes of this block's rows
    uint8_t* p0 = block_mask + ((long long)h * NB + (long long)tq * Sp) * NB;
    const int lead = (int)((32u - (unsigned)(reinterpret_cast<uintptr_t>(p0) & 31u)) & 31u);   // first aligned offset
    // up to `limit` mask bytes from region offset r on (bit i of the result = byte r + i); *got = bytes that exist
    auto gen = [&](int r, int limit, int* got) -> unsigned {
      int hh = h, tq_ = tq;
      int sq = div_magic(r, magic_nb), kb = r - sq * NB;
      int tk = div_magic(kb, magic_sp), sk = kb - tk * Sp;
      unsigned long long sT = setT, sT_hi = setT_hi, sS = setS, mT_ = mT;
      unsigned mS = (unsigned)(sS >> (Sp - 1 - sq)) & maskS;
      unsigned bits = 0u;
      int n = 0;
      while (n < limit && hh < n_heads_here) {
        const unsigned grp = ((mT_ >> tk) & 1ull) ? (mS >> sk) : 0u;   // Sp - sk key blocks of temporal group tk
        int take = Sp - sk;
        if (take > limit - n) take = limit - n;
        bits |= (take >= 32 ? grp : (grp & ((1u << take) - 1u))) << n;
        n += take;
        sk += take;
        if (sk == Sp) {
          sk = 0;
          if (++tk == Tp) {
            tk = 0;
            if (++sq == Sp) {   // rare: the chunk runs on into the next region
              sq = 0;
              if (++tq_ == Tp) {
                tq_ = 0;
                if (++hh < n_heads_here) { sT = hs.setT[hh]; sT_hi = hs.setT_hi[hh]; sS = hs.setS[hh]; }
              }
              const int sh = Tp - 1 - tq_;
              mT_ = ((sT >> sh) | (sh ? (sT_hi << (64 - sh)) : 0ull)) & maskT;
            }
            mS = (unsigned)(sS >> (Sp - 1 - sq)) & maskS;
          }
        }
      }
      *got = n;
      return bits;
    };
    const int nchunks = len > lead ? (len - lead + 31) >> 5 : 0;
    // Closed form of a window that stays inside the block's rows: the temporal bits tk, tk + 1, ...
    // are spread to a spacing of S' bits by one multiplication, widened to runs of S' ones
    // ((x << S') - x), and combined with the spatial pattern repeated with period S'; the window
    // starts sk bits in.  A window that leaves the block's rows takes the general loop above.
    auto periodic = [&](unsigned m) -> unsigned long long {
      unsigned long long r = m;
      for (int wd = Sp; wd < 64; wd <<= 1) r |= r << wd;
      return r;
    };
    auto runs = [&](int tk) -> unsigned long long {
      const unsigned long long tw = (mT >> tk) & ((1ull << wc.groups) - 1ull);
      const unsigned long long spread = (tw * wc.mul) & wc.keep;
      return (spread << Sp) - spread;
    };
    const unsigned long long runs0 = runs(0);
    for (int c = threadIdx.x; c < nchunks; c += blockDim.x) {
      const int r = lead + 32 * c;
      int n = 32;
      unsigned bits;
      const int sq = div_magic(r, magic_nb), kb = r - sq * NB;
      if (wc.enabled && (kb + 32 <= NB || sq + 1 < Sp)) {
        const int tk = div_magic(kb, magic_sp), sk = kb - tk * Sp;
        bits = (unsigned)((runs(tk) & periodic(rowS(sq))) >> sk);
        if (kb + 32 > NB) bits |= (unsigned)(runs0 & periodic(rowS(sq + 1))) << (NB - kb);   // on into the next row
      } else {
        bits = gen(r, 32, &n);
      }
      if (n == 32) {
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = (((bits >> (4 * k)) & 15u) * 0x00204081u) & 0x01010101u;
        uint4* dst = reinterpret_cast<uint4*>(p0 + r);
        dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
        dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
      } else {
        for (int i = 0; i < n; ++i) p0[r + i] = (uint8_t)((bits >> i) & 1u);   // the end of the whole mask
      }
    }
    if (h == 0 && tq == 0 && lead > 0 && threadIdx.x == blockDim.x - 1) {   // unaligned start of the whole mask
      int n;
      const unsigned bits = gen(0, lead, &n);
      for (int i = 0; i < n; ++i) p0[i] = (uint8_t)((bits >> i) & 1u);
    }
  }
  __syncthreads();

  if (col_idx) {
    // Sub-groups of 8, 16 or 32 lanes take one row each, so that the S' rows of the block are
    // all in flight at once (S' <= 8, 16, 32 with eight warps).
    const int cT = s_hdr[0], pos0 = s_hdr[1];
    const int lg = Sp > 16 ? 2 : (Sp > 8 ? 1 : 0);          // log2 of the sub-groups per warp
    const int W = 32 >> lg, grp = lane >> (5 - lg), sl = lane & (W - 1);
    int* strip = s_strip + ((warp << 2) + grp) * 32;         // the r-th attended spatial coordinate of the row
    for (int sq0 = warp << lg; sq0 < Sp && cT > 0; sq0 += nwarps << lg) {
      const int sq = sq0 + grp;
      const bool act = sq < Sp;
      const int cS = act ? s_cS[sq] : 0;
      const int pos = pos0 + cT * (act ? s_preS[sq] : 0);
      const unsigned mS = act ? rowS(sq) : 0u;
      for (int b = sl; b < 32; b += W)
        if ((mS >> b) & 1u) strip[__popc(mS & ((1u << b) - 1u))] = b;
      __syncwarp();
      const int count = cT * cS;
      const unsigned inv = s_inv[cS];
      for (int e = sl; e < count; e += W) {
        const int it = (int)(((unsigned)e * inv) >> 20), is = e - it * cS;
        col_idx[pos + e] = s_tsel[it] * Sp + strip[is];
      }
      __syncwarp();
    }
  }
}

bool mask_build_small(const Geom& g) { return g.Tp <= 64 && g.Sp <= 32; }

// sets: the two axis sets of every head (temporal, spatial), when mask_build_small(g).
cudaError_t launch_mask_build(const HeadParamsArray& hp, const AxisSet* sets, const int* head_bases, const Geom& g, int n_heads_here,
                              uint8_t* block_mask, int* row_ptr, int* col_idx, int total_nnz_through_chunk,
                              int n_sms, cudaStream_t stream, int* launches) {
  if (mask_build_small(g)) {
    HeadSets hs;   // entries beyond n_heads_here are never read
    for (int h = 0; h < n_heads_here; ++h) {
      hs.setT[h] = sets[2 * h].lo;
      hs.setT_hi[h] = sets[2 * h].hi;
      hs.setS[h] = sets[2 * h + 1].lo;
      hs.base[h] = head_bases[h];
    }
    const unsigned long long two40 = 1ull << 40;
    const unsigned long long magic_nb = (two40 + (unsigned long long)g.NB - 1ull) / (unsigned long long)g.NB;
    const unsigned long long magic_sp = (two40 + (unsigned long long)g.Sp - 1ull) / (unsigned long long)g.Sp;
    // the closed-form window needs its partial products on distinct bits and at most one row end per window
    WindowConsts wc;
    wc.groups = (g.Sp - 1 + 31) / g.Sp + 1;
    wc.enabled = (wc.groups <= g.Sp - 1 && g.NB >= 32) ? 1 : 0;
    wc.mul = 0;
    wc.keep = 0;
    if (wc.enabled)
      for (int i = 0; i < wc.groups; ++i) {
        wc.mul |= 1ull << (i * (g.Sp - 1));
        if (i * g.Sp < 64) wc.keep |= 1ull << (i * g.Sp);
      }
    dim3 grid(g.Tp, n_heads_here);   // one block per (head, temporal query coordinate)
    mask_build_small_kernel<<<grid, 256, 0, stream>>>(
        hs, g, n_heads_here, magic_nb, magic_sp, wc, block_mask, row_ptr, col_idx, total_nnz_through_chunk);
    ++*launches;
    return cudaGetLastError();
  }
  HeadBases hb;
  for (int h = 0; h < kMaxHeads; ++h) hb.base[h] = h < n_heads_here ? head_bases[h] : 0;
  const size_t smem = axis_bytes(g.Sp) + axis_bytes(g.Tp);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(mask_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  // four blocks per SM, all at once, with at least 8 rows (one per warp) each: 6 heads of 21 x 60 blocks take 12.4 us (14.8
  // with two, 14.4 with three or five), 20 of 32 x 36 take 28.6 (32.9, 28.4, 26.7)
  int blocks_per_head = 4 * n_sms / n_heads_here;
  if (blocks_per_head < 1) blocks_per_head = 1;
  int rows_per_block = (g.NB + blocks_per_head - 1) / blocks_per_head;
  if (rows_per_block < 8) rows_per_block = 8;
  blocks_per_head = (g.NB + rows_per_block - 1) / rows_per_block;
  dim3 grid(blocks_per_head, n_heads_here);
  mask_build_kernel<<<grid, 256, smem, stream>>>(hp, hb, g, n_heads_here, rows_per_block, block_mask, row_ptr, col_idx,
                                                 total_nnz_through_chunk);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace psa
