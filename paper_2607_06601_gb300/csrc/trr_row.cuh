#pragma once
// trr_row.cuh - the attention kernels: mode-routed split-K decode attention over the
// mixed-precision paged cache (Sec. 3.2(A), Eq. 2; Sec. 3.8; Sec. 7).
//
// A work unit is a split of a query for one query head (MHA, per-head modes, small calls of wide
// groups) or for one KV head and heads of its query group, and belongs to one warp from its plan to
// its row: the warp plans the unit (plan_pages), streams its pages' KV slices through a ring of
// shared memory of its own with 1-D bulk copies (one per page as a rule, cp.async.bulk +
// mbarrier), and computes on them.  Nothing but the call's start and end synchronises warps.
// The kernels are bound by instructions issued and by the latency of a unit's chain (plan,
// copies, tiles, merge), not by memory: batch 256 of the sweep shape streams at 3.9 TB/s, at 5.9
// with the tile arithmetic left out.  (A step of 3 such layers 762 us; 828 with a producer warp that
// fed four consumer warps through one ring and binary32 arithmetic on the CUDA cores.)
//
// Two CTAs of eight warps fill an SM; while some of the places are free or a CTA has ended,
// the next layer's kernel is resident, so that its plans and its first page copies come before
// its wait on this kernel.
//
// One query head per warp: the arithmetic runs on the tensor cores (mma.sync m16n8k16, f32
// accumulation) though only one query head shares a key, because the codes then need one mask per
// two elements (a pair of codes in the halves of a word, read as f16 subnormals) in place of one
// per element, and the multiply-adds come free:
//   q.k   A = 16 keys' codes, B = the query row, its column n holding quantiser group
//         n % NG (zero outside it); each lane then takes one key of a tile of 32 and adds
//         up s * (group sum) + z * (group's query sum) in binary32.
//   P.V   A = V^T codes paired along keys, B = p * s of the tile's keys, exchanged through
//         shared memory: column (group, hi | lo), the weight split into two f16 parts
//         (22 bits and the sign, as many as exp2's approximation has; scaled by a power of
//         two per group that follows the weights, far from f16's limits).
//         Width 16 uses m16n8k8 with tf32 operands (bf16 values are exact in tf32), its
//         weights split the same way.
// The running maximum is the warp's, raised only when a score exceeds it by 2^8.
#include <type_traits>

#include "trr_attn.cuh"

namespace trr {

// What a work unit is: a query head; a query head of a cache with per-head modes; a KV head and its
// query group (g * d/G <= 8); a KV head and up to 8 / (d/G) heads of a wider query group.
enum Kind { kRow, kHeads, kGroup, kWide };

constexpr int kRowWarps = 8;   // warps per CTA
constexpr int kRowSlots = 8;   // tiles a warp may have in flight
constexpr int kRowCtasPerSm = 2;
// A grid leaves num_sms / kRowSpare places of the chip free: the next layer's kernel then
// starts, and plans, while the last CTAs of this one still run.  (160M, 4 steps 796 us, 799 with a
// full grid; the 1.3B shape 666 and 653, per-head modes 666 and 645.)
constexpr int kRowSpare = 32;
constexpr int kRowSmemLimit = 110 * 1024;
constexpr float kLoScale = 2048.f;  // the low part of a weight is stored times 2^11

constexpr int kRowRed = 8 * kRowWarps * 2 + 4 * 32;  // plan_rows' sums and counts
struct RowSmem {  // byte offsets of one CTA's shared memory
  int full, fac, q, w, pre, qinf, ord, red, ent, flag, ring, total;
  // heads: query heads of a unit (query groups)
  __host__ __device__ RowSmem(int D, int heads, int n, int step, int ring_bytes)
      : full(0),
        fac(full + kRowWarps * kRowSlots * 8),
        q(fac + 16 * (D / 8) * 4),
        w(q + kRowWarps * row_q_bytes(D, heads)),
        pre(w + kRowWarps * row_w_bytes(heads)),
        qinf(pre + align16(4 * (n + 2))),
        ord(qinf + 16 * n),
        red(ord + align16(2 * n)),
        ent(red + kRowRed),
        flag(ent + (step ? align16(4 * step_ints(n)) : 0)),
        ring((flag + 16 + 8 * kRowWarps + 127) & ~127),
        total(ring + kRowWarps * ring_bytes) {}
  // a unit's query rows; one head: the row as the class's operand, as given, its groups' exponents
  __host__ __device__ static constexpr int row_q_bytes(int D, int heads) { return heads > 1 ? heads * D * 2 : 4 * D + 16; }
  // the weights of a tile: 32 rows of 8 f16 (width 16: of 2 tf32; query groups: of 8 bf16,
  // high parts, then low parts)
  __host__ __device__ static constexpr int row_w_bytes(int heads) { return heads > 1 ? 1024 : 512; }
};

// The largest tile in a ring: 16-bit rows (at d 128 sixteen of them) or 32 8-bit ones, with a
// presence mask and positions.
constexpr int row_tile_bytes(int D, int NG) {
  const int wide = (D == 64 ? 32 : 16) * 4 * D, b8 = 32 * (2 * D + 8 * NG);
  return (((wide > b8 ? wide : b8) + 16 + 127) & ~127) + 128;
}

// Rows (work units per query split): full heads, local heads and the others of a query.
struct HeadCounts {
  int full, local, skip;
};
__device__ __forceinline__ HeadCounts head_counts(const AttnKernelArgs& ka, int q) {
  const uint8_t* row = ka.modes + static_cast<int64_t>(q) * ka.a.Hq;
  HeadCounts c{0, 0, 0};
#pragma unroll 1
  for (int h = 0; h < ka.a.Hq; ++h) {
    c.full += row[h] == TRR_MODE_FULL;
    c.local += row[h] == TRR_MODE_LOCAL;
  }
  c.skip = ka.a.Hq - c.full - c.local;
  return c;
}

// x / y for 0 <= x < 2^24, 0 < y < 2^24: the binary32 quotient is within one of it.
__device__ __forceinline__ int div24(int x, int y) {
  const int q = static_cast<int>(__fdividef(static_cast<float>(x), static_cast<float>(y)));
  const int r = x - q * y;
  return r < 0 ? q - 1 : r >= y ? q + 1 : q;
}

// The work units of a call, computed the same way by every CTA.  Queries are taken in the
// order of their units' size (those that read everything, those that read a window, zero
// rows), so that units handed out on demand end with short ones: place k holds query ord[k];
// pre[k] numbers its first unit, pre[n] counts them all, pre[n + 1] is the call's key
// positions per split; qinf[k] = {sequence, position, first key position (per-head modes: of
// a local head), splits of a row (per-head modes: of a full head) | query error << 24 | zero
// row << 28}.  A query has one unit per (row, split); with per-head modes each head its own
// splits (one for a skip head, which writes its zero row).
template <bool HM, bool GQ>
__device__ __forceinline__ void plan_rows(const AttnKernelArgs& ka, int rows, int* pre, int4* qinf, uint16_t* ord, long long* red) {
  const LayerArgs& a = ka.a;
  const int n = ka.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int* counts = reinterpret_cast<int*>(red + 2 * kRowWarps);  // per 32 queries: full | local << 16
  auto facts = [&](int q, int4& qi, int& r) -> int {  // returns the query's class: 0 full, 1 local, 2 zero
    bool any_local;
    const int seq = ka.seq_ids[q], t = ka.q_positions[q], mode = query_mode(ka, q, any_local);
    const int w = ka.windows ? ka.windows[q] : ka.window_scalar;
    const int err = query_error(a, seq, t, mode, any_local, w);
    r = err ? 0 : query_range(t, mode, w);
    const bool local_lo = HM ? any_local : mode == TRR_MODE_LOCAL;
    qi = make_int4(seq, t, local_lo ? max(0, t - w + 1) : 0, err << 24 | (r == 0) << 28);
    return r == 0 ? 2 : mode == TRR_MODE_LOCAL ? 1 : 0;
  };
  if (threadIdx.x < 32) counts[threadIdx.x] = 0;
  __syncthreads();
  long long rsum = 0;
  int4 qi;
  int r = 0, cls = 3;
#pragma unroll 1
  for (int q0 = 0; q0 < n; q0 += 32 * kRowWarps) {
    const int q = q0 + threadIdx.x;
    cls = 3;
    if (q < n) {
      cls = facts(q, qi, r);
      if (HM && r > 0) {
        const HeadCounts c = head_counts(ka, q);
        rsum += static_cast<long long>(c.full) * (qi.y + 1) + static_cast<long long>(c.local) * (qi.y + 1 - qi.z);
      } else {
        rsum += static_cast<long long>(r) * rows;
      }
    }
    const unsigned f = __ballot_sync(0xffffffffu, cls == 0), l = __ballot_sync(0xffffffffu, cls == 1);
    if (lane == 0) counts[(q0 >> 5) + warp] = __popc(f) | __popc(l) << 16;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
  if (lane == 0) red[warp] = rsum;
  __syncthreads();
  int incl = counts[lane];  // counts of each class in the query blocks before lane's
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int all = __shfl_sync(0xffffffffu, incl, 31), nf = all & 0xffff, nl = all >> 16;
#pragma unroll 1
  for (int q0 = 0; q0 < n; q0 += 32 * kRowWarps) {
    const int q = q0 + threadIdx.x, blk = (q0 >> 5) + warp;
    if (n > 32 * kRowWarps) cls = q < n ? facts(q, qi, r) : 3;
    const unsigned f = __ballot_sync(0xffffffffu, cls == 0), l = __ballot_sync(0xffffffffu, cls == 1);
    const unsigned below = (1u << lane) - 1u;
    const int before = __shfl_sync(0xffffffffu, incl, blk) - (__popc(f) | __popc(l) << 16);
    const int bf = (before & 0xffff) + __popc(f & below), bl = (before >> 16) + __popc(l & below);
    const int k = cls == 0 ? bf : cls == 1 ? nf + bl : nf + nl + q - bf - bl;
    if (q < n) {
      ord[k] = static_cast<uint16_t>(q);
      qinf[k] = qi;
      pre[k] = r;
    }
  }
  __syncthreads();
  rsum = 0;
#pragma unroll
  for (int k = 0; k < kRowWarps; ++k) rsum += red[k];
  // Split size: about one unit per warp while a unit then stays short, else up to three per
  // warp, of 700 positions at least, handed out on demand; never below pos_split.  (1.3B shape,
  // batch 64, contexts to 8192, 2 steps of 4 layers 666 us, units from 512 positions 685; 8 queries
  // of 32 sequences 269 and 292.  A query group's positions weigh about twice as much: gqa_long
  // shape 663 us for 4 steps of 3 layers, 673 with units from 250 positions.)  The tiles' bound of
  // splits_of cuts finer where tiles are of 16 keys: at head size 128 and in pages of 16 a unit has
  // 350 to 450 positions at most, whatever this asks for.  Binary32 arithmetic: the same result in
  // every CTA, and it only sizes the splits.
  const float warps = static_cast<float>(gridDim.x * kRowWarps), rs = static_cast<float>(rsum);
  const float one = rs / (0.85f * warps);
  const float most = GQ ? 600.f : 1000.f, least = GQ ? 350.f : 700.f;
  const float by_work = ceilf(one > most ? fmaxf(least, rs / (3.f * warps)) : one);
  const int pos_split = by_work > static_cast<float>(a.pos_split) ? static_cast<int>(fminf(by_work, 1073741824.f))
                                                                   : a.pos_split;
  const int chunk = (n + 32 * kRowWarps - 1) / (32 * kRowWarps);
  const int q0 = min(n, static_cast<int>(threadIdx.x) * chunk), q1 = min(n, q0 + chunk);
  int mine = 0;
#pragma unroll 1
  for (int k = q0; k < q1; ++k) {  // pre[k] becomes the query's unit count
    const int range = pre[k];
    int ns = 1, units = rows;
    if (range > 0) {
      ns = splits_of(range, pos_split, a.split_keys, a.split_extra, a.split_most, a.s_cap);
      units = rows * ns;
      if (HM) {
        const HeadCounts c = head_counts(ka, ord[k]);
        const int4 x = qinf[k];
        ns = splits_of(x.y + 1, pos_split, a.split_keys, a.split_extra, a.split_most, a.s_cap);
        units = c.full * ns + c.skip +
                c.local * splits_of(x.y + 1 - x.z, pos_split, a.split_keys, a.split_extra, a.split_most, a.s_cap);
      }
    }
    qinf[k].w |= ns;
    pre[k] = units;
    mine += units;
  }
  incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) red[8 + warp] = incl;
  __syncthreads();
  int off = incl - mine;
#pragma unroll 1
  for (int k = 0; k < warp; ++k) off += static_cast<int>(red[8 + k]);
#pragma unroll 1
  for (int q = q0; q < q1; ++q) {
    const int units = pre[q];
    pre[q] = off;
    off += units;
  }
  if (threadIdx.x == 32 * kRowWarps - 1) {
    pre[n] = off;
    pre[n + 1] = pos_split;
  }
  __syncthreads();
}

// mbar_wait_or out of line: a tile that has arrived is found by one test.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, volatile int* abort, uint64_t limit_ns) {
  return mbar_wait_or(bar, parity, abort, limit_ns);
}

// One unit as its warp plans it.
struct RowUnit {
  int q, h;         // query, query head
  int sp, ns;       // split, splits of the row
  int base;         // the row's first partial
  int t, lo;        // key range [lo, t]
  int err;          // the query's error: a zero row
  int T;            // pages; none for a zero row
  bool zero;        // a skip head or a failed query
};

// A split's share of a row is a run of its pages, listed from the widest class down and each
// class's in position order: the row's tiles (and kNewTiles for the query's own token of a
// decode step at the end) are cut evenly, at page boundaries.  So a split meets one or two
// classes (a share of every class made four switches a unit), and the warps of a CTA, which
// as a rule have the same split of neighbouring heads, run the same class's code at a time.
constexpr int kNewTiles = 3;

// Pages of split sp (of ns) of a query of sequence seq over key positions [lo, t]: returns
// their number (<= kItemMaxTiles); lane j below it gets page j's id in wid and class |
// fill << 2 | kMask in wmeta.  own: whether the query's own token joins the last split.  RUNS: a
// split may have more tiles than a warp has lanes and comes in runs of pages; skip is where the run
// starts in the split's share, and becomes where the next one does (0: this was the last).
// Eight lanes per class: a rolled nine-way search of the pages' first or last positions where
// the range needs it (small code: a unit's plan competes with its tiles for the instruction
// cache).
template <bool RUNS>
__device__ __forceinline__ int plan_pages(const LayerArgs& a, int seq, int lo, int t, int sp, int ns, bool own,
                                          int kt_most, int kt_wide, int lane, int& skip, int& wid, int& wmeta) {
  const int c8 = lane >> 3, sub = lane & 7, lg = __ffs(a.P) - 1;
  const int nt = a.ntok[seq * 4 + c8];
  const bool upper_mask = t < a.last_pos[seq];  // keys after t may be stored
  const int pages = (nt + a.P - 1) >> lg;
  const int64_t row0 = (static_cast<int64_t>(seq) * 4 + c8) * a.MP;
  int first = 0, end = pages;
#pragma unroll 1
  for (int side = lo > 0 ? 0 : 1; side < (upper_mask ? 2 : 1); ++side) {
    const int* arr = (side ? a.pfirst : a.plast) + row0;
    const int x = side ? t + 1 : lo;  // entries below x
    int l = 0, h = pages;             // the count lies in [l, h]
    // first the end of the list, where decode queries look: a window's pages and a few more
    int step = side ? 1 : (((t + 1 - lo) >> lg) + 8) >> 3, p1 = max(0, pages - 8 * step);
    int probe = p1 + sub * step;
#pragma unroll 1
    while (__any_sync(0xffffffffu, l < h)) {
      const bool below = probe < h && arr[probe] < x;
      const int cnt = __popc((__ballot_sync(0xffffffffu, below) >> (8 * c8)) & 255u);
      const int p0 = probe - sub * step;
      if (l < h) {
        if (cnt < 8) h = min(h, p0 + cnt * step);  // probe cnt is not below (or past the end)
        if (cnt > 0) l = max(l, p0 + (cnt - 1) * step + 1);
      }
      step = max(1, (h - l + 8) / 9);
      probe = l + sub * step + (step > 1 ? step - 1 : 0);
    }
    if (side) end = l;
    else first = l;
  }
  const int npr = max(0, end - first);
  int lw = lg + 1 - __ffs(c8 == 3 ? kt_wide : kt_most);  // log2 of a page's tiles
  const int mass = npr << lw;
  int before = 0, all = own ? kNewTiles : 0;  // tiles of the wider classes; of the row
#pragma unroll
  for (int k = 0; k < kClasses; ++k) {
    const int m = __shfl_sync(0xffffffffu, mass, 8 * k);
    all += m;
    before += k > c8 ? m : 0;
  }
  // 16-bit tiles count twice where a split's tiles then stay within a warp's lanes: a warp's
  // ring holds one of 8 KB, so that each waits out a copy, and a split of nothing else ended
  // last.  (160M, 4 steps 796 us, 832 counted once; batch 256 of the sweep 1575 and 1631, 1.3B 666 and
  // 707; head size 128, batch 64 of contexts 4000 251 and 247.)
  const int wide = __shfl_sync(0xffffffffu, mass, 24);
  if (div24(all + wide, ns) + 1 + 2 * (a.P >> (__ffs(kt_wide) - 1)) <= kItemMaxTiles) {
    all += wide;
    if (c8 == 3) ++lw;
    else before += wide;
  }
  const int w = 1 << lw;
  // the split's pages: those that start in its share [b0, b1) of the tiles, all / ns and one
  // more for the first all % ns splits (all < 2^24)
  const int each = div24(all, ns), extra = all - each * ns;
  const int share = sp * each + min(sp, extra), b2 = share + each + (sp < extra ? 1 : 0);
  int b0 = share, b1 = b2;
  if (RUNS) {
    b0 += skip;
    b1 = min(b2, b0 + kItemMaxTiles + 1 - (1 << __shfl_sync(0xffffffffu, lw, 24)));  // (the widest pages are class 3's)
    skip = b1 < b2 ? b1 - share : 0;
  }
  const int beg = min(npr, max(0, (b0 - before + w - 1) >> lw));
  const int tc = min(npr, max(0, (b1 - before + w - 1) >> lw)) - beg;
  const int t1 = __shfl_sync(0xffffffffu, tc, 24), t2 = t1 + __shfl_sync(0xffffffffu, tc, 16);
  const int t3 = t2 + __shfl_sync(0xffffffffu, tc, 8);
  const int T = min(t3 + __shfl_sync(0xffffffffu, tc, 0), kItemMaxTiles);  // (the split bound, or the run's, keeps it within)
  const int r = (lane >= t1) + (lane >= t2) + (lane >= t3), c = 3 - r;
  const int kid = __shfl_sync(0xffffffffu, first + beg, 8 * c) + lane - (r == 0 ? 0 : r == 1 ? t1 : r == 2 ? t2 : t3);
  const int f = __shfl_sync(0xffffffffu, first, 8 * c), e = __shfl_sync(0xffffffffu, end, 8 * c);
  const int ntc = __shfl_sync(0xffffffffu, nt, 8 * c);
  wid = 0;
  wmeta = 0;
  if (lane < T) {
    wid = a.pt[(static_cast<int64_t>(seq) * 4 + c) * a.MP + kid];
    // slot positions are needed on a page that may hold keys outside [lo, t]
    const bool mask = (lo > 0 && kid == f) || (upper_mask && kid == e - 1);
    wmeta = c | (min(a.P, ntc - kid * a.P) << 2) | (mask ? kMask : 0);
  }
  return T;
}

// ------------------------------------------------------------------- tile arithmetic --

// c = a * b with a zero accumulator
template <int B>
__device__ __forceinline__ void mma_cls0(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  if (B == 16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// The eight keys i = 0 .. 7 of a tile whose V rows a lane (its lane % 4 = tig) reads, chosen
// per row length so that the lanes' rows fall into different banks; the first four are keys
// below 16 in each map.  (Key order is free in P.V as long as the weights follow it.)
__host__ __device__ constexpr int row_map(int D, int B) { return B == 16 || (D == 128 && B == 8) ? 2 : B == 8 ? 1 : 0; }
template <int MAP>
__device__ __forceinline__ int v_key(int tig, int i) {
  return MAP == 0 ? tig + 4 * i : MAP == 1 ? 4 * tig + (i & 3) + 16 * (i >> 2) : 2 * tig + (i & 1) + 8 * (i >> 1);
}
// A tile's weights lie in shared memory as one 16-byte row of eight f16 per key (columns
// group * 2 + (hi | lo)), read as the mma's B operands by one ldmatrix.x4.trans: lane l gives
// the address of row l % 8 of matrix l / 8, the key that this place of the contraction has.
template <int MAP>
__device__ __forceinline__ int w_row(int lane) {
  const int r = lane & 7, m = lane >> 3;  // matrices: keys i = 0, 1 | 2, 3 | 4, 5 | 6, 7 of lanes r / 2
  return v_key<MAP>(r >> 1, 2 * m + (r & 1));
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t (&r)[4], const uint8_t* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p))
               : "memory");
}

// Where a lane's bytes lie in a tile's K rows (rows gid + 8 h + 16 u, dims tig D/4 ..) and V
// rows (row v_key(tig, i), dims gid D/8 ..): a lane offset, then per load one exclusive-or of
// a constant (8- and 16-bit rows keep the chunks of a line in the order chunk ^ (line % 8))
// and a constant to add.  q, hf: the 16-byte chunk of a lane's part.
template <int D, int B>
__device__ __forceinline__ uint32_t k_lane(int gid, int tig) {
  constexpr int rowb = D * B / 8;
  if (B < 8) return gid * rowb + tig * (rowb / 4);
  if (rowb == 64) return (gid >> 1) * 128 + (((((gid & 1) << 2) | tig) ^ (gid >> 1)) << 4);
  if (rowb == 128) return gid * 128 + (((2 * tig) ^ gid) << 4);
  return (2 * gid + (tig >> 1)) * 128 + ((((tig & 1) << 2) ^ ((2 * gid + (tig >> 1)) & 7)) << 4);
}
template <int D, int B>
__device__ __forceinline__ uint32_t k_off(uint32_t lane_off, int h, int u, int q) {
  constexpr int rowb = D * B / 8;
  const uint32_t x = B < 8 ? lane_off : lane_off ^ (rowb == 64 ? h << 6 : q << 4);
  return x + (8 * h + 16 * u) * rowb + (B < 8 ? 16 * q : 0);
}
template <int D, int B>
__device__ __forceinline__ uint32_t v_lane(int gid, int tig) {
  constexpr int rowb = D * B / 8;
  if (B < 8) return tig * rowb + (rowb >= 32 ? gid * (rowb / 8) : (gid * (rowb / 8)) & ~3);
  if (rowb == 64) return tig * 256 + (((gid >> 1) ^ (2 * tig)) << 4) + ((gid & 1) << 3);
  if (rowb == 128) return tig * 256 + ((gid ^ (2 * tig)) << 4);
  return (4 * tig + (gid >> 2)) * 128 + ((((gid & 3) << 1) ^ ((4 * tig) & 7) ^ (gid >> 2)) << 4);
}
template <int D, int B>
__device__ __forceinline__ uint32_t v_off(uint32_t lane_off, int i, int hf) {
  constexpr int rowb = D * B / 8;
  if (B < 8) return lane_off + 4 * i * rowb;
  if (rowb == 64) return (lane_off ^ ((((i & 1) << 2) | ((i >> 1) & 1)) << 4)) + ((i & 3) >> 1) * 128 + (i >> 2) * 1024;
  if (rowb == 128) return (lane_off ^ ((i & 1) << 4)) + (i & 1) * 128 + (i >> 1) * 1024;
  return (lane_off ^ (((2 * (i & 1)) ^ hf) << 4)) + (i & 1) * 256 + (i >> 1) * 2048;
}

// NW words at p (a shared-memory pointer, aligned for one load of up to 16 bytes).
template <int NW>
__device__ __forceinline__ void load_words(const uint8_t* p, uint32_t* w) {
  if (NW % 4 == 0) {
#pragma unroll
    for (int k = 0; k < NW; k += 4) {
      const uint4 u = *reinterpret_cast<const uint4*>(p + 4 * k);
      w[k] = u.x; w[k + 1] = u.y; w[k + 2] = u.z; w[k + 3] = u.w;
    }
  } else if (NW == 2) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    w[0] = u.x; w[1] = u.y;
  } else {
    w[0] = *reinterpret_cast<const uint32_t*>(p);
  }
}

__device__ __forceinline__ void mma_tf32(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int D, int NG>
struct RowState {
  static constexpr int NP = D / 8, MT = D / 16;
  uint32_t kb[NP];    // the query as q.k's B operand in the current class
  float acc[MT][4];   // V sums: dims gid D/8 + 2 t (+ 1) x columns (group tig % NG, hi | lo),
                      // times 2^vfac_log2 and the group's ws for codes, 1 for width 16
  float qsum[NG];     // softmax scale * log2(e) * sum of the query over each group
  float m, l;         // running maximum (the warp's, log2 units); this lane's sum of weights
  float zacc[NG];     // this lane's sums of p * z
  float ws[NG];       // codes' weights are p * s * ws (a power of two per group)
  float kfac[NG];     // the current class's factors of the group sums
  uint32_t kl, vl;    // the current class's lane offsets (k_lane, v_lane)
  int wl;             // the byte offset of the lane's row of weights as ldmatrix reads it
  int zoff;           // the offset in a tile of the V scales of the lane's key
  int cls;
};

// The query row in the order and scale of class cls's B operand, to qs: widths 2, 4 and 8 as
// f16 pairs times 2^(15 - E - the code's bit offset), E of the values' group: the largest are just
// below f16's end, and what is 2^-24 of them still has all of its 8 bits; width 16 the bf16 values.
// Lane holds dims lane * D/32 .. (raw, bf16).
template <int D>
__device__ __forceinline__ void store_query_row(uint8_t* qs, uint2 raw, int cls, int E, int lane) {
  constexpr int DPL = D / 32;
  const int d0 = lane * DPL, part = d0 / (D / 4), dd0 = d0 % (D / 4);
  uint8_t* row = qs + part * (D / 2);
  if (cls == 3) {
    if (D == 64) *reinterpret_cast<uint32_t*>(row + 2 * dd0) = raw.x;
    else *reinterpret_cast<uint2*>(row + 2 * dd0) = raw;
    return;
  }
#pragma unroll
  for (int j = 0; j < DPL; ++j) {
    const uint32_t w = j < 2 ? raw.x : raw.y;
    const int dd = dd0 + j;
    // the word and half of dim dd, and the bit offset of its code: width 8 pairs (2 i, 2 i + 1);
    // width 4 (8 k + i, + 4), offset 4 (i % 2); width 2 (16 k + i, + 8), offset 2 (i < 5 ? i : i - 5)
    const int lg = cls == 0 ? 3 : 2, i = dd & ((1 << lg) - 1);
    const int word = cls == 2 ? dd >> 1 : ((dd >> (lg + 1)) << lg) + i, half = cls == 2 ? dd & 1 : (dd >> lg) & 1;
    const int pos = cls == 2 ? 0 : cls == 1 ? 4 * (i & 1) : 2 * (i < 5 ? i : i - 5);
    const float v = ((j & 1) ? bf_hi(w) : bf_lo(w)) * __int_as_float((127 + 15 - E - pos) << 23);
    *reinterpret_cast<__half*>(row + 4 * word + 2 * half) = __float2half_rn(v);
  }
}

// log2 of the factor the accumulators of dim j (of a lane's D/8) carry in class c, without
// the codes' ws
__host__ __device__ constexpr int row_fac(int c, int j) { return c == 3 ? 0 : vfac_log2(c, j); }

template <int D>
__device__ __forceinline__ uint2 load_row(const uint16_t* src, int lane) {
  uint2 r = make_uint2(0, 0);
  if (D == 64) r.x = reinterpret_cast<const uint32_t*>(src)[lane];
  else r = reinterpret_cast<const uint2*>(src)[lane];
  return r;
}

// What a code's weight p * s * ws may reach (f16 ends at 2^16), and the largest ws: with the
// largest factor of a code's bit offset it takes sums of width 16 into a code's domain unchanged.
constexpr float kWeightTop = 32768.f;
constexpr int kWeightScale = 16;  // log2

// The element of a per-group array for the group whose columns this lane's accumulators have.
template <int NG>
__device__ __forceinline__ float lane_group(const float (&x)[NG], int lane) {
  float r = x[0];
#pragma unroll
  for (int i = 1; i < NG; ++i)
    if ((lane & 3) % NG == i) r = x[i];
  return r;
}
// 1 / x of a power of two
__device__ __forceinline__ float pow2_inverse(float x) { return __int_as_float((254 << 23) - __float_as_int(x)); }

// What a lane keeps of class B while it works on its tiles.
template <int D, int NG, int B>
__device__ __forceinline__ void row_class(RowState<D, NG>& st, int lane) {
  st.kl = k_lane<D, B>(lane >> 2, lane & 3);
  st.vl = v_lane<D, B>(lane >> 2, lane & 3);
  st.wl = 16 * w_row<row_map(D, B)>(lane);
}

// Class st.cls -> to: the query's operand (lane (gid, tig) holds dims tig D/4 .. of group
// gid % NG), the accumulators' factors (fac: a table [from][to][dim of the lane]).
template <int D, int NG>
__device__ __forceinline__ void row_switch(RowState<D, NG>& st, int to, bool fresh, uint8_t* qs, const float* fac,
                                           float qscale, int kt, int lane) {
  constexpr int NP = D / 8, MT = D / 16;
  const int gid = lane >> 2, tig = lane & 3;
  const bool ok = (tig * NG) / 4 == gid % NG;
  switch (to) {
    case 0: row_class<D, NG, 2>(st, lane); break;
    case 1: row_class<D, NG, 4>(st, lane); break;
    case 2: row_class<D, NG, 8>(st, lane); break;
    default: row_class<D, NG, 16>(st, lane); break;
  }
  const int b = bits_of_class(to);
  st.zoff = kt * (2 * (D * b / 8) + 4 * NG) + min(8 * tig + gid, kt - 1) * NG * 4;
  const int* qe = reinterpret_cast<const int*>(qs + 4 * D);  // largest exponents of the groups
  store_query_row<D>(qs, load_row<D>(reinterpret_cast<const uint16_t*>(qs + 2 * D), lane), to, qe[lane / (32 / NG)], lane);
#pragma unroll
  for (int i = 0; i < NG; ++i)
    // finite: 0 * kfac of a scale of 0 is 0; above 2^118 q's scores are beyond binary32 anyway
    st.kfac[i] = to == 3 ? qscale : fminf(__int_as_float((127 + qe[i]) << 23) * qscale * pow2f(9), 3.4028235e38f);
  __syncwarp();
  load_words<NP>(qs + tig * (D / 2), st.kb);
#pragma unroll
  for (int i = 0; i < NP; ++i) st.kb[i] = ok ? st.kb[i] : 0u;
  if (!fresh) {
    const float ws = lane_group<NG>(st.ws, lane);
    const float g = (to == 3) == (st.cls == 3) ? 1.f : to == 3 ? pow2_inverse(ws) : ws;
    float f[2 * MT];
    load_words<2 * MT>(reinterpret_cast<const uint8_t*>(fac + (st.cls * 4 + to) * (D / 8)), reinterpret_cast<uint32_t*>(f));
#pragma unroll
    for (int t = 0; t < MT; ++t) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float x = f[2 * t + r] * g;
        st.acc[t][2 * r] *= x;
        st.acc[t][2 * r + 1] *= x;
      }
    }
  }
  st.cls = to;
}

// A tile: kt (16 or 32) rows at `tile` (K rows, V rows, K (s, z), V (s, z)).  Its work is in
// three parts, so that only what depends on the width has a copy per width (the four widths'
// loops and the rest of the kernel compete for the instruction cache: with whole tiles per
// width a seventh of the fetches missed it).

// The A operands of P.V of 16 keys (half u of the tile) and this lane's D/8 dims.
template <int D, int NG, int B>
__device__ __forceinline__ void value_words(const RowState<D, NG>& st, const uint8_t* v0, int u, uint32_t* va, int lane) {
  constexpr int MT = D / 16;
  constexpr int VB = D * B / 64;   // V bytes per lane and key (D/8 dims)
  constexpr int VW = VB >= 4 ? VB / 4 : 1;
  uint32_t x[4][VW];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    load_words<VW>(v0 + v_off<D, B>(st.vl, 4 * u + i, 0), x[i]);
    if (VB < 4) x[i][0] >>= (((lane >> 2) * VB) & 3) * 8;
  }
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    va[4 * t] = v_pair<B>(x[0], x[1], 2 * t);
    va[4 * t + 1] = v_pair<B>(x[0], x[1], 2 * t + 1);
    va[4 * t + 2] = v_pair<B>(x[2], x[3], 2 * t);
    va[4 * t + 3] = v_pair<B>(x[2], x[3], 2 * t + 1);
  }
}

// 1. The group sums of q.c of the lane's key: lane (gid, tig) takes key 8 tig + gid, which is
// in half tig % 2 of the 16 keys tig / 2.
template <int D, int NG, int B>
__device__ __forceinline__ void tile_scores(const RowState<D, NG>& st, const uint8_t* tile, int kt, float (&g)[NG], int lane) {
  constexpr int KS = D / 16;
  constexpr int KW = D * B / 128;  // K words per lane and key (D/4 dims)
  const int tig = lane & 3;
  const bool h1 = tig & 1, u1 = tig & 2;
  float o0 = 0.f, o1 = 0.f;  // NG = 4: the partner's key, this lane's groups
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && kt == 16) break;
    float c[4], c2[4];
    constexpr int KH = KW >= 8 ? KW / 4 : 1, KWH = KW / KH, KSH = KS / KH;  // 16 bytes of a row at a time when long
#pragma unroll
    for (int hf = 0; hf < KH; ++hf) {
      uint32_t k1[KWH], k2[KWH];
      load_words<KWH>(tile + k_off<D, B>(st.kl, 0, u, hf), k1);
      load_words<KWH>(tile + k_off<D, B>(st.kl, 1, u, hf), k2);
#pragma unroll
      for (int s = hf * KSH; s < (hf + 1) * KSH; ++s) {
        const int i0 = 2 * (s - hf * KSH);
        const uint32_t a0 = k_pair<B>(k1, i0), a1 = k_pair<B>(k2, i0), a2 = k_pair<B>(k1, i0 + 1), a3 = k_pair<B>(k2, i0 + 1);
        if (s == 0) mma_cls0<B>(c, a0, a1, a2, a3, st.kb[0], st.kb[1]);
        else if (D == 128 && s == 1) mma_cls0<B>(c2, a0, a1, a2, a3, st.kb[2], st.kb[3]);
        else mma_cls<B>((D == 128 && (s & 1)) ? c2 : c, a0, a1, a2, a3, st.kb[2 * s], st.kb[2 * s + 1]);
      }
    }
    if (D == 128) {
#pragma unroll
      for (int i = 0; i < 4; ++i) c[i] += c2[i];
    }
    if (u == 0 || u1) {
      g[0] = h1 ? c[2] : c[0];
      if (NG > 1) g[NG > 1 ? 1 : 0] = h1 ? c[3] : c[1];
      if (NG == 4) {
        o0 = h1 ? c[0] : c[2];
        o1 = h1 ? c[1] : c[3];
      }
    }
  }
  if (NG == 4) {  // this lane's columns are groups 0 and 1 (tig even) or 2 and 3: trade with tig ^ 1
    const float x0 = __shfl_xor_sync(0xffffffffu, o0, 1), x1 = __shfl_xor_sync(0xffffffffu, o1, 1);
    g[NG > 2 ? 2 : 0] = h1 ? g[0] : x0;
    g[NG > 3 ? 3 : 0] = h1 ? g[NG > 1 ? 1 : 0] : x1;
    g[0] = h1 ? x0 : g[0];
    g[NG > 1 ? 1 : 0] = h1 ? x1 : g[NG > 1 ? 1 : 0];
  }
}

// 2. The key's weight (ok: it counts): the score from the group sums, p, and p * s * ws as the
// operand rows at wb.  The running maximum and the groups' ws are set anew when a key asks for it:
// its score is above the maximum by more than kTau, or its weight in a group above kWeightTop.  ws
// follows the weights, not the scales alone, and each group its own: a group with scales 2^26 below
// another's, or keys with such scales beside one of no weight, keep all of their bits.
// kw, zw: the key's K and V (s, z); (1, 0) where the width has none (has_sz).
template <int D, int NG>
__device__ __forceinline__ void tile_weights(RowState<D, NG>& st, float (&g)[NG], bool ok, bool has_sz,
                                             const uint32_t (&kw)[NG], uint32_t (&zw)[NG], int key, uint8_t* wb, int lane) {
  constexpr int MT = D / 16;
  float sc = 0.f, w[NG];
  float2 vz[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const float2 sz = __half22float2(*reinterpret_cast<const __half2*>(&kw[i]));
    sc = fmaf(sz.x * st.kfac[i], g[i], fmaf(sz.y, st.qsum[i], sc));
    if (!ok) zw[i] = 0u;  // a slot that does not count may hold any bytes
    vz[i] = __half22float2(*reinterpret_cast<const __half2*>(&zw[i]));
  }
  if (!ok) sc = kNegInf;
  float p = fast_exp2(sc - st.m);  // 0 for a key that does not count
  bool ask = p > 256.f;            // 2^kTau
  if (has_sz) {
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      w[i] = p * vz[i].x * st.ws[i];
      ask |= w[i] > kWeightTop;
    }
  }
  if (__any_sync(0xffffffffu, ask)) {
    float top = sc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    top = fmaxf(top, st.m);
    const float alpha = top == st.m ? 1.f : fast_exp2(st.m - top);
    float f = alpha;
    st.m = top;
    p = fast_exp2(sc - top);
    st.l *= alpha;
#pragma unroll
    for (int i = 0; i < NG; ++i) st.zacc[i] *= alpha;
    if (has_sz) {
      const float before = lane_group<NG>(st.ws, lane);
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        float big = p * vz[i].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
        // big * ws < 2^6 (width 2), 2^3, 2^0 (width 8): p may rise by 2^8, and the scales of the
        // narrower classes that follow are larger by the ratio of the levels
        const int e = 5 - 3 * st.cls - (static_cast<int>(__float_as_uint(big) >> 23) - 127);
        if (big > 0.f) st.ws[i] = __int_as_float((127 + min(kWeightScale, e)) << 23);
        w[i] = p * vz[i].x * st.ws[i];
      }
      f *= lane_group<NG>(st.ws, lane) * pow2_inverse(before);
    }
#pragma unroll
    for (int t = 0; t < MT; ++t)
#pragma unroll
      for (int i = 0; i < 4; ++i) st.acc[t][i] *= f;
  }
  st.l += p;
  if (has_sz) {
    uint32_t w2[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      st.zacc[i] = fmaf(p, vz[i].y, st.zacc[i]);
      const float wh = __half2float(__float2half_rn(w[i]));
      w2[i] = pack_f16x2(wh, (w[i] - wh) * kLoScale);
    }
    uint32_t* at = reinterpret_cast<uint32_t*>(wb + 16 * key);
    if (NG == 1) at[0] = w2[0];
    else if (NG == 2) *reinterpret_cast<uint2*>(at) = make_uint2(w2[0], w2[NG > 1 ? 1 : 0]);
    else *reinterpret_cast<uint4*>(at) = make_uint4(w2[0], w2[NG > 1 ? 1 : 0], w2[NG > 2 ? 2 : 0], w2[NG > 3 ? 3 : 0]);
  } else {
    const uint32_t hi = __float_as_uint(p) & 0xffffe000u;  // 11 bits, exact remainder
    *reinterpret_cast<float2*>(wb + 8 * key) = make_float2(__uint_as_float(hi), (p - __uint_as_float(hi)) * kLoScale);
  }
}

// 3. P.V of a tile of width B < 16.
template <int D, int NG, int B>
__device__ __forceinline__ void tile_values(RowState<D, NG>& st, const uint8_t* tile, int kt, const uint8_t* wb, int lane) {
  constexpr int MT = D / 16;
  uint32_t w[4];
  ldmatrix4_trans(w, wb + st.wl);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && kt == 16) break;
    uint32_t x[4 * MT];
    value_words<D, NG, B>(st, tile + kt * (D * B / 8), u, x, lane);
#pragma unroll
    for (int t = 0; t < MT; ++t) mma_f16(st.acc[t], x[4 * t], x[4 * t + 1], x[4 * t + 2], x[4 * t + 3], w[2 * u], w[2 * u + 1]);
  }
}

// The same for width 16.  all: lanes whose key counts (part: not every one does).
template <int D, int NG>
__device__ __forceinline__ void tile_values16(RowState<D, NG>& st, const uint8_t* tile, int kt, bool part, unsigned all,
                                              const uint8_t* wb, int lane) {
  constexpr int VB = D / 4, MAP = row_map(D, 16);  // V bytes per lane and key (D/8 dims)
  const int gid = lane >> 2, tig = lane & 3;
  const uint8_t* v0 = tile + kt * 2 * D;
  const uint8_t* wa = wb + (gid & 1) * 4;
#pragma unroll
  for (int s = 0; s < 4; ++s) {  // 8 keys
    if (s == 2 && kt == 16) break;
    const int ka = v_key<MAP>(tig, 2 * s), kb = v_key<MAP>(tig, 2 * s + 1);
    const uint32_t wx = *reinterpret_cast<const uint32_t*>(wa + 8 * ka), wy = *reinterpret_cast<const uint32_t*>(wa + 8 * kb);
#pragma unroll
    for (int hf = 0; hf < VB / 16; ++hf) {
      uint32_t x[4], y[4];
      load_words<4>(v0 + v_off<D, 16>(st.vl, 2 * s, hf), x);
      load_words<4>(v0 + v_off<D, 16>(st.vl, 2 * s + 1, hf), y);
      if (part) {  // values of keys that do not count read as 0 (they may be NaN)
        const bool oka = (all >> ((ka & 7) * 4 + (ka >> 3))) & 1u, okb = (all >> ((kb & 7) * 4 + (kb >> 3))) & 1u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (!oka) x[i] = 0u;
          if (!okb) y[i] = 0u;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        mma_tf32(st.acc[hf * 4 + i], x[i] << 16, x[i] & 0xffff0000u, y[i] << 16, y[i] & 0xffff0000u, wx, wy);
    }
  }
}

// ------------------------------------------------------------------- query groups --
//
// A KV head with its g >= 2 query heads (g * NG <= 8) per unit: column n of the B operands is
// head n / NG and quantiser group n % NG, so that lane (gid, tig) has the scores of keys
// gid + 8 h + 16 u for its columns 2 tig and 2 tig + 1 (two groups of a head, or two heads at
// NG = 1).  Weights p * s are two f16 parts, width 16's p two bf16 parts (one f16 part rounds by
// 2^-12, which leaves rows 1 to 2 % further off; the second takes 1 to 4 % of the time).  A
// running maximum is raised when a score exceeds it by 2^3 (any excess where a scale could then
// take p * s out of f16's range): raised at every new maximum, nine tiles in ten would rescale
// the accumulators.  Narrow groups' rows are stored plainly.
//
// f16 ends at 2^-25, which p * s of small values would come near: p is therefore taken relative to
// 2^-lift of the maximum, lift (0 to 16) lowered when a larger V scale comes.  (V of size 2^-10: rows
// 5e-3 off without it, 2^-14 8 %; gqa_long shape 646 us for 4 steps, 630 without.)
constexpr float kGroupTau = 3.f, kGroupWide = 8000.f;
constexpr float kLift = 16.f;  // at first
//
// Groups wider than the operand's 8 columns are taken 8 / NG heads at a time, so that a page is
// copied and its codes unpacked once for those heads, where a call's work is bound by that.  (64 heads
// on 8 of 128, batch 128, context 4096, 2 steps of 2 layers: 953 us; 1998 with a query head per warp,
// each copying the pages for itself.)  They keep more of the weights' and sums' bits: a power of two
// per column in place of the lift, chosen from the V scales of keys with weight, and the zero points
// folded in.  Their rows are stored as MHA's.
constexpr float kGroupTop = 4096.f;     // s * ws at most: p <= 2^3 keeps p * s * ws below f16's end
constexpr float kGroupWeight = -17.f;   // log2 of the p from which on a key's scale counts: a smaller
                                        // p takes no s * ws (at most 2^32) past f16's end
template <int D, int NG, bool WIDE>
struct GroupState {
  static constexpr int NP = D / 8, MT = D / 16;
  uint32_t kb[NP];
  float acc[MT][4];  // dims gid D/8 + 2 t (+ 1) x the lane's columns, times 2^vfac_log2
  float qsum[2], m[2], l[2], zacc[2];  // per column (m: its head's maximum - lift)
  float lift, lim;   // and the largest V scale that lift allows (wide groups: 0, not used)
  float ws[2];       // wide groups, per column: codes' weights are p * s * ws (a power of two)
  float kfac[2];     // per column: the current class's factor of the group sums
  uint32_t kl, vl;
  int wl, zoff, cls;
  int E;             // exponent of the largest query value of the head and group of column gid
};

template <int D, int NG, int B, bool WIDE>
__device__ __forceinline__ void group_class(GroupState<D, NG, WIDE>& st, const uint8_t* qs, int heads, int lane) {
  constexpr int NP = D / 8, rowb = D * B / 8;
  const int gid = lane >> 2, tig = lane & 3, r = gid / NG;
  const bool ok = r < heads && (tig * NG) / 4 == gid % NG;
  uint32_t raw[NP];
  load_words<NP>(qs + (r < heads ? r : 0) * D * 2 + tig * (D / 2), raw);
  const float escale = __int_as_float((127 + 15 - st.E) << 23);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    uint32_t w = raw[i];
    if (B != 16) {
      const int lo = kp_lo<B>(i), hi = kp_hi<B>(i);
      const float f = pow2f(-kp_pos<B>(i)) * escale;
      w = pack_f16x2(((lo & 1) ? bf_hi(raw[lo >> 1]) : bf_lo(raw[lo >> 1])) * f,
                     ((hi & 1) ? bf_hi(raw[hi >> 1]) : bf_lo(raw[hi >> 1])) * f);
    }
    st.kb[i] = ok ? w : 0u;
  }
  st.kl = WIDE ? k_lane<D, B>(gid, tig) : gid * rowb + tig * (rowb / 4);
  st.vl = WIDE ? v_lane<D, B>(gid, tig) : tig * rowb + (rowb >= 32 ? gid * (rowb / 8) : (gid * (rowb / 8)) & ~3);
  st.wl = 16 * w_row<WIDE ? row_map(D, B) : 0>(lane);
}

template <int D, int NG, bool WIDE>
__device__ __forceinline__ void group_switch(GroupState<D, NG, WIDE>& st, int to, bool fresh, const uint8_t* qs, int heads,
                                             const float* fac, float qscale, int kt, int lane) {
  constexpr int MT = D / 16;
  switch (to) {
    case 0: group_class<D, NG, 2, WIDE>(st, qs, heads, lane); break;
    case 1: group_class<D, NG, 4, WIDE>(st, qs, heads, lane); break;
    case 2: group_class<D, NG, 8, WIDE>(st, qs, heads, lane); break;
    default: group_class<D, NG, 16, WIDE>(st, qs, heads, lane); break;
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {  // as in row_switch
    const float e = __int_as_float((127 + __shfl_sync(0xffffffffu, st.E, 4 * (2 * (lane & 3) + j))) << 23);
    st.kfac[j] = to == 3 ? qscale : fminf(e * qscale * pow2f(9), 3.4028235e38f);
  }
  st.zoff = kt * (2 * (D * bits_of_class(to) / 8) + 4 * NG) + (lane >> 2) * NG * 4 + (NG == 4 ? (lane & 1) * 8 : 0);
  if (!fresh) {
    float f[2 * MT];
    load_words<2 * MT>(reinterpret_cast<const uint8_t*>(fac + (st.cls * 4 + to) * (D / 8)), reinterpret_cast<uint32_t*>(f));
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float g = !WIDE || (to == 3) == (st.cls == 3) ? 1.f : to == 3 ? pow2_inverse(st.ws[j]) : st.ws[j];
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        st.acc[t][j] *= f[2 * t] * g;
        st.acc[t][2 + j] *= f[2 * t + 1] * g;
      }
    }
  }
  st.cls = to;
}

// 1. The columns' group sums of q.c: c[u][2 h + j] is key gid + 8 h + 16 u, column 2 tig + j.
template <int D, int NG, int B, bool WIDE>
__device__ __forceinline__ void group_scores(const GroupState<D, NG, WIDE>& st, const uint8_t* tile, int kt, float (&c)[2][4]) {
  constexpr int KS = D / 16, rowb = D * B / 8;
  constexpr int KW = D * B / 128;  // K words per lane and key (D/4 dims)
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && kt == 16) break;
    float c2[4];
    constexpr int KH = KW >= 8 ? KW / 4 : 1, KWH = KW / KH, KSH = KS / KH;
#pragma unroll
    for (int hf = 0; hf < KH; ++hf) {
      uint32_t k1[KWH], k2[KWH];
      load_words<KWH>(tile + (WIDE ? k_off<D, B>(st.kl, 0, u, hf) : st.kl + 16 * u * rowb + 16 * hf), k1);
      load_words<KWH>(tile + (WIDE ? k_off<D, B>(st.kl, 1, u, hf) : st.kl + (16 * u + 8) * rowb + 16 * hf), k2);
#pragma unroll
      for (int s = hf * KSH; s < (hf + 1) * KSH; ++s) {
        const int i0 = 2 * (s - hf * KSH);
        const uint32_t a0 = k_pair<B>(k1, i0), a1 = k_pair<B>(k2, i0), a2 = k_pair<B>(k1, i0 + 1), a3 = k_pair<B>(k2, i0 + 1);
        if (s == 0) mma_cls0<B>(c[u], a0, a1, a2, a3, st.kb[0], st.kb[1]);
        else if (D == 128 && s == 1) mma_cls0<B>(c2, a0, a1, a2, a3, st.kb[2], st.kb[3]);
        else mma_cls<B>((D == 128 && (s & 1)) ? c2 : c[u], a0, a1, a2, a3, st.kb[2 * s], st.kb[2 * s + 1]);
      }
    }
    if (D == 128) {
#pragma unroll
      for (int i = 0; i < 4; ++i) c[u][i] += c2[i];
    }
  }
}

// 2. The weights of the lane's four keys (ok: bit 2 u + h) for its columns, as operand rows at
// wb.  has_sz: the width has scales (at sz: the key gid's V scales, K's kt keys before).
template <int D, int NG, bool WIDE>
__device__ __forceinline__ void group_weights(GroupState<D, NG, WIDE>& st, const float (&c)[2][4], unsigned ok, bool has_sz,
                                              const uint8_t* sz, int kt, int heads, uint8_t* wb, int lane) {
  constexpr int MT = D / 16, J = NG == 1 ? 2 : 1;  // heads of a lane
  const int gid = lane >> 2, tig = lane & 3;
  float sc[4][J], big = 0.f;
  uint32_t zw[4][2];
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // key gid + 8 k
    uint32_t kw[2] = {0x3c00u, 0x3c00u};
    zw[k][0] = zw[k][1] = 0x3c00u;
    const bool good = (ok >> k) & 1u;
    if (has_sz && (k < 2 || kt > 16)) {
      if (NG == 1) {
        load_words<1>(sz + (8 * k - kt) * NG * 4, kw);
        load_words<1>(sz + 8 * k * NG * 4, zw[k]);
        kw[1] = kw[0];
        zw[k][1] = zw[k][0];
      } else {
        load_words<2>(sz + (8 * k - kt) * NG * 4, kw);
        load_words<2>(sz + 8 * k * NG * 4, zw[k]);
      }
    }
    float cp[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&kw[j]));
      cp[j] = fmaf(f.x * st.kfac[j], c[k >> 1][2 * (k & 1) + j], f.y * st.qsum[j]);
      if (!good) zw[k][j] = 0u;  // a slot that does not count may hold any bytes
    }
    if (NG == 1) {
      sc[k][0] = cp[0];
      sc[k][J - 1] = cp[1];
    } else {
      sc[k][0] = cp[0] + cp[1];
      if (NG == 4) sc[k][0] += __shfl_xor_sync(0xffffffffu, sc[k][0], 1);
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if (!good || (2 * tig + j) / NG >= heads) sc[k][j] = kNegInf;
    }
  }
  float over = kNegInf;  // the largest excess over the lane's maxima
#pragma unroll
  for (int j = 0; j < J; ++j)
    over = fmaxf(over, fmaxf(fmaxf(sc[0][j], sc[1][j]), fmaxf(sc[2][j], sc[3][j])) - st.m[j]);
  if constexpr (!WIDE) {
    over -= st.lift;
    if (has_sz) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        big = fmaxf(big, fmaxf(__half2float(__ushort_as_half(zw[k][0] & 0xffff)), __half2float(__ushort_as_half(zw[k][1] & 0xffff))));
    }
    if (__any_sync(0xffffffffu, over > kGroupTau || (big > st.lim && (st.lift > 0.f || over > 0.f)))) {  // (the keys' lanes share a maximum)
      const float lift = st.lift;
      if (has_sz) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
        if (big > st.lim) {
          // big * 2^lift < 2^6, 2^3, 2^0 as in tile_weights, lift >= 0; 2^(lift + 3) * lim < 2^16
          const int e = 5 - 3 * st.cls - (static_cast<int>(__float_as_uint(big) >> 23) - 127);
          st.lift = static_cast<float>(max(0, min(static_cast<int>(lift), e)));
          st.lim = st.lift > 0.f ? __int_as_float((127 + 12 - static_cast<int>(st.lift)) << 23) : kGroupWide;
        }
      }
#pragma unroll
      for (int j = 0; j < J; ++j) {
        float mx = fmaxf(fmaxf(sc[0][j], sc[1][j]), fmaxf(sc[2][j], sc[3][j]));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mx = fmaxf(mx, __fadd_rd(st.m[j], lift));
        const float m = __fadd_ru(mx, -st.lift);  // rounded up: p <= 2^lift also where a score's ulp is larger
        const float alpha = fast_exp2(st.m[j] - m);
        st.m[j] = m;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (NG == 1 && i != j) continue;
          st.l[i] *= alpha;
          st.zacc[i] *= alpha;
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            st.acc[t][i] *= alpha;
            st.acc[t][i + 2] *= alpha;
          }
        }
        if (NG > 1) st.m[1] = st.m[0];
      }
    }
  } else {
    if (__any_sync(0xffffffffu, over > kGroupTau)) {  // (the keys' lanes share a maximum)
#pragma unroll
      for (int j = 0; j < J; ++j) {
        float mx = fmaxf(fmaxf(sc[0][j], sc[1][j]), fmaxf(sc[2][j], sc[3][j]));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mx = fmaxf(mx, st.m[j]);
        const float alpha = fast_exp2(st.m[j] - mx);
        st.m[j] = mx;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (NG == 1 && i != j) continue;
          float f = alpha;
          if (has_sz && alpha < pow2f(-12)) {  // little is left of what ws was chosen for
            f *= pow2f(kWeightScale) * pow2_inverse(st.ws[i]);
            st.ws[i] = pow2f(kWeightScale);
          }
          st.l[i] *= alpha;
          st.zacc[i] *= alpha;
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            st.acc[t][i] *= f;
            st.acc[t][i + 2] *= f;
          }
        }
        if (NG > 1) st.m[1] = mx;
      }
    }
    if (has_sz) {
      float big[2] = {0.f, 0.f};  // per column: the largest V scale of a key with weight
#pragma unroll
      for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float x = __half2float(__ushort_as_half(zw[k][j] & 0xffff));
          if (sc[k][J == 2 ? j : 0] - st.m[j] > kGroupWeight) big[j] = fmaxf(big[j], x);
        }
      }
      if (__any_sync(0xffffffffu, big[0] * st.ws[0] > kGroupTop || big[1] * st.ws[1] > kGroupTop)) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) big[j] = fmaxf(big[j], __shfl_xor_sync(0xffffffffu, big[j], o));
          // big * ws < 2^6, 2^3, 2^0 as in tile_weights
          const int e = 5 - 3 * st.cls - (static_cast<int>(__float_as_uint(big[j]) >> 23) - 127);
          const float ws = big[j] > 0.f ? __int_as_float((127 + min(kWeightScale, e)) << 23) : st.ws[j];
          const float f = ws * pow2_inverse(st.ws[j]);
          st.ws[j] = ws;
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            st.acc[t][j] *= f;
            st.acc[t][j + 2] *= f;
          }
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float p[2], w[2];
    p[0] = fast_exp2(sc[k][0] - st.m[0]);
    p[1] = NG == 1 ? fast_exp2(sc[k][J - 1] - st.m[1]) : p[0];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&zw[k][j]));
      st.l[j] += p[j];
      st.zacc[j] = fmaf(p[j], f.y, st.zacc[j]);
      w[j] = WIDE && has_sz ? p[j] * f.x * st.ws[j] : p[j] * f.x;
    }
    uint32_t* at = reinterpret_cast<uint32_t*>(wb + 16 * (gid + 8 * k)) + tig;
    if (has_sz) {  // high and low part (finite: p <= 1 where a scale is above kGroupWide, then lift is 0)
      const uint32_t hi = pack_f16x2(w[0], w[1]);
      const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&hi));
      at[0] = hi;
      at[128] = pack_f16x2(w[0] - h.x, w[1] - h.y);
    } else {
      const uint32_t hi = pack_bf16x2(w[0], w[1]);
      at[0] = hi;
      at[128] = pack_bf16x2(w[0] - bf_lo(hi), w[1] - bf_hi(hi));
    }
  }
}

// Infinite bf16 values (and NaN) as the largest finite ones.
__device__ __forceinline__ uint32_t finite_bf16x2(uint32_t x) {
  const uint32_t top = 0x7f7f7f7fu, low = 0xff7fff7fu;
  const __nv_bfloat162 m = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&x), *reinterpret_cast<const __nv_bfloat162*>(&top));
  const __nv_bfloat162 r = __hmax2(m, *reinterpret_cast<const __nv_bfloat162*>(&low));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// 3. P.V.  all[k]: lanes whose key gid + 8 k counts (width 16: other keys' values read as 0).
template <int D, int NG, int B, bool WIDE>
__device__ __forceinline__ void group_values(GroupState<D, NG, WIDE>& st, const uint8_t* tile, int kt, bool part,
                                             const unsigned (&all)[4], const uint8_t* wb, int lane) {
  constexpr int MT = D / 16, rowb = D * B / 8;
  constexpr int VB = D * B / 64, VW = VB >= 4 ? VB / 4 : 1;  // V bytes per lane and key (D/8 dims)
  constexpr int VH = VW > 4 ? VW / 4 : 1, VWH = VW / VH, MTH = MT / VH;
  const int gid = lane >> 2, tig = lane & 3;
  constexpr int MAP = WIDE ? row_map(D, B) : 0;
  const uint8_t* v0 = tile + kt * rowb;
  uint32_t w[4], wlo[4];
  ldmatrix4_trans(w, wb + st.wl);
  ldmatrix4_trans(wlo, wb + 512 + st.wl);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && kt == 16) break;
#pragma unroll
    for (int hf = 0; hf < VH; ++hf) {
      uint32_t x[4][VWH];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        load_words<VWH>(v0 + (WIDE ? v_off<D, B>(st.vl, 4 * u + i, hf) : st.vl + 4 * (4 * u + i) * rowb + 16 * hf), x[i]);
        if (VB < 4) x[i][0] >>= ((gid * VB) & 3) * 8;
        if (B == 16 && part) {
          const int key = v_key<MAP>(tig, 4 * u + i);  // its ok: lane 4 (key % 8)'s bit of all[key / 8]
          const unsigned bits = key & 16 ? (key & 8 ? all[3] : all[2]) : (key & 8 ? all[1] : all[0]);
          if (!((bits >> (4 * (key & 7))) & 1u)) {
#pragma unroll
            for (int y = 0; y < VWH; ++y) x[i][y] = 0u;
          }
        }
      }
#pragma unroll
      for (int t = 0; t < MTH; ++t) {
        const uint32_t a0 = v_pair<B>(x[0], x[1], 2 * t), a1 = v_pair<B>(x[0], x[1], 2 * t + 1);
        const uint32_t a2 = v_pair<B>(x[2], x[3], 2 * t), a3 = v_pair<B>(x[2], x[3], 2 * t + 1);
        mma_cls<B>(st.acc[hf * MTH + t], a0, a1, a2, a3, w[2 * u], w[2 * u + 1]);
        if (B == 16)  // an infinite value times a low part of 0 or below would make its sum a NaN
          mma_bf16(st.acc[hf * MTH + t], finite_bf16x2(a0), finite_bf16x2(a1), finite_bf16x2(a2), finite_bf16x2(a3),
                   wlo[2 * u], wlo[2 * u + 1]);
        else
          mma_f16(st.acc[hf * MTH + t], a0, a1, a2, a3, wlo[2 * u], wlo[2 * u + 1]);
      }
    }
  }
}

// The tensor core truncates its sums, and codes are not negative: running sums of p * s * c come
// out low by up to 2^-23 of themselves per 16 keys, and p * z, about as large with the other sign,
// leaves that in a row a hundred times smaller.  The zero points are therefore added every
// kFoldTiles tiles, so that the running sums stay near the row itself.  (8-bit tokens, 670 keys a
// split: 1.1e-4 of the row off before its rounding, 2.4e-5 so.  Batch 256 of the sweep 1576 us, 1524
// without; every 4 or 16 tiles takes as long.  Sums begun at zero for each tile, or codes made
// normal and centred, take 12 % more.)
constexpr int kFoldTiles = 8;
template <int D, int NG>
__device__ __forceinline__ void fold_zero_points(RowState<D, NG>& st, const float* fac, int lane) {
  constexpr int MT = D / 16;
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int i = 0; i < NG; ++i) st.zacc[i] += __shfl_xor_sync(0xffffffffu, st.zacc[i], o);
  }
  float z = lane_group<NG>(st.zacc, lane);
#pragma unroll
  for (int i = 0; i < NG; ++i) st.zacc[i] = 0.f;
  if (st.cls != 3) z *= lane_group<NG>(st.ws, lane);
  float f[2 * MT];
  load_words<2 * MT>(reinterpret_cast<const uint8_t*>(fac + (12 + st.cls) * (D / 8)), reinterpret_cast<uint32_t*>(f));
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    st.acc[t][0] = fmaf(z, f[2 * t], st.acc[t][0]);
    st.acc[t][2] = fmaf(z, f[2 * t + 1], st.acc[t][2]);
  }
}

template <int D, int NG>
__device__ __forceinline__ void fold_zero_points(GroupState<D, NG, true>& st, const float* fac, int lane) {
  constexpr int MT = D / 16;
  float f[2 * MT];
  load_words<2 * MT>(reinterpret_cast<const uint8_t*>(fac + (12 + st.cls) * (D / 8)), reinterpret_cast<uint32_t*>(f));
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    float z = st.zacc[j];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    st.zacc[j] = 0.f;
    if (st.cls != 3) z *= st.ws[j];
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      st.acc[t][j] = fmaf(z, f[2 * t], st.acc[t][j]);
      st.acc[t][j + 2] = fmaf(z, f[2 * t + 1], st.acc[t][j + 2]);
    }
  }
}

// --------------------------------------------------------------------------- rows --

// A partial: the sums (lane holds dims lane * D/32 ..), their maximum and the weights' sum.
template <int D>
__device__ __forceinline__ void store_partial(float* pp, const float (&v)[D / 32], float M, float L, int lane) {
  constexpr int DPL = D / 32;
#pragma unroll
  for (int j = 0; j < DPL; j += 2) __stcg(reinterpret_cast<float2*>(pp + lane * DPL + j), make_float2(v[j], v[j + 1]));
  if (lane == 0) __stcg(reinterpret_cast<float2*>(pp + D), make_float2(M, L));
}
// Adds one that this warp stored.
template <int D>
__device__ __forceinline__ void take_partial(const float* pp, float (&v)[D / 32], float& M, float& L, int lane) {
  constexpr int DPL = D / 32;
  const float2 ml = __ldcg(reinterpret_cast<const float2*>(pp + D));
  const float top = fmaxf(M, ml.x), f = fast_exp2(M - top), fp = fast_exp2(ml.x - top);
#pragma unroll
  for (int j = 0; j < DPL; ++j) v[j] = fmaf(v[j], f, fp * __ldcg(pp + lane * DPL + j));
  L = fmaf(L, f, fp * ml.y);
  M = top;
  __syncwarp();  // the sums are read before they are overwritten
}

// A row at its unit's end (lane holds dims lane * D/32 .. of the unnormalised sum, relative to
// max M, with weight sum L).  One split: the bf16 row.  Otherwise the split's fp32 partial,
// partial base + sp, merged in two levels: the last split of each group of kMergeGroup to
// arrive folds the group into its first partial, and the last group to arrive merges the
// groups into the row (one level when ns <= kMergeGroup).
template <int D>
__device__ __forceinline__ void store_row(const AttnKernelArgs& ka, float (&v)[D / 32], float M, float L, int sp, int qi,
                                          int qh, int ns, int base, int lane) {
  constexpr int DPL = D / 32;
  constexpr int64_t kRow = D + 4;
  const LayerArgs& a = ka.a;
  if (ns > 1) {
    float* p0 = a.part + static_cast<int64_t>(base) * kRow;  // the level's first partial
    int* counters = a.cnt + (static_cast<int64_t>(qi) * a.Hq + qh) * a.cnt_stride;
    const bool two = ns > kMergeGroup;
    const int gr = two ? sp / kMergeGroup : 0;
    int* counter = two ? counters + 1 + gr : counters;       // the group's arrivals, then the row's
    int count = two ? min(kMergeGroup, ns - gr * kMergeGroup) : ns, stride = 1;
    float* from = two ? p0 + gr * kMergeGroup * kRow : p0;
    float* pp = p0 + sp * kRow;
#pragma unroll 1
    for (int level = two ? 0 : 1; level < 2; ++level) {
      store_partial<D>(pp, v, M, L, lane);
      if (!arrive_last(counter, count, lane)) return;
      merge_partials<D>(from, kRow * stride, count, lane, M, L, v);
      __syncwarp();  // every lane has read the group's rows before the first is overwritten
      pp = from;
      from = p0;
      counter = counters;
      count = (ns + kMergeGroup - 1) / kMergeGroup;
      stride = kMergeGroup;
    }
  }
  __nv_bfloat162* out =
      reinterpret_cast<__nv_bfloat162*>(ka.out + (static_cast<int64_t>(qi) * a.Hq + qh) * D + lane * DPL);
  const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
  for (int j = 0; j < DPL; j += 2) out[j / 2] = __floats2bfloat162_rn(v[j] * inv, v[j + 1] * inv);
}

// The accumulators of a unit as lane's dims lane * D/32 .., with the zero points added.
template <int D, int NG>
__device__ __forceinline__ void row_values(RowState<D, NG>& st, float (&v)[D / 32], const float* fac, int lane) {
  constexpr int DPL = D / 32, MT = D / 16;
  const int gid = lane >> 2, tig = lane & 3, grp = gid * NG / 8;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    st.l += __shfl_xor_sync(0xffffffffu, st.l, o);
#pragma unroll
    for (int i = 0; i < NG; ++i) st.zacc[i] += __shfl_xor_sync(0xffffffffu, st.zacc[i], o);
  }
  float z = st.zacc[0];
#pragma unroll
  for (int i = 1; i < NG; ++i)
    if (grp == i) z = st.zacc[i];
  // dims gid D/8 + 2 t + r are in lane (gid, grp)'s acc[t][2 r] (hi) and [2 r + 1] (lo);
  // this lane wants t = tig DPL/2 ..
  const float g = st.cls == 3 ? 1.f : pow2_inverse(lane_group<NG>(st.ws, lane));
  float f[2 * MT];
  load_words<2 * MT>(reinterpret_cast<const uint8_t*>(fac + (st.cls * 4 + 3) * (D / 8)), reinterpret_cast<uint32_t*>(f));
#pragma unroll
  for (int t = 0; t < MT; ++t) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float inv = f[2 * t + r] * g;
      const float hi = st.acc[t][2 * r], lo = st.acc[t][2 * r + 1];
      // an infinite sum (16-bit values may be infinite) has no low part
      const float x = (fabsf(hi) <= 3.4028235e38f ? fmaf(lo, 1.f / kLoScale, hi) : hi) * inv;
      const float got = __shfl_sync(0xffffffffu, x, (lane & ~3) + grp);
      if (t / (DPL / 2) == tig) v[(t % (DPL / 2)) * 2 + r] = got + z;
    }
  }
}

// ----------------------------------------------------------------------- new token --

// Decode step: K or V row (raw: this lane's D/32 bf16 values) of entry e's KV head j at class
// c: stored to slot `slot` of page pid when `own`; x: the values as stored, in binary32.
template <int D>
__device__ __forceinline__ void step_row(const AttnKernelArgs& ka, uint2 raw, int kv, int j, int c, int pid, int slot,
                                         bool own, float (&x)[D / 32], int lane) {
  const LayerArgs& a = ka.a;
  const int P = a.P, b = bits_of_class(c), rowb = D * b / 8, ng = D >> (__ffs(a.G) - 1);
  uint8_t* sl = a.pool[c] + static_cast<int64_t>(pid) * a.page_bytes[c] + a.hdr + static_cast<int64_t>(j) * a.slice[c];
  const int64_t off = static_cast<int64_t>(kv * P + slot) * rowb;
  const bool sw = a.swz && b >= 8;
  if (b == 16) {
    x[0] = bf16lo(raw.x);
    x[1] = bf16hi(raw.x);
    if (D == 128) {
      x[D == 128 ? 2 : 0] = bf16lo(raw.y);
      x[D == 128 ? 3 : 1] = bf16hi(raw.y);
    }
    if (own) {
      const int64_t o = off + lane * (D / 16);
      uint8_t* dst = sl + (sw ? swz_off(o) : o);
      if (D == 64) *reinterpret_cast<uint32_t*>(dst) = raw.x;
      else *reinterpret_cast<uint2*>(dst) = raw;
    }
    return;
  }
  const RowCodes r = quantise_row_codes<D>(raw, b, a.G, lane, x);
  if (own) {
    const int64_t o = off + 4 * r.code_idx;
    if (r.code_idx >= 0) *reinterpret_cast<uint32_t*>(sl + (sw ? swz_off(o) : o)) = r.code_word;
    if (r.sz_idx >= 0)
      reinterpret_cast<uint32_t*>(sl + 2 * static_cast<int64_t>(P) * rowb + static_cast<int64_t>(kv * P + slot) * ng * 4)[r.sz_idx] =
          r.sz_word;
    if (__any_sync(0xffffffffu, r.bad) && lane == 0) set_status(a.ctrl, TRR_ERR_BAD_VALUE);
  }
}

// Every CTA: validates the entries and plans where each token goes (the same plan as the
// append kernels: the token takes index ntok of its (sequence, class) list; index % P == 0
// opens a page, whose id is next_page + the class's openers before it).  Errors, lowest
// entry first: sequence id, bit-width or mode not allowed, or a sequence named by an
// earlier entry (INVALID_ARG); position outside [0, max_context) or not above the
// sequence's last one (BAD_POSITION); a local query with a window below 1 (INVALID_ARG).
// Built with one thread per entry (n <= kStepMax threads).
__device__ __forceinline__ void plan_entries_cta(const AttnKernelArgs& ka, int* ent) {
  const LayerArgs& a = ka.a;
  const int n = ka.n, e = threadIdx.x, lane = e & 31, warp = e >> 5, H = 2 * n;
  static_assert(kStepMax <= 32 * kRowWarps, "one thread per entry");
  int* hs = ent + 2 * n;  // [H][2]: sequence + 1, lowest entry index naming it
  int* sc = ent + 6 * n;
#pragma unroll 1
  for (int i = e; i < 2 * H; i += 32 * kRowWarps) hs[i] = (i & 1) ? INT_MAX : 0;
  if (e < kSScalars) sc[e] = e == kSErr ? INT_MAX : 0;
  const bool act = e < n;
  int seq = -1, pos = 0, m = 0, b = 0, w = 0;
  if (act) {
    seq = ka.seq_ids[e];
    pos = ka.q_positions[e];
    m = ka.modes[e];
    b = ka.bits[e];
    w = ka.windows ? ka.windows[e] : ka.window_scalar;
  }
  const bool in = act && seq >= 0 && seq < a.S;
  const int c = b == 2 ? 0 : b == 4 ? 1 : b == 8 ? 2 : b == 16 ? 3 : -1;
  int last = -1, tok = -1, lp = -1;
  if (in) {
    last = a.last_pos[seq];
    if (c >= 0) {
      tok = a.ntok[seq * 4 + c];
      lp = a.lastpg[seq * 4 + c];
    }
  }
  __syncthreads();
  unsigned h = 0;
  if (in) {
    h = seq_hash(seq, H);
#pragma unroll 1
    for (int probe = 0; probe < H; ++probe) {
      const int old = atomicCAS(&hs[2 * h], 0, seq + 1);
      if (old == 0 || old == seq + 1) {
        atomicMin(&hs[2 * h + 1], e);
        break;
      }
      h = h + 1 == static_cast<unsigned>(H) ? 0u : h + 1;
    }
  }
  __syncthreads();
  int err = 0;
  if (act) {
    if (!in || c < 0 || m > TRR_MODE_FULL) err = TRR_ERR_INVALID_ARG;
    else if (pos < 0 || pos >= a.maxctx) err = TRR_ERR_BAD_POSITION;
    else if (hs[2 * h + 1] != e) err = TRR_ERR_INVALID_ARG;
    else if (pos <= last) err = TRR_ERR_BAD_POSITION;
    else if (m == TRR_MODE_LOCAL && w < 1) err = TRR_ERR_INVALID_ARG;
  }
  const bool stores = act && !err && (m != TRR_MODE_SKIP || a.skip_writes_kv);
  const bool opens = stores && tok % a.P == 0;
  if (act && err) atomicMin(&sc[kSErr], e * 16 + err);
  int before = 0, mine = 0;  // openers of the class in earlier lanes; of class `lane` in the warp
#pragma unroll
  for (int cc = 0; cc < kClasses; ++cc) {
    const unsigned bal = __ballot_sync(0xffffffffu, opens && c == cc);
    if (c == cc) before = __popc(bal & ((1u << lane) - 1u));
    if (lane == cc) mine = __popc(bal);
  }
  if (lane < kClasses && mine) atomicAdd(&sc[kSOpeners + lane], mine);
  __syncthreads();  // the hash is read no more
  if (act) {
    ent[2 * e] = stores ? tok : -1;
    hs[e] = lp;
  }
  if (n > 32 && lane < kClasses && 32 * warp < n) hs[n + 4 * warp + lane] = mine;
  __syncthreads();
  if (act) {
    if (opens)
#pragma unroll 1
      for (int w2 = 0; w2 < warp; ++w2) before += hs[n + 4 * w2 + c];
    ent[2 * e + 1] = (c & 3) | (opens ? 4 | (before << 3) : 0);
  }
  __syncthreads();
}

// The tiles of a unit's run of pages: their number, and per lane its tile's copy.
struct TilePlan {
  int T, skip;      // tiles; where the split's next run starts (plan_pages), 0: this is the last
  uint64_t src;     // the tile's page's slice of the unit's KV head
  uint32_t geo;     // class | keys << 2 | kMask | ring offset / 128 << 10 | first key / 16 << 20
  int bytes, cum;   // bytes to copy; ring bytes used from the run's start to the tile's end
};
// Bytes of a tile of kt keys: rows, scales, presence mask.
template <int D, int NG, bool HM>
__device__ __forceinline__ int tile_bytes(int cls, int kt) {
  const int b = bits_of_class(cls);
  return kt * (b == 16 ? 4 * D : 2 * (D * b / 8) + 8 * NG) + (HM ? 16 : 0);
}
template <int D, int NG, bool HM, bool STEP, bool RUNS>
__device__ __forceinline__ TilePlan plan_tiles(const AttnKernelArgs& ka, int seq, const RowUnit& un, int kvh, int skip, int lane) {
  const LayerArgs& a = ka.a;
  const int P = a.P, R = ka.ring_bytes;
  const int kt_most = min(P, 32), kt_wide = min(P, D == 128 ? 16 : 32);
  auto tile_keys = [&](int cls) { return D == 128 && cls == 3 ? kt_wide : kt_most; };
  TilePlan tp;
  tp.skip = skip;
  int wid = -1, wmeta = 0;
  tp.T = un.zero ? 0 : plan_pages<RUNS>(a, seq, un.lo, un.t, un.sp, un.ns, STEP, kt_most, kt_wide, lane, tp.skip, wid, wmeta);
  if (kt_wide < P || kt_most < P) {  // pages to tiles
    const int kt = tile_keys(wmeta & 3), nt = lane < tp.T ? (((wmeta >> 2) & 127) + kt - 1) / kt : 0;
    int incl = nt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    int page = 0, key0 = 0;
#pragma unroll 1
    for (int p = 0; p < tp.T; ++p) {
      const int e = __shfl_sync(0xffffffffu, incl, p), m = __shfl_sync(0xffffffffu, nt, p);
      if (lane >= e - m && lane < e) {
        page = p;
        key0 = lane - (e - m);
      }
    }
    tp.T = min(32, __shfl_sync(0xffffffffu, incl, 31));  // (as in plan_pages)
    wid = __shfl_sync(0xffffffffu, wid, page);
    const int pm = __shfl_sync(0xffffffffu, wmeta, page), k = tile_keys(pm & 3);
    key0 *= k;
    wmeta = (pm & ~(127 << 2)) | min(k, ((pm >> 2) & 127) - key0) << 2 | (key0 >> 4) << 20;
  }
  const int cls = wmeta & 3, rows = tile_bytes<D, NG, HM>(cls, tile_keys(cls)), posb = (wmeta & kMask) ? 4 * tile_keys(cls) : 0;
  const int need = ((rows + 127) & ~127) + ((posb + 127) & ~127);
  tp.src = 0;
  tp.cum = 0;
  if (lane < tp.T)
    tp.src = reinterpret_cast<uint64_t>(a.pool[cls] + static_cast<int64_t>(wid) * a.page_bytes[cls] + a.hdr +
                                      static_cast<int64_t>(kvh) * a.slice[cls]);
  tp.bytes = rows + posb;
  int off = 0, cum = 0, woff = 0;
#pragma unroll 1
  for (int j = 0; j < tp.T; ++j) {
    const int nd = __shfl_sync(0xffffffffu, need, j);
    if (off + nd > R) {
      cum += R - off;
      off = 0;
    }
    cum += nd;
    if (lane == j) {
      woff = off;
      tp.cum = cum;
    }
    off += nd;
  }
  tp.geo = static_cast<uint32_t>(wmeta) | static_cast<uint32_t>(woff >> 7) << 10;
  return tp;
}
// ------------------------------------------------------------------------- kernel --

template <int D, int NG, Kind K, bool STEP, bool RUNS>
__global__ void __launch_bounds__(32 * kRowWarps, 2) row_kernel(const __grid_constant__ AttnKernelArgs ka) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int DPL = D / 32;
  constexpr bool HM = K == kHeads, WIDE = K == kWide;
  constexpr bool GQ = K == kGroup || WIDE;  // the combine kernel merges a query's splits
  const LayerArgs& a = ka.a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = ka.n, P = a.P, R = ka.ring_bytes;
  const int g = a.Hq / a.Hkv, hmost = WIDE ? 8 / NG : GQ ? g : 1;  // query heads of a unit, at most
  const int blocks = WIDE ? (g + hmost - 1) / hmost : 1;           // units of a KV head's group
  const int rows = GQ ? a.Hkv * blocks : a.Hq;                     // units of a query's split
  const RowSmem lay(D, hmost, n, STEP, R);
  int* pre = reinterpret_cast<int*>(smem + lay.pre);
  int* ent = reinterpret_cast<int*>(smem + lay.ent);
  int* sc = ent + 6 * n;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + lay.flag);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + lay.full) + warp * kRowSlots;
  uint8_t* ring = smem + lay.ring + warp * R;
  uint8_t* qs = smem + lay.q + warp * RowSmem::row_q_bytes(D, hmost);
  float* fac = reinterpret_cast<float*>(smem + lay.fac);
#pragma unroll 1
  for (int i = threadIdx.x; i < 16 * (D / 8); i += 32 * kRowWarps) {
    const int j = i % (D / 8), from = i / (4 * (D / 8)), to = (i / (D / 8)) & 3;
    fac[i] = __int_as_float((127 + row_fac(to, j) - row_fac(from, j)) << 23);
  }
  uint8_t* wb = smem + lay.w + warp * RowSmem::row_w_bytes(GQ ? 2 : 1);
  if (threadIdx.x < kRowWarps * kRowSlots) mbar_init(reinterpret_cast<uint64_t*>(smem + lay.full) + threadIdx.x, 1);
  if (threadIdx.x == 0) *abort_flag = 0;
  if (RUNS && threadIdx.x < 2 * kRowWarps) reinterpret_cast<int*>(smem + lay.flag + 16)[threadIdx.x] = 0;
  fence_barrier_init();
  // The unit plan reads only the call's own index arrays, which no kernel of this library
  // writes, so it overlaps the previous kernel of the stream.  The layer's cache state is
  // read before the wait only when `early` says that no kernel still running can write it.
  int4* qinf = reinterpret_cast<int4*>(smem + lay.qinf);
  uint16_t* ord = reinterpret_cast<uint16_t*>(smem + lay.ord);
  plan_rows<HM, GQ>(ka, rows, pre, qinf, ord, reinterpret_cast<long long*>(smem + lay.red));
  bool waited = !(STEP && ka.early);
  if (waited) {
    pdl_wait();
    pdl_trigger();
  }
  const int total = pre[n], nwarps = gridDim.x * kRowWarps;

  // ------------------------------------------------------------------- unit and ring state
  // A unit's tiles (a page's keys, 32 at a time) are worked out once, one per lane (TilePlan): what
  // to copy, where in the ring, and how far the ring is used up to the tile's end (the ring
  // is filled and freed in tile order; a tile that would pass its end starts at 0).
  RowUnit un = {};
  uint64_t wsrc = 0;                  // lane j: tile j
  uint32_t wgeo = 0;
  int wbytes = 0, wcum = 0;
  uint32_t base = 0;                  // tiles of the units before
  int inext = 0;                      // next tile to issue
  bool good = true;                   // no wait gave up
  int kvh = 0;                        // the unit's KV head
  const int kt_most = min(P, 32), kt_wide = min(P, D == 128 ? 16 : 32);
  auto tile_keys = [&](int cls) { return D == 128 && cls == 3 ? kt_wide : kt_most; };
  auto tile_rows = [&](int cls) { return tile_bytes<D, NG, HM>(cls, tile_keys(cls)); };
  // RUNS: a split of more tiles than a warp plans at once (plan_pages) is worked on in runs, as one
  // unit after another: every run but the last leaves its sums as the split's partial, every run but
  // the first takes them up.  run[0]: where this run starts, run[1]: the next one (0: there is none).
  // (Kernels of their own for the caches that can meet one: a step with them in took 3 to 8 % longer.)
  int* run = reinterpret_cast<int*>(smem + lay.flag + 16) + 2 * warp;
  // issues the copies of the tiles that fit, each by its lane: tile c is the next to be
  // consumed, `freed` the ring bytes used up to the end of tile c - 1 (tile c itself always
  // fits: the ring is empty then)
  auto issue = [&](int c, int freed) {
    const bool can = lane >= inext && lane < min(un.T, c + kRowSlots) && (wcum - freed <= R || lane == c);
    inext += __popc(__ballot_sync(0xffffffffu, can));
    if (can) {
      const int cls = wgeo & 3, kt = tile_keys(cls);
      uint64_t* bar = &full[(base + lane) % kRowSlots];
      uint8_t* dst = ring + ((wgeo >> 3) & (1023u << 7));
      const uint8_t* sl = reinterpret_cast<const uint8_t*>(wsrc);
      mbar_arrive_expect_tx(bar, wbytes);
      const int posb = (wgeo & kMask) ? 4 * kt : 0, key0 = static_cast<int>(wgeo >> 20) << 4;
      if (kt == P) {  // the whole slice
        bulk_g2s(dst, sl, wbytes - posb, bar);
      } else {  // kt of the page's keys: K rows, V rows, their scales, the presence mask
        const int b = bits_of_class(cls), rowb = D * b / 8, szb = kt * NG * 4;
        bulk_g2s(dst, sl + key0 * rowb, kt * rowb, bar);
        bulk_g2s(dst + kt * rowb, sl + (P + key0) * rowb, kt * rowb, bar);
        if (b != 16) {
          bulk_g2s(dst + 2 * kt * rowb, sl + 2 * P * rowb + key0 * NG * 4, szb, bar);
          bulk_g2s(dst + 2 * kt * rowb + szb, sl + 2 * P * rowb + (P + key0) * NG * 4, szb, bar);
        }
        if (HM) bulk_g2s(dst + tile_rows(cls) - 16, sl + a.slice[cls] - 16, 16, bar);
      }
      if (posb) bulk_g2s(dst + ((tile_rows(cls) + 127) & ~127), sl - a.hdr - kvh * a.slice[cls] + 4 * key0, posb, bar);
    }
  };
  // waits for tile c's copies; false (and not good) when the wait gave up
  auto tile_in = [&](int c) -> bool {
    const uint32_t slot = (base + c) % kRowSlots, parity = ((base + c) / kRowSlots) & 1;
    bool arrived = mbar_test_at(smem_u32(&full[slot]), parity);
    if (!arrived) arrived = mbar_wait_slow(&full[slot], parity, abort_flag, a.wait_ns);
    good = __all_sync(0xffffffffu, arrived);  // give up together, never half a warp
    return good;
  };
  // the unit u: its query, head, split and pages
  auto plan = [&](int u) {
    int q = 0, span = n;  // the query's place: pre[q] <= u < pre[q + 1]
#pragma unroll 1
    while (span > 1) {
      const int step = (span + 31) >> 5, at = q + lane * step;
      q += (__popc(__ballot_sync(0xffffffffu, lane * step < span && pre[at] <= u)) - 1) * step;
      span = min(step, n - q);
    }
    const int4 qi = qinf[q];
    un.q = ord[q];
    un.t = qi.y;
    un.lo = qi.z;
    un.ns = qi.w & 0xffffff;
    un.err = (qi.w >> 24) & 15;
    un.zero = qi.w >> 28;
    const int r = u - pre[q];
    if (HM && !un.err) {
      // full heads first, then local, then skip ones: the k-th head of its mode
      HeadCounts c{0, 0, 0};
      const uint8_t* row = ka.modes + static_cast<int64_t>(un.q) * a.Hq;
#pragma unroll 1
      for (int h0 = 0; h0 < a.Hq; h0 += 32) {
        const int hm = h0 + lane < a.Hq ? row[h0 + lane] : -1;
        c.full += __popc(__ballot_sync(0xffffffffu, hm == TRR_MODE_FULL));
        c.local += __popc(__ballot_sync(0xffffffffu, hm == TRR_MODE_LOCAL));
      }
      const int nsf = un.ns;
      const int nsl = c.local ? splits_of(un.t + 1 - un.lo, pre[n + 1], a.split_keys, a.split_extra, a.split_most, a.s_cap) : 1;
      int k, first = 0, hmode;
      if (r < c.full * nsf) {
        hmode = TRR_MODE_FULL;
        un.lo = 0;
        un.sp = div24(r, c.full);
        k = r - un.sp * c.full;
      } else if (r < c.full * nsf + c.local * nsl) {
        first = c.full * nsf;
        hmode = TRR_MODE_LOCAL;
        un.ns = nsl;
        un.sp = div24(r - first, c.local);
        k = r - first - un.sp * c.local;
      } else {
        first = c.full * nsf + c.local * nsl;
        hmode = TRR_MODE_SKIP;
        un.ns = 1;
        un.sp = 0;
        k = r - first;
      }
      un.base = pre[q] + first + k * un.ns;
      un.h = 0;
#pragma unroll 1
      for (int h0 = 0; h0 < a.Hq; h0 += 32) {
        const int hm = h0 + lane < a.Hq ? row[h0 + lane] : -1;
        const unsigned same = __ballot_sync(0xffffffffu, hm == hmode);
        const int cnt = __popc(same);
        const unsigned hit =
            __ballot_sync(0xffffffffu, hm == hmode && __popc(same & ((1u << lane) - 1u)) == k);  // its k-th
        if (hit) un.h = h0 + __ffs(hit) - 1;
        k -= cnt;
        if (k < 0) break;
      }
      un.zero = hmode == TRR_MODE_SKIP;
    } else {
      un.sp = div24(r, rows);
      un.h = r - un.sp * rows;
      // (wide groups: the units of the queries before are `rows` for each of their splits)
      un.base = WIDE ? pre[q] / rows * a.Hq : (pre[q] + un.h * un.ns) * hmost;
    }
    kvh = WIDE ? div24(un.h, blocks) : GQ || g == 1 ? un.h : div24(un.h, g);
    if (WIDE) un.base += (kvh * g + (un.h - kvh * blocks) * hmost) * un.ns;
    const TilePlan tp = plan_tiles<D, NG, HM, STEP, RUNS>(ka, qi.x, un, kvh, RUNS ? run[0] : 0, lane);
    un.T = tp.T;
    wsrc = tp.src;
    wgeo = tp.geo;
    wbytes = tp.bytes;
    wcum = tp.cum;
    if (RUNS) {
      __syncwarp();
      if (lane == 0) run[1] = tp.skip;
    }
    inext = 0;
    // a limit shorter than a suspended wait covers the first copies from before they are issued
    // (from after it, instructions not yet fetched may take as long as the copies)
    const bool brief = a.wait_ns < kShortWaitNs;
    const uint64_t t0 = brief ? global_ns() : 0;
    issue(0, 0);
    if (brief && un.T > 0) {
      const uint32_t bar = smem_u32(&full[base % kRowSlots]);
      bool in = false;
      while (!in && global_ns() - t0 < a.wait_ns) in = mbar_test_at(bar, (base / kRowSlots) & 1);
      good = __all_sync(0xffffffffu, in);
    }
  };

  // The first unit is planned and its copies issued before the rest of the call's start.
  // Units that do not fill half of the CTAs, one per SM, are dealt evenly to these; more fill
  // CTA after CTA, which leaves places for the next layer's kernel.  (Head size 128, batch 8, 2 steps
  // of 12 layers 392 us, 420 without the deal; a group of 4, batch 8, 440 and 466.  Dealing up to
  // a unit per warp evenly to all CTAs: the 160M steps 847 in place of 796, pages of 16 418 for 367.)
  const int cta = static_cast<int>(blockIdx.x), half = (gridDim.x + 1) / 2;
  int per = kRowWarps, more = 0;
  if (total < half * kRowWarps) {
    per = div24(total, half);
    more = total - per * half;
    if (cta >= half) per = more = 0;
  }
  int u = warp < per + (cta < more) ? cta * per + min(cta, more) + warp : total;
  int consumed = 0;      // tiles of the unit
  int next_page = 0;     // decode step: the pools' counters (lanes 0 .. 3)
  bool failed = false;   // and whether the call fails (it then stores nothing, and the last
                         // CTA zeroes every row)
  bool started = false;
#pragma unroll 1
  for (;;) {
    if (u < total && good) plan(u);
    const bool first = !started;
    if (first) {
      started = true;
      if (STEP) plan_entries_cta(ka, ent);
      if (!waited) {
        pdl_wait();
        pdl_trigger();
      }
      if (STEP) {
        next_page = lane < 4 ? a.ctrl[kNextPage + lane] : 0;
        const int lim = lane == 0 ? a.cap[0] : lane == 1 ? a.cap[1] : lane == 2 ? a.cap[2] : a.cap[3];
        failed = sc[kSErr] != INT_MAX || __any_sync(0xffffffffu, lane < 4 && sc[kSOpeners + (lane & 3)] > 0 &&
                                                                      next_page + sc[kSOpeners + (lane & 3)] > lim);
      }
    }
    if (GQ && ka.defer_merge && first && blockIdx.x == 0) {  // for the combine kernel: a query's first partial, splits
      int2* qtab = reinterpret_cast<int2*>(a.qtab);
#pragma unroll 1
      for (int k = threadIdx.x; k < n; k += 32 * kRowWarps) qtab[ord[k]] = make_int2(WIDE ? pre[k] / rows * a.Hq : pre[k] * hmost, qinf[k].w & 0xffffff);
    }
    if (u >= total || !good) break;
    if (RUNS) __syncwarp();
    const bool last_run = !RUNS || run[1] == 0;
    int u_next = total;
    if (total > nwarps && lane == 0 && last_run) u_next = nwarps + atomicAdd(&a.lctl[kNextUnit], 1);  // read at the unit's end
    const int blk = WIDE ? un.h - kvh * blocks : 0;
    const int heads = WIDE ? min(hmost, g - blk * hmost) : hmost;  // of the unit, from h0 on
    const int h0 = WIDE ? kvh * g + blk * hmost : un.h * hmost;
    const bool own = WIDE ? blk == 0 : GQ || un.h == kvh * g;  // stores a new token's rows of its KV head
    // decode step: the entry's own token joins the row's last split; a skip token that
    // stores KV is written by its zero row's unit
    const bool has_new = STEP && !failed && last_run && un.sp == un.ns - 1 && ent[2 * un.q] >= 0 && (!un.zero || own);
    uint2 rk = make_uint2(0, 0), rv = rk;
    if (has_new) {
      const int64_t src = (static_cast<int64_t>(un.q) * a.Hkv + kvh) * D;
      rk = load_row<D>(ka.k + src, lane);
      rv = load_row<D>(ka.v + src, lane);
    }
    const int64_t qrow = (static_cast<int64_t>(un.q) * a.Hq + h0) * D;  // its first head's
    uint2 qraw = make_uint2(0, 0);
    if (!GQ && !un.zero) qraw = load_row<D>(ka.q + qrow, lane);
    float kx[DPL] = {}, vx[DPL] = {}, new_score = kNegInf;
    if (has_new) {
      const int tok = ent[2 * un.q], info = ent[2 * un.q + 1], c = info & 3;
      const int np = __shfl_sync(0xffffffffu, next_page, c);
      const int pid = (info & 4) ? np + (info >> 3) : ent[2 * n + un.q];
#pragma unroll 1
      for (int kv = 0; kv < 2; ++kv) {  // one copy of the quantiser (its code runs once a unit)
        float y[DPL];
        step_row<D>(ka, kv ? rv : rk, kv, kvh, c, pid, tok % P, own, y, lane);
#pragma unroll
        for (int j = 0; j < DPL; ++j) {
          kx[j] = kv ? kx[j] : y[j];
          vx[j] = y[j];
        }
      }
    }
    if (un.zero) {
      if (un.sp == 0) {
        uint32_t* o = reinterpret_cast<uint32_t*>(ka.out + qrow);
#pragma unroll 1
        for (int i = lane; i < heads * D / 2; i += 32) o[i] = 0u;
      }
      if (!STEP && un.err && un.sp == 0 && lane == 0) atomicMin(&a.lctl[kFirstBadQuery], (ka.q0 + un.q) * 16 + un.err);
    } else if constexpr (GQ) {
      // the group's query rows to shared memory; each column's sum and largest exponent
      GroupState<D, NG, WIDE> st;
      const int gid = lane >> 2, tig = lane & 3;
      float new_score[2] = {kNegInf, kNegInf};
      st.E = -85;
      st.qsum[0] = st.qsum[1] = 0.f;
      constexpr int kMost = 8 / NG;  // heads of a group, at most
      uint2 raws[kMost];
#pragma unroll
      for (int r = 0; r < kMost; ++r)
        raws[r] = r < heads ? load_row<D>(ka.q + qrow + r * D, lane) : make_uint2(0, 0);
#pragma unroll
      for (int r = 0; r < kMost; ++r) {
        if (r >= heads) break;
        const uint2 raw = raws[r];
        float x[DPL], sum = 0.f, dot = 0.f, qmax = 0.f;
        x[0] = bf_lo(raw.x);
        x[1] = bf_hi(raw.x);
        if (D == 128) {
          x[D == 128 ? 2 : 0] = bf_lo(raw.y);
          x[D == 128 ? 3 : 1] = bf_hi(raw.y);
          reinterpret_cast<uint2*>(qs + r * D * 2)[lane] = raw;
        } else {
          reinterpret_cast<uint32_t*>(qs + r * D * 2)[lane] = raw.x;
        }
#pragma unroll
        for (int j = 0; j < DPL; ++j) {
          qmax = fmaxf(qmax, fabsf(x[j]));
          sum += x[j];
          dot = fmaf(x[j], kx[j], dot);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          if (o < 32 / NG) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if (o < 32 / NG) qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, o));
          dot += __shfl_xor_sync(0xffffffffu, dot, o);
        }
        qmax = __shfl_sync(0xffffffffu, qmax, (gid % NG) * (32 / NG));
        if (gid / NG == r) st.E = max(-85, static_cast<int>((__float_as_uint(qmax) >> 23) & 0xff) - 127);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float v = __shfl_sync(0xffffffffu, sum, ((2 * tig + j) % NG) * (32 / NG));
          if ((2 * tig + j) / NG == r) {
            st.qsum[j] = v * ka.qscale;
            new_score[j] = has_new ? dot * ka.qscale : kNegInf;
          }
        }
      }
      st.cls = 3;
      st.lift = WIDE ? 0.f : kLift;
      st.lim = pow2f(12 - static_cast<int>(kLift));
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        st.m[j] = kNoMax;
        st.l[j] = st.zacc[j] = 0.f;
        st.ws[j] = pow2f(kWeightScale);
      }
#pragma unroll
      for (int t = 0; t < D / 16; ++t) st.acc[t][0] = st.acc[t][1] = st.acc[t][2] = st.acc[t][3] = 0.f;
      __syncwarp();
      int c = 0;  // next tile to consume
#pragma unroll 1
      for (; c < un.T; ++c) {
        const uint32_t geo = __shfl_sync(0xffffffffu, wgeo, c);
        const int cls = geo & 3, kt = tile_keys(cls);
        if (c == 0 || cls != st.cls) group_switch<D, NG, WIDE>(st, cls, c == 0, qs, heads, fac, ka.qscale, kt, lane);
        if (!tile_in(c)) break;
        const uint8_t* tile = ring + ((geo >> 3) & (1023u << 7));
        const int fill = (geo >> 2) & 127;
        unsigned ok = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) ok |= static_cast<unsigned>(gid + 8 * k < fill) << k;
        if (geo & kMask) {
          const int* pos = reinterpret_cast<const int*>(tile + ((tile_rows(cls) + 127) & ~127));
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int p = pos[min(gid + 8 * k, kt - 1)];
            if (p < un.lo || p > un.t) ok &= ~(1u << k);
          }
        }
        float sc[2][4] = {};
        switch (cls) {
          case 0: group_scores<D, NG, 2, WIDE>(st, tile, kt, sc); break;
          case 1: group_scores<D, NG, 4, WIDE>(st, tile, kt, sc); break;
          case 2: group_scores<D, NG, 8, WIDE>(st, tile, kt, sc); break;
          default: group_scores<D, NG, 16, WIDE>(st, tile, kt, sc); break;
        }
        group_weights<D, NG, WIDE>(st, sc, ok, cls != 3, tile + st.zoff, kt, heads, wb, lane);
        unsigned all[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) all[k] = __ballot_sync(0xffffffffu, (ok >> k) & 1u);
        __syncwarp();
        switch (cls) {
          case 0: group_values<D, NG, 2, WIDE>(st, tile, kt, false, all, wb, lane); break;
          case 1: group_values<D, NG, 4, WIDE>(st, tile, kt, false, all, wb, lane); break;
          case 2: group_values<D, NG, 8, WIDE>(st, tile, kt, false, all, wb, lane); break;
          default: group_values<D, NG, 16, WIDE>(st, tile, kt, fill < kt || (geo & kMask), all, wb, lane); break;
        }
        __syncwarp();  // the tile's bytes and weights are read
        if (inext < un.T) issue(c + 1, __shfl_sync(0xffffffffu, wcum, c));
        if constexpr (WIDE) {
          if (c % kFoldTiles == kFoldTiles - 1) fold_zero_points<D, NG>(st, fac, lane);
        }
      }
      consumed = c;
      if (!good) break;
      // the heads' rows: lane (gid, tig) has dims gid D/8 .. of the columns whose group they are in
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          st.l[j] += __shfl_xor_sync(0xffffffffu, st.l[j], o);
          st.zacc[j] += __shfl_xor_sync(0xffffffffu, st.zacc[j], o);
        }
      }
      float* vnew = reinterpret_cast<float*>(wb);  // the new token's V row
      if (has_new) {
#pragma unroll
        for (int j = 0; j < DPL; ++j) vnew[lane * DPL + j] = vx[j];
      }
      __syncwarp();
      float f[D / 8];
      load_words<D / 8>(reinterpret_cast<const uint8_t*>(fac + (st.cls * 4 + 3) * (D / 8)), reinterpret_cast<uint32_t*>(f));
      float2 old[2];  // an earlier run's maximum and sum of the lane's columns
      if (RUNS) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          old[j] = make_float2(kNegInf, 0.f);
          if (run[0] && (2 * tig + j) / NG < heads)
            old[j] = __ldcg(reinterpret_cast<const float2*>(
                a.part + static_cast<int64_t>(un.base + (2 * tig + j) / NG * un.ns + un.sp) * (D + 4) + D));
        }
        __syncwarp();
      }
      auto finish = [&](auto column) {
        constexpr int j = decltype(column)::value;
        const int r = (2 * tig + j) / NG, gi = (2 * tig + j) % NG;
        const float g = st.cls == 3 ? 1.f : pow2_inverse(st.ws[j]);
        float M = st.m[j], L = st.l[j], fo = 1.f, fn = 0.f;
        if (has_new) {  // fold the new token in
          M = fmaxf(st.m[j], new_score[j]);
          fo = fast_exp2(st.m[j] - M);
          fn = fast_exp2(new_score[j] - M);
          L = fmaf(L, fo, fn);
        }
        if (r >= heads || gid * NG / 8 != gi) return;
        auto partial = [&] { return a.part + static_cast<int64_t>(un.base + r * un.ns + un.sp) * (D + 4); };
        float fp = 0.f;
        if (RUNS && run[0]) {
          const float top = fmaxf(M, old[j].x), d = fast_exp2(M - top);
          fp = fast_exp2(old[j].x - top);
          L = fmaf(L, d, fp * old[j].y);
          fo *= d;
          fn *= d;
          M = top;
        }
        const bool part = un.ns > 1 || !last_run;
        const float inv = part ? 1.f : L > 0.f ? 1.f / L : 0.f;
        float y[D / 8];
#pragma unroll
        for (int i = 0; i < D / 8; ++i) {
          float v = fmaf(st.acc[i / 2][2 * (i % 2) + j], WIDE ? f[i] * g : f[i], st.zacc[j]) * fo;
          if (has_new) v = fmaf(fn, vnew[gid * (D / 8) + i], v);
          if (RUNS && run[0]) v = fmaf(fp, __ldcg(partial() + gid * (D / 8) + i), v);
          y[i] = v * inv;
        }
        if (!part) {
          uint4* o = reinterpret_cast<uint4*>(ka.out + qrow + r * D + gid * (D / 8));
#pragma unroll
          for (int i = 0; i < D / 8; i += 8)
            o[i / 8] = make_uint4(pack_bf16x2(y[i], y[i + 1]), pack_bf16x2(y[i + 2], y[i + 3]), pack_bf16x2(y[i + 4], y[i + 5]),
                                  pack_bf16x2(y[i + 6], y[i + 7]));
        } else {  // the split's partial; the combine kernel merges them
          float* pp = partial();
#pragma unroll
          for (int i = 0; i < D / 8; i += 4)
            *reinterpret_cast<float4*>(pp + gid * (D / 8) + i) = make_float4(y[i], y[i + 1], y[i + 2], y[i + 3]);
          if (gid == 0) *reinterpret_cast<float2*>(pp + D) = make_float2(M, L);  // (group 0's column)
        }
      };
      finish(std::integral_constant<int, 0>());
      finish(std::integral_constant<int, 1>());
      __syncwarp();  // vnew is read
    } else {
      // the query row's largest exponents and sums per group
      float x[DPL];
      x[0] = bf_lo(qraw.x);
      x[1] = bf_hi(qraw.x);
      if (D == 128) {
        x[D == 128 ? 2 : 0] = bf_lo(qraw.y);
        x[D == 128 ? 3 : 1] = bf_hi(qraw.y);
      }
      float qmax = 0.f, qsum = 0.f, dot = 0.f;
#pragma unroll
      for (int j = 0; j < DPL; ++j) {
        qmax = fmaxf(qmax, fabsf(x[j]));
        qsum += x[j];
        if (has_new) dot = fmaf(x[j], kx[j], dot);
      }
      const int gl = 32 / NG;  // lanes of a group
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (o < gl) qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, o));
        if (o < gl) qsum += __shfl_xor_sync(0xffffffffu, qsum, o);
      }
      RowState<D, NG> st;
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        st.qsum[i] = __shfl_sync(0xffffffffu, qsum, i * gl) * ka.qscale;
        st.zacc[i] = 0.f;
        st.ws[i] = pow2f(kWeightScale);
      }
      if (has_new) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        new_score = dot * ka.qscale;
      }
      if (D == 64) reinterpret_cast<uint32_t*>(qs + 2 * D)[lane] = qraw.x;
      else reinterpret_cast<uint2*>(qs + 2 * D)[lane] = qraw;
      if (lane % gl == 0)
        reinterpret_cast<int*>(qs + 4 * D)[lane / gl] = max(-85, static_cast<int>((__float_as_uint(qmax) >> 23) & 0xff) - 127);
      st.m = kNoMax;
      st.l = 0.f;
      st.cls = 3;
#pragma unroll
      for (int t = 0; t < D / 16; ++t) st.acc[t][0] = st.acc[t][1] = st.acc[t][2] = st.acc[t][3] = 0.f;
      __syncwarp();
      int c = 0;  // next tile to consume
#pragma unroll 1
      for (; c < un.T; ++c) {
        const uint32_t geo = __shfl_sync(0xffffffffu, wgeo, c);
        const int cls = geo & 3, kt = tile_keys(cls);
        if (c == 0 || cls != st.cls) row_switch<D, NG>(st, cls, c == 0, qs, fac, ka.qscale, kt, lane);
        if (!tile_in(c)) break;
        const uint8_t* tile = ring + ((geo >> 3) & (1023u << 7));
        uint32_t there = 0xffffffffu;
        if (HM) {  // the KV head's presence mask, which ends the tile's rows
          const uint2 m2 = *reinterpret_cast<const uint2*>(tile + tile_rows(cls) - 16);
          there = static_cast<uint32_t>(((static_cast<uint64_t>(m2.y) << 32) | m2.x) >> ((geo >> 20) << 4));
        }
        uint32_t kw[NG], zw[NG];
#pragma unroll
        for (int i = 0; i < NG; ++i) kw[i] = zw[i] = 0x3c00u;  // s = 1, z = 0
        if (cls != 3) {
          load_words<NG>(tile + st.zoff - kt * NG * 4, kw);
          load_words<NG>(tile + st.zoff, zw);
        }
        float gs[NG];
        switch (cls) {
          case 0: tile_scores<D, NG, 2>(st, tile, kt, gs, lane); break;
          case 1: tile_scores<D, NG, 4>(st, tile, kt, gs, lane); break;
          case 2: tile_scores<D, NG, 8>(st, tile, kt, gs, lane); break;
          default: tile_scores<D, NG, 16>(st, tile, kt, gs, lane); break;
        }
        const int key = 8 * (lane & 3) + (lane >> 2);
        bool ok = key < ((geo >> 2) & 127) && ((there >> key) & 1u);
        if (geo & kMask) {  // the page may hold keys outside [lo, t]: positions follow the rows
          const int pos = reinterpret_cast<const int*>(tile + ((tile_rows(cls) + 127) & ~127))[min(key, kt - 1)];
          ok = ok && pos >= un.lo && pos <= un.t;
        }
        const unsigned all = __ballot_sync(0xffffffffu, ok);
        tile_weights<D, NG>(st, gs, ok, cls != 3, kw, zw, key, wb, lane);
        __syncwarp();
        if (cls == 3) {
          tile_values16<D, NG>(st, tile, kt, all != (kt == 32 ? 0xffffffffu : 0x33333333u), all, wb, lane);
        } else {
          switch (cls) {
            case 0: tile_values<D, NG, 2>(st, tile, kt, wb, lane); break;
            case 1: tile_values<D, NG, 4>(st, tile, kt, wb, lane); break;
            default: tile_values<D, NG, 8>(st, tile, kt, wb, lane); break;
          }
        }
        __syncwarp();  // the tile's bytes and weights are read
        if (inext < un.T) issue(c + 1, __shfl_sync(0xffffffffu, wcum, c));
        if (c % kFoldTiles == kFoldTiles - 1) fold_zero_points<D, NG>(st, fac, lane);
      }
      consumed = c;
      if (!good) break;
      float v[DPL];
      row_values<D, NG>(st, v, fac, lane);
      float M = st.m, L = st.l;
      if (has_new) {  // fold the new token in
        M = fmaxf(st.m, new_score);
        const float f = fast_exp2(st.m - M), fn = fast_exp2(new_score - M);
        L = fmaf(L, f, fn);
#pragma unroll
        for (int j = 0; j < DPL; ++j) v[j] = fmaf(v[j], f, fn * vx[j]);
      }
      if (RUNS) {
        float* pp = a.part + static_cast<int64_t>(un.base + un.sp) * (D + 4);
        if (run[0]) take_partial<D>(pp, v, M, L, lane);
        if (run[1]) store_partial<D>(pp, v, M, L, lane);
      }
      if (last_run) store_row<D>(ka, v, M, L, un.sp, un.q, un.h, un.ns, un.base, lane);
    }
    base += un.T;
    un.T = inext = consumed = 0;
    if (RUNS) {
      __syncwarp();
      const int next = run[1];
      __syncwarp();
      if (lane == 0) run[0] = next;
      __syncwarp();
      if (next) continue;
    }
    u = __shfl_sync(0xffffffffu, u_next, 0);
  }
  if (!good) {  // a wait gave up: stop the CTA's warps, then let this one's copies land
    if (lane == 0) {
      *abort_flag = 1;
      set_status(a.ctrl, TRR_ERR_TIMEOUT);
    }
    // copies in flight always land (they only read memory): the default bound
#pragma unroll 1
    for (uint32_t s = base + consumed; s < base + inext; ++s) mbar_wait(&full[s % kRowSlots], (s / kRowSlots) & 1);
  }

  // The last CTA to finish records the error of the lowest failing query, readies the
  // layer's counters for the next call and, for a decode step, commits the tokens' metadata.
  // Its arrival tells it all: the count of CTAs, with 2^16 added by each that gave up a wait.
  __shared__ int s_done;
  __syncthreads();
  if (threadIdx.x == 0) s_done = atom_add_acq_rel(&a.lctl[kDoneCtas], *abort_flag ? 0x10001 : 1) + (*abort_flag ? 0x10001 : 1);
  if (STEP && warp == 0) {
    if (lane < 4) sc[kSNextPage + lane] = next_page;
    __syncwarp();
    step_pages_error(ka, ent, lane);
  }
  __syncthreads();
  const int done = s_done;
  if ((done & 0xffff) != static_cast<int>(gridDim.x)) return;
  if (threadIdx.x == 0) {
    a.lctl[kDoneCtas] = 0;
    a.lctl[kNextUnit] = 0;
    if (!STEP) {
      const int bad = atomicExch(&a.lctl[kFirstBadQuery], INT_MAX);
      if (bad != INT_MAX) set_status(a.ctrl, bad & 15);
    }
  }
  if (!STEP) return;
  if (sc[kSErr] != INT_MAX) {  // a call error: every row zero
    uint4* o = reinterpret_cast<uint4*>(ka.out);
    const int64_t n16 = static_cast<int64_t>(n) * a.Hq * D / 8;
#pragma unroll 1
    for (int64_t i = threadIdx.x; i < n16; i += blockDim.x) o[i] = make_uint4(0, 0, 0, 0);
    if (GQ && ka.defer_merge) {  // nothing to merge
      int2* qtab = reinterpret_cast<int2*>(a.qtab);
#pragma unroll 1
      for (int q = threadIdx.x; q < n; q += blockDim.x) qtab[q] = make_int2(0, 1);
    }
  }
  if (done < 0x10000) step_commit(ka, ent);  // a call that gave up a wait stores nothing
}

// ------------------------------------------------------------------------- launch --
// A kernel family (compiled side by side, one translation unit each): launches the instance of a
// layout's head size and groups per head, and sets its shared-memory limit.

template <Kind K, bool STEP, bool RUNS>
auto row_instance(const Layout& l) {
  using Kernel = void (*)(AttnKernelArgs);
  const int ng = l.d / l.G;
  if (l.d == 64) return ng == 1 ? Kernel(row_kernel<64, 1, K, STEP, RUNS>) : Kernel(row_kernel<64, 2, K, STEP, RUNS>);
  return ng == 1   ? Kernel(row_kernel<128, 1, K, STEP, RUNS>)
         : ng == 2 ? Kernel(row_kernel<128, 2, K, STEP, RUNS>)
                   : Kernel(row_kernel<128, 4, K, STEP, RUNS>);
}
template <Kind K, bool STEP, bool RUNS>
cudaError_t launch_rows(const Layout& l, dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  return launch_pdl(row_instance<K, STEP, RUNS>(l), grid, dim3(32 * kRowWarps), smem, s, k);
}
template <Kind K, bool STEP, bool RUNS>
cudaError_t configure_rows(const Layout& l) {
  return cudaFuncSetAttribute(reinterpret_cast<const void*>(row_instance<K, STEP, RUNS>(l)),
                              cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemLimit);
}
#define TRR_ROW_FAMILY(prefix, K, STEP, RUNS)                                                                        \
  prefix template cudaError_t launch_rows<K, STEP, RUNS>(const Layout&, dim3, size_t, cudaStream_t,                  \
                                                         const AttnKernelArgs&);                                     \
  prefix template cudaError_t configure_rows<K, STEP, RUNS>(const Layout&);

}  // namespace trr
