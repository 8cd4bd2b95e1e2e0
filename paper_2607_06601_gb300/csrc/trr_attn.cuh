#pragma once
// trr_attn.cuh - what the attention kernels of trr_decode_attn and trr_decode_step share:
// mode-routed split-K decode attention over the mixed-precision paged cache (Sec. 3.2(A),
// Eq. 2; Sec. 3.8; Sec. 7).  trr_row.cuh holds the kernel; here are its arguments, a query's
// mode, range and errors, a decode step's token bookkeeping, the operands of the tensor-core
// products, the merge of split partials and the combine kernel of query groups.
//
// One persistent kernel per call cuts it into work units: a query gets splits from the length
// of its key range (full: [0, t]; local: [t-w+1, t]; skip or invalid: one that writes the zero
// rows), and a unit is a split of a query head, or of a KV head and its query group.  The same
// deterministic computation in every CTA takes the place of a planning kernel.  A query with
// one split gets its bf16 rows from that unit; otherwise splits write binary32 partials, which
// the last arrival merges (query heads) or the combine kernel (query groups).  The last CTA to
// finish records the error of the lowest failing query.
//
// Per-head modes (a cache with head_modes): each head has its own range, splits and units;
// every slice of a page ends with its KV head's presence mask, which is applied per key; a
// skip head writes its zero row.
#include <algorithm>
#include <climits>

#include "trr_internal.cuh"

namespace trr {

#define kNegInf (-__int_as_float(0x7f800000))
constexpr float kNoMax = -3.4028235e38f;  // a running maximum before the first key: no score is below
                                          // it, and finite (a key that does not count weighs 0)
constexpr float kTau = 8.f;    // lazy rescale threshold (log2 units)

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// exact 2^e, -126 <= e <= 127 (folds to a constant for constant e)
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// 2^x with the hardware approximation (relative error about 2^-22; results below the
// binary32 normal range flush to zero, far below a softmax sum's resolution).
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A shared-memory load at a 32-bit shared address (volatile: it is not kept from a loop).
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// -------------------------------------------------------------------- kernel --

constexpr int kMask = 1 << 9;  // a page's flag: it may hold keys outside the range

struct AttnKernelArgs {
  LayerArgs a;
  int n;                       // queries of the call
  const int32_t* seq_ids;
  const int32_t* q_positions;
  const uint8_t* modes;        // per-query modes, or null: mode_logits
  const float* mode_logits;    // [n][3] router logits (skip, local, full), or null
  const int32_t* windows;      // per-query windows, or null: window_scalar
  int window_scalar;
  const uint16_t* q;
  uint16_t* out;
  float qscale;      // softmax scale * log2(e)
  int q0;            // index of the launch's first query in the call (error reports)
  int ring_bytes;    // bytes of a warp's ring of shared memory
  int defer_merge;   // 1: split partials are merged by the combine kernel (query groups)
  int early;         // 1: the layer's cache state may be read before the previous kernel ends
  int fused;         // 1: a decode step: entry i appends its token (k, v, bits), then query i
                     // attends at the same position with the same mode
  const uint16_t* k;      // fused: K rows [n][Hkv][d] (bf16)
  const uint16_t* v;      // fused: V rows [n][Hkv][d] (bf16)
  const uint8_t* bits;    // fused: bit-widths [n]
};

// Fused decode step: the per-entry table every CTA builds in shared memory (2 ints per
// entry: the entry's token index in its (sequence, class) list, or -1 when it stores
// nothing; class | opens << 2 | openers of the class before it << 3), a hash of the
// entries' sequences (2 slots per entry: sequence + 1, lowest entry index; once the
// entries are checked, its first n ints hold the page of each token that goes into its
// class's last page), then the call's scalars.
constexpr int kStepMax = 256;  // entries of one decode-step call, at most
enum StepScalar : int {
  kSNextPage = 0,   // [4] pages handed out per class before the call (read after the wait)
  kSOpeners = 4,    // [4] entries opening a page, per class
  kSErr = 8,        // lowest failing entry * 16 + error, INT_MAX = none
  kSScalars = 16
};
__host__ __device__ constexpr int step_ints(int n) { return 2 * n + 4 * n + kSScalars; }

// Mode of query q: the caller's, or the hard decision of its mode logits.  With
// per-head modes (modes[n][Hq]) the largest of its heads' modes, which sets the query's
// key range (above full when a head's value is not a mode); any_local tells whether a
// head is local (its window must then be valid).
__device__ __forceinline__ int query_mode(const AttnKernelArgs& ka, int q, bool& any_local) {
  if (ka.mode_logits) {
    const int m = hard_decision<3>(ka.mode_logits + 3 * q);
    any_local = m == TRR_MODE_LOCAL;
    return m;
  }
  if (!ka.a.head_modes) {
    const int m = ka.modes[q];
    any_local = m == TRR_MODE_LOCAL;
    return m;
  }
  const uint8_t* row = ka.modes + static_cast<int64_t>(q) * ka.a.Hq;
  int m = 0;
  any_local = false;
#pragma unroll 1
  for (int h = 0; h < ka.a.Hq; ++h) {
    const int v = row[h];
    m = max(m, v);
    any_local |= v == TRR_MODE_LOCAL;
  }
  return m;
}

// Error of a query's arguments, 0 when it is valid.
__device__ __forceinline__ int query_error(const LayerArgs& a, int seq, int t, int mode, bool any_local, int w) {
  if (seq < 0 || seq >= a.S || mode > TRR_MODE_FULL) return TRR_ERR_INVALID_ARG;
  if (t < 0 || t >= a.maxctx) return TRR_ERR_BAD_POSITION;
  if (any_local && w < 1) return TRR_ERR_INVALID_ARG;
  return 0;
}

// Key positions in range (Eq. 2): full [0, t]; local the last w positions up to t.
__device__ __forceinline__ int query_range(int t, int mode, int w) {
  return mode == TRR_MODE_FULL ? t + 1 : mode == TRR_MODE_LOCAL ? min(w, t + 1) : 0;
}

__host__ __device__ constexpr int align16(int x) { return (x + 15) & ~15; }

// Bounded wait (limit_ns on the global timer) that also gives up once *abort is set (by
// a warp that gave up).
__device__ __forceinline__ bool mbar_wait_or(uint64_t* bar, uint32_t parity, volatile int* abort, uint64_t limit_ns) {
  const uint32_t addr = smem_u32(bar), aaddr = smem_u32(const_cast<int*>(abort));
  if (mbar_poll(addr, parity, limit_ns)) return true;
  const uint64_t t0 = global_ns();
  for (;;) {
    if (mbar_poll(addr, parity, limit_ns)) return true;
    if (lds32(aaddr)) return false;
    if (global_ns() - t0 >= limit_ns) return false;
  }
}

// ------------------------------------------------------------ decode step --
//
// A decode-step call (trr_decode_step) appends entry i's token (Sec. 3.2(C), Eq. 4: K and
// V stored at the entry's bit-width; nothing for a skip token unless skip tokens store
// KV) and attends with query i at the same position in the same mode (Eq. 2), in one
// kernel.  The attention reads the cache as the call finds it and takes each query's own
// new token from its K and V rows, quantised in registers; one unit per KV head writes the
// token's bytes to its slot in the page; the last CTA to finish commits the metadata.  The
// entries name distinct sequences (one token per sequence).

__device__ __forceinline__ unsigned seq_hash(int seq, int slots) {
  return (static_cast<unsigned>(seq) * 2654435761u) % static_cast<unsigned>(slots);
}

// One warp, the pools' page counters known: the first opener beyond its pool's capacity
// (OUT_OF_PAGES) as a call error.
__device__ __forceinline__ void step_pages_error(const AttnKernelArgs& ka, int* ent, int lane) {
  int* sc = ent + 6 * ka.n;
  for (int e = lane; e < ka.n; e += 32) {
    const int tok = ent[2 * e], info = ent[2 * e + 1], c = info & 3;
    if (tok >= 0 && (info & 4) && sc[kSNextPage + c] + (info >> 3) >= ka.a.cap[c])
      atomicMin(&sc[kSErr], e * 16 + TRR_ERR_OUT_OF_PAGES);
  }
}

// Page and slot of entry e's token (an entry that stores KV).
__device__ __forceinline__ void step_slot(const AttnKernelArgs& ka, const int* ent, int e, int& c, int& pid,
                                          int& slot) {
  const LayerArgs& a = ka.a;
  const int tok = ent[2 * e], info = ent[2 * e + 1];
  const int* sc = ent + 6 * ka.n;
  c = info & 3;
  slot = tok % a.P;
  pid = (info & 4) ? sc[kSNextPage + c] + (info >> 3) : ent[2 * ka.n + e];  // the class's last page
}

// The last CTA of a decode-step call: records the call's error, or commits every entry's
// metadata (page tables, page first / last positions, counts, the slot's position,
// presence, last positions, the pools' counters).  Nothing of the call's old metadata is
// read after this: every other CTA has finished.
static __device__ void step_commit(const AttnKernelArgs& ka, const int* ent) {
  const LayerArgs& a = ka.a;
  const int n = ka.n;
  const int* sc = ent + 6 * n;
  if (sc[kSErr] != INT_MAX) {
    if (threadIdx.x == 0) set_status(a.ctrl, sc[kSErr] & 15);
    return;
  }
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int seq = ka.seq_ids[e], pos = ka.q_positions[e], tok = ent[2 * e];
    if (tok >= 0) {
      int c, pid, slot;
      step_slot(ka, ent, e, c, pid, slot);
      const int64_t row = (static_cast<int64_t>(seq) * 4 + c) * a.MP + tok / a.P;
      if (ent[2 * e + 1] & 4) {
        a.pt[row] = pid;
        a.pfirst[row] = pos;
      }
      a.plast[row] = pos;
      a.ntok[seq * 4 + c] = tok + 1;
      a.lastpg[seq * 4 + c] = pid;
      reinterpret_cast<int32_t*>(a.pool[c] + static_cast<int64_t>(pid) * a.page_bytes[c])[slot] = pos;
      atomicOr(&a.presence[static_cast<int64_t>(seq) * a.W32 + pos / 32], 1u << (pos % 32));
    }
    a.last_pos[seq] = pos;
  }
  if (threadIdx.x < 4) a.ctrl[kNextPage + threadIdx.x] = sc[kSNextPage + threadIdx.x] + sc[kSOpeners + threadIdx.x];
}

// ------------------------------------------------------------------ partials --

// Merges `count` partial rows at p0, p0 + stride, ...: the common maximum Mx, the
// weighted sum of L and the weighted rows (lane holds dims lane * DPL ..).
template <int D>
__device__ __forceinline__ void merge_partials(const float* p0, int64_t stride, int count, int lane, float& Mx,
                                               float& Ls, float (&acc_o)[D / 32]) {
  // Chunks of CH partials: each chunk's (max, sum) words and rows are loaded together
  // (one round trip to L2 for up to CH splits), then folded into the running result;
  // CH keeps the rows within the registers that are free at this point.
  constexpr int DPL = D / 32, CH = D == 64 ? 16 : 8;
  Mx = kNegInf;
  float lsum = 0.f;  // lane s: the weighted sums of the partials it reads the words of
#pragma unroll
  for (int j = 0; j < DPL; ++j) acc_o[j] = 0.f;
#pragma unroll 1
  for (int s0 = 0; s0 < count; s0 += CH) {
    const int cnt = min(CH, count - s0);
    float2 ml = make_float2(kNegInf, 0.f);
    if (lane < cnt) ml = __ldcg(reinterpret_cast<const float2*>(p0 + (s0 + lane) * stride + D));
    float rows[CH][DPL];
#pragma unroll
    for (int s = 0; s < CH; ++s) {
#pragma unroll
      for (int j = 0; j < DPL; ++j) rows[s][j] = 0.f;
      const float* row = p0 + (s0 + s) * stride + lane * DPL;
      if (s < cnt) {
        if (DPL == 4) {
          const float4 x = __ldcg(reinterpret_cast<const float4*>(row));
          rows[s][0] = x.x; rows[s][1] = x.y; rows[s][DPL - 2] = x.z; rows[s][DPL - 1] = x.w;
        } else {
          const float2 x = __ldcg(reinterpret_cast<const float2*>(row));
          rows[s][0] = x.x; rows[s][1] = x.y;
        }
      }
    }
    float cm = ml.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
    const float nm = fmaxf(Mx, cm);
    if (nm != kNegInf) {
      const float f = Mx == kNegInf ? 0.f : fast_exp2(Mx - nm);  // the earlier chunks' scale
#pragma unroll
      for (int j = 0; j < DPL; ++j) acc_o[j] *= f;
      lsum *= f;
      const float wl = ml.x == kNegInf ? 0.f : fast_exp2(ml.x - nm);  // lane s: weight of row s0 + s
      lsum = fmaf(wl, ml.y, lsum);
#pragma unroll
      for (int s = 0; s < CH; ++s) {
        const float wgt = __shfl_sync(0xffffffffu, wl, s);
#pragma unroll
        for (int j = 0; j < DPL; ++j) acc_o[j] = fmaf(wgt, rows[s][j], acc_o[j]);
      }
      Mx = nm;
    }
  }
  Ls = lsum;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
}

// Counts this warp's arrival on *counter (release of its partial stores, acquire of
// the others'); true for the last of `expected` arrivals, which resets the counter.
__device__ __forceinline__ bool arrive_last(int* counter, int expected, int lane) {
  __syncwarp();
  int arrivals = 0;
  if (lane == 0) arrivals = atom_add_acq_rel(counter, 1);
  __syncwarp();
  arrivals = __shfl_sync(0xffffffffu, arrivals, 0);
  if (arrivals != expected - 1) return false;
  if (lane == 0) *counter = 0;  // ready for the next call
  return true;
}

// ----------------------------------------------------- tensor-core operands --
//
// mma.sync m16n8k16 (f16 or bf16 operands, f32 accumulation); thread (gid, tig) =
// (lane / 4, lane % 4) as in the PTX fragment layouts.
//
// q.k: D_s[key][col] = sum_k A[key][k] B[k][col] with A the K codes of 16 keys and B
// the query rows, column col = (head r, quantiser group gi) = (col / NG, col % NG)
// holding head r's query on group gi's dimensions (zero elsewhere), so every column
// gets its own group sum and s, z apply per group.  A code is masked in place and
// read as an f16 subnormal c * 2^(pos - 24) (pos = its bit offset in the 16-bit half);
// the query is pre-scaled in f16 by 2^(15 - E - pos), E the exponent of the column's largest
// query value, so that every product of a column carries the same factor 2^(-9 - E).  Width 16
// uses bf16 operands (the query is bf16 already).
//
// P.V: O^T[dim][col] = sum_k V^T[dim][key] W[key][col] with W = p * s (two f16 parts; for width 16,
// whose values are raw bf16, two bf16 or tf32 parts).  Pairs along keys for the A
// operand come from byte permutes of two keys' code words.  Each accumulator row keeps
// its class's factor 2^(pos - 24) until the class changes.

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
template <int B>
__device__ __forceinline__ void mma_cls(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  if (B == 16) mma_bf16(c, a0, a1, a2, a3, b0, b1);
  else mma_f16(c, a0, a1, a2, a3, b0, b1);
}

__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// K side: pair i of a thread's D/4 dims of one key, as an A-operand word.
template <int B>
__device__ __forceinline__ uint32_t k_pair(const uint32_t* kw, int i) {
  if (B == 16) return kw[i];
  if (B == 8) return __byte_perm(kw[i >> 1], 0u, (i & 1) ? 0x4342 : 0x4140);
  if (B == 4) {
    const int k = i & 3;
    const uint32_t w = k < 2 ? kw[i >> 2] : (kw[i >> 2] >> 8);
    return w & ((k & 1) ? 0x00F000F0u : 0x000F000Fu);
  }
  const int k = i & 7;
  const uint32_t w = k < 5 ? kw[i >> 3] : (kw[i >> 3] >> 10);
  return w & (0x00030003u << (2 * (k < 5 ? k : k - 5)));
}
// the two dims (relative to the thread's first) of K pair i and their bit offset
template <int B> __host__ __device__ constexpr int kp_lo(int i) {
  return B >= 8 ? 2 * i : B == 4 ? 8 * (i / 4) + i % 4 : 16 * (i / 8) + i % 8;
}
template <int B> __host__ __device__ constexpr int kp_hi(int i) {
  return B >= 8 ? 2 * i + 1 : B == 4 ? 8 * (i / 4) + i % 4 + 4 : 16 * (i / 8) + 8 + i % 8;
}
template <int B> __host__ __device__ constexpr int kp_pos(int i) {
  return B >= 8 ? 0 : B == 4 ? 4 * (i % 2) : 2 * ((i % 8) < 5 ? i % 8 : i % 8 - 5);
}

// V side: dim j of the thread's D/8 dims for keys (a, b) as an A-operand word (key a
// in the low half).  The tensor core lines products up by their operands' exponents, and all
// subnormals have the same: what a product has below 2^-24 of the largest operand exponents is
// cut off, which costs a code at bit offset 0 ten bits.  Codes of 2 and 4 bits are therefore
// moved up to offsets 4, 6, 8 and 2, 6, two shifts a half word in place of one (offsets 0, 2, ..
// and 0, 4: rows of 2-bit tokens with outlier channels were 1e-4 to 3e-4 of their size off
// before rounding, of 4-bit ones 7e-5 to 2e-4).
__host__ __device__ constexpr int v2_pos(int k) { return 4 + 2 * ((k + 1) % 3); }  // width 2: field k of 8
template <int B>
__device__ __forceinline__ uint32_t v_pair(const uint32_t* wa, const uint32_t* wb, int j) {
  if (B == 16) return __byte_perm(wa[j >> 1], wb[j >> 1], (j & 1) ? 0x7632 : 0x5410);
  if (B == 8) {
    const int k = j & 3;
    const uint32_t x = __byte_perm(wa[j >> 2], wb[j >> 2], k < 2 ? 0x5140 : 0x7362);
    return __byte_perm(x, 0u, (k & 1) ? 0x4342 : 0x4140);
  }
  if (B == 4) {
    const int k = j & 7;
    uint32_t x = __byte_perm(wa[j >> 3], wb[j >> 3], k < 4 ? 0x5410 : 0x7632);
    x = (k & 3) < 2 ? x << 2 : x >> 6;
    return x & ((k & 1) ? 0x03C003C0u : 0x003C003Cu);
  }
  const int k = j & 15, kk = k & 7;
  uint32_t x = __byte_perm(wa[j >> 4], wb[j >> 4], k < 8 ? 0x5410 : 0x7632);
  if (kk < 2) x <<= 6;
  if (kk >= 5) x >>= 6;
  return x & (0x00030003u << v2_pos(kk));
}
// log2 of the factor a V accumulator row carries in class index c (dim j of the
// thread's D/8): 2^(pos - 24) for codes, 1 for bf16
__host__ __device__ constexpr int vfac_log2(int c, int j) {
  return c == 3 ? 0 : c == 2 ? -24 : c == 1 ? 2 + 4 * (j & 1) - 24 : v2_pos(j & 7) - 24;
}

// ------------------------------------------------------------------ combine --
// Merges the split partials of every (query, head) of a query-group launch whose query has
// more than one split, and writes the bf16 row.  `wpr` warps share a row, each folding every
// wpr-th split over its own maximum; the row's first warp then folds the warps.  Chained after
// the attention kernel (programmatic dependent launch): it reads nothing before that kernel
// has finished, and the next layer's kernel waits for all of it, so it is bound by its round
// trips to L2.  Each warp therefore has a chunk of rows and its (max, sum) words in flight at
// once (merge_partials).  (gqa_long shape, 3 full queries of 16, 93 splits of 32768 positions:
// 5.2 us; 17 with four warps a row that read the maxima, then the sums, then row after row.)
// A row gets as many warps, up to the CTA's 8, as keep the CTAs within what the chip
// holds at once (8 per SM): with 2048 rows of 0 to 3 splits, 8 warps a row took 16 us more
// per 6 layers than 4.
constexpr int kCombineWarps = 8;  // of a CTA

struct CombineArgs {
  const float* part;  // partials of the launch: a head's splits one after another, D + 4 floats each
  const int2* qtab;   // [n] first partial and splits per head of each query (written by CTA 0 of the
                      // attention kernel)
  uint16_t* out;      // [n][Hq][D] bf16 rows of the launch
  int Hq, rows;       // rows: n * Hq
  int wpr;            // warps of a row: 1, 2, 4 or 8
};

template <int D>
__global__ void __launch_bounds__(32 * kCombineWarps) attn_combine_kernel(const __grid_constant__ CombineArgs ca) {
  constexpr int DPL = D / 32;
  __shared__ float sacc[kCombineWarps][D];
  __shared__ float2 sml[kCombineWarps];
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp & (ca.wpr - 1);
  const int row = (blockIdx.x * kCombineWarps + warp) / ca.wpr;
  const int qi = min(row, ca.rows - 1) / ca.Hq, qh = row - qi * ca.Hq;
  const int2 e = ca.qtab[qi];
  const bool act = row < ca.rows && e.y > 1;  // one split: written by the attention kernel
  float M = kNegInf, L = 0.f, acc[DPL];
  if (act) {
    const int64_t stride = D + 4;
    const float* p0 = ca.part + (static_cast<int64_t>(e.x) + static_cast<int64_t>(qh) * e.y + part) * stride;
    merge_partials<D>(p0, stride * ca.wpr, (e.y - part + ca.wpr - 1) / ca.wpr, lane, M, L, acc);
    if (part > 0) {
#pragma unroll
      for (int j = 0; j < DPL; ++j) sacc[warp][lane * DPL + j] = acc[j];
      if (lane == 0) sml[warp] = make_float2(M, L);
    }
  }
  if (ca.wpr > 1) __syncthreads();
  if (!act || part > 0) return;
  if (ca.wpr > 1) {
    const float own = M;
#pragma unroll 1
    for (int w = 1; w < ca.wpr; ++w) M = fmaxf(M, sml[warp + w].x);
    float f = own == kNegInf ? 0.f : fast_exp2(own - M);
    L *= f;
#pragma unroll
    for (int j = 0; j < DPL; ++j) acc[j] *= f;
#pragma unroll 1
    for (int w = 1; w < ca.wpr; ++w) {
      const float2 ml = sml[warp + w];
      f = ml.x == kNegInf ? 0.f : fast_exp2(ml.x - M);
      L = fmaf(f, ml.y, L);
#pragma unroll
      for (int j = 0; j < DPL; ++j) acc[j] = fmaf(f, sacc[warp + w][lane * DPL + j], acc[j]);
    }
  }
  const float inv = L > 0.f ? 1.f / L : 0.f;
  uint16_t* orow = ca.out + static_cast<int64_t>(row) * D + lane * DPL;
#pragma unroll
  for (int j = 0; j < DPL; j += 2)
    *reinterpret_cast<__nv_bfloat162*>(orow + j) = __floats2bfloat162_rn(acc[j] * inv, acc[j + 1] * inv);
}

cudaError_t launch_attn_combine(int d, int ctas, cudaStream_t s, const CombineArgs& ca);

}  // namespace trr
