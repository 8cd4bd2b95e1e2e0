// trr_append.cu - trr_kv_append: quantise-on-write into the width-class page pools.
//
// One kernel, append_kernel (below), for calls of up to 1024 entries: validates every
// entry, ranks it among the earlier entries of its (sequence, class), hands out page ids in
// entry order, quantises the rows (Q_b of Sec. 3.2(C), Eq. 4, or a bf16 copy for b = 16)
// and commits the metadata only when the whole call is valid (Sec. 3.8: each token's KV is
// stored at its chosen width in a paged cache).
#include <algorithm>
#include <climits>

#include "trr_internal.cuh"

namespace trr {

__device__ __forceinline__ int class_of_bits(int b) {
  return b == 2 ? 0 : b == 4 ? 1 : b == 8 ? 2 : b == 16 ? 3 : -1;
}

// An entry's attention mode and bit-width: the caller's, or the hard decisions of its
// router logits (Sec. 3.8), taken here in the append's own planning step.  With
// per-head modes (modes[n][Hq]) the largest of the entry's head modes: skip only when
// every head skips, above full when any head's value is not a mode.
__device__ __forceinline__ int entry_mode(const LayerArgs& a, const uint8_t* modes, const float* mode_logits, int e) {
  if (mode_logits) return hard_decision<3>(mode_logits + 3 * e);
  if (!a.head_modes) return modes[e];
  int m = 0;
  const uint8_t* row = modes + static_cast<int64_t>(e) * a.Hq;
  for (int h = 0; h < a.Hq; ++h) m = max(m, static_cast<int>(row[h]));
  return m;
}

// Per-head modes: whether entry e stores KV head j, i.e. whether a query head reading it
// (h / (Hq / Hkv) == j) does not skip, or skip tokens store KV.
__device__ __forceinline__ bool head_stores(const LayerArgs& a, const uint8_t* modes, int e, int j) {
  if (a.skip_writes_kv) return true;
  const int g = a.Hq / a.Hkv;
  const uint8_t* row = modes + static_cast<int64_t>(e) * a.Hq + j * g;
  for (int h = 0; h < g; ++h)
    if (row[h] != TRR_MODE_SKIP) return true;
  return false;
}

// Per-head modes: KV head j's presence mask in a page, the first 8 of the 16 bytes that
// end its slice.
__device__ __forceinline__ unsigned long long* head_mask(const LayerArgs& a, int c, int pid, int j) {
  return reinterpret_cast<unsigned long long*>(a.pool[c] + static_cast<int64_t>(pid) * a.page_bytes[c] + a.hdr +
                                               static_cast<int64_t>(j + 1) * a.slice[c] - a.maskb);
}
__device__ __forceinline__ int entry_bits(const uint8_t* bits, const float* bit_logits, int e) {
  return bit_logits ? 2 << hard_decision<4>(bit_logits + 4 * e) : bits[e];
}

// Entries of the small instance: a decode step's calls plan with 256 threads, larger ones
// with 1024.  The instance is chosen by n alone.
constexpr int kSmallAppend = 256;

// Per-entry facts of a call, indexed by entry, that every CTA works out for itself.
template <int T>
struct AppendShared {
  unsigned long long prefix[T];  // inclusive counts of the four classes' tokens in sorted order (16 bits each)
  unsigned long long wsum[32], wmax[32], wopen[32];  // per warp (the rest zero): see the prefix passes
  uint32_t key[T];  // sequence << 10 | entry, sorted
  int pos[T];       // position; later the page that the list slot's token opens
  int cls[T];       // width class when the entry stores KV, else -1
  int tok[T];       // token index in its (sequence, class) list
  int pid[T];       // page of the token
  int end[T];       // by first sorted index of a sequence: its last one
  int whead[32];
  int next[kClasses];
  int first_err, last;
};

// Sorts the T keys (one per thread, all distinct) ascending: bitonic, exchanges inside a
// warp by shuffles.
template <int T>
__device__ __forceinline__ uint32_t sort_keys(uint32_t key, uint32_t* sh) {
  const int i = threadIdx.x;
#pragma unroll 1
  for (int k = 2; k <= T; k <<= 1) {
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
      uint32_t other;
      if (j >= 32) {
        sh[i] = key;
        __syncthreads();
        other = sh[i ^ j];
        __syncthreads();
      } else {
        other = __shfl_xor_sync(0xffffffffu, key, j);
      }
      const bool low = (i & j) == 0, up = (i & k) == 0;
      key = low == up ? min(key, other) : max(key, other);
    }
  }
  return key;
}

// The warp's sum of four 16-bit counts (each sum below 65536).
__device__ __forceinline__ unsigned long long add_packed(unsigned long long x) {
  const uint32_t lo = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(x));
  const uint32_t hi = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(x >> 32));
  return static_cast<unsigned long long>(hi) << 32 | lo;
}

// 8 consecutive values of a row (raw, bf16) by one lane of the G/8 that hold the group:
// Eq. 4 at b < 16 bits, the 8 codes packed LSB-first into `codes`, (s, z) into `sz`.  A
// group holding a value binary16 cannot carry (non-finite or |x| > 65504) gets zeros and
// bad = true.  Every lane of the warp calls it.
__device__ __forceinline__ void quantise_8(const uint4 raw, int b, int GL, unsigned long long& codes, uint32_t& sz,
                                           bool& bad) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  float x[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = bf16lo(w[i]);
    x[2 * i + 1] = bf16hi(w[i]);
  }
  float mn = x[0], mx = x[0];
  bad = false;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    bad |= !(fabsf(x[i]) <= 65504.f);  // also true for NaN
    mn = fminf(mn, x[i]);
    mx = fmaxf(mx, x[i]);
  }
  for (int o = 1; o < GL; o <<= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    bad |= __shfl_xor_sync(0xffffffffu, static_cast<int>(bad), o) != 0;
  }
  codes = 0;
  sz = 0;
  if (bad) return;
  const int levels = (1 << b) - 1;
  const __half z16 = __float2half_rn(mn);                                                        // z = min(x)
  const __half s16 = __float2half_rn(__fdiv_rn(__fsub_rn(mx, mn), static_cast<float>(levels)));  // s
  const float z = __half2float(z16), s = __half2float(s16), rs = __frcp_rn(s);
  if (s != 0.f) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      codes |= static_cast<unsigned long long>(static_cast<uint32_t>(code_of(x[i], z, s, rs, levels))) << (i * b);
  }
  sz = static_cast<uint32_t>(__half_as_ushort(s16)) | (static_cast<uint32_t>(__half_as_ushort(z16)) << 16);
}

// One kernel per call.  Every CTA plans every entry the same way from the metadata as the
// call found it and writes its share of the rows; the last CTA to finish planning commits
// the metadata: every other CTA has read all it needs of them by then.
//
// The plan sorts the entries by (sequence, entry) unless they come that way, so that what
// an entry needs of the earlier entries of its sequence (largest position, tokens per
// class) is one prefix pass instead of a scan of all entries: O(n log n) in place of
// O(n^2).  In the small instance everything up to the first read of metadata comes before
// the wait on the previous kernel and overlaps it.  Rows are quantised by d/8 lanes each,
// 16 bytes a lane.
//
// Bound by latency: the chain from the wait (metadata, page ids, first rows).  The second
// row of a lane is loaded while the first is quantised, and the arrival's round trip and the
// commit overlap the rows: 11.8 us a call of 1024 entries of 12 x 64 KV heads, on the GPU alone
// (13.9 without either; 122 with a plan kernel that scans all entries for each entry and a second
// kernel of one thread per group).  The large instance waits before it reads its entries
// (reading them early would save 2.4 us).
template <int D, int T>
__global__ void __launch_bounds__(T) append_kernel(LayerArgs a, int n, const int32_t* __restrict__ seq_ids,
                                                   const int32_t* __restrict__ positions,
                                                   const uint8_t* __restrict__ bits,
                                                   const uint8_t* __restrict__ modes,
                                                   const float* __restrict__ bit_logits,
                                                   const float* __restrict__ mode_logits,
                                                   const uint16_t* __restrict__ k, const uint16_t* __restrict__ v) {
  __shared__ AppendShared<T> sh;
  constexpr int LPR = D / 8;  // lanes per row
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  const unsigned below = (1u << lane) - 1u;

  // ------------------------------------------- the entries, and what follows from them alone
  // lanes LPR r .. of the grid hold row r = (entry, KV head, K | V), 8 values each
  const int nlanes = n * a.Hkv * 2 * LPR, step = gridDim.x * T;
  auto row_src = [&](int x) {
    const int r = x / LPR, e = r / (2 * a.Hkv), j = (r >> 1) % a.Hkv;
    return reinterpret_cast<const uint4*>(((r & 1) ? v : k) + (static_cast<int64_t>(e) * a.Hkv + j) * D) + x % LPR;
  };
  const int x0 = blockIdx.x * T + i;
  if (T > kSmallAppend) pdl_wait();
  int err = 0;  // of entry i until the sort, then of the entry this thread has
  uint32_t key = 0xffffffffu - (1023u - i);  // past the entries
  if (i < n) {
    const int seq = seq_ids[i], pos = positions[i], m = entry_mode(a, modes, mode_logits, i);
    const int c = class_of_bits(entry_bits(bits, bit_logits, i));
    const bool in = seq >= 0 && seq < a.S;
    if (!in || c < 0 || m > TRR_MODE_FULL) err = TRR_ERR_INVALID_ARG;
    else if (pos < 0 || pos >= a.maxctx) err = TRR_ERR_BAD_POSITION;
    key = ((in ? static_cast<uint32_t>(seq) : 1u << 20) << 10) | static_cast<uint32_t>(i);
    sh.pos[i] = pos;
    sh.cls[i] = !err && (m != TRR_MODE_SKIP || a.skip_writes_kv) ? c : -1;
    sh.tok[i] = err;
  }
  sh.key[i] = key;
  if (i < 32) {
    sh.wsum[i] = sh.wmax[i] = sh.wopen[i] = 0ull;
    sh.whead[i] = -1;
  }
  if (i == 0) sh.first_err = INT_MAX;
  __syncthreads();
  if (__syncthreads_or(i > 0 && sh.key[i - 1] > key)) {
    key = sort_keys<T>(key, sh.key);
    __syncthreads();
    sh.key[i] = key;
    __syncthreads();
  }
  const bool act = key < (2u << 30);            // an entry ..
  const int e = static_cast<int>(key & 1023u);  // .. this one ..
  const bool has_seq = key < (1u << 30);        // .. whose sequence id is valid
  const int seq = has_seq ? static_cast<int>(key >> 10) : -1;
  const int pos = act ? sh.pos[e] : 0, c = act ? sh.cls[e] : -1;
  err = act ? sh.tok[e] : 0;
  const bool writes = c >= 0;
  // prefix passes over the sorted entries: tokens per class (16 bits each), the largest
  // position so far (with the sequence above it: sequences ascend), the sequence's start
  const bool head = i == 0 || (sh.key[i - 1] >> 10) != (key >> 10);
  const bool tail = i == T - 1 || (sh.key[i + 1] >> 10) != (key >> 10);
  unsigned long long sum = writes ? 1ull << (16 * c) : 0ull;
  unsigned long long top = (static_cast<unsigned long long>(key >> 10) << 32) |
                           (static_cast<uint32_t>(pos) ^ 0x80000000u);  // order of int32
  const unsigned heads = __ballot_sync(0xffffffffu, head) & (below | (1u << lane));
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long s1 = __shfl_up_sync(0xffffffffu, sum, o), t1 = __shfl_up_sync(0xffffffffu, top, o);
    if (lane >= o) {
      sum += s1;
      top = max(top, t1);
    }
  }
  if (lane == 31) {
    sh.wsum[warp] = sum;
    sh.wmax[warp] = top;
    sh.whead[warp] = heads ? 32 * warp + 31 - __clz(heads) : -1;
  }
  __syncthreads();
  // the warps before this one: their sum, largest and last start, one warp per lane
  const bool earlier = lane < warp;
  const unsigned long long before = add_packed(earlier ? sh.wsum[lane] : 0ull);
  const unsigned long long wt = earlier ? sh.wmax[lane] : 0ull;
  const uint32_t th = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(wt >> 32));
  const uint32_t tl = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(wt >> 32) == th ? static_cast<uint32_t>(wt) : 0u);
  const unsigned long long top_before = static_cast<unsigned long long>(th) << 32 | tl;
  const int hb = __reduce_max_sync(0xffffffffu, earlier ? sh.whead[lane] : -1);
  const int first = heads ? 32 * warp + 31 - __clz(heads) : hb;
  sum += before;
  // the largest position before this entry: the previous lane's, or the previous warps'
  unsigned long long prev = __shfl_up_sync(0xffffffffu, top, 1);
  prev = lane == 0 ? top_before : max(prev, top_before);
  const bool has_prev = i > 0 && static_cast<uint32_t>(prev >> 32) == (key >> 10);
  const int prev_max = has_prev ? static_cast<int>(static_cast<uint32_t>(prev) ^ 0x80000000u) : -1;
  sh.prefix[i] = sum;
  if (tail) sh.end[first] = i;
  __syncthreads();  // sh.pos (by entry) is read no more
  const unsigned long long start = first > 0 ? sh.prefix[first - 1] : 0ull;
  const unsigned long long mine = sum - start, all = sh.prefix[sh.end[first]] - start;
  auto field = [](unsigned long long x, int cc) { return static_cast<int>((x >> (16 * cc)) & 0xffffu); };
  const int rank = writes ? field(mine, c) - 1 : 0;  // earlier entries of the (sequence, class) that store KV
  const bool last_cls = writes && rank + 1 == field(all, c);
  int slot0 = first;  // where the class's tokens of this sequence are listed: first, then rank
  for (int cc = 0; cc < c; ++cc) slot0 += field(all, cc);

  // ----------------------------------- after the wait: the metadata, this lane's first row
  if (T <= kSmallAppend) pdl_wait();
  pdl_trigger();
  uint4 raw = make_uint4(0, 0, 0, 0);
  if (x0 < nlanes) raw = *row_src(x0);
  if (i < kClasses) sh.next[i] = a.ctrl[kNextPage + i];
  int tok = 0, nt_old = 0, last_page = -1;
  if (act && !err) {
    const int lp = a.last_pos[seq];
    if (writes) {
      nt_old = a.ntok[seq * 4 + c];
      last_page = a.lastpg[seq * 4 + c];
    }
    if (pos <= max(prev_max, lp)) err = TRR_ERR_BAD_POSITION;
    tok = nt_old + rank;
  }
  const bool opens = writes && !err && tok % a.P == 0;
  if (act) sh.pid[e] = opens;
  __syncthreads();
  // page ids in entry order: next_page + openers of the same class before the entry
  {
    const int cc = i < n && sh.pid[i] ? sh.cls[i] : -1;
    unsigned long long mine4 = cc >= 0 ? 1ull << (16 * cc) : 0ull;
    int rk = 0;
#pragma unroll
    for (int q = 0; q < kClasses; ++q) {
      const unsigned bal = __ballot_sync(0xffffffffu, cc == q);
      if (cc == q) rk = __popc(bal & below);
    }
    mine4 = add_packed(mine4);
    if (lane == 0) sh.wopen[warp] = mine4;
    __syncthreads();
    const unsigned long long wo = add_packed(lane < warp ? sh.wopen[lane] : 0ull);
    if (cc >= 0) sh.pid[i] = sh.next[cc] + field(wo, cc) + rk;
  }
  __syncthreads();
  int pid = -1;
  if (opens) {
    pid = sh.pid[e];
    if (pid >= a.cap[c]) err = TRR_ERR_OUT_OF_PAGES;
    sh.pos[slot0 + rank] = pid;
  }
  if (act && err) atomicMin(&sh.first_err, e);
  __syncthreads();
  if (sh.first_err != INT_MAX) {  // the call is a no-op; record the lowest failing entry
    if (blockIdx.x == 0 && act && e == sh.first_err) set_status(a.ctrl, err);
    return;
  }
  const int kidx = tok / a.P;
  if (writes && !opens)  // a page opened by an earlier call (then the class's last one), or
                         // by an earlier entry of this one
    pid = kidx * a.P < nt_old ? last_page : sh.pos[slot0 + kidx * a.P - nt_old];
  if (act) {
    sh.pid[e] = pid;
    sh.tok[e] = tok;
  }
  __syncthreads();

  // This CTA has read its last metadata.  The last one to get here commits them (after its
  // own rows, so that the arrival's round trip is hidden): its acquire follows the release
  // of every other CTA.
  if (i == 0) sh.last = atom_add_acq_rel(&a.ctrl[kAppendDone], 1) == static_cast<int>(gridDim.x) - 1;

  // ------------------------------------------------------------------------ the rows
  const int ng = D / a.G, GL = a.G / 8;
  uint4 next = raw;
  for (int x = x0; x - lane < nlanes; x += step) {  // warps stay together
    raw = next;
    if (x + step < nlanes) next = *row_src(x + step);
    const int r = min(x, nlanes - 1) / LPR, re = r / (2 * a.Hkv), j = (r >> 1) % a.Hkv, which = r & 1, l = x % LPR;
    const int rc = x < nlanes ? sh.cls[re] : -1, b = bits_of_class(rc & 3);
    unsigned long long codes;
    uint32_t sz;
    bool bad;
    quantise_8(raw, min(b, 8), GL, codes, sz, bad);
    if (rc < 0) continue;
    const int slot = sh.tok[re] % a.P;
    uint8_t* sl = a.pool[rc] + static_cast<int64_t>(sh.pid[re]) * a.page_bytes[rc] + a.hdr +
                  static_cast<int64_t>(j) * a.slice[rc];
    const int64_t off = static_cast<int64_t>(which * a.P + slot) * (D * b / 8) + l * b;
    uint8_t* dst = sl + (a.swz && b >= 8 ? swz_off(off) : off);  // stays inside a 16-byte chunk
    if (b == 16) {  // native precision: the bf16 bits
      *reinterpret_cast<uint4*>(dst) = raw;
      continue;
    }
    if (b == 2) *reinterpret_cast<uint16_t*>(dst) = static_cast<uint16_t>(codes);
    else if (b == 4) *reinterpret_cast<uint32_t*>(dst) = static_cast<uint32_t>(codes);
    else *reinterpret_cast<unsigned long long*>(dst) = codes;
    if (l % GL == 0) {
      reinterpret_cast<uint32_t*>(sl + 2 * static_cast<int64_t>(a.P) * (D * b / 8) +
                                  static_cast<int64_t>(which * a.P + slot) * ng * 4)[l / GL] = sz;
      if (bad) set_status(a.ctrl, TRR_ERR_BAD_VALUE);
    }
  }

  // ---------------------------------------------------------------------- the commit
  __syncthreads();
  if (!sh.last) return;
  if (writes) {
    const int slot = tok % a.P;
    const int64_t prow = (static_cast<int64_t>(seq) * 4 + c) * a.MP + kidx;
    if (opens) {
      a.pt[prow] = pid;
      a.pfirst[prow] = pos;
    }
    if (last_cls || slot == a.P - 1) a.plast[prow] = pos;
    if (last_cls) {
      a.ntok[seq * 4 + c] = tok + 1;
      a.lastpg[seq * 4 + c] = pid;
    }
    reinterpret_cast<int32_t*>(a.pool[c] + static_cast<int64_t>(pid) * a.page_bytes[c])[slot] = pos;
    atomicOr(&a.presence[static_cast<int64_t>(seq) * a.W32 + pos / 32], 1u << (pos % 32));
  }
  if (act && tail) a.last_pos[seq] = pos;
  if (a.head_modes) {  // presence masks: openers clear their new pages, then every entry
                       // sets its slot's bit for the KV heads it stores
    if (opens)
      for (int j = 0; j < a.Hkv; ++j) {
        head_mask(a, c, pid, j)[0] = 0ull;
        head_mask(a, c, pid, j)[1] = 0ull;
      }
    __syncthreads();
    if (writes)
      for (int j = 0; j < a.Hkv; ++j)
        if (head_stores(a, modes, e, j)) atomicOr(head_mask(a, c, pid, j), 1ull << (tok % a.P));
  }
  if (warp == 0) {
    const unsigned long long opened = add_packed(sh.wopen[lane]);
    if (i < kClasses) a.ctrl[kNextPage + i] = sh.next[i] + field(opened, i);
  }
  if (i == 0) a.ctrl[kAppendDone] = 0;
}

template <int D, int T>
static cudaError_t launch_append(const LayerArgs& a, int num_sms, cudaStream_t s, int n, const int32_t* seq_ids,
                                 const int32_t* positions, const uint8_t* bits, const uint8_t* modes,
                                 const float* bit_logits, const float* mode_logits, const uint16_t* k,
                                 const uint16_t* v) {
  // a lane per 8 values, at most one CTA per SM
  const int64_t work = static_cast<int64_t>(n) * a.Hkv * 2 * (D / 8);
  const unsigned grid = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((work + T - 1) / T, num_sms)));
  return launch_pdl(append_kernel<D, T>, dim3(grid), dim3(T), 0, s, a, n, seq_ids, positions, bits, modes, bit_logits,
                    mode_logits, k, v);
}

}  // namespace trr

using namespace trr;

// One append call: the entries' modes and widths come from `bits` / `modes`, or (with
// those null) from the router logits.
static trr_status append_call(trr_cache* cache, int32_t layer, int32_t n, const int32_t* seq_ids,
                              const int32_t* positions, const void* k_bf16, const void* v_bf16, const uint8_t* bits,
                              const uint8_t* modes, const float* bit_logits, const float* mode_logits,
                              void* stream) {
  if (!cache) return TRR_ERR_INVALID_ARG;
  const Layout& l = cache_layout(cache);
  if (layer < 0 || layer >= l.L || n < 0 || n > l.max_append) return TRR_ERR_INVALID_ARG;
  cache_set_launches(cache, 0);
  if (n == 0) return TRR_OK;
  if (!seq_ids || !positions || !k_bf16 || !v_bf16 || !(bits || bit_logits) || !(modes || mode_logits))
    return TRR_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(k_bf16) | reinterpret_cast<uintptr_t>(v_bf16)) & 15)
    return TRR_ERR_INVALID_ARG;  // rows are read 16 bytes at a time
  if ((reinterpret_cast<uintptr_t>(bit_logits) | reinterpret_cast<uintptr_t>(mode_logits)) & 3)
    return TRR_ERR_INVALID_ARG;
  if (mode_logits && l.head_modes) return TRR_ERR_UNSUPPORTED;  // router decisions are per token
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const LayerArgs a = layer_args(l, cache_views(cache), layer);
  cache_note_call(cache, layer);
  const uint16_t* k = static_cast<const uint16_t*>(k_bf16);
  const uint16_t* v = static_cast<const uint16_t*>(v_bf16);
  auto* launch = n <= kSmallAppend ? (l.d == 64 ? launch_append<64, kSmallAppend> : launch_append<128, kSmallAppend>)
                                   : (l.d == 64 ? launch_append<64, 1024> : launch_append<128, 1024>);
  const cudaError_t e = launch(a, cache_num_sms(cache), s, n, seq_ids, positions, bits, modes, bit_logits, mode_logits, k, v);
  cache_set_launches(cache, 1);
  return e == cudaSuccess ? TRR_OK : TRR_ERR_CUDA;
}

extern "C" trr_status trr_kv_append(trr_cache* cache, int32_t layer, int32_t n, const int32_t* seq_ids,
                                    const int32_t* positions, const void* k_bf16, const void* v_bf16,
                                    const uint8_t* bits, const uint8_t* modes, void* stream) {
  return append_call(cache, layer, n, seq_ids, positions, k_bf16, v_bf16, bits, modes, nullptr, nullptr, stream);
}

extern "C" trr_status trr_kv_append_routed(trr_cache* cache, int32_t layer, int32_t n, const int32_t* seq_ids,
                                           const int32_t* positions, const void* k_bf16, const void* v_bf16,
                                           const float* bit_logits, const float* mode_logits, void* stream) {
  return append_call(cache, layer, n, seq_ids, positions, k_bf16, v_bf16, nullptr, nullptr, bit_logits, mode_logits,
                     stream);
}
