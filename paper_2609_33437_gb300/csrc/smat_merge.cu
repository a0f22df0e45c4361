// Merging over K experts (the evaluation side, Eq. merged-state):
// theta_merge = theta0 + sum_j alpha_j (.) m_j (.) Delta_j, Delta_j = theta_j -
// theta0, for weight averaging, Task Arithmetic, DARE followed by Task
// Arithmetic and TIES (the merging methods of Sec. 5). Elementwise and bound
// by HBM bandwidth: each element reads theta0 and the K experts once and
// writes the result once (TIES first reads every expert once or twice more, at
// most four times, to select its per-tensor trim thresholds exactly).
//
// Arithmetic, identical to the CPU oracle: Delta_j one fp32 subtraction;
// experts accumulated in index order, one fused multiply-add each (WA 1/K,
// TA gamma, DARE gamma / p_keep on the kept coordinates); TIES sums the kept
// values, elects the sign of that sum, averages the kept values of that sign
// (one fp32 division) and scales by gamma; then fl(theta0 + acc) rounded to
// the storage dtype. DARE's mask of expert j is the library's Mask stream
// with step = j.
//
// TIES trim threshold of each (tensor, expert) slot: the r-th largest key of
// |Delta_j| (key = the bits of the magnitude as uint32, r = ceil(retention
// n)), selected exactly. A sample of the slot's keys gives an interval that
// holds the threshold almost surely (small tensors are sampled whole, which
// decides them); a pass over the inputs then counts the keys in 2046 equal
// bins of that interval and in one bin below and one above it, and one CTA
// per slot picks the bin that holds the r-th largest. A bin of one key, or the
// first key of a bin (bf16 differences lie on coarse grids) if that is
// where the r-th lies, is the threshold; any other bin, also the two outer
// ones when the sample missed, is the next pass's interval. Passes skip decided
// slots.

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <unordered_set>
#include <vector>

#include "smat.h"
#include "smat_device.cuh"

namespace smat {
namespace {

constexpr int kMergeMaxExperts = SMAT_MERGE_MAX_EXPERTS;
// Elements per chunk of a merge: 2^16, or for lists of fewer than kFewChunks
// such chunks (16 per SM of a GB300's 152; a tuning value, any other count works)
// a smaller power of two down to 2^13, so that a small merge is spread over the
// chip (61 chunks of 2^16 left most SMs idle: TIES of 4 experts of 4e6 fp32
// elements spent 55 us in the merge pass, 14 at HBM speed).
constexpr int64_t kMergeChunkMax = int64_t(1) << 16;
constexpr int64_t kMergeChunkMin = int64_t(1) << 13;
constexpr int64_t kFewChunks = 16 * 152;
int64_t merge_chunk_for(int64_t total) {
  int64_t c = kMergeChunkMax;
  while (c > kMergeChunkMin && total / c < kFewChunks) c /= 2;
  return c;
}
constexpr int kHistBins = 2048;  // an interval's 2046 bins, one below it and one above it
constexpr int kInner = kHistBins - 2;
// Passes over the inputs: one or two when the sample's interval holds the
// threshold. An interval never reaches past kInfKey (NaN keys count in the bin
// above it), so it is at most kInfKey + 1 <= 2046 2^20 keys wide and three passes
// decide it (bins of at most 2^20, 2^10 and 1 keys); a miss costs one pass more.
constexpr int kPasses = 4;
constexpr uint32_t kInfKey = 0x7F800000u;
static_assert((uint64_t(kInner) << 20) >= uint64_t(kInfKey) + 1 && (uint64_t(kInner) << 10) >= (1u << 20) && kInner >= 1 << 10,
              "kPasses passes decide every slot");
constexpr size_t kMergeAlign = 256;

struct MTensor {
  const void* theta0;
  void* out;
  int64_t numel;
  int64_t elem_offset;
  uint32_t tid, flags, t_hi, t_lo;
  int32_t dtype, pad;
};

// Threshold selection of one (tensor, expert) slot.
struct TiesSlot {  // 16 bytes
  uint32_t lo;     // first key of the interval, a multiple of 2^shift
  int32_t shift;   // its bins hold 2^shift keys each
  uint32_t done;   // the threshold is decided
  uint32_t pad;
};

// A list cut into chunks of `elems` elements, one tensor after the other: first[t]
// is tensor t's first chunk, first[n_tensors] == n the number of chunks.
struct ChunkSplit {
  const int32_t* first;
  int64_t elems;
  int64_t n;
};

struct MArgs {
  const MTensor* tensors;
  ChunkSplit chunks;           // of the merge kernels
  ChunkSplit hist_chunks;      // of the TIES threshold passes
  const void* const* experts;  // [tensor * K + e]
  uint32_t* thr;               // [tensor * K + e] TIES threshold keys
  TiesSlot* slots;             // [tensor * K + e]
  int64_t* rank;               // r of each slot (1 = the largest key)
  uint32_t* n_done;            // slots decided so far
  unsigned long long* hist;    // [(tensor * K + e) * kHistBins], see ties_hist_kernel
  RoundKeys key;
  int32_t K, method;
  int32_t n_tensors;
  float gamma, c;              // c: per-expert coefficient (WA 1/K, TA gamma, DARE gamma / p_keep)
  int32_t n_slots;
};

// Chunk c of the split, by a binary search of the tensors' first chunks (they stay in
// L1: the streaming loads allocate no lines there). A table with a record per chunk took
// one load, but beyond 64 KB its upload from pageable memory waits for the stream,
// and a merge call then does not return before the work ahead of it is done (two
// experts of 3.5e7 fp32 elements, called in a row: 111 us each with 102 KB of records,
// 93 now). Without a barrier: finding it together, with one load per thread, made the
// DARE kernel's warps wait for each other at every chunk (0.5B decoder 2366 -> 2407 us).
__device__ __forceinline__ Chunk chunk_of(const MArgs& m, const ChunkSplit& split, int64_t c) {
  int lo = 0, hi = m.n_tensors;  // first[lo] <= c < first[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (split.first[mid] <= c) lo = mid;
    else hi = mid;
  }
  Chunk ch;
  ch.tensor = lo;
  ch.pad = 0;
  ch.begin = (c - split.first[lo]) * split.elems;
  ch.end = min(ch.begin + split.elems, m.tensors[lo].numel);
  return ch;
}

__device__ __forceinline__ uint32_t abs_key(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

// An expert's contribution to a 16-element group: acc += c Delta.
template <int DT>
__device__ __forceinline__ void merge_acc16(float c, const Raw16<DT>& x, const Raw16<DT>& t0, float2 (&acc)[8]) {
  const float2 c2 = splat(c);
#pragma unroll
  for (int h = 0; h < 8; ++h) acc[h] = fma2_rn(c2, sub2_rn(x.pair(h), t0.pair(h)), acc[h]);
}

template <int DT>
__device__ __forceinline__ void store_merged16(const MTensor& T, int64_t i, const Raw16<DT>& t0,
                                               const float2 (&acc)[8]) {
  float out[16];
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    const float2 o = add2_rn(t0.pair(h), acc[h]);
    out[2 * h] = o.x;
    out[2 * h + 1] = o.y;
  }
  store16<DT>(T.out, i, out);
}

// Experts are loaded four at a time (all four loads in flight before the
// first is used) and accumulated in index order.
constexpr int kExpertBatch = 4;

// WA / TA on one 16-element group (vector path).
template <int DT>
__device__ __forceinline__ void merge_linear16(const MArgs& m, const MTensor& T, int t, int64_t i) {
  Raw16<DT> t0;
  load16<DT>(T.theta0, i, t0);
  float2 acc[8];
#pragma unroll
  for (int h = 0; h < 8; ++h) acc[h] = splat(0.0f);
  const void* const* xp = m.experts + t * m.K;
  int e = 0;
#pragma unroll 1
  for (; e + kExpertBatch <= m.K; e += kExpertBatch) {
    Raw16<DT> x[kExpertBatch];
#pragma unroll
    for (int b = 0; b < kExpertBatch; ++b) load16<DT>(xp[e + b], i, x[b]);
#pragma unroll
    for (int b = 0; b < kExpertBatch; ++b) merge_acc16<DT>(m.c, x[b], t0, acc);
  }
#pragma unroll 1
  for (; e < m.K; ++e) {
    Raw16<DT> x;
    load16<DT>(xp[e], i, x);
    merge_acc16<DT>(m.c, x, t0, acc);
  }
  store_merged16<DT>(T, i, t0, acc);
}

// DARE keep masks. A warp first draws the masks of its 32 groups for all K
// experts (expert e's mask is the Mask stream at step e) into shared memory:
// bit 8b + 7 of word q of (expert e, thread t) is element 4q + b of t's group.
// A group with an element whose mask byte equals the threshold's high byte
// (probability 1/256 per element and expert; its low 24 bits, MASK_LO stream,
// decide) goes to the warp's queue: a ballot gives every such lane its slot,
// so the main loop has no branch for it. The whole warp then draws the queued
// groups together, about K / 16 per lane; most warps meet such a group for
// every expert, and resolving it where it was met took as many instructions
// as the expert's Philox block.
// Dynamic shared memory: uint4 keep flags [K][kBlock], then the queues,
// 32 K entries (lane << 4 | expert) per warp.
size_t dare_smem_bytes(int K) {
  return (size_t)K * kBlock * sizeof(uint4) + (size_t)K * kBlock * sizeof(uint16_t);
}

struct DareShared {
  uint4* keep;      // keep[e * kBlock + thread]
  uint16_t* queue;  // this warp's
};

// Called by all 32 lanes of the warp (full: this lane has a vector group at
// element index g0; gw0: lane 0's group). Two experts' Mask blocks are drawn
// together (two independent Philox chains per thread). On return the warp's
// keep flags are complete.
template <int R>
__device__ __forceinline__ void dare_masks(const MArgs& m, const MTensor& T, bool full, uint64_t g0, uint64_t gw0,
                                           const DareShared& s) {
  const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
  const bool low = full && T.t_lo != 0u;
  const uint32_t below = (1u << lane) - 1u;
  int n = 0;
  auto draw = [&](const uint4& w, int e) {
    uint32_t kw[4];
    const bool tie = keep_bytes16(w, T.t_hi, kw) && low;
    s.keep[e * kBlock + threadIdx.x] = make_uint4(kw[0], kw[1], kw[2], kw[3]);
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, tie);
    if (tie) s.queue[n + __popc(b & below)] = (uint16_t)((lane << 4) | e);
    n += __popc(b);
  };
#pragma unroll 1
  for (int e = 0; e < m.K; e += 2) {
    const uint4 w0 = stream_block_at<R>(m.key, (uint32_t)e, S_MASK, T.tid, g0 >> 4);
    const uint4 w1 = stream_block_at<R>(m.key, (uint32_t)e + 1u, S_MASK, T.tid, g0 >> 4);
    draw(w0, e);
    if (e + 1 < m.K) draw(w1, e + 1);
  }
  __syncwarp();
#pragma unroll 1
  for (int j = lane; j < n; j += 32) {
    const uint32_t it = s.queue[j];
    const int owner = (int)(it >> 4), e = (int)(it & 15u);
    const uint64_t g = gw0 + 16 * (uint64_t)owner;
    uint32_t tb = tie_bits16(stream_block_at<R>(m.key, (uint32_t)e, S_MASK, T.tid, g >> 4), T.t_hi);
    uint32_t* kwp = reinterpret_cast<uint32_t*>(&s.keep[e * kBlock + wbase + owner]);
    while (tb) {
      const int k = __ffs(tb) - 1;
      tb &= tb - 1u;
      const uint4 l = stream_block_at<R>(m.key, (uint32_t)e, S_MASK_LO, T.tid, (g + (uint64_t)k) >> 2);
      if ((pick(l, (unsigned)(k & 3)) >> 8) < T.t_lo) kwp[k >> 2] |= 0x80u << (8 * (k & 3));  // one lane per group
    }
  }
  __syncwarp();
}

// prmt.b32 with sign-replicating selectors (nibble bit 3): two keep flags of
// a word spread over the 16-bit lanes of a mask.
template <int SEL>
__device__ __forceinline__ uint32_t spread_flags(uint32_t kw) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(kw), "n"(SEL));
  return r;
}

// Expert e's DARE contribution to a bf16 group: the expert's bf16 words are
// blended with theta0's by the keep masks (a dropped element takes theta0's
// bits), so a dropped element's Delta is fl(theta0 - theta0) = +0 and its
// multiply-add leaves acc unchanged (acc is never -0: it starts at +0 and a
// sum rounds to -0 only from two -0). This is exact while theta0 is finite;
// the caller takes the select path below for a group with an infinite or NaN
// theta0 (whose Delta would be NaN instead of unused).
__device__ __forceinline__ void dare_acc16_blend(float c, const uint4& km, const Raw16<DT_BF16>& x,
                                                 const Raw16<DT_BF16>& t0, const float2 (&b0)[8], float2 (&acc)[8]) {
  const float2 c2 = splat(c);
  const uint32_t kmw[4] = {km.x, km.y, km.z, km.w};
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    // 16-bit lanes of the word's two elements: flags 0, 1 (even h) or 2, 3 (odd h) of flag word h / 2
    const uint32_t lm = (h & 1) ? spread_flags<0xBBAA>(kmw[h >> 1]) : spread_flags<0x9988>(kmw[h >> 1]);
    const uint32_t xw = (x.r[h] & lm) | (t0.r[h] & ~lm);
    const float2 d = sub2_rn(make_float2(__uint_as_float(xw << 16), __uint_as_float(xw & 0xFFFF0000u)), b0[h]);
    acc[h] = fma2_rn(c2, d, acc[h]);
  }
}

// The same with a select per element after the multiply-add (fp32 groups, and
// bf16 groups whose theta0 is not finite).
template <int DT>
__device__ __forceinline__ void dare_acc16_select(float c, const uint4& km, const Raw16<DT>& x, const Raw16<DT>& t0,
                                                  float2 (&acc)[8]) {
  const float2 c2 = splat(c);
  const uint32_t kw[4] = {km.x, km.y, km.z, km.w};
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    const float2 b = t0.pair(h);
    const float2 d = sub2_rn(x.pair(h), b);
    const float2 f = fma2_rn(c2, d, acc[h]);
    acc[h] = make_float2(kept_of(kw, 2 * h) ? f.x : acc[h].x, kept_of(kw, 2 * h + 1) ? f.y : acc[h].y);
  }
}

// Some element of a bf16 group is infinite or NaN (exponent all ones).
__device__ __forceinline__ bool nonfinite16(const Raw16<DT_BF16>& v) {
  uint32_t nf = 0u;
#pragma unroll
  for (int h = 0; h < 8; ++h) nf |= (v.r[h] & 0x7F807F80u) + 0x00800080u;  // 0x8000 in a half iff its exponent is 0xFF
  return (nf & 0x80008000u) != 0u;
}

// Experts loaded together, the first of them before the keep masks are drawn.
template <int DT>
constexpr int kDareBatch = DT == DT_BF16 ? 4 : 2;

// DARE + TA on one 16-element group whose t0 and first kDareBatch experts are
// already loaded; keep flags from shared memory (masked) or all kept.
template <int DT>
__device__ __forceinline__ void dare_linear16(const MArgs& m, const MTensor& T, int t, int64_t i, bool masked,
                                              const Raw16<DT>& t0, Raw16<DT> (&x)[kDareBatch<DT>],
                                              const DareShared& s) {
  float2 acc[8], b0[8];
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    acc[h] = splat(0.0f);
    b0[h] = t0.pair(h);
    asm volatile("" : "+f"(b0[h].x), "+f"(b0[h].y));  // kept unpacked, not unpacked again for every expert
  }
  const void* const* xp = m.experts + t * m.K;
  bool blend = false;
  if (DT == DT_BF16) blend = !nonfinite16(*reinterpret_cast<const Raw16<DT_BF16>*>(&t0));
#pragma unroll 1
  for (int e = 0; e < m.K; e += kDareBatch<DT>) {
    if (e > 0) {
#pragma unroll
      for (int b = 0; b < kDareBatch<DT>; ++b)
        if (e + b < m.K) load16<DT>(xp[e + b], i, x[b]);
    }
#pragma unroll
    for (int b = 0; b < kDareBatch<DT>; ++b) {
      if (e + b < m.K) {
        const uint4 km = masked ? s.keep[(e + b) * kBlock + threadIdx.x]
                                : make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        if (DT == DT_BF16 && blend)
          dare_acc16_blend(m.c, km, *reinterpret_cast<const Raw16<DT_BF16>*>(&x[b]),
                           *reinterpret_cast<const Raw16<DT_BF16>*>(&t0), b0, acc);
        else
          dare_acc16_select<DT>(m.c, km, x[b], t0, acc);
      }
    }
  }
  store_merged16<DT>(T, i, t0, acc);
}

// ------------------------------------------------------------ TIES merge pass ---
// Eight consecutive elements as loaded (bf16: 16 bytes, fp32: 32).
template <int DT>
struct Raw8 {
  uint32_t r[DT == DT_BF16 ? 4 : 8];
  __device__ __forceinline__ float2 pair(int m) const {
    if (DT == DT_BF16) return make_float2(__uint_as_float(r[m] << 16), __uint_as_float(r[m] & 0xFFFF0000u));
    return make_float2(__uint_as_float(r[2 * m]), __uint_as_float(r[2 * m + 1]));
  }
};

template <int DT>
__device__ __forceinline__ void load8(const void* base, int64_t i, Raw8<DT>& v) {
  if constexpr (DT == DT_BF16) {
    asm("ld.global.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
        : "=r"(v.r[0]), "=r"(v.r[1]), "=r"(v.r[2]), "=r"(v.r[3])
        : "l"(static_cast<const uint16_t*>(base) + i));
  } else {
    ld32B(static_cast<const float*>(base) + i, v.r);
  }
}

// One expert's Delta of one element into the running sums: kept positive values
// (Delta >= lo), kept negative ones (Delta <= -lo), both together, and the two
// counts (positive in the low byte, negative in the next). Written out so that
// the additions are predicated: as C++ conditions they became branches (three
// times the merge pass's time), and as factors 1 and 0 of multiply-adds a
// comparison and a select each.
__device__ __forceinline__ void ties_add(float d, float lo, float& sum, float& pos, float& neg, uint32_t& cnt) {
  asm("{\n\t.reg .pred p, n;\n\t"
      "setp.ge.f32 p, %4, %5;\n\tsetp.le.f32 n, %4, %6;\n\t"
      "@p add.rn.f32 %0, %0, %4;\n\t@p add.rn.f32 %1, %1, %4;\n\t@p add.u32 %3, %3, 1;\n\t"
      "@n add.rn.f32 %0, %0, %4;\n\t@n add.rn.f32 %2, %2, %4;\n\t@n add.u32 %3, %3, 256;\n\t}"
      : "+f"(sum), "+f"(pos), "+f"(neg), "+r"(cnt)
      : "f"(d), "f"(lo), "f"(-lo));
}

// TIES on an 8-element group in one reading of the experts: beside the sum of
// the kept values that elects the sign, the kept positive values and the kept
// negative ones are summed and counted by themselves, each in expert order, so
// that the elected one's sum is the disjoint mean's numerator whatever the
// sign. Kept: key >= lo = max(thr, 1): a zero Delta changes no sum and agrees
// with no sign. A NaN Delta passes neither test, where the oracle's sum
// becomes NaN and elects nothing: false is returned (nothing is stored) if
// some Delta of the group is NaN, or infinities of both signs meet, and the
// caller takes the element path. BATCH: experts whose loads are in flight
// together; FULL: it divides their number (a build of its own: with the
// remainder's code beside it the loop spilled, and the pass took 7.2 ms
// instead of 4.2 for 8 experts of 1.07e9 bf16 elements).
template <int DT, int BATCH, bool FULL>
__device__ __forceinline__ bool merge_ties8(const MArgs& m, const void* t0_p, void* out_p, const void* const* xp,
                                            const float* lo, int64_t i) {
  Raw8<DT> t0;
  load8<DT>(t0_p, i, t0);
  float sum[8], pos[8], neg[8];
  uint32_t cnt[8];
  float2 all = splat(0.0f);  // NaN if some Delta is
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    sum[k] = pos[k] = neg[k] = 0.0f;
    cnt[k] = 0u;
  }
  auto add = [&](const Raw8<DT>& x, float l) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const float2 d = sub2_rn(x.pair(h), t0.pair(h));
      all = add2_rn(all, d);
      ties_add(d.x, l, sum[2 * h], pos[2 * h], neg[2 * h], cnt[2 * h]);
      ties_add(d.y, l, sum[2 * h + 1], pos[2 * h + 1], neg[2 * h + 1], cnt[2 * h + 1]);
    }
  };
#pragma unroll 1
  for (int e = 0; e < m.K; e += BATCH) {
    Raw8<DT> x[BATCH];
#pragma unroll
    for (int b = 0; b < BATCH; ++b)
      if (FULL || e + b < m.K) load8<DT>(xp[e + b], i, x[b]);
#pragma unroll
    for (int b = 0; b < BATCH; ++b)
      if (FULL || e + b < m.K) add(x[b], lo[e + b]);
  }
  if (isnan(__fadd_rn(all.x, all.y))) return false;
  float out[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float part = sum[k] > 0.0f ? pos[k] : neg[k];
    const uint32_t n = sum[k] > 0.0f ? (cnt[k] & 0xFFu) : (cnt[k] >> 8);
    const float mean = n && (sum[k] > 0.0f || sum[k] < 0.0f) ? __fdiv_rn(part, (float)n) : 0.0f;
    const float b = (k & 1) ? t0.pair(k >> 1).y : t0.pair(k >> 1).x;
    out[k] = __fadd_rn(b, __fmul_rn(m.gamma, mean));
  }
  if constexpr (DT == DT_BF16) {
    asm volatile("st.global.v4.b32 [%0], {%1,%2,%3,%4};" ::"l"(static_cast<uint16_t*>(out_p) + i),
                 "r"(pack_bf16x2(out[0], out[1])), "r"(pack_bf16x2(out[2], out[3])),
                 "r"(pack_bf16x2(out[4], out[5])), "r"(pack_bf16x2(out[6], out[7]))
                 : "memory");
  } else {
    uint32_t r[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k] = __float_as_uint(out[k]);
    st32B(static_cast<float*>(out_p) + i, r);
  }
  return true;
}

// Any method, one element (any alignment).
template <int R, int DT, int METHOD>
__device__ __forceinline__ void merge_elem(const MArgs& m, const MTensor& T, int t, int64_t i) {
  const float t0 = load1<DT>(T.theta0, i);
  const uint64_t g = (uint64_t)(T.elem_offset + i);
  float acc = 0.0f;
  if (METHOD == SMAT_MERGE_TIES) {
    float sum = 0.0f, part = 0.0f;
    int n = 0;
    for (int e = 0; e < m.K; ++e) {
      const float d = __fsub_rn(load1<DT>(m.experts[t * m.K + e], i), t0);
      if (abs_key(d) >= m.thr[t * m.K + e]) sum = __fadd_rn(sum, d);
    }
    for (int e = 0; e < m.K; ++e) {
      const float d = __fsub_rn(load1<DT>(m.experts[t * m.K + e], i), t0);
      if (abs_key(d) >= m.thr[t * m.K + e] && ((sum > 0.0f && d > 0.0f) || (sum < 0.0f && d < 0.0f))) {
        part = __fadd_rn(part, d);
        ++n;
      }
    }
    acc = __fmul_rn(m.gamma, n ? __fdiv_rn(part, (float)n) : 0.0f);
  } else {
    for (int e = 0; e < m.K; ++e) {
      const float d = __fsub_rn(load1<DT>(m.experts[t * m.K + e], i), t0);
      const bool kept = METHOD != SMAT_MERGE_DARE_TA || !(T.flags & TF_MASK) ||
                        elem_kept_at<R>(m.key, (uint32_t)e, T.tid, T.t_hi, T.t_lo, g);
      if (kept) acc = __fmaf_rn(m.c, d, acc);
    }
  }
  store1<DT>(T.out, i, __fadd_rn(t0, acc));
}

// TIES merge pass, one CTA per chunk (no draws: one build for all stream variants).
template <int DT, int BATCH, bool FULL>
__global__ void __launch_bounds__(kBlock, DT == DT_BF16 ? 3 : 2) ties_merge_kernel(const __grid_constant__ MArgs m) {
  __shared__ const void* s_x[kMergeMaxExperts];
  __shared__ float s_lo[kMergeMaxExperts];
  const Chunk ch = chunk_of(m, m.chunks, blockIdx.x);
  const MTensor& T = m.tensors[ch.tensor];
  const void* const t0_p = T.theta0;
  void* const out_p = T.out;
  const bool vec = (T.flags & TF_VEC) != 0u;
  if (threadIdx.x < m.K) {
    s_x[threadIdx.x] = m.experts[ch.tensor * m.K + threadIdx.x];
    const uint32_t thr = m.thr[ch.tensor * m.K + threadIdx.x];
    s_lo[threadIdx.x] = __uint_as_float(thr > 1u ? thr : 1u);
  }
  __syncthreads();
  for (int64_t i = ch.begin + 8 * (int64_t)threadIdx.x; i < ch.end; i += 8 * (int64_t)kBlock) {
    if (vec && i + 8 <= ch.end && merge_ties8<DT, BATCH, FULL>(m, t0_p, out_p, s_x, s_lo, i)) continue;
    const int64_t e_end = (i + 8 < ch.end) ? i + 8 : ch.end;
#pragma unroll 1
    for (int64_t e = i; e < e_end; ++e) merge_elem<10, DT, SMAT_MERGE_TIES>(m, T, ch.tensor, e);
  }
}

// WA and TA (they differ in m.c alone), one CTA per chunk. bf16 at three CTAs per SM (76 registers): two left 7% of the copy
// bandwidth unused, four spill (8 experts of 1e8 elements: 332, 309 and 357 us,
// 16 experts 572, 541 and 636 us).
template <int DT>
constexpr int kLinearCtas = DT == DT_BF16 ? 3 : 2;

template <int DT>
__global__ void __launch_bounds__(kBlock, kLinearCtas<DT>) merge_kernel(const __grid_constant__ MArgs m) {
  const Chunk ch = chunk_of(m, m.chunks, blockIdx.x);
  const MTensor& T = m.tensors[ch.tensor];
  const bool vec = (T.flags & TF_VEC) != 0u;
  for (int64_t i = ch.begin + 16 * (int64_t)threadIdx.x; i < ch.end; i += 16 * (int64_t)kBlock) {
    if (vec && i + 16 <= ch.end) {
      merge_linear16<DT>(m, T, ch.tensor, i);
    } else {
      const int64_t e_end = (i + 16 < ch.end) ? i + 16 : ch.end;
      for (int64_t e = i; e < e_end; ++e) merge_elem<10, DT, SMAT_MERGE_TA>(m, T, ch.tensor, e);
    }
  }
}

// DARE + TA. The loop runs the same number of iterations on every lane of
// the CTA (the keep masks are drawn warp-cooperatively); t0 and the first
// experts are loaded before the masks are drawn, so the loads are in flight
// during the Philox work.
template <int R, int DT>
__global__ void __launch_bounds__(kBlock, 2) dare_kernel(const __grid_constant__ MArgs m) {
  extern __shared__ __align__(16) unsigned char dare_smem[];
  const int warp = threadIdx.x >> 5;
  DareShared s;
  s.keep = reinterpret_cast<uint4*>(dare_smem);
  s.queue = reinterpret_cast<uint16_t*>(s.keep + m.K * kBlock) + 32 * m.K * warp;
  for (int64_t ci = blockIdx.x; ci < m.chunks.n; ci += gridDim.x) {
    const Chunk ch = chunk_of(m, m.chunks, ci);
    const MTensor& T = m.tensors[ch.tensor];
    const bool vec = (T.flags & TF_VEC) != 0u;
    const bool masked = (T.flags & TF_MASK) != 0u;
    const void* const* xp = m.experts + ch.tensor * m.K;
    for (int64_t base = ch.begin; base < ch.end; base += 16 * (int64_t)kBlock) {
      const int64_t i = base + 16 * (int64_t)threadIdx.x;
      const bool full = vec && i + 16 <= ch.end;
      Raw16<DT> t0, x[kDareBatch<DT>];
      if (full) {
        load16<DT>(T.theta0, i, t0);
#pragma unroll
        for (int b = 0; b < kDareBatch<DT>; ++b)
          if (b < m.K) load16<DT>(xp[b], i, x[b]);
      }
      if (masked)
        dare_masks<R>(m, T, full, (uint64_t)(T.elem_offset + i),
                      (uint64_t)(T.elem_offset + base + 16 * 32 * (int64_t)warp), s);
      if (full) {
        dare_linear16<DT>(m, T, ch.tensor, i, masked, t0, x, s);
      } else if (i < ch.end) {
        const int64_t e_end = (i + 16 < ch.end) ? i + 16 : ch.end;
        for (int64_t e = i; e < e_end; ++e) merge_elem<R, DT, SMAT_MERGE_DARE_TA>(m, T, ch.tensor, e);
      }
    }
  }
}

// --------------------------------------------------- TIES threshold selection ---
template <int DT>
__device__ __forceinline__ void load_lane(const void* base, int64_t i, Raw16<DT>& v) {
  load16<DT>(base, i, v);
}
template <int DT>
__device__ __forceinline__ void load_lane(const void* base, int64_t i, Raw8<DT>& v) {
  load8<DT>(base, i, v);
}

// A thread's 32 bytes of one array: 16 bf16 or 8 fp32 elements. (16 fp32
// elements of theta0 and four experts took 147 registers, one CTA per SM.)
template <int DT>
using RawLane = std::conditional_t<DT == DT_BF16, Raw16<DT>, Raw8<DT>>;
template <int DT>
constexpr int kLaneElems = DT == DT_BF16 ? 16 : 8;

// Elements sampled per slot, as 16-element groups spread evenly over the
// tensor; a tensor of at most kWholeElems elements is read whole.
constexpr int kSampleElems = 1 << 15;
constexpr int kWholeElems = 1 << 16;

// The interval [lo, lo + width) as the slot's next one: the smallest shift
// whose 2046 bins cover it from a multiple of 2^shift.
__device__ __forceinline__ void set_interval(TiesSlot& S, uint32_t lo, uint64_t width) {
  int s = 0;
  while ((uint64_t(kInner) << s) < width + (lo & ((1u << s) - 1u))) ++s;
  S.lo = lo & ~((1u << s) - 1u);
  S.shift = s;
}

__device__ __forceinline__ unsigned long long count_at(const uint32_t* p) { return *p; }  // shared memory
__device__ __forceinline__ unsigned long long count_at(const unsigned long long* p) {     // global bin (numel < 2^40)
  return __ldcg(p) & ((1ull << 41) - 1u);
}

// The bin that holds the r-th entry counted from the top of a histogram of nb
// bins and the entries above that bin, by all NT threads of the CTA; digit -1
// if there are fewer than r.
template <int NT>
struct SelectShared {
  unsigned long long sum[NT];
  int digit;
  long long above;
};

template <int NT, typename Count>
__device__ __forceinline__ void select_from_top(const Count* hist, int nb, long long r, SelectShared<NT>& sh) {
  const int per = nb / NT;  // bins per thread, highest bins in thread 0
  unsigned long long local = 0;
  const int top = nb - 1 - threadIdx.x * per;
  for (int k = 0; k < per; ++k) local += count_at(hist + top - k);
  sh.sum[threadIdx.x] = local;
  if (threadIdx.x == 0) {
    sh.digit = -1;
    sh.above = 0;
  }
  __syncthreads();
  // inclusive scan from the top (Hillis-Steele)
  for (int o = 1; o < NT; o <<= 1) {
    const unsigned long long v = threadIdx.x >= o ? sh.sum[threadIdx.x - o] : 0ull;
    __syncthreads();
    sh.sum[threadIdx.x] += v;
    __syncthreads();
  }
  const unsigned long long incl = sh.sum[threadIdx.x];
  const unsigned long long excl = incl - local;
  if (r > 0 && (long long)excl < r && r <= (long long)incl) {
    unsigned long long acc = excl;
    for (int k = 0; k < per; ++k) {
      const unsigned long long c = count_at(hist + top - k);
      if ((long long)(acc + c) >= r) {
        sh.digit = top - k;
        sh.above = (long long)acc;
        break;
      }
      acc += c;
    }
  }
  __syncthreads();
}

// The first interval of each slot, one CTA per slot: two order statistics of
// the sample, six standard deviations of the sampled rank to either side of
// r's share, each by a radix select of three digits (11, 11 and 10 bits). The
// sample's keys stay in registers, 32 per thread (65,536 keys read anew for each digit
// took 50 us for an fp32 slot, these take 33); a tensor that is read whole comes from L2
// after the first digit.
constexpr int kSampleThreads = 1024;

template <int DT>
__global__ void __launch_bounds__(kSampleThreads) ties_sample_kernel(const __grid_constant__ MArgs m) {
  __shared__ uint32_t h[2][kHistBins];
  __shared__ SelectShared<kSampleThreads> sh;
  const int slot = blockIdx.x;
  const MTensor& T = m.tensors[slot / m.K];
  const void* x = m.experts[slot];
  const int64_t n = T.numel, r = m.rank[slot];
  if (n <= 0) {
    if (threadIdx.x == 0) {
      m.slots[slot].done = 1u;
      atomicAdd(m.n_done, 1u);
    }
    return;
  }
  const bool all = n <= kWholeElems, vec = (T.flags & TF_VEC) != 0u;
  const int64_t seen = all ? n : kSampleElems;
  // ranks in the sample, counted from the largest key: the upper end of the
  // interval and the lower one
  long long rank[2] = {r, r};
  if (!all) {
    const double p = (double)r / (double)n, at = p * (double)seen;
    const double d = 6.0 * sqrt(at * (1.0 - p)) + 16.0;
    rank[0] = (long long)ceil(at - d);
    rank[1] = (long long)floor(at + d);
  }
  const bool open_top = rank[0] < 1, open_bottom = rank[1] > seen;
  if (open_top) rank[0] = 1;
  if (open_bottom) rank[1] = seen;
  constexpr int kMine = kSampleElems / kSampleThreads, kLane = kLaneElems<DT>;
  uint32_t prefix[2] = {0u, 0u};
  const int shifts[3] = {21, 10, 0}, widths[3] = {11, 11, 10};
  // each(count) calls count for every key of the sample
  auto select = [&](auto&& each) {
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = shifts[pass], nb = 1 << widths[pass];
      const uint32_t decided = pass == 0 ? 0u : ~0u << shifts[pass - 1];
      const bool same = prefix[0] == prefix[1];
      for (int b = threadIdx.x; b < 2 * kHistBins; b += kSampleThreads) (&h[0][0])[b] = 0u;
      __syncthreads();
      each([&](uint32_t key) {
        const uint32_t digit = (key >> shift) & (uint32_t)(nb - 1);
        if ((key & decided) == prefix[0]) atomicAdd(&h[0][digit], 1u);
        if (!same && (key & decided) == prefix[1]) atomicAdd(&h[1][digit], 1u);
      });
      __syncthreads();
      for (int q = 0; q < 2; ++q) {
        select_from_top(h[same ? 0 : q], nb, rank[q], sh);
        prefix[q] |= (uint32_t)sh.digit << shift;
        rank[q] -= sh.above;
        __syncthreads();
      }
    }
  };
  // the keys of the lane of kLane elements at i
  auto lane_keys = [&](int64_t i, uint32_t* keys) {
    RawLane<DT> t0, y;
    load_lane<DT>(T.theta0, i, t0);
    load_lane<DT>(x, i, y);
#pragma unroll
    for (int q = 0; q < kLane / 2; ++q) {
      const float2 d = sub2_rn(y.pair(q), t0.pair(q));
      keys[2 * q] = abs_key(d.x);
      keys[2 * q + 1] = abs_key(d.y);
    }
  };
  auto key_at = [&](int64_t i) { return abs_key(__fsub_rn(load1<DT>(x, i), load1<DT>(T.theta0, i))); };
  if (all) {
    select([&](auto&& count) {
      for (int i = kLane * (int)threadIdx.x; i < (int)n; i += kLane * kSampleThreads) {
        if (vec && i + kLane <= (int)n) {
          uint32_t keys[kLane];
          lane_keys(i, keys);
#pragma unroll
          for (int k = 0; k < kLane; ++k) count(keys[k]);
        } else {
          for (int k = i; k < (int)n && k < i + kLane; ++k) count(key_at(k));
        }
      }
    });
  } else {
    uint32_t mine[kMine];
#pragma unroll
    for (int l = 0; l < kMine / kLane; ++l) {
      const int at = kLane * ((int)threadIdx.x + l * kSampleThreads);  // place in the sample
      const int64_t i = 16 * ((int64_t)(at / 16) * (n / 16) / (kSampleElems / 16)) + at % 16;
      if (vec) {
        lane_keys(i, mine + l * kLane);
      } else {
#pragma unroll
        for (int k = 0; k < kLane; ++k) mine[l * kLane + k] = key_at(i + k);
      }
    }
    select([&](auto&& count) {
#pragma unroll
      for (int k = 0; k < kMine; ++k) count(mine[k]);
    });
  }
  if (threadIdx.x == 0) {
    TiesSlot S;
    S.done = all ? 1u : 0u;
    S.pad = 0u;
    // NaN samples end the interval at kInfKey: from a NaN's key a miss below
    // would span more than the passes can decide
    const uint32_t lo = open_bottom ? 0u : min(prefix[1], kInfKey);
    const uint32_t hi = open_top ? kInfKey : min(prefix[0], kInfKey);
    set_interval(S, lo, (uint64_t)hi - lo + 1);
    m.slots[slot] = S;
    if (all) {
      m.thr[slot] = prefix[0];
      atomicAdd(m.n_done, 1u);
    }
  }
}

// One pass of the selection. A work item is a chunk and up to kHistExperts of
// its experts: theta0 is read once for them, and each thread has theta0's and
// every expert's 32-byte load in flight at once; one shared-memory histogram
// per expert, flushed into the 64-bit global bins.
//
// Every key counts (the outer bins take what lies outside the interval), so
// that no branch surrounds the shared-memory atomic: a pass that tested each
// key against the digits decided so far and branched around the atomic took
// 5.7 ms for 8 experts of 1.07e9 bf16 elements, bound by issue slots; this one
// takes 3.0 (2.9 at HBM speed), bound by the shared-memory atomics (LSU data
// pipe 72% busy).
//
// bf16: a key that is not its bin's first (differences of bf16 values near
// each other are multiples of coarse powers of two, so few keys are) sends its
// group and expert to a list; after the chunk the CTA counts such keys per
// bin. In the loop this is one operation per two keys and a seldom taken
// branch; flagging there took 0.6 of 4.0 ms, and a flag without a count sent most
// bf16 thresholds to a second pass. A shared bin holds the count
// (17 bits, a chunk has at most 2^16 elements) and the count of those keys (15 bits);
// a global bin the sums in bits 0 to 40 and 41 to 62. Where such keys are too
// many to count (the list is full, or kOffMost of them in one chunk's bin)
// bit 63 says so.
constexpr int kHistExperts = 4;
constexpr uint32_t kOffOne = 1u << 17;
constexpr uint32_t kOffMost = 256u;  // sums of 2^14 chunks stay below 2^22
constexpr int64_t kOffChunks = 1 << 14;
constexpr int kOffList = 512;

constexpr int kHistCtas(int dtype) { return dtype == DT_BF16 ? 4 : 3; }  // per SM

template <int DT>
__global__ void __launch_bounds__(kBlock, kHistCtas(DT)) ties_hist_kernel(const __grid_constant__ MArgs m) {
  __shared__ uint32_t h[kHistExperts * kHistBins];
  __shared__ uint16_t list[kOffList];  // (group << 2) | expert of the batch
  __shared__ int n_list;
  if (*m.n_done == (uint32_t)m.n_slots) return;
  const int nbat = (m.K + kHistExperts - 1) / kHistExperts;
  const int64_t items = m.hist_chunks.n * nbat;
  for (int64_t w = blockIdx.x; w < items; w += gridDim.x) {
    const int e0 = (int)(w % nbat) * kHistExperts;
    const int ne = m.K - e0 < kHistExperts ? m.K - e0 : kHistExperts;
    const Chunk ch = chunk_of(m, m.hist_chunks, w / nbat);
    const MTensor& T = m.tensors[ch.tensor];
    const int slot0 = ch.tensor * m.K + e0;
    uint32_t lo[kHistExperts];
    int sh[kHistExperts];
    const void* xp[kHistExperts];
    bool any = false;
#pragma unroll
    for (int b = 0; b < kHistExperts; ++b) {
      xp[b] = nullptr;
      lo[b] = 0u;
      sh[b] = 0;
      if (b < ne) {
        const TiesSlot S = m.slots[slot0 + b];
        if (!S.done) {  // a decided expert is not read again
          any = true;
          xp[b] = m.experts[slot0 + b];
          lo[b] = S.lo;
          sh[b] = S.shift;
        }
      }
    }
    if (!any) continue;  // the same slots in every thread
    for (int b = threadIdx.x; b < kHistExperts * kHistBins; b += kBlock) h[b] = 0u;
    if (threadIdx.x == 0) n_list = 0;
    __syncthreads();
    // bin of a key: 1 + (key - lo) / 2^shift, clamped to [0, 2047]
    auto bin_of = [&](uint32_t key, uint32_t low, int shift) {
      return __viaddmin_s32_relu((int)(key - low) >> shift, 1, kHistBins - 1);
    };
    const bool vec = (T.flags & TF_VEC) != 0u;
    const void* t0p = T.theta0;
    for (int64_t i = ch.begin + kLaneElems<DT> * (int64_t)threadIdx.x; i < ch.end; i += kLaneElems<DT> * (int64_t)kBlock) {
      if (vec && i + kLaneElems<DT> <= ch.end) {
        RawLane<DT> t0, x[kHistExperts];
        load_lane<DT>(t0p, i, t0);
#pragma unroll
        for (int b = 0; b < kHistExperts; ++b)
          if (xp[b]) load_lane<DT>(xp[b], i, x[b]);
#pragma unroll
        for (int b = 0; b < kHistExperts; ++b) {
          if (xp[b]) {
            uint32_t bits = 0u;
#pragma unroll
            for (int q = 0; q < kLaneElems<DT> / 2; ++q) {
              const float2 d = sub2_rn(x[b].pair(q), t0.pair(q));
              const uint32_t k0 = abs_key(d.x), k1 = abs_key(d.y);
              bits |= k0 | k1;
              atomicAdd(&h[b * kHistBins + bin_of(k0, lo[b], sh[b])], 1u);
              atomicAdd(&h[b * kHistBins + bin_of(k1, lo[b], sh[b])], 1u);
            }
            if (DT == DT_BF16 && (bits & ((1u << sh[b]) - 1u)) != 0u) {
              const int at = atomicAdd(&n_list, 1);
              if (at < kOffList) list[at] = (uint16_t)(((uint32_t)(i - ch.begin) >> 4 << 2) | b);
            }
          }
        }
      } else {
        const int64_t e_end = (i + kLaneElems<DT> < ch.end) ? i + kLaneElems<DT> : ch.end;
        for (int64_t k = i; k < e_end; ++k) {
          const float t0 = load1<DT>(t0p, k);
#pragma unroll
          for (int b = 0; b < kHistExperts; ++b) {
            if (xp[b]) {
              const uint32_t key = abs_key(__fsub_rn(load1<DT>(xp[b], k), t0));
              atomicAdd(&h[b * kHistBins + bin_of(key, lo[b], sh[b])], 1u);
              if (DT == DT_BF16 && (key & ((1u << sh[b]) - 1u)) != 0u) {
                const int at = atomicAdd(&n_list, 1);  // the group may be listed more than once: it is counted too often
                if (at < kOffList) list[at] = (uint16_t)(((uint32_t)(i - ch.begin) >> 4 << 2) | b);
              }
            }
          }
        }
      }
    }
    __syncthreads();
    const int listed = n_list;
    if (DT == DT_BF16 && listed > 0 && listed <= kOffList) {
      // sixteen threads per entry, an element each
      for (int j = threadIdx.x >> 4; j < listed; j += kBlock / 16) {
        const uint32_t it = list[j];
        const int b = (int)(it & 3u);
        const int64_t k = ch.begin + 16 * (int64_t)(it >> 2) + (threadIdx.x & 15);
        if (k < ch.end) {
          const TiesSlot S = m.slots[slot0 + b];
          const uint32_t key = abs_key(__fsub_rn(load1<DT>(m.experts[slot0 + b], k), load1<DT>(t0p, k)));
          const int bin = bin_of(key, S.lo, S.shift);
          uint32_t* p = &h[b * kHistBins + bin];
          // past kOffMost the exact count no longer matters (at most 256 threads add beyond it)
          if ((key & ((1u << S.shift) - 1u)) != 0u && bin > 0 && bin < kHistBins - 1 &&
              (*(volatile uint32_t*)p >> 17) < kOffMost)
            atomicAdd(p, kOffOne);
        }
      }
      __syncthreads();
    }
    // the ne histograms are consecutive slots' bins in the global array
    unsigned long long* gh = m.hist + (size_t)slot0 * kHistBins;
    const uint32_t most = T.numel <= kOffChunks * m.hist_chunks.elems ? kOffMost : 1u;
    for (int b = threadIdx.x; b < ne * kHistBins; b += kBlock) {
      const uint32_t c = h[b];
      if (c) {
        const uint32_t off = c >> 17;
        atomicAdd(gh + b, (unsigned long long)(c & (kOffOne - 1u)) | (off < most ? (unsigned long long)off << 41 : 0ull));
        if (off >= most || listed > kOffList) atomicOr(gh + b, 1ull << 63);
      }
    }
    __syncthreads();
  }
}

// After a pass, one CTA per slot: the bin that holds the r-th largest key either
// decides the threshold or is the next pass's interval (and the histogram is
// cleared). A launch of its own, about 6 us: done by the CTA that finishes a
// tensor's last item it lengthened the pass by 0.75 of 3.4 ms (the call's
// registers) and a small list's by 50 us (its slots one after the other).
template <int DT>
__global__ void __launch_bounds__(kBlock) ties_select_kernel(const __grid_constant__ MArgs m) {
  __shared__ SelectShared<kBlock> sh;
  const int slot = blockIdx.x;
  TiesSlot S = m.slots[slot];
  if (S.done) return;
  unsigned long long* gh = m.hist + (size_t)slot * kHistBins;
  const long long r = m.rank[slot];
  select_from_top(gh, kHistBins, r, sh);
  if (threadIdx.x == 0) {
    const int b = sh.digit;
    const uint64_t past = (uint64_t)S.lo + (uint64_t(kInner) << S.shift);  // first key above the interval
    uint32_t thr = 0u;
    if (b <= 0) {
      set_interval(S, 0u, S.lo);
    } else if (b == kHistBins - 1 && past <= kInfKey) {
      set_interval(S, (uint32_t)past, kInfKey + 1u - past);
    } else if (b == kHistBins - 1) {  // NaN keys alone are left: the hardware's NaN
      thr = 0x7FFFFFFFu;
      S.done = 1u;
    } else {
      const uint32_t first = S.lo + ((uint32_t)(b - 1) << S.shift);
      // the bin's keys that are not its first are all larger: r - above is past them
      const unsigned long long c = __ldcg(gh + b);
      const bool counted = DT == DT_BF16 && (c >> 63) == 0ull;
      if (S.shift == 0 || (counted && r - sh.above > (long long)(c >> 41))) {
        thr = first;
        S.done = 1u;
      } else {
        set_interval(S, first, uint64_t(1) << S.shift);
      }
    }
    m.slots[slot] = S;
    // an undecided slot holds its interval's lower end: never a threshold that trims nothing
    m.thr[slot] = S.done ? thr : S.lo;
    if (S.done) atomicAdd(m.n_done, 1u);
  }
  __syncthreads();  // the bins have been read
  for (int b = threadIdx.x; b < kHistBins; b += kBlock) gh[b] = 0ull;
}

template <int R, int DT>
cudaError_t dare_run(const MArgs& m, int grid, cudaStream_t s) {
  const size_t smem = dare_smem_bytes(m.K);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(dare_kernel<R, DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem);
    if (e != cudaSuccess) return e;
  }
  dare_kernel<R, DT><<<grid, kBlock, smem, s>>>(m);
  return cudaGetLastError();
}

// ------------------------------------------------------------------- host ---
struct MLayout {
  size_t tensors, first, experts, thr, slots, n_done, rank, hist, total;
};

size_t align_m(size_t x) { return (x + kMergeAlign - 1) / kMergeAlign * kMergeAlign; }

// What merge_check finds of a list: its elements, chunk size, chunks and dtype
// (one dtype per call).
struct MPlan {
  int64_t total, chunk, n_chunks;
  int32_t dtype;
};

// A workspace's bytes grow with the tensors and experts alone.
MLayout merge_layout(int32_t n, int K, bool ties) {
  MLayout L;
  size_t off = 0;
  const size_t slots = (size_t)n * (size_t)K;
  L.tensors = off; off = align_m(off + sizeof(MTensor) * (size_t)n);
  L.first = off;   off = align_m(off + sizeof(int32_t) * ((size_t)n + 1) * (ties ? 2 : 1));  // chunks, hist_chunks
  L.experts = off; off = align_m(off + sizeof(void*) * slots);
  L.thr = off;     off = align_m(off + sizeof(uint32_t) * slots);
  L.slots = off;   off = align_m(off + sizeof(TiesSlot) * slots);
  L.n_done = off;  off = align_m(off + sizeof(uint32_t));
  L.rank = off;    off = align_m(off + sizeof(int64_t) * slots);
  L.hist = off;    off = align_m(off + (ties ? sizeof(unsigned long long) * kHistBins * slots : 0));
  L.total = off;
  return L;
}

smat_status mfail(smat_status s, const char* fmt, ...) {
  char buf[256];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  return (smat_status)record_error_code((int)s, buf);
}

bool m_overlaps(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + nb && y < x + na;
}

// Host-side validation (no device access).
smat_status merge_check(const smat_merge_tensor* t, int32_t n, const smat_merge_config* cfg, MPlan* plan) {
  if (!cfg) return mfail(SMAT_ERR_INVALID_ARG, "cfg is NULL");
  if (cfg->method < SMAT_MERGE_WA || cfg->method > SMAT_MERGE_TIES)
    return mfail(SMAT_ERR_UNSUPPORTED, "merge method %d not supported", cfg->method);
  if (cfg->n_experts < 1 || cfg->n_experts > kMergeMaxExperts)
    return mfail(SMAT_ERR_INVALID_ARG, "n_experts %d not in [1, %d]", cfg->n_experts, kMergeMaxExperts);
  if (!std::isfinite(cfg->gamma)) return mfail(SMAT_ERR_INVALID_ARG, "gamma not finite");
  if (!(cfg->p_drop >= 0.0f && cfg->p_drop < 1.0f)) return mfail(SMAT_ERR_INVALID_ARG, "p_drop not in [0, 1)");
  if (!(cfg->retention > 0.0f && cfg->retention <= 1.0f))
    return mfail(SMAT_ERR_INVALID_ARG, "retention not in (0, 1]");
  if (cfg->philox_rounds != 0 && cfg->philox_rounds != 7 && cfg->philox_rounds != 10)
    return mfail(SMAT_ERR_UNSUPPORTED, "philox_rounds %d not supported (7 or 10)", cfg->philox_rounds);
  if (cfg->flags != 0) return mfail(SMAT_ERR_UNSUPPORTED, "unknown flags 0x%x", cfg->flags);
  if (n < 0 || (n > 0 && !t)) return mfail(SMAT_ERR_INVALID_ARG, "bad tensor list");
  std::unordered_set<uint32_t> ids;
  int64_t nc = 0, total = 0;
  for (int32_t k = 0; k < n; ++k) {
    const smat_merge_tensor& d = t[k];
    if (d.numel < 0 || d.numel >= (int64_t(1) << 40))
      return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: numel out of range", k);
    if (d.elem_offset < 0 || d.elem_offset >= (int64_t(1) << 62) - d.numel)
      return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: elem_offset out of range", k);
    if (d.tensor_id >= kGlobalAlphaTensor) return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: tensor_id too large", k);
    if (!ids.insert(d.tensor_id).second) return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: duplicate tensor_id", k);
    if (d.dtype != SMAT_F32 && d.dtype != SMAT_BF16)
      return mfail(SMAT_ERR_UNSUPPORTED, "tensor %d: dtype %d not supported", k, d.dtype);
    if (d.dtype != t[0].dtype) return mfail(SMAT_ERR_UNSUPPORTED, "tensor %d: one dtype per merge call", k);
    if (d.numel > 0) {
      const size_t es = d.dtype == SMAT_BF16 ? 2 : 4, bytes = es * (size_t)d.numel;
      if (!d.theta0 || !d.out || !d.experts) return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: NULL pointer", k);
      if ((uintptr_t)d.theta0 % es || (uintptr_t)d.out % es)
        return mfail(SMAT_ERR_ALIGNMENT, "tensor %d: pointer not aligned to its element size", k);
      if (d.out != d.theta0 && m_overlaps(d.out, bytes, d.theta0, bytes))
        return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: out overlaps theta0 without being equal to it", k);
      for (int e = 0; e < cfg->n_experts; ++e) {
        const void* x = d.experts[e];
        if (!x) return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: expert %d is NULL", k, e);
        if ((uintptr_t)x % es) return mfail(SMAT_ERR_ALIGNMENT, "tensor %d: expert %d misaligned", k, e);
        if (m_overlaps(d.out, bytes, x, bytes))
          return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: out overlaps expert %d", k, e);
      }
    }
    total = std::min(total + d.numel, int64_t(1) << 62);
  }
  const int64_t chunk = merge_chunk_for(total);
  for (int32_t k = 0; k < n; ++k) nc += (t[k].numel + chunk - 1) / chunk;
  if (nc >= (int64_t(1) << 31)) return mfail(SMAT_ERR_INVALID_ARG, "too many chunks");
  *plan = {total, chunk, nc, n > 0 ? t[0].dtype : SMAT_F32};
  return SMAT_OK;
}

// Chunk of the threshold passes: their CTAs clear and flush up to 32 KB of bins per
// item, so items are as long as they can be (2^16 elements) while they fill whole
// rounds of the resident CTAs, of which the tensors' short last chunks take at most
// half. Two experts of 1.8e7 fp32 elements: 52 and 48 us for the two passes that
// count in the merge kernels' chunks of 2^13, 44 and 41 in one round.
int64_t hist_chunk_for(const MPlan& p, int32_t n, int K, int sms) {
  const int64_t nbat = (K + kHistExperts - 1) / kHistExperts;
  const int64_t resident = std::max<int64_t>(kHistCtas(p.dtype) * (int64_t)sms / nbat, 1);
  int64_t chunk = kMergeChunkMax + 1;
  for (int64_t rounds = 1; chunk > kMergeChunkMax; ++rounds) {
    const int64_t items = resident * rounds - n;
    if (2 * items >= resident * rounds) chunk = (p.total + items - 1) / items;
  }
  const int64_t step = 16 * (int64_t)kBlock;
  return std::min(std::max((chunk + step - 1) / step * step, kMergeChunkMin), kMergeChunkMax);
}

template <int DT, int BATCH, bool FULL>
cudaError_t ties_merge_run(const MArgs& m, cudaStream_t s) {
  ties_merge_kernel<DT, BATCH, FULL><<<(int)m.chunks.n, kBlock, 0, s>>>(m);
  return cudaGetLastError();
}

template <int DT>
cudaError_t merge_launch(MArgs m, int64_t slots, int64_t largest, int rounds, int sms, cudaStream_t s) {
  if (m.method == SMAT_MERGE_TIES) {
    const int64_t items = m.hist_chunks.n * ((m.K + kHistExperts - 1) / kHistExperts);  // one CTA each
    m.n_slots = (int32_t)slots;
    ties_sample_kernel<DT><<<(int)slots, kSampleThreads, 0, s>>>(m);
    // no pass where every tensor is small enough for the sample to decide
    for (int p = 0; p < (largest > kWholeElems ? kPasses : 0); ++p) {
      ties_hist_kernel<DT><<<(int)std::min(items, int64_t(INT32_MAX)), kBlock, 0, s>>>(m);
      ties_select_kernel<DT><<<(int)slots, kBlock, 0, s>>>(m);
    }
    if constexpr (DT == DT_BF16)
      if (m.K % 8 == 0) return ties_merge_run<DT, 8, true>(m, s);
    if (m.K % 4 == 0) return ties_merge_run<DT, 4, true>(m, s);
    if (m.K == 2) return ties_merge_run<DT, 2, true>(m, s);
    return ties_merge_run<DT, 4, false>(m, s);
  }
  // one CTA per chunk, started by the hardware as others end (8 experts of 1e8 bf16
  // elements 309 -> 306 us, 16 experts 542 -> 534 us); DARE's CTAs, with their
  // shared memory, are worth keeping (4e7 elements: 175 against 187 us)
  if (m.method == SMAT_MERGE_DARE_TA) {
    const int grid = (int)std::min(m.chunks.n, 2 * (int64_t)sms);
    return rounds == 7 ? dare_run<7, DT>(m, grid, s) : dare_run<10, DT>(m, grid, s);
  }
  merge_kernel<DT><<<(int)m.chunks.n, kBlock, 0, s>>>(m);
  return cudaGetLastError();
}

}  // namespace
}  // namespace smat

using namespace smat;

extern "C" size_t smat_merge_workspace_bytes(const smat_merge_tensor* tensors, int32_t n_tensors,
                                             const smat_merge_config* cfg) {
  MPlan plan;
  if (merge_check(tensors, n_tensors, cfg, &plan) != SMAT_OK) return 0;
  return merge_layout(n_tensors, cfg->n_experts, cfg->method == SMAT_MERGE_TIES).total;
}

extern "C" smat_status smat_merge(const smat_merge_tensor* tensors, int32_t n_tensors, const smat_merge_config* cfg,
                                  void* d_workspace, size_t workspace_bytes, smat_stream_t stream) {
  MPlan plan;
  smat_status st = merge_check(tensors, n_tensors, cfg, &plan);
  if (st != SMAT_OK) return st;
  const int K = cfg->n_experts;
  const bool ties = cfg->method == SMAT_MERGE_TIES;
  const MLayout L = merge_layout(n_tensors, K, ties);
  if (!d_workspace || (uintptr_t)d_workspace % kMergeAlign)
    return mfail(SMAT_ERR_WORKSPACE, "workspace NULL or not 256-byte aligned");
  if (workspace_bytes < L.total) return mfail(SMAT_ERR_WORKSPACE, "workspace %zu < %zu bytes", workspace_bytes, L.total);
  GpuAccess access;
  for (int32_t k = 0; k < n_tensors; ++k) {
    if (tensors[k].numel <= 0) continue;
    int ok = access.check(tensors[k].theta0) == 1 && access.check(tensors[k].out) == 1;
    for (int e = 0; ok && e < K; ++e) ok = access.check(tensors[k].experts[e]) == 1;
    if (!ok) return mfail(SMAT_ERR_INVALID_ARG, "tensor %d: a pointer is not accessible from the GPU", k);
  }
  if (n_tensors == 0 || plan.n_chunks == 0) return SMAT_OK;
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return mfail(SMAT_ERR_CUDA, "device query failed");

  // tables (host), then one upload each
  const float keep = 1.0f - cfg->p_drop;
  const uint64_t T = (uint64_t)std::floor((double)keep * 4294967296.0);
  std::vector<MTensor> ht((size_t)n_tensors);
  const int64_t hist_chunk = hist_chunk_for(plan, n_tensors, K, sms);
  std::vector<int32_t> first(((size_t)n_tensors + 1) * (ties ? 2 : 1), 0);
  std::vector<const void*> hx((size_t)n_tensors * (size_t)K, nullptr);
  std::vector<int64_t> hrank((size_t)n_tensors * (size_t)K, 0);
  for (int32_t k = 0; k < n_tensors; ++k) {
    const smat_merge_tensor& d = tensors[k];
    MTensor& M = ht[(size_t)k];
    std::memset(&M, 0, sizeof(M));
    M.theta0 = d.theta0;
    M.out = d.out;
    M.numel = d.numel;
    M.elem_offset = d.elem_offset;
    M.tid = d.tensor_id;
    M.dtype = d.dtype;
    bool vec = d.numel > 0 && (uintptr_t)d.theta0 % 32 == 0 && (uintptr_t)d.out % 32 == 0 && d.elem_offset % 16 == 0;
    for (int e = 0; e < K; ++e) {
      hx[(size_t)k * K + e] = d.numel > 0 ? d.experts[e] : nullptr;
      vec = vec && (uintptr_t)d.experts[e] % 32 == 0;
    }
    M.flags = vec ? TF_VEC : 0u;
    if (cfg->method == SMAT_MERGE_DARE_TA && T < (uint64_t(1) << 32)) {
      M.flags |= TF_MASK;
      M.t_hi = (uint32_t)(T >> 24);
      M.t_lo = (uint32_t)(T & 0xFFFFFFu);
    }
    if (ties && d.numel > 0) {
      int64_t r = (int64_t)std::ceil((double)cfg->retention * (double)d.numel);
      r = r < 1 ? 1 : (r > d.numel ? d.numel : r);
      for (int e = 0; e < K; ++e) hrank[(size_t)k * K + e] = r;
    }
    first[(size_t)k + 1] = first[(size_t)k] + (int32_t)((d.numel + plan.chunk - 1) / plan.chunk);
    if (ties) {
      int32_t* f = first.data() + n_tensors + 1 + k;
      f[1] = f[0] + (int32_t)((d.numel + hist_chunk - 1) / hist_chunk);
    }
  }
  char* ws = static_cast<char*>(d_workspace);
  MArgs m;
  std::memset(&m, 0, sizeof(m));
  m.tensors = reinterpret_cast<const MTensor*>(ws + L.tensors);
  m.chunks = {reinterpret_cast<const int32_t*>(ws + L.first), plan.chunk, plan.n_chunks};
  if (ties) m.hist_chunks = {m.chunks.first + n_tensors + 1, hist_chunk, first.back()};
  m.experts = reinterpret_cast<const void* const*>(ws + L.experts);
  m.thr = reinterpret_cast<uint32_t*>(ws + L.thr);
  m.slots = reinterpret_cast<TiesSlot*>(ws + L.slots);
  m.n_done = reinterpret_cast<uint32_t*>(ws + L.n_done);
  m.rank = reinterpret_cast<int64_t*>(ws + L.rank);
  m.hist = ties ? reinterpret_cast<unsigned long long*>(ws + L.hist) : nullptr;
  m.n_tensors = n_tensors;
  m.key = make_round_keys(cfg->seed);
  m.K = K;
  m.method = cfg->method;
  m.gamma = cfg->gamma;
  const float inv_keep = (float)(1.0 / (double)keep);
  m.c = cfg->method == SMAT_MERGE_WA ? (float)(1.0 / (double)K)
        : cfg->method == SMAT_MERGE_DARE_TA ? cfg->gamma * inv_keep : cfg->gamma;
  const size_t slots = (size_t)n_tensors * (size_t)K;
  cudaError_t e = cudaMemcpyAsync(ws + L.tensors, ht.data(), sizeof(MTensor) * ht.size(), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.first, first.data(), sizeof(int32_t) * first.size(), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.experts, hx.data(), sizeof(void*) * slots, cudaMemcpyHostToDevice, stream);
  if (e != cudaSuccess) return mfail(SMAT_ERR_CUDA, "merge table upload failed");
  const int rounds = cfg->philox_rounds == 7 ? 7 : 10;
  if (ties) {
    e = cudaMemsetAsync(ws + L.n_done, 0, sizeof(uint32_t), stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + L.thr, 0, sizeof(uint32_t) * slots, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + L.hist, 0, sizeof(unsigned long long) * kHistBins * slots, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ws + L.rank, hrank.data(), sizeof(int64_t) * slots, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return mfail(SMAT_ERR_CUDA, "TIES state initialisation failed");
  }
  const int64_t slots64 = (int64_t)slots;
  int64_t largest = 0;
  for (int32_t k = 0; k < n_tensors; ++k) largest = tensors[k].numel > largest ? tensors[k].numel : largest;
  if (plan.dtype == SMAT_BF16)
    e = merge_launch<DT_BF16>(m, slots64, largest, rounds, sms, stream);
  else
    e = merge_launch<DT_F32>(m, slots64, largest, rounds, sms, stream);
  if (e != cudaSuccess) return mfail(SMAT_ERR_CUDA, "merge launch failed");
  return SMAT_OK;
}

extern "C" smat_status smat_merge_ties_thresholds(const smat_merge_tensor* tensors, int32_t n_tensors,
                                                  const smat_merge_config* cfg, const void* d_workspace,
                                                  uint32_t* d_out, smat_stream_t stream) {
  MPlan plan;
  smat_status st = merge_check(tensors, n_tensors, cfg, &plan);
  if (st != SMAT_OK) return st;
  if (cfg->method != SMAT_MERGE_TIES) return mfail(SMAT_ERR_STATE, "not a TIES configuration");
  if (!d_workspace || !d_out) return mfail(SMAT_ERR_INVALID_ARG, "NULL pointer");
  const MLayout L = merge_layout(n_tensors, cfg->n_experts, true);
  const size_t bytes = sizeof(uint32_t) * (size_t)n_tensors * (size_t)cfg->n_experts;
  if (bytes && cudaMemcpyAsync(d_out, static_cast<const char*>(d_workspace) + L.thr, bytes,
                               cudaMemcpyDeviceToDevice, stream) != cudaSuccess)
    return mfail(SMAT_ERR_CUDA, "threshold copy failed");
  return SMAT_OK;
}
