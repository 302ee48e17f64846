#pragma once

// Streaming fast path of the SJD-PAC verify-and-draft step for sm_103a
// (the kernel templates; sjd_fast_part.cu instantiates them).
//
// One CTA per logit row, in one of three layouts (plan() in sjd_api.cu): 128
// threads and about 32 KB of shared memory, so seven CTAs share an SM and every
// row of a 1024-row step is in flight at once; 256 threads, two rows per SM; or
// 512 threads, one row per SM. What bounds a row is the chain of its phases,
// most of them a few round trips and barriers long (a 16-row step of 32768 ids
// takes 27 us, of which its bytes are 0.4), so the phases are few, their
// barriers fewer, and what a phase does not need is not done. Each row is read
// once from HBM, with 128-bit loads two to four rounds ahead of the arithmetic:
//
//  1. guidance in fp32 as the definition has it (fl(c - u), then one fused
//     multiply-add), temperature, the allowed-range mask;
//  2. a shared running maximum (atomicMax on order-preserving keys; a stale
//     value is never above the final maximum m) filters candidates on the
//     fly: ids with l - m_running > -34 go to a dense shared-memory list
//     (continued in the workspace). exp(-34) 2^47 < 0.5, so every other id
//     has weight 0. A sample of the first round also gives a conservative
//     bound of the k-th largest logit that keeps the list short, checked once
//     the row is in (and the row streamed again without it when it excluded
//     too much), and says whether a top-p row needs more than its ids with
//     t = l - m > -22;
//  3. the top-k cut, where there are more than k candidates: counts over the
//     window of values where the sample expects the cut, then an exact ranking
//     in the bin that holds it (an exact select where the window misses);
//  4. the top-p cut, from a head buffer (t > -9) weighed exactly and bounds on
//     the other members' total; from the exact total where the bounds leave it
//     open; by a weighted select where it lies below the head;
//  5. kept ids in id order with their precise weights, verification, residual
//     resampling and the proactive-drafting draws (one warp for up to 32 kept
//     ids, the block otherwise; decisions and fp64 operations by one thread),
//     and the per-batch epilogue shared with the general kernel.
//
// The code of a row runs once, so fetching it is part of its time: loops of a
// few iterations stay rolled (the compiler's unrolling of the kept row's loops
// cost 3 % of a 16-row step of 32768 ids, 37.5 against 36.3 us a pass).
//
// Steps 1-4 read the step's logits alone: with the caller's early-logits
// guarantee they run while the previous step finishes (programmatic
// dependent launch), and only step 5 waits for it.
//
// Results are bit-identical to the general kernel (sjd_kernels.cu), which
// handles the configurations this path does not cover.


#include <cuda_bf16.h>

#include "sjd_device.cuh"

namespace sjd {
namespace {

constexpr int kMaxWarps = 16;           // scratch sized for up to 512 threads per CTA
__device__ __forceinline__ int nthr() { return static_cast<int>(blockDim.x); }
__device__ __forceinline__ int nwarp() { return static_cast<int>(blockDim.x >> 5); }
constexpr int NB = kFastBins;           // select bins
constexpr int CMAX = NB / 2;            // select candidates (16 bytes each) in the histogram space
constexpr int HCAP = 128;               // head buffer
constexpr float kTCut = -34.0f;         // t <= -34 => weight 0
constexpr float kTHead = -9.0f;         // head: t > -9
constexpr float kTShort = -22.0f;       // short list of a top-p row: t > -22
// upper bound of the weight of an id with t <= -22: 2^47 e^-22 (1 + 2e-6) + 1/2 < 39260
constexpr unsigned long long kShortWeight = 39260ull;
constexpr float kTHead2 = -6.0f;        // rebuilt head (too many ids above -9)
constexpr float kBinScale = static_cast<float>(NB) / 34.0f;

// ---------------------------------------------------------------------------
// Per-CTA scratch and block-wide operations (one warp combines the per-warp
// partials; results are broadcast through shared memory).

struct FScratch {
  unsigned long long red[kMaxWarps];
  unsigned long long red2[kMaxWarps];
  // partials of the one-barrier reductions: a call's values stay until the
  // call after the next (alternating halves)
  unsigned long long pa[2][kMaxWarps], pb[2][kMaxWarps];
  uint32_t pc[2][kMaxWarps];
  unsigned long long bc64[8];
  int bi[24];
  uint32_t mkey;          // running maximum (order-preserving key)
  uint32_t list_count;    // candidates appended (may exceed the capacity)
  uint32_t head_count;
  uint32_t cand_count, cand_kmin, cand_kmax;
  uint32_t rnd[5][4];     // Philox blocks of the row: ACCEPT lanes 0-3 / 4-7, RESIDUAL, PD 0-3 / 4-7
  float lbound;           // lower bound estimate of the k-th largest logit (-inf: none)
  float win_lo, win_hi;   // where the k-th largest logit is expected (-inf / +inf: open)
  int short_list;         // top-p row expected to need only the ids with t > -22: they alone are listed
  int interval;           // top-p row expected to have at most k ids with t > -22
  int g, qlen, slot;      // the row's state: group size, stored draft row's length (-1: uniform), ring slot,
  uint32_t pos, t;        // position and step
  int cands[kMaxK];       // draft group of the row
  int gpidx[kMaxK];       // its positions in the kept row (-1: absent)
  float gqc[kMaxK];       // q at the group's tokens
  float2 exp2[65];        // kExp2Table
  int32_t dq_id[32];      // first entries of the stored draft row
  float dq_p[32];
  int alts[kMaxK], altf[kMaxK];  // proactive-drafting draws (warp 0), and the vanilla-SJD tail's
  unsigned long long lvA[kMaxK];  // level k's scale q^(k) -> weight (level_scale), k >= 2 at k - 1
  int lvG[kMaxK];
};
static_assert(sizeof(FScratch) + sizeof(Scratch) <= kFastStaticSmem, "plan() counts with it");

__device__ __forceinline__ int lane() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp() { return threadIdx.x >> 5; }

// Sum over a warp of a u64 per lane: three 32-bit reductions of 24-, 24- and
// 16-bit pieces instead of ten dependent shuffles.
__device__ __forceinline__ unsigned long long wadd64(unsigned long long v) {
  const uint32_t a = __reduce_add_sync(0xFFFFFFFFu, static_cast<uint32_t>(v) & 0xFFFFFFu);
  const uint32_t b = __reduce_add_sync(0xFFFFFFFFu, static_cast<uint32_t>(v >> 24) & 0xFFFFFFu);
  const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, static_cast<uint32_t>(v >> 48));
  return a + (static_cast<unsigned long long>(b) << 24) + (static_cast<unsigned long long>(c) << 48);
}

__device__ unsigned long long fsum(unsigned long long v, FScratch& s) {
  v = wadd64(v);
  if (lane() == 0) s.red[warp()] = v;
  __syncthreads();
  if (warp() == 0) {
    unsigned long long x = lane() < nwarp() ? s.red[lane()] : 0ull;
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    if (lane() == 0) s.bc64[7] = x;
  }
  __syncthreads();
  return s.bc64[7];
}

// Block sums with one barrier; `ph` alternates from call to call (a half is
// written again only two barriers later).
__device__ __forceinline__ void bsum3(uint32_t c, unsigned long long a, unsigned long long b, FScratch& s, int& ph,
                                      uint32_t* rc, unsigned long long* ra, unsigned long long* rb) {
  c = __reduce_add_sync(0xFFFFFFFFu, c);
  a = wadd64(a);
  b = wadd64(b);
  ph ^= 1;
  if (lane() == 0) {
    s.pc[ph][warp()] = c;
    s.pa[ph][warp()] = a;
    s.pb[ph][warp()] = b;
  }
  __syncthreads();
  uint32_t x = 0;
  unsigned long long y = 0, z = 0;
#pragma unroll 4
  for (int w = 0; w < nwarp(); ++w) {
    x += s.pc[ph][w];
    y += s.pa[ph][w];
    z += s.pb[ph][w];
  }
  *rc = x;
  *ra = y;
  *rb = z;
}

// Length of each thread's contiguous run over n positions: odd, so that a
// warp's reads of 8-byte elements a run apart fall into different banks (runs
// of 16 put all lanes on one bank: 12 us for the prefix of 4096 weights by 256
// threads).
__device__ __forceinline__ int run_of(int n, int threads) { return ((n + threads - 1) / threads) | 1; }

// Exclusive scan of one u64 per thread in thread order and the sum, with one
// barrier.
struct Scan {
  unsigned long long ex, total;
};
__device__ Scan bscan(unsigned long long v, FScratch& s, int ph) {
  unsigned long long incl = v;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane() >= o) incl += y;
  }
  if (lane() == 31) s.pa[ph][warp()] = incl;
  __syncthreads();
  unsigned long long base = 0, tot = 0;
#pragma unroll 4
  for (int w = 0; w < nwarp(); ++w) {
    const unsigned long long x = s.pa[ph][w];
    if (w < warp()) base += x;
    tot += x;
  }
  return Scan{base + incl - v, tot};
}

// First position i in [0, n) with pcum[i] > T (T below pcum[n - 1]), by one
// warp: each step tests 32 evenly spaced positions at once (three steps up to
// 32768).
__device__ __forceinline__ int warp_search(const unsigned long long* pcum, int n, unsigned long long T) {
  int lo = 0, len = n;
#pragma unroll 1
  for (;;) {
    const int step = (len + 31) >> 5;
    const int i = lo + min((lane() + 1) * step, len) - 1;
    const uint32_t hit = __ballot_sync(0xFFFFFFFFu, pcum[i] > T);
    const int f = hit ? __ffs(hit) - 1 : (len - 1) / step;
    lo += f * step;
    len = min(step, len - f * step);
    if (step == 1) return lo;
  }
}

// Exclusive scan of one u64 per thread in thread order; *total = the sum.
__device__ unsigned long long fexscan(unsigned long long v, FScratch& s, unsigned long long* total) {
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane() >= o) incl += y;
  }
  if (lane() == 31) s.red[warp()] = incl;
  __syncthreads();
  if (warp() == 0) {
    const int nw = nwarp();
    const unsigned long long w = lane() < nw ? s.red[lane()] : 0ull;
    unsigned long long x = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane() >= o) x += y;
    }
    if (lane() < nw) s.red2[lane()] = x - w;
    if (lane() == nw - 1) s.bc64[4] = x;
  }
  __syncthreads();
  *total = s.bc64[4];
  return s.red2[warp()] + incl - v;
}

// ---------------------------------------------------------------------------
// Shared-memory views and the kept-row arrays.

struct KeptArrays {           // kept row (capacity S) and its verification arrays
  uint16_t* pidx;             // local index (id - al0), ascending
  unsigned long long* pcum;   // inclusive prefix of the weights
  float* qP;                  // q at the kept ids
  unsigned long long* Rw;     // residual weights of the group levels
};

struct FSmem {
  uint2* list;                // candidates: {logit bits, local index}; the general kept pass
                              // replaces an entry by its precise weight and index
  unsigned long long* hist;   // histogram / select candidates / word prefix counts
  unsigned long long* head;   // head buffer: HCAP x {key, idx, E} (16 bytes)
  uint32_t* bitmap;           // one bit per local index
  KeptArrays small;           // kept arrays in shared memory (capacity f_kcap)
};

__device__ __forceinline__ FSmem fsmem_views(const DevParams& P, unsigned char* base) {
  FSmem s;
  s.list = reinterpret_cast<uint2*>(base + P.f_list_l);
  s.hist = reinterpret_cast<unsigned long long*>(base + P.f_hist);
  s.head = reinterpret_cast<unsigned long long*>(base + P.f_list_w);
  s.bitmap = reinterpret_cast<uint32_t*>(base + P.f_bitmap);
  s.small.pidx = reinterpret_cast<uint16_t*>(base + P.f_pidx);
  s.small.pcum = reinterpret_cast<unsigned long long*>(base + P.f_pcum);
  s.small.qP = reinterpret_cast<float*>(base + P.f_qP);
  s.small.Rw = reinterpret_cast<unsigned long long*>(base + P.f_Rw);
  return s;
}

// Kept arrays of row `row` in the workspace (for kept rows above f_kcap).
__device__ __forceinline__ KeptArrays global_kept(const DevParams& P, int row) {
  unsigned char* base = reinterpret_cast<unsigned char*>(P.f_scratch) + static_cast<size_t>(row) * P.f_row_bytes;
  const size_t S = static_cast<size_t>(P.S);
  KeptArrays k;
  k.pcum = reinterpret_cast<unsigned long long*>(base);
  k.Rw = reinterpret_cast<unsigned long long*>(base + 8 * S);
  k.qP = reinterpret_cast<float*>(base + 16 * S);
  k.pidx = reinterpret_cast<uint16_t*>(base + 20 * S);
  return k;
}

struct FCand {
  uint32_t key;
  int idx;
  unsigned long long w;
};

// First-level bin over t in (-34, 0]: linear in -t, monotone in l.
__device__ __forceinline__ int fbin0(float t) {
  const float x = __fmul_rn(-t, kBinScale);
  return (x < static_cast<float>(NB - 1)) ? static_cast<int>(x) : NB - 1;
}

// Weight of a member: E = rint(2^47 exp(t)) (the exponential of the shared
// exp_neg definition) and E 2^-47 as fp32, without conversion instructions.
// rint(a) for |a| <= 64 is fl(a + 1.5 2^23) - 1.5 2^23 (the sum lies in a
// binade of spacing 1, so the addition rounds to an integer, ties to even),
// and its integer value is the difference of the bit patterns. For
// y >= 2^-24, y 2^47 is an integer and E is y's significand shifted; below,
// fl(y + 2^-24) rounds y to the grid 2^-47 (ties to even on the significand,
// whose last bit is E's), E is the difference of the bit patterns and
// E 2^-47 = fl(y + 2^-24) - 2^-24 exactly (Sterbenz). Both identities hold
// for every input float (checked exhaustively against rintf and against the
// integer rounding of quant()).
__device__ __forceinline__ float exp_weight(float t, unsigned long long* E) {
  const float a = __fmul_rn(t, 0x1.715476p+0f);  // fl32(log2 e)
  if (!(a >= -64.0f)) {
    *E = 0ull;
    return 0.0f;
  }
  const float r = __fadd_rn(a, 0x1.8p23f);
  const float n = __fsub_rn(r, 0x1.8p23f);
  const int ni = static_cast<int>(__float_as_uint(r) - __float_as_uint(0x1.8p23f));
  const float f = __fsub_rn(a, n);
  float y = 0x1.ffcbfcp-17f;
  y = __fmaf_rn(y, f, 0x1.430912p-13f);
  y = __fmaf_rn(y, f, 0x1.5d87fep-10f);
  y = __fmaf_rn(y, f, 0x1.3b2ab6p-7f);
  y = __fmaf_rn(y, f, 0x1.c6b08ep-5f);
  y = __fmaf_rn(y, f, 0x1.ebfbe0p-3f);
  y = __fmaf_rn(y, f, 0x1.62e430p-1f);
  y = __fmaf_rn(y, f, 1.0f);
  y = __fmul_rn(y, __int_as_float((ni + 127) << 23));
  const uint32_t b = __float_as_uint(y);
  if (y >= 0x1p-24f) {
    *E = static_cast<unsigned long long>((b & 0x7FFFFFu) | 0x800000u) << ((b >> 23) - 103u);
    return y;
  }
  const float sg = __fadd_rn(y, 0x1p-24f);
  *E = static_cast<unsigned long long>(__float_as_uint(sg) - __float_as_uint(0x1p-24f));
  return __fsub_rn(sg, 0x1p-24f);
}

// Index of the need-th set bit (1-based) of the bitmap (nwords words).
__device__ int nth_set_bit(const uint32_t* bitmap, int nwords, unsigned long long need, FScratch& s) {
  const int per = (nwords + nthr() - 1) / nthr();
  const int w0 = min(nwords, static_cast<int>(threadIdx.x) * per), w1 = min(nwords, w0 + per);
  unsigned long long c = 0;
  for (int w = w0; w < w1; ++w) c += __popc(bitmap[w]);
  if (threadIdx.x == 0) s.bi[5] = INT_MAX;
  unsigned long long total;
  unsigned long long run = fexscan(c, s, &total);
  if (run < need && need <= run + c) {
    for (int w = w0; w < w1; ++w) {
      const uint32_t word = bitmap[w];
      const unsigned long long pc = __popc(word);
      if (run + pc >= need) {
        s.bi[5] = w * 32 + __fns(word, 0, static_cast<int>(need - run));
        break;
      }
      run += pc;
    }
  }
  __syncthreads();
  const int r = s.bi[5];
  __syncthreads();
  return r;
}

// Select the cut at which the running count (or weight) of the active
// elements, in the order (key desc, local index asc), first reaches `need`.
// src.each(f) calls f(key, idx, t, w) for this thread's active elements.
template <bool WEIGHTED, class Src>
__device__ Cut fast_select(const Src src, float m, unsigned long long need_in, const FSmem sm, int nwords,
                           FScratch& s) {
  uint32_t* h32 = reinterpret_cast<uint32_t*>(sm.hist);
  unsigned long long* h64 = sm.hist;
  FCand* cands = reinterpret_cast<FCand*>(sm.hist);
  unsigned long long need = need_in;
  uint32_t klo = 0, khi = 0xFFFFFFFFu;
  for (int level = 0; level < 8; ++level) {
    const int sh = level == 0 ? 0 : max(0, 32 - __clz(khi - klo) - 8);
    for (int k = threadIdx.x; k < NB; k += nthr()) {
      if (WEIGHTED) h64[k] = 0; else h32[k] = 0;
    }
    __syncthreads();
    src.each([&](uint32_t key, int idx, float t, unsigned long long w) {
      if (key < klo || key > khi) return;
      const int bk = level == 0 ? fbin0(t) : static_cast<int>((khi - key) >> sh);
      if (WEIGHTED) {
        if (w) atomicAdd(&h64[bk], w);
      } else {
        atomicAdd(&h32[bk], 1u);
      }
    });
    __syncthreads();
    // thread t owns bins [t kPer, t kPer + kPer) (kPer = 2 for 128 threads, 1 for more)
    const int kPer = nthr() >= NB ? 1 : NB / nthr();
    unsigned long long loc[2];
    unsigned long long lsum = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = threadIdx.x * kPer + q;
      loc[q] = (q < kPer && k < NB) ? (WEIGHTED ? h64[k] : h32[k]) : 0ull;
      lsum += loc[q];
    }
    if (threadIdx.x == 0) {
      s.bi[1] = -1;
      s.bc64[0] = 0;
    }
    unsigned long long tot;
    const unsigned long long ex = fexscan(lsum, s, &tot);
    if (ex < need && need <= ex + lsum) {
      unsigned long long run = ex;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q < kPer && run < need && need <= run + loc[q]) {
          s.bi[1] = threadIdx.x * kPer + q;
          s.bc64[0] = run;
        }
        run += loc[q];
      }
    }
    if (threadIdx.x == 0) {
      s.cand_count = 0;
      s.cand_kmin = 0xFFFFFFFFu;
      s.cand_kmax = 0;
    }
    __syncthreads();
    const int bstar = s.bi[1];
    need -= s.bc64[0];
    uint32_t kmn = 0xFFFFFFFFu, kmx = 0;
    src.each([&](uint32_t key, int idx, float t, unsigned long long w) {
      if (key < klo || key > khi) return;
      const int bk = level == 0 ? fbin0(t) : static_cast<int>((khi - key) >> sh);
      if (bk != bstar) return;
      kmn = min(kmn, key);
      kmx = max(kmx, key);
      const uint32_t slot = atomicAdd(&s.cand_count, 1u);
      if (slot < static_cast<uint32_t>(CMAX)) {
        cands[slot].key = key;
        cands[slot].idx = idx;
        cands[slot].w = w;
      }
    });
    kmn = __reduce_min_sync(0xFFFFFFFFu, kmn);
    kmx = __reduce_max_sync(0xFFFFFFFFu, kmx);
    if (lane() == 0) {
      atomicMin(&s.cand_kmin, kmn);
      atomicMax(&s.cand_kmax, kmx);
    }
    __syncthreads();
    const uint32_t nc = s.cand_count;
    const uint32_t bkmin = s.cand_kmin, bkmax = s.cand_kmax;
    if (nc <= static_cast<uint32_t>(CMAX)) {
      for (uint32_t c = threadIdx.x; c < nc; c += nthr()) {
        const FCand me = cands[c];
        uint32_t rank = 0;
        unsigned long long wsum = 0;
        for (uint32_t d = 0; d < nc; ++d) {
          const FCand o = cands[d];
          const bool better = o.key > me.key || (o.key == me.key && o.idx < me.idx);
          rank += better ? 1u : 0u;
          wsum += better ? o.w : 0ull;
        }
        bool pick;
        if (WEIGHTED) pick = wsum < need && need <= wsum + me.w;
        else pick = static_cast<unsigned long long>(rank) + 1 == need;
        if (pick) {
          s.bi[2] = static_cast<int>(me.key);
          s.bi[3] = me.idx;
        }
      }
      __syncthreads();
      const Cut c{static_cast<uint32_t>(s.bi[2]), s.bi[3]};
      __syncthreads();
      return c;
    }
    __syncthreads();
    klo = bkmin;
    khi = bkmax;
    if (klo == khi) {
      // every remaining element has the same value: the order is by index
      unsigned long long nth = need;
      if (WEIGHTED) {
        const unsigned long long wt = quant(exp_neg(__fsub_rn(key2f(klo), m)));
        nth = (need + wt - 1) / wt;
      }
      src.each([&](uint32_t key, int idx, float t, unsigned long long w) {
        if (key == klo) atomicOr(&sm.bitmap[idx >> 5], 1u << (idx & 31));
      });
      __syncthreads();
      const Cut c{klo, nth_set_bit(sm.bitmap, nwords, nth, s)};
      for (int k = threadIdx.x; k < nwords; k += nthr()) sm.bitmap[k] = 0u;  // (empty again for the kept ids)
      __syncthreads();
      return c;
    }
  }
  return Cut{khi, INT_MAX};
}

// ---------------------------------------------------------------------------
// Streaming loads.

template <int DT>
struct Chunk {  // one 16-byte chunk of cond and of uncond
  uint4 c, u;
};

// One 4-byte word to shared memory without waiting for it.
__device__ __forceinline__ void copy_word(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

// The row in memory: chunk c holds the ids al0 + c EPC .. at the 16-byte
// boundary cr + c. Rows that do not start on such a boundary have a grid of
// their own, from the boundary at or below their first allowed id (cond and
// uncond lie alike there), and only the allowed elements of their first and
// last chunk are read.
struct RowMem {
  const uint4* cr;
  const uint4* ur;
  int al0, nL;   // first id, ids up to the last chunk's end
  bool ragged;
};

// Elements [e0, e1) of the chunk at p (zeros elsewhere), read one by one.
template <int DT>
__device__ __noinline__ uint4 edge_chunk(const uint4* p, int e0, int e1) {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
  if (DT == SJD_BF16) {
    const unsigned short* h = reinterpret_cast<const unsigned short*>(p);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (e >= e0 && e < e1) w[e >> 1] |= static_cast<uint32_t>(__ldcs(h + e)) << (16 * (e & 1));
  } else {
    const unsigned int* f = reinterpret_cast<const unsigned int*>(p);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e >= e0 && e < e1) w[e] = __ldcs(f + e);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

template <int DT, bool CFG>
__device__ __forceinline__ Chunk<DT> load_chunk(const DevParams& P, const RowMem& R, int c) {
  constexpr int EPC = DT == SJD_BF16 ? 8 : 4;
  Chunk<DT> k;
  k.c = make_uint4(0u, 0u, 0u, 0u);
  k.u = make_uint4(0u, 0u, 0u, 0u);
  const int v0 = R.al0 + c * EPC;
  if (v0 < P.hi) {
    if (R.ragged && (v0 < P.lo || v0 + EPC > P.hi)) {
      const int e0 = max(P.lo - v0, 0), e1 = min(P.hi - v0, EPC);
      k.c = edge_chunk<DT>(R.cr + c, e0, e1);
      if (CFG) k.u = edge_chunk<DT>(R.ur + c, e0, e1);
    } else {
      k.c = __ldcs(R.cr + c);
      if (CFG) k.u = __ldcs(R.ur + c);
    }
  }
  return k;
}

// NaN-propagating maximum of three values.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Guidance of two values at once: fl(c - u), then one fused multiply-add
// s (c - u) + u, element by element as the definition has it.
__device__ __forceinline__ void guide2(float c0, float c1, float u0, float u1, float s, float& x0, float& x1) {
  asm("{\n\t.reg .b64 c2, u2, s2;\n\t"
      "mov.b64 c2, {%2, %3};\n\t"
      "mov.b64 u2, {%4, %5};\n\t"
      "mov.b64 s2, {%6, %6};\n\t"
      "sub.rn.f32x2 c2, c2, u2;\n\t"
      "fma.rn.f32x2 c2, s2, c2, u2;\n\t"
      "mov.b64 {%0, %1}, c2;\n\t}"
      : "=f"(x0), "=f"(x1)
      : "f"(c0), "f"(c1), "f"(u0), "f"(u1), "f"(s));
}

// Logits of one chunk (EPC values; ids outside the allowed range, and chunks
// past the row, get the padding value) and their NaN-propagating maximum
// (-inf if none).
template <int DT, bool CFG>
__device__ __forceinline__ void chunk_logits(const DevParams& P, int al0, const Chunk<DT>& k, int c, float* out,
                                             float* cmax) {
  constexpr int EPC = DT == SJD_BF16 ? 8 : 4;
  float cv[EPC], uv[EPC];
  if (DT == SJD_BF16) {
    const uint32_t cw[4] = {k.c.x, k.c.y, k.c.z, k.c.w};
    const uint32_t uw[4] = {k.u.x, k.u.y, k.u.z, k.u.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cv[2 * q] = __uint_as_float(cw[q] << 16);
      cv[2 * q + 1] = __uint_as_float(cw[q] & 0xFFFF0000u);
      uv[2 * q] = __uint_as_float(uw[q] << 16);
      uv[2 * q + 1] = __uint_as_float(uw[q] & 0xFFFF0000u);
    }
  } else {
    cv[0] = __uint_as_float(k.c.x); cv[1] = __uint_as_float(k.c.y);
    cv[2] = __uint_as_float(k.c.z); cv[3] = __uint_as_float(k.c.w);
    uv[0] = __uint_as_float(k.u.x); uv[1] = __uint_as_float(k.u.y);
    uv[2] = __uint_as_float(k.u.z); uv[3] = __uint_as_float(k.u.w);
  }
#pragma unroll
  for (int q = 0; q < EPC; q += 2) {
    if (CFG) {
      guide2(cv[q], cv[q + 1], uv[q], uv[q + 1], P.cfg, out[q], out[q + 1]);
    } else {
      out[q] = cv[q];
      out[q + 1] = cv[q + 1];
    }
  }
  if (P.temp != 1.0f) {
#pragma unroll
    for (int q = 0; q < EPC; ++q) out[q] = __fdiv_rn(out[q], P.temp);
  }
  const int v0 = al0 + c * EPC;
  if (v0 >= P.lo && v0 + EPC <= P.hi) {
    float x = max3_nan(out[0], out[1], out[2]);
#pragma unroll
    for (int q = 3; q + 1 < EPC; q += 2) x = max3_nan(x, out[q], out[q + 1]);
    *cmax = max_nan(x, out[EPC - 1]);
  } else {
    float x = -INFINITY;
#pragma unroll
    for (int q = 0; q < EPC; ++q) {
      const bool ok = v0 + q >= P.lo && v0 + q < P.hi;
      x = ok ? max_nan(x, out[q]) : x;
      out[q] = ok ? out[q] : pad_value();
    }
    *cmax = x;
  }
}

// ---------------------------------------------------------------------------
// Element sources for the selects.

// Candidates (t > -34) of the whole row, read again (128-bit loads, mostly
// from L2) with the final maximum.
template <int DT, bool CFG>
struct GlobalRow {
  const DevParams* P;
  const RowMem* R;
  float m;
  template <class F>
  __device__ __forceinline__ void each(F f) const {
    constexpr int EPC = DT == SJD_BF16 ? 8 : 4;
    const int nch = R->nL / EPC;
    for (int c = threadIdx.x; c < nch; c += nthr()) {
      float lv[EPC], cm;
      chunk_logits<DT, CFG>(*P, R->al0, load_chunk<DT, CFG>(*P, *R, c), c, lv, &cm);
#pragma unroll
      for (int q = 0; q < EPC; ++q) {
        const float t = __fsub_rn(lv[q], m);
        if (t > kTCut) f(f2key(lv[q]), c * EPC + q, t, 0ull);
      }
    }
  }
};

// The candidate list: entries [0, lcap) in shared memory (logit, local
// index), the rest in the row's workspace scratch (8 bytes each; written and
// read by this CTA only, ordered by its barriers).
struct ListView {
  uint2* sh;
  uint2* g;
  int lcap;
  bool early;  // the grid may still overlap the previous one: wait before writing g
  static __device__ __forceinline__ uint2 entry(float l, int idx) {
    return make_uint2(__float_as_uint(l), static_cast<uint32_t>(idx));
  }
  __device__ __forceinline__ uint2& at(int i) const { return i < lcap ? sh[i] : g[i - lcap]; }
  __device__ __forceinline__ void put(int i, float l, int idx) const {
    // the previous step's CTA of this row may still read this scratch
    if (i >= lcap && early) griddep_wait();
    at(i) = entry(l, idx);
  }
  // the kept pass replaces an entry by (precise weight << 16) | local index
  static __device__ __forceinline__ uint2 weight_entry(unsigned long long E, int idx) {
    return make_uint2(static_cast<uint32_t>(E << 16) | static_cast<uint32_t>(idx), static_cast<uint32_t>(E >> 16));
  }
  static __device__ __forceinline__ unsigned long long weight_of(uint2 e) {
    return (static_cast<unsigned long long>(e.y) << 16) | (e.x >> 16);
  }
  static __device__ __forceinline__ int index_of(uint2 e) { return static_cast<int>(e.x & 0xFFFFu); }
  // f(entry) for this thread's entries: one loop over the shared part, one
  // over the rest (rolled: for a body of some length, run over a few entries)
  template <class F>
  __device__ __forceinline__ void each(int n, F f) const {
    const int ns = min(n, lcap);
    for (int i = threadIdx.x; i < ns; i += nthr()) f(sh[i]);
    for (int i = lcap + static_cast<int>(threadIdx.x); i < n; i += nthr()) f(g[i - lcap]);
  }
  template <class F>
  __device__ __forceinline__ void each_rolled(int n, F f) const {
    const int ns = min(n, lcap);
#pragma unroll 1
    for (int i = threadIdx.x; i < ns; i += nthr()) f(sh[i]);
#pragma unroll 1
    for (int i = lcap + static_cast<int>(threadIdx.x); i < n; i += nthr()) f(g[i - lcap]);
  }
};

// Hits of the streaming filter, without branches (a branch per value costs
// more than the filter): counts a hit; stores one at `at` (a shared-memory
// address) and moves on.
__device__ __forceinline__ void count_hit(float l, float thr, uint32_t& n) {
  asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %1, %2;\n\t@p add.u32 %0, %0, 1;\n\t}" : "+r"(n) : "f"(l), "f"(thr));
}
__device__ __forceinline__ void store_hit(float l, float thr, uint32_t idx, uint32_t& at) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %1, %2;\n\t@p st.shared.v2.b32 [%0], {%3, %4};\n\t@p add.u32 %0, %0, 8;\n\t}"
      : "+r"(at)
      : "f"(l), "f"(thr), "r"(__float_as_uint(l)), "r"(idx)
      : "memory");
}

// The raw inputs of the id at local index idx of the row, read again (mostly
// from L2) for its precise weight (sjd_device.cuh).
template <int DT, bool CFG>
__device__ __forceinline__ void raw_logits(const RowMem& R, int idx, float& c, float& u) {
  const uint4 *cr = R.cr, *ur = R.ur;
  u = 0.0f;
  if (DT == SJD_BF16) {
    c = bf16_bits_to_f32(__ldg(reinterpret_cast<const unsigned short*>(cr) + idx));
    if (CFG) u = bf16_bits_to_f32(__ldg(reinterpret_cast<const unsigned short*>(ur) + idx));
  } else {
    c = __ldg(reinterpret_cast<const float*>(cr) + idx);
    if (CFG) u = __ldg(reinterpret_cast<const float*>(ur) + idx);
  }
}
// Every list entry (the list of a stream pass that overflowed).
struct ListAll {
  ListView L;
  int n;
  float m;
  template <class F>
  __device__ __forceinline__ void each(F f) const {
    L.each(n, [&](uint2 e) {
      const float lv = __uint_as_float(e.x);
      f(f2key(lv), static_cast<int>(e.y), __fsub_rn(lv, m), 0ull);
    });
  }
};

// Candidate list (entries with t > -34 under the final maximum).
struct ListCand {
  ListView L;
  int n;
  float m;
  template <class F>
  __device__ __forceinline__ void each(F f) const {
    L.each(n, [&](uint2 e) {
      const float lv = __uint_as_float(e.x);
      const float t = __fsub_rn(lv, m);
      if (t > kTCut) f(f2key(lv), static_cast<int>(e.y), t, 0ull);
    });
  }
};

// Members of the candidate list (t > -34, inside the top-k cut) with their
// weights recomputed.
struct ListMembers {
  ListView L;
  int n;
  float m;
  Cut kcut;
  template <class F>
  __device__ __forceinline__ void each(F f) const {
    L.each(n, [&](uint2 en) {
      const float lv = __uint_as_float(en.x);
      const int id = static_cast<int>(en.y);
      const float t = __fsub_rn(lv, m);
      if (!(t > kTCut)) return;
      const uint32_t key = f2key(lv);
      if (!in_cut(key, id, kcut)) return;
      unsigned long long E;
      exp_weight(t, &E);
      f(key, id, t, E);
    });
  }
};

// What a sample of the row says of it (warp 0): h[NB] counts its values with t
// > -34 below the sample's maximum mth. Sets s.short_list, s.interval,
// s.lbound, s.win_lo and s.win_hi. Everyone waits for it, so what does not
// depend on the row (the ranks) comes with the parameters.
__device__ __forceinline__ void sample_bounds(const DevParams& P, const uint32_t* h, float mth, FScratch& s) {
  constexpr int PER = NB / 32;
  constexpr float kWidth = 34.0f / NB;
  uint32_t c = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) c += h[lane() * PER + q];
  uint32_t ci = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, ci, o);
    if (lane() >= o) ci += y;
  }
  const uint32_t total = __shfl_sync(0xFFFFFFFFu, ci, 31);  // candidates in the sample
  // ranks in the sample where the cut is expected, with a quarter and 16 to both sides
  const uint32_t kp = P.f_kp;
  const uint32_t ks = kp + kp / 4 + 16;
  const uint32_t kh = kp > kp / 4 + 16 ? kp - kp / 4 - 16 : 0u;
  uint32_t ce = ci - c;
  bool shortl = false;
  // A top-p row's cut is first sought among the ids with t > -22 when the
  // sample has fewer than k's share of them, and only they are listed when it
  // has 15 % and two standard deviations less. Counted under the row's maximum
  // as far as the sample tells it: its own, or, where higher, as far above its
  // top 1/128 as that is above its top 1/16, less 2.5 units.
  if (P.top_p < 1.0f) {
    int b1 = -1, b2 = -1;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const uint32_t nq = h[lane() * PER + q];
      if (ce < P.f_ns / 128u && P.f_ns / 128u <= ce + nq) b1 = lane() * PER + q;
      if (ce < P.f_ns / 16u && P.f_ns / 16u <= ce + nq) b2 = lane() * PER + q;
      ce += nq;
    }
    b1 = __reduce_max_sync(0xFFFFFFFFu, b1);
    b2 = __reduce_max_sync(0xFFFFFFFFu, b2);
    const int tb = static_cast<int>(24.5f * kBinScale) + (b2 >= 0 ? min(0, 2 * b1 - b2) : 0);
    uint32_t near = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) near += lane() * PER + q < tb ? h[lane() * PER + q] : 0u;
    near = __reduce_add_sync(0xFFFFFFFFu, near);
    const int spare = static_cast<int>(kp - kp / 7u) - static_cast<int>(near) - 2;
    shortl = spare >= 0 && static_cast<uint32_t>(spare) * static_cast<uint32_t>(spare) >= 4u * near;
    if (lane() == 0) {
      s.short_list = shortl ? 1 : 0;
      s.interval = near < kp ? 1 : 0;
    }
    ce = ci - c;
  }
  // Only rows whose sample projects more than 1.5 k candidates need the bound.
  const bool want = !shortl && total > P.f_want;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const uint32_t nq = h[lane() * PER + q];
    const float edge = -static_cast<float>(lane() * PER + q) * kWidth;
    if (ce < ks && ks <= ce + nq) {
      const float e = __fadd_rn(mth, edge - kWidth);
      s.win_lo = e;
      if (want) s.lbound = e;
    }
    if (ce < kh && kh <= ce + nq) s.win_hi = __fadd_rn(mth, edge);
    ce += nq;
  }
}

// The top-k cut of a row from its list (every candidate, or every value above
// a bound of the k-th largest; more than k entries): counts over NB bins of the
// window [wlo, whi] where the sample expects the k-th largest, then an exact
// ranking inside the bin that holds it (a window of a quarter of k to both
// sides gives about k / 512 entries per bin). Listed values with t <= -34 take
// part harmlessly: a cut among them keeps every candidate. The general select
// is the way out when the window misses the cut or a bin is crowded (ties), and
// from |m| = 4e6 on, where fp32 can no longer name a value between the
// candidates and m - 34.5 (at 1e8 that rounds to m - 32, a candidate).
// Bound by barriers and shared-memory latency. The cut used to be taken from
// counts of the weights, or 128 bins over the whole range, after a pass over
// all weights; flat rows overflowed the bins and took two more passes (cut
// phase of 8x32x16384 rows with k = 4096: 0.8 us median, 15 us in a tenth of the rows).
__device__ Cut topk_cut(const ListView L, int n, float m, int topk, float wlo, float whi, const FSmem sm,
                        int nwords, FScratch& s) {
  uint32_t* h32 = reinterpret_cast<uint32_t*>(sm.hist);
  const float floor_l = __fadd_rn(m, kTCut - 0.5f);  // below every candidate (|m| < 4e6)
  const bool lo_open = !(wlo > floor_l);
  const float lo = lo_open ? floor_l : wlo;
  const float hi = fminf(whi, m);
  const float scale = __fdiv_rn(static_cast<float>(NB), __fsub_rn(hi, lo));
  if (hi > lo && scale < 1e30f && fabsf(m) < 4.0e6f) {
    for (int k = threadIdx.x; k < NB; k += nthr()) h32[k] = 0u;
    if (threadIdx.x == 0) {
      s.bi[1] = -1;
      s.bi[4] = 0;
      s.cand_count = 0u;
    }
    __syncthreads();
    // bin of a value at most hi: non-increasing in l; NB and above: below the window
    auto bin = [&](float l) { return static_cast<int>(fminf(__fmul_rn(__fsub_rn(hi, l), scale), 2.0f * NB)); };
    int above = 0;
    L.each(n, [&](uint2 e) {
      const float l = __uint_as_float(e.x);
      if (l > hi) {
        ++above;
      } else {
        const int b = bin(l);
        if (b < NB) atomicAdd(&h32[b], 1u);
      }
    });
    above = __reduce_add_sync(0xFFFFFFFFu, above);
    if (lane() == 0 && above) atomicAdd(&s.bi[4], above);
    __syncthreads();
    if (warp() == 0) {
      constexpr int PER = NB / 32;
      uint32_t c[PER], sum = 0;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        c[q] = h32[lane() * PER + q];
        sum += c[q];
      }
      uint32_t ci = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, ci, o);
        if (lane() >= o) ci += y;
      }
      const uint32_t total = __shfl_sync(0xFFFFFFFFu, ci, 31);
      const int need = topk - s.bi[4];  // rank of the cut inside the window (1-based)
      if (lane() == 0 && need > static_cast<int>(total) && lo_open) s.bi[1] = -2;  // fewer than k candidates
      uint32_t ce = ci - sum;
      if (need > 0) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          if (ce < static_cast<uint32_t>(need) && static_cast<uint32_t>(need) <= ce + c[q]) {
            s.bi[1] = c[q] <= static_cast<uint32_t>(CMAX) ? lane() * PER + q : -1;
            s.bi[2] = need - static_cast<int>(ce);
          }
          ce += c[q];
        }
      }
    }
    __syncthreads();
    const int bstar = s.bi[1];
    if (bstar == -2) return no_cut();
    if (bstar >= 0) {
      const uint32_t need = static_cast<uint32_t>(s.bi[2]);
      // keys over the dead histogram: every thread is past the barrier that ended its reading
      unsigned long long* ck = sm.hist;  // (key << 32) | ~index: larger is earlier in the order
      L.each(n, [&](uint2 e) {
        const float l = __uint_as_float(e.x);
        if (!(l > hi) && bin(l) == bstar) {
          const uint32_t at = atomicAdd(&s.cand_count, 1u);
          ck[at] = (static_cast<unsigned long long>(f2key(l)) << 32) | ~e.y;
        }
      });
      __syncthreads();
      const uint32_t nc = s.cand_count;
      if (threadIdx.x < nc) {
        const unsigned long long me = ck[threadIdx.x];
        uint32_t rank = 1;
#pragma unroll 4
        for (uint32_t d = 0; d < nc; ++d) rank += ck[d] > me ? 1u : 0u;
        if (rank == need) s.bc64[2] = me;
      }
      __syncthreads();
      const unsigned long long me = s.bc64[2];
      return Cut{static_cast<uint32_t>(me >> 32), static_cast<int>(~static_cast<uint32_t>(me))};
    }
  }
  // the exact select, when there are more than k candidates
  const ListCand lc{L, n, m};
  uint32_t c = 0;
  lc.each([&](uint32_t, int, float, unsigned long long) { ++c; });
  if (fsum(c, s) <= static_cast<unsigned long long>(topk)) return no_cut();
  return fast_select<false>(lc, m, static_cast<unsigned long long>(topk), sm, nwords, s);
}

// ---------------------------------------------------------------------------
// The row kernel.

// RAG: rows may start off 16-byte boundaries. (Seven CTAs of 128 threads an SM
// leave 72 registers a thread, so that layout has a kernel of its own for rows
// that do not, whose chunk grid is a constant: 42.2 us a pass at 16x64x65536
// with top-p, 42.7 without it, and 217 against 221 for eight chained steps.)
template <int DT, int MODE, bool CFG, int NT, bool RAG>
__global__ void __launch_bounds__(NT, NT == 128 ? 7 : NT == 256 ? 2 : 1)
stream_row_kernel(const __grid_constant__ DevParams P, const void* __restrict__ cond, const void* __restrict__ uncond,
                  int32_t* out_committed, int32_t* out_ncommit, int32_t* out_firstrej) {
  constexpr int ST = NT;         // threads per CTA: 128 (7 CTAs per SM), 256 (2 or more) or 512 (one)
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ FScratch s;
  __shared__ Scratch esc;  // for the per-batch epilogue shared with the general kernel
  // Programmatic dependent launch: this grid may start while the previous
  // kernel of the stream drains, and the next launch may start as soon as
  // every CTA of this grid has begun. Everything below may depend on the
  // previous kernel (the window state of the previous step, or logits a
  // forward has just written), so the wait comes before the first global
  // read; when the caller guarantees that the logits were written before
  // that kernel started (P.early_logits), S1-S4 (which read the logits
  // alone) run at once, and the wait comes before the first read or write
  // of the decode state or of the row's workspace scratch. Whether a tree node
  // exists is decode state, so its row waits in either case.
  if (P.early_logits == 0) griddep_wait();
  griddep_launch_dependents();
  const FSmem sm = fsmem_views(P, smem_raw);
  constexpr int EPC = DT == SJD_BF16 ? 8 : 4;
  // row: logit row; window row j of batch element b, or (tree) a node row,
  // whose children sit at window row j, with that row's draft row and uniforms
  constexpr bool TREE = MODE == kModeTree;
  const int row = blockIdx.x;
  const int b = row / (TREE ? P.rows_b : P.W);
  const int jr = row - b * (TREE ? P.rows_b : P.W);
  const bool node_row = TREE && jr >= P.W;
  int nd = 0, ni = 0;  // node ni >= 1 at depth nd
  if (node_row) {
    int e = jr - P.W, kd = P.K;
    nd = 1;
#pragma unroll 1
    while (e >= kd - 1) {
      e -= kd - 1;
      kd *= P.K;
      ++nd;
    }
    ni = e + 1;
  }
  const int j = node_row ? nd : jr;
  const bool early = P.early_logits != 0 && !node_row;
  RowMem R;
  if constexpr (!RAG) {
    const size_t first = (static_cast<size_t>(row) * static_cast<size_t>(P.row_stride) +
                          static_cast<size_t>(P.al0 - P.col0)) * (DT == SJD_BF16 ? 2 : 4);  // id al0
    R.cr = reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(cond) + first);
    R.ur = CFG ? reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(uncond) + first) : nullptr;
    R.al0 = P.al0;
    R.nL = P.nL;
    R.ragged = false;
  } else {
    const int esz = DT == SJD_BF16 ? 2 : 4;
    const size_t lo_e = static_cast<size_t>(row) * static_cast<size_t>(P.row_stride) +
                        static_cast<size_t>(P.lo - P.col0);  // element of id lo
    const uintptr_t at = reinterpret_cast<uintptr_t>(cond) + lo_e * esz;
    const int shift = static_cast<int>(at & 15u) / esz;  // elements before it in its 16 bytes
    R.al0 = P.lo - shift;
    R.nL = (P.hi - R.al0 + EPC - 1) / EPC * EPC;
    R.cr = reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(cond) + (lo_e - shift) * esz);
    R.ur = CFG ? reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(uncond) + (lo_e - shift) * esz) : nullptr;
    R.ragged = P.f_ragged != 0;
  }
  const int nch = R.nL / EPC;
  // DEPTH rounds of the stream are on their way at a time, the first requested
  // before anything else: in registers, or with 256 threads through a ring in
  // shared memory, where every thread copies the 16 bytes of cond and of uncond
  // that it will process itself (no barrier). A pass of 256 rows: 31.7 us
  // through the ring, 33.3 through registers (drafting from 16384 logits), 26.4
  // against 29.0 (8996 of 10007 ids). With 128 threads the ring's space is
  // taken from the candidate list (46.9 against 42.3 us at 1024 rows), with 512
  // it gains nothing (41.9 against 42.4, 62.1 against 60.5).
  constexpr int RP = NT == 128 ? 1 : 2;     // rounds taken at once (one list reservation for both)
  constexpr int DEPTH = NT == 128 ? 2 : 4;
  constexpr bool RING = NT == 256;
  Chunk<DT> buf[RING ? RP : DEPTH];
  [[maybe_unused]] unsigned char* const ring = smem_raw + P.f_ring + 16 * threadIdx.x;
  constexpr int SLOT = 16 * NT * (CFG ? 2 : 1);
  [[maybe_unused]] auto request = [&](int r, int slot) {
    const int c = threadIdx.x + r * ST, v0 = R.al0 + c * EPC;
    unsigned char* const at = ring + slot * SLOT;
    if (v0 < P.hi) {  // (past the row: what the slot holds is masked)
      if (RAG && R.ragged && (v0 < P.lo || v0 + EPC > P.hi)) {
        const Chunk<DT> k = load_chunk<DT, CFG>(P, R, c);
        *reinterpret_cast<uint4*>(at) = k.c;
        if (CFG) *reinterpret_cast<uint4*>(at + 16 * NT) = k.u;
      } else {
        const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(at));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(R.cr + c) : "memory");
        if (CFG) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * NT), "l"(R.ur + c) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto request_first = [&]() {
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) {
      if constexpr (RING) request(d, d);
      else buf[d] = load_chunk<DT, CFG>(P, R, threadIdx.x + d * ST);
    }
  };
  // (tree) the row's ticket, once everything the block has stored is ordered
  // before it; the last one of the batch element walks the tree and commits
  auto tree_ticket = [&]() {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      s.bi[0] = atomicAdd(P.ticket + b, 1u) == static_cast<uint32_t>(P.rows_b - 1) ? 1 : 0;
    }
    __syncthreads();
    if (s.bi[0]) {
      __threadfence();
      batch_epilogue_tree(P, b, out_committed, out_ncommit, out_firstrej, esc,
                          reinterpret_cast<int32_t*>(smem_raw + P.f_list_l));
    }
  };
  int child_at = 0;  // (tree) slot of the node's first child
  if (node_row) {
    if (P.early_logits != 0) griddep_wait();
    int off = 0, kd = P.K;
#pragma unroll 1
    for (int d = 1; d < nd; ++d, kd *= P.K) off += kd;  // off: depth nd's first slot, kd = K^nd
    child_at = off + kd + ni * P.K;
    // The row of a node that does not exist is not read: it only takes its
    // ticket. (One round trip to L2 before the row's first request; both words
    // are the same for the whole block.)
    const int32_t tok = P.tree_tok[static_cast<size_t>(b) * P.tree_n + SJD_IDX(off + ni, P.tree_n)];
    if (!(nd < P.tree_depth[b] && tok >= 0)) {
      tree_ticket();
      return;
    }
  }
  request_first();
  const int nwords = (R.nL + 31) >> 5;
  if (threadIdx.x == 0) {
    s.mkey = 0u;
    s.lbound = -INFINITY;
    s.win_lo = -INFINITY;
    s.win_hi = INFINITY;
    s.short_list = 0;
    s.interval = 0;
    s.list_count = 0u;
    s.head_count = 0u;
  }
  for (int k = threadIdx.x; k < NB; k += ST) reinterpret_cast<uint32_t*>(smem_raw + P.f_hist)[k] = 0u;
  for (int k = threadIdx.x; k < nwords; k += ST) sm.bitmap[k] = 0u;
  for (int k = threadIdx.x; k < 130; k += ST)
    copy_word(reinterpret_cast<float*>(s.exp2) + k, reinterpret_cast<const float*>(kExp2Table) + k);
  // The row's decode state (position, step, draft group, the stored draft
  // row's length) and its random words, into shared memory by the last warp:
  // two dependent round trips to L2. The first (load_position) is under way
  // with the first rounds of the stream, the second (row_setup, asynchronous
  // copies) behind the first round.
  int abs0 = 0;
  uint32_t step_t = 0;
  auto load_position = [&]() {
    if (warp() != ST / 32 - 1) return;
    abs0 = P.abs_pos[b];
    step_t = P.step_t[b];
  };
  auto row_setup = [&]() {
    if (warp() != ST / 32 - 1) return;
    const int slot = (abs0 + j) % P.W;
    const size_t bs = static_cast<size_t>(b) * P.W + slot;
    const uint32_t pos = static_cast<uint32_t>(abs0 + j);
    if (node_row) {
      // the node's children: depth nd + 1, slots ni K .. ni K + K - 1
      const int c = lane() < P.K
                        ? P.tree_tok[static_cast<size_t>(b) * P.tree_n + SJD_IDX(child_at + lane(), P.tree_n)]
                        : -1;
      const int g = __ffs(~__ballot_sync(0xFFFFFFFFu, c >= 0)) - 1;
      if (lane() < P.K) s.cands[lane()] = c;
      if (lane() == 0) s.g = g;
    } else if (MODE != kModeFromLogits) {
      if (lane() < P.K) copy_word(&s.cands[lane()], P.cand + bs * P.K + lane());  // (those past the group are not used)
      if (lane() == 0) copy_word(&s.g, P.gsize + bs);
    }
    if (MODE != kModeFromLogits && lane() < 5) {
      const uint32_t purpose[5] = {kAccept, kAccept + 8u, kResidual, kPd, kPd + 8u};
      const uint4 r = philox4x32_10(make_uint4(pos, step_t, static_cast<uint32_t>(b), purpose[lane()]), P.seed_lo,
                                    P.seed_hi);
      s.rnd[lane()][0] = r.x;
      s.rnd[lane()][1] = r.y;
      s.rnd[lane()][2] = r.z;
      s.rnd[lane()][3] = r.w;
    }
    if (lane() == 0) {
      if (MODE != kModeFromLogits) copy_word(&s.qlen, P.q_len + bs);
      s.slot = slot;
      s.pos = pos;
      s.t = step_t;
    }
  };
  // the stored draft row's first entries (usually all of a short row)
  auto fetch_draft = [&]() {
    if (MODE == kModeFromLogits || warp() != 0 || lane() >= min(s.qlen, P.S)) return;
    const size_t at = (static_cast<size_t>(b) * P.W + s.slot) * P.S + lane();
    copy_word(&s.dq_id[lane()], P.q_ids + at);
    copy_word(&s.dq_p[lane()], P.q_prob + at);
  };
  if (!early) load_position();
  // ---- S1-S2 streaming pass: logits, running maximum, candidate list.
  // Bound by instruction issue where many rows share an SM.
  const int rounds = (nch + ST - 1) / ST;
  volatile uint32_t* mkey_v = &s.mkey;
  float nan_acc = -INFINITY;  // NaN once a NaN has been read
  float mfix = 0.0f;  // second pass: the final maximum
  // Listed values are >= lmin. The first pass sets it from the first
  // round: a conservative estimate of the row's k-th largest logit (the
  // sample's rank k*ns/nL, plus a quarter and 16 for safety). The estimate is
  // checked once the row is streamed: when fewer than k candidates were
  // listed while it excluded some, the row is streamed again without it.
  float lmin_below = -INFINITY;  // the float below lmin
  float toff = kTCut - 0.5f;     // listed: l above the running maximum plus toff
  uint32_t* hsamp = reinterpret_cast<uint32_t*>(sm.hist);  // [NB] sample histogram (first pass)
  const int lcap = P.f_lcap;
  const ListView Lst{sm.list,
                     reinterpret_cast<uint2*>(P.f_scratch + static_cast<size_t>(row) * P.f_row_bytes + P.f_glist),
                     lcap, early};
  const int lmax = lcap + P.f_gcap;  // list capacity
  // RP rounds (chunks c = threadIdx.x + r ST and the next). First pass: filter with the
  // running maximum (never above the final one), published when a warp
  // exceeds it. Second pass: filter with the final maximum, so that exactly
  // the candidates are listed.
  auto process = [&](const Chunk<DT>* k, int r, bool fixed) {
    const int c = threadIdx.x + r * ST;
    if (r > 0 && (c & ~31) >= nch) return;  // a whole warp past the row (r = 0 has barriers)
    float lv[RP][EPC];
    float cm;
    chunk_logits<DT, CFG>(P, R.al0, k[0], c, lv[0], &cm);
    if constexpr (RP == 2) {
      float c2;
      chunk_logits<DT, CFG>(P, R.al0, k[1], c + ST, lv[1], &c2);
      cm = max_nan(cm, c2);
    }
    float mth = mfix;
    if (!fixed) {
      nan_acc = max_nan(nan_acc, cm);
      mth = key2f(*mkey_v);
      // (a NaN compares false: it is dealt with after the pass)
      if (r == 0 || __any_sync(0xFFFFFFFFu, cm > mth)) {
        const uint32_t wk = __reduce_max_sync(0xFFFFFFFFu, f2key(cm == cm ? cm : -INFINITY));
        if (lane() == 0) atomicMax(&s.mkey, wk);
        mth = fmaxf(mth, key2f(wk));
      }
      if (r == 0) {
        __syncthreads();  // the first round sets a good threshold for everyone
        mth = key2f(*mkey_v);
        // histogram of a sample (512 values of the round for 128 threads, up
        // to 2048 for more) over t in (-34, 0] below its maximum
        constexpr int SPT = fast_sample_per_thread(ST, EPC);
#pragma unroll
        for (int q = 0; q < EPC; q += EPC / SPT) {
          const float tq = __fsub_rn(lv[0][q], mth);
          if (tq > kTCut) atomicAdd(&hsamp[fbin0(tq)], 1u);
        }
        __syncthreads();
        if (warp() == 0) sample_bounds(P, hsamp, mth, s);
        __syncthreads();
        lmin_below = s.lbound == -INFINITY ? -INFINITY : nextafterf(s.lbound, -INFINITY);
        if (s.short_list) toff = kTShort - 0.5f;
        if (!early) row_setup();
      }
    }
    // One comparison lists every id that can have t > -34 under the final
    // maximum m >= mth: such an id has l > m - 34 - 2^-18 (fl(l - m) > -34),
    // while fl(mth - 34.5) <= mth - 34.25 for |mth| < 4e6 (the short list: t >
    // -22 and 22.5 in the same way). Listed ids are tested exactly later.
    // Values below the bound lmin are not listed (l >= lmin is l > the float
    // below lmin); padding and NaN compare false.
    const float thr = fmaxf(fabsf(mth) < 4.0e6f ? __fadd_rn(mth, toff) : -INFINITY, lmin_below);
    // append to the list: one reservation per warp, consecutive entries per lane
    uint32_t cnt = 0;
#pragma unroll
    for (int h = 0; h < RP; ++h)
#pragma unroll
      for (int q = 0; q < EPC; ++q) count_hit(lv[h][q], thr, cnt);
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane() >= o) incl += y;
    }
    uint32_t base = 0;  // (lane 31's count is the warp's)
    if (lane() == 31 && incl) base = atomicAdd(&s.list_count, incl);
    const uint32_t wend = __shfl_sync(0xFFFFFFFFu, base + incl, 31);
    uint32_t at = __shfl_sync(0xFFFFFFFFu, base, 31) + incl - cnt;
    if (wend <= static_cast<uint32_t>(lcap)) {
      uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(sm.list + at));
#pragma unroll
      for (int h = 0; h < RP; ++h)
#pragma unroll
        for (int q = 0; q < EPC; ++q) store_hit(lv[h][q], thr, static_cast<uint32_t>((c + h * ST) * EPC + q), dst);
    } else {
#pragma unroll
      for (int h = 0; h < RP; ++h)
#pragma unroll
        for (int q = 0; q < EPC; ++q)
          if (lv[h][q] > thr) {
            if (at < static_cast<uint32_t>(lmax)) Lst.put(static_cast<int>(at), lv[h][q], (c + h * ST) * EPC + q);
            ++at;
          }
    }
  };
  bool bad = false;  // the row holds a NaN
  int ph = 0;        // parity of the one-barrier reductions
  // Streams the row (again, with the final maximum, when `fixed`); returns the
  // number of listed values (which may exceed the list's capacity).
  auto stream = [&](bool fixed) -> uint32_t {
    __syncthreads();  // counters initialised (first pass) or reset (second)
    if (fixed) request_first();
    [[maybe_unused]] int slot = 0;
    // (one copy of the processing keeps the hot code small)
#pragma unroll 1
    for (int r = 0; r < rounds; r += RP) {
      if constexpr (RING) {
        asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH - RP) : "memory");
#pragma unroll
        for (int h = 0; h < RP; ++h) {
          const unsigned char* const at = ring + (slot + h) * SLOT;
          buf[h].c = *reinterpret_cast<const uint4*>(at);
          buf[h].u = CFG ? *reinterpret_cast<const uint4*>(at + 16 * NT) : make_uint4(0u, 0u, 0u, 0u);
        }
      }
      process(buf, r, fixed);
      if constexpr (RING) {
#pragma unroll
        for (int h = 0; h < RP; ++h) request(r + DEPTH + h, slot + h);
        slot = slot + RP == DEPTH ? 0 : slot + RP;
      } else {
#pragma unroll
        for (int d = 0; d + RP < DEPTH; ++d) buf[d] = buf[d + RP];
#pragma unroll
        for (int h = 0; h < RP; ++h)
          buf[DEPTH - RP + h] = load_chunk<DT, CFG>(P, R, threadIdx.x + (r + DEPTH + h) * ST);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // (the table; row_setup)
    if (__syncthreads_or(nan_acc != nan_acc ? 1 : 0) && !fixed) {
      // A NaN in the allowed range (rare; flagged, then it acts as -inf): its
      // chunk's maximum was lost, so the row's is taken again without NaNs and
      // the row streamed once more.
      bad = true;
      float mx = -INFINITY;
      for (int c2 = threadIdx.x; c2 < nch; c2 += ST) {
        float lv[EPC], cm;
        chunk_logits<DT, CFG>(P, R.al0, load_chunk<DT, CFG>(P, R, c2), c2, lv, &cm);
#pragma unroll
        for (int q = 0; q < EPC; ++q)
          if (lv[q] == lv[q]) mx = fmaxf(mx, lv[q]);
      }
      const uint32_t wk = __reduce_max_sync(0xFFFFFFFFu, f2key(mx));
      if (lane() == 0) atomicMax(&s.mkey, wk);
      __syncthreads();
    }
    return s.list_count;
  };

  uint32_t* const word_base = reinterpret_cast<uint32_t*>(sm.hist);  // kept ids before each bitmap word
  int n = 0;                  // kept ids
  unsigned long long Zk = 0;  // their total weight
  KeptArrays K = sm.small;    // aliases the candidate list: used once the list is dead
  bool short_row = false;     // at most 32 kept ids from the head: warp 0 finishes the row
  bool valid_row = false;     // the row has a finite maximum
  bool head_done = false;     // the kept ids are all in the head
  int nlist = 0;              // entries of the list
  Cut kcut = no_cut(), pcut = no_cut();
  float m = 0.0f;
  // The row is streamed once; again, with the final maximum, when the list
  // overflowed, the sampled bound excluded too much, or the short list of a
  // top-p row left its cut open.
#pragma unroll 1
  for (bool fixed = false;;) {
    const uint32_t appended = stream(fixed);
    if (!early && !fixed) fetch_draft();
    m = key2f(s.mkey);
    valid_row = m < INFINITY && s.mkey > 0x007FFFFFu;
    if (!valid_row) break;  // +inf logit, or no finite logit at all
    bool again = bad && !fixed;
    const bool short_list = !fixed && s.short_list;  // a top-p row that listed only t > -22 (the top-p cut below)
    const float lmin = s.lbound;
    const bool full_list = appended > static_cast<uint32_t>(lmax);
    nlist = full_list ? lmax : static_cast<int>(appended);
    // the estimate excluded candidates (the top-k cut lies well above -34)
    const bool tau_active = !fixed && lmin > __fadd_rn(m, -(34.0f + fmaxf(1.0f, fabsf(m) * 0x1p-20f)));
    if (!fixed) {
      mfix = m;
      if (bad) {
        lmin_below = -INFINITY;
      } else if (full_list) {
        // The list overflowed. Its k-th largest value is at most the row's
        // k-th largest, so streaming the row again (mostly from L2) and listing
        // only the candidates at or above it keeps every top-k member.
        again = true;
        const ListAll la{Lst, nlist, m};
        lmin_below = nextafterf(
            key2f(fast_select<false>(la, m, static_cast<unsigned long long>(P.topk), sm, nwords, s).key), -INFINITY);
      } else if (tau_active) {
        // The estimate may have excluded candidates: it holds when at least k
        // candidates (under the final maximum) are listed above it. With lmin
        // above fl(m - 33.5) (>= m - 33.625 for |m| < 4e6), every listed value
        // has fl(l - m) > -34: the listed entries are the candidates.
        bool holds;
        if (lmin >= __fadd_rn(m, -33.5f) && fabsf(m) < 4.0e6f) {
          holds = appended >= static_cast<uint32_t>(P.topk);
        } else {
          uint32_t nc = 0;
          const ListCand lc0{Lst, nlist, m};
          lc0.each([&](uint32_t, int, float, unsigned long long) { ++nc; });
          holds = fsum(nc, s) >= static_cast<unsigned long long>(P.topk);
        }
        if (!holds) {
          lmin_below = -INFINITY;
          again = true;
        }
      }
    }
    if (!again) {
      // ---- S3: the top-k cut. The list holds every candidate, or every one
      // at or above a bound of the k-th largest: in both cases every top-k
      // member (a top-p row may not need the cut: below).
      const bool may_cut = !full_list && appended > static_cast<uint32_t>(P.topk);
      bool interval = short_list || (may_cut && !fixed && s.interval);
      if (full_list) {
        // More values than the list holds (massive ties): the top-k cut is
        // taken over the row (read again), then only the members are listed.
        // From |m| = 4e6 on, where the list takes values of any size, there may
        // be fewer candidates than k among them, and no cut.
        const GlobalRow<DT, CFG> gr{&P, &R, m};
        uint32_t c = 0;
        gr.each([&](uint32_t, int, float, unsigned long long) { ++c; });
        if (fsum(c, s) > static_cast<unsigned long long>(P.topk))
          kcut = fast_select<false>(gr, m, static_cast<unsigned long long>(P.topk), sm, nwords, s);
        if (threadIdx.x == 0) s.list_count = 0u;
        __syncthreads();
        gr.each([&](uint32_t key, int idx, float, unsigned long long) {
          if (!in_cut(key, idx, kcut)) return;
          const uint32_t at = atomicAdd(&s.list_count, 1u);
          if (at < static_cast<uint32_t>(lmax)) Lst.put(static_cast<int>(at), key2f(key), idx);
        });
        __syncthreads();
        if (s.list_count > static_cast<uint32_t>(lmax) && threadIdx.x == 0) atomicOr(P.err, err_bit(SJD_ERR_CAPACITY));
        nlist = min(static_cast<int>(s.list_count), lmax);
        if (threadIdx.x == 0) atomicAdd(P.stats + kStatsPaths + 1, 1ull);
      }
      if (may_cut && !interval) kcut = topk_cut(Lst, nlist, m, P.topk, s.win_lo, s.win_hi, sm, nwords, s);
      if (!(P.top_p < 1.0f)) break;
      // ---- S3-S4 of a top-p row: the cut is the entry where the running
      // weight reaches target = ceil(tau Z), Z the members' exact total. Where
      // it falls depends on Z only through that target, so Z is first bounded:
      // the head (t > -9) weighed exactly, the other members by the hardware
      // exponential with a margin (2^-13 relative, 2^-22 its error, and one
      // unit each), and, when only ids with t > -22 are taken (interval: at
      // most k of them, so that all are members), the largest weight of the
      // others that may be members. Both bounds give targets, and the cut is
      // decided when one head entry holds both. Of 1024 rows of 8192 ids about
      // one in 10^4 is left open and takes the next step: the top-k cut, the
      // row again (if only t > -22 were listed), the exact Z. Weighing every
      // listed id exactly took 2.8 us of the median row at 1024 rows, and 7.4
      // of rows with 2500 listed ids; the bounds take 2.1 and 5.1. (Without
      // top-p nothing depends on these weights.)
      bool exact = false;
      float thead = kTHead;
#pragma unroll 1
      for (;;) {
        const bool cut_on = kcut.key != no_cut().key || kcut.id != no_cut().id;
        const uint32_t kk = static_cast<uint32_t>(P.topk);
        unsigned long long Zlo, Zhi, z2;  // bounds of Z, without the head until exact
        uint32_t ncand;
        bool open = false;
        if (!exact) {
          const float tlim = interval ? kTShort : kTCut;
          if (threadIdx.x == 0) {
            s.head_count = 0u;
            s.bi[9] = -1;
          }
          __syncthreads();
          float tail = 0.0f;
          uint32_t cpart = 0;
          Lst.each(nlist, [&](uint2 en) {
            const float lv = __uint_as_float(en.x);
            const float tt = __fsub_rn(lv, m);
            if (!(tt > tlim) || (cut_on && !in_cut(f2key(lv), static_cast<int>(en.y), kcut))) return;
            ++cpart;
            if (tt > thead) {
              const uint32_t h = atomicAdd(&s.head_count, 1u);
              if (h < static_cast<uint32_t>(HCAP))
                sm.head[2 * h] = (static_cast<unsigned long long>(f2key(lv)) << 32) | ~en.y;
            } else {
              float e;
              asm("ex2.approx.f32 %0, %1;" : "=f"(e) : "f"(tt * 0x1.715476p+0f));
              tail += e;
            }
          });
          bsum3(cpart, static_cast<unsigned long long>(tail * 0x1p47f), 0ull, s, ph, &ncand, &Zlo, &z2);
          if (s.head_count > static_cast<uint32_t>(HCAP) && thead == kTHead) {
            thead = kTHead2;  // too many ids above -9: the head is t > -6
            __syncthreads();
            continue;
          }
          if (threadIdx.x < min(s.head_count, static_cast<uint32_t>(HCAP))) {
            const uint32_t key = static_cast<uint32_t>(sm.head[2 * threadIdx.x] >> 32);
            unsigned long long E;
            exp_weight(__fsub_rn(key2f(key), m), &E);
            sm.head[2 * threadIdx.x + 1] = E;
          }
          __syncthreads();
          const unsigned long long margin = (Zlo >> 13) + ncand + ST;
          open = interval && ncand > kk;  // the top-k cut may lie among them
          Zhi = Zlo + margin + (interval && !open ? static_cast<unsigned long long>(kk - ncand) * kShortWeight : 0ull);
          Zlo = Zlo > margin ? Zlo - margin : 0ull;
        } else {
          unsigned long long zpart = 0;
          const ListMembers mz{Lst, nlist, m, kcut};
          mz.each([&](uint32_t, int, float, unsigned long long E) { zpart += E; });
          bsum3(0u, zpart, 0ull, s, ph, &ncand, &Zlo, &z2);
          Zhi = Zlo;
        }
        const uint32_t nh = s.head_count;
        if (!open && nh <= static_cast<uint32_t>(HCAP)) {
          // one head entry per thread, ranked (key desc, index asc); the raw
          // values that a kept entry needs are on their way meanwhile
          const bool mine = threadIdx.x < nh;
          unsigned long long me = 0, before = 0, head_mass = 0;
          float rc = 0.0f, ru = 0.0f;
          if (mine) {
            me = sm.head[2 * threadIdx.x];
            raw_logits<DT, CFG>(R, static_cast<int>(~static_cast<uint32_t>(me)), rc, ru);
          }
#pragma unroll 4
          for (uint32_t d = 0; d < nh; ++d) {
            const unsigned long long E = sm.head[2 * d + 1];
            head_mass += E;
            if (sm.head[2 * d] > me) before += E;
          }
          if (!exact) {
            Zlo += head_mass;
            Zhi += head_mass;
          }
          const unsigned long long t_lo = scale_ceil(Zlo, P.tau_mant, P.tau_shift);
          const unsigned long long t_hi = exact ? t_lo : scale_ceil(Zhi, P.tau_mant, P.tau_shift);
          if (mine && before < t_lo && t_hi <= before + sm.head[2 * threadIdx.x + 1]) {
            s.bc64[0] = me;
            s.bi[9] = 1;
          }
          __syncthreads();
          head_done = s.bi[9] >= 0;
          if (head_done) {
            // ---- S4: the kept ids (in the top-p cut, precise weight > 0) in id
            // order; K.pcum holds their weights until the prefix pass
            unsigned long long E = 0;
            if (mine && me >= s.bc64[0])
              E = precise_weight(rc, ru, CFG, P.cfg, P.temp != 1.0f, P.temp, m, s.exp2);
            if (mine) sm.head[2 * threadIdx.x + 1] = E;
            n = __syncthreads_count(E != 0 ? 1 : 0);
            if (E != 0) {
              const uint32_t mi = static_cast<uint32_t>(me);  // ~index
              int rank = 0;
#pragma unroll 4
              for (uint32_t d = 0; d < nh; ++d)
                rank += (sm.head[2 * d + 1] != 0 && static_cast<uint32_t>(sm.head[2 * d]) > mi) ? 1 : 0;
              K.pidx[SJD_IDX(rank, P.f_kcap)] = static_cast<uint16_t>(~mi);
              K.pcum[SJD_IDX(rank, P.f_kcap)] = E;
            }
            __syncthreads();
            break;
          }
        }
        if (interval) {
          // A short list of more than k ids with t > -22 holds every member all
          // the same: it only takes the top-k cut. (Streaming such rows again,
          // four of 1024 in a step of 12288 ids, took 115 us a step against 64.)
          if (short_list && !open) {
            again = true;
            break;
          }
          interval = false;
          kcut = topk_cut(Lst, nlist, m, P.topk, s.win_lo, s.win_hi, sm, nwords, s);
        } else if (!exact) {
          exact = true;
        } else {
          // the cut lies below the head: weighted select over every member
          const ListMembers mg{Lst, nlist, m, kcut};
          pcut = fast_select<true>(mg, m, scale_ceil(Zlo, P.tau_mant, P.tau_shift), sm, nwords, s);
          break;
        }
      }
      if (!again) break;
    }
    // once more: no bound unless the overflowed list gave one, the whole list
    toff = kTCut - 0.5f;
    fixed = true;
    __syncthreads();  // (the count has been read by everyone)
    if (threadIdx.x == 0) {
      s.list_count = 0u;
      atomicAdd(P.stats + kStatsPaths, 1ull);  // this row is streamed a second time
    }
  }
  if (bad && threadIdx.x == 0) atomicOr(P.err, err_bit(SJD_ERR_NONFINITE));
  if (!valid_row) {
    if (threadIdx.x == 0) atomicOr(P.err, err_bit(SJD_ERR_NONFINITE));
  } else {
    // ---- S4 of a row whose kept ids are not all in the head: members in the
    // top-p cut with precise weight > 0, in id order
    if (!head_done) {
      // general: the list's logits become kept weights (-1 otherwise), then a
      // bitmap over the local indices, word prefix counts and ranks
      // four entries at a time, their raw values requested together (a round
      // trip to L2 each)
      for (int i0 = threadIdx.x; i0 < nlist; i0 += 4 * ST) {
        uint2 en[4];
        float rc[4], ru[4];
        bool keep[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * ST;
          en[u] = Lst.at(min(i, nlist - 1));
          const float lv = __uint_as_float(en[u].x);
          const int idx = static_cast<int>(en[u].y);
          const uint32_t key = f2key(lv);
          keep[u] = i < nlist && __fsub_rn(lv, m) > kTCut && in_cut(key, idx, kcut) &&
                    (!(P.top_p < 1.0f) || in_cut(key, idx, pcut));
          rc[u] = ru[u] = 0.0f;
          if (keep[u]) raw_logits<DT, CFG>(R, idx, rc[u], ru[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * ST;
          if (i >= nlist) break;
          const int idx = static_cast<int>(en[u].y);
          unsigned long long E = 0;
          if (keep[u]) {
            E = precise_weight(rc[u], ru[u], CFG, P.cfg, P.temp != 1.0f, P.temp, m, s.exp2);
            if (E) atomicOr(&sm.bitmap[idx >> 5], 1u << (idx & 31));
          }
          Lst.at(i) = ListView::weight_entry(E, idx);
        }
      }
      __syncthreads();
      {
        const int per = (nwords + ST - 1) / ST;
        const int w0 = min(nwords, static_cast<int>(threadIdx.x) * per), w1 = min(nwords, w0 + per);
        unsigned long long c = 0;
#pragma unroll 1
        for (int w = w0; w < w1; ++w) c += __popc(sm.bitmap[w]);
        ph ^= 1;
        const Scan sc = bscan(c, s, ph);
        unsigned long long run = sc.ex;
#pragma unroll 1
        for (int w = w0; w < w1; ++w) {
          word_base[w] = static_cast<uint32_t>(run);
          run += __popc(sm.bitmap[w]);
        }
        n = static_cast<int>(sc.total);
      }
      if (n > P.S) {
        if (threadIdx.x == 0) atomicOr(P.err, err_bit(SJD_ERR_CAPACITY));
        n = P.S;
      }
      // the kept arrays: in shared memory when the layout holds them apart
      // from the list, else in the row's workspace scratch
      const bool k_shared = P.f_kwide && n <= P.f_kcap;
      // the previous step's CTA of this row may still use the row's scratch
      if (early && !k_shared) griddep_wait();
      K = k_shared ? sm.small : global_kept(P, row);
      __syncthreads();
      Lst.each_rolled(nlist, [&](uint2 en) {
        const unsigned long long E = ListView::weight_of(en);
        if (E == 0) return;
        const int idx = ListView::index_of(en);
        const uint32_t word = sm.bitmap[idx >> 5];
        const int r = static_cast<int>(word_base[idx >> 5] + __popc(word & ((1u << (idx & 31)) - 1u)));
        if (r < n) {
          K.pidx[r] = static_cast<uint16_t>(idx);
          K.pcum[r] = E;
        }
      });
      __syncthreads();
    }
    // inclusive prefix of the kept weights (a short kept row from the head does
    // it in warp 0, with verification)
    short_row = head_done && MODE != kModeFromLogits && !TREE && n <= 32;
    if (!short_row) {
      const int per = run_of(n, ST);  // each thread owns a run of kept positions
      const int i0 = min(n, static_cast<int>(threadIdx.x) * per), i1 = min(n, i0 + per);
      unsigned long long loc = 0;
#pragma unroll 2
      for (int i = i0; i < i1; ++i) loc += K.pcum[i];
      ph ^= 1;
      const Scan sc = bscan(loc, s, ph);
      Zk = sc.total;
      unsigned long long run = sc.ex;
#pragma unroll 2
      for (int i = i0; i < i1; ++i) {
        run += K.pcum[i];
        K.pcum[i] = run;
      }
    }
  }
  auto id_of = [&](int i) { return R.al0 + static_cast<int>(K.pidx[SJD_IDX(i, n)]); };
  if (early) {
    griddep_wait();  // the previous step is complete: its state may be read
    load_position();
    row_setup();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();  // the row's state, and the kept row's prefix
  if (early) fetch_draft();
  const int g = MODE == kModeFromLogits ? 1 : node_row ? s.g : min(max(s.g, 1), P.K);
  const int qlen = MODE == kModeFromLogits ? -1 : min(s.qlen, P.S);
  const uint32_t pos = s.pos, t = s.t;
  const size_t bs = static_cast<size_t>(b) * P.W + s.slot;
  const int32_t* qids_g = P.q_ids + bs * P.S;
  const float* qpr_g = P.q_prob + bs * P.S;

  // P^t, the row's stored draft distribution of the next step: ids and
  // p = fl(fl(E) 2^-47 / Wz), Wz = fl(Zk 2^-47)
  auto write_row = [&](int first, int step) {
    const float Wz = fix_to_f32(Zk);
    // (tree: a row that node rows read is held apart until they have)
    const bool held = TREE && tree_holds(P, j);
    int32_t* const ids = (held ? P.tq_ids : P.q_ids) + bs * P.S;
    float* const pr = (held ? P.tq_prob : P.q_prob) + bs * P.S;
#pragma unroll 1
    for (int i = first; i < n; i += step) {
      ids[i] = id_of(i);
      pr[i] = prob_of(weight_at(K.pcum, i), Wz);
    }
  };

  if (MODE == kModeFromLogits) {
    if (warp() == 0) {
      int x = P.lo;
      if (n > 0) {
        const uint32_t odd = odd24(rand32(P, pos, t, static_cast<uint32_t>(b), kSynth, 0));
        x = id_of(warp_search(K.pcum, n, scale_floor(Zk, odd)));
      }
      if (lane() == 0) {
        P.q_len[bs] = n;
        unsigned long long* st = P.stats + kStatsSpread + 3 * (row & (kStatsSlots - 1));
        atomicAdd(st + 0, 1ull);
        atomicAdd(st + 2, static_cast<unsigned long long>(n));
        P.cand[bs * P.K] = x;
        P.gsize[bs] = 1;
        P.win_tok[static_cast<size_t>(b) * P.W + j] = x;
      }
    }
    write_row(threadIdx.x, ST);
    return;
  }

  // ---- S5/S7: verify the draft group (Sec. 3.2, Thm. 2), residual resample.
  // One thread takes every decision (and every fp64 operation); all threads
  // share the per-element residual passes.
  // kept position of local index lc (-1: not kept)
  auto pos_of = [&](int lc) -> int {
    if (n == 0 || lc < 0 || lc >= R.nL) return -1;
    if (!head_done) {
      const uint32_t word = sm.bitmap[lc >> 5], bit = 1u << (lc & 31);
      const int r = static_cast<int>(word_base[lc >> 5]) + __popc(word & (bit - 1u));
      return (word & bit) && r < n ? r : -1;
    }
    int lo = 0, hi = n;
#pragma unroll 1
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (static_cast<int>(K.pidx[mid]) < lc) lo = mid + 1; else hi = mid;
    }
    return (lo < n && static_cast<int>(K.pidx[lo]) == lc) ? lo : -1;
  };
  // The stored draft row against the kept row and the draft group: K.qP, the
  // candidates' draft probabilities s.gqc and kept positions s.gpidx. The
  // draft row's entries are spread over the threads first, first + step, ...
  // and find their kept position (the other way round, every kept id searched
  // the draft row, which had to be in shared memory: 8 S bytes). `sync` waits
  // for those threads.
  auto merge_draft = [&](int first, int step, auto sync) {
#pragma unroll 1
    for (int i = first; i < n; i += step) K.qP[i] = qlen < 0 ? P.uniform_q : 0.0f;
    asm volatile("cp.async.wait_all;" ::: "memory");  // (fetch_draft, by warp 0, which runs this first or alone)
    if (first < g) {
      const int c = s.cands[first];
      s.gpidx[first] = pos_of(c - R.al0);
      s.gqc[first] = qlen < 0 && c >= P.lo && c < P.hi ? P.uniform_q : 0.0f;
    }
    sync();
    if (qlen <= 0) return;
#pragma unroll 1
    for (int i = first; i < qlen; i += step) {
      const int v = i < 32 ? s.dq_id[i] : __ldcg(qids_g + i);
      const float q = i < 32 ? s.dq_p[i] : __ldcg(qpr_g + i);
      const int r = pos_of(v - R.al0);
      if (r >= 0) K.qP[r] = q;
#pragma unroll 1
      for (int k = 0; k < g; ++k)
        if (v == s.cands[k]) s.gqc[k] = q;
    }
    sync();
  };
  // The row's results, then its ticket: by warp 0 (every lane), with its own
  // fence, so that the other warps' stores of P^t are not waited for. The
  // last ticket of the batch element runs the epilogue below.
  auto publish = [&](int x, int na, int xf, int naf) {
    const int Km1 = P.K - 1, ln = lane();
    if (ln < na) P.res_alt[bs * Km1 + ln] = s.alts[ln];
    if (!P.ac && ln < naf) P.res_altf[bs * Km1 + ln] = s.altf[ln];
    if (ln == 0) {
      P.res_altn[bs] = na;
      P.res_x[bs] = x;
      P.res_dev[bs] = x != s.cands[0] ? 1 : 0;
      if (!P.ac) {
        P.res_altfn[bs] = naf;
        P.res_xf[bs] = xf;
      }
      P.q_len[bs] = n;
    }
    __syncwarp();
    if (ln == 0) {
      __threadfence();
      const uint32_t done = atomicAdd(P.ticket + b, 1u);
      s.bi[0] = done == static_cast<uint32_t>(P.W - 1) ? 1 : 0;
      unsigned long long* st = P.stats + kStatsSpread + 3 * (row & (kStatsSlots - 1));
      atomicAdd(st + 0, 1ull);
      atomicAdd(st + 1, static_cast<unsigned long long>(max(qlen, 0)));
      atomicAdd(st + 2, static_cast<unsigned long long>(n));
    }
  };
  // One warp finishes a row of at most 32 kept ids, and merges a short draft
  // row too; the ids of a longer one are looked for by the block (by one warp,
  // 128 rows that turn from 1900 kept ids to a few: 53.4 us a step against
  // 37.0).
  const bool warp_row = !TREE && n > 0 && n <= 32;
  const bool warp_merge = warp_row && qlen <= 128;
  if (n > 0 && !warp_merge) merge_draft(threadIdx.x, ST, [] { __syncthreads(); });
  if (warp_row) {
    // ---- a short kept row (the common case: top-p keeps a few ids): warp 0
    // verifies, resamples and draws with one kept position per lane and the
    // same operations as the block path below, without block barriers
    if (warp() == 0) {
      const int ln = lane();
      const bool mine = ln < n;
      // inclusive prefix over the lanes (positions) of a u64
      auto lane_incl = [&](unsigned long long v) {
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, v, o);
          if (ln >= o) v += y;
        }
        return v;
      };
      if (short_row) {
        // inclusive prefix of the kept weights
        const unsigned long long inc = lane_incl(mine ? K.pcum[ln] : 0ull);
        Zk = __shfl_sync(0xFFFFFFFFu, inc, 31);
        __syncwarp();
        if (mine) K.pcum[ln] = inc;
      }
      __syncwarp();
      if (warp_merge) merge_draft(ln, 32, [] { __syncwarp(); });
      int x = s.cands[0], xidx = -1;
      const unsigned long long pc = mine ? K.pcum[ln] : 0ull;
      const unsigned long long w = mine ? weight_at(K.pcum, ln) : 0ull;
      unsigned long long Wk = w, Wsum = Zk;  // p^(k) as integer weights (my position; total)
      const float qP = mine ? K.qP[ln] : 0.0f;
      bool accepted = false;
      double S = 0.0;  // draft mass of the rejected candidates
      unsigned long long R = 0, Rsum = 0;
      const int grp = (P.group_of && mine) ? __ldg(P.group_of + id_of(ln)) : 0;  // relaxed test: my id's group
#pragma unroll 1
      for (int k = 1; k <= g; ++k) {
        const int pi = s.gpidx[k - 1];
        unsigned long long Wc = __shfl_sync(0xFFFFFFFFu, Wk, max(pi, 0) & 31);
        if (P.group_of) {  // the weight of the candidate's whole group (relaxed, lossy)
          const int gc = __ldg(P.group_of + s.cands[k - 1]);
          Wc = wadd64(mine && grp == gc ? Wk : 0ull);
        }
        const double d = __dsub_rn(1.0, S);
        int acc = 0;
        if (ln == 0) {
          const float q_c = s.gqc[k - 1];
          if (q_c == 0.0f && !P.group_of) {
            atomicOr(P.err, err_bit(SJD_ERR_INVALID_DRAFT));
          } else {
            acc = accept_exact(odd24(s.rnd[(k - 1) >> 2][(k - 1) & 3]), q_c, Wsum,
                               (pi >= 0 || P.group_of) ? Wc : 0ull, d) ? 1 : 0;
          }
        }
        if (__shfl_sync(0xFFFFFFFFu, acc, 0)) {
          x = s.cands[k - 1];
          xidx = pi;
          accepted = true;
          break;
        }
        if (k == 1) {
          R = mine ? residual_first(Wk, qP, Wsum) : 0ull;
        } else {
          // the tokens of the rejected levels leave the draft's support
          unsigned long long A_fix = 0;
          int G = 0;
          if (ln == 0) level_scale(Wsum, d, &A_fix, &G);
          A_fix = __shfl_sync(0xFFFFFFFFu, A_fix, 0);
          G = __shfl_sync(0xFFFFFFFFu, G, 0);
          bool rem = false;
#pragma unroll 1
          for (int e = 0; e < k - 1; ++e) rem |= s.gpidx[e] == ln;
          R = mine ? (rem ? Wk : residual_level(Wk, qP, A_fix, G)) : 0ull;
        }
        Rsum = wadd64(R);
        if (Rsum == 0) {  // only reachable through rounding: sample from p^(k)
          R = Wk;
          Rsum = Wsum;
        }
        if (k == g) break;
        S = __dadd_rn(S, f32_to_f64(s.gqc[k - 1]));
        if (!(__dsub_rn(1.0, S) > 0.0)) break;
        Wk = R;
        Wsum = Rsum;
      }
      // first position whose value exceeds T (the last one when none does)
      auto first_over = [&](unsigned long long v, unsigned long long T) {
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, mine && v > T);
        return hit ? __ffs(hit) - 1 : n - 1;
      };
      if (!accepted) {
        const unsigned long long T = scale_floor(Rsum, odd24(s.rnd[2][0]));
        const unsigned long long incl = lane_incl(R);  // every lane takes part in the shuffles
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, mine && incl > T);
        xidx = hit ? __ffs(hit) - 1 : -1;
        if (xidx >= 0) x = id_of(xidx);
      }
      // ---- S8: proactive-drafting alternates and the vanilla-SJD tail draw
      auto draw = [&](int first_idx, int32_t* out) {
        unsigned long long tot = Zk, cx = pc;  // cx: C'(i), pcum minus the excluded weights up to i
        if (first_idx >= 0) {
          const unsigned long long wi = __shfl_sync(0xFFFFFFFFu, w, first_idx);
          if (ln >= first_idx) cx -= wi;
          tot -= wi;
        }
        int drawn = 0;
#pragma unroll 1
        for (int kk = 1; kk <= P.K - 1; ++kk) {
          if (tot == 0) break;
          const int i = first_over(cx, scale_floor(tot, odd24(s.rnd[3 + (kk >> 2)][kk & 3])));
          if (ln == 0) out[drawn] = id_of(i);
          ++drawn;
          const unsigned long long wi = __shfl_sync(0xFFFFFFFFu, w, i);
          if (ln >= i) cx -= wi;
          tot -= wi;
        }
        return drawn;
      };
      const int na = draw(xidx, s.alts);
      int xf = x, naf = 0;
      if (!P.ac) {
        const int fidx = first_over(pc, scale_floor(Zk, odd24(s.rnd[2][0])));
        xf = id_of(fidx);
        naf = draw(fidx, s.altf);
      }
      __syncwarp();
      publish(x, na, xf, naf);
      write_row(ln, 32);
    }
  } else {
    // ---- the block path. Every thread owns the kept positions [i0, i1)
    // through all levels, so that a level is one pass over them and one scan;
    // the deciding thread is in the last warp, whose share is the smallest.
    // Bound by the chain of levels (the acceptance test in fp64, the pass, the
    // scan): a row of n = 2000 rejected at four levels takes 15.1 us with 512
    // threads, and 21.3 where each residual is computed twice around a
    // two-barrier sum with the level's scale between them.
    int x = s.cands[0];
    int xidx = -1;
    if (n > 0) {
      const int per = run_of(n, ST);
      const int i0 = min(n, static_cast<int>(threadIdx.x) * per), i1 = min(n, i0 + per);
      const bool decider = threadIdx.x == ST - 32, scaler = threadIdx.x == ST - 64;
      if (decider) s.bi[7] = -1;
      // residual weight of position i at level k from its weight w there
      auto residual = [&](int k, int i, unsigned long long w, unsigned long long Z1) {
        if (k == 1) return residual_first(w, K.qP[i], Z1);
        // the tokens of the rejected levels leave the draft's support
        bool rem = false;
#pragma unroll 1
        for (int e = 0; e < k - 1; ++e) rem |= s.gpidx[e] == i;
        return rem ? w : residual_level(w, K.qP[i], s.lvA[k - 1], s.lvG[k - 1]);
      };
      // p^(k) as integer weights: the kept weights (differences of K.pcum) at
      // k = 1, then K.Rw; the total is Wsum
      unsigned long long Wsum = Zk, Rsum = 0, run = 0, loc = 0;
      double S = 0.0, d = 1.0;  // draft mass of the rejected candidates and 1 - S (decider and scaler)
      uint32_t kept_levels = 0;  // levels whose residual was empty: p^(k+1) = p^(k)
      bool accepted = false;
#pragma unroll 1
      for (int k = 1; k <= g; ++k) {
        unsigned long long WG = 0;
        if (P.group_of) {  // the weight of the candidate's whole group (relaxed, lossy)
          const int gc = __ldg(P.group_of + s.cands[k - 1]);
          unsigned long long part = 0;
#pragma unroll 1
          for (int i = i0; i < i1; ++i)
            if (__ldg(P.group_of + id_of(i)) == gc) part += k == 1 ? weight_at(K.pcum, i) : K.Rw[i];
          WG = fsum(part, s);
        }
        if (decider) {
          const float q_c = s.gqc[k - 1];
          const int pi = s.gpidx[k - 1];
          const unsigned long long Wc =
              P.group_of ? WG : (pi < 0 ? 0ull : (k == 1 ? weight_at(K.pcum, pi) : K.Rw[pi]));
          int acc = 0;
          if (q_c == 0.0f && !P.group_of) {
            atomicOr(P.err, err_bit(SJD_ERR_INVALID_DRAFT));
          } else {
            const uint32_t odd = odd24(s.rnd[(k - 1) >> 2][(k - 1) & 3]);
            acc = accept_exact(odd, q_c, Wsum, Wc, d) ? 1 : 0;
          }
          s.bi[6] = acc;
        }
        if (scaler && k > 1) level_scale(Wsum, d, &s.lvA[k - 1], &s.lvG[k - 1]);
        __syncthreads();
        if (s.bi[6]) {
          x = s.cands[k - 1];
          xidx = s.gpidx[k - 1];
          accepted = true;
          break;
        }
        loc = 0;
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
          const unsigned long long R = residual(k, i, k == 1 ? weight_at(K.pcum, i) : K.Rw[i], Wsum);
          K.Rw[i] = R;
          loc += R;
        }
        if (decider || scaler) {
          S = __dadd_rn(S, f32_to_f64(s.gqc[k - 1]));
          d = __dsub_rn(1.0, S);
          if (decider) s.bi[18] = d > 0.0 ? 0 : 1;  // the group's draft mass is spent
        }
        ph ^= 1;
        Scan sc = bscan(loc, s, ph);
        if (sc.total == 0) {
          // only reachable through rounding: sample from p^(k), formed again from the levels before
          kept_levels |= 1u << k;
          loc = 0;
#pragma unroll 1
          for (int i = i0; i < i1; ++i) {
            unsigned long long w = weight_at(K.pcum, i);
#pragma unroll 1
            for (int e = 1; e < k; ++e)
              if (!((kept_levels >> e) & 1u)) w = residual(e, i, w, Zk);
            K.Rw[i] = w;
            loc += w;
          }
          ph ^= 1;
          sc = bscan(loc, s, ph);
        }
        run = sc.ex;
        Rsum = sc.total;
        if (k == g || s.bi[18]) break;
        Wsum = Rsum;
      }
      if (!accepted) {
        const unsigned long long T = scale_floor(Rsum, odd24(s.rnd[2][0]));
        if (run <= T && T < run + loc) {
#pragma unroll 1
          for (int i = i0; i < i1; ++i) {
            run += K.Rw[i];
            if (run > T) {
              s.bi[7] = i;
              break;
            }
          }
        }
        __syncthreads();
        xidx = s.bi[7];
        if (xidx >= 0) x = id_of(xidx);
      }
    }
    // ---- S8: proactive-drafting alternates and the vanilla-SJD tail draw, by
    // warp 0 while the others store P^t.
    // (count tokens without replacement, word(k) their random words, put(k, i)
    // takes the position of the k-th)
    auto draw = [&](int first_idx, int count, auto word, auto put) {
      unsigned long long tot = Zk;
      int nex = 0, drawn = 0;
      // lane e holds the e-th excluded position's weight interval [ea, ea + ew) of pcum
      unsigned long long ea = ~0ull, ew = 0;
      auto exclude = [&](int i) {
        const unsigned long long end = K.pcum[i], wi = weight_at(K.pcum, i);
        if (lane() == nex) {
          ea = end - wi;
          ew = wi;
        }
        tot -= wi;
        ++nex;
      };
      if (first_idx >= 0) exclude(first_idx);
#pragma unroll 1
      for (int kk = 1; kk <= count; ++kk) {
        if (tot == 0) break;
        // T among the weights left is T plus the excluded intervals that
        // begin at or before it (each one added may reach the next)
        unsigned long long T = scale_floor(tot, odd24(word(kk)));
        uint32_t used = 0;
#pragma unroll 1
        for (;;) {
          const bool reach = ea <= T && !((used >> lane()) & 1u);
          const uint32_t hit = __ballot_sync(0xFFFFFFFFu, reach);
          if (!hit) break;
          T += wadd64(reach ? ew : 0ull);
          used |= hit;
        }
        const int i = warp_search(K.pcum, n, T);
        put(drawn, i);
        ++drawn;
        if (kk < count) exclude(i);
      }
      return drawn;
    };
    auto pd_word = [&](int kk) { return s.rnd[3 + (kk >> 2)][kk & 3]; };
    if constexpr (TREE) {
      // The groups of the next tree off the main path as well, for whichever
      // depth this row takes in it: group gi (lanes gi K .. gi K + K - 1) by
      // warp gi mod the warps, group 0 being the alternates.
      if (node_row) {
        if (threadIdx.x == 0) P.res_node[static_cast<size_t>(b) * P.X + SJD_IDX(jr - P.W, P.X)] = x;
      } else {
        const int Km1 = P.K - 1;
#pragma unroll 1
        for (int gi = warp(); gi <= P.tree_g; gi += ST / 32) {
          int32_t* const out = gi == 0 ? P.res_alt + bs * Km1
                                       : P.res_tree + (bs * static_cast<size_t>(P.tree_g) + (gi - 1)) * P.K;
          const int count = gi == 0 ? Km1 : P.K;
          const int na = n == 0 ? 0
                                : draw(gi == 0 ? xidx : -1, count,
                                       [&](int kk) {
                                         return gi == 0 ? pd_word(kk)
                                                        : rand32(P, pos, t, static_cast<uint32_t>(b), kTree,
                                                                 static_cast<uint32_t>(gi * P.K + kk - 1));
                                       },
                                       [&](int k, int i) {
                                         if (lane() == 0) out[k] = id_of(i);
                                       });
          if (lane() == 0) {
            if (gi == 0) P.res_altn[bs] = na;
            else
              for (int k = na; k < P.K; ++k) out[k] = -1;
          }
        }
        if (threadIdx.x == 0) {
          P.res_x[bs] = x;
          P.res_dev[bs] = x != s.cands[0] ? 1 : 0;
          P.tq_len[bs] = n;
          unsigned long long* st = P.stats + kStatsSpread + 3 * (row & (kStatsSlots - 1));
          atomicAdd(st + 0, 1ull);
          atomicAdd(st + 1, static_cast<unsigned long long>(max(qlen, 0)));
          atomicAdd(st + 2, static_cast<unsigned long long>(n));
        }
        write_row(threadIdx.x, ST);
      }
      tree_ticket();
      return;
    }
    if (warp() == 0) {
      const int na = n > 0 ? draw(xidx, P.K - 1, pd_word, [&](int k, int i) { if (lane() == 0) s.alts[k] = id_of(i); }) : 0;
      int xf = x, naf = 0;
      if (!P.ac && n > 0) {
        const int fidx = warp_search(K.pcum, n, scale_floor(Zk, odd24(s.rnd[2][0])));
        xf = id_of(fidx);
        naf = draw(fidx, P.K - 1, pd_word, [&](int k, int i) { if (lane() == 0) s.altf[k] = id_of(i); });
      }
      __syncwarp();
      publish(x, na, xf, naf);
    } else {
      write_row(static_cast<int>(threadIdx.x) - 32, ST - 32);
    }
  }

  // ---- last row of the batch element: S6 (+ S9 in the fused step)
  __syncthreads();
  if (s.bi[0]) {
    __threadfence();
    batch_epilogue_staged(P, b, static_cast<int>(pos) - j, t, MODE == kModeStep, out_committed, out_ncommit,
                          out_firstrej, esc, reinterpret_cast<int32_t*>(smem_raw + P.f_list_l), P.f_region_bytes / 4);
  }
}

// Raise (never lower) the dynamic shared-memory limit of one kernel.
template <class Kern>
cudaError_t raise_limit(Kern* k, int bytes) {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, k);
  if (e != cudaSuccess || a.maxDynamicSharedSizeBytes >= bytes) return e;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// The kernels of one layout: a context launches no others. (Host steps of a
// ragged configuration run on compact aligned rows, on the same kernels.)
template <int DT, int MODE>
cudaError_t set_one(int nt, bool ragged, int bytes) {
  auto both = [&](auto* with, auto* without) {
    const cudaError_t e = raise_limit(with, bytes);
    return e == cudaSuccess ? raise_limit(without, bytes) : e;
  };
  switch (nt) {
    case 512: return both(stream_row_kernel<DT, MODE, true, 512, true>, stream_row_kernel<DT, MODE, false, 512, true>);
    case 256: return both(stream_row_kernel<DT, MODE, true, 256, true>, stream_row_kernel<DT, MODE, false, 256, true>);
    default:
      return ragged ? both(stream_row_kernel<DT, MODE, true, 128, true>, stream_row_kernel<DT, MODE, false, 128, true>)
                    : both(stream_row_kernel<DT, MODE, true, 128, false>, stream_row_kernel<DT, MODE, false, 128, false>);
  }
}


// Launched with programmatic stream serialization: the grid may begin while
// the previous kernel in the stream finishes (the kernel waits for it before
// its first global read).
template <int DT, int MODE, bool CFG, int NT, bool RAG>
cudaError_t launch_pdl(const DevParams& p, const void* cond, const void* uncond, int32_t* oc, int32_t* on,
                       int32_t* of, cudaStream_t s) {
  return launch_overlapped(stream_row_kernel<DT, MODE, CFG, NT, RAG>, dim3(p.B * p.rows_b), dim3(NT), p.f_smem_bytes, s, p, cond,
                           uncond, oc, on, of);
}

template <int DT, int MODE, int NT, bool RAG>
cudaError_t launch_n(const DevParams& p, const void* cond, const void* uncond, bool use_cfg, int32_t* oc,
                     int32_t* on, int32_t* of, cudaStream_t s) {
  return use_cfg ? launch_pdl<DT, MODE, true, NT, RAG>(p, cond, uncond, oc, on, of, s)
                 : launch_pdl<DT, MODE, false, NT, RAG>(p, cond, uncond, oc, on, of, s);
}

template <int DT, int MODE>
cudaError_t launch_m(const DevParams& p, const void* cond, const void* uncond, bool use_cfg, int32_t* oc,
                     int32_t* on, int32_t* of, cudaStream_t s) {
  switch (p.f_nt) {
    case 512: return launch_n<DT, MODE, 512, true>(p, cond, uncond, use_cfg, oc, on, of, s);
    case 256: return launch_n<DT, MODE, 256, true>(p, cond, uncond, use_cfg, oc, on, of, s);
    default:
      return p.f_ragged_kernel ? launch_n<DT, MODE, 128, true>(p, cond, uncond, use_cfg, oc, on, of, s)
                               : launch_n<DT, MODE, 128, false>(p, cond, uncond, use_cfg, oc, on, of, s);
  }
}

}  // namespace

// The (dtype, mode) variants, instantiated one pair per translation unit
// (sjd_fast_part.cu) so that they compile in parallel.
template <int DT, int MODE>
cudaError_t fast_launch(const DevParams& p, const void* cond, const void* uncond, bool use_cfg, int32_t* oc,
                        int32_t* on, int32_t* of, cudaStream_t s) {
  return launch_m<DT, MODE>(p, cond, uncond, use_cfg, oc, on, of, s);
}

template <int DT, int MODE>
cudaError_t fast_raise_smem(int nt, bool ragged, int bytes) {
  return set_one<DT, MODE>(nt, ragged, bytes);
}

}  // namespace sjd
