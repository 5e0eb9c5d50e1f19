// Selection helpers shared by the retrieval kernels: shared-memory histogram walks, the radix select of the top-k
// (Eq. 8), the union with the persistent selection (Sec. 3.5), the host-memory pager's cache policy, token ranges.
#pragma once

#include "common.cuh"

namespace ltri {

// Warp-parallel walks over a shared-memory histogram (all 32 lanes of one warp call them).
// pick_from_top: the largest bin b with  sum(hist[b+1..nb-1]) < need <= sum(hist[b..nb-1]);  `need` becomes the rank
// inside that bin.  pick_from_bottom: the smallest bin b with  rank < sum(hist[0..b]);  `rank` becomes the rank inside
// the bin.  Both clamp to the last bin they look at when the counts do not reach the target.  nb is a multiple of 32.
__device__ __forceinline__ int pick_from_top(const unsigned* hist, int nb, unsigned& need) {
  const int lane = threadIdx.x & 31, per = nb >> 5;
  const int b1 = nb - lane * per;  // lane 0 owns the top `per` bins
  unsigned mine = 0;
  for (int i = 1; i <= per; ++i) mine += hist[b1 - i];
  unsigned incl = mine;  // counts of this lane's bins and of all higher ones
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, incl >= need);
  const int src = hit ? __ffs(hit) - 1 : 31;
  int bin = 0;
  unsigned left = 0;
  if (lane == src) {
    left = need - (incl - mine);
    bin = b1 - 1;
    for (; bin > b1 - per; --bin) {
      if (left <= hist[bin]) break;
      left -= hist[bin];
    }
    if (!hit && left > hist[bin]) left = hist[bin];
  }
  need = __shfl_sync(0xffffffffu, left, src);
  return __shfl_sync(0xffffffffu, bin, src);
}

__device__ __forceinline__ unsigned pick_from_bottom(const unsigned* hist, int nb, long long& rank) {
  const int lane = threadIdx.x & 31, per = nb >> 5;
  const int b0 = lane * per;
  long long mine = 0;
  for (int i = 0; i < per; ++i) mine += hist[b0 + i];
  long long incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = shfl_up_ll(incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, rank < incl);
  const int src = hit ? __ffs(hit) - 1 : 31;
  unsigned bin = 0;
  long long left = 0;
  if (lane == src) {
    left = rank - (incl - mine);
    bin = (unsigned)b0;
    for (; bin < (unsigned)(b0 + per - 1); ++bin) {
      if (left < (long long)hist[bin]) break;
      left -= hist[bin];
    }
  }
  rank = shfl_ll(left, src);
  return __shfl_sync(0xffffffffu, bin, src);
}

// Counting one radix digit of many keys with few shared-memory atomics.  Scores of one head share their leading bits,
// so in the first passes nearly every key falls into the same bin and one atomic per key would serialise on it.  A
// thread adds up runs of equal digits among its own keys; when all lanes of a warp end on the same digit, the warp
// adds their last runs with one atomic.  flush() is called by all 32 lanes of a warp, converged.
struct DigitRuns {
  int cur = -1;
  unsigned run = 0;
  __device__ __forceinline__ void add(unsigned* hist, int d) {
    if (d == cur) {
      ++run;
    } else {
      if (run) atomicAdd(&hist[cur], run);
      cur = d;
      run = 1;
    }
  }
  __device__ __forceinline__ void flush(unsigned* hist) {
    const int top = __reduce_max_sync(0xffffffffu, cur);  // (-1: a lane without a matching key)
    if (__all_sync(0xffffffffu, cur == top || cur < 0)) {
      const unsigned sum = __reduce_add_sync(0xffffffffu, run);
      if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&hist[top], sum);
    } else if (run) {
      atomicAdd(&hist[cur], run);
    }
    cur = -1;
    run = 0;
  }
};

// Exclusive scan of the nt (a multiple of 32, at most 1024) counts in s_scan by the first warp of the CTA; returns the
// total to every thread of that warp.  The caller brackets it with __syncthreads().
__device__ __forceinline__ int warp0_exclusive_scan(int* s_scan, int nt) {
  const int lane = threadIdx.x & 31;
  int run = 0;
  for (int blk = 0; blk < nt; blk += 32) {
    const int v = s_scan[blk + lane];
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    s_scan[blk + lane] = run + inc - v;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  return run;
}

// Union of this step's selection (s_ids[0..cnt), ascending) with the selection the last prefill call left in
// persist_sel (ascending, -1 padded): the persistent mechanism of Sec. 3.5.  Writes the ascending, duplicate-free id
// list to s_all and returns its length.  Called by every thread of the CTA; s_tmp has room for kMaxTopK ints.
__device__ __forceinline__ int union_with_persistent(const DevCtx& c, size_t unit, int g, const int* s_ids, int cnt,
                                                     int* s_tmp, int* s_all) {
  // an element's place is the number of smaller ones in both lists, a thread each (walking the two lists with one thread took
  // some 6K cycles of every decode step)
  const int tid = threadIdx.x, b = tid - kMaxTopK;  // threads 0..63: this step's ids, 64..127: the kept ones
  const bool kept = b >= 0 && b < c.topk;
  int v = -1;
  if (tid < min(cnt, kMaxTopK)) v = s_ids[tid];
  if (kept) {
    v = c.persist ? c.persist_sel[(unit * c.Hkv + g) * (size_t)c.topk + b] : -1;
    for (int i = 0; i < cnt; ++i) v = s_ids[i] == v ? -1 : v;  // (named by both: counted once)
    s_tmp[b] = v;
  }
  const int n = __syncthreads_count(v >= 0);
  if (v >= 0) {
    int at = 0;
    for (int i = 0; i < cnt; ++i) at += s_ids[i] < v;
    for (int i = 0; i < c.topk; ++i) at += s_tmp[i] >= 0 && s_tmp[i] < v;
    s_all[at] = v;
  }
  __syncthreads();
  return n;
}

__device__ __forceinline__ unsigned order_key(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Bin (0..254, 255: further away) of how far the upper 16 bits of a key lie below those of the largest key.  The upper 16 bits
// have 128 steps per power of two: one step per bin for the nearest 128, then 4, 16 and 64, so that a K-th score
// 2^22 times smaller than the best is still found by one histogram (with one step per bin throughout, two powers of two, the
// planted streams of 128K tokens sent every other retrieval to the passes of the general select: 28K cycles instead of 9K).
__device__ __forceinline__ unsigned dist_bin(unsigned d) {
  // bins 0..127 | 128..191 from d = 128 | 192..223 from 384 | 224..254 from 896 | 255 from 2880
  return min(min(d, 96u + (d >> 2)), min(min(168u + (d >> 4), 210u + (d >> 6)), 255u));
}
// the largest distance that falls into bin b
__device__ __forceinline__ unsigned dist_last(unsigned b) {
  return b < 128u ? b : b < 192u ? 4u * b - 381u : b < 224u ? 16u * b - 2673u : b < 255u ? 64u * b - 13377u : 0xffffffffu;
}

// Radix select of the K largest keys among KEY(0..N) (ties: lower index first), one 8-bit digit per pass from the top.
// Writes the chosen indices, unordered, to s_ids and their number to *s_cnt (which the caller has zeroed).  Called by
// every thread of the CTA; K < N.  R > 0 (keys that are expensive to read, 32-bit): up to R keys per thread are read
// once and kept in registers (thread t holds keys t, t + nt, ...); with more keys than that, or R = 0, every pass
// reads them through KEY.  s_scan has room for one word per thread, and with s_ckey for at least 64 + kSelCand words.
constexpr int kSelCand = 256;  // keys the short cut of radix_select_top ranks against each other

template <typename KT, int R, typename KeyF>
__device__ __forceinline__ void radix_select_top(KeyF&& KEY, int N, int K, unsigned* hist, KT* s_prefix,
                                                 unsigned* s_need, int* s_scan, int* s_cnt, int* s_ids,
                                                 unsigned* s_ckey = nullptr) {
  static_assert(R == 0 || sizeof(KT) == 4, "register copies are kept of 32-bit keys only");
  const int tid = threadIdx.x, nt = blockDim.x;
  constexpr int kPasses = (int)sizeof(KT);
  const bool inreg = R > 0 && N <= R * nt;
  unsigned kr[R > 0 ? R : 1];
  if (inreg) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int s = tid + i * nt;
      kr[i] = s < N ? (unsigned)KEY(s) : 0u;
    }
  }
  // f(index, key) for every key of this thread
  auto for_each_key = [&](auto&& f) {
    if (inreg) {
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int s = tid + i * nt;
        if (s < N) f(s, (KT)kr[i]);
      }
    } else {
      // eight keys in flight per thread (KEY may be a load from global memory)
      for (int base = tid; base < N; base += 8 * nt) {
        KT k8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int s = base + u * nt;
          k8[u] = s < N ? (KT)KEY(s) : (KT)0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int s = base + u * nt;
          if (s < N) f(s, k8[u]);
        }
      }
    }
  };
  if (sizeof(KT) == 4 && s_ckey != nullptr) {
    // Short cut for 32-bit keys (K is small against N): with the block's largest key M known, one histogram of how far a
    // key's upper 16 bits lie below M's (dist_bin) gives the smallest bin b within which at least K keys lie; those keys --
    // usually a few more than K -- are listed in shared memory and ranked against each other (key, then lower index).  Four
    // barriers instead of twelve and about a third of the instructions of the four radix passes.  The radix passes below
    // remain for the cases this does not cover: the K-th key in the last bin, or more than kSelCand keys within b (many
    // equal keys).
    int* s_cid = s_scan + 64;  // (s_scan[32..34]: scratch words)
    const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    unsigned m = 0;
    for_each_key([&](int, KT key) { m = max(m, (unsigned)key); });
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) s_scan[wid] = (int)m;
    if (tid < 256) hist[tid] = 0;
    if (tid == 0) s_scan[34] = 0;
    __syncthreads();
    m = __reduce_max_sync(0xffffffffu, (unsigned)s_scan[lane < nw ? lane : 0]);
    const unsigned M16 = m >> 16;
    DigitRuns dr;
    for_each_key([&](int, KT key) { dr.add(hist, (int)dist_bin(M16 - ((unsigned)key >> 16))); });
    dr.flush(hist);
    __syncthreads();
    if (tid < 32) {
      long long rank = K - 1;  // (0-based from the top = from bin 0)
      const unsigned b = pick_from_bottom(hist, 256, rank);
      if (tid == 0) s_scan[33] = (int)b;
    }
    __syncthreads();
    const unsigned bcut = (unsigned)s_scan[33];
    if (bcut < 255u) {
      const unsigned dcut = dist_last(bcut);
      for_each_key([&](int s, KT key) {
        if (M16 - ((unsigned)key >> 16) <= dcut) {
          const int j = atomicAdd(&s_scan[34], 1);
          if (j < kSelCand) {
            s_ckey[j] = (unsigned)key;
            s_cid[j] = s;
          }
        }
      });
      __syncthreads();
      const int nc = s_scan[34];
      if (nc <= kSelCand) {
        for (int j = tid; j < nc; j += nt) {
          const unsigned key = s_ckey[j];
          const int id = s_cid[j];
          int rank = 0;
          for (int i = 0; i < nc; ++i) rank += (s_ckey[i] > key) || (s_ckey[i] == key && s_cid[i] < id);
          if (rank < K) {
            const int slot = atomicAdd(s_cnt, 1);
            if (slot < kMaxTopK) s_ids[slot] = id;
          }
        }
        return;
      }
    }
    __syncthreads();  // (the scratch words are free again)
  }
  if (tid == 0) {
    *s_prefix = 0;
    *s_need = K;  // rank from the top, 1-based: find key T with #(key > T) < K <= #(key >= T)
  }
  for (int pass = 0; pass < kPasses; ++pass) {
    const int shift = 8 * (kPasses - 1 - pass);
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const KT prefix = *s_prefix;
    const KT himask = pass == 0 ? (KT)0 : (KT)(~(KT)0 << (shift + 8));
    DigitRuns dr;
    for_each_key([&](int, KT key) {
      if ((key & himask) == prefix) dr.add(hist, (int)((unsigned)(key >> shift) & 255u));
    });
    dr.flush(hist);
    __syncthreads();
    if (tid < 32) {
      unsigned need = *s_need;
      const int bin = pick_from_top(hist, 256, need);
      if (tid == 0) {
        *s_need = need;
        *s_prefix = prefix | ((KT)bin << shift);
      }
    }
    __syncthreads();
  }
  const KT T = *s_prefix;
  const unsigned need_eq = *s_need;  // how many of the == T elements are taken (lowest ids first)
  // the last pass counted the keys equal to T in the bin of T's low digit (the histogram is still there)
  if (hist[(unsigned)T & 255u] == need_eq) {
    // every key equal to the threshold is taken: no order among them is needed
    for_each_key([&](int s, KT key) {
      if (key >= T) {
        const int slot = atomicAdd(s_cnt, 1);
        if (slot < kMaxTopK) s_ids[slot] = s;
      }
    });
    return;
  }
  // ties at the cut: contiguous id partition so that they are picked in id order
  const int per = (N + nt - 1) / nt;
  const int lo = min(N, tid * per), hi = min(N, lo + per);
  int eq = 0;
  for (int s = lo; s < hi; ++s) eq += KEY(s) == T;
  s_scan[tid] = eq;
  __syncthreads();
  if (tid < 32) warp0_exclusive_scan(s_scan, nt);
  __syncthreads();
  int eqrank = s_scan[tid];
  for (int s = lo; s < hi; ++s) {
    const KT key = KEY(s);
    bool take = key > T;
    if (key == T) {
      take = (unsigned)eqrank < need_eq;
      ++eqrank;
    }
    if (take) {
      const int slot = atomicAdd(s_cnt, 1);
      if (slot < kMaxTopK) s_ids[slot] = s;
    }
  }
}

// Host-memory pager (Sec. 3.4): which slot of the (sequence, layer, KV head)'s unit cache every named unit lives in.  Every
// slot's usage score decays, a unit named now gains 1; a missing unit takes the slot with the lowest score among the
// slots not named now (lowest slot among equals).  A unit that reaches beyond grow_end is still growing and is not
// cached.  s_src[t]: slot of named unit t, -1 = straight from the host; s_fill[t]: its rows have to be pulled first.
// Called by every thread of the CTA.
__device__ __forceinline__ void unit_cache_policy(const DevCtx& c, size_t unit, int g, const int* ids, int nall,
                                                  int grow_end, int* s_tag, float* s_sco, unsigned char* s_named,
                                                  int* s_src, int* s_fill) {
  const int tid = threadIdx.x, CU = c.cache_units, U = c.unit;
  const size_t cb = (unit * c.Hkv + g) * (size_t)CU;
  if (tid < CU) {
    s_tag[tid] = c.ctag[cb + tid];
    s_sco[tid] = __fmul_rn(c.cscore[cb + tid], c.score_decay);
    s_named[tid] = 0;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long hits = 0, misses = 0;
    auto growing = [&](int id) { return (long long)(id + 1) * U > grow_end; };
    for (int t = 0; t < nall; ++t) {  // first the units that are there, so that none of them is pushed out
      const int id = ids[t];
      s_src[t] = -1;
      s_fill[t] = 0;
      if (growing(id)) continue;
      for (int sl = 0; sl < CU; ++sl)
        if (s_tag[sl] == id) {
          s_src[t] = sl;
          s_named[sl] = 1;
          s_sco[sl] = __fadd_rn(s_sco[sl], 1.f);
          ++hits;
          break;
        }
    }
    for (int t = 0; t < nall; ++t) {
      const int id = ids[t];
      if (growing(id) || s_src[t] >= 0) continue;
      int victim = -1;
      for (int sl = 0; sl < CU; ++sl)
        if (!s_named[sl] && (victim < 0 || s_sco[sl] < s_sco[victim])) victim = sl;
      if (victim < 0) continue;  // (cannot happen: cache_units >= the units one retrieval names)
      s_tag[victim] = id;
      s_sco[victim] = 1.f;
      s_named[victim] = 1;
      s_src[t] = victim;
      s_fill[t] = 1;
      ++misses;
    }
    atomicAdd(&c.cstat[unit * 2], hits);
    atomicAdd(&c.cstat[unit * 2 + 1], misses);
  }
  __syncthreads();
  if (tid < CU) {
    c.ctag[cb + tid] = s_tag[tid];
    c.cscore[cb + tid] = s_sco[tid];
  }
}

// Decode: the rows [st, st + ln) of a missing unit go from the host mirror to the same row offsets of its cache slot.
__device__ __forceinline__ void pull_unit(const DevCtx& c, size_t unit, int g, int id, int slot, int st, int ln) {
  const size_t drow = ((unit * c.Hkv + g) * (size_t)c.cache_units + slot) * (size_t)c.unit + (st - id * c.unit);
  const size_t hrow = (unit * c.Hkv + g) * (size_t)c.Tpad + st;
  const uint4* hk = reinterpret_cast<const uint4*>(c.hostK + hrow * kD);
  const uint4* hv = reinterpret_cast<const uint4*>(c.hostV + hrow * kD);
  uint4* dk = reinterpret_cast<uint4*>(c.Kcache + drow * kD);
  uint4* dv = reinterpret_cast<uint4*>(c.Vcache + drow * kD);
  for (int i = threadIdx.x; i < ln * 16; i += blockDim.x) {
    dk[i] = hk[i];
    dv[i] = hv[i];
  }
}

// Token ranges of the attention kernels from M items (start, length) in ascending order of start: items of length
// zero are dropped, an item that starts at or before the end of what came before it (adjacent spans, or overlapping
// ones under NMS with phi > 0) extends the current range.  One warp, 32 items per round: an item opens a range iff it
// starts beyond the largest end seen so far (a prefix maximum), its range number is the count of such items up to
// it, and a range's end is the prefix maximum in front of the next opener.  Returns the number of ranges; s_rs / s_rl
// receive their starts and lengths.  Called by all 32 lanes of one warp.
template <typename ItemF>
__device__ __forceinline__ int merge_ranges_warp(int M, ItemF&& item, int* s_rs, int* s_rl) {
  const int lane = threadIdx.x & 31;
  constexpr int kNone = -0x7fffffff;
  int far = kNone, nr = 0;  // largest end so far, ranges so far
  for (int base = 0; base < M; base += 32) {
    const int i = base + lane;
    int st = 0, ln = 0;
    if (i < M) item(i, st, ln);
    const bool valid = i < M && ln > 0;
    const int en = valid ? st + ln : kNone;
    int inc = en;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc = max(inc, t);
    }
    int before = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) before = kNone;
    before = max(before, far);
    const bool opens = valid && st > before;
    const unsigned ob = __ballot_sync(0xffffffffu, opens);
    if (opens) {
      const int idx = nr + __popc(ob & ((2u << lane) - 1u)) - 1;
      s_rs[idx] = st;
      if (idx > 0) s_rl[idx - 1] = before;  // (the end of the range before it; turned into a length below)
    }
    far = max(far, __shfl_sync(0xffffffffu, inc, 31));
    nr += __popc(ob);
  }
  if (lane == 0 && nr > 0) s_rl[nr - 1] = far;
  __syncwarp();
  for (int r = lane; r < nr; r += 32) s_rl[r] -= s_rs[r];
  __syncwarp();
  return nr;
}

// a0 inside the one-launch decode kernels: one CTA of (sequence, layer, KV head) also stores that head's new K and V row
// (threads 0-31: sixteen 16-byte pieces each; in a sliding slab the window row, and the sink's own row for a sink token), so a
// decode step needs no separate append launch.  Other CTAs of the same launch must not read the row from the slab: the
// retrievers leave it to the attention kernel launched next, the one-launch step takes it from the caller's tensors.
__device__ __forceinline__ void append_decode_row(const DevCtx& c, const DecBatch& b, int bi, int l, int layer_count,
                                                  size_t unit, int g, const __nv_bfloat16* __restrict__ k,
                                                  const __nv_bfloat16* __restrict__ v) {
  const int tid = threadIdx.x;
  if (tid < 32) {
    const int c16 = tid & 15, pos = b.pos[bi];
    const __nv_bfloat16* src = (tid < 16 ? k : v) + (((size_t)b.src[bi] * layer_count + l) * c.Hkv + g) * kD + c16 * 8;
    __nv_bfloat16* slab = (tid < 16 ? c.Kc : c.Vc) + (unit * c.Hkv + g) * (size_t)c.SR * kD + c16 * 8;
    const long long wrow = c.paged ? pos - b.shift[bi] : pos;
    if (wrow < 0 || wrow >= c.SR) {  // cannot happen: the host keeps the window inside the slab
      set_status(c, -2, pos);
    } else {
      const uint4 w = *reinterpret_cast<const uint4*>(src);
      *reinterpret_cast<uint4*>(slab + wrow * kD) = w;
      if (c.paged && pos < c.Ls) *reinterpret_cast<uint4*>(slab + (size_t)pos * kD) = w;  // the sink's permanent row
    }
    if (g == 0 && tid == 0) c.votes[unit * c.Tpad + pos] = 0;
  }
}

}  // namespace ltri
