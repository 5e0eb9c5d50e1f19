// State kernels: cache append, eviction + span index build (Sec. 3.3.1, Eq. 6), span segmenter
// (Eq. 4-5, App. "NMS Input Filtration"), query representatives, similarity scores (Eq. 7) and
// top-k selection (Eq. 8).  All segmentation arithmetic is integer and order-independent.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "mma_util.cuh"
#include "select_util.cuh"

namespace ltri {

// ------------------------------------------------------------------------------------------
__global__ void k_init(DevCtx c, int seq) {
  const int s0 = seq < 0 ? 0 : seq, s1 = seq < 0 ? c.NS : seq + 1;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int s = s0; s < s1; ++s) {
    const size_t u0 = (size_t)s * c.NL;
    for (size_t i = tid; i < (size_t)c.NL; i += stride) {
      c.n_spans[u0 + i] = 0;
    }
    for (size_t i = tid; i < (size_t)c.NL * c.Hkv; i += stride) c.sel_tokens[u0 * c.Hkv + i] = 0;
    for (size_t i = tid; i < (size_t)c.NL * c.slots; i += stride) c.pend_cnt[u0 * c.slots + i] = 0;
    for (size_t i = tid; i < (size_t)c.NL * c.Hkv * c.topk; i += stride) {
      c.sel[u0 * c.Hkv * c.topk + i] = -1;
      c.persist_sel[u0 * c.Hkv * c.topk + i] = -1;
    }
    for (size_t i = tid; i < (size_t)c.NL * c.Hkv; i += stride) c.rng_cnt[u0 * c.Hkv + i] = 0;
    for (size_t i = tid; i < (size_t)c.NL * c.topk; i += stride) c.ballot[u0 * c.topk + i] = -1;
    if (c.host_kv) {  // empty unit caches
      const size_t nslot = (size_t)c.NL * c.Hkv * c.cache_units;
      for (size_t i = tid; i < nslot; i += stride) {
        c.ctag[u0 * c.Hkv * c.cache_units + i] = -1;
        c.cscore[u0 * c.Hkv * c.cache_units + i] = 0.f;
      }
      for (size_t i = tid; i < (size_t)c.NL * 2; i += stride) c.cstat[u0 * 2 + i] = 0ull;
    }
  }
  if (seq < 0 && tid < 4) c.status[tid] = 0;
  if (seq < 0) {
    for (size_t i = tid; i < (size_t)c.NL; i += stride) c.Jcnt[i] = 0;
    for (size_t i = tid; i < ((size_t)c.NL * kSegPasses << kSegHistBits); i += stride) c.seg_hist[i] = 0u;
    for (size_t i = tid; i < (size_t)c.NL * 2 * c.chunk; i += stride) c.seg_best[i] = 0;
  }
}

cudaError_t launch_init(const DevCtx& c, int seq, cudaStream_t s) {
  k_init<<<64, 256, 0, s>>>(c, seq);
  return cudaGetLastError();
}


// ------------------------------------------------------------------------------------------
// a0: copy the call's K/V rows into the cache slabs; 16 threads move one 256-byte row.  The threads behind the copy
// (zero_vec of them, 16 bytes each) clear the region maps of the call's layers, which the tensor-core map pass
// accumulates into with integer reductions: nothing reads a layer's map between the segmenter of the layer's previous
// call and that pass, so clearing it here, in the first kernel of the call, keeps a memset out of the kernel chain.
__global__ void k_append_prefill(DevCtx c, PrefillArgs a, unsigned long long zero_vec) {
  chain_wait();
  const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int c16 = gid & 15;
  size_t row = gid >> 4;  // over [layer_count][n][Hkv]
  const size_t nrows = (size_t)a.layer_count * a.n * c.Hkv;
  if (row >= nrows) {
    const size_t zi = gid - nrows * 16;
    if (zi < zero_vec)
      reinterpret_cast<uint4*>(c.Mq + (size_t)a.layer_begin * c.chunk * c.chunk)[zi] = make_uint4(0u, 0u, 0u, 0u);
  } else {
    const int g = row % c.Hkv;
    const int r = (row / c.Hkv) % a.n;
    const int l = row / ((size_t)c.Hkv * a.n);
    const size_t unit = unit_of(c, a.seq, a.layer_begin + l);
    const long long tok = a.t0 + r;
    const long long wrow = c.paged ? tok - a.shift : tok;  // window row (a sink token has one too while it is current)
    if (wrow < 0 || wrow >= c.SR) {                         // cannot happen: the host keeps the window inside the slab
      set_status(c, -2, (int)tok);
    } else {
      const size_t dst = ((unit * c.Hkv + g) * c.SR + wrow) * kD + c16 * 8;
      const size_t src = row * kD + c16 * 8;
      const uint4 kv = *reinterpret_cast<const uint4*>(a.k + src), vv = *reinterpret_cast<const uint4*>(a.v + src);
      *reinterpret_cast<uint4*>(c.Kc + dst) = kv;
      *reinterpret_cast<uint4*>(c.Vc + dst) = vv;
      if (c.paged && tok < c.Ls) {  // the sink's permanent rows
        const size_t sd = ((unit * c.Hkv + g) * c.SR + tok) * kD + c16 * 8;
        *reinterpret_cast<uint4*>(c.Kc + sd) = kv;
        *reinterpret_cast<uint4*>(c.Vc + sd) = vv;
      }
      if (g == 0 && c16 == 0) c.votes[unit * c.Tpad + a.t0 + r] = 0;
    }
  }
}

cudaError_t launch_append_prefill(const DevCtx& c, const PrefillArgs& a, bool clear_maps, cudaStream_t s) {
  const unsigned long long zero_vec = clear_maps ? (unsigned long long)a.layer_count * c.chunk * c.chunk / 4 : 0ull;
  const size_t threads = (size_t)a.layer_count * a.n * c.Hkv * 16 + zero_vec;
  return launch_chained(k_append_prefill, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, s, c, a, zero_vec);
}

__global__ void k_append_decode(DevCtx c, DecBatch b, int layer_begin, int layer_count,
                                const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v) {
  chain_wait();
  const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int c16 = gid & 15;
  size_t row = gid >> 4;  // over [b.n][layer_count][Hkv]
  if (row >= (size_t)b.n * layer_count * c.Hkv) return;
  const int g = row % c.Hkv;
  const int l = (row / c.Hkv) % layer_count;
  const int bi = row / ((size_t)c.Hkv * layer_count);
  const size_t unit = unit_of(c, b.seq[bi], layer_begin + l);
  const long long tok = b.pos[bi];
  const long long wrow = c.paged ? tok - b.shift[bi] : tok;
  if (wrow < 0 || wrow >= c.SR) {  // cannot happen: the host keeps the window inside the slab
    set_status(c, -2, (int)tok);
    return;
  }
  const size_t dst = ((unit * c.Hkv + g) * c.SR + wrow) * kD + c16 * 8;
  const size_t src = (((size_t)b.src[bi] * layer_count + l) * c.Hkv + g) * kD + c16 * 8;
  const uint4 kv = *reinterpret_cast<const uint4*>(k + src), vv = *reinterpret_cast<const uint4*>(v + src);
  *reinterpret_cast<uint4*>(c.Kc + dst) = kv;
  *reinterpret_cast<uint4*>(c.Vc + dst) = vv;
  if (c.paged && tok < c.Ls) {  // the sink's permanent rows
    const size_t sd = ((unit * c.Hkv + g) * c.SR + tok) * kD + c16 * 8;
    *reinterpret_cast<uint4*>(c.Kc + sd) = kv;
    *reinterpret_cast<uint4*>(c.Vc + sd) = vv;
  }
  if (g == 0 && c16 == 0) {
    c.votes[unit * c.Tpad + b.pos[bi]] = 0;
  }
}

cudaError_t launch_append_decode(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count, int,
                                 const __nv_bfloat16* k, const __nv_bfloat16* v, cudaStream_t s) {
  const size_t threads = (size_t)b.n * layer_count * c.Hkv * 16;
  return launch_chained(k_append_decode, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, s, c, b, layer_begin,
                        layer_count, k, v);
}

// ------------------------------------------------------------------------------------------
// a1: regions that left the window: every span gets its index vector, the bf16 sum of the keys of
// its most voted token(s), and is appended to the span table.  Eight CTAs of eight warps (a cluster, so that the span
// count is moved on only when all have read it) share a layer, one warp per span, four key rows in flight per warp.
// Bound: latency (votes -> token -> key rows); with one CTA of 32 warps per layer, two or three rounds of it: 12 us for
// one region of 512 tokens, 18 us of 1024.
constexpr int kEvictCluster = 8;
__global__ void __cluster_dims__(kEvictCluster, 1, 1) __launch_bounds__(256) k_evict_index(DevCtx c, EvictArgs a) {
  chain_wait();
  if (a.release) chain_release();
  const int layer = a.layer_begin + blockIdx.x / kEvictCluster, part = blockIdx.x % kEvictCluster;
  const size_t unit = unit_of(c, a.seq, layer);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = (blockDim.x >> 5) * kEvictCluster;
  const int base = c.n_spans[unit];
  const long long* votes = c.votes + unit * c.Tpad;
  int off = 0;
  for (int si = 0; si < a.nslots; ++si) {
    const size_t ps = (unit * c.slots + a.slot[si]) * c.Jmax;
    const int cnt = c.pend_cnt[unit * c.slots + a.slot[si]];
    for (int i = part + kEvictCluster * warp; i < cnt; i += nwarps) {
      const int start = c.pend_start[ps + i], len = c.pend_len[ps + i];
      const int dst = base + off + i;
      if (dst >= c.cap) {
        if (lane == 0) set_status(c, -2, dst);
        continue;
      }
      if (lane == 0) {
        c.span_start[unit * c.cap + dst] = start;
        c.span_len[unit * c.cap + dst] = len;
      }
      int toks[kMaxReps];
      const int nrep = select_reps(votes, start, len, c.rep_mode == 1 ? c.pend_nrep[ps + i] : c.reps, toks);
      for (int g0 = 0; g0 < c.Hkv; g0 += 4) {
        float acc[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = acc[u][2] = acc[u][3] = 0.f;
        for (int r = 0; r < nrep; ++r) {
          const size_t row = (size_t)slab_row(c, toks[r], a.shift) * kD + lane * 4;
          uint2 raw[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            raw[u] = g0 + u < c.Hkv
                         ? *reinterpret_cast<const uint2*>(c.Kc + ((unit * c.Hkv + g0 + u) * c.SR) * kD + row)
                         : make_uint2(0u, 0u);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const __nv_bfloat162 p0 = *reinterpret_cast<const __nv_bfloat162*>(&raw[u].x);
            const __nv_bfloat162 p1 = *reinterpret_cast<const __nv_bfloat162*>(&raw[u].y);
            acc[u][0] += __bfloat162float(p0.x);
            acc[u][1] += __bfloat162float(p0.y);
            acc[u][2] += __bfloat162float(p1.x);
            acc[u][3] += __bfloat162float(p1.y);
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (g0 + u >= c.Hkv) continue;
          __nv_bfloat162 o0 = __floats2bfloat162_rn(acc[u][0], acc[u][1]);
          __nv_bfloat162 o1 = __floats2bfloat162_rn(acc[u][2], acc[u][3]);
          uint2 w;
          w.x = *reinterpret_cast<uint32_t*>(&o0);
          w.y = *reinterpret_cast<uint32_t*>(&o1);
          *reinterpret_cast<uint2*>(c.KR + ((unit * c.Hkv + g0 + u) * c.cap + dst) * kD + lane * 4) = w;
        }
      }
    }
    off += cnt;
  }
  cooperative_groups::this_cluster().sync();
  if (part == 0 && threadIdx.x == 0) c.n_spans[unit] = min(base + off, c.cap);
}

cudaError_t launch_evict_index(const DevCtx& c, const EvictArgs& a, int layer_count, cudaStream_t s) {
  return launch_chained(k_evict_index, dim3(layer_count * kEvictCluster), dim3(256), 0, s, c, a);
}

// ------------------------------------------------------------------------------------------
// a3 segmenter, step 1: exact rank selection of theta (quantile mode) over the causal entries of Mq.
// Pass 1 counts negatives (only hand-built maps have any) and zeros (a sparse map is mostly zeros) and builds a
// log-scale histogram of the positive entries: bin = (position of the leading one, next four bits), which is monotone
// in the value and spreads a heavy-tailed map over many bins.  If the rank falls among the positives, the remaining
// low bits of the selected bin are resolved by MSB radix passes of 9 bits.  One histogram per few warps, four loads
// in flight per lane; a thread-block cluster of eight CTAs shares a layer: each counts its share of the rows, then
// every CTA adds up the eight histograms through distributed shared memory and takes the same decision.
constexpr int kThetaBits = 9;
constexpr int kThetaBins = 1 << kThetaBits;

// visits the causal entries of the m x m map: f(value) for every (i, j <= i).  The rows are dealt to the warps of the
// `nparts` CTAs that share a map in pairs (i, m-1-i), so every warp sees about the same number of entries.
template <typename F>
__device__ __forceinline__ void for_each_causal(const int* __restrict__ Mq, int ld, int m, int part, int nparts, F&& f) {
  const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int gw = part * nwarps + (threadIdx.x >> 5), step = nparts * nwarps;
  for (int idx = gw; 2 * idx < m; idx += step) {
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
      const int i = side == 0 ? idx : m - 1 - idx;
      if (side == 1 && i == idx) break;
      const int* row = Mq + (size_t)i * ld;
      for (int j0 = 0; j0 <= i; j0 += 128) {
        int v[4];
        bool ok[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = j0 + u * 32 + lane;
          ok[u] = j <= i;
          v[u] = ok[u] ? row[j] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ok[u]) f(v[u]);
      }
    }
  }
}

// monotone log-scale bin of a positive value: 16 bins per power of two
__device__ __forceinline__ unsigned log_bin(unsigned v) {
  const int e = 31 - __clz(v);
  const unsigned frac = e >= 4 ? (v >> (e - 4)) & 15u : (v << (4 - e)) & 15u;
  return ((unsigned)e << 4) | frac;
}

// rank of theta among the causal entries of a layer's map under its own quantile level: the same double arithmetic as on
// the host
__device__ __forceinline__ long long layer_rank(const DevCtx& c, int layer, int m) {
  const long long N = (long long)m * (m + 1) / 2;
  const long long rank = (long long)floor((double)c.theta_l[layer] * (double)(N - 1));
  return rank < 0 ? 0 : (rank > N - 1 ? N - 1 : rank);
}
// absolute threshold of a layer under its own theta
__device__ __forceinline__ long long layer_theta_q(const DevCtx& c, int layer, bool one_head) {
  return (long long)rint((double)c.theta_l[layer] * (one_head ? 1.0 : (double)c.Hq) * (double)kQScale);
}

constexpr int kThetaThreads = 512;


__global__ void __launch_bounds__(kThetaThreads)
    k_theta_select(DevCtx c, int layer_begin, int m, long long rank, int tables) {
  chain_wait();
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ unsigned hist[];  // [warps][kThetaBins]
  const int CL = (int)cluster.num_blocks(), NW = blockDim.x >> 5;
  const int layer = layer_begin + blockIdx.x / CL;
  const int part = (int)cluster.block_rank();
  if (tables && c.theta_l) rank = layer_rank(c, layer, m);
  const int* Mq = c.Mq + (size_t)layer * c.chunk * c.chunk;
  // this CTA's histogram, then its counts of negatives and zeros: two copies that the passes use in turn, so that one
  // cluster barrier per pass is enough
  __shared__ unsigned loc[2][kThetaBins + 2];
  __shared__ unsigned tot[kThetaBins];  // the cluster's histogram (every CTA builds its own copy)
  __shared__ unsigned s_red[32][2];
  __shared__ unsigned s_prefix, s_lo_bits;
  __shared__ long long s_rank, s_cn, s_cz;
  __shared__ int s_cls;  // 0: answer found, 1: among positives (bin chosen), -1: among negatives
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned* myhist = hist + warp * kThetaBins;
  auto visit = [&](auto&& f) { for_each_causal(Mq, c.chunk, m, part, CL, f); };
  int pass = 0;
  // sums the per-warp histograms into loc, then the cluster's loc arrays into tot
  auto combine = [&](bool with_counts) {
    unsigned* mine = loc[pass & 1];
    __syncthreads();
    if (threadIdx.x < kThetaBins) {
      unsigned sum = 0;
#pragma unroll 8
      for (int w = 0; w < NW; ++w) sum += hist[w * kThetaBins + threadIdx.x];
      mine[threadIdx.x] = sum;
    }
    if (with_counts && threadIdx.x < 2) {
      unsigned n = 0;
      for (int w = 0; w < NW; ++w) n += s_red[w][threadIdx.x];
      mine[kThetaBins + threadIdx.x] = n;
    }
    cluster.sync();
    if (threadIdx.x < kThetaBins) {
      unsigned sum = 0;
#pragma unroll 8
      for (int r = 0; r < CL; ++r) sum += cluster.map_shared_rank(mine, r)[threadIdx.x];
      tot[threadIdx.x] = sum;
    }
    if (with_counts && threadIdx.x < 2) {
      long long n = 0;
#pragma unroll 8
      for (int r = 0; r < CL; ++r) n += cluster.map_shared_rank(mine, r)[kThetaBins + threadIdx.x];
      if (threadIdx.x == 0)
        s_cn = n;
      else
        s_cz = n;
    }
    ++pass;
    __syncthreads();
  };
  for (int t = threadIdx.x; t < NW * kThetaBins; t += blockDim.x) hist[t] = 0;
  __syncthreads();
  unsigned nneg = 0, nzero = 0;
  visit([&](int v) {
    if (v > 0)
      atomicAdd(&myhist[log_bin((unsigned)v)], 1u);
    else if (v == 0)
      ++nzero;
    else
      ++nneg;
  });
  nneg = __reduce_add_sync(0xffffffffu, nneg);
  nzero = __reduce_add_sync(0xffffffffu, nzero);
  if (lane == 0) {
    s_red[warp][0] = nneg;
    s_red[warp][1] = nzero;
  }
  combine(true);
  if (threadIdx.x < 32) {
    const long long cn = s_cn, cz = s_cz;
    if (rank < cn) {
      if (lane == 0) {
        s_cls = -1;
        s_rank = rank;
      }
    } else if (rank < cn + cz) {
      if (lane == 0) {
        s_cls = 0;
        if (part == 0) c.thetaq[layer] = 0;
      }
    } else {
      long long r = rank - cn - cz;
      const unsigned b = pick_from_bottom(tot, kThetaBins, r);
      const int e = (int)(b >> 4);
      const unsigned frac = b & 15u;
      if (lane == 0) {
        s_rank = r;
        if (e <= 4) {  // the bin holds a single value
          s_cls = 0;
          if (part == 0) c.thetaq[layer] = (long long)((1u << e) | (frac >> (4 - e)));
        } else {
          s_cls = 1;
          s_prefix = (1u << e) | (frac << (e - 4));  // leading one and the next four bits
          s_lo_bits = (unsigned)(e - 4);             // bits still unknown
        }
      }
    }
  }
  __syncthreads();
  const int cls = s_cls;
  // remaining bits: [0, hi).  Negatives: plain MSB radix over the sign-flipped key.
  int hi = cls > 0 ? (int)s_lo_bits : (cls < 0 ? 31 : 0);
  if (cls < 0 && threadIdx.x == 0) s_prefix = 0;
  __syncthreads();
  while (hi > 0) {  // (the same decisions in every CTA of the cluster)
    const int lo = max(0, hi - kThetaBits);
    const unsigned dmask = (1u << (hi - lo)) - 1u;
    for (int t = threadIdx.x; t < NW * kThetaBins; t += blockDim.x) hist[t] = 0;
    __syncthreads();
    const unsigned prefix = s_prefix;
    visit([&](int v) {
      const bool in_cls = cls > 0 ? v > 0 : v < 0;
      const unsigned key = cls > 0 ? (unsigned)v : ((unsigned)v ^ 0x80000000u);
      if (in_cls && (key >> hi) == (prefix >> hi)) atomicAdd(&myhist[(key >> lo) & dmask], 1u);
    });
    combine(false);
    if (threadIdx.x < 32) {
      long long r = s_rank;
      unsigned b = pick_from_bottom(tot, kThetaBins, r);  // bins above dmask are empty
      if (b > dmask) b = dmask;
      if (threadIdx.x == 0) {
        s_rank = r;
        s_prefix = prefix | (b << lo);
      }
    }
    __syncthreads();
    hi = lo;
  }
  if (cls != 0 && threadIdx.x == 0 && part == 0)
    c.thetaq[layer] = cls > 0 ? (long long)s_prefix : (long long)(int)(s_prefix ^ 0x80000000u);
  cluster.sync();  // nobody leaves while its histogram may still be read
}

// rank of theta among the m (m + 1) / 2 causal entries
static long long quantile_rank(float theta, int m) {
  const long long N = (long long)m * (m + 1) / 2;
  const long long rank = (long long)floor((double)theta * (double)(N - 1));
  return rank < 0 ? 0 : (rank > N - 1 ? N - 1 : rank);
}

// absolute threshold: thq in units of the map summed over all heads, thq1 in units of a single (retrieval) head's map;
// with per-layer tables the layer's own theta, scaled here
__global__ void k_theta_set(DevCtx c, int layer_begin, long long thq, long long thq1, int tables) {
  chain_wait();
  const int layer = layer_begin + blockIdx.x;
  const bool one = ret_head_of(c, layer) >= 0;
  long long t = one ? thq1 : thq;
  if (tables && c.theta_l) t = layer_theta_q(c, layer, one);
  c.thetaq[layer] = t;
}

// step 2: suffix sums along each row of D = Mq - theta ("sum the right elements", Fig. 2):
// Rsuf[i][x] = sum_{j=x..i} D[i][j].  One warp per row.  A lane holds four consecutive entries of every block of 128, all
// of them requested before the first is used (one load at a time, a row of 1024 was 32 dependent round trips: 24 us for
// one layer's map); B = blocks of 128 in a row.
template <int B>
__global__ void __launch_bounds__(256) k_seg_rowscan(DevCtx c, int layer_begin, int m) {
  chain_wait();
  const int layer = layer_begin + blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + warp;
  if (blockIdx.x == 0)
    for (int t = threadIdx.x; t < 2 * c.chunk; t += blockDim.x) c.best[(size_t)layer * 2 * c.chunk + t] = 0;
  if (i >= m) return;
  const int* row = c.Mq + ((size_t)layer * c.chunk + i) * c.chunk;
  long long* out = c.Rsuf + ((size_t)layer * c.chunk + i) * c.chunk;
  // 16-byte accesses need rows that start on 16 bytes and whose groups of four never leave them: always so in a context
  // (chunk is a multiple of 16), not for a caller's dense map of any size and alignment
  const bool vec = (c.chunk & 3) == 0 && (reinterpret_cast<uintptr_t>(c.Mq) & 15) == 0;
  int4 v[B];
#pragma unroll
  for (int k = 0; k < B; ++k) {
    const int x = k * 128 + lane * 4;
    v[k] = make_int4(0, 0, 0, 0);
    if (vec) {
      if (x <= i) v[k] = *reinterpret_cast<const int4*>(row + x);
    } else {
      if (x <= i) v[k].x = row[x];
      if (x + 1 <= i) v[k].y = row[x + 1];
      if (x + 2 <= i) v[k].z = row[x + 2];
      if (x + 3 <= i) v[k].w = row[x + 3];
    }
  }
  const long long thq = c.thetaq[layer];
  long long carry = 0;
#pragma unroll
  for (int k = B - 1; k >= 0; --k) {
    if (k * 128 > i) continue;  // (uniform over the warp)
    const int x = k * 128 + lane * 4;
    long long s3 = x + 3 <= i ? (long long)v[k].w - thq : 0;
    long long s2 = s3 + (x + 2 <= i ? (long long)v[k].z - thq : 0);
    long long s1 = s2 + (x + 1 <= i ? (long long)v[k].y - thq : 0);
    long long s0 = s1 + (x <= i ? (long long)v[k].x - thq : 0);
    long long inc = s0;  // sum over this lane's entries and those of the lanes to its right
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_down_sync(0xffffffffu, inc, o);
      if (lane + o < 32) inc += t;
    }
    const long long right = carry + inc - s0;
    if (vec) {
      if (x <= i) {
        *reinterpret_cast<longlong2*>(out + x) = make_longlong2(right + s0, right + s1);
        *reinterpret_cast<longlong2*>(out + x + 2) = make_longlong2(right + s2, right + s3);
      }
    } else {
      if (x <= i) out[x] = right + s0;
      if (x + 1 <= i) out[x + 1] = right + s1;
      if (x + 2 <= i) out[x + 2] = right + s2;
      if (x + 3 <= i) out[x + 3] = right + s3;
    }
    carry += __shfl_sync(0xffffffffu, inc, 0);
  }
}

// step 3: prefix sums down each column ("sum the upper elements"): S(x,y) = sum_{i=x..y} Rsuf[i][x], and the
// best point of every anti-diagonal x+y=c (max S, ties -> shorter span), kept only when S > 0.
// A CTA owns CX columns; thread (cx, ry) scans a group of at most 16 rows of its column, whose entries it keeps in
// registers, a scan over the row groups supplies the offsets, and a second pass emits S.
// key = (S << 10) | (1023 - (y-x)).  CX = 32 for regions of up to 512 tokens (32 row groups), 16 for longer ones (64).
// seg_unit > 0 (segmentation per memory unit): only intervals inside one unit of seg_unit tokens on the absolute grid
// are candidates; `origin` is the absolute position of the region's first token.
template <int CX>
__global__ void __launch_bounds__(1024) k_seg_colscan(DevCtx c, int layer_begin, int m, int seg_unit, int origin) {
  chain_wait();
  constexpr int RY = 1024 / CX, K = RY / 32;
  extern __shared__ long long sm[];
  long long* part = sm;                  // [RY][CX + 1]
  long long* sbest = sm + RY * (CX + 1); // [m + CX]
  const int layer = layer_begin + blockIdx.y;
  const int cx = threadIdx.x % CX, ry = threadIdx.x / CX;
  const int x0 = blockIdx.x * CX, x = x0 + cx;
  const int R = (m + RY - 1) / RY;
  const long long* Rs = c.Rsuf + (size_t)layer * c.chunk * c.chunk;
  const int ylo = ry * R, yhi = min(m, ylo + R);
  long long cv[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int y = ylo + k;
    cv[k] = (x < m && y >= x && y < yhi) ? Rs[(size_t)y * c.chunk + x] : 0;
  }
  for (int t = threadIdx.x; t < m + CX; t += blockDim.x) sbest[t] = 0;
  long long acc = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) acc += cv[k];
  part[ry * (CX + 1) + cx] = acc;
  __syncthreads();
  // exclusive scan over the row groups, a warp per column, K groups per lane
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid < CX) {
    long long v[K], inc = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      v[k] = part[(lane * K + k) * (CX + 1) + wid];
      inc += v[k];
    }
    const long long own = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    long long run = inc - own;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      part[(lane * K + k) * (CX + 1) + wid] = run;
      run += v[k];
    }
  }
  __syncthreads();
  if (x < m) {
    long long S = part[ry * (CX + 1) + cx];
    // last token of the unit that holds x (region-relative)
    const int ymax = seg_unit > 0 ? ((origin + x) / seg_unit + 1) * seg_unit - origin - 1 : m;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int y = ylo + k;
      if (y < x || y >= yhi) continue;
      S += cv[k];
      if (S > 0 && y <= ymax) {
        const long long key = (S << 10) | (long long)(1023 - (y - x));
        atomicMax(&sbest[x + y - 2 * x0], key);
      }
    }
  }
  __syncthreads();
  long long* gbest = c.best + (size_t)layer * 2 * c.chunk;
  for (int t = threadIdx.x; t < m + CX; t += blockDim.x) {
    const long long key = sbest[t];
    const int cd = 2 * x0 + t;
    if (key > 0 && cd <= 2 * m - 2) atomicMax(&gbest[cd], key);
  }
}

// step 4: the <= 2m-1 candidates in the order (S desc, length asc, start asc), greedy non-maximum suppression with
// IoU threshold 0 until max_spans are kept, gap fill, store the region's spans in its pending slot; then the
// query representatives of every span (Sec. 3.4 step 2): u[g][j] = sum_{h in g} sum_{rep tokens} q_h[tok].
// NMS on the squares (x, x, y+1, y+1): a candidate is suppressed by a kept span when their IoU exceeds phi_milli/1000;
// two spans that share `inter` tokens have IoU = inter^2 / (L1^2 + L2^2 - inter^2).  Integer arithmetic; phi = 0
// means any overlap suppresses.
__device__ __forceinline__ bool nms_suppressed(int x, int y, int kx, int ky, int phi_milli) {
  const int inter = min(y, ky) - max(x, kx) + 1;
  if (inter <= 0 || phi_milli == 0) return inter > 0;
  // lengths of at most 1024: every product fits 32 bits (in 64 bits the test was most of a round's instructions)
  const unsigned l1 = y - x + 1, l2 = ky - kx + 1, i2 = (unsigned)inter * (unsigned)inter;
  return i2 * 1000u > (unsigned)phi_milli * (l1 * l1 + l2 * l2 - i2);
}

struct NmsArgs {
  int seq, layer_begin, m, reg_start, slot, max_spans;
  int n, t0;                 // query tensor geometry (q == nullptr: skip the representatives)
  const __nv_bfloat16* q;
  int tables;                // use the context's per-layer phi and lambda tables where it has them
  int seg_unit;              // > 0: every unit of this many tokens (absolute grid) keeps max_spans spans of its own
};

// Steps 4 and the representatives, by all CTAs of a cluster (CL of them, this one is `part`): the first CTA runs the NMS
// and the gap fill, then the spans are dealt to all of them for the representatives.  gbest: the candidates; votes: the
// votes of token t at votes[t], for the region's tokens.
__device__ __forceinline__ void spans_and_reps(const DevCtx& c, const NmsArgs& a, cooperative_groups::cluster_group& cluster,
                                               int CL, int part, int lidx, const long long* gbest, const long long* votes) {
  __shared__ long long skey[768];  // scratch of the query representatives: token lists and counts per span
  __shared__ int kx[kMaxTopK], ky[kMaxTopK], ox[kMaxTopK], oy[kMaxTopK];  // kept spans, as found and by start
  __shared__ int out_start[2 * kMaxTopK + 1], out_len[2 * kMaxTopK + 1];
  __shared__ int s_nout;
  __shared__ int s_ucnt[kMaxTopK + 2];  // segmentation per unit: spans kept in every unit the region touches
  const int layer = a.layer_begin + lidx;
  const size_t unit = unit_of(c, a.seq, layer);
  const int m = a.m;
  const int SU = a.seg_unit;
  auto unit_idx = [&](int x) { return (a.reg_start + x) / SU - a.reg_start / SU; };
  const int cap_total = SU > 0 ? kMaxTopK : a.max_spans;
  const int phi_milli = a.tables && c.phi_l ? c.phi_l[layer] : c.phi_milli;
  const float rep_lambda = a.tables && c.lambda_l ? c.lambda_l[layer] : c.rep_lambda;
  const int ncand = 2 * m - 1;
  // Greedy NMS without a sort: the candidate the sorted sweep would reach next is the best one that is still alive
  // (key larger, or equal key and smaller anti-diagonal), so every round takes the block-wide maximum over the alive
  // candidates, keeps it, and lets every thread strike out its own candidates that the new span suppresses (or whose
  // unit is full).  At most max_spans rounds instead of sorting up to 2047 keys.
  // Candidate of anti-diagonal cd: key = (S << 10) | (1023 - len) > 0; x = (cd - len) / 2, y = x + len.
  // The rounds run in the first 8 warps, one barrier each (three where units fill up): the warps' best meet in one of two arrays
  // that the rounds use in turn.  A key is held as its upper 32 significant bits (of the largest key) and the rest, so that one
  // warp-wide maximum nearly always names the winner.  (Bound: latency of the chain suppress - warp maximum - barrier - maximum.  With three
  // warp-wide reductions per maximum and a branch per candidate a round took 1300 cycles, now 750.)
  constexpr int NT = 256, NW = NT / 32;
  __shared__ uint4 s_wbest[2][NW];
  __shared__ int s_kept;
  __shared__ unsigned s_bits;  // bits of the largest key
  const int tid = threadIdx.x, wlane = tid & 31, wid = tid >> 5;
  if (SU > 0)
    for (int t = tid; t < kMaxTopK + 2; t += blockDim.x) s_ucnt[t] = 0;
  if (tid == 0) s_bits = 0u;
  __syncthreads();
  if (part == 0 && tid < NT) {
    auto round_barrier = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };
    // CU candidates per thread: tid, tid + NT, ...
    auto rounds = [&](auto cu_tag, auto plain_tag) {
      constexpr int CU = decltype(cu_tag)::value;
      constexpr bool PLAIN = decltype(plain_tag)::value;  // any overlap suppresses, no limit per unit
      unsigned khi[CU], klo[CU], bits = 0u;
      int cx[CU], cy[CU];
      {
        long long key[CU];
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          const int cd = tid + u * NT;
          key[u] = cd < ncand ? max(__ldcg(gbest + cd), 0ll) : 0;  // (0: not alive)
          const int len = 1023 - (int)(key[u] & 1023);
          cx[u] = (cd - len) >> 1;
          cy[u] = cx[u] + len;
          bits = max(bits, 64u - (unsigned)__clzll(key[u]));
        }
        bits = __reduce_max_sync(0xffffffffu, bits);
        if (wlane == 0) atomicMax(&s_bits, bits);
        round_barrier();
        const unsigned sh = max(s_bits, 32u) - 32u;
#pragma unroll
        for (int u = 0; u < CU; ++u) {
          khi[u] = (unsigned)(key[u] >> sh);
          klo[u] = (unsigned)key[u] & ((1u << sh) - 1u);
        }
      }
      const unsigned sh = max(s_bits, 32u) - 32u;
      // the lane that holds the warp-wide best of (hi, lo) descending, then cd ascending
      auto winner = [&](unsigned hi, unsigned lo, int cd) {
        const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
        unsigned at = __ballot_sync(0xffffffffu, hi == mh);
        if (at & (at - 1u)) {
          const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
          const int mc = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? cd : 0x7fffffff);
          at = __ballot_sync(0xffffffffu, hi == mh && lo == ml && cd == mc);
        }
        return __ffs(at) - 1;
      };
      int kept = 0;
      while (kept < cap_total) {
        unsigned bh = khi[0], bl = klo[0];
        int bc = tid;
#pragma unroll
        for (int u = 1; u < CU; ++u) {
          const bool more = khi[u] > bh || (khi[u] == bh && klo[u] > bl);  // (ascending: an equal one does not replace)
          bh = more ? khi[u] : bh;
          bl = more ? klo[u] : bl;
          bc = more ? tid + u * NT : bc;
        }
        uint4* buf = s_wbest[kept & 1];
        if (wlane == winner(bh, bl, bc)) buf[wid] = make_uint4(bh, bl, (unsigned)bc, 0u);
        round_barrier();
        uint4 w = wlane < NW ? buf[wlane] : make_uint4(0u, 0u, 0x7fffffffu, 0u);
        w = buf[winner(w.x, w.y, (int)w.z) & (NW - 1)];  // (nothing alive: any of the empty entries)
        if ((w.x | w.y) == 0u) break;  // nothing alive is left (the same decision in every thread)
        const int wl = 1023 - (int)(((w.x << sh) | w.y) & 1023u);
        const int wx = ((int)w.z - wl) >> 1, wy = wx + wl;
        if (tid == 0) {
          kx[kept] = wx;
          ky[kept] = wy;
          if (!PLAIN && SU > 0) ++s_ucnt[unit_idx(wx)];
        }
        ++kept;
        if (PLAIN) {
#pragma unroll
          for (int u = 0; u < CU; ++u) {
            const bool apart = cy[u] < wx || cx[u] > wy;
            khi[u] = apart ? khi[u] : 0u;
            klo[u] = apart ? klo[u] : 0u;
          }
        } else {
          if (SU > 0) round_barrier();  // the unit counts are up to date
#pragma unroll
          for (int u = 0; u < CU; ++u)
            if ((khi[u] | klo[u]) != 0u &&
                (tid + u * NT == (int)w.z || nms_suppressed(cx[u], cy[u], wx, wy, phi_milli) ||
                 (SU > 0 && s_ucnt[unit_idx(cx[u])] >= a.max_spans)))
              khi[u] = klo[u] = 0u;
          if (SU > 0) round_barrier();  // (everybody has read them)
        }
      }
      if (tid == 0) s_kept = kept;
    };
    using four = std::integral_constant<int, 4>;
    using eight = std::integral_constant<int, 8>;
    const bool plain = SU == 0 && phi_milli == 0, few = ncand <= 4 * NT;
    if (plain && few)
      rounds(four(), std::true_type());
    else if (plain)
      rounds(eight(), std::true_type());
    else if (few)
      rounds(four(), std::false_type());
    else
      rounds(eight(), std::false_type());
  }
  __syncthreads();
  // order the kept spans by start, a warp per span; with phi > 0 two of them may share their start: then the shorter first
  if (part == 0)
    for (int w = wid; w < s_kept; w += blockDim.x >> 5) {
      const int x = kx[w], y = ky[w];
      int rank = 0;
#pragma unroll
      for (int b = 0; b < kMaxTopK; b += 32) {
        const int q = b + wlane;
        rank += __popc(__ballot_sync(0xffffffffu, q < s_kept && (kx[q] < x || (kx[q] == x && ky[q] < y))));
      }
      if (wlane == 0) {
        ox[rank] = x;
        oy[rank] = y;
      }
    }
  __syncthreads();
  if (part == 0 && threadIdx.x < 32) {
    const int lane = threadIdx.x, kept = s_kept;
    if (SU == 0) {
      // two entries per lane: the end of everything covered in front of a span (a prefix maximum: with phi > 0 kept spans
      // may overlap) tells whether an uncovered run precedes it, the number of such runs where it goes
      int covered = 0, no = 0;
      for (int base = 0; base < kept; base += 32) {
        const int q = base + lane;
        const int sx = q < kept ? ox[q] : 0x7fffffff, sy = q < kept ? oy[q] + 1 : 0;
        int inc = sy;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc = max(inc, t);
        }
        int before = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) before = 0;
        before = max(before, covered);
        const unsigned gaps = __ballot_sync(0xffffffffu, q < kept && sx > before);
        const int at = no + lane + __popc(gaps & ((2u << lane) - 1u));
        if (q < kept) {
          if (sx > before) {
            out_start[at - 1] = before;
            out_len[at - 1] = sx - before;
          }
          out_start[at] = sx;
          out_len[at] = sy - sx;
        }
        covered = max(covered, __shfl_sync(0xffffffffu, inc, 31));
        no += min(32, kept - base) + __popc(gaps);
      }
      if (lane == 0) {
        if (covered < m) {
          out_start[no] = covered;
          out_len[no++] = m - covered;
        }
        s_nout = no;
      }
    } else if (lane == 0) {
      int pos = 0, no = 0;
      // an uncovered run [g0, g1) becomes a span; under segmentation per unit it is cut at the unit boundaries
      auto emit_gap = [&](int g0, int g1) {
        while (g0 < g1 && no < 2 * kMaxTopK + 1) {
          const int e = SU > 0 ? min(g1, ((a.reg_start + g0) / SU + 1) * SU - a.reg_start) : g1;
          out_start[no] = g0;
          out_len[no++] = e - g0;
          g0 = e;
        }
      };
      for (int q = 0; q < kept; ++q) {
        if (ox[q] > pos) emit_gap(pos, ox[q]);
        if (no < 2 * kMaxTopK + 1) {
          out_start[no] = ox[q];
          out_len[no++] = oy[q] - ox[q] + 1;
        }
        pos = max(pos, oy[q] + 1);  // kept spans may overlap when phi > 0
      }
      if (pos < m) emit_gap(pos, m);
      s_nout = no;
    }
  }
  __syncthreads();
  if (CL > 1) {  // pushed to the others, not fetched by them: one barrier and no round trip
    if (part == 0) {
      const int n = min(s_nout, 2 * kMaxTopK + 1);
      for (int t = tid; t < (n + 1) * CL; t += blockDim.x) {
        const int r = t % CL, i = t / CL;
        if (i == n) {
          if (r > 0) *cluster.map_shared_rank(&s_nout, r) = s_nout;
        } else if (r > 0) {
          cluster.map_shared_rank(out_start, r)[i] = out_start[i];
          cluster.map_shared_rank(out_len, r)[i] = out_len[i];
        }
      }
    }
    cluster.sync();  // (from here on a CTA reads its own shared memory only)
  }
  const int nout = s_nout;
  const size_t ps = (unit * c.slots + a.slot) * c.Jmax;
  if (nout > c.Jmax) {
    if (threadIdx.x == 0) set_status(c, -5, nout);
    return;
  }
  if (part == 0)
    for (int t = threadIdx.x; t < nout; t += blockDim.x) {
      c.pend_start[ps + t] = a.reg_start + out_start[t];
      c.pend_len[ps + t] = out_len[t];
    }
  if (part == 0 && threadIdx.x == 0) {
    c.pend_cnt[unit * c.slots + a.slot] = nout;
    c.Jcnt[layer] = a.q ? nout : 0;
  }
  // query representatives.  First one warp per span picks the representative tokens, then one warp per
  // (span, KV head) sums their query rows with all loads of the head group in flight at once.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const __nv_bfloat16* q = a.q + (size_t)lidx * a.n * c.Hq * kD;
  int* rep_tok = reinterpret_cast<int*>(skey);          // [Jmax][kMaxReps]
  int* rep_cnt = rep_tok + (2 * kMaxTopK + 1) * kMaxReps;
  __syncthreads();
  // representative count of every span: static, or from the area ratio of Sec. 3.3.2 on the raw region map.  The
  // row-suffix table holds sums of (Mq - theta), so a raw sum over w entries is the table value + theta * w.
  int* nrep_of = rep_cnt + (2 * kMaxTopK + 1);
  // (the spans part, part + CL, ... are this CTA's)
  for (int j = part + CL * warp; j < nout; j += CL * nwarps) {
    int cnt = min(c.reps, out_len[j]);
    if (c.rep_mode == 1) {
      const long long* Rs = c.Rsuf + (size_t)layer * c.chunk * c.chunk;
      const long long th = c.thetaq[layer];
      const int x = out_start[j], y = x + out_len[j] - 1;
      long long T = 0, TR = 0, Cn = 0;
      for (int i = x + lane; i <= y; i += 32) {
        T += Rs[(size_t)i * c.chunk + x] + th * (i - x + 1);
        TR += Rs[(size_t)i * c.chunk] + th * (i + 1);
      }
      for (int i = y + 1 + lane; i < m; i += 32)
        Cn += Rs[(size_t)i * c.chunk + x] - Rs[(size_t)i * c.chunk + y + 1] + th * (y - x + 1);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        T += shfl_xor_ll(T, o);
        TR += shfl_xor_ll(TR, o);
        Cn += shfl_xor_ll(Cn, o);
      }
      const long long R = TR - T;
      const long long nb = c.ratio_kind == 0 ? R : c.ratio_kind == 1 ? Cn : R + Cn;
      const double ra = (T + nb) > 0 ? (double)T / (double)(T + nb) : 1.0;
      const double rv = 1.0 / exp((double)rep_lambda * (1.0 - ra));
      cnt = (int)rint((double)out_len[j] * rv);  // to nearest even
      cnt = max(cnt, c.min_reps);
      cnt = min(cnt, c.max_reps);
      cnt = min(cnt, out_len[j]);
      cnt = max(cnt, 1);
    }
    if (lane == 0) {
      nrep_of[j] = cnt;
      if (c.pend_nrep) c.pend_nrep[ps + j] = cnt;  // (absent in the scratch-only context of the static entry)
      if (c.nrep_last) c.nrep_last[(size_t)layer * c.Jmax + j] = cnt;
    }
  }
  __syncthreads();
  if (!a.q) return;
  for (int j = part + CL * warp; j < nout; j += CL * nwarps) {
    int toks[kMaxReps];
    const int nrep = select_reps(votes, a.reg_start + out_start[j], out_len[j], nrep_of[j], toks);
    if (lane == 0) {
      rep_cnt[j] = nrep;
      for (int r = 0; r < nrep; ++r) rep_tok[j * kMaxReps + r] = toks[r];
    }
  }
  __syncthreads();
  // a half-warp per (span, KV head): sixteen lanes x eight dimensions; the rows of the heads of the group are all in
  // flight before they are added up, per head over the representative tokens (ascending) and then over the heads in
  // ascending order
  const int hw = lane >> 4, hl = lane & 15;
  const int rh = ret_head_of(c, layer);
  const int nmine = nout > part ? (nout - part + CL - 1) / CL : 0;
  for (int task = 2 * warp + hw; task < nmine * c.Hkv; task += 2 * nwarps) {
    const int j = part + CL * (task / c.Hkv), g = task % c.Hkv;
    const int nrep = rep_cnt[j];
    const __nv_bfloat16* qg = q + (size_t)g * c.G * kD + hl * 8;
    // a layer with a retrieval head (Sec. 3.5) has one representative per span, that head's: the other heads add zero
    auto counts = [&](int hh) { return hh < c.G && (rh < 0 || g * c.G + hh == rh); };
    auto add8 = [](float (&acc)[8], const uint4& w) {
      const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&w);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(p2[i]);
        acc[2 * i] += f.x;
        acc[2 * i + 1] += f.y;
      }
    };
    float ug[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) ug[e] = 0.f;
    if (nrep == 1) {
      // (four heads at a time, added as they are: a short loop body, because a kernel that runs once per call fetches
      // every instruction line from L2 and spends more time on that than on the rows)
      const __nv_bfloat16* row = qg + (size_t)(rep_tok[j * kMaxReps] - a.t0) * c.Hq * kD;
#pragma unroll 1
      for (int h0 = 0; h0 < c.G; h0 += 4) {
        uint4 raw[4];
#pragma unroll
        for (int hh = 0; hh < 4; ++hh)
          raw[hh] = counts(h0 + hh) ? *reinterpret_cast<const uint4*>(row + (size_t)(h0 + hh) * kD) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int hh = 0; hh < 4; ++hh) add8(ug, raw[hh]);
      }
    } else {
      for (int hh = 0; hh < c.G; ++hh) {
        if (!counts(hh)) continue;
        uint4 raw[kMaxReps];
#pragma unroll
        for (int r = 0; r < kMaxReps; ++r)
          raw[r] = r < nrep ? *reinterpret_cast<const uint4*>(qg + ((size_t)(rep_tok[j * kMaxReps + r] - a.t0) * c.Hq + hh) * kD)
                            : make_uint4(0u, 0u, 0u, 0u);
        float one[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) one[e] = 0.f;
#pragma unroll
        for (int r = 0; r < kMaxReps; ++r)
          if (r < nrep) add8(one, raw[r]);
#pragma unroll
        for (int e = 0; e < 8; ++e) ug[e] += one[e];
      }
    }
    float* up = c.u + (((size_t)layer * c.Hkv + g) * c.Jmax + j) * kD + hl * 8;
    *reinterpret_cast<float4*>(up) = make_float4(ug[0], ug[1], ug[2], ug[3]);
    *reinterpret_cast<float4*>(up + 4) = make_float4(ug[4], ug[5], ug[6], ug[7]);
  }
}

// A cluster of CTAs may share a layer (its launch says how many).
__global__ void __launch_bounds__(1024) k_seg_nms(DevCtx c, NmsArgs a) {
  chain_wait();
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int CL = (int)cluster.num_blocks(), lidx = blockIdx.x / CL, layer = a.layer_begin + lidx;
  if (CL > 1) cluster.sync();  // (every CTA runs before the first store to another)
  spans_and_reps(c, a, cluster, CL, (int)cluster.block_rank(), lidx, c.best + (size_t)layer * 2 * c.chunk,
                 c.votes + unit_of(c, a.seq, layer) * c.Tpad);
}

// The segmenter of a few layers in one launch: threshold, both cumulative sums, candidates, NMS and representatives.  A
// cluster of 16 CTAs shares a layer's m x m map: CTA p holds the row blocks p and 31 - p of 32 (33 column blocks whatever
// p is) and keeps the raw row suffix sums RS[i][x] = sum_{j=x..i} Mq[i][j] in shared memory.  With T(x,y) the sum of RS
// over the rows x..y of column x, the score of Fig. 2 is S(x,y) = T(x,y) - theta * len (len + 1) / 2, so the map is read
// once, and the column sums of the 32 row blocks and the histograms of the entries cross the cluster behind one barrier.
// Both go through L2: gathered from the other CTAs' shared memory, 64 KB a CTA, they took 8K cycles each time.
// Bound: latency, a dozen dependent steps.  As four launches, with the map and a 64-bit table of sums going through L2 between
// them, a layer took 36 us (256 tokens), 45 (512) and 66 (1024); now 20, 30 and 55.
// The map's entries are not negative and a row's sum over all heads is at most Hq * kRowSumQ, so RS fits 32 bits; PT, the
// type of a block's column sums (at most 32 rows), is 32 bits up to 64 heads.
constexpr int kSegThreads = 1024, kSegCluster = kSegSms, kSegBlocks = 2 * kSegCluster;
constexpr int kSegFrac = 7;                         // the first histogram has 2^7 bins per power of two,
constexpr int kSegBits = kSegHistBits;              // the others resolve 12 bits a pass
constexpr int kSegBins = 1 << kSegBits;             // (four per thread)
constexpr int kSegRowVec = 1024 / 128;              // 128-entry groups of the longest row
static_assert(kSegBins == 4 * kSegThreads, "four bins per thread");

struct SegArgs {
  NmsArgs nms;
  int theta_mode;         // 1: quantile (of rank `rank`), otherwise the threshold is given
  int bh;                 // rows of a block: m / 32, rounded up
  int release;            // lets the kernel launched behind this one start at once
  long long rank, thq, thq1;
};

// monotone log-scale bin of a positive value: exponent and first bits of its fp32 form (rounded towards zero)
__device__ __forceinline__ unsigned seg_bin(unsigned v) {
  return (__float_as_uint(__uint2float_rz(v)) >> (23 - kSegFrac)) - (127u << kSegFrac);
}

__host__ __device__ inline int seg_stride(int blocks, int bh) { return (blocks * bh + 3) & ~3; }
// dynamic shared memory: histogram | T above each half of the two blocks, per column | candidates [2m + 1] | votes [m] (8 bytes
// each) | row sums
__host__ __device__ inline size_t seg_rows_at(int m, int bh) {
  return kSegBins * 4 + (((size_t)2 * (kSegBlocks + 1) * bh + 3 * m + 2) & ~(size_t)1) * 8;
}
static size_t seg_smem(int m, int bh) {  // (two row strides, each rounded up by at most three words)
  return seg_rows_at(m, bh) + (size_t)bh * ((kSegBlocks + 1) * bh + 6) * sizeof(unsigned);
}

template <typename PT>
__global__ void __launch_bounds__(kSegThreads, 1) k_segment(DevCtx c, SegArgs a) {
  chain_wait();
  if (a.release) chain_release();
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int part = (int)cluster.block_rank(), lidx = blockIdx.x / kSegCluster, layer = a.nms.layer_begin + lidx;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NW = kSegThreads / 32;
  const int m = a.nms.m, BH = a.bh;
  const size_t unit = unit_of(c, a.nms.seq, layer);
  // blocks A = part and B = 31 - part: columns (up to the block's last row), row strides of the sums
  const int bA = part, bB = kSegBlocks - 1 - part;
  const int nA = (bA + 1) * BH, nB = (bB + 1) * BH, ldA = seg_stride(bA + 1, BH), ldB = seg_stride(bB + 1, BH);
  extern __shared__ __align__(16) unsigned char dyn[];
  unsigned* hist = reinterpret_cast<unsigned*>(dyn);                    // [kSegBins]
  long long* above = reinterpret_cast<long long*>(hist + kSegBins);     // [2][nA + nB]: first half, second half of the rows
  long long* sbest = above + 2 * (kSegBlocks + 1) * BH;                 // [2m - 1]
  long long* svotes = sbest + (2 * m + 1);                              // [m]
  unsigned* RS = reinterpret_cast<unsigned*>(dyn + seg_rows_at(m, BH));  // A's rows, then B's
  __shared__ unsigned s_wsum[NW], s_bin;
  __shared__ long long s_rank;
  // what the cluster adds up: histograms [pass][bin] and candidates; clear at the start, left clear at the end
  unsigned* ghist = c.seg_hist + (size_t)layer * kSegPasses * kSegBins;
  long long* gbest = c.seg_best + (size_t)layer * 2 * c.chunk;
  PT* gsum = reinterpret_cast<PT*>(c.Rsuf + (size_t)layer * c.chunk * c.chunk);  // [block][m] column sums of the blocks
  const int* Mq = c.Mq + (size_t)layer * c.chunk * c.chunk;
  const long long* votes = c.votes + unit * c.Tpad + a.nms.reg_start;
  const bool quant = a.theta_mode == 1;

  reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (a.nms.q)  // (on their way until the representatives are chosen)
    for (int t = tid; t < m; t += kSegThreads) cp_async8(smem_u32(svotes + t), votes + t);
  cp_async_commit();
  for (int t = tid; t < 2 * m - 1; t += kSegThreads) sbest[t] = 0;
  __syncthreads();

  // ---- the rows: histogram of the entries, suffix sums.  A warp per row; a lane holds four consecutive entries of every
  // group of 128, all of them requested before the first is used.
  const int bh2 = 2 * BH;
  auto row_of = [&](int lr) { return lr < BH ? bA * BH + lr : bB * BH + lr - BH; };
  auto sums_of = [&](int lr) { return lr < BH ? RS + lr * ldA : RS + BH * ldA + (lr - BH) * ldB; };
#pragma unroll 1
  for (int lr = warp; lr < bh2; lr += NW) {
    const int i = row_of(lr), ld = lr < BH ? ldA : ldB;
    const int last = i < m ? i : -1;  // (rows behind the map: zeros)
    const int* row = Mq + (size_t)i * c.chunk;
    unsigned* rs = sums_of(lr);
    int4 v[kSegRowVec];
#pragma unroll
    for (int k = 0; k < kSegRowVec; ++k) {
      const int x = k * 128 + lane * 4;
      v[k] = x <= last ? *reinterpret_cast<const int4*>(row + x) : make_int4(0, 0, 0, 0);
    }
    unsigned carry = 0;
#pragma unroll
    for (int k = kSegRowVec - 1; k >= 0; --k) {
      if (k * 128 >= ld) continue;  // (uniform over the warp)
      const int x = k * 128 + lane * 4;
      const unsigned e0 = (unsigned)v[k].x, e1 = x + 1 <= last ? (unsigned)v[k].y : 0u,
                     e2 = x + 2 <= last ? (unsigned)v[k].z : 0u, e3 = x + 3 <= last ? (unsigned)v[k].w : 0u;
      const unsigned s3 = e3, s2 = s3 + e2, s1 = s2 + e1, s0 = s1 + e0;
      unsigned inc = s0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_down_sync(0xffffffffu, inc, o);
        if (lane + o < 32) inc += t;
      }
      const unsigned right = carry + inc - s0;
      if (x < ld) *reinterpret_cast<uint4*>(rs + x) = make_uint4(right + s0, right + s1, right + s2, right + s3);
      carry += __shfl_sync(0xffffffffu, inc, 0);
      if (quant) {
        if (e0 != 0u) atomicAdd(&hist[seg_bin(e0)], 1u);
        if (e1 != 0u) atomicAdd(&hist[seg_bin(e1)], 1u);
        if (e2 != 0u) atomicAdd(&hist[seg_bin(e2)], 1u);
        if (e3 != 0u) atomicAdd(&hist[seg_bin(e3)], 1u);
      }
    }
  }
  __syncthreads();
  // adds this CTA's histogram to the cluster's
  auto flush = [&](int pass) {
    const uint4 h = reinterpret_cast<const uint4*>(hist)[tid];
    unsigned* g = ghist + pass * kSegBins + tid * 4;
    if (h.x) atomicAdd(g, h.x);
    if (h.y) atomicAdd(g + 1, h.y);
    if (h.z) atomicAdd(g + 2, h.z);
    if (h.w) atomicAdd(g + 3, h.w);
  };
  if (quant) flush(0);
  // ---- column sums of the two blocks; the sum over the first half of a block's rows stays here
  const int hb = (BH + 1) >> 1;
  for (int t = tid; t < nA + nB; t += kSegThreads) {
    const bool inA = t < nA;
    const int ld = inA ? ldA : ldB, x = inA ? t : t - nA, b = inA ? bA : bB;
    const unsigned* col = inA ? RS + x : RS + BH * ldA + x;
    PT sum = 0;
#pragma unroll 8
    for (int y = 0; y < hb; ++y) sum += col[y * ld];
    above[nA + nB + t] = (long long)sum;
#pragma unroll 8
    for (int y = hb; y < BH; ++y) sum += col[y * ld];
    if (x < m && b * BH < m) gsum[(size_t)b * m + x] = sum;
  }
  cluster.sync();

  // ---- what the cluster knows: the histogram, and the column sums of the row blocks above this CTA's
  // the bin of the cluster's histogram in which rank `rank` falls (-1: among the zeros), and its rank inside it, to every thread
  auto pick = [&](int pass, long long rank) {
    const uint4 h = __ldcg(reinterpret_cast<const uint4*>(ghist + pass * kSegBins) + tid);
    const unsigned own = h.x + h.y + h.z + h.w;
    unsigned inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    if (lane == 31) s_wsum[warp] = inc;
    __syncthreads();
    const unsigned w = s_wsum[lane];
    if (pass == 0) rank -= (long long)m * (m + 1) / 2 - __reduce_add_sync(0xffffffffu, w);  // the zeros are not counted
    inc += __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
    const long long at = rank - (long long)(inc - own);  // rank counted from this thread's first bin
    if (at >= 0 && at < (long long)own) {
      const unsigned r = (unsigned)at, c1 = h.x, c2 = c1 + h.y, c3 = c2 + h.z;
      s_bin = tid * 4 + (r >= c1) + (r >= c2) + (r >= c3);
      s_rank = r - (r >= c3 ? c3 : r >= c2 ? c2 : r >= c1 ? c1 : 0u);
    }
    if (rank < 0 && tid == 0) s_bin = 0xffffffffu;
    __syncthreads();
  };
  long long thq = a.thq;
  unsigned prefix = 0;
  int hi = 0;  // bits of theta still unknown
  if (quant) {
    pick(0, a.nms.tables && c.theta_l ? layer_rank(c, layer, m) : a.rank);
    const unsigned bin = s_bin;  // (the same in every CTA)
    if (bin == 0xffffffffu) {
      thq = 0;
    } else {
      const int e = (int)(bin >> kSegFrac);
      const unsigned frac = bin & ((1u << kSegFrac) - 1u);
      if (e <= kSegFrac) {  // the bin holds a single value
        thq = (long long)((1u << e) | (frac >> (kSegFrac - e)));
      } else {
        hi = e - kSegFrac;
        prefix = (1u << e) | (frac << hi);  // the leading one and the bits behind it
      }
    }
  } else {
    const bool one = ret_head_of(c, layer) >= 0;
    if (one) thq = a.thq1;
    if (a.nms.tables && c.theta_l) thq = layer_theta_q(c, layer, one);
  }
  // T(x, y) of the row above a block: the sums of the blocks from column x's own down to it
  for (int t = tid; t < nA + nB; t += kSegThreads) {
    const bool inA = t < nA;
    const int x = inA ? t : t - nA, b = inA ? bA : bB;
    long long sum = 0;
    const int q0 = x / BH, n = x < m ? min(b, (m + BH - 1) / BH) - q0 : 0;  // (sixteen in flight)
    const PT* from = gsum + (size_t)q0 * m + x;
#pragma unroll 1
    for (int q = 0; q < n; q += 16, from += (size_t)16 * m)
#pragma unroll
      for (int i = 0; i < 16; ++i) sum += q + i < n ? __ldcg(from + (size_t)i * m) : (PT)0;
    above[t] = sum;
    above[nA + nB + t] += sum;
  }
  // ---- theta: the low bits over the entries that share the bits found so far
  for (int pass = 1; hi > 0; ++pass) {  // (the same decisions in every CTA of the cluster)
    const int lo = max(0, hi - kSegBits);
    const unsigned dmask = (1u << (hi - lo)) - 1u;
    const long long left = s_rank;
    reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
#pragma unroll 1
    for (int lr = warp; lr < bh2; lr += NW) {
      const int ld = lr < BH ? ldA : ldB;
      const unsigned* rs = sums_of(lr);
#pragma unroll 4
      for (int x = lane * 4; x - lane * 4 < ld; x += 128) {
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (x < ld) r = *reinterpret_cast<const uint4*>(rs + x);
        unsigned next = __shfl_down_sync(0xffffffffu, r.x, 1);
        if (lane == 31) next = x + 4 < ld ? rs[x + 4] : 0u;
        auto count = [&](unsigned val) {
          if ((val >> hi) == (prefix >> hi)) atomicAdd(&hist[(val >> lo) & dmask], 1u);
        };
        count(r.x - r.y);
        count(r.y - r.z);
        count(r.z - r.w);
        count(r.w - next);
      }
    }
    __syncthreads();
    flush(pass);
    cluster.sync();
    pick(pass, left);
    prefix |= s_bin << lo;
    hi = lo;
    thq = (long long)prefix;
  }
  __syncthreads();
  if (part == 0 && tid == 0) c.thetaq[layer] = thq;
  if (c.rep_mode == 1) {  // the table that the area ratios are read from (see k_seg_rowscan), over the blocks' column sums
    cluster.sync();
    for (int lr = warp; lr < bh2; lr += NW) {
      const int i = row_of(lr);
      if (i >= m) continue;
      long long* out = c.Rsuf + ((size_t)layer * c.chunk + i) * c.chunk;
      for (int x = lane; x <= i; x += 32) out[x] = (long long)sums_of(lr)[x] - thq * (i - x + 1);
    }
  }
  // ---- S(x, y) and the best point of every anti-diagonal (see k_seg_colscan).  A warp takes 32 columns of half a block, a
  // column per lane, row by row; the best of an anti-diagonal moves one lane down with every row, so that only what leaves
  // the warp takes an atomic (64-bit maxima in shared memory are loops).  Bound: issue slots, some 25 instructions an entry.
  const int SU = a.nms.seg_unit;
  const int gA = (nA + 31) >> 5, gB = (nB + 31) >> 5;
#pragma unroll 1
  for (int w = warp; w < 2 * (gA + gB); w += NW) {
    const int half = w & 1, grp = w >> 1;
    const bool inA = grp < gA;
    const int x0 = (inA ? grp : grp - gA) * 32, x = x0 + lane, n = inA ? nA : nB, ld = inA ? ldA : ldB;
    const int yb = (inA ? bA : bB) * BH, y1 = min(min(m, yb + BH), half ? yb + BH : yb + hb);
    const bool col_ok = x < n;
    const int ymax = !col_ok ? -1 : SU > 0 ? ((a.nms.reg_start + x) / SU + 1) * SU - a.nms.reg_start - 1 : m;
    const unsigned* col = (inA ? RS : RS + BH * ldA) + min(x, n - 1);
    long long* out = reinterpret_cast<long long*>(hist) + warp * 16;  // what leaves the warp, a row's at a time
    long long best = 0;
    const int y0 = max(half ? yb + hb : yb, x0);  // (above the diagonal of the first column there is nothing)
    if (y0 >= y1) continue;
    // S = D + the half block's own rows, D = T above the half block - theta * len (len + 1) / 2 from row to row (the recurrence
    // holds for len <= 0 too); the own rows above the diagonal are zeros
    const int len0 = y0 - x + 1;
    long long step = thq * len0;
    long long D = (col_ok ? above[(half ? nA + nB : 0) + (inA ? x : nA + x)] : 0) - ((thq * len0 * (len0 - 1)) >> 1);
    PT own = 0;
    unsigned low = (unsigned)(1024 - len0);
#pragma unroll 2
    for (int y = y0; y < y1; ++y) {
      own += col[(y - yb) * ld];
      D -= step;
      step += thq;
      const long long S = D + (long long)own;
      if (y >= x && y <= ymax && S > 0) best = max(best, (S << 10) | (long long)low);
      --low;
      if (lane == 0) out[y - y0] = best;
      best = __shfl_down_sync(0xffffffffu, best, 1);
      if (lane == 31) best = 0;
    }
    __syncwarp();
    const long long left = lane < y1 - y0 ? out[lane] : 0;  // what left the warp after row y0 + lane
    __syncwarp();
    // (lane l now holds the anti-diagonal of column x + 1 in the last row)
    auto give = [&](long long key, int cd) {
      if (key > 0 && key > *reinterpret_cast<volatile long long*>(&sbest[cd])) atomicMax(&sbest[cd], key);
    };
    give(left, min(x0 + y0 + lane, 2 * m - 2));
    give(best, min(x + y1, 2 * m - 2));
  }
  __syncthreads();
  for (int t = tid; t < 2 * m - 1; t += kSegThreads) {
    const long long key = sbest[t];
    if (key > 0) atomicMax(&gbest[t], key);
  }
  cp_async_wait<0>();  // (this thread's votes; the barriers below order all of them)
  cluster.sync();
  if (part > 0)
    for (int t = (part - 1) * kSegThreads + tid; t < kSegPasses * kSegBins / 4; t += (kSegCluster - 1) * kSegThreads)
      reinterpret_cast<uint4*>(ghist)[t] = make_uint4(0u, 0u, 0u, 0u);
  spans_and_reps(c, a.nms, cluster, kSegCluster, part, lidx, gbest, svotes - a.nms.reg_start);
  if (part == 0)  // (read by this CTA only, before the barriers in there)
    for (int t = tid; t < 2 * m - 1; t += kSegThreads) gbest[t] = 0;
}

constexpr int kSegWideLayers = 7;    // most layers that get a cluster of 16 (as many run at once on a whole GPU)
constexpr int kSegShareLayers = 16;  // up to here four CTAs share a layer's representatives

static bool seg_wide_sums(const DevCtx& c) { return c.Hq > 64; }

int segment_wide_clusters(const DevCtx& c) {
  const int smem = (int)seg_smem(c.chunk, (c.chunk + kSegBlocks - 1) / kSegBlocks);
  return std::min(kSegWideLayers, seg_wide_sums(c) ? active_clusters(k_segment<unsigned long long>, kSegCluster, kSegThreads, smem)
                                                   : active_clusters(k_segment<unsigned>, kSegCluster, kSegThreads, smem));
}

// A cluster of 16 needs a GPC to itself, so seven run at once; more layers keep the GPU busy as separate launches.
bool segment_in_one(const DevCtx& c, int layer_count) { return layer_count <= c.seg_wide; }

cudaError_t launch_segment_in_one(const DevCtx& c, int seq, int layer_begin, int layer_count, int m, int reg_start, int slot,
                                  int theta_mode, float theta, long long theta_q_abs, int max_spans, int n, int t0,
                                  const __nv_bfloat16* q, bool release, cudaStream_t s, bool tables, int seg_unit) {
  SegArgs a;
  a.nms = NmsArgs{seq, layer_begin, m, reg_start, slot, max_spans, n, t0, q, tables ? 1 : 0, seg_unit};
  a.theta_mode = theta_mode;
  a.bh = (m + kSegBlocks - 1) / kSegBlocks;
  a.release = release ? 1 : 0;
  a.rank = quantile_rank(theta, m);
  a.thq = theta_q_abs;
  a.thq1 = (long long)nearbyint((double)theta * (double)kQScale);
  return launch_chained_cluster(seg_wide_sums(c) ? k_segment<unsigned long long> : k_segment<unsigned>,
                                dim3(layer_count * kSegCluster), dim3(kSegThreads), kSegCluster, seg_smem(m, a.bh), s, c, a);
}

cudaError_t launch_segment(const DevCtx& c, int seq, int layer_begin, int layer_count, int m, int reg_start,
                             int slot, int theta_mode, float theta, long long theta_q_abs, int max_spans, int n,
                             int t0, const __nv_bfloat16* q, cudaStream_t s, bool tables, int seg_unit) {
  cudaError_t e;
  if (theta_mode == 1) {
    const int hsmem = (kThetaThreads / 32) * kThetaBins * (int)sizeof(unsigned);
    e = launch_chained_cluster(k_theta_select, dim3(layer_count * 8), dim3(kThetaThreads), 8, hsmem, s, c, layer_begin, m,
                               quantile_rank(theta, m), tables ? 1 : 0);
  } else {
    e = launch_chained(k_theta_set, dim3(layer_count), dim3(1), 0, s, c, layer_begin, theta_q_abs,
                       (long long)nearbyint((double)theta * (double)kQScale), tables ? 1 : 0);
  }
  if (e != cudaSuccess) return e;
  e = launch_chained(m <= 256 ? k_seg_rowscan<2> : m <= 512 ? k_seg_rowscan<4> : k_seg_rowscan<8>,
                     dim3((m + 7) / 8, layer_count), dim3(256), 0, s, c, layer_begin, m);
  if (e != cudaSuccess) return e;
  const int cx = m <= 512 ? 32 : 16;  // columns per CTA; 1024 / cx row groups
  e = launch_chained(m <= 512 ? k_seg_colscan<32> : k_seg_colscan<16>, dim3((m + cx - 1) / cx, layer_count), dim3(1024),
                     (size_t)(1024 / cx * (cx + 1) + m + cx) * sizeof(long long), s, c, layer_begin, m, seg_unit, reg_start);
  if (e != cudaSuccess) return e;
  NmsArgs a{seq, layer_begin, m, reg_start, slot, max_spans, n, t0, q, tables ? 1 : 0, seg_unit};
  const int cl = q && layer_count <= kSegShareLayers ? 4 : 1;
  return launch_chained_cluster(k_seg_nms, dim3(layer_count * cl), dim3(1024), cl, 0, s, c, a);
}

// ------------------------------------------------------------------------------------------
// a4 scores (Eq. 7 with summed representatives, max over the call's query spans):
// score[g][s] = max_j u[g][j] . K^R[g][s].  One warp per span, 4 dims per lane.
template <bool DECODE>
__global__ void __launch_bounds__(256) k_score(DevCtx c, int seq, int layer_begin, DecBatch b, int layer_count,
                                               const __nv_bfloat16* __restrict__ q) {
  extern __shared__ float su[];  // [J][128]
  int layer, sq, J;
  const int g = blockIdx.y;
  if (DECODE) {
    const int bi = blockIdx.z / layer_count;
    layer = layer_begin + blockIdx.z % layer_count;
    sq = b.seq[bi];
    J = 1;
    if (threadIdx.x < kD) {
      const __nv_bfloat16* qp =
          q + (((size_t)b.src[bi] * layer_count + (layer - layer_begin)) * c.Hq + g * c.G) * kD + threadIdx.x;
      float acc = 0.f;
      for (int hh = 0; hh < c.G; ++hh) acc += __bfloat162float(qp[(size_t)hh * kD]);
      su[threadIdx.x] = acc;
    }
  } else {
    layer = layer_begin + blockIdx.z;
    sq = seq;
    J = c.Jcnt[layer];
    const float* up = c.u + ((size_t)layer * c.Hkv + g) * c.Jmax * kD;
    for (int t = threadIdx.x; t < J * kD; t += blockDim.x) su[t] = up[t];
  }
  const size_t unit = unit_of(c, sq, layer);
  __syncthreads();
  const int N = c.n_spans[unit];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s0 = blockIdx.x * 64;
  const __nv_bfloat16* KR = c.KR + (unit * c.Hkv + g) * (size_t)c.cap * kD;
  float* sc = c.scores + (unit * c.Hkv + g) * (size_t)c.cap;
  for (int s = s0 + warp; s < min(s0 + 64, N); s += 8) {
    const uint2 raw = *reinterpret_cast<const uint2*>(KR + (size_t)s * kD + lane * 4);
    const __nv_bfloat162 p0 = *reinterpret_cast<const __nv_bfloat162*>(&raw.x);
    const __nv_bfloat162 p1 = *reinterpret_cast<const __nv_bfloat162*>(&raw.y);
    const float k0 = __bfloat162float(p0.x), k1 = __bfloat162float(p0.y), k2 = __bfloat162float(p1.x),
                k3 = __bfloat162float(p1.y);
    float best = -INFINITY;
    for (int j = 0; j < J; ++j) {
      const float4 uv = *reinterpret_cast<const float4*>(su + j * kD + lane * 4);
      float d = uv.x * k0;
      d = fmaf(uv.y, k1, d);
      d = fmaf(uv.z, k2, d);
      d = fmaf(uv.w, k3, d);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      best = fmaxf(best, d);
    }
    if (lane == 0) sc[s] = best;
  }
}

cudaError_t launch_score_prefill(const DevCtx& c, const PrefillArgs& a, int span_bound, cudaStream_t s) {
  DecBatch dummy;
  dummy.n = 0;
  const size_t smem = (size_t)c.Jmax * kD * sizeof(float);
  k_score<false><<<dim3((span_bound + 63) / 64, c.Hkv, a.layer_count), 256, smem, s>>>(c, a.seq, a.layer_begin, dummy,
                                                                                       a.layer_count, nullptr);
  return cudaGetLastError();
}

// decode scores, memory-bound index scan: one query representative per KV head (the summed query of the group).
// Half-warp per 256-byte index row, 16 bytes per lane, four rows in flight; grid (span tiles of 256, Hkv, units).
__global__ void __launch_bounds__(256) k_score_dec(DevCtx c, int layer_begin, DecBatch b, int layer_count,
                                                   const __nv_bfloat16* __restrict__ q) {
  chain_wait();
  __shared__ float su[kD];
  const int g = blockIdx.y;
  const int bi = blockIdx.z / layer_count, l = blockIdx.z % layer_count, layer = layer_begin + l;
  const size_t unit = unit_of(c, b.seq[bi], layer);
  const int tid = threadIdx.x;
  const int N = c.n_spans[unit];
  // a layer with a retrieval head (Sec. 3.5) scores that head's query against the index of its KV head, for every g
  const int rh = ret_head_of(c, layer), gk = rh >= 0 ? rh / c.G : g;
  const int s0 = blockIdx.x * 256;
  if (s0 >= N) return;
  if (tid < kD) {
    const __nv_bfloat16* qp = q + (((size_t)b.src[bi] * layer_count + l) * c.Hq + gk * c.G) * kD + tid;
    float acc = 0.f;
    for (int hh = 0; hh < c.G; ++hh)
      if (rh < 0 || gk * c.G + hh == rh) acc += __bfloat162float(qp[(size_t)hh * kD]);
    su[tid] = acc;
  }
  __syncthreads();
  const int hw = tid >> 4, hl = tid & 15;  // 16 half-warps
  float uf[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) uf[e] = su[hl * 8 + e];
  const __nv_bfloat16* KR = c.KR + (unit * c.Hkv + gk) * (size_t)c.cap * kD + hl * 8;
  float* sc = c.scores + (unit * c.Hkv + g) * (size_t)c.cap;
#pragma unroll
  for (int rep = 0; rep < 4; ++rep) {
    uint4 raw[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int s = s0 + rep * 64 + t * 16 + hw;
      raw[t] = s < N ? __ldg(reinterpret_cast<const uint4*>(KR + (size_t)s * kD)) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&raw[t]);
      float d = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(p2[i]);
        d = fmaf(uf[2 * i], f.x, d);
        d = fmaf(uf[2 * i + 1], f.y, d);
      }
      d += __shfl_xor_sync(0xffffffffu, d, 1);
      d += __shfl_xor_sync(0xffffffffu, d, 2);
      d += __shfl_xor_sync(0xffffffffu, d, 4);
      d += __shfl_xor_sync(0xffffffffu, d, 8);
      const int s = s0 + rep * 64 + t * 16 + hw;
      if (hl == 0 && s < N) sc[s] = d;
    }
  }
}

cudaError_t launch_score_decode(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count, int,
                                const __nv_bfloat16* q, int span_bound, cudaStream_t s) {
  if (span_bound <= 0) span_bound = 1;
  return launch_chained(k_score_dec, dim3((span_bound + 255) / 256, c.Hkv, b.n * layer_count), dim3(256), 0, s, c,
                        layer_begin, b, layer_count, q);
}

// ------------------------------------------------------------------------------------------
// a4 top-k (Eq. 8 with unit = span): the min(k, N_s) largest scores, ties -> lower span id.  4-pass radix select on
// order-preserving keys, then an id-ordered pick of the threshold ties.  Writes the ascending id list and the token
// ranges the attention kernels walk (adjacent spans merged).  One CTA per (unit, KV head).
// What a launch of k_topk does.  kTopkSelect: the selection, the token ranges and (prefill) the gather.  The other
// two are the collaborative voting of Sec. 3.5: kTopkBallot only records the own top-k units of every layer that has a
// retrieval head; kTopkVote then ranks a layer's units by the tally of the ballots of the layers up to it before
// their own scores and goes on like kTopkSelect.
enum { kTopkSelect = 0, kTopkBallot = 1, kTopkVote = 2 };
constexpr int kTopkSelRegs = 24;  // scores of up to 12K spans (512 threads) are read from global memory once

template <bool DECODE>
__global__ void __launch_bounds__(512) k_topk(DevCtx c, int seq, int layer_begin, DecBatch b, int layer_count,
                                              int evicted_end, int mode, int parts, int stage) {
  chain_wait();
  __shared__ unsigned hist[256];
  __shared__ unsigned s_prefix, s_need;
  __shared__ unsigned long long s_prefix64;
  __shared__ int s_ids[kMaxTopK];
  __shared__ int s_cnt;
  __shared__ int s_scan[512];
  __shared__ unsigned s_ckey[kSelCand];
  __shared__ int s_rs[kMaxRanges], s_rl[kMaxRanges], s_pre[kMaxRanges + 1], s_nr;  // merged ranges, packed-row prefix
  __shared__ int s_sst[2 * kMaxTopK], s_sln[2 * kMaxTopK];  // extents of the selected spans
  __shared__ int s_all[2 * kMaxTopK];            // decode: this step's selection united with the persistent one
  __shared__ int s_ko[kMaxRanges];  // pager, decode: first K row of every range, counted from the start of the K slabs
  // `parts` CTAs make the same selection for a (layer, KV head) and share the rows to be packed; the first one stores it
  const int g = blockIdx.x / parts, my_part = blockIdx.x % parts;
  int layer, sq, pos = 0, loc_begin = 0;
  if (DECODE) {
    const int bi = blockIdx.y / layer_count;
    layer = layer_begin + blockIdx.y % layer_count;
    sq = b.seq[bi];
    pos = b.pos[bi];
    loc_begin = b.loc_begin[bi];
  } else {
    layer = layer_begin + blockIdx.y;
    sq = seq;
  }
  // a layer with a retrieval head (Sec. 3.5) has one selection, made from the scores of that head's KV head
  const int rh = ret_head_of(c, layer);
  if (mode == kTopkBallot && (rh < 0 || g != 0)) return;
  const size_t unit = unit_of(c, sq, layer);
  const int nspans = c.n_spans[unit];
  const float* sc = c.scores + (unit * c.Hkv + (rh >= 0 ? rh / c.G : g)) * (size_t)c.cap;
  const int tid = threadIdx.x, nt = blockDim.x;
  // What is ranked: the spans themselves, or (Eq. 8 as printed) fixed units of c.unit tokens on the absolute token
  // grid, each scored by the maximum over the spans it meets.  N = number of candidates, KEY(i) = order key of
  // candidate i.
  extern __shared__ unsigned ukey[];  // unit mode: order key of every unit that meets the indexed range [Ls, E)
  const int U = c.unit;
  int N = nspans, u0 = 0, Eend = 0;
  if (U > 0) {
    Eend = nspans > 0 ? (DECODE ? loc_begin : evicted_end) : c.Ls;  // end of the indexed range
    u0 = c.Ls / U;
    N = Eend > c.Ls ? (Eend + U - 1) / U - u0 : 0;
    for (int i = tid; i < N; i += nt) ukey[i] = 0u;  // below the key of every real score
    __syncthreads();
    // (four spans a thread in flight)
    for (int base = tid; base < nspans; base += 4 * nt) {
      int st[4], ln[4];
      float v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int s = base + t * nt;
        st[t] = s < nspans ? c.span_start[unit * c.cap + s] : 0;
        ln[t] = s < nspans ? c.span_len[unit * c.cap + s] : 0;
        v[t] = s < nspans ? sc[s] : 0.f;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (base + t * nt < nspans)
          for (int u = st[t] / U; u <= (st[t] + ln[t] - 1) / U; ++u) atomicMax(&ukey[u - u0], order_key(v[t]));
    }
    __syncthreads();
  }
  // voting: tally of every unit = summed weights of the ballots that name it, layers in ascending order (fp32)
  float* utally = reinterpret_cast<float*>(ukey + ((N + 3) & ~3));
  if (mode == kTopkVote) {
    for (int i = tid; i < N; i += nt) utally[i] = 0.f;
    __syncthreads();
    for (int l = 0; l <= layer; ++l) {
      if (ret_head_of(c, l) < 0) continue;
      const float w = c.head_w[l];
      if (tid < c.topk) {
        const int id = c.ballot[unit_of(c, sq, l) * c.topk + tid];  // distinct within a ballot
        if (id >= u0 && id - u0 < N) utally[id - u0] += w;
      }
      __syncthreads();
    }
  }
  // the order keys are staged in shared memory where the launch left room for `stage` of them
  const bool staged = !DECODE && U == 0 && N <= stage;
  if (staged) {
    for (int base = tid; base < N; base += 16 * nt) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = base + u * nt < N ? sc[base + u * nt] : 0.f;
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (base + u * nt < N) ukey[base + u * nt] = order_key(v[u]);
    }
    __syncthreads();
  }
  auto KEY = [&](int i) -> unsigned { return U > 0 || staged ? ukey[i] : order_key(sc[i]); };
  auto KEY64 = [&](int i) -> unsigned long long {
    return ((unsigned long long)order_key(utally[i]) << 32) | ukey[i];
  };
  const int K = min(c.topk, N);
  if (tid == 0) s_cnt = 0;
  __syncthreads();
  if (K == N) {
    for (int t = tid; t < K; t += nt) s_ids[t] = t;
    if (tid == 0) s_cnt = K;
  } else if (mode == kTopkVote) {
    radix_select_top<unsigned long long, 0>(KEY64, N, K, hist, &s_prefix64, &s_need, s_scan, &s_cnt, s_ids);
  } else if (!DECODE && (staged || U > 0)) {
    radix_select_top<unsigned, 0>([&](int i) { return ukey[i]; }, N, K, hist, &s_prefix, &s_need, s_scan, &s_cnt, s_ids,
                                  s_ckey);
  } else {
    radix_select_top<unsigned, kTopkSelRegs>(KEY, N, K, hist, &s_prefix, &s_need, s_scan, &s_cnt, s_ids, s_ckey);
  }
  __syncthreads();
  const int cnt = min(s_cnt, K);
  // rank sort ascending
  int myid = -1, rank = 0;
  if (tid < cnt) {
    myid = s_ids[tid];
    for (int t = 0; t < cnt; ++t) rank += s_ids[t] < myid;
  }
  __syncthreads();
  if (tid < cnt) s_ids[rank] = myid;
  __syncthreads();
  if (U > 0 && tid < cnt) s_ids[tid] += u0;  // absolute unit ids
  __syncthreads();
  if (mode == kTopkBallot) {
    for (int t = tid; t < c.topk; t += nt) c.ballot[unit * c.topk + t] = t < cnt ? s_ids[t] : -1;
    return;
  }
  int* sel = c.sel + (unit * c.Hkv + g) * (size_t)c.topk;
  if (my_part == 0)
    for (int t = tid; t < c.topk; t += nt) sel[t] = t < cnt ? s_ids[t] : -1;
  // token ranges of the attention kernels: the spans' extents are fetched in parallel, merged (adjacent spans become
  // one range) by one thread in shared memory and written out in parallel
  const int* ids_all = s_ids;
  int nall = cnt;
  if (DECODE && c.persist) {
    nall = union_with_persistent(c, unit, g, s_ids, cnt, s_scan, s_all);
    ids_all = s_all;
  }
  if (tid < nall) {
    if (U > 0) {  // the unit's tokens inside the indexed range
      const int st = max(ids_all[tid] * U, c.Ls);
      s_sst[tid] = st;
      s_sln[tid] = min((ids_all[tid] + 1) * U, Eend) - st;
    } else {
      s_sst[tid] = c.span_start[unit * c.cap + ids_all[tid]];
      s_sln[tid] = c.span_len[unit * c.cap + ids_all[tid]];
    }
  }
  __syncthreads();
  // Host-memory pager (Sec. 3.4).  The units named by this retrieval are looked up in this (sequence, layer, KV
  // head)'s unit cache; every slot's usage score decays, a unit named now gains 1; a missing unit takes the slot with
  // the lowest score among the slots not named now (lowest slot among equals) and its rows are pulled from the host
  // mirror.  A prefill call caches only whole units: the unit the indexed range ends in, while it is still growing,
  // is read from the mirror every time.  (During decode the indexed range no longer grows, so that unit is cached
  // like the others.)  s_src[t]: slot of named unit t, -1 = straight from the host.
  __shared__ int s_tag[128], s_src[2 * kMaxTopK], s_fill[2 * kMaxTopK];
  __shared__ float s_sco[128];
  __shared__ unsigned char s_named[128];
  if (c.host_kv) {
    unit_cache_policy(c, unit, g, ids_all, nall, DECODE ? 0x7fffffff : Eend, s_tag, s_sco, s_named, s_src, s_fill);
    if (!DECODE) {
      // A prefill call leaves the data movement to k_pull_pack, which runs on a stream of its own while the kernels
      // of the call's other layers compute: this kernel only records what has to be brought in and from where.
      const size_t pb = (unit * c.Hkv + g) * (size_t)(2 * kMaxTopK);
      if (tid < nall) {
        c.pl_id[pb + tid] = ids_all[tid];
        c.pl_src[pb + tid] = s_src[tid] < 0 ? -1 : (s_src[tid] | (s_fill[tid] ? 0x10000 : 0));
        c.pl_start[pb + tid] = s_sst[tid];
        c.pl_len[pb + tid] = s_sln[tid];
      }
      if (tid == 0) c.pl_cnt[unit * c.Hkv + g] = nall;
    }
    if (DECODE) {
      // a decode step pulls its missing units here: the unit's valid rows [s_sst, s_sst + s_sln) go to the same row
      // offsets of its slot (the attention kernel, launched next, reads the slots in place)
      for (int t = 0; t < nall; ++t)
        if (s_fill[t]) pull_unit(c, unit, g, ids_all[t], s_src[t], s_sst[t], s_sln[t]);
    }
  }
  if (!(DECODE && c.host_kv)) {
    // (ranges in place, adjacent spans merged: one warp)
    if (tid < 32) {
      const int first = DECODE ? 1 : 0;  // decode: the sink in front of the spans, the recent tokens behind them
      const int rbeg = DECODE ? min(loc_begin, pos + 1) : 0;
      const int nr = merge_ranges_warp(
          nall + 2 * first,
          [&](int i, int& st, int& ln) {
            if (i < first) {
              st = 0;
              ln = min(c.Ls, pos + 1);
            } else if (i - first < nall) {
              st = s_sst[i - first];
              ln = s_sln[i - first];
            } else {
              st = rbeg;
              ln = pos + 1 - rbeg;
            }
          },
          s_rs, s_rl);
      long long tokens = 0;
      for (int t = tid; t < nall; t += 32) tokens += s_sln[t];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tokens += shfl_xor_ll(tokens, o);
      // packed-row prefix of the ranges
      int run = 0;
      for (int base = 0; base < nr; base += 32) {
        const int i = base + tid;
        const int v = i < nr ? s_rl[i] : 0;
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (tid >= o) inc += t;
        }
        if (i < nr) s_pre[i] = run + inc - v;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (tid == 0) {
        s_pre[nr] = run;
        s_nr = nr;
        if (my_part == 0) {
          c.rng_cnt[unit * c.Hkv + g] = nr;
          c.sel_tokens[unit * c.Hkv + g] = tokens;  // (summed over the KV heads by ltri_get_stats)
          if (!DECODE) c.gcnt[(size_t)layer * c.Hkv + g] = run;
        }
      }
    }
  } else
  if (tid == 0) {
    int nr = 0;
    long long tokens = 0;
    // under the pager a decode step reads every named unit from its cache slot, so the units stay ranges of their own
    // and every range carries the K row it starts at, counted from the start of the K slabs (the V row follows from it)
    const bool paged = DECODE && c.host_kv;
    const long long slab0 = (long long)((unit * c.Hkv + g) * (size_t)c.SR);
    auto push = [&](int st, int ln, int slot) {
      if (ln <= 0) return;
      if (!paged && nr > 0 && s_rs[nr - 1] + s_rl[nr - 1] >= st)  // adjacent, or (NMS with phi > 0) overlapping
        s_rl[nr - 1] = max(s_rl[nr - 1], st + ln - s_rs[nr - 1]);
      else {
        s_rs[nr] = st;
        s_rl[nr] = ln;
        if (paged) {
          if (slot >= 0) {
            const long long crow =
                (long long)(((unit * c.Hkv + g) * (size_t)c.cache_units + slot) * (size_t)U) + (st - (st / U) * U);
            s_ko[nr] = (int)((long long)((c.Kcache - c.Kc) / kD) + crow);
          } else {
            s_ko[nr] = (int)(slab0 + slab_row(c, st, DECODE ? b.shift[blockIdx.y / layer_count] : 0));
          }
        }
        ++nr;
      }
    };
    if (DECODE) push(0, min(c.Ls, pos + 1), -1);
    for (int t = 0; t < nall; ++t) {
      tokens += s_sln[t];
      push(s_sst[t], s_sln[t], paged ? s_src[t] : -1);
    }
    if (DECODE) push(min(loc_begin, pos + 1), pos + 1 - min(loc_begin, pos + 1), -1);
    int run = 0;
    for (int i = 0; i < nr; ++i) {
      s_pre[i] = run;
      run += s_rl[i];
    }
    s_pre[nr] = run;
    s_nr = nr;
    c.rng_cnt[unit * c.Hkv + g] = nr;
    c.sel_tokens[unit * c.Hkv + g] = tokens;  // (summed over the KV heads by ltri_get_stats)
    if (!DECODE) c.gcnt[(size_t)layer * c.Hkv + g] = run;
  }
  __syncthreads();
  if (my_part == 0) {
    const size_t rb = (unit * c.Hkv + g) * (size_t)c.rcap;
    for (int t = tid; t < s_nr; t += nt) {
      c.rng_start[rb + t] = s_rs[t];
      c.rng_len[rb + t] = s_rl[t];
      if (DECODE && c.host_kv) c.rng_koff[rb + t] = s_ko[t];
    }
  }
  if (!DECODE && c.host_kv) {
    // (a5 gather from the unit cache / the host mirror: k_pull_pack)
  } else if (!DECODE) {
    // a5 gather: pack the K and V rows of the selected spans into one contiguous slab per (layer, KV head), so the
    // attention kernel that continues over them reads whole 128-row tiles.  16 threads per 256-byte row, four rows
    // of K and of V in flight per thread; the rows up to the next multiple of 8 are zero-filled.
    const int nr = s_nr, R = s_pre[nr], Rz = (R + 7) & ~7;
    const size_t slab = (unit * c.Hkv + g) * (size_t)c.SR;  // (resident contexts only: row = token)
    const uint4* Ksrc = reinterpret_cast<const uint4*>(c.Kc + slab * kD);
    const uint4* Vsrc = reinterpret_cast<const uint4*>(c.Vc + slab * kD);
    const size_t gslab = ((size_t)layer * c.Hkv + g) * (size_t)c.Rcap;
    uint4* Kdst = reinterpret_cast<uint4*>(c.Kg + gslab * kD);
    uint4* Vdst = reinterpret_cast<uint4*>(c.Vg + gslab * kD);
    const int ch = tid & 15, rpp = nt >> 4;  // 16-byte chunk of the row, rows per pass
    // (rows dealt to the CTAs rpp at a time, so that few rows reach all of them)
    const int step = parts * rpp;
    for (int r0 = my_part * rpp + (tid >> 4); r0 < Rz; r0 += 4 * step) {
      uint4 kv[4], vv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + i * step;
        kv[i] = vv[i] = make_uint4(0u, 0u, 0u, 0u);
        if (r < R) {
          int lo = 0, hi = nr - 1;  // last range whose first packed row is <= r
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= r) lo = mid; else hi = mid - 1;
          }
          const size_t tok = (size_t)(s_rs[lo] + (r - s_pre[lo]));
          kv[i] = __ldg(Ksrc + tok * 16 + ch);
          vv[i] = __ldg(Vsrc + tok * 16 + ch);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + i * step;
        if (r < Rz) {
          Kdst[(size_t)r * 16 + ch] = kv[i];
          Vdst[(size_t)r * 16 + ch] = vv[i];
        }
      }
    }
  }
}

// Host-memory pager (Sec. 3.4), data movement of a prefill call.  A task = one (named unit, KV head, layer): bring
// the unit's rows to the slab the retrieved attention reads (a5 gather) -- from its cache slot, or over the bus from
// the host mirror, in which case the rows also go into the slot the top-k kernel chose for the unit (unless the unit
// is the one the indexed range ends in and still grows: that one is never cached).  A few small persistent CTAs walk the tasks:
// small and few on purpose, so that each fits onto an SM beside the one large CTA of the attention and map kernels and the
// bus transfer really runs under the computation of the call's other layers instead of taking SMs away from it.
// Registers decide whether one fits: those kernels' 18 warps of 96 leave 1024 free on two of an SM's four partitions, which is
// a warp of 32 registers a thread.  With 64 a thread a CTA found room only where a large one had just left, and all of them
// crowded onto four to eight SMs, which takes twice as long.  Four 16-byte loads per thread in flight, K rows first, then V rows.
// 512-token calls of 8 / 12 / 16 / 32 layers, 32 CTAs of 64 registers a thread: 1.32 / 2.58 / 3.72 / 8.26 ms, 64 of 32: 1.29 /
// 1.89 / 2.42 / 4.86.
constexpr int kPullThreads = 128;
constexpr int kPullCtas = 64;

__global__ void __launch_bounds__(kPullThreads, 65536 / (kPullThreads * 32))
    k_pull_pack(DevCtx c, int seq, int layer_begin, int layer_count, int max_units) {
  __shared__ int s_off;
  const int tid = threadIdx.x;
  const int ntasks = max_units * c.Hkv * layer_count;
  for (int task = blockIdx.x; task < ntasks; task += gridDim.x) {
  const int t = task % max_units, g = (task / max_units) % c.Hkv, layer = layer_begin + task / (max_units * c.Hkv);
  const size_t unit = unit_of(c, seq, layer);
  const int nall = min(c.pl_cnt[unit * c.Hkv + g], 2 * kMaxTopK);
  if (t >= nall) continue;
  __syncthreads();  // (s_off of the previous task has been read by everyone)
  const size_t pb = (unit * c.Hkv + g) * (size_t)(2 * kMaxTopK);
  // first packed row of this unit: the units are packed in ascending order, every token once
  if (tid < 32) {
    int part = 0;
    for (int i = tid; i < t; i += 32) part += c.pl_len[pb + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (tid == 0) s_off = part;
  }
  __syncthreads();
  const int U = c.unit;
  const int id = c.pl_id[pb + t], src = c.pl_src[pb + t], st = c.pl_start[pb + t], ln = c.pl_len[pb + t];
  const size_t gslab = ((size_t)layer * c.Hkv + g) * (size_t)c.Rcap + s_off;
  uint4* Kdst = reinterpret_cast<uint4*>(c.Kg + gslab * kD);
  uint4* Vdst = reinterpret_cast<uint4*>(c.Vg + gslab * kD);
  const int n16 = ln * 16;
  const size_t hslab = (unit * c.Hkv + g) * (size_t)c.Tpad;
  const size_t row = ((unit * c.Hkv + g) * (size_t)c.cache_units + (src & 0xffff)) * (size_t)U + (st - id * U);
  const bool bus = src < 0 || (src & 0x10000);  // not in the cache: over the bus, and into its slot if it has one
#pragma unroll 1
  for (int kv = 0; kv < 2; ++kv) {
    uint4* slot = src < 0 ? nullptr : reinterpret_cast<uint4*>((kv ? c.Vcache : c.Kcache) + row * kD);
    const uint4* from = bus ? reinterpret_cast<const uint4*>((kv ? c.hostV : c.hostK) + (hslab + st) * kD) : slot;
    uint4* to = kv ? Vdst : Kdst;
    if (!bus) slot = nullptr;
    for (int i0 = tid; i0 < n16; i0 += 4 * kPullThreads) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kPullThreads;
        if (i < n16) v[u] = from[i];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kPullThreads;
        if (i < n16) {
          to[i] = v[u];
          if (slot) slot[i] = v[u];
        }
      }
    }
  }
  if (t == nall - 1) {
    // the packed rows up to the next multiple of eight are zero (tile pieces are eight rows high)
    const int R = s_off + ln, pad = ((R + 7) & ~7) - R;
    for (int i = tid; i < pad * 16; i += kPullThreads) {
      Kdst[n16 + i] = make_uint4(0u, 0u, 0u, 0u);
      Vdst[n16 + i] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  }  // task
}

cudaError_t launch_pull_pack(const DevCtx& c, const PrefillArgs& a, cudaStream_t s) {
  k_pull_pack<<<kPullCtas, kPullThreads, 0, s>>>(c, a.seq, a.layer_begin, a.layer_count, c.topk);
  return cudaGetLastError();
}

// Decode retrieval in one launch: a CTA owns one (sequence, layer, KV head), streams that head's index once
// (half-warp per 256-byte row, 16 bytes per lane, four rows in flight), keeps the scores in shared memory, selects the
// top-k there (same radix select as k_topk) and writes the selection and the token ranges of the attention kernel.
constexpr int kFusedMaxSpans = 12288;  // scores kept in shared memory (48 KB)
constexpr int kDecSelRegs = 16;        // keys per thread the select holds in registers (8K spans at 512 threads)

__global__ void __launch_bounds__(1024) k_dec_retrieve(DevCtx c, int layer_begin, DecBatch b, int layer_count,
                                                       const __nv_bfloat16* __restrict__ q,
                                                       const __nv_bfloat16* __restrict__ knew,
                                                       const __nv_bfloat16* __restrict__ vnew) {
  chain_wait();
  extern __shared__ unsigned sck[];  // [N] order-preserving keys of the scores
  __shared__ float su[kD];
  __shared__ unsigned hist[256];
  __shared__ unsigned s_prefix, s_need;
  __shared__ int s_ids[kMaxTopK];
  __shared__ int s_cnt;
  __shared__ int s_scan[1024];
  __shared__ unsigned s_ckey[kSelCand];
  __shared__ int s_rs[kMaxRanges], s_rl[kMaxRanges], s_nr, s_sst[2 * kMaxTopK], s_sln[2 * kMaxTopK];
  __shared__ int s_all[2 * kMaxTopK];
  const int g = blockIdx.x;
  const int bi = blockIdx.y / layer_count, l = blockIdx.y % layer_count, layer = layer_begin + l;
  const int sq = b.seq[bi], pos = b.pos[bi], loc_begin = b.loc_begin[bi];
  const size_t unit = unit_of(c, sq, layer);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int N = min(c.n_spans[unit], kFusedMaxSpans);
  const int rh = ret_head_of(c, layer), gk = rh >= 0 ? rh / c.G : g;  // retrieval head of the layer (Sec. 3.5)
  append_decode_row(c, b, bi, l, layer_count, unit, g, knew, vnew);
  // ---- scores.  The first four index rows of every half-warp are requested before the query sum below is formed,
  // so that their latency and that of the query loads pass together.
  const int hw = tid >> 4, hl = tid & 15, nhw = nt >> 4;  // half-warps of the CTA (the launch picks its size)
  const __nv_bfloat16* KR = c.KR + (unit * c.Hkv + gk) * (size_t)c.cap * kD + hl * 8;
  // software pipeline: the next four rows are in flight while the current four are reduced
  auto fetch = [&](int base, uint4 (&raw)[4]) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int s = base + t * nhw + hw;
      raw[t] = s < N ? __ldg(reinterpret_cast<const uint4*>(KR + (size_t)s * kD)) : make_uint4(0, 0, 0, 0);
    }
  };
  uint4 cur[4], nxt[4];
  fetch(0, cur);
  if (tid < kD) {
    const __nv_bfloat16* qp = q + (((size_t)b.src[bi] * layer_count + l) * c.Hq + gk * c.G) * kD + tid;
    float acc = 0.f;
    for (int hh = 0; hh < c.G; ++hh)
      if (rh < 0 || gk * c.G + hh == rh) acc += __bfloat162float(qp[(size_t)hh * kD]);
    su[tid] = acc;
  }
  if (tid == 0) s_cnt = 0;
  __syncthreads();
  {
    float uf[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) uf[e] = su[hl * 8 + e];
    for (int base = 0; base < N; base += nhw * 4) {  // uniform trip count (shuffles inside)
      fetch(base + nhw * 4, nxt);                    // past the end: zeros, no loads
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&cur[t]);
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __bfloat1622float2(p2[i]);
          d = fmaf(uf[2 * i], f.x, d);
          d = fmaf(uf[2 * i + 1], f.y, d);
        }
        d += __shfl_xor_sync(0xffffffffu, d, 1);
        d += __shfl_xor_sync(0xffffffffu, d, 2);
        d += __shfl_xor_sync(0xffffffffu, d, 4);
        d += __shfl_xor_sync(0xffffffffu, d, 8);
        const int s = base + t * nhw + hw;
        if (hl == 0 && s < N) sck[s] = order_key(d);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) cur[t] = nxt[t];
    }
  }
  __syncthreads();
  // ---- top-k over the shared-memory scores
  const int K = min(c.topk, N);
  if (K == N) {
    for (int t = tid; t < K; t += nt) s_ids[t] = t;
    if (tid == 0) s_cnt = K;
  } else {
    radix_select_top<unsigned, kDecSelRegs>([&](int i) { return sck[i]; }, N, K, hist, &s_prefix, &s_need, s_scan,
                                            &s_cnt, s_ids, s_ckey);
  }
  __syncthreads();
  const int cnt = min(s_cnt, K);
  int myid = -1, rank = 0;
  if (tid < cnt) {
    myid = s_ids[tid];
    for (int t = 0; t < cnt; ++t) rank += s_ids[t] < myid;
  }
  __syncthreads();
  if (tid < cnt) s_ids[rank] = myid;
  __syncthreads();
  int* sel = c.sel + (unit * c.Hkv + g) * (size_t)c.topk;
  for (int t = tid; t < c.topk; t += nt) sel[t] = t < cnt ? s_ids[t] : -1;
  const int* ids_all = s_ids;
  int nall = cnt;
  if (c.persist) {
    nall = union_with_persistent(c, unit, g, s_ids, cnt, s_scan, s_all);
    ids_all = s_all;
  }
  if (tid < nall) {
    s_sst[tid] = c.span_start[unit * c.cap + ids_all[tid]];
    s_sln[tid] = c.span_len[unit * c.cap + ids_all[tid]];
  }
  __syncthreads();
  if (tid < 32) {
    // items: the sink, the selected spans, the recent tokens
    const int rb = min(loc_begin, pos + 1);
    const int nr = merge_ranges_warp(
        nall + 2,
        [&](int i, int& st, int& ln) {
          if (i == 0) {
            st = 0;
            ln = min(c.Ls, pos + 1);
          } else if (i <= nall) {
            st = s_sst[i - 1];
            ln = s_sln[i - 1];
          } else {
            st = rb;
            ln = pos + 1 - rb;
          }
        },
        s_rs, s_rl);
    long long tokens = 0;
    for (int t = tid; t < nall; t += 32) tokens += s_sln[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tokens += shfl_xor_ll(tokens, o);
    if (tid == 0) {
      s_nr = nr;
      c.rng_cnt[unit * c.Hkv + g] = nr;
      c.sel_tokens[unit * c.Hkv + g] = tokens;  // (summed over the KV heads by ltri_get_stats)
    }
  }
  __syncthreads();
  const size_t rbb = (unit * c.Hkv + g) * (size_t)c.rcap;
  for (int t = tid; t < s_nr; t += nt) {
    c.rng_start[rbb + t] = s_rs[t];
    c.rng_len[rbb + t] = s_rl[t];
  }
}

// Decode retrieval in one launch for an index too large for one CTA's shared memory (up to 98K spans, the 1M-token
// workload): a thread-block cluster of eight CTAs owns one (sequence, layer, KV head).  Each
// CTA streams its eighth of that head's index once (half-warp per 256-byte row, 16 bytes per lane, four rows in
// flight, the next four prefetched) and keeps its scores in shared memory; the cluster then selects the top-k with
// the radix select of k_topk, every CTA counting its own scores and all of them adding the eight histograms up
// through distributed shared memory; the selected ids meet in the first CTA, which writes the selection and the
// token ranges of the attention kernel.
constexpr int kRetCluster = 8;
constexpr int kRetThreads = 512;
constexpr int kRetSliceMax = 12288;  // scores a CTA keeps in shared memory (48 KB)

__global__ void __cluster_dims__(kRetCluster, 1, 1) __launch_bounds__(kRetThreads)
    k_dec_retrieve_cl(DevCtx c, int layer_begin, DecBatch b, int layer_count, const __nv_bfloat16* __restrict__ q,
                      const __nv_bfloat16* __restrict__ knew, const __nv_bfloat16* __restrict__ vnew) {
  chain_wait();
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ float ssc[];  // this CTA's slice of the scores
  __shared__ float su[kD];
  __shared__ unsigned hist[256];  // this CTA's histogram (read by the whole cluster)
  __shared__ unsigned tot[256];   // the cluster's histogram (every CTA builds its own copy)
  __shared__ unsigned s_prefix, s_need;
  __shared__ int s_eq, s_take;    // this CTA's count of scores equal to the threshold / of selected scores
  __shared__ int s_ids[kMaxTopK]; // first CTA: all selected ids, ascending
  __shared__ int s_loc[kMaxTopK]; // this CTA's selected ids
  __shared__ int s_scan[kRetThreads];
  __shared__ int s_rs[kMaxRanges], s_rl[kMaxRanges], s_nr, s_sst[2 * kMaxTopK], s_sln[2 * kMaxTopK];
  __shared__ int s_all[2 * kMaxTopK];
  const int rank = (int)cluster.block_rank();
  const int g = blockIdx.x / kRetCluster;
  const int bi = blockIdx.y / layer_count, l = blockIdx.y % layer_count, layer = layer_begin + l;
  const int sq = b.seq[bi], pos = b.pos[bi], loc_begin = b.loc_begin[bi];
  const size_t unit = unit_of(c, sq, layer);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int N = min(c.n_spans[unit], kRetCluster * kRetSliceMax);
  const int per = (N + kRetCluster - 1) / kRetCluster;
  const int lo = min(N, rank * per), hi = min(N, lo + per), nloc = hi - lo;  // this CTA's spans [lo, hi)
  const int rh = ret_head_of(c, layer), gk = rh >= 0 ? rh / c.G : g;  // retrieval head of the layer (Sec. 3.5)
  if (rank == 0) append_decode_row(c, b, bi, l, layer_count, unit, g, knew, vnew);
  if (tid < kD) {
    const __nv_bfloat16* qp = q + (((size_t)b.src[bi] * layer_count + l) * c.Hq + gk * c.G) * kD + tid;
    float acc = 0.f;
    for (int hh = 0; hh < c.G; ++hh)
      if (rh < 0 || gk * c.G + hh == rh) acc += __bfloat162float(qp[(size_t)hh * kD]);
    su[tid] = acc;
  }
  __syncthreads();
  // ---- scores of the slice
  {
    constexpr int HW = kRetThreads / 16;  // half-warps
    const int hw = tid >> 4, hl = tid & 15;
    float uf[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) uf[e] = su[hl * 8 + e];
    const __nv_bfloat16* KR = c.KR + ((unit * c.Hkv + gk) * (size_t)c.cap + lo) * kD + hl * 8;
    auto fetch = [&](int base, uint4 (&raw)[4]) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int s = base + t * HW + hw;
        raw[t] = s < nloc ? __ldg(reinterpret_cast<const uint4*>(KR + (size_t)s * kD)) : make_uint4(0, 0, 0, 0);
      }
    };
    uint4 cur[4], nxt[4];
    fetch(0, cur);
    for (int base = 0; base < nloc; base += HW * 4) {  // uniform trip count (shuffles inside)
      fetch(base + HW * 4, nxt);                       // past the end: zeros, no loads
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&cur[t]);
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __bfloat1622float2(p2[i]);
          d = fmaf(uf[2 * i], f.x, d);
          d = fmaf(uf[2 * i + 1], f.y, d);
        }
        d += __shfl_xor_sync(0xffffffffu, d, 1);
        d += __shfl_xor_sync(0xffffffffu, d, 2);
        d += __shfl_xor_sync(0xffffffffu, d, 4);
        d += __shfl_xor_sync(0xffffffffu, d, 8);
        const int s = base + t * HW + hw;
        if (hl == 0 && s < nloc) ssc[s] = d;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) cur[t] = nxt[t];
    }
  }
  __syncthreads();
  // ---- top-k over the cluster's scores
  const int K = min(c.topk, N);
  if (tid == 0) s_take = 0;
  __syncthreads();
  if (K == N) {
    for (int t = tid; t < nloc; t += nt) s_loc[t] = lo + t;  // (N <= top_k <= 64)
    if (tid == 0) s_take = nloc;
  } else {
    if (tid == 0) {
      s_prefix = 0;
      s_need = K;  // rank from the top, 1-based: find key T with #(key > T) < K <= #(key >= T)
    }
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      if (tid < 256) hist[tid] = 0;
      __syncthreads();
      const unsigned prefix = s_prefix;
      const unsigned himask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
      DigitRuns dr;
      for (int s = tid; s < nloc; s += nt) {
        const unsigned key = order_key(ssc[s]);
        if ((key & himask) == prefix) dr.add(hist, (int)((key >> shift) & 255u));
      }
      dr.flush(hist);
      cluster.sync();
      if (tid < 256) {
        unsigned sum = 0;
        for (int r = 0; r < kRetCluster; ++r) sum += cluster.map_shared_rank(hist, r)[tid];
        tot[tid] = sum;
      }
      cluster.sync();  // every CTA has read every histogram: they may be reset
      if (tid < 32) {
        unsigned need = s_need;
        const int bin = pick_from_top(tot, 256, need);
        if (tid == 0) {
          s_need = need;
          s_prefix = prefix | ((unsigned)bin << shift);
        }
      }
      __syncthreads();
    }
    const unsigned T = s_prefix;
    const unsigned need_eq = s_need;  // how many of the == T elements are taken (lowest ids first, cluster-wide)
    if (tot[T & 255u] == need_eq) {
      // (the last pass counted the cluster's keys equal to T; every CTA holds the same tot) every key at the
      // threshold is taken: no order among them is needed, and no exchange of counts
      for (int s = tid; s < nloc; s += nt)
        if (order_key(ssc[s]) >= T) {
          const int slot = atomicAdd(&s_take, 1);
          if (slot < kMaxTopK) s_loc[slot] = lo + s;
        }
    } else {
    // contiguous id partition so that ties are picked in id order: inside the CTA by thread, across CTAs by rank
    const int pt = (nloc + nt - 1) / nt;
    const int tlo = min(nloc, tid * pt), thi = min(nloc, tlo + pt);
    int eq = 0;
    for (int s = tlo; s < thi; ++s) eq += order_key(ssc[s]) == T;
    s_scan[tid] = eq;
    __syncthreads();
    if (tid < 32) {
      const int run = warp0_exclusive_scan(s_scan, nt);
      if (tid == 0) s_eq = run;
    }
    cluster.sync();
    int eqrank = s_scan[tid];
    for (int r = 0; r < rank; ++r) eqrank += *cluster.map_shared_rank(&s_eq, r);
    for (int s = tlo; s < thi; ++s) {
      const unsigned key = order_key(ssc[s]);
      bool take = key > T;
      if (key == T) {
        take = (unsigned)eqrank < need_eq;
        ++eqrank;
      }
      if (take) {
        const int slot = atomicAdd(&s_take, 1);
        if (slot < kMaxTopK) s_loc[slot] = lo + s;
      }
    }
    }
  }
  __syncthreads();
  // this CTA's ids in ascending order (rank sort), then into the first CTA's list behind those of the lower ranks
  const int ntake = min(s_take, kMaxTopK);
  int myid = -1, myrank = 0;
  if (tid < ntake) {
    myid = s_loc[tid];
    for (int t = 0; t < ntake; ++t) myrank += s_loc[t] < myid;
  }
  cluster.sync();  // every CTA's s_take is final
  int offset = 0, total = 0;
  for (int r = 0; r < kRetCluster; ++r) {
    const int v = min(*cluster.map_shared_rank(&s_take, r), kMaxTopK);
    if (r < rank) offset += v;
    total += v;
  }
  if (tid < ntake && offset + myrank < kMaxTopK) cluster.map_shared_rank(s_ids, 0)[offset + myrank] = myid;
  cluster.sync();  // the list is complete; the other CTAs' shared memory is not read after this point
  if (rank != 0) return;
  const int cnt = min(total, K);
  int* sel = c.sel + (unit * c.Hkv + g) * (size_t)c.topk;
  for (int t = tid; t < c.topk; t += nt) sel[t] = t < cnt ? s_ids[t] : -1;
  const int* ids_all = s_ids;
  int nall = cnt;
  if (c.persist) {
    nall = union_with_persistent(c, unit, g, s_ids, cnt, s_scan, s_all);
    ids_all = s_all;
  }
  if (tid < nall) {
    s_sst[tid] = c.span_start[unit * c.cap + ids_all[tid]];
    s_sln[tid] = c.span_len[unit * c.cap + ids_all[tid]];
  }
  __syncthreads();
  if (tid < 32) {
    // items: the sink, the selected spans, the recent tokens
    const int rbeg = min(loc_begin, pos + 1);
    const int nr = merge_ranges_warp(
        nall + 2,
        [&](int i, int& st, int& ln) {
          if (i == 0) {
            st = 0;
            ln = min(c.Ls, pos + 1);
          } else if (i <= nall) {
            st = s_sst[i - 1];
            ln = s_sln[i - 1];
          } else {
            st = rbeg;
            ln = pos + 1 - rbeg;
          }
        },
        s_rs, s_rl);
    long long tokens = 0;
    for (int t = tid; t < nall; t += 32) tokens += s_sln[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tokens += shfl_xor_ll(tokens, o);
    if (tid == 0) {
      s_nr = nr;
      c.rng_cnt[unit * c.Hkv + g] = nr;
      c.sel_tokens[unit * c.Hkv + g] = tokens;  // (summed over the KV heads by ltri_get_stats)
    }
  }
  __syncthreads();
  const size_t rbb = (unit * c.Hkv + g) * (size_t)c.rcap;
  for (int t = tid; t < s_nr; t += nt) {
    c.rng_start[rbb + t] = s_rs[t];
    c.rng_len[rbb + t] = s_rl[t];
  }
}

cudaError_t launch_dec_retrieve_fused(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count,
                                      const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                      int span_bound, bool force_cluster, int threads, cudaStream_t s) {
  span_bound = max(span_bound, 1);
  if (span_bound <= kFusedMaxSpans && !force_cluster) {  // one CTA per head: no cluster barriers
    return launch_chained(k_dec_retrieve, dim3(c.Hkv, b.n * layer_count), dim3(threads), sizeof(float) * span_bound, s,
                          c, layer_begin, b, layer_count, q, k, v);
  }
  const int per = (span_bound + kRetCluster - 1) / kRetCluster;
  if (per > kRetSliceMax) return cudaErrorInvalidValue;
  return launch_chained(k_dec_retrieve_cl, dim3(c.Hkv * kRetCluster, b.n * layer_count), dim3(kRetThreads),
                        sizeof(float) * per, s, c, layer_begin, b, layer_count, q, k, v);
}
int dec_retrieve_fused_max_spans() { return kRetCluster * kRetSliceMax; }

// dynamic shared memory of k_topk: one order key per unit in unit mode (at most 12K units: 48 KB), nothing otherwise;
// under collaborative voting a tally per unit behind the keys
static int topk_unit_smem(const DevCtx& c) {
  if (c.unit <= 0) return 0;
  const int n = (int)(c.Tmax / c.unit + 2);
  return (int)sizeof(unsigned) * (c.vote ? 2 * n + 4 : n);
}

constexpr int kTopkStage = 48 * 1024;  // most order keys a prefill select keeps in shared memory

cudaError_t prepare_state() {
  cudaError_t e = cudaSuccess;
  for (auto fn : {k_segment<unsigned>, k_segment<unsigned long long>})
    e = first_error(e, first_error(allow_smem(fn, -1),
                                   cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)));
  for (auto fn : {k_topk<false>, k_topk<true>}) e = first_error(e, allow_smem(fn, -1));
  // (48 KB of keys beside the static arrays: more than a kernel may use without asking)
  e = first_error(e, first_error(allow_smem(k_dec_retrieve, kFusedMaxSpans * (int)sizeof(unsigned)),
                                 allow_smem(k_dec_retrieve_cl, kRetSliceMax * (int)sizeof(float))));
  return first_error(e, allow_smem(k_score<false>, -1));
}

// Top-k of the call.  Under collaborative voting (Sec. 3.5) two launches: the ballots of the layers with a retrieval
// head, then the vote (a layer reads the ballots of the layers up to its own, also those of earlier calls for the same
// chunk or step).
template <bool DECODE>
static cudaError_t launch_topk(const DevCtx& c, int seq, int layer_begin, const DecBatch& b, int layer_count, int gy,
                               int evicted_end, int span_bound, cudaStream_t s) {
  int smem = topk_unit_smem(c), stage = 0, parts = 1;
  if (!DECODE && !c.host_kv && !c.vote) {
    // Few (layer, KV head) pairs: several CTAs repeat the selection (it costs them nothing: the GPU is idle) and share the
    // packing, which one CTA of 512 threads alone does at some 60 GB/s (one layer, 512 tokens a KV head: 33 us).
    parts = max(1, min(16, c.sms / (c.Hkv * gy)));
    // With a CTA per SM to spare the scores are read once into shared memory: any number of them that fits, in short
    // loops (unrolled over 24 registers per thread, the select is 12 KB of instructions that a lone launch fetches cold)
    if (c.unit == 0 && span_bound <= kTopkStage && c.Hkv * gy <= c.sms) {
      stage = span_bound;
      smem = stage * (int)sizeof(unsigned);
    }
  }
  if (c.vote) {
    const cudaError_t e = launch_chained(k_topk<DECODE>, dim3(c.Hkv, gy), dim3(512), smem, s, c, seq, layer_begin, b,
                                         layer_count, evicted_end, (int)kTopkBallot, 1, 0);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(k_topk<DECODE>, dim3(c.Hkv * parts, gy), dim3(512), smem, s, c, seq, layer_begin, b, layer_count,
                        evicted_end, (int)(c.vote ? kTopkVote : kTopkSelect), parts, stage);
}

cudaError_t launch_topk_prefill(const DevCtx& c, const PrefillArgs& a, int span_bound, cudaStream_t s) {
  DecBatch dummy;
  dummy.n = 0;
  return launch_topk<false>(c, a.seq, a.layer_begin, dummy, a.layer_count, a.layer_count, a.loc_begin,
                            span_bound, s);
}

cudaError_t launch_topk_decode(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count, cudaStream_t s) {
  return launch_topk<true>(c, 0, layer_begin, b, layer_count, b.n * layer_count, 0, 0, s);
}

}  // namespace ltri
