// A whole decode step in one launch (Sec. 3.5: while decoding, the current block is one token), for steps whose
// (sequence, layer, KV head) units are too few to fill the GPU: append, scores against the index (Eq. 7), top-k (Eq. 8),
// token ranges, split-KV attention and the merge of the splits.
//
// A thread-block cluster of S CTAs owns one unit.  Every CTA scans 1/S of the unit's index; the cluster finds the top-k
// together: the largest score, one summed histogram of how far the other scores lie below it, and the few candidates
// within the cut, which every CTA receives from the others and ranks by itself (the same integers in every CTA, so
// nothing has to be sent back).  A CTA then attends over 1/S of the sink and recent tokens, whose first tiles were
// requested before the scan began, and over 1/S of the selected tokens; the partial softmaxes are pushed through
// distributed shared memory to the CTAs that write the outputs.
//
// Bound: latency.  As five (or three) launches a step of one layer costs 20 to 50 us whatever it reads, because each
// kernel is a dependent chain of a few memory round trips between a launch and a drain and uses 8 to 72 of 148 SMs.
// Two CTAs of 256 threads fit an SM (<= 113 KB of shared memory, 128 registers): clusters of 16 are then available for
// the eight units of one layer with eight KV heads (with one CTA per SM only seven such clusters fit the GPU).
#include <cooperative_groups.h>

#include "common.cuh"
#include "decode_util.cuh"
#include "select_util.cuh"

namespace ltri {

namespace cg = cooperative_groups;

constexpr int kStThreads = 256;
constexpr int kStWarps = kStThreads / 32;
constexpr int kStTileBytes = 2 * kDTile * 256;  // K and V rows of a 16-token tile
constexpr int kStRing = kStWarps * kStTileBytes;
constexpr int kStMaxCluster = 16;
constexpr int kStList = 1024;         // candidates of a cluster: room for kStList / S per CTA
constexpr int kStCand = kStThreads;   // candidates ranked against each other, one per thread
constexpr int kStAhead = 4;           // batches of index rows requested ahead of the scan
constexpr int kStMaxSlots = 5120;     // order keys a CTA can keep (20 KB)
static_assert(kStRing >= (int)(kStWarps * 8 * (kD + 2) * sizeof(float)), "the warps' partials reuse the ring");
static_assert(kStMaxCluster * kMaxTopK <= kStList, "the lists of the general select reuse the candidates'");

// dynamic shared memory: K/V ring | candidates | order keys
static int dec_step_smem(int key_slots) { return kStRing + kStList * 8 + key_slots * 4; }

template <int G>
__global__ void __launch_bounds__(kStThreads, 2)
    k_dec_step(DevCtx c, int layer_begin, DecBatch b, int layer_count, const __nv_bfloat16* __restrict__ q,
               const __nv_bfloat16* __restrict__ knew, const __nv_bfloat16* __restrict__ vnew,
               __nv_bfloat16* __restrict__ out, int key_slots) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  // [S][kStList / S] (key, id) of the candidates, larger key first, then lower id: one descending order
  unsigned long long* s_list = reinterpret_cast<unsigned long long*>(dsm + kStRing);
  unsigned* g_key = reinterpret_cast<unsigned*>(s_list);  // general select: the cluster's lists, keys then ids
  int* g_id = reinterpret_cast<int*>(g_key + kStMaxCluster * kMaxTopK);
  unsigned* sck = reinterpret_cast<unsigned*>(dsm + kStRing + kStList * 8);  // [key_slots] this CTA's order keys
  __shared__ float su[kD];
  __shared__ unsigned hist[256];
  __shared__ unsigned r_hist[256];  // added up by the CTAs of the cluster: the histogram over all their keys
  __shared__ unsigned s_prefix, s_need;
  __shared__ int s_ids[kMaxTopK], s_cnt, s_cut;
  __shared__ int s_scan[64 + kSelCand];
  __shared__ unsigned s_ckey[kSelCand];
  __shared__ unsigned long long s_rank[kStCand];
  __shared__ unsigned l_key[kMaxTopK];  // general select: this CTA's candidates, ascending span ids
  __shared__ int l_id[kMaxTopK];
  __shared__ unsigned r_max[kStMaxCluster];  // written by the other CTAs: their largest keys, their candidate counts
  __shared__ int r_cnt[kStMaxCluster];
  __shared__ int s_all[2 * kMaxTopK];
  __shared__ int s_sst[2 * kMaxTopK], s_sln[2 * kMaxTopK];
  __shared__ int s_rs[kMaxRanges], s_rl[kMaxRanges], s_rp[kMaxRanges + 1], s_nr;
  // host-memory pager: the unit cache as the first CTA sees it, the named units' slots
  __shared__ int s_tag[128], s_src[2 * kMaxTopK], s_fill[2 * kMaxTopK];
  __shared__ float s_sco[128];
  __shared__ unsigned char s_named[128];
  // written by the other CTAs: their partial softmaxes -- (m, l) of every head, O of this CTA's share of the outputs
  __shared__ float2 r_ml[kStMaxCluster][G];
  __shared__ float r_o[G * kD];
  cg::cluster_group cluster = cg::this_cluster();
  chain_wait();
  cluster.barrier_arrive();  // (waited for in front of the first access to another CTA's shared memory)
  const int S = (int)gridDim.x, rank = (int)blockIdx.x, g = blockIdx.y;
  const int bi = blockIdx.z / layer_count, l = blockIdx.z % layer_count, layer = layer_begin + l;
  const int pos = b.pos[bi], loc_begin = b.loc_begin[bi];
  const size_t unit = unit_of(c, b.seq[bi], layer);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int nt = kStThreads;
  const int nsp = c.n_spans[unit];
  const int U = c.unit;
  const int rh = ret_head_of(c, layer), gk = rh >= 0 ? rh / c.G : g;  // retrieval head of the layer (Sec. 3.5)
  const size_t qrow = ((size_t)b.src[bi] * layer_count + l) * c.Hq;
  const size_t nrow = ((size_t)b.src[bi] * layer_count + l) * c.Hkv + g;  // the new token's K/V row

  // ---- the tokens known without a retrieval: the sink and everything since the last eviction
  const int a0 = min(c.Ls, pos + 1), rb = min(loc_begin, pos + 1);
  const int nA = a0 + (pos + 1 - rb), perA = (nA + S - 1) / S;
  const int tA0 = min(nA, rank * perA), tA1 = min(nA, tA0 + perA);
  const int ntA = (tA1 - tA0 + kDTile - 1) / kDTile;
  const __nv_bfloat16* Kslab = c.Kc + (unit * c.Hkv + g) * (size_t)c.SR * kD;
  const __nv_bfloat16* Vslab = c.Vc + (unit * c.Hkv + g) * (size_t)c.SR * kD;
  const uint32_t sk = smem_u32(dsm) + warp * kStTileBytes, sv = sk + kDTile * 256;  // this warp's tile: K rows, V rows
  const int ch = lane & 15;
  // A tile is copied in two steps: every lane finds the row of one of its tokens (lane & 15), then copies 16 bytes at chunk ch
  // of the rows (lane >> 4) + 2i, whose numbers it gets from the lanes that found them.  (A kernel this short fetches each of
  // its instructions once, at some ten cycles apiece, so what counts on the way is their number: with every lane working out
  // eight addresses for the keys and eight for the values at each place, requesting a tile took 3K cycles.)
  constexpr int kNoRow = -1, kNewRow = -2;  // the new token's row comes from the caller's tensors: another CTA stores it
  auto known_row = [&](int t) {
    const int v = tA0 + t * kDTile + ch, tok = v < a0 ? v : rb + (v - a0);
    return v >= tA1 ? kNoRow : tok == pos ? kNewRow : (int)slab_row(c, tok, b.shift[bi]);
  };
  auto copy_rows = [&](int rows, const __nv_bfloat16* base, const __nv_bfloat16* fresh, uint32_t dst) {
#pragma unroll
    for (int i = 0; i < kDTile / 2; ++i) {
      const int row = 2 * i + (lane >> 4), r = __shfl_sync(0xffffffffu, rows, row);
      const __nv_bfloat16* src = r == kNewRow ? fresh : base + (size_t)max(r, 0) * kD;
      cp_async16(dst + tile_off(row, ch), src + ch * 8, r == kNoRow ? 0 : 16);
    }
  };
  const bool early = warp < ntA;  // this warp's first tile is requested before the retrieval
  if (early) {
    const int rows = known_row(warp);
#pragma unroll 1
    for (int kv = 0; kv < 2; ++kv) {
      copy_rows(rows, kv ? Vslab : Kslab, (kv ? vnew : knew) + nrow * kD, kv ? sv : sk);
      cp_async_commit();
    }
  }
  // the new token's rows go to the cache at the end: their load is not waited for on the way (by the CTA with the fewest tokens)
  const bool appends = rank == S - 1 && warp == kStWarps - 1;
  uint4 new_row = make_uint4(0u, 0u, 0u, 0u);
  if (appends) new_row = *reinterpret_cast<const uint4*>((lane < 16 ? knew : vnew) + nrow * kD + ch * 8);

  // ---- retrieval
  int nall = 0;
  const int* ids_all = s_ids;
  uint32_t qa[8][2];     // query fragments: rows 0..G-1 of the 16-row A operand are the heads of the group
  const int r = lane >> 2, qd = lane & 3;
  auto load_q = [&]() {
    const __nv_bfloat16* qp = q + (qrow + (size_t)g * G + (r < G ? r : 0)) * kD;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      qa[ks][0] = r < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 2 * qd) : 0u;
      qa[ks][1] = r < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8 + 2 * qd) : 0u;
    }
  };
  if (nsp > 0) {
    // the cluster's slices of the index, and what is ranked: the spans, or (Eq. 8 as printed) fixed token units
    const int per = (nsp + S - 1) / S;
    const int lo = min(nsp, rank * per), nloc = min(nsp, lo + per) - lo;
    const int u0 = U > 0 ? c.Ls / U : 0;
    const int Nu = U > 0 && loc_begin > c.Ls ? min((loc_begin + U - 1) / U - u0, key_slots / 2) : 0;
    unsigned* utot = sck + Nu;  // unit mode: this CTA's keys of the units, then the cluster's
    if (U > 0)
      for (int i = tid; i < Nu; i += nt) sck[i] = 0u;  // below the key of every real score
    constexpr int HW = kStThreads / 16, R = 8;  // half-warps, rows in flight per half-warp
    const int hw = tid >> 4, hl = tid & 15;
    const __nv_bfloat16* KR = c.KR + ((unit * c.Hkv + gk) * (size_t)c.cap + lo) * kD + hl * 8;
    auto fetch = [&](int base, uint4 (&raw)[R]) {
#pragma unroll
      for (int t = 0; t < R; ++t) {
        const int s = base + t * HW + hw;
        raw[t] = s < nloc ? __ldg(reinterpret_cast<const uint4*>(KR + (size_t)s * kD)) : make_uint4(0, 0, 0, 0);
      }
    };
    // A register batch is 32 KB per CTA, less than the bytes that have to be on their way to keep the memory busy (a
    // loaded DRAM round trip is about 2K cycles: 15 B/clk per SM), so a thread asks for the rows four batches ahead to
    // be brought into L2, whose round trip is a third of that.
    auto ahead = [&](int base) {
      const int n = min(nloc - base, HW * R);
      if (tid == 0 && n > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                         c.KR + ((unit * c.Hkv + gk) * (size_t)c.cap + lo + base) * kD),
                     "r"(n * kD * 2)
                     : "memory");
    };
    uint4 cur[R], nxt[R];
    fetch(0, cur);
#pragma unroll
    for (int i = 1; i <= kStAhead; ++i) ahead(i * HW * R);
    if (tid < kD) {
      const __nv_bfloat16* qp = q + (qrow + (size_t)gk * c.G) * kD + tid;
      float acc = 0.f;
      for (int hh = 0; hh < c.G; ++hh)
        if (rh < 0 || gk * c.G + hh == rh) acc += __bfloat162float(qp[(size_t)hh * kD]);
      su[tid] = acc;
    }
    if (tid == 0) s_cnt = 0;
    hist[tid] = 0;
    r_hist[tid] = 0;
    __syncthreads();
    unsigned kmax = 0u;
    {
      float2 uf[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) uf[e] = make_float2(su[hl * 8 + 2 * e], su[hl * 8 + 2 * e + 1]);
      float* sc = c.scores + (unit * c.Hkv + g) * (size_t)c.cap + lo;
      // the eight rows are reduced over the sixteen lanes together: a lane passes half of its partial sums on in every
      // step (8 shuffles instead of 32) and ends with the score of row myrow (lanes 2i and 2i + 1 hold the same one)
      const bool h8 = hl & 8, h4 = hl & 4, h2 = hl & 2;
      const int myrow = (h8 ? 4 : 0) + (h4 ? 2 : 0) + (h2 ? 1 : 0);
      for (int base = 0; base < nloc; base += HW * R) {  // uniform trip count (shuffles inside)
        fetch(base + HW * R, nxt);                       // past the end: zeros, no loads
        ahead(base + (kStAhead + 1) * HW * R);
        float d[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
          const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&cur[t]);
          float2 a2 = __fmul2_rn(uf[0], __bfloat1622float2(p2[0]));
#pragma unroll
          for (int i = 1; i < 4; ++i) a2 = __ffma2_rn(uf[i], __bfloat1622float2(p2[i]), a2);
          d[t] = a2.x + a2.y;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float give = h8 ? d[i] : d[i + 4];
          d[i] = (h8 ? d[i + 4] : d[i]) + __shfl_xor_sync(0xffffffffu, give, 8);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float give = h4 ? d[i] : d[i + 2];
          d[i] = (h4 ? d[i + 2] : d[i]) + __shfl_xor_sync(0xffffffffu, give, 4);
        }
        {
          const float give = h2 ? d[0] : d[1];
          d[0] = (h2 ? d[1] : d[0]) + __shfl_xor_sync(0xffffffffu, give, 2);
        }
        const float mine = d[0] + __shfl_xor_sync(0xffffffffu, d[0], 1);
        const int s = base + myrow * HW + hw;
        if (!(hl & 1) && s < nloc) {
          sc[s] = mine;
          const unsigned key = order_key(mine);
          kmax = max(kmax, key);
          if (U == 0) {
            if (s < key_slots) sck[s] = key;  // (the launch gives every slice room; never index past it)
          } else {
            const int st = c.span_start[unit * c.cap + lo + s], ln = c.span_len[unit * c.cap + lo + s];
            for (int u = max(st / U - u0, 0); u <= min((st + ln - 1) / U - u0, Nu - 1); ++u) atomicMax(&sck[u], key);
          }
        }
#pragma unroll
        for (int t = 0; t < R; ++t) cur[t] = nxt[t];
      }
    }
    // the rest of this CTA's share of the recent tokens comes into L2 while the cluster selects
    if (tid == 0) {
      const int v0 = max(tA0, a0);
      if (v0 < tA1) {
        const size_t row = (size_t)slab_row(c, rb + (v0 - a0), b.shift[bi]);
        for (const __nv_bfloat16* slab : {Kslab, Vslab})
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(slab + row * kD), "r"((tA1 - v0) * kD * 2)
                       : "memory");
      }
    }
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) s_scan[warp] = (int)kmax;
    load_q();
    __syncthreads();
    cluster.barrier_wait();  // every CTA of the cluster runs
    int cnt = 0;
    // ascending order of the s_cnt ids a select left in s_ids
    auto sort_ids = [&](int K) {
      __syncthreads();
      const int n = min(s_cnt, K);
      int myid = -1, rk = 0;
      if (tid < n) {
        myid = s_ids[tid];
        for (int t = 0; t < n; ++t) rk += s_ids[t] < myid;
      }
      __syncthreads();
      if (tid < n) s_ids[rk] = myid;
      __syncthreads();
      return n;
    };
    auto take_all = [&](int n) {
      for (int t = tid; t < n; t += nt) s_ids[t] = t;
      if (tid == 0) s_cnt = n;
    };
    if (U == 0) {
      const int K = min(c.topk, nsp);
      const int cap = kStList / S;
      unsigned bcut = 255u, M16 = 0xffffu;  // (K == nsp: every span is a candidate)
      bool general = false;
      if (K < nsp) {
        if (tid < S) {
          unsigned m = 0u;
#pragma unroll
          for (int w = 0; w < kStWarps; ++w) m = max(m, (unsigned)s_scan[w]);
          *cluster.map_shared_rank(&r_max[rank], tid) = m;
        }
        cluster.sync();
        unsigned m = 0u;
        for (int t = 0; t < S; ++t) m = max(m, r_max[t]);
        M16 = m >> 16;
        // how far the upper 16 bits of the keys lie below those of the largest (dist_bin), counted here and added to every
        // CTA's total; few bins hold anything
        for (int s = tid; s < nloc; s += nt) {
          const unsigned d = dist_bin(M16 - (sck[s] >> 16));
          if (d < 255u) atomicAdd(&hist[d], 1u);
        }
        if (tid == 0) s_cut = 255;
        __syncthreads();
        if (const unsigned n = hist[tid])
          for (int t = 0; t < S; ++t) atomicAdd(cluster.map_shared_rank(&r_hist[tid], t), n);
        cluster.sync();
        const unsigned tot = r_hist[tid];
        // the first bin at which the running count reaches K
        unsigned inc = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += t;
        }
        if (lane == 31) s_scan[32 + warp] = (int)inc;
        __syncthreads();
        for (int w = 0; w < warp; ++w) inc += (unsigned)s_scan[32 + w];
        if (inc >= (unsigned)K && inc - tot < (unsigned)K) s_cut = tid;
        __syncthreads();
        bcut = (unsigned)s_cut;
        general = bcut >= 255u;  // the K-th key lies further below (the same decision in every CTA)
      }
      if (!general) {
        // the candidates go to every CTA of the cluster
        const unsigned dcut = dist_last(bcut);
        for (int s = tid; s < nloc; s += nt) {
          const unsigned key = sck[s];
          if (M16 - (key >> 16) <= dcut) {
            const int j = atomicAdd(&s_cnt, 1);
            if (j < cap) {
              const unsigned long long e = ((unsigned long long)key << 32) | (unsigned)~(lo + s);
              for (int t = 0; t < S; ++t) cluster.map_shared_rank(s_list, t)[rank * cap + j] = e;
            }
          }
        }
        __syncthreads();
        if (tid < S) *cluster.map_shared_rank(&r_cnt[rank], tid) = s_cnt;
        cluster.sync();
        int nc = 0, most = 0;  // all candidates, the longest list
        for (int t = 0; t < S; ++t) {
          const int n = r_cnt[t];
          most = max(most, n);
          nc += n;
        }
        general = most > cap || nc > kStCand;  // many equal scores
        if (!general) {
          for (int t = warp; t < S; t += kStWarps) {  // the lists behind each other
            int at = 0;
            for (int w = 0; w < t; ++w) at += r_cnt[w];
            for (int j = lane; j < r_cnt[t]; j += 32) s_rank[at + j] = s_list[t * cap + j];
          }
          __syncthreads();
          int rk = 0x7fffffff;
          unsigned long long mine = 0;
          if (tid < nc) {
            mine = s_rank[tid];
            rk = 0;
            for (int i = 0; i < nc; ++i) rk += s_rank[i] > mine;
          }
          const int id = (int)~(unsigned)mine;
          if (rk < K) s_scan[rk] = id;
          __syncthreads();
          if (rk < K) {
            int at = 0;
            for (int i = 0; i < K; ++i) at += s_scan[i] < id;
            s_ids[at] = id;
          }
          cnt = K;
        }
      }
      if (general) {
        // this CTA's best k of its slice in ascending id order, then the best k of the cluster's lists, which take the place of
        // the candidates' (their last remote writes lie before the cluster barrier that counted them)
        if (tid == 0) s_cnt = 0;
        __syncthreads();
        const int cf = min(c.topk, per);  // candidates of every full slice
        const int kl = min(c.topk, nloc);
        if (kl == nloc)
          take_all(nloc);
        else
          radix_select_top<unsigned, 0>([&](int i) { return sck[i]; }, nloc, kl, hist, &s_prefix, &s_need, s_scan, &s_cnt,
                                        s_ids);
        const int n = sort_ids(kl);
        if (tid < n) {
          l_key[tid] = sck[s_ids[tid]];
          l_id[tid] = lo + s_ids[tid];
        }
        cluster.sync();
        // slices in front of a non-empty one are full, so the candidates of rank t start at t * cf; the ids ascend
        // with the list index, so "lower index first" among equal keys is "lower id first"
        int NG = 0;
        for (int t = 0; t < S; ++t) NG += min(c.topk, max(0, min(per, nsp - t * per)));
        for (int i = tid; i < NG; i += nt) {
          const int t = i / cf, j = i - t * cf;
          g_key[i] = cluster.map_shared_rank(l_key, t)[j];
          g_id[i] = cluster.map_shared_rank(l_id, t)[j];
        }
        if (tid == 0) s_cnt = 0;
        __syncthreads();
        if (K == NG)
          take_all(NG);
        else
          radix_select_top<unsigned, 0>([&](int i) { return g_key[i]; }, NG, K, hist, &s_prefix, &s_need, s_scan, &s_cnt,
                                        s_ids);
        cnt = sort_ids(K);
        int id = 0;
        if (tid < cnt) id = g_id[s_ids[tid]];
        __syncthreads();
        if (tid < cnt) s_ids[tid] = id;
      }
    } else {
      cluster.sync();
      for (int i = tid; i < Nu; i += nt) {
        unsigned key = 0u;
#pragma unroll
        for (int t = 0; t < kStMaxCluster; ++t)
          if (t < S) key = max(key, cluster.map_shared_rank(sck, t)[i]);
        utot[i] = key;
      }
      __syncthreads();
      const int K = min(c.topk, Nu);
      if (K == Nu)
        take_all(Nu);
      else
        radix_select_top<unsigned, 4>([&](int i) { return utot[i]; }, Nu, K, hist, &s_prefix, &s_need, s_scan, &s_cnt,
                                      s_ids, s_ckey);
      cnt = sort_ids(K);
      if (tid < cnt) s_ids[tid] += u0;  // absolute unit ids
    }
    __syncthreads();
    nall = cnt;
    if (rank == S - 1) {
      int* sel = c.sel + (unit * c.Hkv + g) * (size_t)c.topk;
      for (int t = tid; t < c.topk; t += nt) sel[t] = t < cnt ? s_ids[t] : -1;
    }
    if (c.persist) {
      nall = union_with_persistent(c, unit, g, s_ids, cnt, s_scan, s_all);
      ids_all = s_all;
    }
    if (tid < nall) {
      if (U > 0) {  // the unit's tokens inside the indexed range
        const int st = max(ids_all[tid] * U, c.Ls);
        s_sst[tid] = st;
        s_sln[tid] = min((ids_all[tid] + 1) * U, loc_begin) - st;
      } else {
        s_sst[tid] = c.span_start[unit * c.cap + ids_all[tid]];
        s_sln[tid] = c.span_len[unit * c.cap + ids_all[tid]];
      }
    }
  } else {
    load_q();
    if (rank == S - 1) {
      int* sel = c.sel + (unit * c.Hkv + g) * (size_t)c.topk;
      for (int t = tid; t < c.topk; t += nt) sel[t] = -1;
    }
    cluster.barrier_wait();
  }
  __syncthreads();
  if (c.host_kv && nall > 0) {
    // the first CTA looks the units up and assigns the slots, the cluster shares the pulls of the missing ones
    if (rank == 0)
      unit_cache_policy(c, unit, g, ids_all, nall, 0x7fffffff, s_tag, s_sco, s_named, s_src, s_fill);
    cluster.sync();
    if (tid < nall && rank > 0) {
      s_src[tid] = cluster.map_shared_rank(s_src, 0)[tid];
      s_fill[tid] = cluster.map_shared_rank(s_fill, 0)[tid];
    }
    __syncthreads();
    for (int t = rank; t < nall; t += S)
      if (s_fill[t]) pull_unit(c, unit, g, ids_all[t], s_src[t], s_sst[t], s_sln[t]);
    cluster.sync();  // (orders the pulled rows before the cluster's reads)
  }
  // ranges of the selected tokens and the prefix of their lengths
  if (nall == 0) {  // (the same in every CTA)
    if (tid == 0) s_rp[0] = s_nr = 0;
  } else if (warp == 0) {
    int nr = nall;
    if (U == 0 && (c.phi_milli > 0 || c.phi_l)) {  // kept spans may overlap: every token once
      nr = merge_ranges_warp(
          nall,
          [&](int i, int& st, int& ln) {
            st = s_sst[i];
            ln = s_sln[i];
          },
          s_rs, s_rl);
    } else {
      for (int i = lane; i < nall; i += 32) {
        // (host-memory pager: the range starts at a row of the unit cache)
        s_rs[i] = c.host_kv ? (int)((unit * c.Hkv + g) * (size_t)c.cache_units + s_src[i]) * U + (s_sst[i] - ids_all[i] * U)
                            : s_sst[i];
        s_rl[i] = s_sln[i];
      }
      __syncwarp();
    }
    int run = 0;
    for (int base = 0; base < nr; base += 32) {
      const int i = base + lane;
      const int v = i < nr ? s_rl[i] : 0;
      int inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (i < nr) s_rp[i] = run + inc - v;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) {
      s_rp[nr] = run;
      s_nr = nr;
    }
  }
  if (rank == S - 1 && warp == 1) {
    long long tokens = 0;
    for (int t = lane; t < nall; t += 32) tokens += s_sln[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tokens += shfl_xor_ll(tokens, o);
    if (lane == 0) c.sel_tokens[unit * c.Hkv + g] = tokens;  // (summed over the KV heads by ltri_get_stats)
  }
  __syncthreads();

  // ---- attention: the CTA's share of the sink and recent tokens, then of the selected ones
  const int nB = s_rp[s_nr], perB = (nB + S - 1) / S;
  const int tB0 = min(nB, rank * perB), tB1 = min(nB, tB0 + perB);
  const int ntiles = ntA + (tB1 - tB0 + kDTile - 1) / kDTile;
  const __nv_bfloat16* Ksel = c.host_kv ? c.Kcache : Kslab;  // what the ranges' rows are counted from
  const __nv_bfloat16* Vsel = c.host_kv ? c.Vcache : Vslab;
  int ri = 0;  // range of this lane's last row (a warp's tiles ascend)
  auto any_row = [&](int t) {
    if (t < ntA) return known_row(t);
    const int v = tB0 + (t - ntA) * kDTile + ch;
    if (v >= tB1) return kNoRow;
    while (v >= s_rp[ri + 1]) ++ri;
    return s_rs[ri] + (v - s_rp[ri]);
  };
  auto issue = [&](int t, int rows, bool values) {
    copy_rows(rows, t < ntA ? (values ? Vslab : Kslab) : (values ? Vsel : Ksel), (values ? vnew : knew) + nrow * kD,
              values ? sv : sk);
  };
  // One tile buffer per warp: the next K rows are requested as soon as the tile's logits are formed, the next V rows
  // after its P.V product, so that one of the two is always on its way (a second buffer would cost the second CTA).
  const int my_tiles = ntiles > warp ? (ntiles - warp + kStWarps - 1) / kStWarps : 0;
  if (!early && my_tiles > 0) {
    const int rows = any_row(warp);
#pragma unroll 1
    for (int kv = 0; kv < 2; ++kv) {
      issue(warp, rows, kv != 0);
      cp_async_commit();
    }
  }
  const float c2 = c.scale * kLog2eD;
  DecAcc acc;
  acc.clear();
  for (int it = 0; it < my_tiles; ++it) {
    const int t = warp + kStWarps * it, next = t + kStWarps;
    const int left = t < ntA ? (tA1 - tA0) - t * kDTile : (tB1 - tB0) - (t - ntA) * kDTile;
    cp_async_wait<1>();
    __syncwarp();
    float Sl[2][4];
    dec_tile_logits(Sl, qa, sk, lane);
    __syncwarp();
    int rows = kNoRow;
    if (next < ntiles) {
      rows = any_row(next);
      issue(next, rows, false);
    }
    cp_async_commit();
    uint32_t pa[4];
    dec_tile_softmax(acc, Sl, pa, left, c2, lane);
    cp_async_wait<1>();
    __syncwarp();
    dec_tile_values(acc, pa, sv, lane);
    __syncwarp();
    if (next < ntiles) issue(next, rows, true);
    cp_async_commit();
  }
  cp_async_wait<0>();
  acc.lsum += __shfl_xor_sync(0xffffffffu, acc.lsum, 1);
  acc.lsum += __shfl_xor_sync(0xffffffffu, acc.lsum, 2);
  __syncthreads();  // every warp is done with the ring: it now holds the warps' partial softmaxes
  float* w_o = reinterpret_cast<float*>(dsm);  // [warp][G][128]
  float* w_m = w_o + kStWarps * G * kD;        // [warp][G]
  float* w_l = w_m + kStWarps * G;
  if (r < G) {
    if (qd == 0) {
      w_m[warp * G + r] = acc.m;
      w_l[warp * G + r] = acc.lsum;
    }
#pragma unroll
    for (int n8 = 0; n8 < 16; ++n8)
      *reinterpret_cast<float2*>(&w_o[(warp * G + r) * kD + n8 * 8 + 2 * qd]) = make_float2(acc.O[n8][0], acc.O[n8][1]);
  }
  __syncthreads();
  const int share = G * kD / S;  // outputs of the unit that a CTA of the cluster writes (S divides 128)
  for (int idx = tid; idx < G * kD; idx += nt) {
    const int hh = idx / kD, e = idx % kD;
    float mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < kStWarps; ++w) mx = fmaxf(mx, w_m[w * G + hh]);
    float lt = 0.f, ot = 0.f;
#pragma unroll
    for (int w = 0; w < kStWarps; ++w) {
      const float mw = w_m[w * G + hh];
      const float sc = mw == -INFINITY ? 0.f : exp2f(mw - mx);
      lt += w_l[w * G + hh] * sc;
      ot += w_o[(w * G + hh) * kD + e] * sc;
    }
    const int to = idx / share;
    cluster.map_shared_rank(r_o, to)[rank * share + idx - to * share] = ot;
    if (e < S) *cluster.map_shared_rank(&r_ml[rank][hh], e) = make_float2(mx, lt);
  }
  if (appends) {
    const long long wrow = c.paged ? pos - b.shift[bi] : pos;
    __nv_bfloat16* slab = (lane < 16 ? c.Kc : c.Vc) + (unit * c.Hkv + g) * (size_t)c.SR * kD + ch * 8;
    if (wrow < 0 || wrow >= c.SR) {  // cannot happen: the host keeps the window inside the slab
      set_status(c, -2, pos);
    } else {
      *reinterpret_cast<uint4*>(slab + wrow * kD) = new_row;
      if (c.paged && pos < c.Ls) *reinterpret_cast<uint4*>(slab + (size_t)pos * kD) = new_row;  // the sink's permanent row
    }
    if (g == 0 && lane == 0) c.votes[unit * c.Tpad + pos] = 0;
  }
  cluster.sync();  // (from here on a CTA reads its own shared memory only)
  for (int i = tid; i < share; i += nt) {
    const int idx = rank * share + i, hh = idx / kD, e = idx % kD;
    float mx = -INFINITY;
    for (int s = 0; s < S; ++s) mx = fmaxf(mx, r_ml[s][hh].x);
    float lt = 0.f, ot = 0.f;
    for (int s = 0; s < S; ++s) {
      const float2 ml = r_ml[s][hh];
      const float sc = ml.x == -INFINITY ? 0.f : exp2f(ml.x - mx);
      lt += ml.y * sc;
      ot += r_o[s * share + i] * sc;
    }
    out[(qrow + (size_t)g * G + hh) * kD + e] = __float2bfloat16(ot / lt);
  }
}

typedef void (*DecStepFn)(DevCtx, int, DecBatch, int, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                          __nv_bfloat16*, int);
static DecStepFn dec_step_fn(int G) {
  return G == 1 ? k_dec_step<1> : G == 2 ? k_dec_step<2> : G == 4 ? k_dec_step<4> : k_dec_step<8>;
}

cudaError_t prepare_dec_step(const DevCtx& c) {
  const DecStepFn fn = dec_step_fn(c.G);
  return first_error(allow_smem(fn, dec_step_smem(kStMaxSlots)),
                     cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
}

// CTAs of k_dec_step that fit the GPU at once as clusters of `cluster` CTAs (after prepare_dec_step).
int dec_step_capacity(const DevCtx& c, int cluster) {
  return cluster * active_clusters(dec_step_fn(c.G), cluster, kStThreads, dec_step_smem(kStMaxSlots));
}

// order keys a CTA of the cluster needs: its slice of the spans, or two tables of the units of the indexed range
static long long dec_step_slots(const DevCtx& c, int span_bound, int indexed_end, int cluster) {
  if (c.unit > 0) return 2ll * (indexed_end / c.unit + 2);
  return ((long long)span_bound + cluster - 1) / cluster;
}

bool dec_step_fits(const DevCtx& c, int span_bound, int indexed_end, int cluster) {
  return dec_step_slots(c, span_bound, indexed_end, cluster) <= kStMaxSlots;
}

cudaError_t launch_dec_step(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count, const __nv_bfloat16* q,
                            const __nv_bfloat16* k, const __nv_bfloat16* v, __nv_bfloat16* out, int span_bound,
                            int indexed_end, int cluster, cudaStream_t s) {
  const int slots = (int)((dec_step_slots(c, span_bound, indexed_end, cluster) + 31) / 32 * 32);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster, c.Hkv, b.n * layer_count);
  cfg.blockDim = dim3(kStThreads);
  cfg.dynamicSmemBytes = dec_step_smem(slots);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, dec_step_fn(c.G), c, layer_begin, b, layer_count, q, k, v, out, slots);
}

}  // namespace ltri
