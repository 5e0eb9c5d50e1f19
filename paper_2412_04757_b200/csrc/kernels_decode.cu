// Decode attention (Sec. 3.5: while decoding, the current block is one token): memory-bound split-KV flash-decoding over the
// token ranges [sink | selected spans | tokens since the last eviction].  Every K/V row is read once with 16-byte
// loads and shared by the G query heads of its KV group; softmax reductions use warp shuffles.
#include "common.cuh"
#include "decode_util.cuh"

namespace ltri {

constexpr int kDecThreads = 128;  // 4 warps = 8 half-warps, each half-warp owns one token at a time

// grid (nsplit, Hkv, b.n*layer_count), 4 warps.  Each warp walks 16-token tiles of the CTA's slice of the virtual
// token list (sink | selected spans | recent tokens): the tile's K and V rows (two contiguous 256-byte rows per
// cp.async instruction, 16 bytes per lane) land in a warp-private, XOR-swizzled 2-stage ring; QK^T and PV run as
// m16n8k16 tensor-core MMAs with the G query heads of the group in the first rows of the 16-row operand, so the
// per-token ALU cost is a handful of instructions and the kernel stays bound by the K/V stream.
// Partial results (m, l, O[128]) per (unit, head, split) go to dec_part.
constexpr int kDStages = 2;     // two stages of 8 KB per warp: three CTAs (12 warps) fit an SM, which hides more latency
constexpr int kDecCtasPerSm = 3;  // than a deeper ring at two CTAs per SM
constexpr int kDWarpBytes = kDStages * 2 * kDTile * 256;  // K and V rows of every stage

template <int G>
__global__ void __launch_bounds__(kDecThreads, kDecCtasPerSm) k_decode_attn(DevCtx c, DecBatch b, int layer_begin, int layer_count,
                                                                const __nv_bfloat16* __restrict__ q, int nsplit) {
  chain_wait();
  extern __shared__ __align__(1024) unsigned char dsm[];
  // rs: first token of every range -- in a paged context (host-memory pager) its first K row, counted from the start
  // of the K slabs, instead: there a range lives in a sliding slab or in a slot of the unit cache
  __shared__ int rs[kMaxRanges], rp[kMaxRanges + 1];
  __shared__ float sm_m[4][G], sm_l[4][G];
  __shared__ float sm_o[4][G][kD];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x, g = blockIdx.y;
  const int bi = blockIdx.z / layer_count, l = blockIdx.z % layer_count, layer = layer_begin + l;
  const size_t unit = unit_of(c, b.seq[bi], layer);
  const size_t rb = (unit * c.Hkv + g) * (size_t)c.rcap;
  const int nr = min(c.rng_cnt[unit * c.Hkv + g], c.rcap);
  // (a warp reads 32 ranges at a time and adds up their lengths: one thread reading one range after the other took as long as
  // several tiles, in every CTA)
  if (warp == 0) {
    int run = 0;
    for (int base = 0; base < nr; base += 32) {
      const int i = base + lane;
      const int start = i < nr ? (c.host_kv ? (int)c.rng_koff[rb + i] : c.rng_start[rb + i]) : 0;
      const int len = i < nr ? c.rng_len[rb + i] : 0;
      int inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (i < nr) {
        rs[i] = start;
        rp[i] = run + inc - len;
      }
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) rp[nr] = run;
  }
  __syncthreads();
  const int total = rp[nr];
  const int per = (total + nsplit - 1) / nsplit;
  const int v0 = split * per, v1 = min(total, v0 + per);
  const int ntiles = v1 > v0 ? (v1 - v0 + kDTile - 1) / kDTile : 0;

  // query fragments: rows 0..G-1 of the 16-row A operand are the heads of the group, the rest are zero
  const int r = lane >> 2, qd = lane & 3;
  uint32_t qa[8][2];
  {
    const __nv_bfloat16* qp = q + (((size_t)b.src[bi] * layer_count + l) * c.Hq + (size_t)g * G + (r < G ? r : 0)) * kD;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      qa[ks][0] = r < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 2 * qd) : 0u;
      qa[ks][1] = r < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8 + 2 * qd) : 0u;
    }
  }
  // (resident contexts: row = token; paged contexts address every range through rko / rvo below)
  const __nv_bfloat16* Kslab = c.Kc + (unit * c.Hkv + g) * (size_t)c.SR * kD;
  const __nv_bfloat16* Vslab = c.Vc + (unit * c.Hkv + g) * (size_t)c.SR * kD;
  const size_t cache_k0 = c.host_kv ? (size_t)((c.Kcache - c.Kc) / kD) : 0;
  const size_t cache_dv = c.host_kv ? (size_t)((c.Vcache - c.Vc) / kD) - cache_k0 : 0;
  const uint32_t wbase = smem_u32(dsm) + warp * kDWarpBytes;
  const float c2 = c.scale * kLog2eD;

  // this lane copies rows (lane>>4) + 2i of every tile, 16 bytes at chunk (lane&15)
  int ri = 0;  // range of this lane's last row: at first that of the warp's first token
  for (int base = 0; base < nr; base += 32)
    ri += __popc(__ballot_sync(0xffffffffu, base + lane < nr && rp[base + lane + 1] <= v0 + warp * kDTile));
  ri = min(ri, max(nr - 1, 0));
  const int ch = lane & 15;
  auto issue = [&](int t, int stage) {
    const uint32_t sk = wbase + stage * (2 * kDTile * 256), sv = sk + kDTile * 256;
    const int vb = v0 + t * kDTile;
#pragma unroll
    for (int i = 0; i < kDTile / 2; ++i) {
      const int row = 2 * i + (lane >> 4);
      const int v = vb + row;
      const bool okr = v < v1;
      size_t tok = 0;
      if (okr) {
        while (v >= rp[ri + 1]) ++ri;
        tok = (size_t)(rs[ri] + (v - rp[ri]));
      }
      const __nv_bfloat16* kp = Kslab + tok * kD;
      const __nv_bfloat16* vp = Vslab + tok * kD;
      if (c.host_kv) {
        // tok is a K row counted from c.Kc; its V row has the same number counted from c.Vc inside the slabs and is
        // cache_dv rows further inside the unit caches
        kp = c.Kc + tok * kD;
        vp = c.Vc + (tok >= cache_k0 ? tok + cache_dv : tok) * kD;
      }
      cp_async16(sk + tile_off(row, ch), kp + ch * 8, okr ? 16 : 0);
      cp_async16(sv + tile_off(row, ch), vp + ch * 8, okr ? 16 : 0);
    }
  };

  DecAcc acc;
  acc.clear();

  // tiles of this warp: warp, warp + 4, ...
  const int my_tiles = ntiles > warp ? (ntiles - warp + 3) / 4 : 0;
#pragma unroll
  for (int s = 0; s < kDStages - 1; ++s) {
    if (s < my_tiles) issue(warp + 4 * s, s);
    cp_async_commit();
  }
  for (int it = 0; it < my_tiles; ++it) {
    const int stage = it % kDStages;
    if (it + kDStages - 1 < my_tiles) issue(warp + 4 * (it + kDStages - 1), (it + kDStages - 1) % kDStages);
    cp_async_commit();
    cp_async_wait<kDStages - 1>();
    __syncwarp();
    const uint32_t sk = wbase + stage * (2 * kDTile * 256), sv = sk + kDTile * 256;
    const int vb = v0 + (warp + 4 * it) * kDTile;
    dec_tile_16(acc, qa, sk, sv, v1 - vb, c2, lane);
    __syncwarp();
  }
  cp_async_wait<0>();
  acc.lsum += __shfl_xor_sync(0xffffffffu, acc.lsum, 1);
  acc.lsum += __shfl_xor_sync(0xffffffffu, acc.lsum, 2);
  if (r < G) {
    if (qd == 0) {
      sm_m[warp][r] = acc.m;
      sm_l[warp][r] = acc.lsum;
    }
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) {
      sm_o[warp][r][nt * 8 + 2 * qd] = acc.O[nt][0];
      sm_o[warp][r][nt * 8 + 2 * qd + 1] = acc.O[nt][1];
    }
  }
  __syncthreads();
  for (int idx = tid; idx < G * kD; idx += kDecThreads) {
    const int hh = idx / kD, e = idx % kD;
    float mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < 4; ++w) mx = fmaxf(mx, sm_m[w][hh]);
    float lt = 0.f, ot = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float sc = sm_m[w][hh] == -INFINITY ? 0.f : exp2f(sm_m[w][hh] - mx);
      lt += sm_l[w][hh] * sc;
      ot += sm_o[w][hh][e] * sc;
    }
    float* part = c.dec_part + ((unit * c.Hq + g * G + hh) * (size_t)kMaxDecSplit + split) * (kD + 2);
    part[e] = ot;
    if (e == 0) {
      part[kD] = mx;
      part[kD + 1] = lt;
    }
  }
}

// merge of the split partials: grid (Hq, b.n*layer_count), 128 threads (one per output dim).
__global__ void __launch_bounds__(kD) k_decode_merge(DevCtx c, DecBatch b, int layer_begin, int layer_count,
                                                     __nv_bfloat16* __restrict__ out, int nsplit) {
  chain_wait();
  const int h = blockIdx.x, e = threadIdx.x;
  const int bi = blockIdx.y / layer_count, l = blockIdx.y % layer_count;
  const size_t unit = unit_of(c, b.seq[bi], layer_begin + l);
  const float* part = c.dec_part + (unit * c.Hq + h) * (size_t)kMaxDecSplit * (kD + 2);
  float mx = -INFINITY;
  for (int s = 0; s < nsplit; ++s) mx = fmaxf(mx, part[(size_t)s * (kD + 2) + kD]);
  float lt = 0.f, ot = 0.f;
  for (int s = 0; s < nsplit; ++s) {
    const float ms = part[(size_t)s * (kD + 2) + kD];
    const float sc = ms == -INFINITY ? 0.f : exp2f(ms - mx);
    lt += part[(size_t)s * (kD + 2) + kD + 1] * sc;
    ot += part[(size_t)s * (kD + 2) + e] * sc;
  }
  out[(((size_t)b.src[bi] * layer_count + l) * c.Hq + h) * kD + e] = __float2bfloat16(ot / lt);
}

constexpr int kDecSmem = 4 * kDWarpBytes;

cudaError_t prepare_decode(const DevCtx& c) {
  switch (c.G) {
    case 1: return allow_smem(k_decode_attn<1>, kDecSmem);
    case 2: return allow_smem(k_decode_attn<2>, kDecSmem);
    case 4: return allow_smem(k_decode_attn<4>, kDecSmem);
    case 8: return allow_smem(k_decode_attn<8>, kDecSmem);
  }
  return cudaErrorInvalidValue;
}

template <int G>
static cudaError_t launch_dec_g(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count,
                                const __nv_bfloat16* q, __nv_bfloat16* out, int nsplit, cudaStream_t s) {
  const cudaError_t e = launch_chained(k_decode_attn<G>, dim3(nsplit, c.Hkv, b.n * layer_count), dim3(kDecThreads), kDecSmem,
                                       s, c, b, layer_begin, layer_count, q, nsplit);
  if (e != cudaSuccess) return e;
  return launch_chained(k_decode_merge, dim3(c.Hq, b.n * layer_count), dim3(kD), 0, s, c, b, layer_begin, layer_count, out,
                        nsplit);
}

cudaError_t launch_decode_attn(const DevCtx& c, const DecBatch& b, int layer_begin, int layer_count, int,
                               const __nv_bfloat16* q, __nv_bfloat16* out, int nsplit, cudaStream_t s) {
  switch (c.G) {
    case 1: return launch_dec_g<1>(c, b, layer_begin, layer_count, q, out, nsplit, s);
    case 2: return launch_dec_g<2>(c, b, layer_begin, layer_count, q, out, nsplit, s);
    case 4: return launch_dec_g<4>(c, b, layer_begin, layer_count, q, out, nsplit, s);
    case 8: return launch_dec_g<8>(c, b, layer_begin, layer_count, q, out, nsplit, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ltri
