// One 16-token tile of the decode attention (Sec. 3.4 step 3 for a single query token), shared by the split-KV kernel
// and the one-launch decode step.
#pragma once

#include "common.cuh"
#include "mma_util.cuh"

namespace ltri {

constexpr float kLog2eD = 1.4426950408889634f;
constexpr int kDTile = 16;

// Running softmax state of one warp: row r = lane / 4 of the 16-row operand is head r of the KV group (r < G).
struct DecAcc {
  float O[16][4];
  float m, lsum;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 16; ++i) O[i][0] = O[i][1] = O[i][2] = O[i][3] = 0.f;
    m = -INFINITY;
    lsum = 0.f;
  }
};

// Logits of the tile's 16 tokens (K rows at sk, swizzled by tile_off): row r of a lane, tokens nt * 8 + 2 * qd + e.
__device__ __forceinline__ void dec_tile_logits(float (&S)[2][4], const uint32_t (&qa)[8][2], uint32_t sk, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i) S[i][0] = S[i][1] = S[i][2] = S[i][3] = 0.f;
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    uint32_t bf[4];
    ldsm_x4(bf, sk + tile_off((lane & 7) + ((lane >> 4) << 3), ks * 2 + ((lane >> 3) & 1)));
    const uint32_t a[4] = {qa[ks][0], 0u, qa[ks][1], 0u};
    mma_bf16(S[0], a, bf[0], bf[1]);
    mma_bf16(S[1], a, bf[2], bf[3]);
  }
}

// Moves the running maximum and row sum to include the tile's first `nvalid` tokens, rescales O and leaves the
// probabilities in pa (bf16 A operand of the P.V product).
__device__ __forceinline__ void dec_tile_softmax(DecAcc& acc, float (&S)[2][4], uint32_t (&pa)[4], int nvalid, float c2,
                                                 int lane) {
  const int qd = lane & 3;
  float tmax = -INFINITY;
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (nt * 8 + 2 * qd + e >= nvalid) S[nt][e] = -INFINITY;
      tmax = fmaxf(tmax, S[nt][e]);
    }
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 1));
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 2));
  const float mnew = fmaxf(acc.m, tmax * c2);
  const float mu = mnew == -INFINITY ? 0.f : mnew;
  const float alpha = exp2f(acc.m - mu);
  acc.m = mnew;
  float p[2][2];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) p[nt][e] = exp2f(fmaf(S[nt][e], c2, -mu));
  acc.lsum = acc.lsum * alpha + (p[0][0] + p[0][1] + p[1][0] + p[1][1]);
#pragma unroll
  for (int nt = 0; nt < 16; ++nt) {
    acc.O[nt][0] *= alpha;
    acc.O[nt][1] *= alpha;
  }
  pa[0] = pack_bf16(p[0][0], p[0][1]);
  pa[1] = 0u;
  pa[2] = pack_bf16(p[1][0], p[1][1]);
  pa[3] = 0u;
}

// O += P V for the tile's 16 tokens (V rows at sv, swizzled by tile_off).
__device__ __forceinline__ void dec_tile_values(DecAcc& acc, const uint32_t (&pa)[4], uint32_t sv, int lane) {
#pragma unroll
  for (int dp = 0; dp < 8; ++dp) {
    uint32_t bf[4];
    ldsm_x4_t(bf, sv + tile_off((lane & 7) + (((lane >> 3) & 1) << 3), dp * 2 + (lane >> 4)));
    mma_bf16(acc.O[2 * dp], pa, bf[0], bf[1]);
    mma_bf16(acc.O[2 * dp + 1], pa, bf[2], bf[3]);
  }
}

// Adds the tile's first `nvalid` tokens to the state.
__device__ __forceinline__ void dec_tile_16(DecAcc& acc, const uint32_t (&qa)[8][2], uint32_t sk, uint32_t sv, int nvalid,
                                            float c2, int lane) {
  float S[2][4];
  uint32_t pa[4];
  dec_tile_logits(S, qa, sk, lane);
  dec_tile_softmax(acc, S, pa, nvalid, c2, lane);
  dec_tile_values(acc, pa, sv, lane);
}

}  // namespace ltri
