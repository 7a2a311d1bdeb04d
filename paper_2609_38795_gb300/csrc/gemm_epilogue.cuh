// Store of a GEMM tile from tensor memory: C = acc or C += acc, fp32, row-major.
//
// A thread holds one tensor-memory lane, i.e. one row of the tile; written straight from there a
// warp's 16-byte accesses fall on 32 different rows, half a sector each, and the accumulating
// form waits for every one of its reads.  Each warp therefore turns 32 x 32 blocks around in its
// own 4 KB of shared memory (16-byte columns XOR-swizzled by the row, conflict-free both ways)
// and touches global memory as whole 128-byte lines, four rows per instruction; the accumulating
// form has the old values of the next two blocks in flight while it adds one, the first two
// already while the tile is being computed.  Bound by the 8 bytes per element of C when K is
// small: dW += H_d^T G at d = 4096, V = 151936 (5 GB of C) takes 1189 us with 128 rows and 1619
// us with 1920, against 2968 and 3242 us written straight from the lanes.
#pragma once

#include "kernels.h"
#include "tc_common.cuh"

namespace alr {

constexpr int kEpiBlock = 32;                          // rows and columns turned around at a time
constexpr int kEpiStageBytes = kEpiBlock * kEpiBlock * 4;   // per warp

// This lane's eight vectors of the 32 x 32 block of C whose first element is (m0, n0): row
// m0 + 4 i + lane / 8, columns n0 + 4 (lane % 8) ..+3 (Nc is a multiple of 4).
struct CBlock {
  float4 v[8];

  ALR_DEV void load(const GemmArgs& a, int m0, int n0, int lane) {
    const int m = m0 + (lane >> 3), n = n0 + 4 * (lane & 7);
    const float* p = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (m + 4 * i < a.M && n < a.Nc)
        v[i] = __ldcs(reinterpret_cast<const float4*>(p + size_t(4 * i) * size_t(a.ldc)));
  }
};

// A 32 x 32 block in shared memory: put row `lane` there, and the index of this lane's i-th
// vector of it (row 4 i + lane / 8, columns 4 (lane % 8) ..+3).
ALR_DEV void put_row(const uint32_t (&r)[32], uint8_t* stage, int lane) {
  float4* s = reinterpret_cast<float4*>(stage);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    s[lane * 8 + (j ^ (lane & 7))] =
        make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                    __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
}

ALR_DEV int block_vector(int i, int lane) {
  const int row = 4 * i + (lane >> 3);
  return row * 8 + ((lane & 7) ^ (row & 7));
}

// Write (kAcc: add) one block whose row `lane` this thread holds in r; `stage` is the warp's own.
template <bool kAcc>
ALR_DEV void store_block(const uint32_t (&r)[32], const CBlock& old, const GemmArgs& a, int m0,
                         int n0, uint8_t* stage, int lane) {
  const float4* s = reinterpret_cast<const float4*>(stage);
  put_row(r, stage, lane);
  __syncwarp();
  const int m = m0 + (lane >> 3), n = n0 + 4 * (lane & 7);
  float* p = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float4 v = s[block_vector(i, lane)];
    if (kAcc) {
      v.x += old.v[i].x;
      v.y += old.v[i].y;
      v.z += old.v[i].z;
      v.w += old.v[i].w;
    }
    if (m + 4 * i < a.M && n < a.Nc) {
      float4* q = reinterpret_cast<float4*>(p + size_t(4 * i) * size_t(a.ldc));
      if (kAcc) __stcs(q, v);
      else *q = v;
    }
  }
  __syncwarp();
}

// The old values of a warp's 32 x kCols strip of C, two blocks ahead of their use.
template <bool kAcc, int kCols>
struct CStrip {
  static constexpr int kBlocks = kCols / kEpiBlock;
  CBlock old[3];

  // Before the tile's accumulator is ready.
  ALR_DEV void begin(const GemmArgs& a, int m0, int n0, int lane) {
    if (kAcc) {
      old[0].load(a, m0, n0, lane);
      old[1].load(a, m0, n0 + kEpiBlock, lane);
    }
  }

  // The accumulator (tensor-memory address `taddr`, this warp's lanes) is ready; `release` is
  // called once it has been read.
  template <class Release>
  ALR_DEV void finish(const GemmArgs& a, int m0, int n0, uint32_t taddr, uint8_t* stage, int lane,
                      Release release) {
#pragma unroll
    for (int c = 0; c < kBlocks; ++c) {
      if (kAcc && c + 2 < kBlocks) old[(c + 2) % 3].load(a, m0, n0 + (c + 2) * kEpiBlock, lane);
      uint32_t r[32];
      tmem_ld32(taddr + c * kEpiBlock, r);
      tmem_ld_wait();
      reg_fence(r);
      if (c == kBlocks - 1) release();
      store_block<kAcc>(r, old[c % 3], a, m0, n0 + c * kEpiBlock, stage, lane);
    }
  }
};

// Split-K: each CTA of a cluster holds the partial sums of the same kRowBlocks x kColBlocks tile
// of 32 x 32 blocks in its own shared memory at `tile` (block (q, c) at q * kColBlocks + c).  The
// blocks are dealt over the CTAs and their warps; a block's sum is taken in CTA order, so the
// result does not depend on timing.  Blocks wholly outside C are neither put there nor read.
// Between cluster barriers.
template <bool kAcc, int kRowBlocks, int kColBlocks>
ALR_DEV void reduce_split(const GemmArgs& a, int m0, int n0, const uint8_t* tile, int rank,
                          int n_cta, int warp, int n_warps, int lane) {
  for (int b = rank + n_cta * warp; b < kRowBlocks * kColBlocks; b += n_cta * n_warps) {
    const int bm = m0 + (b / kColBlocks) * kEpiBlock, bn = n0 + (b % kColBlocks) * kEpiBlock;
    if (bm >= a.M || bn >= a.Nc) continue;
    CBlock old;
    if (kAcc) old.load(a, bm, bn, lane);
    float4 sum[8];
    for (int p = 0; p < n_cta; ++p) {
      const uint32_t base = cluster_smem_addr(tile + b * kEpiStageBytes, uint32_t(p));
      float4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = ld_cluster_v4(base + 16u * uint32_t(block_vector(i, lane)));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (p == 0) {
          sum[i] = v[i];
        } else {
          sum[i].x += v[i].x;
          sum[i].y += v[i].y;
          sum[i].z += v[i].z;
          sum[i].w += v[i].w;
        }
      }
    }
    const int m = bm + (lane >> 3), n = bn + 4 * (lane & 7);
    float* q = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (kAcc) {
        sum[i].x += old.v[i].x;
        sum[i].y += old.v[i].y;
        sum[i].z += old.v[i].z;
        sum[i].w += old.v[i].w;
      }
      if (m + 4 * i < a.M && n < a.Nc)
        *reinterpret_cast<float4*>(q + size_t(4 * i) * size_t(a.ldc)) = sum[i];
    }
  }
}

}  // namespace alr
