// Store of a GEMM tile from tensor memory: C = acc or C += acc, fp32, row-major.
//
// A thread holds one tensor-memory lane, i.e. one row of the tile; written straight from there a
// warp's 16-byte accesses fall on 32 different rows, half a sector each, and the accumulating
// form waits for every one of its reads.  Each warp therefore turns 32 x 64 blocks around in its
// own 8 KB of shared memory (16-byte columns XOR-swizzled by the row, conflict-free both ways)
// and touches global memory in 256-byte row pieces, two rows per instruction.  The accumulating
// form has the old values of the next 16-row half in flight while it adds one, and where K is so
// small that C's traffic sets the time it asks for the next tile's rows, 1 KB each, to be brought
// into L2 a tile ahead (prefetch_row).
// Bound by the 8 bytes per element of C when K is small: dW += H_d^T G at d = 4096, V = 151936 (5
// GB of C) takes 922 us with 128 rows, against 2968 us written straight from the lanes, 1197 in
// 128-byte pieces without the L2 prefetch and 1002 with it, 1060 in 256-byte pieces without it.
// DRAM serves short pieces of scattered rows badly: the same traffic alone, without products,
// takes 1286, 980 and, in 256-byte pieces with the prefetch, 803 us; one stream over C takes 701.
// More reads in flight only queue up: 968 us with two halves ahead, 1044 with none, 1105 with
// eight epilogue warps.
#pragma once

#include "kernels.h"
#include "tc_common.cuh"

namespace alr {

constexpr int kEpiBlock = 32;                          // rows turned around at a time
constexpr int kEpiWide = 64;                           // and columns
constexpr int kEpiStageBytes = kEpiBlock * kEpiWide * 4;    // per warp

// This lane's eight vectors of a 16 x 64 piece of C whose first element is (m0, n0): row m0 + 2 i
// + lane / 16, columns n0 + 4 (lane % 16) ..+3 (Nc is a multiple of 4).
struct CPiece {
  float4 v[8];

  ALR_DEV void load(const GemmArgs& a, int m0, int n0, int lane) {
    const int m = m0 + (lane >> 4), n = n0 + 4 * (lane & 15);
    const float* p = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (m + 2 * i < a.M && n < a.Nc)
        v[i] = __ldcs(reinterpret_cast<const float4*>(p + size_t(2 * i) * size_t(a.ldc)));
  }
};

// Ask for this lane's row of a warp's 32-row strip of C, columns n0 .. n0 + cols, to be brought
// into L2 (Nc and n0 are multiples of 4, so the piece is whole 16-byte units).
ALR_DEV void prefetch_row(const GemmArgs& a, int m0, int n0, int cols, int lane) {
  const int m = m0 + lane, n = min(cols, a.Nc - n0);
  if (m < a.M && n > 0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                     a.C + size_t(m) * size_t(a.ldc) + size_t(n0)),
                 "r"(n * 4)
                 : "memory");
}

ALR_DEV float4 vec4(const uint32_t (&r)[32], int j) {
  return make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                     __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
}

// Columns 32 h .. 32 h + 31 of this lane's row of the 32 x 64 block, into the warp's staging.
ALR_DEV void put_half_row(const uint32_t (&r)[32], int h, uint8_t* stage, int lane) {
  float4* s = reinterpret_cast<float4*>(stage);
#pragma unroll
  for (int j = 0; j < 8; ++j) s[lane * 16 + 8 * h + (j ^ (lane & 7))] = vec4(r, j);
}

// Write (kAcc: add) rows 16 h .. 16 h + 15 of the staged block; (m0, n0): the piece's first
// element.
template <bool kAcc>
ALR_DEV void store_piece(const CPiece& old, const GemmArgs& a, int m0, int n0, int h,
                         const uint8_t* stage, int lane) {
  const float4* s = reinterpret_cast<const float4*>(stage);
  const int m = m0 + (lane >> 4), j = lane & 15, n = n0 + 4 * j;
  float* p = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = 16 * h + 2 * i + (lane >> 4);
    float4 v = s[row * 16 + (j ^ (row & 7))];
    if (kAcc) {
      v.x += old.v[i].x;
      v.y += old.v[i].y;
      v.z += old.v[i].z;
      v.w += old.v[i].w;
    }
    if (m + 2 * i < a.M && n < a.Nc) {
      float4* q = reinterpret_cast<float4*>(p + size_t(2 * i) * size_t(a.ldc));
      if (kAcc) __stcs(q, v);
      else *q = v;
    }
  }
}

// A warp's 32 x kCols strip of C, with its old values one piece ahead of their use.
template <bool kAcc, int kCols>
struct CStrip {
  static constexpr int kPieces = 2 * kCols / kEpiWide;
  CPiece old[2];

  ALR_DEV void load(int s, const GemmArgs& a, int m0, int n0, int lane) {
    old[s & 1].load(a, m0 + 16 * (s & 1), n0 + (s >> 1) * kEpiWide, lane);
  }

  // Before the tile's accumulator is ready.
  ALR_DEV void begin(const GemmArgs& a, int m0, int n0, int lane) {
    if (kAcc) load(0, a, m0, n0, lane);
  }

  // The accumulator (tensor-memory address `taddr`, this warp's lanes) is ready; `release` is
  // called once it has been read.
  template <class Release>
  ALR_DEV void finish(const GemmArgs& a, int m0, int n0, uint32_t taddr, uint8_t* stage, int lane,
                      Release release) {
#pragma unroll
    for (int s = 0; s < kPieces; ++s) {
      if (kAcc && s + 1 < kPieces) load(s + 1, a, m0, n0, lane);
      if ((s & 1) == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t r[32];
          tmem_ld32(taddr + (s >> 1) * kEpiWide + 32 * h, r);
          tmem_ld_wait();
          reg_fence(r);
          if (h == 1 && s + 2 == kPieces) release();
          put_half_row(r, h, stage, lane);
        }
        __syncwarp();
      }
      store_piece<kAcc>(old[s & 1], a, m0 + 16 * (s & 1), n0 + (s >> 1) * kEpiWide, s & 1, stage,
                        lane);
      if ((s & 1) == 1) __syncwarp();   // the staging is read before the next block goes in
    }
  }
};

// Split-K's partial sums: 32 x 32 blocks of 4 KB, this lane's row put there, and the index of this
// lane's i-th vector of a block (row 4 i + lane / 8, columns 4 (lane % 8) ..+3).
constexpr int kSplitBlock = 32;
constexpr int kSplitBlockBytes = kSplitBlock * kSplitBlock * 4;

ALR_DEV void put_row(const uint32_t (&r)[32], uint8_t* block, int lane) {
  float4* s = reinterpret_cast<float4*>(block);
#pragma unroll
  for (int j = 0; j < 8; ++j) s[lane * 8 + (j ^ (lane & 7))] = vec4(r, j);
}

ALR_DEV int block_vector(int i, int lane) {
  const int row = 4 * i + (lane >> 3);
  return row * 8 + ((lane & 7) ^ (row & 7));
}

// Split-K: each CTA of a cluster holds the partial sums of the same kRowBlocks x kColBlocks tile
// of 32 x 32 blocks in its own shared memory at `tile` (block (q, c) at q * kColBlocks + c).  The
// blocks are dealt over the CTAs and their warps; a block's sum is taken in CTA order, so the
// result does not depend on timing.  Blocks wholly outside C are neither put there nor read.
// Between cluster barriers.
template <bool kAcc, int kRowBlocks, int kColBlocks>
ALR_DEV void reduce_split(const GemmArgs& a, int m0, int n0, const uint8_t* tile, int rank,
                          int n_cta, int warp, int n_warps, int lane) {
  for (int b = rank + n_cta * warp; b < kRowBlocks * kColBlocks; b += n_cta * n_warps) {
    const int bm = m0 + (b / kColBlocks) * kSplitBlock, bn = n0 + (b % kColBlocks) * kSplitBlock;
    if (bm >= a.M || bn >= a.Nc) continue;
    const int m = bm + (lane >> 3), n = bn + 4 * (lane & 7);
    float* q = a.C + size_t(m) * size_t(a.ldc) + size_t(n);
    float4 sum[8], old[8];
    if (kAcc) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (m + 4 * i < a.M && n < a.Nc)
          old[i] = *reinterpret_cast<const float4*>(q + size_t(4 * i) * size_t(a.ldc));
    }
    for (int p = 0; p < n_cta; ++p) {
      const uint32_t base = cluster_smem_addr(tile + b * kSplitBlockBytes, uint32_t(p));
      float4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        v[i] = ld_cluster_v4(base + 16u * uint32_t(block_vector(i, lane)));
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
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (kAcc) {
        sum[i].x += old[i].x;
        sum[i].y += old[i].y;
        sum[i].z += old[i].z;
        sum[i].w += old[i].w;
      }
      if (m + 4 * i < a.M && n < a.Nc)
        *reinterpret_cast<float4*>(q + size_t(4 * i) * size_t(a.ldc)) = sum[i];
    }
  }
}

}  // namespace alr
