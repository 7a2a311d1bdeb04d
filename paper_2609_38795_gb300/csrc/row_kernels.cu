// Row-level kernels of the slot-loss path: the IRA gather, block plan, draws and context, L from
// reduced sums, the accepted-length statistic and the erase-gate weights.  (The merge of the
// forward's partial records is in combine_kernels.cu, the logit gradient from kept logits in
// grad_kernels.cu.)

#include "kernels.h"
#include "launch.h"
#include "tc_common.cuh"

namespace alr {
namespace {

// ------------------------------------------------------------------ IRA gather ---
// One warp per output row; each lane moves 16-byte vectors, issuing a batch of loads before
// the matching stores so that many requests are in flight per SM.
constexpr int kGatherBatch = 16;

__global__ void __launch_bounds__(256) gather_kernel(const uint4* feat, int S, int L,
                                                     int vec_per_row, const int32_t* seq,
                                                     const int32_t* pos, const int32_t* valid_len,
                                                     int A, int B, uint4* out, float* row_valid) {
  pdl_wait_and_release();
  const long long r = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (r >= (long long)A * B) return;
  const int a = int(r / B), s = int(r - (long long)a * B);
  const int sq = seq[a], p0 = pos[a];
  int lim = L;
  if (valid_len != nullptr) lim = min(lim, valid_len[a]);
  const bool ok = sq >= 0 && sq < S && p0 >= 0 && (long long)p0 + s < lim;   // no int overflow
  uint4* dst = out + r * vec_per_row;
  if (lane == 0 && row_valid != nullptr) row_valid[r] = ok ? 1.f : 0.f;
  if (!ok) {
    const uint4 z = make_uint4(0, 0, 0, 0);
    for (int i = lane; i < vec_per_row; i += 32) dst[i] = z;
    return;
  }
  const uint4* src = feat + ((long long)sq * L + p0 + s) * vec_per_row;
  for (int base = 0; base < vec_per_row; base += 32 * kGatherBatch) {
    uint4 v[kGatherBatch];
#pragma unroll
    for (int j = 0; j < kGatherBatch; ++j) {
      const int i = base + j * 32 + lane;
      if (i < vec_per_row) v[j] = src[i];
    }
#pragma unroll
    for (int j = 0; j < kGatherBatch; ++j) {
      const int i = base + j * 32 + lane;
      if (i < vec_per_row) __stcs(dst + i, v[j]);
    }
  }
}

// ------------------------------------------------------------- gate (Eq. 2) ---
// Warp-level survival gate for one anchor: lane s holds row a*B+s (lanes >= B inactive).
// soft: g_s = exp(sum_{s'<s} logp_x[s']); hard: g_s = prod_{s'<s} 1[x == argmax_t].
__device__ __forceinline__ float gate_for_lane(bool active, int lane, bool hard, float logp,
                                               bool match) {
  if (hard) {
    const unsigned bad = __ballot_sync(0xffffffffu, active && !match);
    const unsigned below = (lane == 0) ? 0u : (0xffffffffu >> (32 - lane));
    return (bad & below) ? 0.f : 1.f;
  }
  float v = active ? logp : 0.f;
  float incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += t;
  }
  return expf(incl - v);
}

// Eq. 1 from sums that the caller reduced over the shards of a batch: L = lambda * wl / ws,
// 0 when ws = 0 (no supervised slot anywhere in the batch).
__global__ void loss_from_sums_kernel(const float* wl_sum, const float* weight_sum, float lam,
                                      float* loss_total) {
  pdl_wait_and_release();
  const double ws = *weight_sum;
  *loss_total = ws > 0.0 ? float(double(lam) * double(*wl_sum) / ws) : 0.f;
}

// ------------------------------------------------------------- accepted length ---
// One warp per anchor: the count of leading slots whose greedy drafter token equals the
// greedy target token (and whose row is active).
ALR_DEV int accepted_slots(const int32_t* am_d, const int32_t* am_t, const float* active_w, int a,
                           int B, int lane) {
  bool ok = false;
  if (lane < B) {
    const int r = a * B + lane;
    ok = am_d[r] == am_t[r];
    if (active_w != nullptr) ok = ok && active_w[r] > 0.f;
  }
  const unsigned bal = __ballot_sync(0xffffffffu, ok);
  return bal == 0xffffffffu ? 32 : __ffs(~bal) - 1;
}

__global__ void __launch_bounds__(256)
    accept_len_kernel(const int32_t* am_d, const int32_t* am_t, const float* active_w, int A,
                      int B, int32_t* acc, unsigned long long* hist) {
  pdl_wait_and_release();
  const int a = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (a >= A) return;
  const int n = accepted_slots(am_d, am_t, active_w, a, B, lane);
  if (lane == 0) {
    acc[a] = n;
    if (hist != nullptr) atomicAdd(hist + n, 1ull);
  }
}

// Few anchors: one block counts them all, its histogram in shared memory, which saves the clear
// of hist as a stream operation of its own (12 anchors: 1.45 us against 1.4 and a 0.9 us clear with
// the gap between them).  Past kAcceptOneBlock anchors the rounds of one block cost more than that.
constexpr int kAcceptOneBlock = 256;

__global__ void __launch_bounds__(1024)
    accept_len_one_block_kernel(const int32_t* am_d, const int32_t* am_t, const float* active_w,
                                int A, int B, int32_t* acc, unsigned long long* hist) {
  __shared__ int count[33];
  pdl_wait_and_release();
  const int lane = threadIdx.x & 31, n_warps = blockDim.x / 32;
  if (threadIdx.x < 32) {
    count[threadIdx.x] = 0;
    if (threadIdx.x == 0) count[32] = 0;
  }
  __syncthreads();
#pragma unroll 4
  for (int a = threadIdx.x / 32; a < A; a += n_warps) {
    const int n = accepted_slots(am_d, am_t, active_w, a, B, lane);
    if (lane == 0) {
      acc[a] = n;
      atomicAdd(&count[n], 1);
    }
  }
  __syncthreads();
  if (hist != nullptr && int(threadIdx.x) <= B) hist[threadIdx.x] = count[threadIdx.x];
}

// ---------------------------------------------------------- erase weights ---
__global__ void __launch_bounds__(256)
    erase_weights_kernel(const float* logp_x, const int32_t* corpus_tok, const int32_t* argmax_t,
                         const float* row_mask, int A, int B, float gamma, int hard,
                         float* weight) {
  pdl_wait_and_release();
  const int a = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (a >= A) return;
  const bool active = lane < B;
  const int r = a * B + (active ? lane : 0);
  float logp = 0.f;
  bool match = true;
  if (active) {
    if (hard) match = corpus_tok[r] == argmax_t[r];
    else logp = logp_x[r];
  }
  const float g = gate_for_lane(active, lane, hard != 0, logp, match);
  if (active) {
    float w = expf(-float(lane) / gamma) * g;
    if (row_mask != nullptr) w *= row_mask[r];
    weight[r] = w;
  }
}

// ------------------------------------------------------------- IRA block plan ---
// One thread per block slot (s, b): sample s keeps m = min(v_s, max_blocks) blocks, the
// first ceil(m/2) primary, the next floor(m/2) secondary (Sec. 3.2); secondary i sits in
// primary i's rollout at offset j.  Emits the label-row gather (seq, pos, valid_len) over
// the primary label buffer [S * P, K, d], the anchor token and the rollout context length.
__global__ void __launch_bounds__(256)
    ira_blocks_kernel(int S, int K, int max_blocks, const int32_t* valid_anchors,
                      const int32_t* rollout_len, const int32_t* offsets,
                      const int32_t* rollout_tok, const int32_t* corpus_anchor_tok, int32_t* seq,
                      int32_t* pos, int32_t* vlen, int32_t* ctx_len, int32_t* anchor_tok) {
  pdl_wait_and_release();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)S * max_blocks) return;
  const int s = int(t / max_blocks), b = int(t - (long long)s * max_blocks);
  const int P = max_blocks - max_blocks / 2, Q = max_blocks / 2;
  const int m = max(0, min(valid_anchors[s], max_blocks));
  const int n_prim = (m + 1) / 2;
  int p = -1, j = 0;
  if (b < n_prim) {
    p = b;
  } else if (b < m) {
    p = b - n_prim;
    j = offsets[size_t(s) * Q + p];
    // an offset outside the rollout leaves the block unused: past K - 1, or past the end of
    // a primary rollout that terminated early (y*_j, the block's anchor token, never existed)
    if (j < 1 || j > K - 1 || j > rollout_len[size_t(s) * P + p]) p = -1;
  }
  if (p < 0) {
    seq[t] = -1;
    pos[t] = 0;
    vlen[t] = 0;
    if (ctx_len) ctx_len[t] = 0;
    if (anchor_tok) anchor_tok[t] = -1;
    return;
  }
  const size_t prim = size_t(s) * P + p;
  seq[t] = int(prim);
  pos[t] = j;
  vlen[t] = rollout_len[prim];
  if (ctx_len) ctx_len[t] = j > 0 ? j - 1 : 0;
  if (anchor_tok) {
    int tok = -1;
    if (j == 0 && corpus_anchor_tok) tok = corpus_anchor_tok[t];
    if (j > 0 && rollout_tok) tok = rollout_tok[prim * K + (j - 1)];   // y*_j
    anchor_tok[t] = tok;
  }
}

// ------------------------------------------------------------------ IRA draws ---
// One block per sample.  The anchor draw is the m = min(v, max_blocks) smallest of the sample's v
// valid (key, position) pairs, in increasing order.  A radix select narrows the pairs to the
// candidates: per 8-bit digit a shared histogram of the pairs still in the running finds the
// digit value that holds the m-th smallest, until at most kDrawSlack pairs more than m are left
// (one pass for random keys; equal keys go on into the position's digits, which tell every pair
// apart).  Each candidate's rank is then counted among the candidates alone, one warp per
// candidate.  Positions live in registers (L <= 16 per thread).  Counting each valid pair's rank
// among all L instead took 380 us for 6 samples of L = 4096; this takes 8.5 us.
// Offsets: j = 2 + floor(u (K - 2) / 2^32).
constexpr int kDrawThreads = 1024;         // most; 256 and 512 for short samples
constexpr int kDrawPer = 16;               // positions per thread: L <= 16384
constexpr int kDrawSlack = 64;
using Pair = unsigned long long;           // key << 32 | position
constexpr Pair kNoPair = ~0ull;            // an invalid position (no valid one: position < 2^14)

__global__ void __launch_bounds__(kDrawThreads)
    ira_draw_kernel(int L, int K, int max_blocks, const uint8_t* anchor_ok, const uint32_t* keys,
                    const uint32_t* offset_u, int32_t* n_valid, int32_t* anchor_pos,
                    int32_t* offsets) {
  extern __shared__ Pair cand[];           // [L]
  __shared__ int hist[256], s_valid, s_cand, s_digit, s_below, s_in;
  pdl_wait_and_release();
  const int s = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t row = size_t(s) * size_t(L);
  if (tid < 256) hist[tid] = 0;
  if (tid == 0) s_valid = s_cand = 0;
  Pair c[kDrawPer];
  int mine = 0;
#pragma unroll
  for (int j = 0; j < kDrawPer; ++j) {
    const int a = tid + j * int(blockDim.x);
    c[j] = kNoPair;
    if (a < L && anchor_ok[row + a] != 0) {
      c[j] = (Pair(keys[row + a]) << 32) | unsigned(a);
      ++mine;
    }
  }
  __syncthreads();
  mine = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0) atomicAdd(&s_valid, mine);
  __syncthreads();
  const int v = s_valid, m = min(v, max_blocks);
  int32_t* out = anchor_pos + size_t(s) * size_t(max_blocks);
  for (int i = m + tid; i < max_blocks; i += blockDim.x) out[i] = -1;

  // candidates: pairs whose bits from `shift` up are at most `prefix` (all valid ones when m = v)
  Pair prefix = kNoPair;
  int shift = 0;
  if (m < v) {                             // uniform over the block
    int below = 0;                         // pairs known to be among the m smallest
    prefix = 0;
    for (int digit = 0; digit < 6; ++digit) {
      // the key's four digits, then the position's two (positions are below 2^14)
      shift = digit < 4 ? 56 - 8 * digit : 8 * (5 - digit);
      // the bits over shift + 8
      const Pair above = digit == 0 ? 0 : digit == 4 ? prefix << 16 : prefix;
#pragma unroll
      for (int j = 0; j < kDrawPer; ++j) {
        if (c[j] == kNoPair) continue;
        if (digit == 0 || (c[j] >> (shift + 8)) == above)
          atomicAdd(&hist[int(c[j] >> shift) & 255], 1);
      }
      __syncthreads();
      if (warp == 0) {                     // the digit value that holds the m-th smallest pair
        int n[8], sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          n[i] = hist[8 * lane + i];
          sum += n[i];
        }
        int incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += t;
        }
        int before = below + incl - sum;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (before < m && m <= before + n[i]) {   // true for exactly one digit value
            s_digit = 8 * lane + i;
            s_below = before;
            s_in = n[i];
          }
          before += n[i];
        }
      }
      __syncthreads();
      prefix = (above << 8) | unsigned(s_digit);
      below = s_below;
      if (below + s_in <= m + kDrawSlack) break;
      if (tid < 256) hist[tid] = 0;
      __syncthreads();
    }
  }
#pragma unroll
  for (int j = 0; j < kDrawPer; ++j)
    if (c[j] != kNoPair && (c[j] >> shift) <= prefix) cand[atomicAdd(&s_cand, 1)] = c[j];
  __syncthreads();
  const int n = s_cand;
  for (int i = warp; i < n; i += int(blockDim.x >> 5)) {
    const Pair mypair = cand[i];
    int rank = 0;
    for (int q = lane; q < n; q += 32) rank += cand[q] < mypair ? 1 : 0;
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0 && rank < m) out[rank] = int(unsigned(mypair));
  }
  const int H = max_blocks / 2;
  for (int i = tid; i < H; i += blockDim.x) {
    const unsigned long long u = offset_u[size_t(s) * H + i];
    offsets[size_t(s) * H + i] = 2 + int((u * unsigned(K - 2)) >> 32);
  }
  if (tid == 0) n_valid[s] = v;
}

// ------------------------------------------------------------------ IRA context ---
// Context rows of the secondary blocks: output row (s, i, r) of [S, H, C, F] is row r of
// primary i's stored rollout features when secondary i of sample s exists and r < j - 1,
// zero otherwise.  One warp per output row, 16-byte vectors in batches as in the gather.
__global__ void __launch_bounds__(256) ira_context_kernel(
    const uint4* store, int C, int vec_per_row, int S, int K, int max_blocks,
    const int32_t* n_valid, const int32_t* rollout_len, const int32_t* offsets,
    const int32_t* anchor_pos, uint4* ctx, int32_t* ctx_len, int32_t* prefix_end) {
  pdl_wait_and_release();
  const int H = max_blocks / 2, P = max_blocks - H;
  const long long t = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (t >= (long long)S * H * C) return;
  const int r = int(t % C);
  const long long si = t / C;
  const int s = int(si / H), i = int(si - (long long)s * H);
  const int m = max(0, min(n_valid[s], max_blocks));
  const int j = offsets[si];
  const size_t prim = size_t(s) * P + i;
  const bool exists = i < m / 2 && j >= 1 && j <= K - 1 && j <= rollout_len[prim];
  const int n = exists ? j - 1 : 0;
  if (r == 0 && lane == 0) {
    if (ctx_len) ctx_len[si] = n;
    if (prefix_end) prefix_end[si] = exists ? anchor_pos[size_t(s) * max_blocks + i] : -1;
  }
  uint4* dst = ctx + t * vec_per_row;
  if (r >= n) {
    const uint4 z = make_uint4(0, 0, 0, 0);
    for (int k = lane; k < vec_per_row; k += 32) __stcs(dst + k, z);
    return;
  }
  const uint4* src = store + ((long long)prim * C + r) * vec_per_row;
  for (int base = 0; base < vec_per_row; base += 32 * kGatherBatch) {
    uint4 v[kGatherBatch];
#pragma unroll
    for (int k = 0; k < kGatherBatch; ++k) {
      const int e = base + k * 32 + lane;
      if (e < vec_per_row) v[k] = src[e];
    }
#pragma unroll
    for (int k = 0; k < kGatherBatch; ++k) {
      const int e = base + k * 32 + lane;
      if (e < vec_per_row) __stcs(dst + e, v[k]);
    }
  }
}

// ------------------------------------------------------------------ transpose ---
// out[c * ld_out + r] = in[r * C + c] for 32-bit elements, 32 x 32 tiles through shared memory; the
// blocks from column tile `tiles` on do the same for in2 [R, C2].  Small matrices only (the fp32
// path), so a launch costs more than its traffic: the fp32 step of 512 x 256 x 4096 takes 81.4 us
// with dW's two operands in one launch, 83.0 with one each.
__global__ void __launch_bounds__(256) transpose32_kernel(const float* in, float* out, int R, int C,
                                                          int ld_out, unsigned tiles,
                                                          const float* in2, float* out2, int C2) {
  __shared__ float tile[32][33];
  pdl_wait_and_release();
  unsigned cb = blockIdx.x;
  if (cb >= tiles) {
    cb -= tiles;
    in = in2;
    out = out2;
    C = C2;
  }
  const int c0 = cb * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[i][threadIdx.x] = in[(long long)r * C + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < C) out[(long long)c * ld_out + r] = tile[threadIdx.x][i];
  }
}

}  // namespace

cudaError_t launch_ira_blocks(int S, int K, int max_blocks, const int32_t* valid_anchors,
                              const int32_t* rollout_len, const int32_t* offsets,
                              const int32_t* rollout_tok, const int32_t* corpus_anchor_tok,
                              int32_t* seq, int32_t* pos, int32_t* vlen, int32_t* ctx_len,
                              int32_t* anchor_tok, cudaStream_t s) {
  const long long n = (long long)S * max_blocks;
  return launch_pdl(ira_blocks_kernel, unsigned((n + 255) / 256), 256, 0, s, S, K, max_blocks,
                    valid_anchors, rollout_len, offsets, rollout_tok, corpus_anchor_tok, seq, pos,
                    vlen, ctx_len, anchor_tok);
}

cudaError_t launch_ira_draw(int S, int L, int K, int max_blocks, const uint8_t* anchor_ok,
                            const uint32_t* keys, const uint32_t* offset_u, int32_t* n_valid,
                            int32_t* anchor_pos, int32_t* offsets, cudaStream_t s) {
  const size_t smem = size_t(L) * sizeof(Pair);
  cudaError_t e = cudaFuncSetAttribute(ira_draw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(smem));
  if (e != cudaSuccess) return e;
  const int threads = L <= 256 ? 256 : L <= 512 ? 512 : kDrawThreads;
  return launch_pdl(ira_draw_kernel, S, threads, smem, s, L, K, max_blocks, anchor_ok, keys,
                    offset_u, n_valid, anchor_pos, offsets);
}

cudaError_t launch_ira_context(const void* store, int C, int F, int elem_bytes, int S, int K,
                               int max_blocks, const int32_t* n_valid, const int32_t* rollout_len,
                               const int32_t* offsets, const int32_t* anchor_pos, void* ctx,
                               int32_t* ctx_len, int32_t* prefix_end, cudaStream_t s) {
  const long long rows = (long long)S * (max_blocks / 2) * C;
  const int vec = int((long long)F * elem_bytes / 16);
  if (rows == 0) return cudaSuccess;
  return launch_pdl(ira_context_kernel, unsigned((rows + 7) / 8), 256, 0, s,
                    static_cast<const uint4*>(store), C, vec, S, K, max_blocks, n_valid,
                    rollout_len, offsets, anchor_pos, static_cast<uint4*>(ctx), ctx_len,
                    prefix_end);
}

cudaError_t launch_transpose32(const float* in, float* out, int R, int C, int ld_out,
                               cudaStream_t s) {
  dim3 grid((C + 31) / 32, (R + 31) / 32);
  return launch_pdl(transpose32_kernel, grid, dim3(32, 8), 0, s, in, out, R, C, ld_out, grid.x,
                    (const float*)nullptr, (float*)nullptr, 0);
}

cudaError_t launch_transpose32_pair(const float* a, float* a_out, int Ca, const float* b,
                                    float* b_out, int Cb, int R, int ld_out, cudaStream_t s) {
  const unsigned tiles = (Ca + 31) / 32;
  dim3 grid(tiles + (Cb + 31) / 32, (R + 31) / 32);
  return launch_pdl(transpose32_kernel, grid, dim3(32, 8), 0, s, a, a_out, R, Ca, ld_out, tiles, b,
                    b_out, Cb);
}

cudaError_t launch_gather(const void* feat, int S, int L, int d, int elem_bytes,
                          const int32_t* seq, const int32_t* pos, const int32_t* valid_len,
                          int A, int B, void* out, float* row_valid, cudaStream_t s) {
  const long long rows = (long long)A * B;
  const int vec = int((long long)d * elem_bytes / 16);
  const long long blocks = (rows + 7) / 8;
  if (blocks == 0) return cudaSuccess;
  return launch_pdl(gather_kernel, unsigned(blocks), 256, 0, s, static_cast<const uint4*>(feat), S,
                    L, vec, seq, pos, valid_len, A, B, static_cast<uint4*>(out), row_valid);
}

cudaError_t launch_loss_from_sums(const float* wl_sum, const float* weight_sum, float lam,
                                  float* loss_total, cudaStream_t s) {
  return launch_pdl(loss_from_sums_kernel, 1, 1, 0, s, wl_sum, weight_sum, lam, loss_total);
}

cudaError_t launch_accept_len(const int32_t* am_d, const int32_t* am_t, const float* active,
                              int A, int B, int32_t* acc, int64_t* hist, cudaStream_t s) {
  unsigned long long* h = reinterpret_cast<unsigned long long*>(hist);
  if (A <= kAcceptOneBlock) {
    // at least 33 threads: one per histogram entry
    const int threads = A < 2 ? 64 : A < 32 ? 32 * A : 1024;
    return launch_pdl(accept_len_one_block_kernel, 1, threads, 0, s, am_d, am_t, active, A, B, acc,
                      h);
  }
  if (hist != nullptr) {
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int64_t) * size_t(B + 1), s);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(accept_len_kernel, (A + 7) / 8, 256, 0, s, am_d, am_t, active, A, B, acc, h);
}

cudaError_t launch_erase_weights(const float* logp_x, const int32_t* corpus_tok,
                                 const int32_t* argmax_t, const float* row_mask, int A, int B,
                                 float gamma, int hard, float* weight, cudaStream_t s) {
  return launch_pdl(erase_weights_kernel, (A + 7) / 8, 256, 0, s, logp_x, corpus_tok, argmax_t,
                    row_mask, A, B, gamma, hard, weight);
}

}  // namespace alr
