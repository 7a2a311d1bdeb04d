// Merge of the fused loss kernels' partial records into the per-row results, the slot weights and
// the batch sums of Eq. 1: the full-vocabulary forward, the label readout and the top-k forward.
//
// A row has one partial record per vocabulary split and column group (up to 608 of them), so
// the merge is a reduction over records as much as a map over rows.  A block takes kRows rows
// (whole anchors) and kWarps warps; a lane holds one row and walks every (kWarps * 32 / kRows)-th
// record of it, the lanes of a row are then merged by shuffles and the warps through shared
// memory, in a fixed order.  Latency-bound (a chain of dependent record loads per lane), so the
// split over records is what sets its time: 23 us at 128 rows and 608 records and 25 us at 4096
// rows and 76 records, against 1087 and 230 us with one warp per anchor (for the readout one
// thread per row: 512 us at 768 rows and 200 records, now 34) walking all records in fp64.
#include <cfloat>

#include "kernels.h"
#include "launch.h"
#include "tc_common.cuh"

namespace alr {
namespace {

ALR_DEV float quiet_nan() { return __int_as_float(0x7fc00000); }

// ------------------------------------------------------------- two-float sums ---
// A sum of exponentials is held as s + c (c: the rounding errors of s), about 2^-44 relative:
// with a sharp softmax its logarithm is the near-zero part of the loss and the entropy.  fp64
// would do the same at 1/64 of the fp32 rate.
ALR_DEV void scale2(float& s, float& c, float f) {
  const float h = s * f;
  c = fmaf(c, f, fmaf(s, f, -h));
  s = h;
}
ALR_DEV void add2(float& s, float& c, float s2, float c2) {
  const float t = s + s2, b = t - s;
  const float e = (s - (t - b)) + (s2 - b);
  s = t;
  c += c2 + e;
}
ALR_DEV double value2(float s, float c) { return double(s) + double(c); }

// (s, c) divided by 2^r, the factor its exponentials carry (r: the exponent residual of their
// reference, |r| <= 4e-3 over the fp16 range of logits): 2^-r = 1 - y, y = x - x^2 / 2 with
// x = r ln 2, within 1e-8 relative (1e-14 for |r| <= 3e-5, |logit| < 1000).
ALR_DEV void unscale_residual(float& s, float& c, float r) {
  const float x = r * kLn2;
  const float y = fmaf(-0.5f * x, x, x);
  add2(s, c, -s * y, -c * y);
}

// Factor exp(m - nm) of a sum moved from reference m to nm >= m (1 when they are equal).
ALR_DEV float rescale(float m, float nm) { return ex2((m - nm) * kLog2e); }

// Top-2 of two disjoint column sets (the leaders' values are the running maxima); equal leaders go
// to the lower token id.
ALR_DEV void merge_top2(float best, float& sec, int& id, float best2, float sec2, int id2) {
  if (best2 > best || (best2 == best && id2 < id)) {
    sec = fmaxf(best, sec2);
    id = id2;
  } else {
    sec = fmaxf(sec, best2);
  }
}

// ------------------------------------------------------------------ row states ---
// Each state is a plain record of 32-bit words: init() is a row with no columns, load() reads one
// partial record (field stride fs), merge() folds in the state of other columns.
struct FullState {
  float md, sd, cd, mt, st, ct, u, w, secd, sect, zx;
  int id, it;

  ALR_DEV void init() {
    md = mt = secd = sect = -INFINITY;
    sd = cd = st = ct = u = w = 0.f;
    zx = quiet_nan();
    id = it = 0x7fffffff;
  }
  ALR_DEV void load(const float* p, size_t fs) {
    md = p[kPMd * fs];
    sd = p[kPSd * fs];
    cd = p[kPSdLo * fs];
    mt = p[kPMt * fs];
    st = p[kPSt * fs];
    ct = p[kPStLo * fs];
    u = p[kPU * fs];
    w = p[kPW * fs];
    secd = p[kPSecd * fs];
    sect = p[kPSect * fs];
    zx = p[kPZx * fs];
    id = __float_as_int(p[kPId * fs]);
    it = __float_as_int(p[kPIt * fs]);
  }
  // u and w are measured from their own maxima (z_d - md, z_t - mt): both sides move to the
  // merged references before they are added.
  ALR_DEV void merge(const FullState& o) {
    if (!(o.mt > -INFINITY)) return;       // no columns: adds nothing
    if (!(mt > -INFINITY)) {
      *this = o;
      return;
    }
    const float nmd = fmaxf(md, o.md), nmt = fmaxf(mt, o.mt);
    const float ft = rescale(mt, nmt), fo = rescale(o.mt, nmt);
    u = fmaf(md - nmd, st, u) * ft + fmaf(o.md - nmd, o.st, o.u) * fo;
    w = fmaf(mt - nmt, st, w) * ft + fmaf(o.mt - nmt, o.st, o.w) * fo;
    float s2 = o.st, c2 = o.ct;
    scale2(st, ct, ft);
    scale2(s2, c2, fo);
    add2(st, ct, s2, c2);
    s2 = o.sd, c2 = o.cd;
    scale2(sd, cd, rescale(md, nmd));
    scale2(s2, c2, rescale(o.md, nmd));
    add2(sd, cd, s2, c2);
    merge_top2(md, secd, id, o.md, o.secd, o.id);
    merge_top2(mt, sect, it, o.mt, o.sect, o.it);
    md = nmd;
    mt = nmt;
    if (o.zx == o.zx) zx = o.zx;
  }
};

// Insert (v, id) into a list sorted by value descending, equal values by id ascending.
ALR_DEV void insert_ranked(float (&t)[kTopK], int (&ti)[kTopK], float v, int id) {
  t[kTopK - 1] = v;
  ti[kTopK - 1] = id;
#pragma unroll
  for (int k = kTopK - 1; k > 0; --k) {
    const bool up = t[k] > t[k - 1] || (t[k] == t[k - 1] && ti[k] < ti[k - 1]);
    const float a = t[k], b = t[k - 1];
    const int ia = ti[k], ib = ti[k - 1];
    t[k - 1] = up ? a : b;
    t[k] = up ? b : a;
    ti[k - 1] = up ? ia : ib;
    ti[k] = up ? ib : ia;
  }
}

struct ReadoutState {
  float m, s, c, zx;
  float t[kTopK];
  int ti[kTopK];

  ALR_DEV void init() {
    m = -INFINITY;
    s = c = 0.f;
    zx = quiet_nan();
#pragma unroll
    for (int i = 0; i < kTopK; ++i) {
      t[i] = -INFINITY;
      ti[i] = 0x7fffffff;
    }
  }
  ALR_DEV void load(const float* p, size_t fs) {
    m = p[kRM * fs];
    s = p[kRS * fs];
    c = p[kRSLo * fs];
    zx = p[kRZx * fs];
#pragma unroll
    for (int i = 0; i < kTopK; ++i) {
      t[i] = p[(kRTop + i) * fs];
      ti[i] = __float_as_int(p[(kRIdx + i) * fs]);
    }
    if (m > -INFINITY) unscale_residual(s, c, exp_residual(m));
  }
  ALR_DEV void merge(const ReadoutState& o) {
    if (!(o.m > -INFINITY)) return;
    if (!(m > -INFINITY)) {
      *this = o;
      return;
    }
    const float nm = fmaxf(m, o.m);
    float s2 = o.s, c2 = o.c;
    scale2(s, c, rescale(m, nm));
    scale2(s2, c2, rescale(o.m, nm));
    add2(s, c, s2, c2);
    m = nm;
    if (o.zx == o.zx) zx = o.zx;
    // the other list's entries largest first: the first that stays out ends the merge.  Entries
    // past a part's columns are -inf with the largest id and never enter.
#pragma unroll
    for (int i = 0; i < kTopK; ++i) {
      const float v = o.t[i];
      const bool in = v > t[kTopK - 1] || (v == t[kTopK - 1] && o.ti[i] < ti[kTopK - 1]);
      if (!in) break;
      insert_ranked(t, ti, v, o.ti[i]);
    }
  }
};

struct TopkState {
  float m, s, c, so, co, sec;   // s + c: all columns; so + co: the columns outside the label
  int id;
  float z[kTopK];               // z_d at the label tokens, NaN until their column is met

  ALR_DEV void init() {
    m = sec = -INFINITY;
    s = c = so = co = 0.f;
    id = 0x7fffffff;
#pragma unroll
    for (int i = 0; i < kTopK; ++i) z[i] = quiet_nan();
  }
  ALR_DEV void load(const float* p, size_t fs) {
    m = p[kKM * fs];
    s = p[kKS * fs];
    c = p[kKSLo * fs];
    const float in = p[kKSIn * fs];
    sec = p[kKSec * fs];
    id = __float_as_int(p[kKIdx * fs]);
#pragma unroll
    for (int i = 0; i < kTopK; ++i) z[i] = p[(kKZ + i) * fs];
    so = s;
    co = 0.f;
    add2(so, co, -in, 0.f);
    const float lo = co + c;               // back to a leading value and its small error
    co = 0.f;
    add2(so, co, lo, 0.f);
    if (m > -INFINITY) {
      const float r = exp_residual(m);
      unscale_residual(s, c, r);
      unscale_residual(so, co, r);
    }
  }
  ALR_DEV void merge(const TopkState& o) {
    if (!(o.m > -INFINITY)) return;
    if (!(m > -INFINITY)) {
      *this = o;
      return;
    }
    const float nm = fmaxf(m, o.m);
    const float f = rescale(m, nm), fo = rescale(o.m, nm);
    float s2 = o.s, c2 = o.c;
    scale2(s, c, f);
    scale2(s2, c2, fo);
    add2(s, c, s2, c2);
    s2 = o.so, c2 = o.co;
    scale2(so, co, f);
    scale2(s2, c2, fo);
    add2(so, co, s2, c2);
    merge_top2(m, sec, id, o.m, o.sec, o.id);
    m = nm;
#pragma unroll
    for (int i = 0; i < kTopK; ++i)
      if (o.z[i] == o.z[i]) z[i] = o.z[i];
  }
};

template <class St>
constexpr int kWords = int(sizeof(St) / 4);

template <class St>
ALR_DEV St shfl_xor_state(const St& s, int mask) {
  St o;
  const uint32_t* a = reinterpret_cast<const uint32_t*>(&s);
  uint32_t* b = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
  for (int i = 0; i < kWords<St>; ++i) b[i] = __shfl_xor_sync(0xffffffffu, a[i], mask);
  return o;
}

// Shared memory of the merge: one state per warp and row, word-major so that a warp's rows are
// consecutive words.
template <class St, int kRows, int kWarps>
struct MergeSmem {
  uint32_t w[kWarps][kWords<St>][kRows];

  ALR_DEV void put(int warp, int rr, const St& s) {
    const uint32_t* a = reinterpret_cast<const uint32_t*>(&s);
#pragma unroll
    for (int i = 0; i < kWords<St>; ++i) w[warp][i][rr] = a[i];
  }
  ALR_DEV St get(int warp, int rr) const {
    St s;
    uint32_t* a = reinterpret_cast<uint32_t*>(&s);
#pragma unroll
    for (int i = 0; i < kWords<St>; ++i) a[i] = w[warp][i][rr];
    return s;
  }
};

// Merge all partial records of this block's rows [row0, row0 + n_rows), n_rows <= kRows, into
// sm.get(0, row - row0).  Every thread of the block calls it; it ends with a block barrier.
template <class St, int kRows, int kWarps>
ALR_DEV void merge_rows(const LossPlan& P, const float* part, int row0, int n_rows,
                        MergeSmem<St, kRows, kWarps>& sm) {
  pdl_wait_and_release();
  constexpr int kSlots = 32 / kRows;       // records of a row read by one warp at a time
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rr = lane % kRows, slot = lane / kRows;
  const size_t fs = size_t(P.n_parts) * size_t(P.N);
  St st;
  st.init();
  if (rr < n_rows) {
#pragma unroll 2
    for (int k = warp * kSlots + slot; k < P.n_parts; k += kWarps * kSlots) {
      St o;
      o.load(part + size_t(k) * size_t(P.N) + size_t(row0 + rr), fs);
      st.merge(o);
    }
  }
#pragma unroll
  for (int off = kRows; off < 32; off <<= 1) st.merge(shfl_xor_state(st, off));
  if (lane < kRows) sm.put(warp, rr, st);
  __syncthreads();
#pragma unroll
  for (int n = kWarps / 2; n >= 1; n >>= 1) {
    if (warp < n && lane < kRows) {
      st.merge(sm.get(warp + n, rr));
      sm.put(warp, rr, st);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------- gate (Eq. 2) ---
// Survival gate of slot s of an anchor whose slots sit in consecutive lanes, slot 0 first.
// soft: g_s = exp(sum_{s'<s} logp[s']); hard: g_s = prod_{s'<s} 1[x == argmax_t].
ALR_DEV float gate_for_slot(bool active, int lane, int s, bool hard, float logp, bool match) {
  if (hard) {
    const unsigned bad = __ballot_sync(0xffffffffu, active && !match);
    const unsigned below = s == 0 ? 0u : ((0xffffffffu >> (32 - s)) << (lane - s));
    return (bad & below) ? 0.f : 1.f;
  }
  const float v = active ? logp : 0.f;
  float incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(0xffffffffu, incl, off);
    if (s >= off) incl += t;
  }
  return expf(incl - v);
}

// ------------------------------------------------------- batch sums (Eq. 1) ---
// The block's sum omega l and sum omega (lanes of its first warp) go to block_part; the block
// that finishes last (a ticket the fused kernel before this one cleared) adds all of them in a
// fixed order and writes L = lambda sum omega l / sum omega (0 when sum omega = 0).  A separate
// one-block reduction launch took 5 us.
struct BatchOut {
  double* block_part;      // [2 * gridDim.x]
  unsigned* ticket;
  float lam;
  float* loss_total;
  float* weight_sum;
  float* wl_sum;           // nullable
};

ALR_DEV double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

template <int kWarps>
ALR_DEV void batch_sums(const BatchOut& b, double wl, double ws) {
  __shared__ double s_wl[kWarps], s_ws[kWarps];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    wl = warp_sum(wl);
    ws = warp_sum(ws);
    if (lane == 0) {
      b.block_part[2 * blockIdx.x] = wl;
      b.block_part[2 * blockIdx.x + 1] = ws;
      __threadfence();
      s_last = atomicAdd(b.ticket, 1u) == gridDim.x - 1 ? 1 : 0;
    }
  }
  __syncthreads();
  if (s_last == 0) return;
  __threadfence();
  wl = ws = 0.0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += kWarps * 32) {
    wl += __ldcg(b.block_part + 2 * i);
    ws += __ldcg(b.block_part + 2 * i + 1);
  }
  wl = warp_sum(wl);
  ws = warp_sum(ws);
  if (lane == 0) {
    s_wl[warp] = wl;
    s_ws[warp] = ws;
  }
  __syncthreads();
  if (warp == 0) {
    wl = warp_sum(lane < kWarps ? s_wl[lane] : 0.0);
    ws = warp_sum(lane < kWarps ? s_ws[lane] : 0.0);
    if (lane == 0) {
      *b.loss_total = ws > 0.0 ? float(double(b.lam) * wl / ws) : 0.f;
      *b.weight_sum = float(ws);
      if (b.wl_sum != nullptr) *b.wl_sum = float(wl);
    }
  }
}

// ------------------------------------------------------- full-vocabulary forward ---
// Per row: the log-sum-exps, l = LSE_d - E_p[z_d], the label entropy, the greedy tokens with
// their top-1/top-2 gaps, log p_t(x) and the slot weight omega (envelope w_k, mask, gate of
// Eq. 2).  rows_per_block = kRows / B * B.
struct FullOut {
  float *loss_row, *ent_row, *lse_d, *lse_t;
  int32_t *argmax_d, *argmax_t;
  float *gap_d, *gap_t, *logp_x, *weight;
};

template <int kRows, int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
    combine_kernel(LossPlan P, const float* part, int rows_per_block, int mode,
                   float gamma, const float* row_mask,
                   const int32_t* corpus_tok, FullOut o, BatchOut bo) {
  __shared__ MergeSmem<FullState, kRows, kWarps> sm;
  __shared__ float s_loss[kRows], s_logp[kRows];
  const int row0 = blockIdx.x * rows_per_block;
  const int n_rows = min(rows_per_block, P.N - row0);
  merge_rows<FullState, kRows, kWarps>(P, part, row0, n_rows, sm);
  const bool erase = mode != 0;
  // one thread per row and side: both are log S - X / S_t with X = u (drafter: the loss) or w
  // (target: the entropy), two non-negative terms, in fp64
  const int side = threadIdx.x / kRows, sr = threadIdx.x % kRows;
  if (side < 2 && sr < n_rows) {
    const FullState st = sm.get(0, sr);
    const int r = row0 + sr;
    const double ls = log(side == 0 ? value2(st.sd, st.cd) : value2(st.st, st.ct));
    const double x = double(side == 0 ? st.u : st.w);
    const float v = float(ls - x / value2(st.st, st.ct));
    const float lse = (side == 0 ? st.md : st.mt) + float(ls);
    if (side == 0) {
      o.loss_row[r] = v;
      s_loss[sr] = v;
      o.lse_d[r] = lse;
      o.argmax_d[r] = st.id;
      if (o.gap_d) o.gap_d[r] = st.md - st.secd;
    } else {
      if (o.ent_row) o.ent_row[r] = v;
      o.lse_t[r] = lse;
      o.argmax_t[r] = st.it;
      if (o.gap_t) o.gap_t[r] = st.mt - st.sect;
      s_logp[sr] = st.zx - lse;
      if (erase && o.logp_x) o.logp_x[r] = st.zx - lse;
    }
  }
  __syncthreads();
  double wl = 0.0, ws = 0.0;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x, s = lane % P.B, r = row0 + lane;
    const bool active = lane < n_rows;
    float gate = 1.f;
    if (erase) {
      const float logp = active ? s_logp[lane] : 0.f;
      const bool match = active && corpus_tok[r] == sm.get(0, active ? lane : 0).it;
      gate = gate_for_slot(active, lane, s, mode == 2, logp, match);
    }
    if (active) {
      float w = expf(-float(s) / gamma) * gate;
      if (row_mask != nullptr) w *= row_mask[r];
      o.weight[r] = w;
      wl = double(w) * double(s_loss[lane]);
      ws = double(w);
    }
  }
  batch_sums<kWarps>(bo, wl, ws);
}

// ------------------------------------------------------------------ label readout ---
// Per row: log-sum-exp, the k best target logits (ties to the lower id), their probabilities
// and the tail mass (S - sum_k exp(t_k - M)) / S, the greedy token with its top-1 minus top-2
// gap, and log p at the corpus token.  Rows are independent.
template <int kRows, int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
    readout_combine_kernel(LossPlan P, const float* part, int has_corpus,
                           int32_t* top_idx, float* top_prob,
                           float* tail, float* lse_t,
                           int32_t* argmax_t, float* gap_t,
                           float* logp_x) {
  static_assert(kRows * kTopK <= 32 * kWarps, "one thread per label");
  __shared__ MergeSmem<ReadoutState, kRows, kWarps> sm;
  __shared__ double s_e[kTopK][kRows];
  const int row0 = blockIdx.x * kRows;
  const int n_rows = min(kRows, P.N - row0);
  merge_rows<ReadoutState, kRows, kWarps>(P, part, row0, n_rows, sm);
  {   // the label's exponentials in fp64, one thread each
    const int rr = threadIdx.x % kRows, i = threadIdx.x / kRows;
    if (i < kTopK && rr < n_rows) {
      const ReadoutState st = sm.get(0, rr);
      float ti = st.t[0];
      int id = st.ti[0];
#pragma unroll
      for (int j = 1; j < kTopK; ++j)
        if (j == i) {
          ti = st.t[j];
          id = st.ti[j];
        }
      const double e = exp(double(ti) - double(st.m));
      s_e[i][rr] = e;
      top_idx[size_t(row0 + rr) * kTopK + i] = id;
      top_prob[size_t(row0 + rr) * kTopK + i] = float(e / value2(st.s, st.c));
    }
  }
  __syncthreads();
  if (int(threadIdx.x) < n_rows) {
    const int rr = threadIdx.x, r = row0 + rr;
    const ReadoutState st = sm.get(0, rr);
    const double S = value2(st.s, st.c), ls = log(S);
    double inside = 0.0;
#pragma unroll
    for (int i = 0; i < kTopK; ++i) inside += s_e[i][rr];
    // with V <= k every token is in the list and the tail is empty by definition
    tail[r] = P.V <= kTopK ? 0.f : float(fmax(0.0, (S - inside) / S));
    if (lse_t) lse_t[r] = st.m + float(ls);
    if (argmax_t) argmax_t[r] = st.ti[0];
    if (gap_t) gap_t[r] = st.t[0] - st.t[1];
    if (has_corpus && logp_x) logp_x[r] = float((double(st.zx) - double(st.m)) - ls);
  }
}

// -------------------------------------------------------------------- top-k forward ---
// Per row: log-sum-exp and greedy top-2 of z_d, the drafter's mass tail_q outside the label
// tokens, the loss l = -sum_i prob_i (z_i - LSE_d) - tail log tail_q (no tail term when tail = 0)
// and the slot weight (given, or envelope times mask).
struct TopkOut {
  float *loss_row, *lse_d, *tail_q;
  int32_t* argmax_d;
  float *gap_d, *weight;
};

template <int kRows, int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
    topk_combine_kernel(LossPlan P, const float* part, int rows_per_block,
                        const float* top_prob, const float* tail,
                        const float* row_mask, const float* weight_in,
                        float gamma, TopkOut o, BatchOut bo) {
  __shared__ MergeSmem<TopkState, kRows, kWarps> sm;
  const int row0 = blockIdx.x * rows_per_block;
  const int n_rows = min(rows_per_block, P.N - row0);
  merge_rows<TopkState, kRows, kWarps>(P, part, row0, n_rows, sm);
  double wl = 0.0, ws = 0.0;
  if (int(threadIdx.x) < n_rows) {         // n_rows <= 32: the first warp
    const int s = threadIdx.x % P.B, r = row0 + threadIdx.x;
    const TopkState st = sm.get(0, threadIdx.x);
    const double S = value2(st.s, st.c), ls = log(S);
    // log q_i = (z_i - M) - log S: the difference z_i - M is exact in fp64
    double ce = 0.0;
#pragma unroll
    for (int i = 0; i < kTopK; ++i)
      ce -= double(top_prob[size_t(r) * kTopK + i]) * ((double(st.z[i]) - double(st.m)) - ls);
    const double tq = fmax(value2(st.so, st.co) / S, 1e-30);
    const float tl = tail[r];
    if (tl > 0.f) ce -= double(tl) * log(tq);
    const float loss = float(ce);
    const float w = weight_in != nullptr
                        ? weight_in[r]
                        : expf(-float(s) / gamma) * (row_mask ? row_mask[r] : 1.f);
    o.loss_row[r] = loss;
    o.lse_d[r] = st.m + float(ls);
    o.tail_q[r] = float(tq);
    o.argmax_d[r] = st.id;
    if (o.gap_d) o.gap_d[r] = st.m - st.sec;
    o.weight[r] = w;
    wl = double(w) * double(loss);
    ws = double(w);
  }
  batch_sums<kWarps>(bo, wl, ws);
}

// ------------------------------------------------------------------ launch shape ---
// Enough 32-row blocks to fill the chip twice over: 32 rows and 8 warps per block, whose record
// reads are whole 128-byte lines.  Fewer: the smallest of 8, 16 or 32 rows that holds a whole
// anchor, with 16 warps over the records (32 warps leave a thread 64 registers
// and spill).
constexpr int kManyBlocks = 304;
constexpr int kReadoutFewRows = 1024;

struct MergeShape {
  int rows, warps, rows_per_block, blocks;
};

MergeShape merge_shape(int N, int B) {
  const int per32 = 32 / B * B;
  MergeShape m{32, 8, per32, (N + per32 - 1) / per32};
  if (m.blocks >= kManyBlocks) return m;
  m.rows = B <= 8 ? 8 : B <= 16 ? 16 : 32;
  m.warps = 16;
  m.rows_per_block = m.rows / B * B;
  m.blocks = (N + m.rows_per_block - 1) / m.rows_per_block;
  return m;
}

}  // namespace

cudaError_t launch_combine(const LossPlan& plan, const float* part, int mode, float gamma,
                           const float* row_mask, const int32_t* corpus_tok, float* loss_row,
                           float* ent_row, float* lse_d, float* lse_t, int32_t* argmax_d,
                           int32_t* argmax_t, float* gap_d, float* gap_t, float* logp_x,
                           float* weight, double* block_part, unsigned* ticket, float lam,
                           float* loss_total, float* weight_sum, float* wl_sum, cudaStream_t s) {
  const MergeShape m = merge_shape(plan.N, plan.B);
  const FullOut o{loss_row, ent_row, lse_d, lse_t, argmax_d, argmax_t, gap_d, gap_t, logp_x, weight};
  const BatchOut b{block_part, ticket, lam, loss_total, weight_sum, wl_sum};
  auto kern = m.warps == 8   ? combine_kernel<32, 8>
              : m.rows == 8  ? combine_kernel<8, 16>
              : m.rows == 16 ? combine_kernel<16, 16>
                             : combine_kernel<32, 16>;
  return launch_pdl(kern, m.blocks, 32 * m.warps, 0, s, plan, part, m.rows_per_block, mode, gamma, row_mask,
                                       corpus_tok, o, b);
}

cudaError_t launch_readout_combine(const LossPlan& plan, const float* part, bool has_corpus,
                                   int32_t* top_idx, float* top_prob, float* tail, float* lse_t,
                                   int32_t* argmax_t, float* gap_t, float* logp_x,
                                   cudaStream_t s) {
  // a merge of two top-8 lists costs several times a plain record's, so with more rows fewer lanes
  // share one: 64, 16 from 1024 rows, 8 (readout with 16 instead of 64: 1920 x 64 x 151936 243 ->
  // 229 us, 9000 x 64 x 20000 231 -> 191; 768 x 64 x 151936 130 -> 131)
  MergeShape m = merge_shape(plan.N, 1);
  auto kern = readout_combine_kernel<32, 8>;
  if (m.rows < 32) {
    const bool few = plan.N < kReadoutFewRows;
    kern = few ? readout_combine_kernel<8, 16> : readout_combine_kernel<16, 8>;
    m = few ? MergeShape{8, 16, 8, (plan.N + 7) / 8} : MergeShape{16, 8, 16, (plan.N + 15) / 16};
  }
  return launch_pdl(kern, m.blocks, 32 * m.warps, 0, s, plan, part, has_corpus ? 1 : 0, top_idx,
                    top_prob, tail, lse_t, argmax_t, gap_t, logp_x);
}

cudaError_t launch_topk_combine(const LossPlan& plan, const float* part, const float* top_prob,
                                const float* tail, const float* row_mask, const float* weight_in,
                                float gamma, float* loss_row, float* lse_d, float* tail_q,
                                int32_t* argmax_d, float* gap_d, float* weight,
                                double* block_part, unsigned* ticket, float lam,
                                float* loss_total, float* weight_sum, float* wl_sum,
                                cudaStream_t s) {
  const MergeShape m = merge_shape(plan.N, plan.B);
  const TopkOut o{loss_row, lse_d, tail_q, argmax_d, gap_d, weight};
  const BatchOut b{block_part, ticket, lam, loss_total, weight_sum, wl_sum};
  auto kern = m.warps == 8   ? topk_combine_kernel<32, 8>
              : m.rows == 8  ? topk_combine_kernel<8, 16>
              : m.rows == 16 ? topk_combine_kernel<16, 16>
                             : topk_combine_kernel<32, 16>;
  return launch_pdl(kern, m.blocks, 32 * m.warps, 0, s, plan, part, m.rows_per_block, top_prob, tail, row_mask,
                                       weight_in, gamma, o, b);
}

}  // namespace alr
