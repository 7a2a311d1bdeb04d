// Merge of the fused loss kernels' partial records into the per-row results, the slot weights and
// the batch sums of Eq. 1: the full-vocabulary forward, the label readout and the top-k forward.
//
// A row has one partial record per vocabulary split and column group (tens to some 2400 of them),
// so the merge is a reduction over records as much as a map over rows.  A block takes kRows rows
// (whole anchors) and kWarps warps; a lane holds one row and walks every (kWarps * 32 / kRows)-th
// record of it, the lanes of a row are then merged by shuffles and the warps through shared
// memory, in a fixed order.  The row's maxima over all records are found first, so every record's
// sums are multiplied by one factor only, and all sums of exponentials are held in fp64.  Bound by
// latency (record loads, three in flight per lane: 31 us with two at 128 rows and 608 records, 25
// with three), so the split over records is what sets its time: 25 us there, 16 us at 2000 rows
// and 76 records, against 1087 us at 128 rows with one warp per anchor walking all records.
#include <cfloat>

#include "kernels.h"
#include "launch.h"
#include "tc_common.cuh"

namespace alr {
namespace {

ALR_DEV float quiet_nan() { return __int_as_float(0x7fc00000); }

// ----------------------------------------------------------------- record sums ---
// A part's sum of exponentials arrives as s + c (c: the rounding errors of s) and is merged in
// fp64: with a sharp softmax its logarithm is the near-zero part of the loss and the entropy.
// fp64 instructions, conversions to it among them, run at 1/64 of the fp32 rate, so a value is
// widened by moving its bits (normal numbers and zero; smaller ones become zero).
ALR_DEV double widen(float x) {
  const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
  const unsigned hi = ((b & 0x7fffffffu) >> 3) + 0x38000000u + (b & 0x80000000u);
  return __hiloint2double(int(e == 0 ? 0u : hi), int(e == 0 ? 0u : b << 29));
}

// acc + f (s + c)
ALR_DEV double add_part(double acc, float f, float s, float c) {
  const double f64 = widen(f);
  return fma(f64, widen(s), fma(f64, widen(c), acc));
}

// The row's sums carry the factor 2^r of its maximum m (exp_residual): its natural logarithm.
constexpr double kLn2Double = 0.6931471805599453;
ALR_DEV double ln_residual(float m) { return double(exp_residual(m)) * kLn2Double; }

// Top-2 of two disjoint column sets; equal leaders go to the lower token id.
ALR_DEV void merge_top2(float& best, float& sec, int& id, float best2, float sec2, int id2) {
  if (best2 > best || (best2 == best && id2 < id)) {
    sec = fmaxf(best, sec2);
    best = best2;
    id = id2;
  } else {
    sec = fmaxf(sec, best2);
  }
}

// ------------------------------------------------------------------ row states ---
// A state holds sums measured from the row's maxima over all records (`ref`, kRefs of them, found
// first), so that every record's sums are multiplied by one factor, whatever the order of the
// merge.  kWords: its 32-bit words, without padding.  init() is a row with no columns, Record one
// partial record (field stride fs), add() folds a record in, merge() another state of the same
// row.
struct FullState {
  double sd, st;
  float u, w, bd, secd, bt, sect, zx;
  int id, it;

  static constexpr int kWords = 13, kRefs = 2;
  static constexpr bool kLongAdd = false;
  static ALR_DEV constexpr int ref_field(int i) { return i == 0 ? kPMd : kPMt; }

  struct Record {
    float md, sd, cd, mt, st, ct, u, w, secd, sect, zx;
    int id, it;

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
    ALR_DEV float ref(int i) const { return i == 0 ? md : mt; }
  };

  ALR_DEV void init() {
    sd = st = 0.0;
    u = w = 0.f;
    bd = bt = secd = sect = -INFINITY;
    zx = quiet_nan();
    id = it = 0x7fffffff;
  }
  // u and w are measured from their part's maxima ((z_d - md) log2 e, (z_t - mt) log2 e): moved to
  // the row's.
  ALR_DEV void add(const Record& o, const float (&ref)[kRefs]) {
    if (!(o.mt > -INFINITY)) return;       // no columns
    const float dd = ref_step(o.md, -ref[0] * kLog2e), dt = ref_step(o.mt, -ref[1] * kLog2e);
    const float ft = ex2(dt);
    sd = add_part(sd, ex2(dd), o.sd, o.cd);
    st = add_part(st, ft, o.st, o.ct);
    u = fmaf(ft, fmaf(dd, o.st, o.u), u);
    w = fmaf(ft, fmaf(dt, o.st, o.w), w);
    merge_top2(bd, secd, id, o.md, o.secd, o.id);
    merge_top2(bt, sect, it, o.mt, o.sect, o.it);
    if (o.zx == o.zx) zx = o.zx;
  }
  ALR_DEV void merge(const FullState& o) {
    sd += o.sd;
    st += o.st;
    u += o.u;
    w += o.w;
    merge_top2(bd, secd, id, o.bd, o.secd, o.id);
    merge_top2(bt, sect, it, o.bt, o.sect, o.it);
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
  double s;
  float zx;
  float t[kTopK];               // t[0]: the row's maximum
  int ti[kTopK];

  static constexpr int kWords = 3 + 2 * kTopK, kRefs = 1;
  static constexpr bool kLongAdd = true;    // a merge of two lists
  static ALR_DEV constexpr int ref_field(int) { return kRM; }

  struct Record {
    float m, s, c, zx;
    float t[kTopK];
    int ti[kTopK];

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
    }
    ALR_DEV float ref(int) const { return m; }
  };

  ALR_DEV void init() {
    s = 0.0;
    zx = quiet_nan();
#pragma unroll
    for (int i = 0; i < kTopK; ++i) {
      t[i] = -INFINITY;
      ti[i] = 0x7fffffff;
    }
  }
  // The other list's entries largest first: the first that stays out ends the merge.  Entries
  // past a part's columns are -inf with the largest id and never enter.
  ALR_DEV void merge_list(const float (&t2)[kTopK], const int (&ti2)[kTopK]) {
#pragma unroll
    for (int i = 0; i < kTopK; ++i) {
      const float v = t2[i];
      const bool in = v > t[kTopK - 1] || (v == t[kTopK - 1] && ti2[i] < ti[kTopK - 1]);
      if (!in) break;
      insert_ranked(t, ti, v, ti2[i]);
    }
  }
  ALR_DEV void add(const Record& o, const float (&ref)[kRefs]) {
    if (!(o.m > -INFINITY)) return;
    s = add_part(s, ex2(ref_step(o.m, -ref[0] * kLog2e)), o.s, o.c);
    if (o.zx == o.zx) zx = o.zx;
    merge_list(o.t, o.ti);
  }
  ALR_DEV void merge(const ReadoutState& o) {
    s += o.s;
    if (o.zx == o.zx) zx = o.zx;
    merge_list(o.t, o.ti);
  }
};

struct TopkState {
  double s, so;                 // all columns; the columns outside the label
  float best, sec;
  int id;
  float z[kTopK];               // z_d at the label tokens, NaN until their column is met

  static constexpr int kWords = 7 + kTopK, kRefs = 1;
  static constexpr bool kLongAdd = false;
  static ALR_DEV constexpr int ref_field(int) { return kKM; }

  struct Record {
    float m, s, c, in, sec;
    int id;
    float z[kTopK];

    ALR_DEV void load(const float* p, size_t fs) {
      m = p[kKM * fs];
      s = p[kKS * fs];
      c = p[kKSLo * fs];
      in = p[kKSIn * fs];
      sec = p[kKSec * fs];
      id = __float_as_int(p[kKIdx * fs]);
#pragma unroll
      for (int i = 0; i < kTopK; ++i) z[i] = p[(kKZ + i) * fs];
    }
    ALR_DEV float ref(int) const { return m; }
  };

  ALR_DEV void init() {
    s = so = 0.0;
    best = sec = -INFINITY;
    id = 0x7fffffff;
#pragma unroll
    for (int i = 0; i < kTopK; ++i) z[i] = quiet_nan();
  }
  ALR_DEV void add(const Record& o, const float (&ref)[kRefs]) {
    if (!(o.m > -INFINITY)) return;
    const float f = ex2(ref_step(o.m, -ref[0] * kLog2e));
    s = add_part(s, f, o.s, o.c);
    so = fma(widen(f), (widen(o.s) - widen(o.in)) + widen(o.c), so);
    merge_top2(best, sec, id, o.m, o.sec, o.id);
#pragma unroll
    for (int i = 0; i < kTopK; ++i)
      if (o.z[i] == o.z[i]) z[i] = o.z[i];
  }
  ALR_DEV void merge(const TopkState& o) {
    s += o.s;
    so += o.so;
    merge_top2(best, sec, id, o.best, o.sec, o.id);
#pragma unroll
    for (int i = 0; i < kTopK; ++i)
      if (o.z[i] == o.z[i]) z[i] = o.z[i];
  }
};

template <class St>
ALR_DEV St shfl_xor_state(const St& s, int mask) {
  St o;
  const uint32_t* a = reinterpret_cast<const uint32_t*>(&s);
  uint32_t* b = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
  for (int i = 0; i < St::kWords; ++i) b[i] = __shfl_xor_sync(0xffffffffu, a[i], mask);
  return o;
}

// Shared memory of the merge: one state per warp and row, word-major so that a warp's rows are
// consecutive words, and the warps' maxima.
template <class St, int kRows, int kWarps>
struct MergeSmem {
  uint32_t w[kWarps][St::kWords][kRows];
  float ref[kWarps][St::kRefs][kRows];

  ALR_DEV void put(int warp, int rr, const St& s) {
    const uint32_t* a = reinterpret_cast<const uint32_t*>(&s);
#pragma unroll
    for (int i = 0; i < St::kWords; ++i) w[warp][i][rr] = a[i];
  }
  ALR_DEV St get(int warp, int rr) const {
    St s;
    uint32_t* a = reinterpret_cast<uint32_t*>(&s);
#pragma unroll
    for (int i = 0; i < St::kWords; ++i) a[i] = w[warp][i][rr];
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
  const float* col = part + size_t(row0 + rr);
  const int k0 = warp * kSlots + slot, step = kWarps * kSlots;
  const bool any = rr < n_rows && k0 < P.n_parts;
  // this lane's first record, on its way while the maxima are found
  typename St::Record first;
  if (any) first.load(col + size_t(k0) * size_t(P.N), fs);
  // the row's maxima
  float ref[St::kRefs];
#pragma unroll
  for (int i = 0; i < St::kRefs; ++i) ref[i] = any ? first.ref(i) : -INFINITY;
  if (rr < n_rows) {
#pragma unroll 8
    for (int k = k0 + step; k < P.n_parts; k += step) {
#pragma unroll
      for (int i = 0; i < St::kRefs; ++i)
        ref[i] = fmaxf(ref[i], col[size_t(k) * size_t(P.N) + size_t(St::ref_field(i)) * fs]);
    }
  }
#pragma unroll
  for (int i = 0; i < St::kRefs; ++i) {
#pragma unroll
    for (int off = kRows; off < 32; off <<= 1)
      ref[i] = fmaxf(ref[i], __shfl_xor_sync(0xffffffffu, ref[i], off));
    if (lane < kRows) sm.ref[warp][i][rr] = ref[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < St::kRefs; ++i)
#pragma unroll
    for (int n = 0; n < kWarps; ++n) ref[i] = fmaxf(ref[i], sm.ref[n][i][rr]);

  St st;
  st.init();
  if constexpr (St::kLongAdd) {
    // one copy of the long add, the next record on its way meanwhile
    if (any) {
#pragma unroll 1
      for (int k = k0;;) {
        const typename St::Record o = first;
        k += step;
        const bool more = k < P.n_parts;
        if (more) first.load(col + size_t(k) * size_t(P.N), fs);
        st.add(o, ref);
        if (!more) break;
      }
    }
  } else {
    if (any) st.add(first, ref);
    if (rr < n_rows) {
#pragma unroll 3
      for (int k = k0 + step; k < P.n_parts; k += step) {
        typename St::Record o;
        o.load(col + size_t(k) * size_t(P.N), fs);
        st.add(o, ref);
      }
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
__global__ void __launch_bounds__(32 * kWarps, kWarps == 8 ? 2 : 1)
    combine_kernel(LossPlan P, const float* part, int rows_per_block, int mode, float gamma,
                   const float* row_mask, const int32_t* corpus_tok, FullOut o, BatchOut bo) {
  __shared__ MergeSmem<FullState, kRows, kWarps> sm;
  __shared__ float s_loss[kRows], s_logp[kRows];
  const int row0 = blockIdx.x * rows_per_block;
  const int n_rows = min(rows_per_block, P.N - row0);
  merge_rows<FullState, kRows, kWarps>(P, part, row0, n_rows, sm);
  const bool erase = mode != 0;
  // one thread per row and side: both are log S - X / S_t with X = u (drafter: the loss) or w
  // (target: the entropy), two non-negative terms, in fp64.  The residual of the side's maximum
  // is in log S and in X / S_t alike (X's terms are the exponents themselves), and cancels.
  const int side = threadIdx.x / kRows, sr = threadIdx.x % kRows;
  if (side < 2 && sr < n_rows) {
    const FullState st = sm.get(0, sr);
    const int r = row0 + sr;
    const double ls = log(side == 0 ? st.sd : st.st);
    const double x = double(side == 0 ? st.u : st.w) * kLn2Double;
    const float v = float(ls - x / st.st);
    const float m = side == 0 ? st.bd : st.bt;
    const float lse = m + float(ls - ln_residual(m));
    if (side == 0) {
      o.loss_row[r] = v;
      s_loss[sr] = v;
      o.lse_d[r] = lse;
      o.argmax_d[r] = st.id;
      if (o.gap_d) o.gap_d[r] = st.bd - st.secd;
    } else {
      if (o.ent_row) o.ent_row[r] = v;
      o.lse_t[r] = lse;
      o.argmax_t[r] = st.it;
      if (o.gap_t) o.gap_t[r] = st.bt - st.sect;
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
__global__ void __launch_bounds__(32 * kWarps, 1)
    readout_combine_kernel(LossPlan P, const float* part, int has_corpus, int32_t* top_idx,
                           float* top_prob, float* tail, float* lse_t, int32_t* argmax_t,
                           float* gap_t, float* logp_x) {
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
      // with the factor that S carries
      const double e = exp(double(ti) - double(st.t[0]) + ln_residual(st.t[0]));
      s_e[i][rr] = e;
      top_idx[size_t(row0 + rr) * kTopK + i] = id;
      top_prob[size_t(row0 + rr) * kTopK + i] = float(e / st.s);
    }
  }
  __syncthreads();
  if (int(threadIdx.x) < n_rows) {
    const int rr = threadIdx.x, r = row0 + rr;
    const ReadoutState st = sm.get(0, rr);
    const double S = st.s, ls = log(S) - ln_residual(st.t[0]);
    double inside = 0.0;
#pragma unroll
    for (int i = 0; i < kTopK; ++i) inside += s_e[i][rr];
    // with V <= k every token is in the list and the tail is empty by definition
    tail[r] = P.V <= kTopK ? 0.f : float(fmax(0.0, (S - inside) / S));
    if (lse_t) lse_t[r] = st.t[0] + float(ls);
    if (argmax_t) argmax_t[r] = st.ti[0];
    if (gap_t) gap_t[r] = st.t[0] - st.t[1];
    if (has_corpus && logp_x) logp_x[r] = float((double(st.zx) - double(st.t[0])) - ls);
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
__global__ void __launch_bounds__(32 * kWarps, kWarps == 8 ? 2 : 1)
    topk_combine_kernel(LossPlan P, const float* part, int rows_per_block, const float* top_prob,
                        const float* tail, const float* row_mask, const float* weight_in,
                        float gamma, TopkOut o, BatchOut bo) {
  __shared__ MergeSmem<TopkState, kRows, kWarps> sm;
  const int row0 = blockIdx.x * rows_per_block;
  const int n_rows = min(rows_per_block, P.N - row0);
  merge_rows<TopkState, kRows, kWarps>(P, part, row0, n_rows, sm);
  double wl = 0.0, ws = 0.0;
  if (int(threadIdx.x) < n_rows) {         // n_rows <= 32: the first warp
    const int s = threadIdx.x % P.B, r = row0 + threadIdx.x;
    const TopkState st = sm.get(0, threadIdx.x);
    const double ls = log(st.s) - ln_residual(st.best);
    // log q_i = (z_i - M) - log S: the difference z_i - M is exact in fp64
    double ce = 0.0;
#pragma unroll
    for (int i = 0; i < kTopK; ++i)
      ce -= double(top_prob[size_t(r) * kTopK + i]) * ((double(st.z[i]) - double(st.best)) - ls);
    const double tq = fmax(st.so / st.s, 1e-30);
    const float tl = tail[r];
    if (tl > 0.f) ce -= double(tl) * log(tq);
    const float loss = float(ce);
    const float w = weight_in != nullptr
                        ? weight_in[r]
                        : expf(-float(s) / gamma) * (row_mask ? row_mask[r] : 1.f);
    o.loss_row[r] = loss;
    o.lse_d[r] = st.best + float(ls);
    o.tail_q[r] = float(tq);
    o.argmax_d[r] = st.id;
    if (o.gap_d) o.gap_d[r] = st.best - st.sec;
    o.weight[r] = w;
    wl = double(w) * double(loss);
    ws = double(w);
  }
  batch_sums<kWarps>(bo, wl, ws);
}

// ------------------------------------------------------------------ launch shape ---
// The smallest of 8, 16 or 32 rows that holds a whole anchor and 16 warps over the records (32
// warps leave a thread 64 registers and spill), as long as every such block has an SM; else 32 rows,
// whose record reads are whole 128-byte lines, and 8 warps.  Forward and top-8 forward, us, first ->
// second shape: 1920 x 64 x 151936 in anchors of 16 (120 blocks) 225 -> 226 and 153 -> 155; 4096 x
// 64 x 60000 in anchors of 16 (256) 226 -> 219 and 158 -> 152; 1600 x 64 x 20000 in anchors of 8
// (200) 51 -> 47 and 56 -> 50; 9000 x 64 x 20000 in anchors of 8 (1125) 197 -> 156 and 209 -> 153.
struct MergeShape {
  int rows, warps, rows_per_block, blocks;
};

MergeShape merge_shape(int N, int B, int sms) {
  MergeShape m{B <= 8 ? 8 : B <= 16 ? 16 : 32, 16, 0, 0};
  m.rows_per_block = m.rows / B * B;
  m.blocks = (N + m.rows_per_block - 1) / m.rows_per_block;
  if (m.blocks <= sms) return m;
  const int per32 = 32 / B * B;
  return MergeShape{32, 8, per32, (N + per32 - 1) / per32};
}

// The readout's rows are independent, and a merge of two top-8 lists costs several times a plain
// record's, so with more rows fewer lanes share one: 64, 16 or 8 (us, 64 -> 16 -> 8 lanes: 768 x 64
// x 151936 129 -> 133 -> 138; 1024 x 64 x 60000 93 -> 93 -> 98; 1920 x 64 x 151936 247 -> 231 ->
// 234; 4096 x 64 x 60000 243 -> 204 -> 203; 9000 x 64 x 20000 243 -> 178 -> 168).
constexpr int kReadoutFewRows = 1024;

MergeShape readout_shape(int N, int sms) {
  if (N < kReadoutFewRows) return MergeShape{8, 16, 8, (N + 7) / 8};
  if ((N + 15) / 16 <= 2 * sms) return MergeShape{16, 8, 16, (N + 15) / 16};
  return MergeShape{32, 8, 32, (N + 31) / 32};
}

}  // namespace

cudaError_t launch_combine(const LossPlan& plan, const float* part, int mode, float gamma,
                           const float* row_mask, const int32_t* corpus_tok, float* loss_row,
                           float* ent_row, float* lse_d, float* lse_t, int32_t* argmax_d,
                           int32_t* argmax_t, float* gap_d, float* gap_t, float* logp_x,
                           float* weight, double* block_part, unsigned* ticket, float lam,
                           float* loss_total, float* weight_sum, float* wl_sum, cudaStream_t s) {
  const MergeShape m = merge_shape(plan.N, plan.B, plan.sms);
  const FullOut o{loss_row, ent_row, lse_d,  lse_t,  argmax_d,
                  argmax_t, gap_d,   gap_t,  logp_x, weight};
  const BatchOut b{block_part, ticket, lam, loss_total, weight_sum, wl_sum};
  auto kern = m.warps == 8   ? combine_kernel<32, 8>
              : m.rows == 8  ? combine_kernel<8, 16>
              : m.rows == 16 ? combine_kernel<16, 16>
                             : combine_kernel<32, 16>;
  return launch_pdl(kern, m.blocks, 32 * m.warps, 0, s, plan, part, m.rows_per_block, mode, gamma,
                    row_mask, corpus_tok, o, b);
}

cudaError_t launch_readout_combine(const LossPlan& plan, const float* part, bool has_corpus,
                                   int32_t* top_idx, float* top_prob, float* tail, float* lse_t,
                                   int32_t* argmax_t, float* gap_t, float* logp_x,
                                   cudaStream_t s) {
  const MergeShape m = readout_shape(plan.N, plan.sms);
  auto kern = m.rows == 8    ? readout_combine_kernel<8, 16>
              : m.rows == 16 ? readout_combine_kernel<16, 8>
                             : readout_combine_kernel<32, 8>;
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
  const MergeShape m = merge_shape(plan.N, plan.B, plan.sms);
  const TopkOut o{loss_row, lse_d, tail_q, argmax_d, gap_d, weight};
  const BatchOut b{block_part, ticket, lam, loss_total, weight_sum, wl_sum};
  auto kern = m.warps == 8   ? topk_combine_kernel<32, 8>
              : m.rows == 8  ? topk_combine_kernel<8, 16>
              : m.rows == 16 ? topk_combine_kernel<16, 16>
                             : topk_combine_kernel<32, 16>;
  return launch_pdl(kern, m.blocks, 32 * m.warps, 0, s, plan, part, m.rows_per_block, top_prob,
                    tail, row_mask, weight_in, gamma, o, b);
}

}  // namespace alr
