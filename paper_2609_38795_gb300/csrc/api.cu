// C ABI of libalr (declared in include/alr.h): argument validation, tensor-map encoding,
// work planning and kernel launches.  No entry point allocates device memory.
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include <nvtx3/nvToolsExt.h>

#include "alr.h"
#include "cluster_forms.h"
#include "kernels.h"

namespace {

thread_local char g_err[1024] = "";

int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}

int cuda_fail(cudaError_t e, const char* what) {
  return fail(ALR_ERR_CUDA, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
}

std::mutex g_mu;

// Every compute entry point opens an NVTX range named after itself, so a profiler attached to
// the process shows each call as a span on the host timeline (and ncu can filter launches by
// it).  With no tool attached, push and pop return after one branch each.
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
  Range(const Range&) = delete;
  Range& operator=(const Range&) = delete;
};
#define ALR_RANGE() const Range alr_nvtx_range_(__func__)

// Test hook state: when set, the next launch of the fused loss kernel by a forward, or of the
// plain GEMM (any form), withholds its first pipeline stage.
std::atomic<int> g_withhold_next{0};

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

struct DevInfo {
  int sms = 0;
  int cc = 0;
};

int device_info(DevInfo* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  static DevInfo cache[64];
  if (dev < 0 || dev >= 64) return fail(ALR_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lk(g_mu);
  if (cache[dev].sms == 0) {
    int sms = 0, major = 0, minor = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev)) !=
            cudaSuccess ||
        (e = cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev)) != cudaSuccess)
      return cuda_fail(e, "cudaDeviceGetAttribute");
    cache[dev].sms = sms;
    cache[dev].cc = major * 10 + minor;
  }
  *out = cache[dev];
  return ALR_OK;
}

int require_sm103(DevInfo* info) {
  int rc = device_info(info);
  if (rc != ALR_OK) return rc;
  if (info->cc != 103)
    return fail(ALR_ERR_UNSUPPORTED,
                "libalr kernels are built for sm_103a only; current device is sm_%d", info->cc);
  return ALR_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

size_t elem_size(int dtype) { return dtype == ALR_BF16 ? 2 : 4; }

size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Element type of the kept logits for bf16 inputs (tensor maps only; not an ALR_* dtype).
constexpr int kMapF16 = 2;

// 2-D tiled tensor map (128-byte swizzle unless stated): `inner` contiguous elements per row,
// `outer` rows `row_bytes` apart; boxes of box_inner x box_outer elements.  dtype: ALR_BF16,
// ALR_F32 or kMapF16.
int make_map(CUtensorMap* m, const void* ptr, int dtype, uint64_t inner, uint64_t outer,
             uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer,
             CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  auto enc = encode_fn();
  if (enc == nullptr) return fail(ALR_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {row_bytes};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapDataType ty = dtype == ALR_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                 : dtype == kMapF16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                    : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  CUresult r = enc(m, ty,
                   2, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fail(ALR_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for %llu x %llu", int(r),
                (unsigned long long)inner, (unsigned long long)outer);
  return ALR_OK;
}

// K elements per 128-byte swizzle row, and MN elements per 128-byte chunk.
uint32_t k_per_row(int dtype) { return uint32_t(128 / elem_size(dtype)); }

int check_params(const alr_params* p) {
  if (p == nullptr) return fail(ALR_ERR_INVALID_ARG, "params is NULL");
  if (p->dtype != ALR_BF16 && p->dtype != ALR_F32)
    return fail(ALR_ERR_UNSUPPORTED, "dtype %d is not ALR_BF16 or ALR_F32", p->dtype);
  if (p->mode < ALR_MODE_ALR || p->mode > ALR_MODE_ERASE_HARD)
    return fail(ALR_ERR_UNSUPPORTED, "mode %d is not an ALR_MODE_* value", p->mode);
  if (p->B < 1 || p->B > 32) return fail(ALR_ERR_INVALID_ARG, "B = %d must lie in [1, 32]", p->B);
  if (p->N < 1 || p->N % p->B != 0)
    return fail(ALR_ERR_INVALID_ARG, "N = %lld must be a positive multiple of B = %d",
                (long long)p->N, p->B);
  if (p->N > (int64_t(1) << 30)) return fail(ALR_ERR_INVALID_ARG, "N = %lld too large", (long long)p->N);
  if (p->d < 8 || p->d % 8 != 0) return fail(ALR_ERR_INVALID_ARG, "d = %d must be a positive multiple of 8", p->d);
  if (p->V < 2 || p->V % 8 != 0) return fail(ALR_ERR_INVALID_ARG, "V = %d must be >= 2 and a multiple of 8", p->V);
  if (!(p->gamma > 0.f)) return fail(ALR_ERR_INVALID_ARG, "gamma must be > 0");
  if (!(p->lambda == p->lambda)) return fail(ALR_ERR_INVALID_ARG, "lambda is NaN");
  return ALR_OK;
}

// A kept logit matrix and its group references: both needed (and 16-byte aligned) for bf16
// inputs, whose logits are kept as fp16 relative to the references; fp32 inputs keep plain
// fp32 logits and ignore `ref`.
int check_kept(const alr_params* p, const void* Z, const void* ref, const char* name) {
  if (Z == nullptr || !aligned16(Z))
    return fail(ALR_ERR_INVALID_ARG, "%s must be non-NULL and 16-byte aligned", name);
  if (p->dtype == ALR_BF16 && (ref == nullptr || !aligned16(ref)))
    return fail(ALR_ERR_INVALID_ARG,
                "%s_ref (the fp16 group references of bf16 inputs) must be non-NULL and "
                "16-byte aligned", name);
  return ALR_OK;
}

// The fused loss kernels run on single CTAs unless the environment variable ALR_LOSS_FORM is
// "mcast" (bf16 inputs): clusters of two CTAs sharing every head tile by TMA multicast, from
// libalr_cluster.so, which only a single-process run loads (alr::cluster_forms() is nullptr in
// a multi-rank process, and then the single form runs).  The dual-product modes already share
// each head tile between z_d and z_t, and at the power cap the multicast form settles ~4 %
// lower in clock for ~1 % fewer L2 bytes per product: it is not faster, so it is not the
// default.  It needs 256-column tiles: where loss_tile_columns takes 128, single CTAs run.  The
// tiles and splits depend on the problem alone, so both forms give bit-identical results and take
// the same workspace.
bool loss_multicast(const alr_params* p) {
  if (p->dtype != ALR_BF16) return false;
  const char* v = getenv("ALR_LOSS_FORM");
  return v != nullptr && strcmp(v, "mcast") == 0 && alr::cluster_forms() != nullptr;
}

enum PlanKind { kPlanFwd, kPlanReadout, kPlanTopk };

// Vocabulary columns per tile.  256-column products read each operand byte from shared memory for
// twice the work, but their two accumulators fill tensor memory, so a tile's epilogue (6000 to
// 10000 cycles) is not hidden; 128-column tiles are double-buffered, their products slower.
// `n_rb`: row blocks (pairs in the two-row modes).
//   More wide tiles than SMs: narrow ones in the forwards up to 10 K blocks.  4096 x d x 32000,
//   us, 256 -> 128 columns: bf16, d = 256 forward 182 -> 160, keeping 245 -> 225, readout 177 ->
//   160; d = 512 239 -> 238, 310 -> 290, 211 -> 190; d = 640 270 -> 279, 341 -> 330, 227 -> 209;
//   d = 1000 404 -> 448; fp32, d = 320 298 -> 303, 641 -> 615, 255 -> 238.  (One row block, whose
//   W is read from memory once: 0.98 to 1.15 of the wide tiles' time.)
//   Otherwise each SM has one tile at most, and a narrow one is half as long, as long as these too
//   are at most one per SM (gradient of 16 x 3072 x 30000, 118 wide or 235 narrow tiles: 44 us
//   wide, 66 narrow; of 512 x 3072 x 4096, 64 or 128: 30 and 21).  In a forward every tile is a
//   split and its records cost the merge time: kMergeCycles a split against half a tile's cycles
//   (16 x 3072 x 4096 41.7 -> 34.3 us; 128 x 1024 x 16000 32.5 -> 36.0, x 3072 52.6 -> 48.7).
//   fp32 forwards have fewer splits than narrow tiles (forward_splits), so these only cost (512 x
//   256 x 4096: 24.2 -> 26.8 us).
constexpr int kNarrowBlocks = 10;

int loss_tile_columns(const alr_params* p, int sms, bool bwd, PlanKind kind, int64_t n_rb) {
  const int64_t n_wide = (p->V + 255) / 256, n_narrow = (p->V + 127) / 128;
  const int n_kb = (p->d + int(k_per_row(p->dtype)) - 1) / int(k_per_row(p->dtype));
  if (n_rb * n_wide > sms) return !bwd && n_kb <= kNarrowBlocks ? 128 : 256;
  if (n_rb * n_narrow > sms) return 256;
  if (bwd) return 128;
  if (p->dtype == ALR_F32) return 256;
  // cycles of a merged split (4, 2 and 2 records a row) and of a wide tile's epilogue
  constexpr int64_t kMergeCycles[] = {380, 295, 150}, kEpilogue[] = {7000, 20000, 7000};
  return 1090 * n_kb + kEpilogue[kind] > 2 * n_wide * kMergeCycles[kind] ? 128 : 256;
}

// Vocabulary splits of a forward over `rb` row blocks (row-block pairs in the two-row modes).
// CTAs take units (row block x split) in turn, so a round that is not full costs a whole unit:
// with 19 splits throughout, 9 row blocks are 171 units on 152 CTAs, two rounds for the work of
// one.  The split count is the one whose rounds times unit length (in vocabulary tiles, plus
// the fixed cost of a unit) is smallest; `base` (one round over `group` row blocks, 19 splits
// for 8) stays unless another promises 2 %.  More splits are more partial records: they take at
// most kPartBytes, or what 19 splits of 256-column tiles take, so every problem the no-workspace
// forward took still fits.
// Measured (us, 19 splits -> chosen): forward of 1152 x 1024 x 60000 358 -> 223, 2176 x 2048 x
// 100000 1443 -> 1150, 8320 x 1024 x 32000 857 -> 760, 1920 x 4096 x 151936 2770 -> 2677; label
// readout of 4096 x 2048 x 32000 533 -> 431.
constexpr int64_t kPartBytes = 48ll << 20;
constexpr int64_t kMaxRecordBytes = 4 * int64_t(sizeof(float)) * alr::kPFields;   // row and split

int forward_splits(const alr_params* p, int sms, int rb, int bn, int n_vt, int group,
                   PlanKind kind) {
  const int round = std::max(1, sms / std::min(rb, group));
  // 19 splits of 256-column tiles, 15 fields: the records the no-workspace limit was set for
  const int64_t wide = std::min((p->V + 255) / 256, round) * 4 * 15 * int64_t(sizeof(float));
  const int64_t fit = std::max((wide * p->N - 2048) / (kMaxRecordBytes * p->N),
                               p->dtype == ALR_BF16 ? kPartBytes / (kMaxRecordBytes * p->N) : 0);
  const int most = int(std::min<int64_t>(n_vt, std::max<int64_t>(1, fit)));
  const int base = std::min(most, round);
  // cycles of one tile: two 128 x 256 products over d (about 1090 per 64 of d) and an epilogue of
  // about 7000; a 128-column tile, its epilogue hidden, 0.65 of such products.  (Alone it takes 0.78
  // of them at d = 1000 to 0.97 at 384, but that weight, 0.87, ranks the split counts worse, taking
  // more of them: 1088 x 640 x 60000 152 -> 159 us, 4320 x 512 x 60000 453 -> 461; 6784 x 640 x
  // 1400 53 -> 51.)  A unit adds its first loads and its record, about 2500, and in the
  // readout the filling of its top-8 lists, about 25000; a split adds its records' trip through
  // memory (at about 2800 bytes a cycle).
  const double products = 1090.0 * ((p->d + 63) / 64) * (p->dtype == ALR_BF16 ? 1 : 2);
  const double tile = bn == 256 ? products + 7000.0 : std::max(0.65 * products, 4500.0);
  const double per_unit = (kind == kPlanReadout ? 27500.0 : 2500.0) / tile;
  const double per_split = 2.0 * double(p->N) * kMaxRecordBytes / 2800.0 / tile;
  auto cost = [&](int vs) {
    const int rounds = int((int64_t(rb) * vs + sms - 1) / sms);
    const double mean = double(n_vt) / vs, longest = (n_vt + vs - 1) / vs;
    // splits differ by one tile at most, and successive groups rotate them over the CTAs
    return std::min(rounds * longest, rounds * mean + 1.0) + rounds * per_unit + vs * per_split;
  };
  int best = base;
  double best_cost = 0.98 * cost(base);
  for (int vs = 1; vs <= most; ++vs)
    if (cost(vs) < best_cost) {
      best_cost = cost(vs);
      best = vs;
    }
  return best;
}

// kind: the readout and the top-k modes are the single-operand ones, whose units hold two row
// blocks.
alr::LossPlan loss_plan(const alr_params* p, int sms, bool bwd, PlanKind kind = kPlanFwd) {
  const bool two_rows = kind != kPlanFwd;
  alr::LossPlan P{};
  P.N = int(p->N);
  P.d = p->d;
  P.V = p->V;
  P.B = p->B;
  P.sms = sms;
  P.products = two_rows ? 1 : 2;
  // row blocks; row-block pairs for the two-row modes and for the multicast form (which
  // places sms / 2 clusters).  Forward: the splits of forward_splits (the same for both
  // forms), in raster groups of up to two rounds of the grid at its base split (16 row blocks).
  // Recomputing backward: one vocabulary tile per unit, raster groups of 16 row blocks as well.
  const int rb = int((p->N + 127) / 128);
  P.bn = loss_tile_columns(p, sms, bwd, kind, two_rows ? (rb + 1) / 2 : rb);
  P.mc = !two_rows && P.bn == 256 && loss_multicast(p) ? 1 : 0;
  const bool pairs = P.mc || two_rows;
  P.n_rb = pairs ? (rb + 1) / 2 : rb;
  const int group = pairs ? 4 : 8;
  P.n_vt = (p->V + P.bn - 1) / P.bn;
  // two rounds per raster group: twice the row blocks share each W split, so W leaves DRAM
  // about half as often, with the same number of units per CTA (forward 49.8 against 50.0 ms at
  // the text8b size, recomputed logit gradient 46.2 against 46.4 ms with 8, three alternating
  // A/B rounds)
  P.group_rows = P.n_rb < 2 * group ? P.n_rb : 2 * group;
  if (bwd) {
    P.n_vs = P.n_vt;  // one tile per unit
  } else {
    P.n_vs = forward_splits(p, sms, two_rows ? P.n_rb : rb, P.bn, P.n_vt, two_rows ? 4 : 8, kind);
    // groups of equal size: 17 row blocks are 9 + 8, not 16 + 1 (in the backward's short units
    // the smaller groups only cost sharing: 2176 x 2048 x 100000 1071 -> 1105 us)
    const int n_groups = (P.n_rb + P.group_rows - 1) / P.group_rows;
    P.group_rows = (P.n_rb + n_groups - 1) / n_groups;
  }
  // partial records per row and split: one per epilogue column group
  P.n_parts = P.n_vs * (two_rows ? 2 : 4);
  P.n_units = P.n_rb * P.n_vs;
  P.grid = sms < P.n_units ? sms : P.n_units;
  return P;
}

// fp32 inputs run tf32 products, which take K-major operands only: the head is then read from
// a transposed copy W^T [V, d] placed in the workspace.
// Forward-type workspace: `fields` partial statistics per row and part, one fp64 pair per
// anchor and the merge kernel's ticket, and W^T for fp32 inputs.
struct FwdLayout {
  size_t part_off, anchor_off, ticket_off, wt_off, total;
};

FwdLayout fwd_layout(const alr_params* p, int sms, PlanKind kind = kPlanFwd) {
  const int fields = kind == kPlanFwd       ? alr::kPFields
                     : kind == kPlanReadout ? alr::kRFields
                                            : alr::kKFields;
  const alr::LossPlan P = loss_plan(p, sms, false, kind);
  FwdLayout L{};
  L.part_off = 0;
  L.anchor_off = round_up(size_t(fields) * P.n_parts * size_t(P.N) * sizeof(float), 1024);
  L.ticket_off = L.anchor_off + 2 * sizeof(double) * size_t(P.N / P.B);
  L.wt_off = round_up(L.ticket_off + 16, 1024);
  L.total = L.wt_off;
  if (p->dtype == ALR_F32) L.total += round_up(size_t(p->V) * p->d * sizeof(float), 1024);
  return L;
}

// Backward workspace: G [N, V]; for fp32 also W^T [V, d], G^T [V, N'] and H_d^T [d, N'] with
// N' = N rounded up to 4 (16-byte rows).
struct BwdLayout {
  size_t g_off, wt_off, gt_off, hdt_off, total;
  int64_t ld_n;
};

// with_g = false: the layout of the backward from kept logits, whose G is the caller's and
// which needs no W^T (G^T and H_d^T only, for fp32).
BwdLayout bwd_layout(const alr_params* p, bool with_g = true) {
  BwdLayout L{};
  const size_t es = p->dtype == ALR_BF16 ? 2 : 4;
  L.g_off = 0;
  L.total = with_g ? round_up(size_t(p->N) * size_t(p->V) * es, 1024) : 0;
  L.ld_n = (p->N + 3) / 4 * 4;
  if (p->dtype == ALR_F32) {
    L.wt_off = L.total;
    L.gt_off = L.wt_off + (with_g ? round_up(size_t(p->V) * p->d * 4, 1024) : 0);
    L.hdt_off = L.gt_off + round_up(size_t(p->V) * L.ld_n * 4, 1024);
    L.total = L.hdt_off + round_up(size_t(p->d) * L.ld_n * 4, 1024);
  }
  return L;
}

// Forms of the products.  The environment variable ALR_GEMM_FORM names one for every bf16 product:
//   "mcast"   clusters of two CTAs, each on a 128 x 256 tile, sharing every B tile by TMA
//             multicast;
//   "mcast4"  as "mcast" with clusters of four CTAs, each loading a quarter of the B tile;
//   "single"  one CTA per 128 x 256 tile, each loading its own B tiles (plain_gemm.cu);
//   "pair"    CTA pairs with M = 256 products.
// Unset, choose_gemm() picks single, mcast or pair, or the split of a tile's K over a cluster, by
// the sizes.  The cluster forms ("mcast", "mcast4", "pair") live in libalr_cluster.so
// (csrc_cluster/), which only a single-process run loads: in a process that is one rank of
// several, or where that library cannot be loaded, every named form runs as "single"
// (alr_kernel_forms reports it).  tf32 products run on single CTAs or split K.
enum GemmForm { kGemmSingle = 0, kGemmMcast = 1, kGemmPair = 2, kGemmMcast4 = 3 };

GemmForm gemm_form(int dtype) {
  if (dtype != ALR_BF16) return kGemmSingle;
  const char* v = getenv("ALR_GEMM_FORM");
  if ((v != nullptr && strcmp(v, "single") == 0) || alr::cluster_forms() == nullptr)
    return kGemmSingle;
  if (v != nullptr && strcmp(v, "pair") == 0) return kGemmPair;
  if (v != nullptr && strcmp(v, "mcast4") == 0) return kGemmMcast4;
  return kGemmMcast;
}

// How one product runs: its form, and the CTAs per tile of the split form (then `form` is
// kGemmSingle).
struct GemmChoice {
  GemmForm form;
  int split;
};

// The form of a product when none is asked for by name: the cheapest by a cost in 0.01 us, from
// the rounds a form needs over the SMs and a fixed time per K block (64 bf16) and per launch,
// fitted to the measurements below (us, random operands, timed alone).
//   pair    27 per K block: six 32 KB stages per CTA ride out more load latency than four 48 KB
//           ones (which take 600-690 cycles per K block, 512 being the tensor pipe's time), and
//           B is read once per pair.  It draws more power per product, though: at
//           the text8b size (4.1e13 flop per product, the step at the power cap throughout) dH
//           and dW gain 1.5 ms and the forward behind them loses 5, 102.5 -> 106.1 ms per step;
//           at 1.0e13 the step gains 1 %, at 2.4e12 4 %, at 5.4e11 5 %.  So: up to kPairFlops,
//           where it turns (step at d = 4096, V = 151936, ms, mcast -> pair: 8192 rows, 1.0e13 flop
//           a product, 26.7 -> 26.4; 12288, 1.5e13, 40.1 -> 40.5; 16384 53.2 -> 54.2; 24576 80.2 ->
//           81.9).
//   mcast   35.5 per K block; single 42, but no cluster has to be placed and an odd row block
//           leaves no CTA idle (128 x 32000 x 512: 9.4 against 15.4 us).
//   split   few tiles, long K: `split` CTAs per tile fill SMs that would idle.  128 x 4096 x
//           151936: 823 (mcast) -> 208 us (6 CTAs); 512 x 4096 x 151936: 632 (pair) -> 460 (2);
//           2000 x 1000 x 60000: 255 (pair) -> 178 (2); 16 x 2048 x 32000: 174 -> 37 (12); 300 x
//           512 x 4000: 23 -> 15 (5).  No gain past one tile per SM (1920 x 4096 x 151936: 1663
//           against 1762).  Taken where it promises 10 %.
constexpr double kPairFlops = 1.5e13;
// Below, the start of a pair's tile costs what it saves (dW at d = 4096, V = 151936: K = 1024 1206
// mcast, 1220 pair; 1920 1831 mcast, 1691 pair).
constexpr int64_t kPairMinBlocks = 24;

GemmChoice choose_gemm(int dtype, int M, int Nc, int K, int sms) {
  GemmChoice best{gemm_form(dtype), 1};
  const char* v = getenv("ALR_GEMM_FORM");
  if (v != nullptr && *v != '\0') return best;
  const int64_t n_mb = (M + 127) / 128, n_nb = (Nc + 255) / 256, tiles = n_mb * n_nb;
  const int64_t n_kb = (int64_t(K) + k_per_row(dtype) - 1) / k_per_row(dtype);
  auto rounds = [](int64_t units, int64_t at_once) { return (units + at_once - 1) / at_once; };

  best = GemmChoice{kGemmSingle, 1};
  int64_t best_cost = rounds(tiles, sms) * n_kb * 42;
  const alr::ClusterForms* cf = dtype == ALR_BF16 ? alr::cluster_forms() : nullptr;
  if (cf != nullptr) {
    const int64_t units = (n_mb + 1) / 2 * n_nb;   // both cluster forms take two row blocks
    const int clusters = cf->gemm_max_clusters(2);
    if (clusters > 0) {
      const int64_t cost = rounds(units, clusters) * n_kb * 71 / 2 + 60;
      if (cost < best_cost) {
        best_cost = cost;
        best = GemmChoice{kGemmMcast, 1};
      }
    }
    if (n_kb >= kPairMinBlocks && 2.0 * M * Nc * K <= kPairFlops) {
      const int pairs = cf->pair_gemm_max_pairs();
      const int64_t cost = pairs > 0 ? rounds(units, pairs) * n_kb * 27 + 150 : best_cost;
      if (cost < best_cost) {
        best_cost = cost;
        best = GemmChoice{kGemmPair, 1};
      }
    }
  }
  if (tiles >= sms) return best;
  best_cost = best_cost * 9 / 10;
  for (int split : {2, 3, 4, 5, 6, 7, 8, 10, 12, 16}) {
    if (split > n_kb) break;
    const int clusters = alr::plain_gemm_split_clusters(split);
    if (clusters < 1) continue;
    const int64_t cost =
        rounds(tiles, clusters) * ((n_kb + split - 1) / split * 36 + 290 + 70 * split);
    if (cost < best_cost) {
      best_cost = cost;
      best = GemmChoice{kGemmSingle, split};
    }
  }
  return best;
}

// Rows of a K-major B box (B columns loaded by one copy).
uint32_t gemm_b_rows(const GemmChoice& c) {
  switch (c.form) {
    case kGemmSingle: return 256;
    case kGemmMcast4: return 64;
    default: return 128;
  }
}

// Up to this K the accumulating products are bound by the traffic of C, which the L2 prefetch helps
// (dW at d = 4096, V = 151936, with two pieces ahead: K = 128 1060 -> 968 us, 512 1091 -> 1079);
// beyond, it only competes with the operands' loads (1024: 1206 -> 1226, 1920: 1691 -> 1780).
// With a tile or two per CTA there is nothing to run ahead of.
constexpr int kPrefetchK = 512;

alr::GemmArgs gemm_plan(int M, int Nc, int K, float* C, int64_t ldc, int sms) {
  alr::GemmArgs g{};
  g.M = M;
  g.Nc = Nc;
  g.K = K;
  g.C = C;
  g.ldc = ldc;
  g.n_mb = (M + 127) / 128;
  g.n_nb = (Nc + 255) / 256;
  g.group_m = g.n_mb < 16 ? g.n_mb : 16;
  g.n_tiles = g.n_mb * g.n_nb;
  g.prefetch_c = K <= kPrefetchK && g.n_tiles >= 2 * sms ? 1 : 0;
  g.grid = sms < g.n_tiles ? sms : g.n_tiles;
  return g;
}

// Plan of the pair GEMM: 256 x 256 tiles over `pairs` resident CTA pairs.
alr::GemmArgs pair_gemm_plan(int M, int Nc, int K, float* C, int64_t ldc, int pairs) {
  alr::GemmArgs g{};
  g.M = M;
  g.Nc = Nc;
  g.K = K;
  g.C = C;
  g.ldc = ldc;
  g.n_mb = (M + 255) / 256;
  g.n_nb = (Nc + 255) / 256;
  g.group_m = g.n_mb < 8 ? g.n_mb : 8;
  g.n_tiles = g.n_mb * g.n_nb;
  g.prefetch_c = K <= kPrefetchK && g.n_tiles >= 2 * pairs ? 1 : 0;
  g.grid = 2 * (pairs < g.n_tiles ? pairs : g.n_tiles);
  return g;
}

// C (+)= A B with the operand maps already encoded (B boxes of gemm_b_rows(c) rows).
int launch_gemm(const GemmChoice& c, int dt, bool a_mn, bool b_mn, bool acc, const CUtensorMap& ma,
                const CUtensorMap& mb, int M, int Nc, int K, float* C, int64_t ldc, int sms,
                cudaStream_t s, const char* what) {
  cudaError_t e;
  const GemmForm form = c.form;
  const alr::ClusterForms* cf = alr::cluster_forms();   // non-NULL for every cluster form
  if (form == kGemmPair) {
    const int pairs = cf->pair_gemm_max_pairs();
    if (pairs < 1) return fail(ALR_ERR_CUDA, "%s: no CTA pair of the GEMM fits on this device", what);
    alr::GemmArgs g = pair_gemm_plan(M, Nc, K, C, ldc, pairs);
    g.status = alr::device_status_ptr();
    if (g.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
    g.withhold_first_stage = g_withhold_next.exchange(0);
    e = cf->launch_pair_gemm(a_mn, b_mn, acc, &ma, &mb, &g, s);
  } else if (form == kGemmMcast || form == kGemmMcast4) {
    const int cl = form == kGemmMcast4 ? 4 : 2;
    const int clusters = cf->gemm_max_clusters(cl);
    if (clusters < 1)
      return fail(ALR_ERR_CUDA, "%s: no CTA cluster of the GEMM fits on this device", what);
    // 128-row blocks in groups of `cl`: n_mb counts groups, raster groups of 16 row blocks
    alr::GemmArgs g = gemm_plan(M, Nc, K, C, ldc, sms);
    g.n_mb = ((M + 127) / 128 + cl - 1) / cl;
    const int gm = 16 / cl;
    g.group_m = g.n_mb < gm ? g.n_mb : gm;
    g.n_tiles = g.n_mb * g.n_nb;
    g.grid = cl * (clusters < g.n_tiles ? clusters : g.n_tiles);
    g.status = alr::device_status_ptr();
    if (g.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
    g.withhold_first_stage = g_withhold_next.exchange(0);
    e = cf->launch_gemm(cl, a_mn, b_mn, acc, &ma, &mb, &g, s);
  } else {
    alr::GemmArgs g = gemm_plan(M, Nc, K, C, ldc, sms);
    g.split = c.split;
    g.status = alr::device_status_ptr();
    if (g.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
    g.withhold_first_stage = g_withhold_next.exchange(0);
    e = alr::launch_plain_gemm(dt, a_mn, b_mn, acc, ma, mb, g, s);
  }
  if (e != cudaSuccess) return cuda_fail(e, what);
  return ALR_OK;
}

// Tensor map of the head operand of the fused loss kernels: MN-major tiles straight from
// W [d, V] for bf16; for fp32, W is first transposed into `wt` and read K-major.
int head_map(CUtensorMap* m, const alr_params* p, const void* W, void* wt, int bn,
             cudaStream_t s) {
  const uint32_t kke = k_per_row(p->dtype);
  if (p->dtype == ALR_BF16) return make_map(m, W, ALR_BF16, p->V, p->d, uint64_t(p->V) * 2, kke, kke);
  cudaError_t e = alr::launch_transpose32(static_cast<const float*>(W), static_cast<float*>(wt),
                                          p->d, p->V, p->d, s);
  if (e != cudaSuccess) return cuda_fail(e, "head transpose launch");
  return make_map(m, wt, ALR_F32, p->d, p->V, uint64_t(p->d) * 4, kke, uint32_t(bn));
}

// The full-vocabulary forward; with Zd / Zt given, the fused kernel also writes both logit
// matrices (kModeFwdKeep).
int fwd_impl(const alr_params* p, const void* Hd, const void* Ht, const void* W,
             const float* row_mask, const int32_t* corpus_tok, void* Zd, void* Zt,
             uint16_t* Zd_ref, uint16_t* Zt_ref, const alr_fwd_outputs* out, void* workspace,
             size_t ws_bytes, void* stream) {
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if (Hd == nullptr || Ht == nullptr || W == nullptr || out == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "Hd, Ht, W and out must be non-NULL");
  if (!aligned16(Hd) || !aligned16(Ht) || !aligned16(W))
    return fail(ALR_ERR_INVALID_ARG, "Hd, Ht and W must be 16-byte aligned");
  if (out->loss_row == nullptr || out->lse_d == nullptr || out->lse_t == nullptr ||
      out->argmax_d == nullptr || out->argmax_t == nullptr || out->weight == nullptr ||
      out->loss_total == nullptr || out->weight_sum == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "a required forward output pointer is NULL");
  if (p->mode != ALR_MODE_ALR && corpus_tok == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "the erase modes need corpus_tok");
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  const FwdLayout lay = fwd_layout(p, info.sms);
  if (workspace == nullptr || ws_bytes < lay.total)
    return fail(ALR_ERR_INVALID_ARG, "workspace of %zu bytes is smaller than the %zu needed",
                ws_bytes, lay.total);
  if (!aligned16(workspace)) return fail(ALR_ERR_INVALID_ARG, "workspace must be 16-byte aligned");

  const int dt = p->dtype;
  const size_t es = elem_size(dt);
  const uint32_t kke = k_per_row(dt);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  CUtensorMap m_hd, m_ht, m_w;
  if ((rc = make_map(&m_hd, Hd, dt, p->d, p->N, p->d * es, kke, 128)) != ALR_OK) return rc;
  if ((rc = make_map(&m_ht, Ht, dt, p->d, p->N, p->d * es, kke, 128)) != ALR_OK) return rc;
  alr::LossArgs args{};
  args.plan = loss_plan(p, info.sms, false);
  if ((rc = head_map(&m_w, p, W, ws + lay.wt_off, args.plan.bn, s)) != ALR_OK) return rc;
  args.part = reinterpret_cast<float*>(ws + lay.part_off);
  args.ticket = reinterpret_cast<unsigned*>(ws + lay.ticket_off);
  args.corpus_tok = p->mode != ALR_MODE_ALR ? corpus_tok : nullptr;
  args.lam = p->lambda;
  args.withhold_first_stage = g_withhold_next.exchange(0);
  args.status = alr::device_status_ptr();
  if (args.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
  args.zd_out = Zd;
  args.zt_out = Zt;
  args.zd_ref = Zd_ref;
  args.zt_ref = Zt_ref;
  // bf16 inputs keep fp16 logits through TMA stores of 16-column x 32-row boxes
  CUtensorMap m_zd = m_w, m_zt = m_w;
  if (Zd != nullptr && dt == ALR_BF16) {
    if ((rc = make_map(&m_zd, Zd, kMapF16, p->V, p->N, uint64_t(p->V) * 2, 16, 32,
                       CU_TENSOR_MAP_SWIZZLE_NONE)) != ALR_OK)
      return rc;
    if ((rc = make_map(&m_zt, Zt, kMapF16, p->V, p->N, uint64_t(p->V) * 2, 16, 32,
                       CU_TENSOR_MAP_SWIZZLE_NONE)) != ALR_OK)
      return rc;
  }
  e = alr::launch_loss_kernel(Zd != nullptr ? alr::kModeFwdKeep : alr::kModeFwd, dt, m_hd, m_ht,
                              m_w, m_zd, m_zt, args, s);
  if (e != cudaSuccess) return cuda_fail(e, "forward loss kernel launch");
  double* anchor = reinterpret_cast<double*>(ws + lay.anchor_off);
  e = alr::launch_combine(args.plan, args.part, p->mode, p->gamma, row_mask, args.corpus_tok,
                          out->loss_row, out->ent_row, out->lse_d, out->lse_t, out->argmax_d,
                          out->argmax_t, out->gap_d, out->gap_t, out->logp_x, out->weight, anchor,
                          args.ticket, p->lambda, out->loss_total, out->weight_sum, out->wl_sum, s);
  if (e != cudaSuccess) return cuda_fail(e, "combine launch");
  return ALR_OK;
}

}  // namespace

namespace alr {
int set_last_error(int code, const char* msg) { return fail(code, "%s", msg); }
}  // namespace alr

extern "C" {

const char* alr_version(void) { return "libalr 0.1 (sm_103a)"; }

int alr_kernel_forms(int32_t* gemm, int32_t* loss) {
  if (gemm == nullptr || loss == nullptr) return fail(ALR_ERR_INVALID_ARG, "gemm and loss must be non-NULL");
  alr_params p{};
  p.dtype = ALR_BF16;
  *gemm = int32_t(gemm_form(ALR_BF16));
  *loss = loss_multicast(&p) ? 1 : 0;
  return ALR_OK;
}

const char* alr_cluster_forms_error(void) {
  return alr::cluster_forms() != nullptr ? "" : alr::cluster_forms_error();
}

int alr_debug_withhold_next_stage(int enable) {
  g_withhold_next.store(enable ? 1 : 0);
  return ALR_OK;
}

const char* alr_last_error(void) { return g_err; }

int alr_device_supported(void) {
  DevInfo info;
  return require_sm103(&info);
}

int alr_device_status(void* stream, int clear) {
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  int* w = alr::device_status_ptr();
  if (w == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
  int v = 0;
  if ((e = cudaMemcpy(&v, w, sizeof(int), cudaMemcpyDeviceToHost)) != cudaSuccess)
    return cuda_fail(e, "reading the status word");
  if (clear) {
    const int z = 0;
    if ((e = cudaMemcpy(w, &z, sizeof(int), cudaMemcpyHostToDevice)) != cudaSuccess)
      return cuda_fail(e, "clearing the status word");
  }
  if (v != 0) return fail(ALR_ERR_TIMEOUT, "a device pipeline wait timed out");
  return ALR_OK;
}

int alr_gather_ira_blocks(const void* feat, int32_t S, int32_t L, int32_t d, int32_t dtype,
                          const int32_t* seq, const int32_t* pos, const int32_t* valid_len,
                          int32_t A, int32_t B, void* out, float* row_valid, void* stream) {
  ALR_RANGE();
  if (dtype != ALR_BF16 && dtype != ALR_F32) return fail(ALR_ERR_UNSUPPORTED, "dtype %d", dtype);
  if (S < 1 || L < 1 || d < 1 || A < 0 || B < 1)
    return fail(ALR_ERR_INVALID_ARG, "bad sizes S=%d L=%d d=%d A=%d B=%d", S, L, d, A, B);
  if ((size_t(d) * elem_size(dtype)) % 16 != 0)
    return fail(ALR_ERR_INVALID_ARG, "d * element size must be a multiple of 16 bytes");
  if (A == 0) return ALR_OK;
  if (feat == nullptr || seq == nullptr || pos == nullptr || out == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "feat, seq, pos and out must be non-NULL");
  if (!aligned16(feat) || !aligned16(out))
    return fail(ALR_ERR_INVALID_ARG, "feat and out must be 16-byte aligned");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_gather(feat, S, L, d, int(elem_size(dtype)), seq, pos, valid_len, A,
                                     B, out, row_valid, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "gather launch");
  return ALR_OK;
}

size_t alr_fwd_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  DevInfo info;
  if (device_info(&info) != ALR_OK) return 0;
  return fwd_layout(p, info.sms).total;
}

int alr_slot_loss_fwd(const alr_params* p, const void* Hd, const void* Ht, const void* W,
                      const float* row_mask, const int32_t* corpus_tok, const alr_fwd_outputs* out,
                      void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  return fwd_impl(p, Hd, Ht, W, row_mask, corpus_tok, nullptr, nullptr, nullptr, nullptr, out,
                  workspace, ws_bytes, stream);
}

int alr_slot_loss_fwd_keep_logits(const alr_params* p, const void* Hd, const void* Ht,
                                  const void* W, const float* row_mask, const int32_t* corpus_tok,
                                  void* Zd, void* Zt, uint16_t* Zd_ref, uint16_t* Zt_ref,
                                  const alr_fwd_outputs* out, void* workspace, size_t ws_bytes,
                                  void* stream) {
  ALR_RANGE();
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if ((rc = check_kept(p, Zd, Zd_ref, "Zd")) != ALR_OK) return rc;
  if ((rc = check_kept(p, Zt, Zt_ref, "Zt")) != ALR_OK) return rc;
  return fwd_impl(p, Hd, Ht, W, row_mask, corpus_tok, Zd, Zt, Zd_ref, Zt_ref, out, workspace,
                  ws_bytes, stream);
}

int32_t alr_kept_ref_groups(int32_t V) {
  return V < 1 ? 0 : (V + alr::kKeepGroup - 1) / alr::kKeepGroup;
}

size_t alr_bwd_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  return bwd_layout(p).total;
}

}  // extern "C"

namespace {

// Checks shared by the backward entry points; fills `info`.
int check_bwd_args(const alr_params* p, const void* Hd, const void* Ht, const void* W,
                   const float* weight, const float* weight_sum, const float* lse_d,
                   const float* lse_t, DevInfo* info) {
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if (Hd == nullptr || Ht == nullptr || W == nullptr || weight == nullptr ||
      weight_sum == nullptr || lse_d == nullptr || lse_t == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "a required backward input pointer is NULL");
  if (!aligned16(Hd) || !aligned16(Ht) || !aligned16(W))
    return fail(ALR_ERR_INVALID_ARG, "Hd, Ht and W must be 16-byte aligned");
  return require_sm103(info);
}

// Compact-label inputs of the top-k path (all NULL for the full-vocabulary loss).
struct TopkLabels {
  const int32_t* idx = nullptr;
  const float* prob = nullptr;
  const float* tail = nullptr;
  const float* tail_q = nullptr;
};

// The fused logit-gradient kernel: G = lambda omega / sum omega (q - p) for the full
// vocabulary (Ht given), or the top-k + tail form (labels given), recomputing the tiles.
int logit_grad_impl(const alr_params* p, const void* Hd, const void* Ht, const void* W,
                    const float* weight, const float* weight_sum, const float* lse_d,
                    const float* lse_t, const TopkLabels& lab, void* G, void* wt,
                    const DevInfo& info, cudaStream_t s) {
  const int dt = p->dtype;
  const size_t es = elem_size(dt);
  const uint32_t kke = k_per_row(dt);
  const bool topk = lab.idx != nullptr;
  int rc;
  CUtensorMap m_hd, m_ht, m_w, m_gs;
  if ((rc = make_map(&m_hd, Hd, dt, p->d, p->N, p->d * es, kke, 128)) != ALR_OK) return rc;
  m_ht = m_hd;
  if (!topk && (rc = make_map(&m_ht, Ht, dt, p->d, p->N, p->d * es, kke, 128)) != ALR_OK) return rc;
  const alr::LossPlan plan = loss_plan(p, info.sms, true, topk ? kPlanTopk : kPlanFwd);
  if ((rc = head_map(&m_w, p, W, wt, plan.bn, s)) != ALR_OK) return rc;
  m_gs = m_w;
  if (dt == ALR_BF16 &&
      (rc = make_map(&m_gs, G, dt, p->V, p->N, p->V * es, 16, 32, CU_TENSOR_MAP_SWIZZLE_NONE)) != ALR_OK)
    return rc;
  alr::LossArgs args{};
  args.plan = plan;
  args.G = G;
  args.lse_d = lse_d;
  args.lse_t = lse_t;
  args.weight = weight;
  args.weight_sum = weight_sum;
  args.lam = p->lambda;
  args.top_idx = lab.idx;
  args.top_prob = lab.prob;
  args.tail = lab.tail;
  args.tail_q = lab.tail_q;
  args.status = alr::device_status_ptr();
  if (args.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
  cudaError_t e = alr::launch_loss_kernel(topk ? alr::kModeTopkBwd : alr::kModeBwd, dt, m_hd, m_ht,
                                          m_w, m_gs, m_gs, args, s);
  if (e != cudaSuccess) return cuda_fail(e, "logit-gradient kernel launch");
  return ALR_OK;
}

// dH_d = G W^T and, when dW is given, dW += H_d^T G (fp32 via transposed workspace copies).
int head_grads_impl(const alr_params* p, const void* Hd, const void* W, const void* G, float* dHd,
                    float* dW, uint8_t* ws, const BwdLayout& lay, const DevInfo& info,
                    cudaStream_t s) {
  const int dt = p->dtype;
  const size_t es = elem_size(dt);
  const uint32_t kke = k_per_row(dt);
  int rc;
  cudaError_t e;
  // dH_d = G W^T: A = G [N, V] K-major, B = W [d, V] K-major.
  CUtensorMap m_ga, m_wk;
  const GemmChoice dh = choose_gemm(dt, int(p->N), p->d, p->V, info.sms);
  if ((rc = make_map(&m_ga, G, dt, p->V, p->N, p->V * es, kke, 128)) != ALR_OK) return rc;
  if ((rc = make_map(&m_wk, W, dt, p->V, p->d, p->V * es, kke, gemm_b_rows(dh))) != ALR_OK)
    return rc;
  if ((rc = launch_gemm(dh, dt, false, false, false, m_ga, m_wk, int(p->N), p->d, p->V, dHd, p->d,
                        info.sms, s, "dH GEMM launch")) != ALR_OK)
    return rc;
  if (dW == nullptr) return ALR_OK;
  CUtensorMap m_ha, m_gb;
  const GemmChoice dw = choose_gemm(dt, p->d, p->V, int(p->N), info.sms);
  if (dt == ALR_BF16) {
    // dW += H_d^T G: A = H_d read as [K = N, M = d] (MN-major), B = G [K = N, V] (MN-major).
    if ((rc = make_map(&m_ha, Hd, dt, p->d, p->N, p->d * es, kke, kke)) != ALR_OK) return rc;
    if ((rc = make_map(&m_gb, G, dt, p->V, p->N, p->V * es, kke, kke)) != ALR_OK) return rc;
    return launch_gemm(dw, dt, true, true, true, m_ha, m_gb, p->d, p->V, int(p->N), dW, p->V,
                       info.sms, s, "dW GEMM launch");
  } else {
    // K-major operands from transposed copies H_d^T [d, N'] and G^T [V, N'].
    float* hdt = reinterpret_cast<float*>(ws + lay.hdt_off);
    float* gt = reinterpret_cast<float*>(ws + lay.gt_off);
    if ((e = alr::launch_transpose32_pair(static_cast<const float*>(Hd), hdt, p->d,
                                          static_cast<const float*>(G), gt, p->V, int(p->N),
                                          int(lay.ld_n), s)) != cudaSuccess)
      return cuda_fail(e, "H_d and G transpose launch");
    if ((rc = make_map(&m_ha, hdt, dt, p->N, p->d, lay.ld_n * 4, kke, 128)) != ALR_OK) return rc;
    if ((rc = make_map(&m_gb, gt, dt, p->N, p->V, lay.ld_n * 4, kke, gemm_b_rows(dw))) != ALR_OK)
      return rc;
    return launch_gemm(dw, dt, false, false, true, m_ha, m_gb, p->d, p->V, int(p->N), dW, p->V,
                       info.sms, s, "dW GEMM launch");
  }
}

int check_workspace(void* workspace, size_t ws_bytes, size_t need) {
  if (need > 0 && (workspace == nullptr || ws_bytes < need))
    return fail(ALR_ERR_INVALID_ARG, "workspace of %zu bytes is smaller than the %zu needed",
                ws_bytes, need);
  if (need > 0 && !aligned16(workspace))
    return fail(ALR_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
  return ALR_OK;
}

// Arguments of the dH / dW products of the backward passes from kept logits.
int check_head_grad_args(const alr_params* p, const void* Hd, const void* W, const float* dHd,
                         const float* dW, void* workspace, size_t ws_bytes) {
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if (Hd == nullptr || W == nullptr || dHd == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "Hd, W and dHd must be non-NULL");
  if (!aligned16(Hd) || !aligned16(W) || !aligned16(dHd) || (dW != nullptr && !aligned16(dW)))
    return fail(ALR_ERR_INVALID_ARG, "Hd, W, dHd and dW must be 16-byte aligned");
  return check_workspace(workspace, ws_bytes, bwd_layout(p, false).total);
}

int check_topk_labels(const alr_params* p, const int32_t* idx, const float* prob,
                      const float* tail) {
  if (p->V < alr::kTopK)
    return fail(ALR_ERR_INVALID_ARG, "V = %d is below the %d label tokens", p->V, alr::kTopK);
  if (idx == nullptr || prob == nullptr || tail == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "top_idx, top_prob and tail must be non-NULL");
  return ALR_OK;
}

}  // namespace

extern "C" {

size_t alr_logit_grad_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  return p->dtype == ALR_F32 ? round_up(size_t(p->V) * p->d * 4, 1024) : 0;
}

int alr_logit_grad(const alr_params* p, const void* Hd, const void* Ht, const void* W,
                   const float* weight, const float* weight_sum, const float* lse_d,
                   const float* lse_t, void* G, void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  DevInfo info;
  int rc = check_bwd_args(p, Hd, Ht, W, weight, weight_sum, lse_d, lse_t, &info);
  if (rc != ALR_OK) return rc;
  if (G == nullptr || !aligned16(G)) return fail(ALR_ERR_INVALID_ARG, "G must be non-NULL and 16-byte aligned");
  const size_t need = alr_logit_grad_workspace_size(p);
  if (need > 0 && (workspace == nullptr || ws_bytes < need || !aligned16(workspace)))
    return fail(ALR_ERR_INVALID_ARG, "workspace of %zu bytes is smaller than the %zu needed",
                ws_bytes, need);
  return logit_grad_impl(p, Hd, Ht, W, weight, weight_sum, lse_d, lse_t, TopkLabels{}, G,
                         workspace, info, static_cast<cudaStream_t>(stream));
}

int alr_slot_loss_bwd(const alr_params* p, const void* Hd, const void* Ht, const void* W,
                      const float* weight, const float* weight_sum, const float* lse_d,
                      const float* lse_t, float* dHd, float* dW, void* workspace, size_t ws_bytes,
                      void* stream) {
  ALR_RANGE();
  DevInfo info;
  int rc = check_bwd_args(p, Hd, Ht, W, weight, weight_sum, lse_d, lse_t, &info);
  if (rc != ALR_OK) return rc;
  if (dHd == nullptr) return fail(ALR_ERR_INVALID_ARG, "dHd is NULL");
  if (!aligned16(dHd) || (dW != nullptr && !aligned16(dW)))
    return fail(ALR_ERR_INVALID_ARG, "dHd and dW must be 16-byte aligned");
  const size_t need = alr_bwd_workspace_size(p);
  if (workspace == nullptr || ws_bytes < need)
    return fail(ALR_ERR_INVALID_ARG, "workspace of %zu bytes is smaller than the %zu needed",
                ws_bytes, need);
  if (!aligned16(workspace)) return fail(ALR_ERR_INVALID_ARG, "workspace must be 16-byte aligned");

  const BwdLayout lay = bwd_layout(p);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  void* G = ws + lay.g_off;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  rc = logit_grad_impl(p, Hd, Ht, W, weight, weight_sum, lse_d, lse_t, TopkLabels{}, G,
                       ws + lay.wt_off, info, s);
  if (rc != ALR_OK) return rc;
  return head_grads_impl(p, Hd, W, G, dHd, dW, ws, lay, info, s);
}

int alr_logit_grad_from_logits(const alr_params* p, const void* Zd, const void* Zt,
                               const uint16_t* Zd_ref, const uint16_t* Zt_ref,
                               const float* weight, const float* weight_sum, const float* lse_d,
                               const float* lse_t, void* G, void* stream) {
  ALR_RANGE();
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if ((rc = check_kept(p, Zd, Zd_ref, "Zd")) != ALR_OK) return rc;
  if ((rc = check_kept(p, Zt, Zt_ref, "Zt")) != ALR_OK) return rc;
  if (G == nullptr || weight == nullptr || weight_sum == nullptr || lse_d == nullptr ||
      lse_t == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned16(G)) return fail(ALR_ERR_INVALID_ARG, "G must be 16-byte aligned");
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  cudaError_t e = alr::launch_logits_grad(p->dtype, Zd, Zt, Zd_ref, Zt_ref, lse_d, lse_t, weight,
                                          weight_sum, p->lambda, int(p->N), p->V, G, info.sms,
                                          static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "logit-gradient launch");
  return ALR_OK;
}

size_t alr_bwd_from_logits_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  return bwd_layout(p, false).total;
}

int alr_slot_loss_bwd_from_logits(const alr_params* p, const void* Hd, const void* W,
                                  const void* Zd, const void* Zt, const uint16_t* Zd_ref,
                                  const uint16_t* Zt_ref, const float* weight,
                                  const float* weight_sum, const float* lse_d, const float* lse_t,
                                  void* G, float* dHd, float* dW, void* workspace,
                                  size_t ws_bytes, void* stream) {
  ALR_RANGE();
  // everything is validated before the gradient kernel overwrites anything
  int rc = check_head_grad_args(p, Hd, W, dHd, dW, workspace, ws_bytes);
  if (rc != ALR_OK) return rc;
  if ((rc = alr_logit_grad_from_logits(p, Zd, Zt, Zd_ref, Zt_ref, weight, weight_sum, lse_d,
                                       lse_t, G, stream)) != ALR_OK)
    return rc;
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  return head_grads_impl(p, Hd, W, G, dHd, dW, static_cast<uint8_t*>(workspace),
                         bwd_layout(p, false), info, static_cast<cudaStream_t>(stream));
}

size_t alr_readout_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  DevInfo info;
  if (device_info(&info) != ALR_OK) return 0;
  return fwd_layout(p, info.sms, kPlanReadout).total;
}

int alr_label_readout(const alr_params* p, const void* Ht, const void* W,
                      const int32_t* corpus_tok, int32_t* top_idx, float* top_prob, float* tail,
                      float* lse_t, int32_t* argmax_t, float* gap_t, float* logp_x,
                      void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if (Ht == nullptr || W == nullptr || top_idx == nullptr || top_prob == nullptr || tail == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "Ht, W, top_idx, top_prob and tail must be non-NULL");
  if (p->V < alr::kTopK)
    return fail(ALR_ERR_INVALID_ARG, "V = %d is below the %d label tokens", p->V, alr::kTopK);
  if (!aligned16(Ht) || !aligned16(W))
    return fail(ALR_ERR_INVALID_ARG, "Ht and W must be 16-byte aligned");
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  const FwdLayout lay = fwd_layout(p, info.sms, kPlanReadout);
  if ((rc = check_workspace(workspace, ws_bytes, lay.total)) != ALR_OK) return rc;
  const int dt = p->dtype;
  const size_t es = elem_size(dt);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CUtensorMap m_h, m_w;
  if ((rc = make_map(&m_h, Ht, dt, p->d, p->N, p->d * es, k_per_row(dt), 128)) != ALR_OK) return rc;
  alr::LossArgs args{};
  args.plan = loss_plan(p, info.sms, false, kPlanReadout);
  if ((rc = head_map(&m_w, p, W, ws + lay.wt_off, args.plan.bn, s)) != ALR_OK) return rc;
  args.part = reinterpret_cast<float*>(ws + lay.part_off);
  args.corpus_tok = corpus_tok;
  args.status = alr::device_status_ptr();
  if (args.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
  cudaError_t e = alr::launch_loss_kernel(alr::kModeReadout, dt, m_h, m_h, m_w, m_w, m_w, args, s);
  if (e != cudaSuccess) return cuda_fail(e, "label readout kernel launch");
  e = alr::launch_readout_combine(args.plan, args.part, corpus_tok != nullptr, top_idx, top_prob,
                                  tail, lse_t, argmax_t, gap_t, logp_x, s);
  if (e != cudaSuccess) return cuda_fail(e, "readout combine launch");
  return ALR_OK;
}

size_t alr_topk_fwd_workspace_size(const alr_params* p) {
  if (check_params(p) != ALR_OK) return 0;
  DevInfo info;
  if (device_info(&info) != ALR_OK) return 0;
  return fwd_layout(p, info.sms, kPlanTopk).total;
}

}  // extern "C"

namespace {

// The top-k + tail forward; with Zd given the fused kernel also writes z_d (kModeTopkFwdKeep).
int topk_fwd_impl(const alr_params* p, const void* Hd, const void* W, const int32_t* top_idx,
                  const float* top_prob, const float* tail, const float* row_mask,
                  const float* weight_in, void* Zd, uint16_t* Zd_ref,
                  const alr_topk_fwd_outputs* out, void* workspace, size_t ws_bytes,
                  void* stream) {
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if ((rc = check_topk_labels(p, top_idx, top_prob, tail)) != ALR_OK) return rc;
  if (Hd == nullptr || W == nullptr || out == nullptr || out->loss_row == nullptr ||
      out->lse_d == nullptr || out->tail_q == nullptr || out->argmax_d == nullptr ||
      out->weight == nullptr || out->loss_total == nullptr || out->weight_sum == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "a required top-k forward pointer is NULL");
  if (!aligned16(Hd) || !aligned16(W))
    return fail(ALR_ERR_INVALID_ARG, "Hd and W must be 16-byte aligned");
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  const FwdLayout lay = fwd_layout(p, info.sms, kPlanTopk);
  if ((rc = check_workspace(workspace, ws_bytes, lay.total)) != ALR_OK) return rc;
  const int dt = p->dtype;
  const size_t es = elem_size(dt);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CUtensorMap m_h, m_w;
  if ((rc = make_map(&m_h, Hd, dt, p->d, p->N, p->d * es, k_per_row(dt), 128)) != ALR_OK) return rc;
  alr::LossArgs args{};
  args.plan = loss_plan(p, info.sms, false, kPlanTopk);
  if ((rc = head_map(&m_w, p, W, ws + lay.wt_off, args.plan.bn, s)) != ALR_OK) return rc;
  args.part = reinterpret_cast<float*>(ws + lay.part_off);
  args.ticket = reinterpret_cast<unsigned*>(ws + lay.ticket_off);
  args.top_idx = top_idx;
  args.zd_out = Zd;
  args.zd_ref = Zd_ref;
  args.status = alr::device_status_ptr();
  if (args.status == nullptr) return fail(ALR_ERR_CUDA, "status word lookup failed");
  CUtensorMap m_zd = m_w;
  if (Zd != nullptr && dt == ALR_BF16 &&
      (rc = make_map(&m_zd, Zd, kMapF16, p->V, p->N, uint64_t(p->V) * 2, 16, 32,
                     CU_TENSOR_MAP_SWIZZLE_NONE)) != ALR_OK)
    return rc;
  cudaError_t e = alr::launch_loss_kernel(Zd != nullptr ? alr::kModeTopkFwdKeep : alr::kModeTopkFwd,
                                          dt, m_h, m_h, m_w, m_zd, m_zd, args, s);
  if (e != cudaSuccess) return cuda_fail(e, "top-k forward kernel launch");
  double* anchor = reinterpret_cast<double*>(ws + lay.anchor_off);
  e = alr::launch_topk_combine(args.plan, args.part, top_prob, tail, row_mask, weight_in, p->gamma,
                               out->loss_row, out->lse_d, out->tail_q, out->argmax_d, out->gap_d,
                               out->weight, anchor, args.ticket, p->lambda, out->loss_total,
                               out->weight_sum, out->wl_sum, s);
  if (e != cudaSuccess) return cuda_fail(e, "top-k combine launch");
  return ALR_OK;
}

}  // namespace

extern "C" {

int alr_topk_loss_fwd(const alr_params* p, const void* Hd, const void* W, const int32_t* top_idx,
                      const float* top_prob, const float* tail, const float* row_mask,
                      const float* weight_in, const alr_topk_fwd_outputs* out, void* workspace,
                      size_t ws_bytes, void* stream) {
  ALR_RANGE();
  return topk_fwd_impl(p, Hd, W, top_idx, top_prob, tail, row_mask, weight_in, nullptr, nullptr,
                       out, workspace, ws_bytes, stream);
}

int alr_topk_loss_fwd_keep_logits(const alr_params* p, const void* Hd, const void* W,
                                  const int32_t* top_idx, const float* top_prob, const float* tail,
                                  const float* row_mask, const float* weight_in, void* Zd,
                                  uint16_t* Zd_ref, const alr_topk_fwd_outputs* out,
                                  void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if ((rc = check_kept(p, Zd, Zd_ref, "Zd")) != ALR_OK) return rc;
  return topk_fwd_impl(p, Hd, W, top_idx, top_prob, tail, row_mask, weight_in, Zd, Zd_ref, out,
                       workspace, ws_bytes, stream);
}

int alr_topk_logit_grad_from_logits(const alr_params* p, const void* Zd, const uint16_t* Zd_ref,
                                    const int32_t* top_idx, const float* top_prob,
                                    const float* tail, const float* weight,
                                    const float* weight_sum, const float* lse_d,
                                    const float* tail_q, void* G, void* stream) {
  ALR_RANGE();
  int rc = check_params(p);
  if (rc != ALR_OK) return rc;
  if ((rc = check_topk_labels(p, top_idx, top_prob, tail)) != ALR_OK) return rc;
  if ((rc = check_kept(p, Zd, Zd_ref, "Zd")) != ALR_OK) return rc;
  if (G == nullptr || weight == nullptr || weight_sum == nullptr || lse_d == nullptr ||
      tail_q == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned16(G)) return fail(ALR_ERR_INVALID_ARG, "G must be 16-byte aligned");
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  cudaError_t e = alr::launch_topk_logits_grad(p->dtype, Zd, Zd_ref, top_idx, top_prob, tail,
                                               tail_q, lse_d, weight, weight_sum, p->lambda,
                                               int(p->N), p->V, G, info.sms,
                                               static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "top-k logit-gradient launch");
  return ALR_OK;
}

int alr_topk_loss_bwd_from_logits(const alr_params* p, const void* Hd, const void* W,
                                  const void* Zd, const uint16_t* Zd_ref,
                                  const int32_t* top_idx, const float* top_prob,
                                  const float* tail, const float* weight, const float* weight_sum,
                                  const float* lse_d, const float* tail_q, void* G, float* dHd,
                                  float* dW, void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  // everything is validated before the gradient kernel overwrites anything
  int rc = check_head_grad_args(p, Hd, W, dHd, dW, workspace, ws_bytes);
  if (rc != ALR_OK) return rc;
  if ((rc = alr_topk_logit_grad_from_logits(p, Zd, Zd_ref, top_idx, top_prob, tail, weight,
                                            weight_sum, lse_d, tail_q, G, stream)) != ALR_OK)
    return rc;
  DevInfo info;
  if ((rc = require_sm103(&info)) != ALR_OK) return rc;
  return head_grads_impl(p, Hd, W, G, dHd, dW, static_cast<uint8_t*>(workspace),
                         bwd_layout(p, false), info, static_cast<cudaStream_t>(stream));
}

int alr_topk_logit_grad(const alr_params* p, const void* Hd, const void* W,
                        const int32_t* top_idx, const float* top_prob, const float* tail,
                        const float* weight, const float* weight_sum, const float* lse_d,
                        const float* tail_q, void* G, void* workspace, size_t ws_bytes,
                        void* stream) {
  ALR_RANGE();
  DevInfo info;
  int rc = check_bwd_args(p, Hd, Hd, W, weight, weight_sum, lse_d, lse_d, &info);
  if (rc != ALR_OK) return rc;
  if ((rc = check_topk_labels(p, top_idx, top_prob, tail)) != ALR_OK) return rc;
  if (tail_q == nullptr) return fail(ALR_ERR_INVALID_ARG, "tail_q is NULL");
  if (G == nullptr || !aligned16(G)) return fail(ALR_ERR_INVALID_ARG, "G must be non-NULL and 16-byte aligned");
  if ((rc = check_workspace(workspace, ws_bytes, alr_logit_grad_workspace_size(p))) != ALR_OK) return rc;
  TopkLabels lab;
  lab.idx = top_idx;
  lab.prob = top_prob;
  lab.tail = tail;
  lab.tail_q = tail_q;
  return logit_grad_impl(p, Hd, nullptr, W, weight, weight_sum, lse_d, nullptr, lab, G, workspace,
                         info, static_cast<cudaStream_t>(stream));
}

int alr_topk_loss_bwd(const alr_params* p, const void* Hd, const void* W, const int32_t* top_idx,
                      const float* top_prob, const float* tail, const float* weight,
                      const float* weight_sum, const float* lse_d, const float* tail_q,
                      float* dHd, float* dW, void* workspace, size_t ws_bytes, void* stream) {
  ALR_RANGE();
  DevInfo info;
  int rc = check_bwd_args(p, Hd, Hd, W, weight, weight_sum, lse_d, lse_d, &info);
  if (rc != ALR_OK) return rc;
  if ((rc = check_topk_labels(p, top_idx, top_prob, tail)) != ALR_OK) return rc;
  if (tail_q == nullptr || dHd == nullptr) return fail(ALR_ERR_INVALID_ARG, "tail_q and dHd must be non-NULL");
  if (!aligned16(dHd) || (dW != nullptr && !aligned16(dW)))
    return fail(ALR_ERR_INVALID_ARG, "dHd and dW must be 16-byte aligned");
  if ((rc = check_workspace(workspace, ws_bytes, alr_bwd_workspace_size(p))) != ALR_OK) return rc;
  const BwdLayout lay = bwd_layout(p);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  void* G = ws + lay.g_off;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  TopkLabels lab;
  lab.idx = top_idx;
  lab.prob = top_prob;
  lab.tail = tail;
  lab.tail_q = tail_q;
  rc = logit_grad_impl(p, Hd, nullptr, W, weight, weight_sum, lse_d, nullptr, lab, G,
                       ws + lay.wt_off, info, s);
  if (rc != ALR_OK) return rc;
  return head_grads_impl(p, Hd, W, G, dHd, dW, ws, lay, info, s);
}

int alr_loss_from_sums(const float* wl_sum, const float* weight_sum, float lambda,
                       float* loss_total, void* stream) {
  ALR_RANGE();
  if (wl_sum == nullptr || weight_sum == nullptr || loss_total == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "wl_sum, weight_sum and loss_total must be non-NULL");
  if (!(lambda == lambda)) return fail(ALR_ERR_INVALID_ARG, "lambda is NaN");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_loss_from_sums(wl_sum, weight_sum, lambda, loss_total,
                                             static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "loss-from-sums launch");
  return ALR_OK;
}

int alr_ira_blocks(int32_t S, int32_t K, int32_t max_blocks, const int32_t* valid_anchors,
                   const int32_t* rollout_len, const int32_t* offsets, const int32_t* rollout_tok,
                   const int32_t* corpus_anchor_tok, int32_t* seq, int32_t* pos,
                   int32_t* valid_len, int32_t* ctx_len, int32_t* anchor_tok, void* stream) {
  ALR_RANGE();
  if (S < 0 || K < 2 || max_blocks < 1)
    return fail(ALR_ERR_INVALID_ARG, "bad sizes S=%d K=%d max_blocks=%d", S, K, max_blocks);
  if (S == 0) return ALR_OK;
  if (valid_anchors == nullptr || rollout_len == nullptr || seq == nullptr || pos == nullptr ||
      valid_len == nullptr || (max_blocks > 1 && offsets == nullptr))
    return fail(ALR_ERR_INVALID_ARG,
                "valid_anchors, rollout_len, offsets, seq, pos and valid_len must be non-NULL");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_ira_blocks(S, K, max_blocks, valid_anchors, rollout_len, offsets,
                                         rollout_tok, corpus_anchor_tok, seq, pos, valid_len,
                                         ctx_len, anchor_tok, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "IRA block plan launch");
  return ALR_OK;
}

int alr_ira_draw(int32_t S, int32_t L, int32_t K, int32_t max_blocks, const uint8_t* anchor_ok,
                 const uint32_t* keys, const uint32_t* offset_u, int32_t* n_valid,
                 int32_t* anchor_pos, int32_t* offsets, void* stream) {
  ALR_RANGE();
  if (S < 0 || L < 1 || L > ALR_IRA_MAX_LEN || K < 3 || max_blocks < 1)
    return fail(ALR_ERR_INVALID_ARG, "bad sizes S=%d L=%d (at most %d) K=%d max_blocks=%d", S, L,
                ALR_IRA_MAX_LEN, K, max_blocks);
  if (S == 0) return ALR_OK;
  if (anchor_ok == nullptr || keys == nullptr || n_valid == nullptr || anchor_pos == nullptr ||
      (max_blocks > 1 && (offset_u == nullptr || offsets == nullptr)))
    return fail(ALR_ERR_INVALID_ARG,
                "anchor_ok, keys, offset_u, n_valid, anchor_pos and offsets must be non-NULL");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_ira_draw(S, L, K, max_blocks, anchor_ok, keys, offset_u, n_valid,
                                       anchor_pos, offsets, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "IRA draw launch");
  return ALR_OK;
}

int alr_ira_context(const void* store, int32_t C, int32_t F, int32_t dtype, int32_t S, int32_t K,
                    int32_t max_blocks, const int32_t* n_valid, const int32_t* rollout_len,
                    const int32_t* offsets, const int32_t* anchor_pos, void* ctx,
                    int32_t* ctx_len, int32_t* prefix_end, void* stream) {
  ALR_RANGE();
  if (dtype != ALR_BF16 && dtype != ALR_F32) return fail(ALR_ERR_UNSUPPORTED, "dtype %d", dtype);
  if (S < 0 || K < 3 || max_blocks < 2 || C < K - 2 || F < 1)
    return fail(ALR_ERR_INVALID_ARG,
                "bad sizes S=%d K=%d max_blocks=%d C=%d (at least K-2) F=%d", S, K, max_blocks, C,
                F);
  if ((size_t(F) * elem_size(dtype)) % 16 != 0)
    return fail(ALR_ERR_INVALID_ARG, "F * element size must be a multiple of 16 bytes");
  if (S == 0) return ALR_OK;
  if (store == nullptr || n_valid == nullptr || rollout_len == nullptr || offsets == nullptr ||
      anchor_pos == nullptr || ctx == nullptr)
    return fail(ALR_ERR_INVALID_ARG,
                "store, n_valid, rollout_len, offsets, anchor_pos and ctx must be non-NULL");
  if (!aligned16(store) || !aligned16(ctx))
    return fail(ALR_ERR_INVALID_ARG, "store and ctx must be 16-byte aligned");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_ira_context(store, C, F, int(elem_size(dtype)), S, K, max_blocks,
                                          n_valid, rollout_len, offsets, anchor_pos, ctx, ctx_len,
                                          prefix_end, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "IRA context launch");
  return ALR_OK;
}

int alr_accept_len(const int32_t* argmax_d, const int32_t* argmax_t, const float* active,
                   int32_t A, int32_t B, int32_t* acc_len, int64_t* hist, void* stream) {
  ALR_RANGE();
  if (A < 0 || B < 1 || B > 32) return fail(ALR_ERR_INVALID_ARG, "bad sizes A=%d B=%d", A, B);
  if (A > 0 && (argmax_d == nullptr || argmax_t == nullptr || acc_len == nullptr))
    return fail(ALR_ERR_INVALID_ARG, "argmax_d, argmax_t and acc_len must be non-NULL");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  if (A == 0) {   // no anchors: an all-zero histogram, no kernel to launch
    if (hist == nullptr) return ALR_OK;
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int64_t) * size_t(B + 1),
                                    static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "histogram clear");
    return ALR_OK;
  }
  cudaError_t e = alr::launch_accept_len(argmax_d, argmax_t, active, A, B, acc_len, hist,
                                         static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "accept_len launch");
  return ALR_OK;
}

int alr_erase_weights(const float* logp_x, const int32_t* corpus_tok, const int32_t* argmax_t,
                      const float* row_mask, int32_t A, int32_t B, float gamma, int32_t hard,
                      float* weight, void* stream) {
  ALR_RANGE();
  if (A < 0 || B < 1 || B > 32) return fail(ALR_ERR_INVALID_ARG, "bad sizes A=%d B=%d", A, B);
  if (!(gamma > 0.f)) return fail(ALR_ERR_INVALID_ARG, "gamma must be > 0");
  if (A == 0) return ALR_OK;
  if (weight == nullptr) return fail(ALR_ERR_INVALID_ARG, "weight must be non-NULL");
  if (hard ? (corpus_tok == nullptr || argmax_t == nullptr) : (logp_x == nullptr))
    return fail(ALR_ERR_INVALID_ARG, "the %s gate needs %s", hard ? "hard" : "soft",
                hard ? "corpus_tok and argmax_t" : "logp_x");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  cudaError_t e = alr::launch_erase_weights(logp_x, corpus_tok, argmax_t, row_mask, A, B, gamma,
                                            hard, weight, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "erase_weights launch");
  return ALR_OK;
}

int alr_gemm_form(int32_t dtype, int32_t M, int32_t Nc, int32_t K, int32_t* form, int32_t* split) {
  if (dtype != ALR_BF16 && dtype != ALR_F32) return fail(ALR_ERR_UNSUPPORTED, "dtype %d", dtype);
  if (M < 1 || Nc < 1 || K < 1)
    return fail(ALR_ERR_INVALID_ARG, "bad sizes M=%d Nc=%d K=%d", M, Nc, K);
  if (form == nullptr || split == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "form and split must be non-NULL");
  DevInfo info;
  const int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  const GemmChoice c = choose_gemm(dtype, M, Nc, K, info.sms);
  *form = int32_t(c.form);
  *split = c.split;
  return ALR_OK;
}

int alr_gemm(int32_t dtype, int32_t a_mn, int32_t b_mn, int32_t accumulate, const void* A,
             const void* B, float* C, int32_t M, int32_t Nc, int32_t K, void* stream) {
  ALR_RANGE();
  if (dtype != ALR_BF16 && dtype != ALR_F32) return fail(ALR_ERR_UNSUPPORTED, "dtype %d", dtype);
  if (M < 1 || Nc < 1 || K < 1) return fail(ALR_ERR_INVALID_ARG, "bad sizes M=%d Nc=%d K=%d", M, Nc, K);
  if (A == nullptr || B == nullptr || C == nullptr)
    return fail(ALR_ERR_INVALID_ARG, "A, B and C must be non-NULL");
  if (!aligned16(A) || !aligned16(B) || !aligned16(C))
    return fail(ALR_ERR_INVALID_ARG, "A, B and C must be 16-byte aligned");
  if (dtype == ALR_F32 && (a_mn || b_mn))
    return fail(ALR_ERR_UNSUPPORTED, "fp32 (tf32) operands must be K-major");
  const size_t es = elem_size(dtype);
  const int64_t a_inner = a_mn ? M : K, b_inner = b_mn ? Nc : K;
  if ((a_inner * es) % 16 != 0 || (b_inner * es) % 16 != 0 || Nc % 4 != 0)
    return fail(ALR_ERR_INVALID_ARG, "row strides must be multiples of 16 bytes and Nc %% 4 == 0");
  DevInfo info;
  int rc = require_sm103(&info);
  if (rc != ALR_OK) return rc;
  const uint32_t kke = k_per_row(dtype);
  const GemmChoice choice = choose_gemm(dtype, M, Nc, K, info.sms);
  CUtensorMap ma, mb;
  if (a_mn) rc = make_map(&ma, A, dtype, M, K, M * es, kke, kke);
  else rc = make_map(&ma, A, dtype, K, M, K * es, kke, 128);
  if (rc != ALR_OK) return rc;
  if (b_mn) rc = make_map(&mb, B, dtype, Nc, K, Nc * es, kke, kke);
  else rc = make_map(&mb, B, dtype, K, Nc, K * es, kke, gemm_b_rows(choice));
  if (rc != ALR_OK) return rc;
  return launch_gemm(choice, dtype, a_mn != 0, b_mn != 0, accumulate != 0, ma, mb, M, Nc, K, C, Nc,
                     info.sms, static_cast<cudaStream_t>(stream), "gemm launch");
}

}  // extern "C"
