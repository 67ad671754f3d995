// C-ABI of the Dion step library: context, argument checks, scratch layout and
// the launch sequence of one step.  All arithmetic runs in the kernels of this
// directory; the host code only validates and launches.
#include <math.h>
#include <stdlib.h>
#include <atomic>
#include <functional>
#include <mutex>
#include <new>
#include <string.h>
#include <vector>

#include "bf16_kernels.cuh"
#include "colnorm.cuh"
#include "dion_common.cuh"
#include "dion_internal.h"
#include "orth_kernels.cuh"
#include "simt_gemm.cuh"
#include "umma_api.cuh"

using namespace dion;

namespace {

constexpr int MAX_GRAPHS = 64;             // cached step graphs per context (least recently used goes first)
constexpr i64 GRAPH_MAX_ELEMS = (i64)2048 * 2048;   // graph replay for matrices up to this many elements (launch-bound steps)
constexpr int MAX_FLAG_SLOTS = 4096;      // step slots of OS_SLOT_INTS ints each; the last MAX_GRAPHS belong to the cached graphs
constexpr int MAX_CHAIN = 64;              // matrices of one shape stepped together by dion_step_grouped
constexpr size_t GROUP_SCRATCH_BYTES = (size_t)16 << 30;  // scratch dion_step_grouped may use for that (or cfg.workspace_bytes)
constexpr int MAX_ROUNDS = 6;             // adaptive Cholesky QR rounds
constexpr float FLOOR_REL = 1e-4f;        // pivot floor relative to the column's squared norm
constexpr float GOOD_REL = 1e-4f;         // smallest relative pivot of a round that one more round can finish
// CholeskyQR2: the second round is skipped when the first round's U1 is orthonormal enough, measured as an
// estimate of |U1^T U1 - I|_F^2 (k_probe_*): done when it is <= ORTH_TAU_F^2 * r, i.e. when the deviation's
// Frobenius norm is what r entries of size ORTH_TAU_F would give.  Measured on the workloads' own panels
// (cond(P) 2-4, r 128-2048, up to 14336 rows): sqrt(estimate / r) is 5e-7 to 9e-6 after one accurate round, and the
// step's outputs then differ from the float64 rule by 3-4e-6 (Q), the same as after two rounds; warm starts
// with nearly parallel columns give 3.6e-5 and more and take the second round.
constexpr float ORTH_TAU_F = 3e-5f;
constexpr float DONE_REL = 0.9f;          // smallest relative pivot of a round whose input was already orthonormal
constexpr i64 PART_CAP_FLOATS = (i64)16 << 20;  // split-K partial sums, at most 64 MiB
constexpr double P_HALF_MIN_MNR = 4e9;          // smallest m n r whose full-rank P runs on scaled half pairs
constexpr double SOLVE_PAIR_MIN_PANEL = 3e7;    // smallest rows x r whose blocked solves run on scaled half pairs
constexpr i64 LAZY_PAIR_MIN_MNR = 50000000;     // smallest m n r whose Lazy-Dion step runs on scaled half pairs (2^25.6: 512 x 768 x 128)
constexpr double GRAM_PAIR_MIN_FLOPS = 2e9;     // smallest rows r^2 whose Gram matrix runs on scaled half pairs
constexpr i64 WIDE_P_WHOLE_K = 1024;            // K up to which the P of a wide range (wide_p) is not split: a tile's K loop is short, and the
                                                // reduction would be one more launch that nearly always finds itself skipped (2 us)
constexpr double P_PAIR_MIN_MNR = 1.5e10;       // smallest m n r whose P = (M + G) Q runs on bf16 operand pairs first

constexpr i64 NBO_COLS = 512;  // = NBO, the outer block of the two-level Cholesky (defined below)

// One launch of k_chol_flow factors Gram matrices up to this order; beyond it blocks of 512 columns, whose products are on the
// tensor cores.  Orthonormalization of rows x r in us, one launch against blocks, and U's distance from float64: 8192 x 2048 686, 958
// (2.93, 2.72e-6); 12288 x 3072 1672, 2100 (2.93, 2.66e-6); 16384 x 3584 2380, 2838 (2.80, 2.57e-6); 16384 x 4096 2842, 3211 (2.95,
// 2.65e-6).  The launch is faster beyond the line too; the line stays for U's distance, which the blocks have 8 to 10 % smaller.
constexpr i64 FLOW_MAX_R = 3072;
// Largest rows r whose panel that launch solves too, against the product with the inverse behind it; in us, the launch's own
// solve first, and U's distance from float64: 2048 x 128 71.7, 81.3 (3.3, 2.5e-7); 1024 x 256 90, 114 (3.9, 5.8e-7); 1536 x 384 113, 139
// (3.7, 8.2e-7); 4096 x 256 98, 117 (3.3, 3.6e-7); beyond the line 8192 x 256 106, 128 (6.1, 4.2e-7); 4096 x 512 147, 170 (9.5, 8.4e-7);
// 4096 x 1024 244, 272 (3.20, 2.97e-6).  The launch is faster on both sides; the line lies where the smaller distance goes from the
// launch (but for 2048 x 128) to the product.  (The helpers of a chain also have as many panels to solve as it has matrices.)
constexpr double FLOW_SOLVE_MAX = 1.1e6;
constexpr i64 FLOW_SOLVE_MAX_TILES = 40000;     // ... in an adaptive round: most 64^3 products of its substitution
constexpr float NEAR_MAX_DEF = 3e-3f;           // largest |P^T P - I|_F whose factor is taken as a series (k_near_identity): third-order error 3e-8
constexpr i64 NEAR_MAX_BLOCKS = 512;
// Partial sums of the Gram product that it adds up itself, of the tensor engine's; twice as many of the FMA engine's.  One CTA reads
// those of the first three tiles; from there on a launch over all SMs reduces them first (4096 x 256, 32 splits: orthonormalization
// 120.8 -> 101.5 us; 1024 x 128, 8 splits of the tensor engine: 79 in the launch, 72 reduced; 640 x 112, 6 of the FMA engine: 65.7 in
// the launch, 66.7 reduced; 1500 x 100, 9 of it: 80 and 77).  Of a Gram matrix of one tile up to sixteen: nothing else waits for that
// CTA's loads (2048 x 16, 11 splits: 55.9 in the launch, 59.0 reduced; 3136 x 48, 14: 68.5 and 70.0; 9888 x 22, 24: 96.0 and 92.4).
constexpr int FLOW_MAX_SPLITS = 4;
constexpr int FLOW_MAX_SPLITS_ONE = 16;
constexpr int FLOW_AHEAD_MAX = 16;              // steps by which its preparations are handed out early
constexpr i64 FLOW_MAX_PANEL_TILES = 800;       // ... and most 64-row blocks of it (the control block holds 64 such matrices)

inline i64 align64(i64 floats) { return (floats + 63) / 64 * 64; }  // 256-byte granules

struct Layout {
  i64 P0, P1, R, Gram, Linv, Tbuf, Dinv, DinvP, part, cn_part, d, gdiag, scal, total;
  i64 Sk, SkV, SkW;         // randomized Cholesky QR: the two stacked panels [S P; P] and a solve temporary
  i64 B16, Q16, U16, R16;   // bf16-operand mode: bf16(M + G) and the bf16 copies of Q, U, R (offsets in floats)
  i64 B32;                  // fp32 mode: M + G formed once per step (0: the products form it on the fly)
  i64 Psave;                // CholeskyQR2: the panel as the product wrote it, kept for the fallback (0: none)
  i64 fb_part, fb_h, fb_n;  // fallback kernel: partial dot products (SMs x r), their sums (r), partial norms (SMs)
  i64 probe_y, probe_part, probe_sums;  // CholeskyQR2's orthogonality probe: U1 z (rows x NPROBE), partial U1^T (U1 z), partial estimates
  i64 probe_cap;            // chunks that probe_part holds
  i64 Bp;                   // fp32 mode, M + G in scratch: the same sum as a bf16 (hi, lo) pair (m x n x 2 bf16) for R; 0: none
  i64 Bh;                   // full rank: M + G as a scaled pair of half arrays for P (m x n x 2 halves), 0: none
  i64 pmax;                 // ... its partial maxima and the product's scale factor (like gmax)
  i64 SolveP, LfP, smax;    // blocked solves on half pairs (r > 512): pair of a rows x 512 right-hand side; pairs of a row block of
                            // the factor (512 x r) and of a diagonal inverse (512 x 512); partial maxima and scales
  i64 lz;                   // steps on half pairs: the scales of their products (HS_*), then the block maxima of R
  i64 XP;                   // scaled half pair of the inverse of the factor
  i64 xmax;                 // largest magnitude of the factor's inverse, then the scale of the product with its pair
  i64 gmax;                 // Gram matrices on half pairs: AMAX_PARTS partial maxima of |P|, then 1 / scale^2
  i64 Qc;                   // fp32 mode, large matrices: dense fp32 copy of Q for the chain-wide recomputation of P (0: none)
  i64 S16;                  // fp32 mode: the bf16 (hi, lo) pair of the error feedback's second factor (max(m,n) x r x 2 bf16)
  i64 part_floats;
  int cn_chunks;
  i64 cn_rows;
};

}  // namespace

struct dion_ctx {
  dion_config cfg;
  int sm_count;
  float* ws;
  size_t ws_bytes;
  int* dev_ints;  // [0] status, [1] skipped, [2..] per-step flags
  int flag_cursor;
  int* flow_ctl = nullptr;   // progress counters of k_chol_flow (zero between launches)
  i64 flow_ctl_cap = 0;
  int64_t launches;
  // per-phase profiling (off by default)
  bool prof_on;
  std::vector<cudaEvent_t> prof_pool;   // reusable events
  size_t prof_used;
  struct ProfRec { int phase; cudaEvent_t e0, e1; int64_t launches; };
  std::vector<ProfRec> prof_recs;
  // second stream for work that can run beside the serial Cholesky chain, and its fork/join events
  bool form_sum = true;   // fp32 mode may keep M + G in scratch (off for the fixed-scratch entry point)
  cudaStream_t side = nullptr;
  cudaEvent_t side_ev[32] = {};
  int side_cursor = 0;
  // Graph replay of launch-bound steps: the launch chain of dion_step on a small matrix is captured once per
  // (descriptor) into a CUDA graph and replayed; the learning rate reaches it through a device scalar.
  struct GraphEntry {
    dion_matrix key;
    cudaGraphExec_t exec;
    int64_t launches;
    int index;            // its state slot and scalar
    uint64_t last_use;
    float scale;          // the scalar's value on the device (NaN: not known)
    bool recorded;        // a write of the scalar may be in a capture of the caller's: it changes behind the library's back
  };
  std::vector<GraphEntry> graphs;
  bool graphs_on = false;
  int flow_lose_cta = 0, flow_lose = 0;      // test hook: see FlowArgs
  bool chain_batch = true;          // tensor-engine products of a grouped chain in one launch over its matrices
  cudaStream_t cap = nullptr;       // the stream the chains are captured on (never the caller's: it may be the legacy stream)
  float* graph_scalars = nullptr;   // MAX_GRAPHS device floats
  uint64_t graph_clock = 0;
};

namespace {

void colnorm_plan(i64 rows, i64 r, int sm, int* chunks, i64* rows_per) {
  const i64 col_blocks = (r + 127) / 128;
  i64 want = (4 * (i64)sm + col_blocks - 1) / col_blocks;
  if (want < 1) want = 1;
  i64 per = (rows + want - 1) / want;
  if (per < 32) per = 32;
  *rows_per = per;
  *chunks = (int)((rows + per - 1) / per);
}

// Row chunks of the probe's second pass: 32 rows (enough blocks to hide a block's few dependent loads; 4096 x 1024: 31 ->
// 12 us against the 55 rows that one wave of blocks would take), more on tall panels (512 chunks of partial sums).
void probe_plan(i64 rows, int* chunks, i64* rows_per) {
  i64 per = (rows + 511) / 512;
  per = (per + 31) / 32 * 32;
  *rows_per = per;
  *chunks = (int)((rows + per - 1) / per);
}
i64 probe_sums(i64 r) { return (r * NPROBE + PD_ENTRIES - 1) / PD_ENTRIES; }

// Both plans are made for the long side when the scratch is laid out and for the panel's or the right factor's rows when they
// are used, and neither grows with the rows: 16384 rows are 512 chunks of the probe, 16448 are 257.  The chunks are made
// larger until they fit what was laid out.
void fit_chunks(i64 rows, i64 cap, i64 step, int* chunks, i64* rows_per) {
  while (*chunks > cap) {
    *rows_per += step;
    *chunks = (int)((rows + *rows_per - 1) / *rows_per);
  }
}

// fp32 mode on the tensor engine: M + G is formed once per step in scratch, as fp32 (4 bytes per element) and as a
// bf16 (hi, lo) pair (4 bytes), and P, R and the error feedback read those.  Forming it inside the two products
// costs their converter warps a second tile and keeps them on three TF32 MMAs per K step; with the pair in
// memory the products take three bf16 MMAs (half the tensor time) and read 4 bytes per element instead of 8, so the
// extra pass pays down to rank fraction 1/64 (measured: 32768^2 at r = 512 22.0 -> 15.9 ms, 16384^2 at r = 256
// 3.4 -> 3.0 ms); below that the step is HBM bound either way and the on-the-fly form moves fewer bytes.
bool sum_in_scratch(const dion_ctx* c, i64 m, i64 n, i64 r) {
  const i64 sd = (m < n) ? m : n;
  return c->form_sum && c->cfg.precision == DION_PREC_FP32 && c->cfg.engine != DION_ENGINE_SIMT &&
         m % 4 == 0 && n % 4 == 0 && m >= 128 && n >= 128 && r >= 64 && 64 * r >= sd;
}

// Above rank fraction 1/4 (the adaptive rounds: ill-conditioned panels) P = (M + G) Q needs its 22 significant
// bits.  On large matrices it takes them from scaled pairs of IEEE half arrays (three kind::f16 MMAs per K step,
// split accumulators) instead of the 3xTF32 split with four kind::tf32 ones: M + G is scaled by a power of two
// found on the device, Q (unit-norm columns) by 2^13.
int resolve_orth(const dion_ctx* c, i64 r, i64 short_dim);
bool p_on_half_pairs(const dion_ctx* c, i64 m, i64 n, i64 r) {
  return c->cfg.precision == DION_PREC_FP32 && c->cfg.engine != DION_ENGINE_SIMT && m % 8 == 0 && n % 8 == 0 && r % 8 == 0 &&
         (double)m * (double)n * (double)r >= P_HALF_MIN_MNR && resolve_orth(c, r, (m < n) ? m : n) == DION_ORTH_SHIFTED3;
}

// A step whose orthonormalization may resolve to CholeskyQR2 keeps the panel for the device-side fallback.
bool may_fallback(const dion_ctx* c, i64 m, i64 n, i64 r) {
  const i64 sd = (m < n) ? m : n;
  const int o = c->cfg.orth;
  return o == DION_ORTH_CHOLQR2 || ((o == DION_ORTH_AUTO || o == DION_ORTH_RCQR) && 4 * r <= sd);
}

Layout make_layout(const dion_ctx* c, i64 m, i64 n, i64 r) {
  Layout L;
  const i64 big = (m > n) ? m : n;
  i64 o = 0;
  L.P0 = o; o += align64(big * r);
  L.P1 = o; o += align64(big * r);
  L.R = o; o += align64(big * r);
  L.Gram = o; o += align64(r * r);
  L.Linv = o; o += align64(r * r);
  L.Tbuf = o; o += align64(r * r);
  const bool gpairs = (double)big * (double)r * (double)r >= GRAM_PAIR_MIN_FLOPS;      // Gram matrices may be formed on half pairs
  L.XP = o; o += gpairs && r <= FLOW_MAX_R ? align64(r * r) : 0;
  L.Dinv = o; o += align64(((r + NB - 1) / NB) * (i64)NB * NB);
  L.DinvP = o; o += align64(((r + NB - 1) / NB) * (i64)NB * NB);
  // split-K partials: the largest plain-store product of a step is max(m,n) x r
  i64 pf = 4 * (i64)c->sm_count * 64 * 64;
  // ... and enough for as many splits as give every SM work: 148 tiles of 64 x 64 held two splits of a 4096 x 256 product, which
  // left more than half of the chip idle (from 4096^2: 50 us with two, 37 with four).  (By the shape's usual tiles; where a launch's
  // own would want more, it takes as many as fit.)  The fixed scratch keeps its size: what fits it is what fitted before.
  if (c->form_sum) {
    const i64 need[4] = {umma_split_floats(m, r, n, false, c->sm_count), umma_split_floats(n, r, m, false, c->sm_count),
                         umma_split_floats(r, r, big, true, c->sm_count), pf};
    for (i64 f : need) if (f > pf) pf = f;
  }
  if (pf > PART_CAP_FLOATS) pf = PART_CAP_FLOATS;
  L.part_floats = pf;
  L.part = o; o += align64(pf);
  colnorm_plan(big, r, c->sm_count, &L.cn_chunks, &L.cn_rows);
  L.cn_chunks += 1;
  L.cn_part = o; o += align64((i64)L.cn_chunks * r + (gpairs ? NEAR_MAX_BLOCKS : 0));
  L.d = o; o += align64(r);
  L.gdiag = o; o += align64(r);
  L.scal = o; o += 64;
  L.Sk = L.SkV = 0;
  L.SkW = 0;
  if (c->cfg.orth == DION_ORTH_RCQR) {
    // two (sketch rows + panel rows) x r buffers for the rounds on the stacked panel [S P; P], and the
    // 512-column temporary of their blocked solves
    L.Sk = o; o += align64((2 * r + big) * r);
    L.SkV = o; o += align64((2 * r + big) * r);
    L.SkW = o; o += align64((2 * r + big) * NBO_COLS);
  }
  L.B16 = L.Q16 = L.U16 = L.R16 = 0;
  if (c->cfg.precision == DION_PREC_BF16_OPERANDS) {
    L.B16 = o; o += align64((m * n + 1) / 2);
    L.Q16 = o; o += align64((big * r + 1) / 2);
    L.U16 = o; o += align64((big * r + 1) / 2);
    L.R16 = o; o += align64((big * r + 1) / 2);
  }
  L.B32 = L.Bp = 0;
  if (sum_in_scratch(c, m, n, r)) {
    L.B32 = o; o += align64(m * n);
    if (m % 8 == 0 && n % 8 == 0 && r % 8 == 0) { L.Bp = o; o += align64(m * n); }
  }
  L.Psave = L.fb_part = L.fb_h = L.fb_n = 0;
  L.gmax = o; o += align64(AMAX_PARTS + 64);
  L.xmax = o; o += 64;
  L.lz = o;
  if (sum_in_scratch(c, m, n, r)) o += align64(8 * (i64)c->sm_count + 64);
  L.SolveP = L.LfP = L.smax = 0;
  if (r > FLOW_MAX_R && (double)big * (double)r >= SOLVE_PAIR_MIN_PANEL) {
    L.SolveP = o; o += align64(big * NBO_COLS);
    L.LfP = o; o += align64(NBO_COLS * r + NBO_COLS * NBO_COLS);
    L.smax = o; o += align64(3 * (AMAX_PARTS + 64));
  }
  L.Bh = L.pmax = 0;
  if (L.Bp > 0 && p_on_half_pairs(c, m, n, r)) {
    L.Bh = o; o += align64(m * n);
    L.pmax = o; o += align64(AMAX_PARTS + 64);
  }
  L.Qc = 0;
  if (L.Bp > 0 && (double)m * (double)n * (double)r >= P_PAIR_MIN_MNR) { L.Qc = o; o += align64(big * r); }
  L.S16 = o; o += align64(big * r);
  L.probe_y = o; o += align64(big * NPROBE);
  {
    int chunks; i64 per;
    probe_plan(big, &chunks, &per);
    L.probe_cap = chunks + 1;
    L.probe_part = o; o += align64(L.probe_cap * r * NPROBE);
    L.probe_sums = o; o += align64(probe_sums(r));
  }
  if (may_fallback(c, m, n, r)) {
    L.Psave = o; o += align64(big * r);
    L.fb_part = o; o += align64((i64)c->sm_count * r);
    L.fb_h = o; o += align64(r);
    L.fb_n = o; o += align64(c->sm_count);
  }
  L.total = o;
  return L;
}

// The plans as a step with the layout L uses them.
void probe_chunks(const Layout& L, i64 rows, int* chunks, i64* rows_per) {
  probe_plan(rows, chunks, rows_per);
  fit_chunks(rows, L.probe_cap, 32, chunks, rows_per);
}
void colnorm_chunks(const dion_ctx* c, const Layout& L, i64 rows, i64 r, int* chunks, i64* rows_per) {
  colnorm_plan(rows, r, c->sm_count, chunks, rows_per);
  fit_chunks(rows, L.cn_chunks, 1, chunks, rows_per);
}

void graphs_clear(dion_ctx* c);

int ensure_ws(dion_ctx* c, size_t bytes) {
  if (bytes <= c->ws_bytes) return DION_OK;
  if (c->ws != nullptr) {
    if (cudaDeviceSynchronize() != cudaSuccess) return DION_ERR_CUDA;
    graphs_clear(c);      // they point into the old scratch
    cudaFree(c->ws);
    c->ws = nullptr;
    c->ws_bytes = 0;
  }
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) { cudaGetLastError(); return DION_ERR_NOMEM; }
  c->ws = (float*)p;
  c->ws_bytes = bytes;
  return DION_OK;
}

#define DION_CHECK_LAUNCH(ctx)                                   \
  do {                                                           \
    (ctx)->launches++;                                           \
    if (cudaGetLastError() != cudaSuccess) return DION_ERR_CUDA; \
  } while (0)
#define DION_TRY(expr)              \
  do {                              \
    const int rc_ = (expr);         \
    if (rc_ != DION_OK) return rc_; \
  } while (0)

GemmArgs gemm_args() {
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.alpha = 1.f;
  g.batch = 1;
  g.batch2 = 1;
  g.splits = 1;
  return g;
}

// Launch with programmatic stream serialization (see pdl_enter in the kernels).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Products on the fp32 FMA engine.
// Splits of K: a K step of 16 takes about as long as the latency of its loads whatever runs beside it, so a product of few tiles is
// cut to two or three steps per block, up to two blocks per SM (1001 x 83 x 333 with the reduction: 28.6 -> 14 us).
// Fewer where the next kernel adds the partial sums up itself (k_chol_flow: one CTA reads those of the first three tiles, which
// costs it as much per split as a K step here: with the square of the splits kept to K / 16, orthonormalizing 1001 x 83 takes 87
// us and 1030 x 190 127, with every split 99 and 148).
constexpr i64 SPLIT_MIN_K = 32;
constexpr i64 SPLIT_MAX = 64;
constexpr i64 SIMT_THIN_N = 32;          // outputs of at most this many columns take 128 x 32 tiles
constexpr i64 SIMT_WIDE_MIN_K = 96;      // updates of C below it are bound by C: 64 x 64 tiles

// tabs != nullptr: the same product on nb matrices (operands from the tables, partial sums part_stride floats apart; outputs too
// where the reduction follows).  Tiles and splits are those of one matrix: the same bits.
int launch_gemm_simt(dion_ctx* c, GemmArgs g, cudaStream_t st, float* part, i64 part_floats,
                     bool force64, const GemmTabs* tabs = nullptr, int nb = 1, i64 part_stride = 0) {
  if (g.M <= 0 || g.N <= 0) return DION_OK;
  const i64 t128 = ((g.M + 127) / 128) * ((g.N + 127) / 128) * g.batch * (g.batch2 > 1 ? g.batch2 : 1);
  const bool thin = !force64 && g.N <= SIMT_THIN_N && g.tri == TRI_FULL && !g.klimit;
  const bool use128 = !force64 && !thin && t128 >= c->sm_count && (g.epi == EPI_STORE || g.K >= SIMT_WIDE_MIN_K);
  const i64 bm = (use128 || thin) ? 128 : 64, bn = use128 ? 128 : thin ? 32 : 64;
  const i64 gm = (g.M + bm - 1) / bm, gn = (g.N + bn - 1) / bn;
  int splits = 1;
  if (!use128 && !force64 && g.epi == EPI_STORE && g.batch == 1 && g.batch2 <= 1 && part != nullptr && g.alpha_dev == nullptr) {
    const i64 tiles = gm * gn;
    i64 want = (2 * (i64)c->sm_count + tiles - 1) / tiles;
    const i64 kmax = g.K / SPLIT_MIN_K;
    if (want > kmax) want = kmax;
    if (want > SPLIT_MAX) want = SPLIT_MAX;
    if (g.splits_out != nullptr) while (want > 1 && want * want * 16 > g.K) --want;
    while (want > 1 && want * g.M * g.N > part_floats) --want;
    if (want > 1) {
      const i64 per = ((g.K + want - 1) / want + 15) / 16 * 16;      // as the kernel cuts K; no empty split
      splits = (int)((g.K + per - 1) / per);
    }
  }
  // (a chain whose tiles fill the chip adds the splits up in the blocks instead of through memory)
  int inner = 1;
  if (tabs != nullptr && splits > 1 && g.splits_out == nullptr && gm * gn * nb >= 2 * c->sm_count) { inner = splits; splits = 1; }
  g.splits = splits;
  g.part = part;
  if (gm > 65535) return DION_ERR_UNSUPPORTED;
  if (g.batch2 < 1) g.batch2 = 1;
  if (splits > 1 && g.batch2 > 1) return DION_ERR_INVALID;
  const dim3 grid((unsigned)gn, (unsigned)gm, (unsigned)(tabs != nullptr ? splits * nb : splits > 1 ? splits : g.batch * g.batch2));
  if (tabs != nullptr) {
    g.bs2 = part_stride;
    if (use128) launch_pdl(k_gemm_simt<128, 128, 8, 8, 8, 1, GemmTabs>, grid, dim3(256), 0, st, g, *tabs, inner);
    else if (thin) launch_pdl(k_gemm_simt<128, 32, 16, 4, 4, 2, GemmTabs>, grid, dim3(256), 0, st, g, *tabs, inner);
    else launch_pdl(k_gemm_simt<64, 64, 16, 4, 4, 2, GemmTabs>, grid, dim3(256), 0, st, g, *tabs, inner);
  } else {
    if (use128) launch_pdl(k_gemm_simt<128, 128, 8, 8, 8, 1, NoTabs>, grid, dim3(256), 0, st, g, NoTabs(), 1);
    else if (thin) launch_pdl(k_gemm_simt<128, 32, 16, 4, 4, 2, NoTabs>, grid, dim3(256), 0, st, g, NoTabs(), 1);
    else launch_pdl(k_gemm_simt<64, 64, 16, 4, 4, 2, NoTabs>, grid, dim3(256), 0, st, g, NoTabs(), 1);
  }
  DION_CHECK_LAUNCH(c);
  if (g.splits_out != nullptr) {      // (the caller sums that many partial products itself)
    if (splits <= *g.splits_out) { *g.splits_out = splits; return DION_OK; }
    *g.splits_out = 1;
  }
  if (splits > 1) {
    const i64 total = g.N % 4 == 0 ? (g.M * g.N + 3) / 4 : g.M * g.N;      // (four elements per thread where rows allow it)
    int blocks = (int)((total + 255) / 256);
    if (blocks > 8 * c->sm_count) blocks = 8 * c->sm_count;
    launch_pdl(k_splitk_reduce, dim3((unsigned)blocks, (unsigned)nb), dim3(256), 0, st, part, splits, g.M, g.N, g.C, g.ldc, g.alpha, g.tri, (int)bm, g.skip_flag,
               part_stride, nb > 1 ? g.skip_stride : (i64)0, (const float*)nullptr, (i64)0);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// Two updates of C of one shape (no split, no batch) in one launch: each as launch_gemm_simt computes it.
int launch_gemm_simt_two(dion_ctx* c, const GemmArgs& a, const GemmArgs& b, cudaStream_t st) {
  const i64 t128 = ((a.M + 127) / 128) * ((a.N + 127) / 128);
  const bool thin = a.N <= SIMT_THIN_N, use128 = !thin && t128 >= c->sm_count && a.K >= SIMT_WIDE_MIN_K;
  const i64 bm = (use128 || thin) ? 128 : 64, bn = use128 ? 128 : thin ? 32 : 64;
  const i64 gm = (a.M + bm - 1) / bm, gn = (a.N + bn - 1) / bn;
  if (gm > 65535) return DION_ERR_UNSUPPORTED;
  const dim3 grid((unsigned)gn, (unsigned)gm, 2);
  const GemmSecond second = {b};
  if (use128) launch_pdl(k_gemm_simt<128, 128, 8, 8, 8, 1, GemmSecond>, grid, dim3(256), 0, st, a, second, 1);
  else if (thin) launch_pdl(k_gemm_simt<128, 32, 16, 4, 4, 2, GemmSecond>, grid, dim3(256), 0, st, a, second, 1);
  else launch_pdl(k_gemm_simt<64, 64, 16, 4, 4, 2, GemmSecond>, grid, dim3(256), 0, st, a, second, 1);
  DION_CHECK_LAUNCH(c);
  return DION_OK;
}

cudaEvent_t prof_event(dion_ctx* c) {
  if (c->prof_used == c->prof_pool.size()) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    c->prof_pool.push_back(e);
  }
  return c->prof_pool[c->prof_used++];
}

// Brackets one phase of a step with events on the step's stream when profiling is on.
struct PhaseScope {
  dion_ctx* c; cudaStream_t st; int phase; cudaEvent_t e0; int64_t l0;
  PhaseScope(dion_ctx* c_, cudaStream_t st_, int phase_) : c(c_), st(st_), phase(phase_), e0(nullptr), l0(c_->launches) {
    if (c->prof_on && phase >= 0) { e0 = prof_event(c); if (e0) cudaEventRecord(e0, st); }
  }
  ~PhaseScope() {
    if (c->prof_on && e0) {
      cudaEvent_t e1 = prof_event(c);
      if (e1) { cudaEventRecord(e1, st); c->prof_recs.push_back({phase, e0, e1, c->launches - l0}); }
    }
  }
};

// One launch chain works on `nb` matrices of identical (m, n, r) at a time (nb = 1 for
// dion_step): the large products are launched per matrix, the small kernels of the
// factorization once for all of them (one block or batch entry per matrix).  Matrix b
// uses the scratch slice that starts b * wstride floats after `ws` and the state slot
// b * OS_SLOT_INTS ints after `os`.
struct StepCtx {
  dion_ctx* c;
  cudaStream_t st;
  float* ws;
  Layout L;
  int nb;
  i64 wstride;
  int* os;    // first device state slot (OS_* ints)
  int* flag;  // = os + OS_FAIL: the step must not write its outputs
  bool tensor;  // tensor-core engine allowed for this matrix
  bool in_orth; // inside the orthonormalization (for the profiling phases)
  const dion_matrix* const* list = nullptr;   // the matrices of the chain (sketch pointers of the RCQR mode)
  i64 wt_off = -1;        // >= 0: scratch offset of the blocked solves' rows x 512 temporary (default: the R panel)
  bool no_split = false;  // launches on the side stream: the split-K scratch belongs to the main stream
  bool quiet_fail = false;  // a failed pivot only sets the step's fail flag: the fallback kernel follows
  const std::function<int()>* redo_p = nullptr;   // the panel came from the fast product: recomputes it accurately
                                                  // (skipped on the device for matrices whose OS_DONE is set)
  float* W(int b, i64 off) const { return ws + (i64)b * wstride + off; }
  int* OS(int b) const { return os + (i64)b * OS_SLOT_INTS; }
};

// Engine dispatch: tensor cores when the product qualifies, else fp32 FMA.
// `b`: the matrix of the batch the product belongs to (selects its split-K scratch).
int launch_gemm(StepCtx& s, const GemmArgs& g, int b = 0, bool force64 = false) {
  if (s.tensor && !force64) {
    PhaseScope ps(s.c, s.st, s.in_orth ? DION_PHASE_ORTH_GEMM : -1);
    // bf16 operands are for the four large contractions only: the Gram matrices, factors and
    // solves of the orthonormalization keep fp32 accuracy in every mode
    const int prec = s.in_orth ? DION_PREC_FP32 : s.c->cfg.precision;
    const int rc = umma_try_launch(g, prec, s.c->sm_count, s.no_split ? nullptr : s.W(b, s.L.part), s.L.part_floats,
                                   s.c->dev_ints, s.st);
    if (rc > 0) { s.c->launches += rc; return DION_OK; }
    if (rc < 0) return rc;
    if (s.c->cfg.engine == DION_ENGINE_TENSOR) return DION_ERR_UNSUPPORTED;
  }
  if (g.ab16) return DION_ERR_UNSUPPORTED;   // bf16 arrays are read by the tensor engine only
  return launch_gemm_simt(s.c, g, s.st, s.no_split ? nullptr : s.W(b, s.L.part), s.L.part_floats, force64);
}

// Shifts the workspace-resident operands of a product to matrix b of the batch.
GemmArgs for_matrix(const StepCtx& s, GemmArgs g, int b, bool a_ws, bool b_ws, bool c_ws) {
  const i64 o = (i64)b * s.wstride;
  if (a_ws) g.A += o;
  if (b_ws) g.B += o;
  if (c_ws) g.C += o;
  if (a_ws && g.A16lo != nullptr) g.A16lo = (const char*)g.A16lo + 4 * o;
  if (b_ws && g.B16lo != nullptr) g.B16lo = (const char*)g.B16lo + 4 * o;
  if (g.alpha_dev != nullptr) g.alpha_dev += (i64)b * g.alpha_dev_stride;
  if (g.skip_flag != nullptr) g.skip_flag += (i64)b * OS_SLOT_INTS;
  if (g.wide_flag != nullptr) g.wide_flag += (i64)b * OS_SLOT_INTS;
  return g;
}

void over_batch(const StepCtx& s, GemmArgs& g);

// One product per matrix of the chain, operands and output in the scratch slices (c2_ws: the second epilogue
// operand too).  The tensor engine takes all matrices in one launch when the product qualifies (its work list
// then runs over (matrix, tile) pairs, which also fills the tail of one matrix's tiles with the next one's);
// otherwise one launch per matrix.
int launch_gemm_chain(StepCtx& s, const GemmArgs& g, bool c2_ws = false) {
  if (s.nb > 1 && s.tensor && s.c->chain_batch) {
    GemmArgs gb = g;
    over_batch(s, gb);
    gb.c2_batched = c2_ws ? 1 : 0;
    PhaseScope ps(s.c, s.st, s.in_orth ? DION_PHASE_ORTH_GEMM : -1);
    const int prec = s.in_orth ? DION_PREC_FP32 : s.c->cfg.precision;
    const int rc = umma_try_launch(gb, prec, s.c->sm_count, s.no_split ? nullptr : s.W(0, s.L.part), s.L.part_floats,
                                   s.c->dev_ints, s.st);
    if (rc > 0) { s.c->launches += rc; return DION_OK; }
    if (rc < 0) return rc;
  }
  if (s.nb > 1 && s.nb <= GEMM_TAB_MAX && s.c->chain_batch && g.batch == 1 && g.batch2 <= 1 && g.alpha_dev == nullptr &&
      s.c->cfg.engine != DION_ENGINE_TENSOR && !(s.tensor && umma_shape_ok(g, s.in_orth ? DION_PREC_FP32 : s.c->cfg.precision)) && !g.ab16) {
    GemmTabs t;      // (shapes that only the FMA engine takes: one launch of it)
    for (int m = 0; m < s.nb; ++m) {
      const i64 o = (i64)m * s.wstride;
      t.A[m] = g.A + o; t.B[m] = g.B + o; t.C[m] = g.C + o; t.A2[m] = g.A2;
      t.C2[m] = g.C2 != nullptr && c2_ws ? (const void*)((const float*)g.C2 + o) : g.C2;
    }
    GemmArgs gb = g;
    gb.skip_stride = OS_SLOT_INTS;
    PhaseScope ps(s.c, s.st, s.in_orth ? DION_PHASE_ORTH_GEMM : -1);
    return launch_gemm_simt(s.c, gb, s.st, s.no_split ? nullptr : s.W(0, s.L.part), s.L.part_floats, false, &t, s.nb, s.wstride);
  }
  for (int m = 0; m < s.nb; ++m) {
    GemmArgs gm = for_matrix(s, g, m, true, true, true);
    if (c2_ws) gm.C2 = (const float*)gm.C2 + (i64)m * s.wstride;
    DION_TRY(launch_gemm(s, gm, m));
  }
  return DION_OK;
}

// The same product on every matrix of the chain, given as one GemmArgs per matrix (as the per-matrix launch would
// take them).  When the tensor engine can run them as ONE launch -- identical shapes and strides, operands in the
// scratch slices (so that one 3-D tensor map covers them), outputs anywhere (a pointer table) -- it does: the work
// list then runs over (matrix, tile) pairs and the last wave of one matrix is filled with the next one's tiles.
// Every element is computed by the same sequence of operations either way.
int launch_gemm_group(StepCtx& s, const std::vector<GemmArgs>& v) {
  const int nb = (int)v.size();
  bool one = nb > 1 && nb <= GEMM_TAB_MAX && s.tensor && s.c->chain_batch;
  const GemmArgs& a = v[0];
  bool c_strided = true, c2_strided = true;
  bool alike = nb > 1 && nb <= GEMM_TAB_MAX && s.c->chain_batch;      // the same product on every matrix, wherever its operands lie
  const i64 wb = s.wstride * 4;   // bytes between scratch slices
  auto at_stride = [&](const void* p0, const void* pb, int b) {
    return (p0 == nullptr && pb == nullptr) ||
           (p0 != nullptr && pb != nullptr && (const char*)pb - (const char*)p0 == (ptrdiff_t)((i64)b * wb));
  };
  for (int b = 1; b < nb && alike; ++b) {
    const GemmArgs& g = v[b];
    alike = alike && g.M == a.M && g.N == a.N && g.K == a.K && g.a_si == a.a_si && g.a_sk == a.a_sk && g.a2_si == a.a2_si &&
            g.a2_sk == a.a2_sk && g.a2_mode == a.a2_mode && g.b_sk == a.b_sk && g.b_sn == a.b_sn && g.ldc == a.ldc &&
            g.epi == a.epi && g.ldc2 == a.ldc2 && g.c2_mode == a.c2_mode && g.alpha == a.alpha &&
            (g.alpha_dev == a.alpha_dev || at_stride(a.alpha_dev, g.alpha_dev, b)) &&
            g.batch == 1 && a.batch == 1 && g.tri == a.tri && g.klimit == a.klimit && g.precise == a.precise &&
            g.ab16 == a.ab16 && g.f16 == a.f16 && g.tf32x1 == a.tf32x1 &&
            ((a.skip_flag == nullptr && g.skip_flag == nullptr) ||
             (a.skip_flag != nullptr && g.skip_flag == a.skip_flag + (i64)b * OS_SLOT_INTS)) &&
            ((a.wide_flag == nullptr && g.wide_flag == nullptr) ||
             (a.wide_flag != nullptr && g.wide_flag == a.wide_flag + (i64)b * OS_SLOT_INTS));
    one = one && alike && at_stride(a.A, g.A, b) && at_stride(a.B, g.B, b) && at_stride(a.A2, g.A2, b) && at_stride(a.A16lo, g.A16lo, b) &&
          at_stride(a.B16lo, g.B16lo, b);
    c_strided = c_strided && at_stride(a.C, g.C, b);
    c2_strided = c2_strided && at_stride(a.C2, g.C2, b);
  }
  if (one && !c_strided && a.epi == EPI_STORE) one = false;   // (a plain store may split K: its reduction wants one stride)
  if (one) {
    GemmArgs gb = a;
    over_batch(s, gb);
    if (nb > 1 && v[1].alpha_dev != a.alpha_dev) gb.alpha_dev_stride = s.wstride;     // a scale per matrix, in its scratch slice
    float* ctab[GEMM_TAB_MAX];
    const void* c2tab[GEMM_TAB_MAX];
    for (int b = 0; b < nb; ++b) { ctab[b] = v[b].C; c2tab[b] = v[b].C2; }
    if (!c_strided) gb.c_tab = ctab;
    if (a.C2 != nullptr) {
      if (c2_strided && a.c2_mode == ADD_F32) gb.c2_batched = 1;
      else gb.c2_tab = c2tab;
    }
    PhaseScope ps(s.c, s.st, s.in_orth ? DION_PHASE_ORTH_GEMM : -1);
    const int prec = s.in_orth ? DION_PREC_FP32 : s.c->cfg.precision;
    const int rc = umma_try_launch(gb, prec, s.c->sm_count, s.no_split ? nullptr : s.W(0, s.L.part), s.L.part_floats,
                                   s.c->dev_ints, s.st);
    if (rc > 0) { s.c->launches += rc; return DION_OK; }
    if (rc < 0) return rc;
  }
  // (not for the tensor engine:) one launch of the FMA engine, with the operands' addresses in tables
  if (alike && !a.ab16 && s.c->cfg.engine != DION_ENGINE_TENSOR && !(s.tensor && umma_shape_ok(a, s.in_orth ? DION_PREC_FP32 : s.c->cfg.precision)) && (c_strided || a.epi != EPI_STORE)) {
    GemmTabs t;
    for (int b = 0; b < nb; ++b) { t.A[b] = v[b].A; t.A2[b] = v[b].A2; t.B[b] = v[b].B; t.C[b] = v[b].C; t.C2[b] = v[b].C2; }
    GemmArgs g = a;
    g.skip_stride = OS_SLOT_INTS;
    if (v[1].alpha_dev != a.alpha_dev) g.alpha_dev_stride = s.wstride;
    PhaseScope ps(s.c, s.st, s.in_orth ? DION_PHASE_ORTH_GEMM : -1);
    return launch_gemm_simt(s.c, g, s.st, s.no_split ? nullptr : s.W(0, s.L.part), s.L.part_floats, false, &t, nb, s.wstride);
  }
  for (int b = 0; b < nb; ++b) DION_TRY(launch_gemm(s, v[b], b));
  return DION_OK;
}

// One-time opt-in to the dynamic shared memory of the kernels that need more than 48 KB.
int configure_kernels() {
  if (umma_configure() != DION_OK) return DION_ERR_CUDA;
  if (cudaFuncSetAttribute(k_probe_y4, cudaFuncAttributeMaxDynamicSharedMemorySize, PY_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(k_probe_fused<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PF_SMEM_MAX) != cudaSuccess ||
      cudaFuncSetAttribute(k_probe_fused<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PF_SMEM_MAX) != cudaSuccess ||
      cudaFuncSetAttribute(k_chol_flow<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FLOW_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(k_chol_flow<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FLOW_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(k_tiny_cholqr2, cudaFuncAttributeMaxDynamicSharedMemorySize, tiny_cholqr2_smem(TINY_MAX_ROWS)) != cudaSuccess) {
    cudaGetLastError();
    return DION_ERR_CUDA;
  }
  return DION_OK;
}

constexpr i64 NBO = NBO_COLS;  // outer block of the two-level Cholesky

// Blocks of 256 threads for `total` items on each of nb matrices: at most one wave (eight per SM) over all of them.
int grid_for(const dion_ctx* c, i64 total, int nb = 1) {
  i64 blocks = (total + 255) / 256;
  const i64 most = (8 * (i64)c->sm_count + nb - 1) / nb;
  if (blocks > most) blocks = most;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

// Marks a small (FMA-engine) product as batched over the nb matrices of the chain.
void over_batch(const StepCtx& s, GemmArgs& g) {
  g.batch2 = s.nb;
  g.bs2 = s.wstride;
  g.skip_stride = OS_SLOT_INTS;
}

// How a Cholesky-QR round runs.
enum : int {
  RM_PLAIN = 0,     // no device-side control
  RM_ADAPTIVE = 1,  // deflating pivots, skipped once the panel is done, split-accumulator products, round statistics
  RM_FIRST = 2,     // first round of CholeskyQR2: plain control, split-accumulator products
  RM_CHECKED = 3,   // second round of CholeskyQR2: the first round's result is measured first (orthogonality probe);
                    // if it is orthonormal to ORTH_TAU_F the whole round is skipped (Pout = Pin)
  RM_REDO = 4       // first round once more, on the panel recomputed with the accurate product: skipped on the device
                    // when the round on the fast panel already passed the probe; split-accumulator products
};
inline bool rm_skips(int mode) { return mode == RM_ADAPTIVE || mode == RM_CHECKED || mode == RM_REDO; }
inline bool rm_precise(int mode) { return mode == RM_ADAPTIVE || mode == RM_FIRST || mode == RM_REDO; }

// ints of the control block per matrix: progress of the rows of L and of the preparations, of D, of the panel's rows
int flow_ctl_ints(i64 sz, i64 rows) {
  const i64 T = (sz + CB - 1) / CB, NR = (rows + CB - 1) / CB;
  return (int)((2 * T + 2 + (NR > T ? NR : T) + 31) / 32 * 32);
}
// Panels that the factorization's launch solves too, beside the factorization.  The rule looks at the shape alone (grouped
// calls compute what single ones do).  CholeskyQR2: small panels; larger ones take one product behind it, before the
// helpers' products outlast the chain of diagonal blocks (more so with several matrices).  Adaptive rounds: up to the
// number of tile products that the blocked solve's tensor-core products take as long for.
bool flow_solves(const StepCtx& s, i64 rows, i64 r, bool adaptive) {
  (void)s;
  const i64 T = (r + CB - 1) / CB, NR = (rows + CB - 1) / CB;
  if (r > FLOW_MAX_R || NR > FLOW_MAX_PANEL_TILES) return false;
  return adaptive ? NR * T * (T + 1) / 2 <= FLOW_SOLVE_MAX_TILES : (double)rows * (double)r <= FLOW_SOLVE_MAX;
}

// One launch of the factorization (k_chol_flow) on the diagonal square [o, o + sz) of the Gram matrices, with either
// the solve of the panel at pin_off into pout_off (rows > 0; the whole Gram matrix, o = 0 and sz = r) or the inverse of its
// factor (transposed: L^-T, upper triangular) into L.Linv.  nsplit > 1: the Gram matrix is still the
// product's partial sums (alpha_dev: their scale).  near: see k_near_identity.
int chol_flow(StepCtx& s, i64 r, i64 o, i64 sz, int mode, i64 pin_off, i64 pout_off, i64 rows, int nsplit, const float* alpha_dev,
              bool round_end, bool near = false) {
  dion_ctx* c = s.c;
  const bool adaptive = (mode == RM_ADAPTIVE);
  FlowArgs f;
  memset(&f, 0, sizeof(f));
  f.A = s.ws + s.L.Gram;
  f.L = s.ws + s.L.Tbuf;
  if (nsplit > 1) { f.part = s.ws + s.L.part; f.nsplit = nsplit; f.alpha_dev = alpha_dev; f.alpha_stride = s.wstride; }
  f.Dinv = s.ws + s.L.Dinv;
  f.DinvP = adaptive ? s.ws + s.L.DinvP : f.Dinv;
  f.gdiag = s.ws + s.L.gdiag;
  f.gdiag_given = (sz < r) ? 1 : 0;
  const bool solve = rows > 0;
  f.Pin = solve ? s.ws + pin_off : nullptr;
  f.Pout = s.ws + (solve ? pout_off : s.L.Linv);
  f.rows = rows;
  f.r = r; f.o = o; f.sz = sz;
  f.floor_rel = adaptive ? FLOOR_REL : 0.f;
  f.os = s.os; f.skips = rm_skips(mode) ? 1 : 0;
  f.status = s.quiet_fail ? nullptr : c->dev_ints;
  f.status_always = c->dev_ints;
  const i64 T = (sz + CB - 1) / CB, NR = (rows + CB - 1) / CB;
  f.ctl = c->flow_ctl;
  f.ctl_stride = flow_ctl_ints(sz, rows);
  f.wstride = s.wstride; f.nb = s.nb;
  f.xmax = solve ? nullptr : s.ws + s.L.xmax;
  f.near = near ? 1 : 0;
  f.round_end = (round_end && adaptive) ? 1 : 0;
  f.good_rel = GOOD_REL; f.done_rel = DONE_REL; f.rounds_total = c->dev_ints + 2;
  f.limit = umma::SPIN_LIMIT_CYCLES;
  f.lose_cta = c->flow_lose_cta; f.lose = c->flow_lose;
  if (FLOW_HEAD_INTS + (i64)s.nb * f.ctl_stride > c->flow_ctl_cap) return DION_ERR_UNSUPPORTED;
  // one runner per matrix; as many helpers as can be resident beside them, at most one per task
  auto blocks = [](i64 n, i64 of) { return (n + of - 1) / of; };
  i64 tasks = (T > 2) ? 2 * (T - 2) : 0, panel[2] = {0, 0};      // (panel[i]: with i + 1 tiles of rows to a task)
  for (i64 k = 0; k + 3 < T; ++k) tasks += blocks(T - 3 - k, FLOW_ROWS);
  for (i64 k = 0; k < T; ++k)
    for (int i = 0; i < 2; ++i) panel[i] += blocks(solve ? NR : flow_inverse_rows((int)T, (int)k, sz < r), i + 1);
  const i64 cap = c->sm_count;      // (one CTA per SM: shared memory)
  // Tasks of two tiles read the tiles of L they meet half as often; where every task has an SM to itself the shorter ones are done
  // sooner (orthonormalization of 768 x 192 82.4 -> 80.7 us, 1024 x 128 71.7 -> 70.5).
  f.prows = (tasks + panel[0]) * s.nb + s.nb <= cap ? 1 : 2;
  tasks += panel[f.prows - 1];
  i64 grid = s.nb + tasks * s.nb;
  if (grid > cap) grid = cap;
  if (grid < s.nb + 1) return DION_ERR_UNSUPPORTED;
  const i64 ahead = (grid - s.nb) / (4 * s.nb) - 1;      // (2 nb (ahead + 1) preparations at most wait for tasks handed out later)
  f.ahead = (int)(ahead < 0 ? 0 : ahead > FLOW_AHEAD_MAX ? FLOW_AHEAD_MAX : ahead);
  void* args[] = {&f};
  const void* fn = (r % 4 == 0) ? (const void*)k_chol_flow<true> : (const void*)k_chol_flow<false>;
  if (cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(FLOW_THREADS), args, FLOW_SMEM, s.st) != cudaSuccess) {
    cudaGetLastError();
    return DION_ERR_CUDA;
  }
  c->launches++;
  return DION_OK;
}

// Cholesky of an r x r Gram matrix (lower) that is too large for one data-flow launch, with the inverses of its diagonal
// squares (L.Linv): outer blocks of 512 columns.  The diagonal square is factored and inverted by k_chol_flow, the panel
// below it is multiplied by that inverse and the trailing matrix is updated with one rank-512 product (tensor cores
// where it qualifies).
int potrf_blocked(StepCtx& s, i64 r, int mode, const std::function<int(i64, i64)>* after_block) {
  dion_ctx* c = s.c;
  float* Gm = s.ws + s.L.Gram;
  float* Linv = s.ws + s.L.Linv;
  float* Tbuf = s.ws + s.L.Tbuf;
  const int* skip = rm_skips(mode) ? (s.os + OS_DONE) : nullptr;
  const int precise = rm_precise(mode) ? 1 : 0;
  for (i64 J0 = 0; J0 < r; J0 += NBO) {
    const i64 sz = (r - J0 < NBO) ? (r - J0) : NBO;
    DION_TRY(chol_flow(s, r, J0, sz, mode, 0, 0, 0, 1, nullptr, false));
    if (after_block != nullptr) DION_TRY((*after_block)(J0, sz));   // block column J of the factor and its inverse are final
    const i64 rem = r - J0 - sz;
    if (rem > 0) {
      float* panel = Gm + (J0 + sz) * r + J0;
      float* ptmp = Tbuf + (J0 + sz) * r + J0;
      GemmArgs g = gemm_args();  // Lpanel = panel * Linv_JJ^T (out of place, then copied back)
      g.M = rem; g.N = sz; g.K = sz;
      g.A = panel; g.a_si = r; g.a_sk = 1;
      g.B = Linv + J0 * r + J0; g.b_sk = r; g.b_sn = 1; g.klimit = 1;
      g.C = ptmp; g.ldc = r; g.epi = EPI_STORE; g.skip_flag = skip; g.precise = precise;
      DION_TRY(launch_gemm_chain(s, g));
      // With the solves on the second stream, the copy of Lpanel into the Gram buffer goes there too: its
      // only readers are the solves of later block columns (queued behind it on that stream); the trailing
      // update reads the temporary, so the copy leaves the serial chain.
      const bool side_copy = after_block != nullptr && c->side != nullptr;
      {
        cudaStream_t cst = s.st;
        if (side_copy) {
          cudaEvent_t e = c->side_ev[c->side_cursor];
          c->side_cursor = (c->side_cursor + 1) % 32;
          if (cudaEventRecord(e, s.st) != cudaSuccess || cudaStreamWaitEvent(c->side, e, 0) != cudaSuccess) return DION_ERR_CUDA;
          cst = c->side;
        }
        dim3 grid((unsigned)grid_for(c, rem * sz, s.nb), (unsigned)s.nb);
        launch_pdl(k_copy_block, grid, dim3(256), 0, cst, ptmp, r, panel, r, rem, sz, skip, s.wstride, (const int*)nullptr, (int*)nullptr, (int*)nullptr);
        DION_CHECK_LAUNCH(c);
      }
      const float* lp = side_copy ? ptmp : panel;
      GemmArgs t = gemm_args();  // A22 -= Lpanel * Lpanel^T (lower tiles)
      t.M = rem; t.N = rem; t.K = sz;
      t.A = lp; t.a_si = r; t.a_sk = 1;
      t.B = lp; t.b_sk = 1; t.b_sn = r;
      t.C = Gm + (J0 + sz) * r + (J0 + sz); t.ldc = r; t.epi = EPI_SUB; t.tri = TRI_LOWER; t.skip_flag = skip;
      t.precise = precise;
      DION_TRY(launch_gemm_chain(s, t));
    }
  }
  return DION_OK;
}

// The orthogonality probe on the rows x r panels at `off` (two passes over the panel instead of its Gram matrix).
// phase: PROBE_CHECK the check of CholeskyQR2's first round; PROBE_FAST the same after a round on a panel from the
// fast product (decides whether the panel is recomputed; counts nothing); PROBE_AFTER_REDO the check that follows a
// possible recomputation (a panel that passed PROBE_FAST is not measured again).
int probe(StepCtx& s, i64 off, i64 rows, i64 r, int phase) {
  dion_ctx* c = s.c;
  int chunks; i64 per;
  probe_chunks(s.L, rows, &chunks, &per);
  const int* keep = (phase == PROBE_AFTER_REDO) ? (const int*)(s.os + OS_DONE) : nullptr;
  const float* U = s.ws + off;
  if (r <= PF_MAX_R) {
    int ct_log = 3;                         // threads by columns: 8 .. 256
    while (4 << ct_log < r) ++ct_log;
    const size_t smem = (size_t)(((r + 127) / 128 * 128) * NPROBE + PF_RED + 32 * NPROBE) * sizeof(float);
    auto go = [&](auto kernel) {
      launch_pdl(kernel, dim3((unsigned)chunks, (unsigned)s.nb), dim3(256), smem, s.st, U, r, rows, r, per, s.ws + s.L.probe_part, s.wstride, keep, ct_log);
    };
    if (r % 4 == 0) go(k_probe_fused<true>); else go(k_probe_fused<false>);
  } else {
    if (r % 4 == 0) {
      i64 blocks = (rows + 31) / 32;          // a block of 8 warps takes 32 rows at a time
      if (blocks > 2 * (i64)c->sm_count) blocks = 2 * (i64)c->sm_count;
      launch_pdl(k_probe_y4, dim3((unsigned)blocks, (unsigned)s.nb), dim3(256), (size_t)PY_SMEM, s.st, U, r, rows, r, s.ws + s.L.probe_y, s.wstride, keep);
      DION_CHECK_LAUNCH(c);
      launch_pdl(k_probe_w4, dim3((unsigned)((r / 4 + 127) / 128), (unsigned)chunks, (unsigned)s.nb), dim3(128), 0, s.st, U, r, rows, r, per,
                 (const float*)(s.ws + s.L.probe_y), s.ws + s.L.probe_part, s.wstride, keep);
    } else {
      launch_pdl(k_probe_y, dim3((unsigned)grid_for(c, rows * 32, s.nb), (unsigned)s.nb), dim3(256), 0, s.st, U, r, rows, r, s.ws + s.L.probe_y, s.wstride, keep);
      DION_CHECK_LAUNCH(c);
      launch_pdl(k_probe_w, dim3((unsigned)((r + 127) / 128), (unsigned)chunks, (unsigned)s.nb), dim3(128), 0, s.st, U, r, rows, r, per,
                 (const float*)(s.ws + s.L.probe_y), s.ws + s.L.probe_part, s.wstride, keep);
    }
  }
  DION_CHECK_LAUNCH(c);
  launch_pdl(k_probe_decide, dim3((unsigned)probe_sums(r), (unsigned)s.nb), dim3(PD_ENTRIES * PD_GROUPS), 0, s.st, (const float*)(s.ws + s.L.probe_part), chunks,
             r, s.os, ORTH_TAU_F, c->dev_ints + 2, s.ws + s.L.probe_sums, s.wstride, phase);
  DION_CHECK_LAUNCH(c);
  return DION_OK;
}

// Tall panels whose blocked triangular solves run on scaled half pairs.
// (where the solves are what the round waits for: CholeskyQR2 on large panels.  In the adaptive rounds they run
// beside the serial chain, and on the panels of the 8B list the extra passes for scales and pairs cost what the
// cheaper products save: measured, 42.1 -> 44.1 ms there, 48.1 -> 42.8 ms on the large squares.)
bool solve_on_pairs(const StepCtx& s, i64 rows, i64 r, int mode) {
  return s.tensor && s.nb <= GEMM_TAB_MAX && mode != RM_ADAPTIVE && rows % 8 == 0 && r % 8 == 0 &&
         (double)rows * (double)r >= SOLVE_PAIR_MIN_PANEL;
}

// Tall panels whose Gram matrix runs on scaled half pairs (the rule looks at the shape alone).
bool gram_on_pairs(const StepCtx& s, i64 rows, i64 r) {
  return s.tensor && rows % 8 == 0 && r % 8 == 0 && r >= 128 &&
         (double)rows * (double)r * (double)r >= GRAM_PAIR_MIN_FLOPS;      // (in either precision mode)
}

// One Cholesky-QR round on every matrix of the chain: Pout = Pin * chol(Pin^T Pin)^-T.
// rows x r panels, ld = r; pin_off / pout_off are offsets in the scratch slice.
// adaptive: columns with negligible pivots are deflated, the round is skipped
// once the panel is orthonormal, and the round statistics are evaluated at the end.
int cholqr_round(StepCtx& s, i64 pin_off, i64 pout_off, i64 rows, i64 r, int mode, i64 gram_rows = 0,
                 int probe_phase = PROBE_CHECK, int round = 0) {      // round: of the adaptive rounds
  // A skipped round leaves Pout untouched (the caller keeps using Pin).
  // gram_rows > 0: the Gram matrix is formed from the first gram_rows rows only (a sketch stacked on
  // top of the panel); the factor is applied to all rows
  dion_ctx* c = s.c;
  const bool adaptive = (mode == RM_ADAPTIVE);
  const bool skips = rm_skips(mode);
  const int* skip = skips ? (s.os + OS_DONE) : nullptr;
  if (mode == RM_CHECKED) {
    // CholeskyQR2, second round: first measure the first round's result; orthonormal enough -> done, and
    // everything below is skipped on the device
    DION_TRY(probe(s, pin_off, rows, r, probe_phase));
  }
  GemmArgs g = gemm_args();
  g.M = r; g.N = r; g.K = gram_rows > 0 ? gram_rows : rows;
  g.A = s.ws + pin_off; g.a_si = 1; g.a_sk = r;
  g.B = s.ws + pin_off; g.b_sk = r; g.b_sn = 1;
  const bool gpairs = gram_rows == 0 && gram_on_pairs(s, rows, r);
  if (gpairs) {
    // The Gram matrix of a tall panel on half pairs: the panel is scaled and split into S16 (free during the
    // orthonormalization) and the product takes three kind::f16 MMAs per K step instead of the three or four
    // kind::tf32 ones; the same 22 significant bits.  1 / scale^2 reaches the epilogue through a device scalar.
    const int* sk = skips ? skip : nullptr;
    __half* hi = reinterpret_cast<__half*>(s.ws + s.L.S16);
    __half* lo = hi + rows * r;
    i64 parts = (rows * r / 4 + 2047) / 2048;
    if (parts > AMAX_PARTS) parts = AMAX_PARTS;
    float* range = s.ws + s.L.part;      // (read before the product writes its partial sums there)
    ChainPtrs t;
    for (int b = 0; b < s.nb; ++b) t.p[b] = s.W(b, pin_off);
    launch_pdl(k_range_partial, dim3((unsigned)parts, (unsigned)s.nb), dim3(256), 0, s.st, t, r, rows, rows, r, range, s.wstride, sk, (i64)OS_SLOT_INTS, (int*)nullptr);
    DION_CHECK_LAUNCH(c);
    launch_pdl(k_split_f16_scaled, dim3((unsigned)grid_for(c, rows * r / 8, s.nb), (unsigned)s.nb), dim3(256), 0, s.st,
               (const float*)(s.ws + pin_off), r, rows, r, (const float*)range, (int)parts, hi, lo, s.ws + s.L.gmax + AMAX_PARTS,
               s.wstride, sk, (i64)OS_SLOT_INTS, -1.f, (const float*)nullptr, (float*)nullptr, s.os, -1, (int)OS_PANEL_WIDE, -1);
    DION_CHECK_LAUNCH(c);
    g.ab16 = 1; g.f16 = 1;
    g.A = reinterpret_cast<const float*>(hi); g.A16lo = lo;
    g.B = reinterpret_cast<const float*>(hi); g.B16lo = lo;
    g.alpha_dev = s.ws + s.L.gmax + AMAX_PARTS; g.alpha_dev_stride = s.wstride;
  }
  g.C = s.ws + s.L.Gram; g.ldc = r; g.epi = EPI_STORE; g.tri = TRI_LOWER; g.skip_flag = skips ? skip : nullptr; g.precise = rm_precise(mode) ? 1 : 0;
  const bool in_flow = flow_solves(s, rows, r, adaptive);      // factorization and solve in one launch
  const bool flow_all = in_flow || (!adaptive && r <= FLOW_MAX_R);      // at least the whole factorization
  const bool on_tensor = g.ab16 || (s.tensor && umma_shape_ok(g, s.in_orth ? DION_PREC_FP32 : c->cfg.precision));
  int nsplit = !flow_all ? 1 : r <= CB ? FLOW_MAX_SPLITS_ONE : on_tensor ? FLOW_MAX_SPLITS : 2 * FLOW_MAX_SPLITS;
  if (flow_all) g.splits_out = &nsplit;       // (which also adds up a few partial products)
  DION_TRY(launch_gemm_chain(s, g));
  const float* part_scale = g.alpha_dev;
  if (flow_all) {
    // The panel's pair that the Gram matrix was formed from times the scaled half pair of L^-T, one product behind the
    // factorization (22 significant bits in three kind::f16 MMAs; without a pair 3xTF32): CholeskyQR2 on large panels.
    // The adaptive rounds solve by substitution instead: an explicit inverse costs a factor cond(L) of backward
    // stability, and their panels are ill conditioned (2048^2 full rank, cond 1e7: Q off by 2.2e-2 against 3.5e-3).  Their
    // finishing round has a factor near the identity, and where that is a short series (k_near_identity) the product
    // replaces the factorization.
    const NearSrc raw = {s.ws + s.L.Gram, s.ws + s.L.part, nsplit, part_scale};
    i64 tiles = (r + 31) / 32 * ((r + 31) / 32) / 4;
    if (tiles < 1) tiles = 1;
    if (tiles > NEAR_MAX_BLOCKS) tiles = NEAR_MAX_BLOCKS;
    const bool series = adaptive && gpairs && round > 0;      // (the first round is never the finishing one)
    if (series) {
      __half* eh = reinterpret_cast<__half*>(s.ws + s.L.Linv);
      __half* fh = eh + r * r;
      launch_pdl(k_near_identity, dim3((unsigned)tiles, (unsigned)s.nb), dim3(256), 0, s.st, raw, r, eh, fh, s.ws + s.L.xmax, s.ws + s.L.cn_part,
                 s.os, NEAR_MAX_DEF, s.wstride);
      DION_CHECK_LAUNCH(c);
      GemmArgs q = gemm_args();      // S = Phi E, lower triangle
      q.M = r; q.N = r; q.K = r;
      q.ab16 = 1; q.f16 = 1;
      q.A = (const float*)fh; q.a_si = r; q.a_sk = 1;
      q.B = (const float*)eh; q.b_sk = 1; q.b_sn = r;
      q.C = s.ws + s.L.Tbuf; q.ldc = r; q.epi = EPI_STORE; q.tri = TRI_LOWER; q.alpha = 1.f / (NEAR_SCALE * NEAR_SCALE);
      q.skip_flag = s.os + OS_NOTNEAR;
      s.no_split = true;      // (the split-K scratch holds the Gram matrix)
      const int rc = launch_gemm_chain(s, q);
      s.no_split = false;
      DION_TRY(rc);
    }
    DION_TRY(chol_flow(s, r, 0, r, mode, pin_off, pout_off, in_flow ? rows : 0, nsplit, part_scale, in_flow, series));
    if (in_flow && !series) return DION_OK;
    const int* uskip = in_flow ? (const int*)(s.os + OS_NOTNEAR) : skip;
    GemmArgs u = gemm_args();
    u.M = rows; u.N = r; u.K = r;
    u.a_si = r; u.a_sk = 1; u.b_sk = r; u.b_sn = 1; u.klimit = 1;
    u.C = s.ws + pout_off; u.ldc = r; u.epi = EPI_STORE; u.skip_flag = uskip;
    u.A = s.ws + pin_off;
    u.B = s.ws + s.L.Linv;
    if (gpairs) {
      __half* ph = reinterpret_cast<__half*>(s.ws + s.L.S16);
      __half* xh = reinterpret_cast<__half*>(s.ws + s.L.XP);
      launch_pdl(k_split_f16_tri, dim3((unsigned)tiles, (unsigned)s.nb), dim3(256), 0, s.st, (const float*)(s.ws + s.L.Linv), r,
                 (const float*)(s.ws + s.L.xmax), (const float*)(s.ws + s.L.gmax + AMAX_PARTS), xh, xh + r * r, s.ws + s.L.xmax + 1, s.wstride,
                 uskip, raw, series ? (const float*)(s.ws + s.L.Tbuf) : (const float*)nullptr, series ? (int*)nullptr : s.os);
      DION_CHECK_LAUNCH(c);
      GemmArgs h = u;
      h.ab16 = 1; h.f16 = 1;
      h.A = (const float*)ph; h.A16lo = ph + rows * r;
      h.B = (const float*)xh; h.B16lo = xh + r * r;
      h.alpha_dev = s.ws + s.L.xmax + 1; h.alpha_dev_stride = s.wstride;
      if (!series) h.skip_flag = s.os + OS_USE32;
      DION_TRY(launch_gemm_chain(s, h));
      u.precise = 1;      // (as accurate as the pairs are on a narrow range)
      u.skip_flag = s.os + OS_USEHALF;
    }
    if (!series) DION_TRY(launch_gemm_chain(s, u));
    if (series) {
      launch_pdl(k_near_end, dim3((unsigned)s.nb), dim3(1), 0, s.st, s.os, c->dev_ints + 2);
      DION_CHECK_LAUNCH(c);
    }
    return DION_OK;
  } else {
    launch_pdl(k_round_begin, dim3((unsigned)(s.nb)), dim3(256), 0, s.st, s.ws + s.L.Gram, r, r, 0.f, s.ws + s.L.gdiag, s.ws + s.L.scal, s.os,
                                          skips ? 1 : 0, s.wstride, c->dev_ints);
    DION_CHECK_LAUNCH(c);
    // Pout_J = (Pin_J - sum_{K<J} Pout_K L_{J,K}^T) Linv_JJ^T, block columns J of 512.
    // The solves run with the plain 3xTF32 product: their rounding error enters U once (~1e-6),
    // whereas an error in the Gram matrix or its factor is amplified by the panel's conditioning.
    // Block column J needs row block J of the factor and the inverse of its diagonal square, both
    // final once the factorization has passed J: the solves run on a second stream beside the rest
    // of the factorization, whose serial 64-column chain leaves most SMs idle.
    const float* Lm = s.ws + s.L.Gram;     // the factor, lower
    float* Wt = s.ws + (s.wt_off >= 0 ? s.wt_off : s.L.R);   // rows x 512 temporary (R is free during the orthonormalization)
    // On tall panels the two products of a block column run on scaled half pairs (22 significant bits in three
    // kind::f16 MMAs; 1024-k chains) like the Gram matrix: the right-hand side, the factor's row block and the
    // diagonal inverse are scaled by powers of two found on the device, the finished columns of Pout (entries of
    // an orthonormal basis; at most 1 / sqrt(pivot floor) = 100 in a deflating round) by 2^6.
    const bool spairs = s.wt_off < 0 && s.L.SolveP > 0 && solve_on_pairs(s, rows, r, mode);
    auto absmax_split = [&](const float* src, i64 ld, i64 nrows, i64 ncols, i64 out_off, i64 slot, float other_inv,
                            const float* other_dev) -> int {
      // pair of the nrows x ncols block at `src` (slice-relative pointer of matrix 0) into scratch at out_off; the
      // scale factor goes to smax slot `slot`
      i64 parts = (nrows * ncols / 4 + 2047) / 2048;
      if (parts < 1) parts = 1;
      if (parts > AMAX_PARTS) parts = AMAX_PARTS;
      float* pm = s.ws + s.L.smax + slot * (AMAX_PARTS + 64);
      launch_pdl(k_absmax_partial, dim3((unsigned)parts, (unsigned)s.nb), dim3(256), 0, s.st, src, ld, nrows, ncols, pm, s.wstride, skip,
                 (i64)OS_SLOT_INTS);
      DION_CHECK_LAUNCH(c);
      __half* hi = reinterpret_cast<__half*>(s.ws + out_off);
      launch_pdl(k_split_f16_scaled, dim3((unsigned)grid_for(c, nrows * ncols / 8, s.nb), (unsigned)s.nb), dim3(256), 0, s.st, src, ld, nrows, ncols,
                 (const float*)pm, (int)parts, hi, hi + nrows * ncols, pm + AMAX_PARTS, s.wstride, skip, (i64)OS_SLOT_INTS, other_inv, other_dev, (float*)nullptr, (int*)nullptr, 0, 0, 0);
      DION_CHECK_LAUNCH(c);
      return DION_OK;
    };
    auto solve_block_pairs = [&](i64 J0, i64 sz) -> int {
      const float* rhs = s.ws + pin_off + J0;
      i64 rhs_ld = r;
      __half* pop = reinterpret_cast<__half*>(s.ws + s.L.S16);          // pair of Pout: rows x r, dense
      const float* sc = s.ws + s.L.smax;
      if (J0 > 0) {
        // W = rhs - Pout[:, :J0] L[J0:J0+sz, :J0]^T
        DION_TRY(absmax_split(Lm + J0 * r, r, sz, J0, s.L.LfP, 0, ldexpf(1.f, -6), nullptr));
        __half* lh = reinterpret_cast<__half*>(s.ws + s.L.LfP);
        GemmArgs w = gemm_args();
        w.M = rows; w.N = sz; w.K = J0;
        w.ab16 = 1; w.f16 = 1;
        w.A = (const float*)pop; w.A16lo = pop + rows * r; w.a_si = r; w.a_sk = 1;
        w.B = (const float*)lh; w.B16lo = lh + sz * J0; w.b_sk = 1; w.b_sn = J0;
        w.C = Wt; w.ldc = NBO; w.epi = EPI_C2_SUB; w.C2 = rhs; w.ldc2 = r; w.c2_mode = ADD_F32;
        w.alpha_dev = sc + AMAX_PARTS; w.alpha_dev_stride = s.wstride;
        w.skip_flag = skip;
        DION_TRY(launch_gemm_chain(s, w, true));
        rhs = Wt; rhs_ld = NBO;
      }
      // V = rhs Linv_JJ^T
      DION_TRY(absmax_split(rhs, rhs_ld, rows, sz, s.L.SolveP, 1, 1.f, nullptr));
      const i64 li_off = s.L.LfP + NBO * r;      // (L^-T: row k, column j of the product's right operand)
      DION_TRY(absmax_split(s.ws + s.L.Linv + J0 * r + J0, r, sz, sz, li_off, 2, 1.f, sc + (AMAX_PARTS + 64) + AMAX_PARTS));
      __half* rh = reinterpret_cast<__half*>(s.ws + s.L.SolveP);
      __half* ih = reinterpret_cast<__half*>(s.ws + li_off);
      GemmArgs v = gemm_args();
      v.M = rows; v.N = sz; v.K = sz;
      v.ab16 = 1; v.f16 = 1;
      v.A = (const float*)rh; v.A16lo = rh + rows * sz; v.a_si = sz; v.a_sk = 1;
      v.B = (const float*)ih; v.B16lo = ih + sz * sz; v.b_sk = sz; v.b_sn = 1; v.klimit = 1;
      v.C = s.ws + pout_off + J0; v.ldc = r; v.epi = EPI_STORE; v.skip_flag = skip;
      v.alpha_dev = sc + 2 * (AMAX_PARTS + 64) + AMAX_PARTS; v.alpha_dev_stride = s.wstride;
      DION_TRY(launch_gemm_chain(s, v));
      if (J0 + sz < r) {      // the new block column of Pout joins the pair (later block columns read it)
        ChainPtrs t;
        for (int b = 0; b < s.nb; ++b) t.p[b] = s.W(b, pout_off + J0);
        launch_pdl(k_split_f16_fixed, dim3((unsigned)grid_for(c, rows * sz / 8, s.nb), (unsigned)s.nb), dim3(256), 0, s.st, t, r, rows, sz,
                   ldexpf(1.f, 6), pop + J0, pop + rows * r + J0, s.wstride, r, skip, (i64)OS_SLOT_INTS, (const int*)nullptr, (__half*)nullptr);
        DION_CHECK_LAUNCH(c);
      }
      return DION_OK;
    };
    auto solve_block = [&](i64 J0, i64 sz) -> int {
      if (spairs && sz >= 64 && sz % 8 == 0) return solve_block_pairs(J0, sz);
      const float* rhs = s.ws + pin_off + J0;
      i64 rhs_ld = r;
      if (J0 > 0) {
        GemmArgs w = gemm_args();
        w.M = rows; w.N = sz; w.K = J0;
        w.A = s.ws + pout_off; w.a_si = r; w.a_sk = 1;
        w.B = Lm + J0 * r; w.b_sk = 1; w.b_sn = r;
        w.C = Wt; w.ldc = NBO; w.epi = EPI_C2_SUB; w.C2 = rhs; w.ldc2 = r; w.c2_mode = ADD_F32;
        w.skip_flag = skip;
        DION_TRY(launch_gemm_chain(s, w, true));
        rhs = Wt; rhs_ld = NBO;
      }
      GemmArgs v = gemm_args();
      v.M = rows; v.N = sz; v.K = sz;
      v.A = rhs; v.a_si = rhs_ld; v.a_sk = 1;
      v.B = s.ws + s.L.Linv + J0 * r + J0; v.b_sk = r; v.b_sn = 1; v.klimit = 1;
      v.C = s.ws + pout_off + J0; v.ldc = r; v.epi = EPI_STORE; v.skip_flag = skip;
      DION_TRY(launch_gemm_chain(s, v));
      return DION_OK;
    };
    if (c->side != nullptr) {
      cudaStream_t main_st = s.st;
      auto next_event = [&]() { cudaEvent_t e = c->side_ev[c->side_cursor]; c->side_cursor = (c->side_cursor + 1) % 32; return e; };
      const std::function<int(i64, i64)> after_block = [&](i64 J0, i64 sz) -> int {
        cudaEvent_t e = next_event();
        if (cudaEventRecord(e, main_st) != cudaSuccess || cudaStreamWaitEvent(c->side, e, 0) != cudaSuccess) return DION_ERR_CUDA;
        s.st = c->side; s.no_split = true;
        const int rc = solve_block(J0, sz);
        s.st = main_st; s.no_split = false;
        return rc;
      };
      DION_TRY(potrf_blocked(s, r, mode, &after_block));
      cudaEvent_t e = next_event();   // join: the round ends when the last solve has finished
      if (cudaEventRecord(e, c->side) != cudaSuccess || cudaStreamWaitEvent(main_st, e, 0) != cudaSuccess) return DION_ERR_CUDA;
    } else {
      DION_TRY(potrf_blocked(s, r, mode, nullptr));
      for (i64 J0 = 0; J0 < r; J0 += NBO) DION_TRY(solve_block(J0, (r - J0 < NBO) ? (r - J0) : NBO));
    }
  }
  if (adaptive) {
    launch_pdl(k_round_end, dim3((unsigned)(s.nb)), dim3(1), 0, s.st, s.os, GOOD_REL, DONE_REL, c->dev_ints + 2);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// Householder factorization of the rows x r matrix A (ld = r): reflectors into V, the triangular
// factor into the rows of A above the diagonal and its diagonal into the matrix's d scratch.
int householder_factor(StepCtx& s, float* A, float* V, i64 rows, i64 r, int b) {
  dion_ctx* c = s.c;
  float* diag = s.W(b, s.L.d);
  for (i64 j = 0; j < r; ++j) {
    k_hh_reflector<<<1, 1024, 0, s.st>>>(A, r, rows, j, V, r, diag);
    DION_CHECK_LAUNCH(c);
    if (j + 1 < r) {
      const unsigned gx = (unsigned)((r - j - 1 + 31) / 32);
      k_hh_apply<<<gx, 256, 0, s.st>>>(A, r, rows, j, V, r, j, j + 1, r);
      DION_CHECK_LAUNCH(c);
    }
  }
  return DION_OK;
}

int householder(StepCtx& s, float* A, float* V, i64 rows, i64 r, int b) {
  dion_ctx* c = s.c;
  float* diag = s.W(b, s.L.d);
  DION_TRY(householder_factor(s, A, V, rows, r, b));
  {
    const i64 total = rows * r;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 8 * c->sm_count) blocks = 8 * c->sm_count;
    k_set_identity<<<blocks, 256, 0, s.st>>>(A, r, rows, r);
    DION_CHECK_LAUNCH(c);
    for (i64 j = r - 1; j >= 0; --j) {
      // columns < j of the partial product are still unit vectors e_c with c < j: untouched
      const unsigned gx = (unsigned)((r - j + 31) / 32);
      k_hh_apply<<<gx, 256, 0, s.st>>>(A, r, rows, j, V, r, j, j, r);
      DION_CHECK_LAUNCH(c);
    }
    k_sign_fix<<<blocks, 256, 0, s.st>>>(A, r, rows, r, diag);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// Adaptive rounds on the panel at off_a (ping-pong with off_b; the result ends at off_a): the device
// decides after each round whether the panel is done.
int adaptive_rounds(StepCtx& s, i64 off_a, i64 off_b, i64 rows, i64 r, i64 gram_rows) {
  static_assert(MAX_ROUNDS % 2 == 0, "the result must end in the first buffer");
  for (int it = 0; it < MAX_ROUNDS; it += 2) {
    DION_TRY(cholqr_round(s, off_a, off_b, rows, r, RM_ADAPTIVE, gram_rows, PROBE_CHECK, it));
    DION_TRY(cholqr_round(s, off_b, off_a, rows, r, RM_ADAPTIVE, gram_rows, PROBE_CHECK, it + 1));
  }
  {   // an odd number of rounds left the result in the second buffer
    dim3 grid((unsigned)grid_for(s.c, rows * r, s.nb), (unsigned)s.nb);
    launch_pdl(k_copy_panel, grid, dim3(256), 0, s.st, (const float*)(s.ws + off_b), r, s.ws + off_a, r, rows, r, (const int*)nullptr,
               (const int*)(s.os + OS_ROUNDS), s.wstride, 1);
    s.c->launches++;
  }
  launch_pdl(k_orth_finish, dim3((unsigned)(s.nb)), dim3(1), 0, s.st, s.os, s.c->dev_ints);
  s.c->launches++;
  if (cudaGetLastError() != cudaSuccess) return DION_ERR_CUDA;
  return DION_OK;
}

// The second round of CholeskyQR2, when it ran, went P0 -> P1: its result back to P0.
int second_round_back(StepCtx& s, i64 rows, i64 r) {
  dim3 grid((unsigned)grid_for(s.c, rows * r, s.nb), (unsigned)s.nb);
  launch_pdl(k_copy_panel, grid, dim3(256), 0, s.st, (const float*)(s.ws + s.L.P1), r, s.ws + s.L.P0, r, rows, r,
             (const int*)(s.os + OS_DONE), (const int*)nullptr, s.wstride, -1);
  DION_CHECK_LAUNCH(s.c);
  return DION_OK;
}

// Randomized Cholesky QR (Algorithm 4 on one device) of the rows x r panel in P0 of every
// matrix of the chain; U ends in P0.
//   Pt = S P (k x r sketch).  R1 = triangular factor of QR(Pt): computed by deflating Cholesky-QR
//   rounds on the sketch, never formed explicitly -- the rounds run on the stacked panel [Pt; P] with
//   their Gram matrices taken from the sketch rows only, so every round's triangular factor is applied
//   to the sketch and to P at once; when the sketch has become orthonormal, the lower rows hold
//   B = P R1^-1.  Then Cholesky QR on B (R2 = Cholesky(B^T B), U = B R2^-1; a second pass only if the
//   device's check asks for it).  All matrices of a chain have the same number of sketch rows.
int rcqr(StepCtx& s, i64 rows, i64 r) {
  dion_ctx* c = s.c;
  if (s.list == nullptr) return DION_ERR_INVALID;
  const i64 k = s.list[0]->sketch_rows;
  for (int b = 0; b < s.nb; ++b) {
    const dion_matrix* a = s.list[b];
    if (a->sketch_rows != k) return DION_ERR_INVALID;
    float* stack = s.W(b, s.L.Sk);
    GemmArgs g = gemm_args();
    g.M = k; g.N = r; g.K = rows;
    g.A = (const float*)a->sketch; g.a_si = a->ld_sketch; g.a_sk = 1;
    g.B = s.W(b, s.L.P0); g.b_sk = r; g.b_sn = 1;
    g.C = stack; g.ldc = r; g.epi = EPI_STORE; g.precise = 1;
    DION_TRY(launch_gemm(s, g, b));
    dim3 grid((unsigned)grid_for(c, rows * r), 1);
    launch_pdl(k_copy_block, grid, dim3(256), 0, s.st, (const float*)s.W(b, s.L.P0), r, stack + k * r, r, rows, r, nullptr, 0, (const int*)nullptr, (int*)nullptr, (int*)nullptr);
    DION_CHECK_LAUNCH(c);
  }
  s.wt_off = s.L.SkW;
  const int rc = adaptive_rounds(s, s.L.Sk, s.L.SkV, k + rows, r, k);
  s.wt_off = -1;
  DION_TRY(rc);
  // B = the panel rows of the stack; the step's state slot starts afresh for its Cholesky QR
  launch_pdl(k_reset_rounds, dim3((unsigned)s.nb), dim3(1), 0, s.st, s.os);
  DION_CHECK_LAUNCH(c);
  DION_TRY(cholqr_round(s, s.L.Sk + k * r, s.L.P0, rows, r, RM_FIRST));
  DION_TRY(cholqr_round(s, s.L.P0, s.L.P1, rows, r, RM_CHECKED));
  return second_round_back(s, rows, r);
}

// The orthonormalization a step on (m, n, r) will use.
int resolve_orth(const dion_ctx* c, i64 r, i64 short_dim) {
  int mode = c->cfg.orth;
  if (mode == DION_ORTH_AUTO) mode = (4 * r <= short_dim) ? DION_ORTH_CHOLQR2 : DION_ORTH_SHIFTED3;
  return mode;
}

// ... for a chain with (step) or without (Lazy-Dion, data-parallel calls) the sketches of the RCQR mode.
int resolve_orth_for(const dion_ctx* c, i64 r, i64 short_dim, bool has_sketches) {
  int mode = resolve_orth(c, r, short_dim);
  if (mode == DION_ORTH_RCQR && !has_sketches) mode = (4 * r <= short_dim) ? DION_ORTH_CHOLQR2 : DION_ORTH_SHIFTED3;
  return mode;
}

// Where the product that forms the panel writes it: CholeskyQR2 reads it from the save buffer (round one goes
// Psave -> P0, round two P0 -> P1), so that the panel is still there if a pivot fails; every other mode works in P0.
i64 panel_offset(const StepCtx& s, i64 r, i64 short_dim) {
  const bool cq2 = resolve_orth_for(s.c, r, short_dim, s.list != nullptr) == DION_ORTH_CHOLQR2;
  return (cq2 && s.L.Psave > 0) ? s.L.Psave : s.L.P0;
}

// The device-side fallback of CholeskyQR2 (k_cgs_fallback): one cooperative launch over the chain's matrices.
// second_off >= 0: where the second round, if it ran, left its result (copied to pout_off by the same launch).
int cgs_fallback(StepCtx& s, i64 pin_off, i64 pout_off, i64 rows, i64 r, i64 second_off = -1) {
  dion_ctx* c = s.c;
  i64 G = rows / 8;
  if (G < 1) G = 1;
  if (G > c->sm_count) G = c->sm_count;
  const float* Pin = s.ws + pin_off;
  float* U = s.ws + pout_off;
  float* part = s.ws + s.L.fb_part;
  float* hvec = s.ws + s.L.fb_h;
  float* npart = s.ws + s.L.fb_n;
  int* os = s.os;
  int* status = c->dev_ints;
  int* fallbacks = c->dev_ints + 3;
  i64 ld = r, wstride = s.wstride;
  int nb = s.nb;
  long long limit = umma::SPIN_LIMIT_CYCLES;
  const float* second = second_off >= 0 ? s.ws + second_off : nullptr;
  void* args[] = {&Pin, &U, &ld, &rows, &r, &part, &hvec, &npart, &os, &status, &fallbacks, &wstride, &nb, &limit, &second};
  if (cudaLaunchCooperativeKernel((const void*)k_cgs_fallback, dim3((unsigned)G), dim3(256), args, 0, s.st) != cudaSuccess) {
    cudaGetLastError();
    return DION_ERR_CUDA;
  }
  c->launches++;
  return DION_OK;
}

bool fallback_fits(const dion_ctx* c, i64 rows) {
  return (rows + c->sm_count - 1) / c->sm_count <= CGS_MAX_ROWS_PER_CTA;
}

// Orthonormalize the rows x r panel at pin_off (= panel_offset) of every matrix of the chain; *U_off is the
// scratch offset of the buffer that holds U afterwards.
int orthonormalize(StepCtx& s, i64 rows, i64 r, i64 short_dim, i64 pin_off, i64* U_off) {
  const int mode = resolve_orth_for(s.c, r, short_dim, s.list != nullptr);
  if (mode == DION_ORTH_CHOLQR2) {
    // the first round with the accurate products; the second one only if the first one's result is
    // not yet orthonormal to ORTH_TAU_F (measured by the probe).  A pivot that is not positive in
    // either round (the paper's "CQR failure") raises the step's fail flag only; the fallback kernel then
    // orthonormalizes the saved panel and clears the flag, or confirms the breakdown.
    const bool fb = pin_off != s.L.P0 && fallback_fits(s.c, rows);
    if (r <= NB && rows <= TINY_MAX_ROWS && s.redo_p == nullptr) {
      // a panel that fits one CTA's shared memory: both rounds and the test between them in one launch
      launch_pdl(k_tiny_cholqr2, dim3((unsigned)s.nb), dim3(TINY_THREADS), (size_t)tiny_cholqr2_smem(rows), s.st, (const float*)(s.ws + pin_off),
                 s.ws + s.L.P0, (int)rows, (int)r, s.os, ORTH_TAU_F, s.c->dev_ints + 2, fb ? (int*)nullptr : s.c->dev_ints, s.c->dev_ints,
                 s.wstride);
      DION_CHECK_LAUNCH(s.c);
      if (fb) DION_TRY(cgs_fallback(s, pin_off, s.L.P0, rows, r));
      *U_off = s.L.P0;
      return DION_OK;
    }
    s.quiet_fail = fb;
    // Round one writes P0, where U is expected; the second round, when it runs, goes P0 -> P1 and is copied
    // back: the common case (one round) moves the panel once.
    int rc = cholqr_round(s, pin_off, s.L.P0, rows, r, RM_FIRST);
    const bool redo = s.redo_p != nullptr;
    if (redo) {
      // The panel came from the fast product (bf16 operand pairs, ~1e-5): good enough exactly when the panel is well
      // conditioned, which the probe of the first round's result shows.  Otherwise the device recomputes the panel
      // with the accurate product and repeats the round; all of that is launched and skipped in the common case.
      if (rc == DION_OK) rc = probe(s, s.L.P0, rows, r, PROBE_FAST);
      if (rc == DION_OK) rc = (*s.redo_p)();
      if (rc == DION_OK) rc = cholqr_round(s, pin_off, s.L.P0, rows, r, RM_REDO);
    }
    if (rc == DION_OK) rc = cholqr_round(s, s.L.P0, s.L.P1, rows, r, RM_CHECKED, 0, redo ? PROBE_AFTER_REDO : PROBE_CHECK);
    s.quiet_fail = false;
    DION_TRY(rc);
    if (fb) DION_TRY(cgs_fallback(s, pin_off, s.L.P0, rows, r, s.L.P1));      // (which also brings the second round's result back)
    else DION_TRY(second_round_back(s, rows, r));                           // (the failed pivot was reported as a breakdown)
    *U_off = s.L.P0;
  } else if (mode == DION_ORTH_SHIFTED3) {
    DION_TRY(adaptive_rounds(s, s.L.P0, s.L.P1, rows, r, 0));
    *U_off = s.L.P0;
  } else if (mode == DION_ORTH_RCQR) {
    DION_TRY(rcqr(s, rows, r));
    *U_off = s.L.P0;
  } else {
    for (int m = 0; m < s.nb; ++m) DION_TRY(householder(s, s.W(m, s.L.P0), s.W(m, s.L.P1), rows, r, m));
    *U_off = s.L.P0;
  }
  return DION_OK;
}

// Columns of W (rows x r) normalized into Q, for `per` matrices of the chain from b on: W (wstride apart), Q and d from pointer
// tables.  x.kind != 0: the operands of the rank-r updates too (offsets in the scratch slices; see k_colnorm_apply).
// sums != nullptr: the columns' sums of squares, given by the caller (sharded form).
int colnorm_launch(StepCtx& s, int b, int per, const float* W, i64 ldw, i64 rows, i64 r, const ChainPtrs& Qs, i64 ldq, const ChainPtrs& ds,
                   const int* skip, ColnormPairs x = ColnormPairs(), const float* sums = nullptr) {
  dion_ctx* c = s.c;
  int chunks; i64 rpc;
  colnorm_chunks(c, s.L, rows, r, &chunks, &rpc);
  const dim3 grid((unsigned)((r + 127) / 128), (unsigned)chunks, (unsigned)per);
  float* part = s.W(b, s.L.cn_part);
  const bool v4 = r % 4 == 0 && ldw % 4 == 0 && !((uintptr_t)W & 15);
  float* amax = nullptr;
  if (x.kind == CN_HALF) {
    x.scal = s.W(b, s.L.lz) + HS_EF;
    if (x.range == nullptr) {
      amax = s.W(b, s.L.lz) + HS_MAX;
      x.amax = amax;
      x.nmax = (int)(grid.x * grid.y);
    }
  }
  if (sums == nullptr) {
    if (v4) launch_pdl(k_colsumsq_partial<true>, grid, dim3(CN_THREADS), 0, s.st, W, ldw, rows, r, rpc, part, amax, (const int*)nullptr, s.wstride);
    else launch_pdl(k_colsumsq_partial<false>, grid, dim3(CN_THREADS), 0, s.st, W, ldw, rows, r, rpc, part, amax, (const int*)nullptr, s.wstride);
    DION_CHECK_LAUNCH(c);
  }
  int qvec = ldq % 4 == 0;
  for (int k = 0; k < per; ++k) qvec = qvec && !((uintptr_t)Qs.p[k] & 15);
  if (sums != nullptr) chunks = 1;
  i64 rpb = (rows * (i64)grid.x * per + 3 * c->sm_count - 1) / (3 * c->sm_count);      // three blocks per SM, all at once
  if (rpb < 32) rpb = 32;
  const dim3 agrid(grid.x, (unsigned)((rows + rpb - 1) / rpb), grid.z);
  const float* sp = sums != nullptr ? sums : (const float*)part;
  auto apply = [&](auto kernel) {
    launch_pdl(kernel, agrid, dim3(CN_THREADS), 0, s.st, W, ldw, rows, r, rpb, chunks, sp, c->cfg.eps, Qs, ldq, qvec, s.W(b, s.L.d), ds,
               c->dev_ints, skip, s.wstride, x, c->dev_ints + 1);
  };
  if (!v4) apply(k_colnorm_apply<false, false>);
  else if (x.qpair != 0) apply(k_colnorm_apply<true, true>);
  else apply(k_colnorm_apply<true, false>);
  DION_CHECK_LAUNCH(c);
  return DION_OK;
}

// ... of one matrix.
int colnorm(StepCtx& s, int b, const float* W, i64 rows, i64 r, float* out, i64 ldo, float* d_out,
            const int* skip = nullptr, ColnormPairs x = ColnormPairs(), const float* sums = nullptr) {
  ChainPtrs Qs, ds;
  Qs.p[0] = out; ds.p[0] = d_out;
  return colnorm_launch(s, b, 1, W, r, rows, r, Qs, ldo, ds, skip != nullptr ? skip : (const int*)(s.OS(b) + OS_FAIL), x, sums);
}

// ---- elementwise kernels over a whole chain -------------------------------------------------------------------
// Each helper makes ONE launch over the chain's matrices (blockIdx.y or .z) when their arrays share leading
// dimensions and alignment, else one launch per matrix; outputs are in the scratch slices either way.

// ColNorm of every matrix's R (scratch, rows x r dense) into its Q, d exported to colnorm_out; kind, qh_off, qscale, pair_off: the
// rank-r updates' operands beside it (offsets in the scratch slices).
int colnorm_chain(StepCtx& s, const dion_matrix* const* list, i64 rows, i64 r, int kind = 0, i64 qh_off = 0, float qscale = 1.f, i64 pair_off = 0) {
  bool one = s.nb <= GEMM_TAB_MAX && (s.nb == 1 || s.c->chain_batch);
  for (int b = 1; b < s.nb && one; ++b)
    one = list[b]->ldq == list[0]->ldq && ((uintptr_t)list[b]->Q & 15) == ((uintptr_t)list[0]->Q & 15);
  const int per = one ? s.nb : 1;
  for (int b = 0; b < s.nb; b += per) {
    ChainPtrs Qs, ds;
    for (int k = 0; k < per; ++k) { Qs.p[k] = list[b + k]->Q; ds.p[k] = list[b + k]->colnorm_out; }
    ColnormPairs x = ColnormPairs();
    x.kind = kind; x.qh = s.W(b, qh_off); x.qscale = qscale; x.hi = s.W(b, pair_off);
    if (kind == CN_HALF) x.os = s.OS(b);
    DION_TRY(colnorm_launch(s, b, per, s.W(b, s.L.R), r, rows, r, Qs, list[b]->ldq, ds, s.OS(b) + OS_FAIL, x));
  }
  return DION_OK;
}

// hi / lo bf16 pair of src[b] (rows x cols, leading dimension ld[b]) into the scratch slices at out_off.
// skip0: the flag of matrix 0 (a state slot apart per matrix), or nullptr.
// copy_off >= 0 (chain launch only): a dense fp32 copy of the sources in the scratch slices too; *copied says whether it was made.
// one_off >= 0: half(one_scale src) too.
int split_chain(StepCtx& s, const float* const* src, const i64* ld, i64 rows, i64 cols, i64 out_off, const int* skip0,
                i64 copy_off = -1, bool* copied = nullptr, i64 one_off = -1, float one_scale = 0.f) {
  dion_ctx* c = s.c;
  bool one = s.nb > 1 && s.nb <= GEMM_TAB_MAX && c->chain_batch;
  for (int b = 1; b < s.nb && one; ++b) one = ld[b] == ld[0];
  const unsigned gx = (unsigned)grid_for(c, rows * cols / 8, one ? s.nb : 1);
  if (one) {
    ChainPtrs t;
    for (int b = 0; b < s.nb; ++b) t.p[b] = src[b];
    __nv_bfloat16* hi = reinterpret_cast<__nv_bfloat16*>(s.ws + out_off);
    launch_pdl(k_split_bf16_chain, dim3(gx, (unsigned)s.nb), dim3(256), 0, s.st, t, ld[0], rows, cols, hi, hi + rows * cols, s.wstride, skip0,
               (i64)OS_SLOT_INTS, copy_off >= 0 ? s.ws + copy_off : (float*)nullptr,
               one_off >= 0 ? reinterpret_cast<__half*>(s.ws + one_off) : (__half*)nullptr, one_scale);
    DION_CHECK_LAUNCH(c);
    if (copied != nullptr) *copied = copy_off >= 0;
    return DION_OK;
  }
  if (copied != nullptr) *copied = false;
  for (int b = 0; b < s.nb; ++b) {
    __nv_bfloat16* hi = reinterpret_cast<__nv_bfloat16*>(s.W(b, out_off));
    launch_pdl(k_split_bf16, dim3(gx), dim3(256), 0, s.st, src[b], ld[b], rows, cols, hi, hi + rows * cols,
               skip0 != nullptr ? skip0 + (i64)b * OS_SLOT_INTS : (const int*)nullptr,
               one_off >= 0 ? reinterpret_cast<__half*>(s.W(b, one_off)) : (__half*)nullptr, one_scale);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// ... as a half pair scaled by 2^bits, or a bf16 pair where a matrix's range is wide (OS_WIDE).  one_off >= 0: the half array
// alone too, whichever pair it is.
int split_half_chain(StepCtx& s, const float* const* src, i64 ld, i64 rows, i64 cols, i64 out_off, int bits, const int* skip0, i64 one_off) {
  dion_ctx* c = s.c;
  const int per = (s.nb <= GEMM_TAB_MAX && c->chain_batch) ? s.nb : 1;
  for (int b = 0; b < s.nb; b += per) {
    ChainPtrs t;
    for (int k = 0; k < per; ++k) t.p[k] = src[b + k];
    __half* hi = reinterpret_cast<__half*>(s.W(b, out_off));
    launch_pdl(k_split_f16_fixed, dim3((unsigned)grid_for(c, rows * cols / 8, per), (unsigned)per), dim3(256), 0, s.st, t, ld, rows, cols, ldexpf(1.f, bits),
               hi, hi + rows * cols, s.wstride, (i64)0, skip0 != nullptr ? skip0 + (i64)b * OS_SLOT_INTS : (const int*)nullptr, (i64)OS_SLOT_INTS,
               (const int*)(s.OS(b) + OS_WIDE), one_off >= 0 ? reinterpret_cast<__half*>(s.W(b, one_off)) : (__half*)nullptr);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// src[b] rounded to TF32 into the scratch slices at out_off.
// half_scale > 0: IEEE half values of half_scale * src instead (see x_half).
int round_chain(StepCtx& s, const float* const* src, const i64* ld, i64 rows, i64 cols, i64 out_off, const int* skip0,
                float half_scale = 0.f) {
  dion_ctx* c = s.c;
  bool one = s.nb > 1 && s.nb <= GEMM_TAB_MAX && c->chain_batch;
  for (int b = 1; b < s.nb && one; ++b) one = ld[b] == ld[0];
  if (half_scale > 0.f) {
    const unsigned g8 = (unsigned)grid_for(c, rows * cols / 8, one ? s.nb : 1);
    if (one) {
      ChainPtrs t;
      for (int b = 0; b < s.nb; ++b) t.p[b] = src[b];
      launch_pdl(k_round_f16_chain, dim3(g8, (unsigned)s.nb), dim3(256), 0, s.st, t, ld[0], rows, cols, half_scale,
                 reinterpret_cast<__half*>(s.ws + out_off), s.wstride, skip0, (i64)OS_SLOT_INTS);
      DION_CHECK_LAUNCH(c);
      return DION_OK;
    }
    for (int b = 0; b < s.nb; ++b) {
      launch_pdl(k_round_f16, dim3(g8), dim3(256), 0, s.st, src[b], ld[b], rows, cols, half_scale, reinterpret_cast<__half*>(s.W(b, out_off)),
                 skip0 != nullptr ? skip0 + (i64)b * OS_SLOT_INTS : (const int*)nullptr);
      DION_CHECK_LAUNCH(c);
    }
    return DION_OK;
  }
  const unsigned gx = (unsigned)grid_for(c, rows * cols / 4, one ? s.nb : 1);
  if (one) {
    ChainPtrs t;
    for (int b = 0; b < s.nb; ++b) t.p[b] = src[b];
    launch_pdl(k_round_tf32_chain, dim3(gx, (unsigned)s.nb), dim3(256), 0, s.st, t, ld[0], rows, cols, s.ws + out_off, s.wstride, skip0,
               (i64)OS_SLOT_INTS);
    DION_CHECK_LAUNCH(c);
    return DION_OK;
  }
  for (int b = 0; b < s.nb; ++b) {
    launch_pdl(k_round_tf32, dim3(gx), dim3(256), 0, s.st, src[b], ld[b], rows, cols, s.W(b, out_off),
               skip0 != nullptr ? skip0 + (i64)b * OS_SLOT_INTS : (const int*)nullptr);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t a0 = (uintptr_t)a, b0 = (uintptr_t)b;
  return a0 < b0 + nb && b0 < a0 + na;
}

// shard: `a` describes a column shard of a wider matrix (the sharded calls): r may exceed its n.
int validate(const dion_matrix* a, bool shard = false) {
  if (a == nullptr) return DION_ERR_INVALID;
  if (a->X == nullptr || a->M == nullptr || a->G == nullptr || a->Q == nullptr) return DION_ERR_INVALID;
  if (a->g_dtype != DION_F32 && a->g_dtype != DION_BF16) return DION_ERR_INVALID;
  if (a->m < 1 || a->n < 1) return DION_ERR_SHAPE;
  if (a->r < 1 || a->r > a->m || (!shard && a->r > a->n)) return DION_ERR_SHAPE;
  if (a->ldx < a->n || a->ldm < a->n || a->ldg < a->n || a->ldq < a->r) return DION_ERR_SHAPE;
  if (a->transposed != 0 && a->transposed != 1) return DION_ERR_INVALID;
  const i64 qrows = a->transposed ? a->m : a->n;
  const size_t gsz = (a->g_dtype == DION_BF16) ? 2 : 4;
  if (((uintptr_t)a->X & 3) || ((uintptr_t)a->M & 3) || ((uintptr_t)a->Q & 3) || ((uintptr_t)a->G & (gsz - 1)))
    return DION_ERR_ALIGN;
  if (a->colnorm_out != nullptr && ((uintptr_t)a->colnorm_out & 3)) return DION_ERR_ALIGN;
  const size_t nx = (size_t)((a->m - 1) * a->ldx + a->n) * 4, nm = (size_t)((a->m - 1) * a->ldm + a->n) * 4;
  const size_t ng = (size_t)((a->m - 1) * a->ldg + a->n) * gsz, nq = (size_t)((qrows - 1) * a->ldq + a->r) * 4;
  if (overlap(a->X, nx, a->M, nm) || overlap(a->X, nx, a->G, ng) || overlap(a->X, nx, a->Q, nq) ||
      overlap(a->M, nm, a->G, ng) || overlap(a->M, nm, a->Q, nq) || overlap(a->G, ng, a->Q, nq))
    return DION_ERR_ALIAS;
  if (a->colnorm_out != nullptr) {
    const size_t nc = (size_t)a->r * 4;
    if (overlap(a->colnorm_out, nc, a->X, nx) || overlap(a->colnorm_out, nc, a->M, nm) ||
        overlap(a->colnorm_out, nc, a->G, ng) || overlap(a->colnorm_out, nc, a->Q, nq))
      return DION_ERR_ALIAS;
  }
  return DION_OK;
}

int begin_step(dion_ctx* c, const dion_matrix* a, int nb, cudaStream_t st, StepCtx* s, int fixed_slot = -1) {
  s->c = c;
  s->st = st;
  s->L = make_layout(c, a->m, a->n, a->r);
  s->ws = c->ws;
  s->nb = nb;
  s->wstride = s->L.total;
  if (fixed_slot >= 0) {
    s->os = c->dev_ints + 8 + (i64)fixed_slot * OS_SLOT_INTS;
  } else {
    if (c->flag_cursor + nb > MAX_FLAG_SLOTS - MAX_GRAPHS) c->flag_cursor = 0;   // the slots of a chain are contiguous
    s->os = c->dev_ints + 8 + (i64)c->flag_cursor * OS_SLOT_INTS;
    c->flag_cursor = (c->flag_cursor + nb) % (MAX_FLAG_SLOTS - MAX_GRAPHS);
  }
  s->flag = s->os + OS_FAIL;
  s->tensor = (c->cfg.engine != DION_ENGINE_SIMT);
  s->in_orth = false;
  return DION_OK;
}

// The state slots of a chain start at zero: cleared by the first kernel of a step where it can (a memset is a launch of its own and
// lets nothing start beside it: 3 us; the step of one data-parallel rank, 4096 x 2048, r = 256: 296 -> 285 us), else here; flag (optional): the caller's flag too.
int clear_slots(const StepCtx& s, int* flag = nullptr) {
  if (cudaMemsetAsync(s.os, 0, sizeof(int) * OS_SLOT_INTS * s.nb, s.st) != cudaSuccess) return DION_ERR_CUDA;
  return flag == nullptr || cudaMemsetAsync(flag, 0, sizeof(int), s.st) == cudaSuccess ? DION_OK : DION_ERR_CUDA;
}

// R = (M + G)^T U on bf16 pairs (transposed form: (M + G) U): where M + G is kept in scratch (sum_in_scratch) the
// product runs on the bf16 (hi, lo) pair of the sum and of U, three bf16 MMAs per K step (1.3 TF32 passes instead of
// three); it is accurate to ~1e-5, which is what Q <- ColNorm(R) and the error feedback need of it.
bool r_on_pairs(const StepCtx& s, i64 m, i64 n, i64 r) {
  return s.tensor && s.c->cfg.precision == DION_PREC_FP32 && s.L.B32 > 0 && s.L.Bp > 0 && m >= 128 && n >= 128 && r >= 64;
}

// The steps whose four products run on scaled half pairs (k_form_sum_amax): CholeskyQR2 panels up to the size from which P
// runs on the bf16 pairs that one pass over M + G makes.
// M + G is read once more (from L2 where it fits), but P leaves the 3xTF32 form, whose converter warps bound it, for three
// half MMAs per K step, U's pair also serves the weight update, and every result carries 22 bits (768^2 to 768 x 3072 at
// r = 192, 72 matrices in one call: P 932 -> 516 us, R 420 -> 194 us with the unsplit chains, weight update 200 -> 173 us;
// errors of Q and M 2 to 5 times smaller).  From P_PAIR_MIN_MNR on the second pass would be over HBM.
// The rule looks at the shape alone, so that a grouped call computes what single calls compute.
bool step_on_half_pairs(const StepCtx& s, i64 m, i64 n, i64 r, i64 short_dim) {
  const i64 mnr = m * n * r;
  return r_on_pairs(s, m, n, r) && s.L.Bh == 0 && (double)mnr < P_PAIR_MIN_MNR &&
         resolve_orth_for(s.c, r, short_dim, s.list != nullptr) == DION_ORTH_CHOLQR2;
}

// M + G and the half pairs of it and of Q (in S16) for every matrix of the chain: in one pair of launches when they share
// leading dimensions and alignment.  ranges: matrices of wide range are flagged and get what the other formats need instead
// (Q dense in P1, a bf16 pair of the sum).  clear: the state slots are cleared here; flag (one matrix): the caller's flag too.
int half_sum_chain(StepCtx& s, const dion_matrix* const* list, i64 qrow, bool clear, bool ranges, int* flag = nullptr) {
  dion_ctx* c = s.c;
  const dion_matrix* a0 = list[0];
  const i64 m = a0->m, n = a0->n, r = a0->r;
  auto vec_ok = [](const dion_matrix* a) {
    return !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 &&
           (a->g_dtype == DION_BF16 ? (!((uintptr_t)a->G & 7) && a->ldg % 4 == 0) : (!((uintptr_t)a->G & 15) && a->ldg % 4 == 0));
  };
  auto qvec_ok = [](const dion_matrix* a) { return !((uintptr_t)a->Q & 15) && a->ldq % 4 == 0; };
  bool one = s.nb <= GEMM_TAB_MAX && (s.nb == 1 || c->chain_batch);
  for (int b = 1; b < s.nb && one; ++b)
    one = list[b]->ldm == a0->ldm && list[b]->ldg == a0->ldg && list[b]->g_dtype == a0->g_dtype && vec_ok(list[b]) == vec_ok(a0) &&
          list[b]->ldq == a0->ldq && qvec_ok(list[b]) == qvec_ok(a0);
  const int per = one ? s.nb : 1;
  for (int b = 0; b < s.nb; b += per) {
    const dion_matrix* a = list[b];
    ChainPtrs Ms, Gs, Qs;
    for (int k = 0; k < per; ++k) { Ms.p[k] = list[b + k]->M; Gs.p[k] = list[b + k]->G; Qs.p[k] = list[b + k]->Q; }
    const int g_mode = (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32;
    const i64 pieces = (m + RANGE_ROWS - 1) / RANGE_ROWS * ((n + 127) / 128);
    const dim3 fg((unsigned)grid_for(c, 32 * pieces, per), (unsigned)per), sg((unsigned)grid_for(c, (m * n + qrow * r) / 8, per), (unsigned)per);
    float* part = s.W(b, s.L.part);      // (the ranges are read before the products write their partial sums there)
    const int qv = qvec_ok(a) ? 1 : 0;
    if (vec_ok(a)) launch_pdl(k_form_sum_amax<true>, fg, dim3(256), 0, s.st, Ms, a->ldm, Gs, a->ldg, g_mode, m, n, Qs, a->ldq, qrow, r, qv, s.W(b, s.L.B32), part, s.wstride, clear ? s.OS(b) : (int*)nullptr, flag);
    else launch_pdl(k_form_sum_amax<false>, fg, dim3(256), 0, s.st, Ms, a->ldm, Gs, a->ldg, g_mode, m, n, Qs, a->ldq, qrow, r, qv, s.W(b, s.L.B32), part, s.wstride, clear ? s.OS(b) : (int*)nullptr, flag);
    DION_CHECK_LAUNCH(c);
    launch_pdl(k_split_sum, sg, dim3(256), 0, s.st, (const float*)s.W(b, s.L.B32), m * n, Qs, a->ldq, qrow, r, qv, (const float*)part, (int)fg.x,
               reinterpret_cast<__half*>(s.W(b, s.L.Bp)), reinterpret_cast<__half*>(s.W(b, s.L.S16)), s.W(b, s.L.P1), s.W(b, s.L.lz),
               ranges ? s.OS(b) : (int*)nullptr, s.wstride);
    DION_CHECK_LAUNCH(c);
  }
  return DION_OK;
}

// P = (M + G) Q of a matrix of a step on half pairs, where its range is wide: the 3xTF32 product of the fp32 sum and the dense
// copy of Q.  (Launched behind the product on half pairs; each of the two finds itself flagged for the other's matrices.)
GemmArgs wide_p(const StepCtx& s, int b, const dion_matrix* a, bool tr, float* P) {
  const i64 n = a->n, r = a->r;
  GemmArgs p = gemm_args();
  p.M = tr ? n : a->m; p.N = r; p.K = tr ? a->m : n;
  p.A = s.W(b, s.L.B32); p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
  p.B = s.W(b, s.L.P1); p.b_sk = r; p.b_sn = 1;
  p.C = P; p.ldc = r; p.epi = EPI_STORE;
  p.skip_flag = s.OS(b) + OS_PHALF;
  p.precise = 1;      // (as accurate as the half pairs are on a narrow range: 1.4e-6; 8e-6 without)
  return p;
}

// Forms M + G in scratch (fp32) and, when `pair`, as a bf16 pair beside it.
int form_sum(StepCtx& s, int b, const dion_matrix* a, bool pair, bool clear = false) {
  dion_ctx* c = s.c;
  const i64 m = a->m, n = a->n;
  const bool vec = !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 &&
                   (a->g_dtype == DION_BF16 ? (!((uintptr_t)a->G & 7) && a->ldg % 4 == 0)
                                            : (!((uintptr_t)a->G & 15) && a->ldg % 4 == 0));
  const int g_mode = (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32;
  const int grid = grid_for(c, m * n / 4);
  __nv_bfloat16* bh = pair ? reinterpret_cast<__nv_bfloat16*>(s.W(b, s.L.Bp)) : nullptr;
  __nv_bfloat16* bl = pair ? bh + m * n : nullptr;
  if (vec) launch_pdl(k_form_b32<true>, grid, dim3(256), 0, s.st, (const float*)a->M, a->ldm, a->G, a->ldg, g_mode, m, n, s.W(b, s.L.B32), bh, bl, clear ? s.OS(b) : (int*)nullptr);
  else launch_pdl(k_form_b32<false>, grid, dim3(256), 0, s.st, (const float*)a->M, a->ldm, a->G, a->ldg, g_mode, m, n, s.W(b, s.L.B32), bh, bl, clear ? s.OS(b) : (int*)nullptr);
  DION_CHECK_LAUNCH(c);
  return DION_OK;
}

// form_sum for every matrix of the chain: one launch when M and G share leading dimensions and alignment.
int form_sum_chain(StepCtx& s, const dion_matrix* const* list, bool pair, bool clear = false) {
  dion_ctx* c = s.c;
  const dion_matrix* a0 = list[0];
  auto vec_ok = [](const dion_matrix* a) {
    return !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 &&
           (a->g_dtype == DION_BF16 ? (!((uintptr_t)a->G & 7) && a->ldg % 4 == 0) : (!((uintptr_t)a->G & 15) && a->ldg % 4 == 0));
  };
  bool one = s.nb > 1 && s.nb <= GEMM_TAB_MAX && c->chain_batch;
  const bool vec = vec_ok(a0);
  for (int b = 1; b < s.nb && one; ++b)
    one = list[b]->ldm == a0->ldm && list[b]->ldg == a0->ldg && list[b]->g_dtype == a0->g_dtype && vec_ok(list[b]) == vec;
  if (!one) {
    for (int b = 0; b < s.nb; ++b) DION_TRY(form_sum(s, b, list[b], pair, clear));
    return DION_OK;
  }
  const i64 m = a0->m, n = a0->n;
  ChainPtrs Ms, Gs;
  for (int b = 0; b < s.nb; ++b) { Ms.p[b] = list[b]->M; Gs.p[b] = list[b]->G; }
  const int g_mode = (a0->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32;
  __nv_bfloat16* bh = pair ? reinterpret_cast<__nv_bfloat16*>(s.ws + s.L.Bp) : nullptr;
  __nv_bfloat16* bl = pair ? bh + m * n : nullptr;
  const dim3 grid((unsigned)grid_for(c, m * n / 4, s.nb), (unsigned)s.nb);
  if (vec) launch_pdl(k_form_b32_chain<true>, grid, dim3(256), 0, s.st, Ms, a0->ldm, Gs, a0->ldg, g_mode, m, n, s.ws + s.L.B32, bh, bl, s.wstride, clear ? s.os : (int*)nullptr);
  else launch_pdl(k_form_b32_chain<false>, grid, dim3(256), 0, s.st, Ms, a0->ldm, Gs, a0->ldg, g_mode, m, n, s.ws + s.L.B32, bh, bl, s.wstride, clear ? s.os : (int*)nullptr);
  DION_CHECK_LAUNCH(c);
  return DION_OK;
}

// The product itself: U (prow x r, dense) is split into the panel buffer `upair`; the pair of M + G must be in place.
int r_pairs(StepCtx& s, int b, const dion_matrix* a, bool tr, const float* U, float* upair, float* out, const int* skip,
            GemmArgs* defer = nullptr, bool split_done = false) {   // defer: the product is handed back instead of launched
  dion_ctx* c = s.c;
  const i64 m = a->m, n = a->n, r = a->r;
  const i64 prow = tr ? n : m, qrow = tr ? m : n;
  __nv_bfloat16* uh = reinterpret_cast<__nv_bfloat16*>(upair);
  __nv_bfloat16* ul = uh + prow * r;
  if (!split_done) {      // (the step splits U for the whole chain beforehand)
    launch_pdl(k_split_bf16, dim3((unsigned)grid_for(c, prow * r / 8)), dim3(256), 0, s.st, U, r, prow, r, uh, ul, skip, (__half*)nullptr, 0.f);
    DION_CHECK_LAUNCH(c);
  }
  __nv_bfloat16* bh = reinterpret_cast<__nv_bfloat16*>(s.W(b, s.L.Bp));
  GemmArgs w = gemm_args();
  w.M = qrow; w.N = r; w.K = prow;
  w.ab16 = 1;
  w.A = (const float*)bh; w.A16lo = bh + m * n; w.a_si = tr ? n : 1; w.a_sk = tr ? 1 : n;
  w.B = (const float*)uh; w.B16lo = ul; w.b_sk = r; w.b_sn = 1;
  w.C = out; w.ldc = r; w.epi = EPI_STORE;
  w.skip_flag = skip;
  if (defer != nullptr) { *defer = w; return DION_OK; }
  return launch_gemm(s, w, b);
}

// The weight update X <- X - alpha F1 F2^T in fp32 mode on the tensor engine (F1: m x r with leading dimension
// ld1, F2: n x r with ld2; U Q^T, or Q U^T in the transposed form).  The update feeds nothing else, so its two
// factors are rounded to TF32 once (to nearest: unbiased) into `r1`, `r2` (scratch, dense) and the product takes
// one MMA per K step instead of three.  Returns false when the shape or the alignment does not qualify.
bool x_single_pass(const StepCtx& s, const dion_matrix* a, const float* F1, i64 ld1, const float* F2, i64 ld2) {
  const i64 m = a->m, n = a->n, r = a->r;
  return s.tensor && s.c->cfg.precision == DION_PREC_FP32 && m >= 128 && n >= 64 && r >= 64 && m % 4 == 0 &&
         n % 4 == 0 && r % 4 == 0 && !((uintptr_t)a->X & 15) && a->ldx % 4 == 0 && !((uintptr_t)F1 & 15) &&
         ld1 % 4 == 0 && !((uintptr_t)F2 & 15) && ld2 % 4 == 0;
}

// ... and with every dimension a multiple of 8 the rounded factors are IEEE half arrays instead: the same 11
// significant bits as TF32, read by one kind::f16 MMA per K step of 16 -- twice the MMA rate and half the operand
// bytes.  Both factors have unit-norm columns (U orthonormal, Q column-normalized), so their entries are at most 1;
// each is scaled by the power of two nearest the square root of its row count (entries around 1: far from half's
// subnormals, at most sqrt(2 rows) < 65504) and alpha takes the scales back exactly.
bool x_half(const dion_matrix* a) { return a->m % 8 == 0 && a->n % 8 == 0 && a->r % 8 == 0; }
float half_scale(i64 rows) { return exp2f(rintf(0.5f * log2f((float)rows))); }

// The error feedback M <- (M + G) - beta F1 F2^T in fp32 mode on the tensor engine (F1: m x r, F2: n x r; U R^T, or
// R U^T in the transposed form).  The product enters M scaled by beta = 1 - mu, so 16 significant bits in its factors
// are plenty (an error of ~1e-5 of the product, ~5e-7 of M): both factors are split once into bf16 pairs
// (hi, lo) in scratch (`p1`, `p2`: max(m,n) x r floats each) and the product takes three bf16 MMAs per K step, 1.3
// TF32 passes instead of three.  Otherwise the 3xTF32 / FMA product of the fp32 factors.
// sum32 != nullptr: M + G comes from scratch (C = sum32 - beta acc); else C = M + G - beta acc with the caller's G.
// ready1 / ready2: that factor's pair already sits in p1 / p2 (the step splits U for R).
bool ef_on_pairs(const StepCtx& s, const dion_matrix* a, const float* F1, i64 ld1, const float* F2, i64 ld2, const float* sum32) {
  const i64 m = a->m, n = a->n, r = a->r;
  return s.tensor && s.c->cfg.precision == DION_PREC_FP32 && m >= 128 && n >= 64 && r >= 64 && m % 8 == 0 &&
         n % 8 == 0 && r % 8 == 0 && !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 && !((uintptr_t)F1 & 15) &&
         ld1 % 4 == 0 && !((uintptr_t)F2 & 15) && ld2 % 4 == 0 &&
         (sum32 != nullptr || (!((uintptr_t)a->G & 15) && a->ldg % ((a->g_dtype == DION_BF16) ? 8 : 4) == 0));
}

int ef_update(StepCtx& s, int b, const dion_matrix* a, const float* F1, i64 ld1, const float* F2, i64 ld2, float* p1,
              float* p2, const float* sum32, const int* skip, bool ready1 = false, bool ready2 = false,
              GemmArgs* defer = nullptr) {
  dion_ctx* c = s.c;
  const i64 m = a->m, n = a->n, r = a->r;
  GemmArgs e = gemm_args();
  e.M = m; e.N = n; e.K = r;
  const bool pairs = ef_on_pairs(s, a, F1, ld1, F2, ld2, sum32);
  if (pairs) {
    __nv_bfloat16* h1 = reinterpret_cast<__nv_bfloat16*>(p1);
    __nv_bfloat16* l1 = h1 + m * r;
    __nv_bfloat16* h2 = reinterpret_cast<__nv_bfloat16*>(p2);
    __nv_bfloat16* l2 = h2 + n * r;
    if (!ready1) {
      launch_pdl(k_split_bf16, dim3((unsigned)grid_for(c, m * r / 8)), dim3(256), 0, s.st, F1, ld1, m, r, h1, l1, skip, (__half*)nullptr, 0.f);
      DION_CHECK_LAUNCH(c);
    }
    if (!ready2) {
      launch_pdl(k_split_bf16, dim3((unsigned)grid_for(c, n * r / 8)), dim3(256), 0, s.st, F2, ld2, n, r, h2, l2, skip, (__half*)nullptr, 0.f);
      DION_CHECK_LAUNCH(c);
    }
    e.ab16 = 1;
    e.A = (const float*)h1; e.A16lo = l1; e.a_si = r; e.a_sk = 1;
    e.B = (const float*)h2; e.B16lo = l2; e.b_sk = 1; e.b_sn = r;
  } else {
    e.A = F1; e.a_si = ld1; e.a_sk = 1;
    e.B = F2; e.b_sk = 1; e.b_sn = ld2;
  }
  e.C = (float*)a->M; e.ldc = a->ldm;
  if (sum32 != nullptr) { e.epi = EPI_C2_SUB; e.C2 = sum32; e.ldc2 = n; e.c2_mode = ADD_F32; }
  else { e.epi = EPI_ADD2_SUB; e.C2 = a->G; e.ldc2 = a->ldg; e.c2_mode = (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32; }
  e.alpha = 1.f - c->cfg.mu;
  e.skip_flag = skip;
  if (defer != nullptr) { *defer = e; return DION_OK; }
  return launch_gemm(s, e, b);
}

int x_update(StepCtx& s, int b, const dion_matrix* a, const float* F1, i64 ld1, const float* F2, i64 ld2, float* r1,
             float* r2, float alpha, const int* skip, const float* alpha_dev = nullptr, GemmArgs* defer = nullptr,
             bool rounded = false, float s1 = 0.f, float s2 = 0.f) {   // rounded: r1 and r2 already hold the rounded factors,
                                                                       // half arrays by the scales s1, s2 (0: half_scale's)
  dion_ctx* c = s.c;
  const i64 m = a->m, n = a->n, r = a->r;
  GemmArgs x = gemm_args();
  x.M = m; x.N = n; x.K = r;
  if (x_single_pass(s, a, F1, ld1, F2, ld2) && x_half(a)) {
    if (s1 == 0.f) s1 = half_scale(m);
    if (s2 == 0.f) s2 = half_scale(n);
    if (!rounded) {
      launch_pdl(k_round_f16, dim3((unsigned)grid_for(c, m * r / 8)), dim3(256), 0, s.st, F1, ld1, m, r, s1, reinterpret_cast<__half*>(r1), skip);
      DION_CHECK_LAUNCH(c);
      launch_pdl(k_round_f16, dim3((unsigned)grid_for(c, n * r / 8)), dim3(256), 0, s.st, F2, ld2, n, r, s2, reinterpret_cast<__half*>(r2), skip);
      DION_CHECK_LAUNCH(c);
    }
    x.ab16 = 1; x.f16 = 1;
    x.A = r1; x.a_si = r; x.a_sk = 1;
    x.B = r2; x.b_sk = 1; x.b_sn = r;
    alpha /= s1 * s2;       // (powers of two: exact)
  } else if (x_single_pass(s, a, F1, ld1, F2, ld2)) {
    if (!rounded) {
      launch_pdl(k_round_tf32, dim3((unsigned)grid_for(c, m * r / 4)), dim3(256), 0, s.st, F1, ld1, m, r, r1, skip);
      DION_CHECK_LAUNCH(c);
      launch_pdl(k_round_tf32, dim3((unsigned)grid_for(c, n * r / 4)), dim3(256), 0, s.st, F2, ld2, n, r, r2, skip);
      DION_CHECK_LAUNCH(c);
    }
    x.tf32x1 = 1;
    x.A = r1; x.a_si = r; x.a_sk = 1;
    x.B = r2; x.b_sk = 1; x.b_sn = r;
  } else {
    x.A = F1; x.a_si = ld1; x.a_sk = 1;
    x.B = F2; x.b_sk = 1; x.b_sn = ld2;
  }
  x.C = (float*)a->X; x.ldc = a->ldx; x.epi = EPI_SUB;
  x.alpha = alpha;
  x.alpha_dev = alpha_dev;      // graph replay: alpha = 1, the factor comes from the device scalar
  x.skip_flag = skip;
  if (defer != nullptr) { *defer = x; return DION_OK; }
  return launch_gemm(s, x, b);
}

// The launch chain of one Dion step (Algorithm 1 + 2) on `nb` matrices of identical
// (m, n, r), phase by phase.  Scratch must hold nb slices.
// x_scale != nullptr (graph capture, nb = 1, fp32 mode): the update's factor lr sqrt(m/n) is read from that device
// scalar and the step uses state slot `fixed_slot`.
int step_batch(dion_ctx* c, const dion_matrix* const* list, int nb, float lr, cudaStream_t st,
               const float* x_scale = nullptr, int fixed_slot = -1) {
  StepCtx s;
  const dion_matrix* a0 = list[0];
  DION_TRY(begin_step(c, a0, nb, st, &s, fixed_slot));
  const i64 m = a0->m, n = a0->n, r = a0->r;
  s.list = list;
  if (c->cfg.orth == DION_ORTH_RCQR) {
    const i64 panel_rows = a0->transposed ? n : m;
    for (int b = 0; b < nb; ++b) {
      const dion_matrix* a = list[b];
      if (a->sketch == nullptr || ((uintptr_t)a->sketch & 3)) return DION_ERR_INVALID;
      if (a->sketch_rows < r || a->sketch_rows > 2 * r || a->ld_sketch < panel_rows) return DION_ERR_SHAPE;
    }
  }

  // Standard form: the power iteration runs on B = M + G (panel P = B Q, m x r; Q is n x r).
  // Transposed form: it runs on B^T (panel P = B^T Q, n x r; Q is m x r), and the rank-r
  // products come out transposed: M <- B - (1 - mu) R U^T, X <- X - lr sqrt(m/n) Q U^T.
  const bool tr = a0->transposed != 0;
  const i64 prow = tr ? n : m;     // rows of the panel that is orthonormalized
  const i64 qrow = tr ? m : n;     // rows of R and Q
  const auto g_mode = [](const dion_matrix* a) { return (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32; };

  // bf16-operand mode on the tensor engine: bf16(M + G) is formed once per step and the four
  // products read bf16 arrays (B16, and the bf16 copies of Q, U, R) straight through TMA.
  bool d16 = s.tensor && c->cfg.precision == DION_PREC_BF16_OPERANDS && m % 8 == 0 && n % 8 == 0 && r % 8 == 0 &&
             m >= 128 && n >= 128 && r >= 64;
  for (int b = 0; b < nb && d16; ++b)
    if (((uintptr_t)list[b]->Q & 15) || (list[b]->ldq % 4)) d16 = false;
  auto bf = [&](int b, i64 off) { return reinterpret_cast<__nv_bfloat16*>(s.W(b, off)); };
  auto to_bf16 = [&](const float* src, i64 lds, i64 rows, i64 cols, __nv_bfloat16* out) -> int {
    launch_pdl(k_to_bf16, dim3((unsigned)(grid_for(c, rows * cols / 8))), dim3(256), 0, st, src, lds, rows, cols, out, nullptr);
    DION_CHECK_LAUNCH(c);
    return DION_OK;
  };

  // fp32 mode: M + G kept in scratch for P, R and the error feedback (see sum_in_scratch)
  const bool b32 = !d16 && s.tensor && s.L.B32 > 0;
  // ... R then runs on bf16 pairs of M + G and of U (three bf16 MMAs per K step: 1.3 TF32 passes instead of 3; the
  // product is accurate to ~1e-5, which is what Q <- ColNorm(R) and the error feedback need of it)
  const bool bpair = b32 && r_on_pairs(s, m, n, r);
  // ... and so does P where the orthonormalization is CholeskyQR2 and the matrix is large enough for the saving to
  // exceed the launches that stand by for the accurate product (see orthonormalize).  The rule looks at the matrix
  // alone, so that a grouped call computes what single calls compute.
  const bool ppair = bpair && (double)m * (double)n * (double)r >= P_PAIR_MIN_MNR &&
                     resolve_orth_for(c, r, (m < n) ? m : n, s.list != nullptr) == DION_ORTH_CHOLQR2;
  bool any_pair = false;
  const bool hstep = step_on_half_pairs(s, m, n, r, (m < n) ? m : n);

  // the large products: one GemmArgs per matrix, then one launch over the chain where that is possible
  std::vector<GemmArgs> group((size_t)nb);

  // P = (M + G) Q   (transposed form: (M + G)^T Q)
  const i64 pin_off = panel_offset(s, r, (m < n) ? m : n);
  bool q_copied = false;      // a dense copy of every Q of the chain sits in scratch (for the recomputation of P)
  {
  PhaseScope ps(c, st, DION_PHASE_P);
  // elementwise preparation for the whole chain: M + G (and its pair), the pair of Q where P takes pairs
  const float* srcs[MAX_CHAIN];
  i64 lds[MAX_CHAIN];
  if (hstep) DION_TRY(half_sum_chain(s, list, qrow, true, true));
  else if (b32) DION_TRY(form_sum_chain(s, list, bpair, true));
  else if (!d16) DION_TRY(clear_slots(s));
  const bool phalf = b32 && s.L.Bh > 0;
  bool p_half_ready = false;
  if (phalf) {      // the scaled half pairs of M + G and of Q, for the whole chain
    bool all_ok = true;
    for (int b = 0; b < nb; ++b) {
      all_ok = all_ok && !((uintptr_t)list[b]->Q & 15) && list[b]->ldq % 4 == 0 && list[b]->ldq == list[0]->ldq;
      srcs[b] = (const float*)list[b]->Q;
    }
    if (all_ok && nb <= GEMM_TAB_MAX) {
      i64 parts = (m * n / 4 + 2047) / 2048;
      if (parts > AMAX_PARTS) parts = AMAX_PARTS;
      __half* bh = reinterpret_cast<__half*>(s.ws + s.L.Bh);
      launch_pdl(k_absmax_partial, dim3((unsigned)parts, (unsigned)nb), dim3(256), 0, st, (const float*)(s.ws + s.L.B32), n, m, n,
                 s.ws + s.L.pmax, s.wstride, (const int*)nullptr, (i64)0);
      DION_CHECK_LAUNCH(c);
      launch_pdl(k_split_f16_scaled, dim3((unsigned)grid_for(c, m * n / 8, nb), (unsigned)nb), dim3(256), 0, st,
                 (const float*)(s.ws + s.L.B32), n, m, n, (const float*)(s.ws + s.L.pmax), (int)parts, bh, bh + m * n,
                 s.ws + s.L.pmax + AMAX_PARTS, s.wstride, (const int*)nullptr, (i64)0, ldexpf(1.f, -13), (const float*)nullptr, (float*)nullptr, (int*)nullptr, 0, 0, 0);
      DION_CHECK_LAUNCH(c);
      ChainPtrs t;
      for (int b = 0; b < nb; ++b) t.p[b] = srcs[b];
      __half* qh = reinterpret_cast<__half*>(s.ws + s.L.S16);
      launch_pdl(k_split_f16_fixed, dim3((unsigned)grid_for(c, qrow * r / 8, nb), (unsigned)nb), dim3(256), 0, st, t, list[0]->ldq, qrow, r,
                 ldexpf(1.f, 13), qh, qh + qrow * r, s.wstride, (i64)0, (const int*)nullptr, (i64)0, (const int*)nullptr, (__half*)nullptr);
      DION_CHECK_LAUNCH(c);
      p_half_ready = true;
    }
  }
  bool q_split = false;
  if (b32 && ppair) {
    bool all_ok = true;
    for (int b = 0; b < nb; ++b) {
      all_ok = all_ok && !((uintptr_t)list[b]->Q & 15) && list[b]->ldq % 4 == 0;
      srcs[b] = (const float*)list[b]->Q; lds[b] = list[b]->ldq;
    }
    if (all_ok) { DION_TRY(split_chain(s, srcs, lds, qrow, r, s.L.S16, nullptr, s.L.Qc > 0 ? s.L.Qc : -1, &q_copied)); q_split = true; }
  }
  // The other products of a chain read the callers' Q; dense copies of them in the scratch slices (S16, free until the
  // error feedback) let one launch take the whole chain: 84 matrices of up to 768 x 3072 at r = 192 went through 147
  // launches of a few tiles each, 1670 us.
  bool q_dense = false;
  if (nb > 1 && nb <= GEMM_TAB_MAX && c->chain_batch && b32 && !ppair && !hstep && !p_half_ready && r % 4 == 0) {
    bool all_ok = true;
    for (int b = 0; b < nb; ++b) {
      all_ok = all_ok && !((uintptr_t)list[b]->Q & 15) && list[b]->ldq == list[0]->ldq && list[b]->ldq % 4 == 0;
      srcs[b] = (const float*)list[b]->Q;
    }
    if (all_ok) {
      ChainPtrs t;
      for (int b = 0; b < nb; ++b) t.p[b] = srcs[b];
      launch_pdl(k_copy_chain, dim3((unsigned)grid_for(c, qrow * r / 4, nb), (unsigned)nb), dim3(256), 0, st, t, list[0]->ldq, qrow, r, s.ws + s.L.S16, s.wstride);
      DION_CHECK_LAUNCH(c);
      q_dense = true;
    }
  }
  for (int b = 0; b < nb; ++b) {
    const dion_matrix* a = list[b];
    GemmArgs p = gemm_args();
    p.M = prow; p.N = r; p.K = qrow;
    if (d16) {
      const bool vec = !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 &&
                       (a->g_dtype == DION_BF16 ? (!((uintptr_t)a->G & 15) && a->ldg % 8 == 0)
                                                : (!((uintptr_t)a->G & 15) && a->ldg % 4 == 0));
      const int grid = grid_for(c, m * n / 8);
      if (vec) launch_pdl(k_form_b16<true>, grid, dim3(256), 0, st, (const float*)a->M, a->ldm, a->G, a->ldg, g_mode(a), m, n, bf(b, s.L.B16), s.OS(b));
      else launch_pdl(k_form_b16<false>, grid, dim3(256), 0, st, (const float*)a->M, a->ldm, a->G, a->ldg, g_mode(a), m, n, bf(b, s.L.B16), s.OS(b));
      DION_CHECK_LAUNCH(c);
      DION_TRY(to_bf16((const float*)a->Q, a->ldq, qrow, r, bf(b, s.L.Q16)));
      p.ab16 = 1;
      p.A = (const float*)bf(b, s.L.B16); p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      p.B = (const float*)bf(b, s.L.Q16); p.b_sk = r; p.b_sn = 1;
    } else if (b32 && ppair && !((uintptr_t)a->Q & 15) && a->ldq % 4 == 0) {
      __nv_bfloat16* qh = reinterpret_cast<__nv_bfloat16*>(s.W(b, s.L.S16));
      __nv_bfloat16* ql = qh + qrow * r;
      if (!q_split) {
        launch_pdl(k_split_bf16, dim3((unsigned)grid_for(c, qrow * r / 8)), dim3(256), 0, st, (const float*)a->Q, a->ldq, qrow, r, qh, ql,
                   (const int*)nullptr, (__half*)nullptr, 0.f);
        DION_CHECK_LAUNCH(c);
      }
      __nv_bfloat16* bh = reinterpret_cast<__nv_bfloat16*>(s.W(b, s.L.Bp));
      p.ab16 = 1;
      p.A = (const float*)bh; p.A16lo = bh + m * n; p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      p.B = (const float*)qh; p.B16lo = ql; p.b_sk = r; p.b_sn = 1;
      any_pair = true;
    } else if (hstep) {
      __half* bh = reinterpret_cast<__half*>(s.W(b, s.L.Bp));
      __half* qh = reinterpret_cast<__half*>(s.W(b, s.L.S16));
      p.ab16 = 1; p.f16 = 1;
      p.A = (const float*)bh; p.A16lo = bh + m * n; p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      p.B = (const float*)qh; p.B16lo = qh + qrow * r; p.b_sk = r; p.b_sn = 1;
      p.alpha_dev = s.W(b, s.L.lz) + HS_P;
      p.skip_flag = s.OS(b) + OS_P32;
    } else if (p_half_ready) {
      __half* bh = reinterpret_cast<__half*>(s.W(b, s.L.Bh));
      __half* qh = reinterpret_cast<__half*>(s.W(b, s.L.S16));
      p.ab16 = 1; p.f16 = 1;
      p.A = (const float*)bh; p.A16lo = bh + m * n; p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      p.B = (const float*)qh; p.B16lo = qh + qrow * r; p.b_sk = r; p.b_sn = 1;
      p.alpha_dev = s.W(b, s.L.pmax) + AMAX_PARTS;
    } else if (b32) {
      p.A = s.W(b, s.L.B32); p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      if (q_dense) { p.B = s.W(b, s.L.S16); p.b_sk = r; p.b_sn = 1; }
      else { p.B = (const float*)a->Q; p.b_sk = a->ldq; p.b_sn = 1; }
    } else {
      p.A = (const float*)a->M; p.a_si = tr ? 1 : a->ldm; p.a_sk = tr ? a->ldm : 1;
      p.A2 = a->G; p.a2_si = tr ? 1 : a->ldg; p.a2_sk = tr ? a->ldg : 1; p.a2_mode = g_mode(a);
      p.B = (const float*)a->Q; p.b_sk = a->ldq; p.b_sn = 1;
    }
    p.C = s.W(b, pin_off); p.ldc = r; p.epi = EPI_STORE;
    // an ill-conditioned panel amplifies the error of P: use the accurate product there
    p.precise = (!d16 && resolve_orth(c, r, (m < n) ? m : n) == DION_ORTH_SHIFTED3) ? 1 : 0;
    group[b] = p;
  }
  DION_TRY(launch_gemm_group(s, group));
  if (hstep) {
    for (int b = 0; b < nb; ++b) group[b] = wide_p(s, b, list[b], tr, s.W(b, pin_off));
    s.no_split = qrow <= WIDE_P_WHOLE_K;
    const int rc_wide = launch_gemm_group(s, group);
    s.no_split = false;
    DION_TRY(rc_wide);
  }
  }

  // U = Orthonormalize(P)
  i64 U_off = 0;
  // (U as a half array for the weight update, made beside U's pair: behind Q's in the panel's save buffer, free by then;
  // a rounding of its own read U again: 4096 x 4096, r = 1024, 619 -> 616 us)
  const i64 u_one = s.L.Psave + ((m > n) ? m : n) * r / 2;
  bool u_one_made = hstep;
  {
  PhaseScope ps(c, st, DION_PHASE_ORTH);
  const std::function<int()> redo = [&]() -> int {
    std::vector<GemmArgs> again((size_t)nb);
    for (int b = 0; b < nb; ++b) {
      const dion_matrix* a = list[b];
      GemmArgs p = gemm_args();
      p.M = prow; p.N = r; p.K = qrow;
      p.A = s.W(b, s.L.B32); p.a_si = tr ? 1 : n; p.a_sk = tr ? n : 1;
      if (q_copied) { p.B = s.W(b, s.L.Qc); p.b_sk = r; p.b_sn = 1; }     // (the same values: one launch over the chain)
      else { p.B = (const float*)a->Q; p.b_sk = a->ldq; p.b_sn = 1; }
      p.C = s.W(b, pin_off); p.ldc = r; p.epi = EPI_STORE;
      p.skip_flag = s.OS(b) + OS_DONE;
      again[b] = p;
    }
    return launch_gemm_group(s, again);
  };
  s.in_orth = true;
  s.redo_p = any_pair ? &redo : nullptr;
  const int rc_orth = orthonormalize(s, prow, r, (m < n) ? m : n, pin_off, &U_off);
  s.redo_p = nullptr;
  s.in_orth = false;
  DION_TRY(rc_orth);
  }

  // R = (M + G)^T U   (transposed form: (M + G) U)
  {
  PhaseScope ps(c, st, DION_PHASE_R);
  const i64 other_off = (U_off == s.L.P0) ? s.L.P1 : s.L.P0;
  if (!d16 && bpair) {   // U as a pair in the other panel buffer, for the whole chain
    const float* srcs[MAX_CHAIN];
    i64 lds[MAX_CHAIN];
    for (int b = 0; b < nb; ++b) { srcs[b] = s.W(b, U_off); lds[b] = r; }
    if (hstep) DION_TRY(split_half_chain(s, srcs, r, prow, r, other_off, HS_U_BITS, s.os + OS_FAIL, u_one));
    else {
      u_one_made = s.L.Psave > 0 && x_half(a0);
      for (int b = 0; b < nb; ++b) {
        const float *Uf = srcs[b], *Qf = (const float*)list[b]->Q;
        u_one_made = u_one_made && (tr ? x_single_pass(s, list[b], Qf, list[b]->ldq, Uf, r) : x_single_pass(s, list[b], Uf, r, Qf, list[b]->ldq));
      }
      DION_TRY(split_chain(s, srcs, lds, prow, r, other_off, s.os + OS_FAIL, -1, nullptr, u_one_made ? u_one : -1, half_scale(prow)));
    }
  }
  for (int b = 0; b < nb; ++b) {
    const dion_matrix* a = list[b];
    GemmArgs w = gemm_args();
    w.M = qrow; w.N = r; w.K = prow;
    if (d16) {
      DION_TRY(to_bf16(s.W(b, U_off), r, prow, r, bf(b, s.L.U16)));
      w.ab16 = 1;
      w.A = (const float*)bf(b, s.L.B16); w.a_si = tr ? n : 1; w.a_sk = tr ? 1 : n;
      w.B = (const float*)bf(b, s.L.U16); w.b_sk = r; w.b_sn = 1;
    } else if (bpair) {
      // U as a bf16 pair in the other panel buffer (the error feedback reuses it)
      DION_TRY(r_pairs(s, b, a, tr, s.W(b, U_off), s.W(b, other_off), s.W(b, s.L.R), s.OS(b) + OS_FAIL, &group[b], true));
      if (hstep) { group[b].f16 = 1; group[b].wide_flag = s.OS(b) + OS_WIDE; group[b].alpha_dev = s.W(b, s.L.lz) + HS_R; }      // (the same place and layout)
      continue;
    } else if (b32) {
      w.A = s.W(b, s.L.B32); w.a_si = tr ? n : 1; w.a_sk = tr ? 1 : n;
      w.B = s.W(b, U_off); w.b_sk = r; w.b_sn = 1;
    } else {
      w.A = (const float*)a->M; w.a_si = tr ? a->ldm : 1; w.a_sk = tr ? 1 : a->ldm;
      w.A2 = a->G; w.a2_si = tr ? a->ldg : 1; w.a2_sk = tr ? 1 : a->ldg; w.a2_mode = g_mode(a);
      w.B = s.W(b, U_off); w.b_sk = r; w.b_sn = 1;
    }
    w.C = s.W(b, s.L.R); w.ldc = r; w.epi = EPI_STORE;
    group[b] = w;
  }
  DION_TRY(launch_gemm_group(s, group));
  }

  // Q <- ColNorm(R), and in the same pass the operands of the two rank-r updates that R and Q become (wherever every matrix of
  // the chain takes them in that form): R's pair in S16, Q rounded in the save buffer of the panel, which nothing reads any more.
  int cn_kind = 0;
  {
  PhaseScope ps(c, st, DION_PHASE_COLNORM);
  if (d16) {
    cn_kind = CN_ONE;
  } else if (hstep) {
    cn_kind = CN_HALF;
  } else if (s.L.Psave > 0 && x_half(a0)) {
    bool all = true;
    for (int b = 0; b < nb; ++b) {
      const dion_matrix* a = list[b];
      const float* sum32 = b32 ? s.W(b, s.L.B32) : nullptr;
      const float *Rf = s.W(b, s.L.R), *Uf = s.W(b, U_off), *Qf = (const float*)a->Q;
      all = all && (tr ? ef_on_pairs(s, a, Rf, r, Uf, r, sum32) && x_single_pass(s, a, Qf, a->ldq, Uf, r)
                       : ef_on_pairs(s, a, Uf, r, Rf, r, sum32) && x_single_pass(s, a, Uf, r, Qf, a->ldq));
    }
    if (all) cn_kind = CN_BF16;
  }
  DION_TRY(colnorm_chain(s, list, qrow, r, cn_kind, cn_kind == CN_ONE ? s.L.Q16 : s.L.Psave, half_scale(qrow), cn_kind == CN_ONE ? s.L.R16 : s.L.S16));
  }

  // On the FMA engine the two rank-r updates, which share nothing that either writes, are one launch (small or ragged matrices:
  // each is a few tens of blocks; 1001 x 333, r = 83: 8 + 11 us one after the other; the step 129.7 -> 119.1 us).
  auto on_simt = [&](const GemmArgs& g) {
    return c->cfg.engine != DION_ENGINE_TENSOR && !g.ab16 && !g.tf32x1 && !(s.tensor && umma_shape_ok(g, c->cfg.precision));
  };
  bool two = false;
  GemmArgs ef_args;
  // Under graph capture (small matrices: a few CTAs each) the two rank-r updates, which share nothing that either writes, are two
  // branches of the graph -- where the update of X has nothing left to prepare (its rounded factors would go where the error
  // feedback's lie).  256 x 512, r = 64, replayed: 77.8 -> 72.4 us.
  const bool fork = x_scale != nullptr && c->side != nullptr && cn_kind != 0 && u_one_made;
  auto order = [&](cudaStream_t from, cudaStream_t to) -> int {      // what follows on `to` waits for what `from` has been given
    cudaEvent_t e = c->side_ev[c->side_cursor];
    c->side_cursor = (c->side_cursor + 1) % 32;
    return cudaEventRecord(e, from) == cudaSuccess && cudaStreamWaitEvent(to, e, 0) == cudaSuccess ? DION_OK : DION_ERR_CUDA;
  };
  if (fork) DION_TRY(order(st, c->side));

  // M <- (M + G) - (1 - mu) U R^T   (transposed form: R U^T)
  {
  PhaseScope ps(c, st, DION_PHASE_EF);
  const i64 other_off = (U_off == s.L.P0) ? s.L.P1 : s.L.P0;
  bool ef_split = false;      // the factors' pairs are made for the whole chain when every matrix takes pairs
  if (!d16) {
    const float* srcs[MAX_CHAIN];
    i64 lds[MAX_CHAIN];
    bool all_pairs = true;
    for (int b = 0; b < nb; ++b) {
      const float* sum32 = b32 ? s.W(b, s.L.B32) : nullptr;
      all_pairs = all_pairs && (tr ? ef_on_pairs(s, list[b], s.W(b, s.L.R), r, s.W(b, U_off), r, sum32)
                                   : ef_on_pairs(s, list[b], s.W(b, U_off), r, s.W(b, s.L.R), r, sum32));
    }
    if (all_pairs || cn_kind != 0) {
      for (int b = 0; b < nb; ++b) { srcs[b] = s.W(b, s.L.R); lds[b] = r; }
      if (cn_kind == 0) DION_TRY(split_chain(s, srcs, lds, qrow, r, s.L.S16, s.os + OS_FAIL));
      if (!bpair) {
        for (int b = 0; b < nb; ++b) srcs[b] = s.W(b, U_off);
        DION_TRY(split_chain(s, srcs, lds, prow, r, other_off, s.os + OS_FAIL));
      }
      ef_split = true;
    }
  }
  for (int b = 0; b < nb; ++b) {
    const dion_matrix* a = list[b];
    if (d16) {
      GemmArgs e = gemm_args();
      e.M = m; e.N = n; e.K = r;
      e.ab16 = 1;
      e.A = (const float*)bf(b, tr ? s.L.R16 : s.L.U16); e.a_si = r; e.a_sk = 1;
      e.B = (const float*)bf(b, tr ? s.L.U16 : s.L.R16); e.b_sk = 1; e.b_sn = r;
      e.C = (float*)a->M; e.ldc = a->ldm;
      e.epi = EPI_ADD2_SUB; e.C2 = a->G; e.ldc2 = a->ldg; e.c2_mode = g_mode(a);
      e.alpha = 1.f - c->cfg.mu;
      e.skip_flag = s.OS(b) + OS_FAIL;
      group[b] = e;
      continue;
    }
    // the bf16 pairs of the two factors go to the other panel buffer and to their own buffer
    float* other = s.W(b, U_off == s.L.P0 ? s.L.P1 : s.L.P0);
    float* sbuf = s.W(b, s.L.S16);
    const float* Uf = s.W(b, U_off);
    const float* Rf = s.W(b, s.L.R);
    const float* sum32 = b32 ? s.W(b, s.L.B32) : nullptr;
    if (tr) DION_TRY(ef_update(s, b, a, Rf, r, Uf, r, sbuf, other, sum32, s.OS(b) + OS_FAIL, ef_split, bpair || ef_split, &group[b]));
    else DION_TRY(ef_update(s, b, a, Uf, r, Rf, r, other, sbuf, sum32, s.OS(b) + OS_FAIL, bpair || ef_split, ef_split, &group[b]));
    if (hstep && group[b].ab16) { group[b].f16 = 1; group[b].wide_flag = s.OS(b) + OS_WIDE; group[b].alpha_dev = s.W(b, s.L.lz) + HS_EF; }
  }
  two = nb == 1 && !c->prof_on && on_simt(group[0]);
  if (two) ef_args = group[0];
  else DION_TRY(launch_gemm_group(s, group));
  }

  // X <- X - lr sqrt(m/n) U Q^T   (transposed form: Q U^T)
  {
  PhaseScope ps(c, st, DION_PHASE_X);
  const float x_alpha = (x_scale != nullptr) ? 1.f : lr * sqrtf((float)((double)m / (double)n));
  const i64 other_off = (U_off == s.L.P0) ? s.L.P1 : s.L.P0;
  if (fork) s.st = c->side;
  float u_half = 0.f;         // scale of U's half array when it is not half_scale's
  bool x_rounded = false;     // the rounded factors are made for the whole chain when every matrix takes the single pass
  if (!d16) {
    const float* srcs[MAX_CHAIN];
    i64 lds[MAX_CHAIN];
    bool all_one = true;
    for (int b = 0; b < nb; ++b) {
      const dion_matrix* a = list[b];
      all_one = all_one && (tr ? x_single_pass(s, a, (const float*)a->Q, a->ldq, s.W(b, U_off), r)
                               : x_single_pass(s, a, s.W(b, U_off), r, (const float*)a->Q, a->ldq));
    }
    if (all_one) {
      for (int b = 0; b < nb; ++b) { srcs[b] = s.W(b, U_off); lds[b] = r; }
      const bool half = x_half(a0);
      if (u_one_made && half) u_half = hstep ? ldexpf(1.f, HS_U_BITS) : half_scale(prow);      // (made beside U's pair)
      else DION_TRY(round_chain(s, srcs, lds, prow, r, other_off, s.os + OS_FAIL, half ? half_scale(prow) : 0.f));
      if (cn_kind == 0) {
        for (int b = 0; b < nb; ++b) { srcs[b] = (const float*)list[b]->Q; lds[b] = list[b]->ldq; }
        DION_TRY(round_chain(s, srcs, lds, qrow, r, s.L.R, s.os + OS_FAIL, half ? half_scale(qrow) : 0.f));
      }
      x_rounded = true;
    }
  }
  for (int b = 0; b < nb; ++b) {
    const dion_matrix* a = list[b];
    if (d16) {
      GemmArgs x = gemm_args();
      x.M = m; x.N = n; x.K = r;
      x.ab16 = 1;
      x.A = (const float*)bf(b, tr ? s.L.Q16 : s.L.U16); x.a_si = r; x.a_sk = 1;
      x.B = (const float*)bf(b, tr ? s.L.U16 : s.L.Q16); x.b_sk = 1; x.b_sn = r;
      x.C = (float*)a->X; x.ldc = a->ldx; x.epi = EPI_SUB;
      x.alpha = x_alpha;
      x.skip_flag = s.OS(b) + OS_FAIL;
      group[b] = x;
      continue;
    }
    // the rounded copies of the single-pass form: in the other panel buffer, and where the normalization put Q's or in R's (free)
    float* other = s.W(b, u_half > 0.f ? u_one : U_off == s.L.P0 ? s.L.P1 : s.L.P0);
    float* rbuf = s.W(b, cn_kind != 0 && x_rounded ? s.L.Psave : s.L.R);
    const float* Uf = s.W(b, U_off);
    const float* Qf = (const float*)a->Q;
    if (tr) DION_TRY(x_update(s, b, a, Qf, a->ldq, Uf, r, rbuf, other, x_alpha, s.OS(b) + OS_FAIL, x_scale, &group[b], x_rounded, 0.f, u_half));
    else DION_TRY(x_update(s, b, a, Uf, r, Qf, a->ldq, other, rbuf, x_alpha, s.OS(b) + OS_FAIL, x_scale, &group[b], x_rounded, u_half, 0.f));
  }
  if (two && on_simt(group[0])) DION_TRY(launch_gemm_simt_two(c, ef_args, group[0], s.st));
  else {
    if (two) DION_TRY(launch_gemm(s, ef_args, 0));
    DION_TRY(launch_gemm_group(s, group));
  }
  s.st = st;
  if (fork) DION_TRY(order(c->side, st));
  }
  return DION_OK;
}

int step_one(dion_ctx* c, const dion_matrix* a, float lr, cudaStream_t st) {
  return step_batch(c, &a, 1, lr, st);
}

// ---- graph replay of launch-bound steps ----------------------------------------------------------------

__global__ void k_set_scalar(float* dst, float v) { *dst = v; }

void graphs_clear(dion_ctx* c) {
  for (auto& g : c->graphs) cudaGraphExecDestroy(g.exec);
  c->graphs.clear();
}

bool same_matrix(const dion_matrix& x, const dion_matrix& y) {
  return x.m == y.m && x.n == y.n && x.r == y.r && x.X == y.X && x.ldx == y.ldx && x.M == y.M && x.ldm == y.ldm &&
         x.G == y.G && x.ldg == y.ldg && x.g_dtype == y.g_dtype && x.Q == y.Q && x.ldq == y.ldq &&
         x.colnorm_out == y.colnorm_out && x.transposed == y.transposed && x.sketch == y.sketch &&
         x.sketch_rows == y.sketch_rows && x.ld_sketch == y.ld_sketch;
}

// A step on a small matrix is a chain of 12 to 30 launches that take longer to issue than to run.  Such steps are
// captured once (on the context's own stream: the caller's may be the legacy stream, which cannot capture) and
// replayed as one graph launch into the caller's stream.
bool graph_eligible(const dion_ctx* c, const dion_matrix* a) {
  return c->graphs_on && !c->prof_on && c->cfg.precision == DION_PREC_FP32 && c->cfg.engine != DION_ENGINE_SIMT &&
         a->m * a->n <= GRAPH_MAX_ELEMS && a->r <= NBO_COLS && a->m >= 128 && a->n >= 64 && a->r >= 64 && a->m % 4 == 0 &&
         a->n % 4 == 0 && a->r % 4 == 0 && !((uintptr_t)a->X & 15) && a->ldx % 4 == 0;     // (the X update must take the tensor engine)
}

// Returns DION_OK when the step was launched as a graph, 1 when the caller should launch it plainly.
int step_graph(dion_ctx* c, const dion_matrix* a, float lr, cudaStream_t st) {
  dion_ctx::GraphEntry* e = nullptr;
  for (auto& g : c->graphs)
    if (same_matrix(g.key, *a)) { e = &g; break; }
  if (e == nullptr) {
    int index = -1;
    if ((int)c->graphs.size() < MAX_GRAPHS) {
      index = (int)c->graphs.size();
    } else {      // evict the least recently used one (its kernels are ordered before ours only on its own stream: wait)
      size_t lru = 0;
      for (size_t i = 1; i < c->graphs.size(); ++i)
        if (c->graphs[i].last_use < c->graphs[lru].last_use) lru = i;
      if (cudaDeviceSynchronize() != cudaSuccess) return DION_ERR_CUDA;
      cudaGraphExecDestroy(c->graphs[lru].exec);
      index = c->graphs[lru].index;
      c->graphs.erase(c->graphs.begin() + (long)lru);
    }
    const int64_t l0 = c->launches;
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(c->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { cudaGetLastError(); return 1; }
    const int rc = step_batch(c, &a, 1, lr, c->cap, c->graph_scalars + index, MAX_FLAG_SLOTS - MAX_GRAPHS + index);
    const cudaError_t ce = cudaStreamEndCapture(c->cap, &graph);
    const int64_t nl = c->launches - l0;
    c->launches = l0;
    if (rc != DION_OK || ce != cudaSuccess || graph == nullptr) {
      cudaGetLastError();
      if (graph != nullptr) cudaGraphDestroy(graph);
      c->graphs_on = false;      // this chain does not capture here: plain launches from now on
      return 1;
    }
    cudaGraphExec_t exec = nullptr;
    const cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess || exec == nullptr) { cudaGetLastError(); c->graphs_on = false; return 1; }
    c->graphs.push_back({*a, exec, nl, index, 0, NAN, false});
    e = &c->graphs.back();
  }
  e->last_use = ++c->graph_clock;
  // The scalar is written when the rate changed (a launch of its own, 2 us).  What a stream that is being captured is given has not
  // run and may run at any time later: nothing is concluded from it, and from then on every call writes.
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &capturing) != cudaSuccess) { cudaGetLastError(); capturing = cudaStreamCaptureStatusActive; }
  if (capturing != cudaStreamCaptureStatusNone) e->recorded = true;
  const float scale = lr * sqrtf((float)((double)a->m / (double)a->n));
  const bool written = !e->recorded && e->scale == scale;
  e->scale = NAN;
  if (!written) {
    k_set_scalar<<<1, 1, 0, st>>>(c->graph_scalars + e->index, scale);
    if (cudaGetLastError() != cudaSuccess) return DION_ERR_CUDA;
    c->launches++;
  }
  if (cudaGraphLaunch(e->exec, st) != cudaSuccess) { cudaGetLastError(); return DION_ERR_CUDA; }
  e->scale = scale;
  c->launches += e->launches;
  return DION_OK;
}

// Lazy-Dion on scaled half pairs (fp32 mode on the tensor engine; the shapes that keep M + G in scratch): M + G is formed once
// per call, in fp32 for the error feedback and as a half pair for the products that read it, and every product takes three
// kind::f16 MMAs per K step on pairs -- the 22 significant bits of the 3xTF32 products it replaces at twice their rate,
// through the kernels with the deeper epilogue (4096^2, r = 256: W 128 -> 35 us + 50 of preparation, error feedback 141 -> 36,
// weight update 85 -> 28).
bool lazy_on_pairs(const StepCtx& s, const dion_matrix* a) {
  return s.tensor && s.L.B32 > 0 && s.L.Bp > 0 && a->r % 8 == 0 && a->m % 8 == 0 && a->n % 8 == 0 && a->m * a->n * a->r >= LAZY_PAIR_MIN_MNR &&
         !((uintptr_t)a->X & 15) && a->ldx % 4 == 0 && !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 && !((uintptr_t)a->Q & 15) && a->ldq % 4 == 0;
}

//
// Where the ranges of M + G, Q or T are too wide for that (k_form_sum_amax), the 3xTF32 product of the fp32 operands takes its
// place: every product is two launches, of which the state slot skips one.
int lazy_pairs(StepCtx& s, const dion_matrix* a, float lr, int refresh) {
  dion_ctx* c = s.c;
  cudaStream_t st = s.st;
  const i64 m = a->m, n = a->n, r = a->r;
  float* sc = s.ws + s.L.lz;      // HS_*
  float* R = s.ws + s.L.R;
  float* sum = s.ws + s.L.B32;
  const float* Q = (const float*)a->Q;
  auto halves = [&](i64 off) { return reinterpret_cast<__half*>(s.ws + off); };
  // the pair of a rows x cols array into scratch at `off`; slot: the scale factor of its product with M + G, own: of itself
  // alone; the flags of the products that read it
  auto pair_of = [&](const float* src, i64 ld, i64 rows, i64 cols, i64 off, int slot, int own, int use32, int usehalf) -> int {
    i64 nparts = (rows * cols / 4 + 2047) / 2048;
    if (nparts > AMAX_PARTS) nparts = AMAX_PARTS;
    float* pm = s.ws + s.L.part;      // (read before the next product writes its partial sums there)
    ChainPtrs t;
    t.p[0] = src;
    launch_pdl(k_range_partial, dim3((unsigned)nparts), dim3(256), 0, st, t, ld, rows, rows, cols, pm, (i64)0, (const int*)nullptr, (i64)0, (int*)nullptr);
    DION_CHECK_LAUNCH(c);
    launch_pdl(k_split_f16_scaled, dim3((unsigned)grid_for(c, rows * cols / 8)), dim3(256), 0, st, src, ld, rows, cols, (const float*)pm, (int)nparts,
               halves(off), halves(off) + rows * cols, sc + slot, (i64)0, (const int*)nullptr, (i64)0, ldexpf(1.f, HS_U_BITS),
               (const float*)(sc + HS_R), own >= 0 ? sc + own : (float*)nullptr, s.os, (int)OS_P32, use32, usehalf);
    DION_CHECK_LAUNCH(c);
    return DION_OK;
  };
  // a product: on the pairs at a_off and b_off, or of A and B (the same shapes, leading dimensions lda and ldb; ta, tb: transposed)
  auto product = [&](GemmArgs g, i64 a_off, const float* A, i64 lda, bool ta, i64 b_off, const float* B, i64 ldb, bool tb, int slot, float half_alpha,
                     int use32, int usehalf) -> int {
    const i64 ac = ta ? g.M : g.K, bc = tb ? g.K : g.N;      // columns of the arrays
    GemmArgs h = g;
    h.ab16 = 1; h.f16 = 1;
    h.A = (const float*)halves(a_off); h.A16lo = halves(a_off) + g.M * g.K; h.a_si = ta ? 1 : ac; h.a_sk = ta ? ac : 1;
    h.B = (const float*)halves(b_off); h.B16lo = halves(b_off) + g.K * g.N; h.b_sk = tb ? 1 : bc; h.b_sn = tb ? bc : 1;
    h.alpha = g.alpha * half_alpha; h.alpha_dev = sc + slot;
    h.skip_flag = s.os + use32;
    DION_TRY(launch_gemm(s, h));
    g.A = A; g.a_si = ta ? 1 : lda; g.a_sk = ta ? lda : 1;
    g.B = B; g.b_sk = tb ? 1 : ldb; g.b_sn = tb ? ldb : 1;
    g.skip_flag = s.os + usehalf;
    if (g.epi == EPI_STORE) g.precise = 1;
    return launch_gemm(s, g);
  };
  auto shape = [&](i64 M_, i64 N_, i64 K_, float* C, i64 ldc, int epi) {
    GemmArgs g = gemm_args();
    g.M = M_; g.N = N_; g.K = K_; g.C = C; g.ldc = ldc; g.epi = epi;
    return g;
  };
  DION_TRY(half_sum_chain(s, &a, n, true, true));      // M + G, its pair and Q's
  if (refresh) {
    PhaseScope ps_orth(c, st, DION_PHASE_ORTH);
    // T = (M + G) Q  (m x r), Z = (M + G)^T T (n x r), Q <- Orthonormalize(Z)
    const int precise = (resolve_orth(c, r, (m < n) ? m : n) == DION_ORTH_SHIFTED3) ? 1 : 0;
    GemmArgs t = shape(m, r, n, R, r, EPI_STORE);
    t.precise = precise;
    DION_TRY(product(t, s.L.Bp, sum, n, false, s.L.S16, Q, a->ldq, false, HS_P, 1.f, OS_P32, OS_PHALF));
    DION_TRY(pair_of(R, r, m, r, s.L.P1, HS_T, -1, OS_USE32, OS_USEHALF));
    const i64 pin_off = panel_offset(s, r, (m < n) ? m : n);
    GemmArgs z = shape(n, r, m, s.ws + pin_off, r, EPI_STORE);
    z.precise = precise;
    DION_TRY(product(z, s.L.Bp, sum, n, true, s.L.P1, R, r, false, HS_T, 1.f, OS_USE32, OS_USEHALF));
    i64 V_off = 0;
    s.in_orth = true;
    const int rc_orth = orthonormalize(s, n, r, (m < n) ? m : n, pin_off, &V_off);
    s.in_orth = false;
    DION_TRY(rc_orth);
    launch_pdl(k_copy_panel, dim3((unsigned)grid_for(c, n * r)), dim3(256), 0, st, (const float*)(s.ws + V_off), r, (float*)a->Q, a->ldq, n, r,
               (const int*)s.flag, (const int*)nullptr, (i64)0, -1);
    DION_CHECK_LAUNCH(c);
  }
  {   // W = (M + G) Q
  PhaseScope ps(c, st, DION_PHASE_P);
  if (refresh) DION_TRY(pair_of(Q, a->ldq, n, r, s.L.S16, HS_P, HS_Q, OS_P32, OS_PHALF));
  DION_TRY(product(shape(m, r, n, R, r, EPI_STORE), s.L.Bp, sum, n, false, s.L.S16, Q, a->ldq, false, HS_P, 1.f, OS_P32, OS_PHALF));
  }
  {   // U = ColNorm(W), as a pair of fixed scale (unit-norm columns) or in fp32, in P0; W's pair in P1
  PhaseScope ps(c, st, DION_PHASE_COLNORM);
  ColnormPairs x = ColnormPairs();
  x.kind = CN_HALF; x.qh = s.ws + s.L.P0; x.qscale = ldexpf(1.f, HS_U_BITS); x.qpair = 1; x.hi = s.ws + s.L.P1; x.other = sc + HS_Q; x.os = s.os;
  DION_TRY(colnorm(s, 0, R, m, r, nullptr, r, a->colnorm_out, nullptr, x));
  }
  {   // M <- (M + G) - (1 - mu) W Q^T
  PhaseScope ps(c, st, DION_PHASE_EF);
  GemmArgs e = shape(m, n, r, (float*)a->M, a->ldm, EPI_C2_SUB);
  e.C2 = sum; e.ldc2 = n; e.c2_mode = ADD_F32;
  e.alpha = 1.f - c->cfg.mu;
  DION_TRY(product(e, s.L.P1, R, r, false, s.L.S16, Q, a->ldq, true, HS_EF, 1.f, OS_USE32, OS_USEHALF));
  }
  // X <- X - lr sqrt(m/n) U Q^T
  PhaseScope ps_x(c, st, DION_PHASE_X);
  GemmArgs x = shape(m, n, r, (float*)a->X, a->ldx, EPI_SUB);
  x.alpha = lr * sqrtf((float)((double)m / (double)n));
  return product(x, s.L.P0, s.ws + s.L.P0, r, false, s.L.S16, Q, a->ldq, true, HS_Q, ldexpf(1.f, -HS_U_BITS), OS_USE32, OS_USEHALF);
}

// One Lazy-Dion step (Algorithm 6).
int lazy_one(dion_ctx* c, const dion_matrix* a, float lr, int refresh, cudaStream_t st) {
  StepCtx s;
  DION_TRY(begin_step(c, a, 1, st, &s));
  if (lazy_on_pairs(s, a)) return lazy_pairs(s, a, lr, refresh);
  DION_TRY(clear_slots(s));
  const i64 m = a->m, n = a->n, r = a->r;
  const int gmode = (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32;
  float* P0 = s.ws + s.L.P0;
  float* R = s.ws + s.L.R;
  const float* Mp = (const float*)a->M;
  // bf16-operand mode on the tensor engine: as in the Dion step, bf16(M + G) is formed once and the
  // products read bf16 arrays (B16, and bf16 copies of Q, T / W, ColNorm(W))
  const bool d16 = s.tensor && c->cfg.precision == DION_PREC_BF16_OPERANDS && m % 8 == 0 && n % 8 == 0 && r % 8 == 0 &&
                   m >= 128 && n >= 128 && r >= 64 && !((uintptr_t)a->Q & 15) && a->ldq % 4 == 0;
  auto bf = [&](i64 off) { return reinterpret_cast<__nv_bfloat16*>(s.ws + off); };
  auto to_bf16 = [&](const float* src, i64 lds, i64 rows, i64 cols, __nv_bfloat16* out) -> int {
    launch_pdl(k_to_bf16, dim3((unsigned)grid_for(c, rows * cols / 8)), dim3(256), 0, st, src, lds, rows, cols, out, nullptr);
    DION_CHECK_LAUNCH(c);
    return DION_OK;
  };
  // B Q -> out (m x r): the fused fp32 path, or B16 Q16
  auto b_times_q = [&](float* out, int precise) -> int {
    GemmArgs t = gemm_args();
    t.M = m; t.N = r; t.K = n;
    if (d16) {
      DION_TRY(to_bf16((const float*)a->Q, a->ldq, n, r, bf(s.L.Q16)));
      t.ab16 = 1;
      t.A = (const float*)bf(s.L.B16); t.a_si = n; t.a_sk = 1;
      t.B = (const float*)bf(s.L.Q16); t.b_sk = r; t.b_sn = 1;
    } else {
      t.A = Mp; t.a_si = a->ldm; t.a_sk = 1;
      t.A2 = a->G; t.a2_si = a->ldg; t.a2_sk = 1; t.a2_mode = gmode;
      t.B = (const float*)a->Q; t.b_sk = a->ldq; t.b_sn = 1;
      t.precise = precise;
    }
    t.C = out; t.ldc = r; t.epi = EPI_STORE;
    return launch_gemm(s, t);
  };
  if (d16) {
    const bool vec = !((uintptr_t)a->M & 15) && a->ldm % 4 == 0 && !((uintptr_t)a->G & 15) &&
                     a->ldg % ((a->g_dtype == DION_BF16) ? 8 : 4) == 0;
    const dim3 grid((unsigned)grid_for(c, m * n / 8));
    if (vec) launch_pdl(k_form_b16<true>, grid, dim3(256), 0, st, Mp, a->ldm, a->G, a->ldg, gmode, m, n, bf(s.L.B16), (int*)nullptr);
    else launch_pdl(k_form_b16<false>, grid, dim3(256), 0, st, Mp, a->ldm, a->G, a->ldg, gmode, m, n, bf(s.L.B16), (int*)nullptr);
    DION_CHECK_LAUNCH(c);
  }

  if (refresh) {
    // profiling: the whole refresh (SymPowerIter1) is booked as the ORTH phase
    PhaseScope ps_orth(c, st, DION_PHASE_ORTH);
    // T = (M + G) Q  (m x r), Z = (M + G)^T T (n x r), Q <- Orthonormalize(Z)
    const int precise = (resolve_orth(c, r, (m < n) ? m : n) == DION_ORTH_SHIFTED3) ? 1 : 0;
    DION_TRY(b_times_q(R, precise));
    GemmArgs z = gemm_args();
    z.M = n; z.N = r; z.K = m;
    if (d16) {
      DION_TRY(to_bf16(R, r, m, r, bf(s.L.U16)));
      z.ab16 = 1;
      z.A = (const float*)bf(s.L.B16); z.a_si = 1; z.a_sk = n;
      z.B = (const float*)bf(s.L.U16); z.b_sk = r; z.b_sn = 1;
    } else {
      z.A = Mp; z.a_si = 1; z.a_sk = a->ldm;
      z.A2 = a->G; z.a2_si = 1; z.a2_sk = a->ldg; z.a2_mode = gmode;
      z.B = R; z.b_sk = r; z.b_sn = 1;
      z.precise = precise;
    }
    const i64 pin_off = panel_offset(s, r, (m < n) ? m : n);
    z.C = s.ws + pin_off; z.ldc = r; z.epi = EPI_STORE;
    DION_TRY(launch_gemm(s, z));
    i64 V_off = 0;
    s.in_orth = true;
    const int rc_orth = orthonormalize(s, n, r, (m < n) ? m : n, pin_off, &V_off);
    s.in_orth = false;
    DION_TRY(rc_orth);
    const float* V = s.ws + V_off;
    // copy V into Q unless the round broke down
    const i64 total = n * r;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 8 * c->sm_count) blocks = 8 * c->sm_count;
    launch_pdl(k_copy_panel, dim3((unsigned)(blocks)), dim3(256), 0, st, V, r, (float*)a->Q, a->ldq, n, r, (const int*)s.flag, (const int*)nullptr, (i64)0, -1);
    DION_CHECK_LAUNCH(c);
  }
  // W = (M + G) Q
  {
  PhaseScope ps(c, st, DION_PHASE_P);
  DION_TRY(b_times_q(R, 0));
  }
  // M <- (M + G) - (1 - mu) W Q^T
  {
  PhaseScope ps(c, st, DION_PHASE_EF);
  GemmArgs e = gemm_args();
  e.M = m; e.N = n; e.K = r;
  if (d16) {   // Q16 was written by b_times_q just above
    DION_TRY(to_bf16(R, r, m, r, bf(s.L.U16)));
    e.ab16 = 1;
    e.A = (const float*)bf(s.L.U16); e.a_si = r; e.a_sk = 1;
    e.B = (const float*)bf(s.L.Q16); e.b_sk = 1; e.b_sn = r;
  } else {
    e.A = R; e.a_si = r; e.a_sk = 1;
    e.B = (const float*)a->Q; e.b_sk = 1; e.b_sn = a->ldq;
  }
  e.C = (float*)a->M; e.ldc = a->ldm; e.epi = EPI_ADD2_SUB;
  e.C2 = a->G; e.ldc2 = a->ldg; e.c2_mode = gmode;
  e.alpha = 1.f - c->cfg.mu;
  e.skip_flag = s.flag;
  DION_TRY(launch_gemm(s, e));
  }
  // U = ColNorm(W)
  {
  PhaseScope ps(c, st, DION_PHASE_COLNORM);
  DION_TRY(colnorm(s, 0, R, m, r, P0, r, a->colnorm_out));
  }
  // X <- X - lr sqrt(m/n) U Q^T
  PhaseScope ps_x(c, st, DION_PHASE_X);
  GemmArgs x = gemm_args();
  x.M = m; x.N = n; x.K = r;
  if (d16) {
    DION_TRY(to_bf16(P0, r, m, r, bf(s.L.R16)));
    x.ab16 = 1;
    x.A = (const float*)bf(s.L.R16); x.a_si = r; x.a_sk = 1;
    x.B = (const float*)bf(s.L.Q16); x.b_sk = 1; x.b_sn = r;
  } else {
    x.A = P0; x.a_si = r; x.a_sk = 1;
    x.B = (const float*)a->Q; x.b_sk = 1; x.b_sn = a->ldq;
  }
  x.C = (float*)a->X; x.ldc = a->ldx; x.epi = EPI_SUB;
  x.alpha = lr * sqrtf((float)((double)m / (double)n));
  x.skip_flag = s.flag;
  DION_TRY(launch_gemm(s, x));
  return DION_OK;
}

}  // namespace

extern "C" {

void dion_default_config(dion_config* cfg) {
  if (cfg == nullptr) return;
  cfg->mu = 0.95f;
  cfg->eps = 1e-8f;
  cfg->precision = DION_PREC_FP32;
  cfg->orth = DION_ORTH_AUTO;
  cfg->engine = DION_ENGINE_AUTO;
  cfg->device = 0;
  cfg->workspace_bytes = 0;
}

int dion_init(dion_ctx** out, const dion_config* cfg) {
  if (out == nullptr) return DION_ERR_INVALID;
  *out = nullptr;
  if (cfg == nullptr) return DION_ERR_INVALID;
  if (cfg->precision != DION_PREC_FP32 && cfg->precision != DION_PREC_BF16_OPERANDS) return DION_ERR_INVALID;
  if (cfg->orth < DION_ORTH_AUTO || cfg->orth > DION_ORTH_RCQR) return DION_ERR_INVALID;
  if (cfg->engine < DION_ENGINE_AUTO || cfg->engine > DION_ENGINE_TENSOR) return DION_ERR_INVALID;
  if (!(cfg->mu >= 0.f && cfg->mu <= 1.f) || !(cfg->eps >= 0.f)) return DION_ERR_INVALID;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device < 0 || cfg->device >= ndev) {
    cudaGetLastError();
    return DION_ERR_CUDA;
  }
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, cfg->device) != cudaSuccess) return DION_ERR_CUDA;
  if (prop.major != 10) return DION_ERR_CUDA;  // built for sm_100a only
  if (cudaSetDevice(cfg->device) != cudaSuccess) return DION_ERR_CUDA;
  dion_ctx* c = new (std::nothrow) dion_ctx();
  if (c == nullptr) return DION_ERR_NOMEM;
  c->ws = nullptr; c->ws_bytes = 0; c->dev_ints = nullptr; c->flag_cursor = 0; c->launches = 0;
  c->prof_on = false; c->prof_used = 0;
  c->cfg = *cfg;
  c->sm_count = prop.multiProcessorCount;
  void* p = nullptr;
  constexpr size_t int_bytes = sizeof(int) * (8 + MAX_FLAG_SLOTS * OS_SLOT_INTS + 24 + FLOW_CTL_INTS);
  if (cudaMalloc(&p, int_bytes) != cudaSuccess) { delete c; return DION_ERR_NOMEM; }
  c->dev_ints = (int*)p;
  c->flow_ctl = c->dev_ints + 8 + MAX_FLAG_SLOTS * OS_SLOT_INTS + 24;      // (128-byte aligned)
  c->flow_ctl_cap = FLOW_CTL_INTS;
  if (cudaMemset(p, 0, int_bytes) != cudaSuccess) { cudaFree(p); delete c; return DION_ERR_CUDA; }
  if (configure_kernels() != DION_OK) { cudaFree(p); delete c; return DION_ERR_CUDA; }
  if (cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); c->side = nullptr; }
  // graph replay of small steps: a capture stream and the scalars the graphs read; off if either cannot be had
  umma::pair_clusters(c->sm_count);      // (asked once per device, outside any capture)
  {
    void* gs = nullptr;
    if (cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking) == cudaSuccess &&
        cudaMalloc(&gs, sizeof(float) * MAX_GRAPHS) == cudaSuccess) {
      c->graph_scalars = (float*)gs;
      c->graphs_on = true;
    } else {
      cudaGetLastError();
      if (c->cap != nullptr) { cudaStreamDestroy(c->cap); c->cap = nullptr; }
    }
  }
  for (int i = 0; i < 32 && c->side != nullptr; ++i)
    if (cudaEventCreateWithFlags(&c->side_ev[i], cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      cudaStreamDestroy(c->side);
      c->side = nullptr;      // no look-ahead: everything runs on the caller's stream
    }
  if (cfg->workspace_bytes > 0) {
    const int rc = ensure_ws(c, cfg->workspace_bytes);
    if (rc != DION_OK) { cudaFree(c->dev_ints); delete c; return rc; }
  }
  *out = c;
  return DION_OK;
}

size_t dion_workspace_bytes(const dion_ctx* ctx, int64_t m, int64_t n, int64_t r) {
  if (ctx == nullptr || m < 1 || n < 1 || r < 1 || r > m || r > n) return 0;
  return (size_t)make_layout(ctx, m, n, r).total * sizeof(float);
}

int dion_step(dion_ctx* ctx, const dion_matrix* a, float lr, void* cuda_stream) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  DION_TRY(validate(a));
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  DION_TRY(ensure_ws(ctx, dion_workspace_bytes(ctx, a->m, a->n, a->r)));
  if (graph_eligible(ctx, a)) {
    const int rc = step_graph(ctx, a, lr, (cudaStream_t)cuda_stream);
    if (rc <= 0) return rc;
  }
  return step_one(ctx, a, lr, (cudaStream_t)cuda_stream);
}

int dion_step_grouped(dion_ctx* ctx, const dion_matrix* list, int count, float lr, void* cuda_stream) {
  if (ctx == nullptr || count < 0) return DION_ERR_INVALID;
  if (count == 0) return DION_OK;
  if (list == nullptr) return DION_ERR_INVALID;
  for (int i = 0; i < count; ++i) DION_TRY(validate(&list[i]));
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  // Matrices of identical (m, n, r) form a class (the paper's batch axis).  A class is
  // stepped in chains of up to `cap` matrices that share each small kernel launch of the
  // factorization; every matrix of a chain has its own scratch slice.
  const size_t budget = ctx->cfg.workspace_bytes > GROUP_SCRATCH_BYTES ? ctx->cfg.workspace_bytes : GROUP_SCRATCH_BYTES;
  std::vector<char> done((size_t)count, 0);
  std::vector<const dion_matrix*> chain;
  size_t need = 0;
  std::vector<std::vector<const dion_matrix*>> chains;
  for (int i = 0; i < count; ++i) {
    if (done[i]) continue;
    const size_t one = dion_workspace_bytes(ctx, list[i].m, list[i].n, list[i].r);
    size_t cap = one > 0 ? budget / one : 1;
    if (cap < 1) cap = 1;
    if (cap > MAX_CHAIN) cap = MAX_CHAIN;
    chain.clear();
    for (int j = i; j < count; ++j) {
      if (done[j] || list[j].m != list[i].m || list[j].n != list[i].n || list[j].r != list[i].r ||
          list[j].transposed != list[i].transposed || list[j].sketch_rows != list[i].sketch_rows) continue;
      done[j] = 1;
      chain.push_back(&list[j]);
      if (chain.size() == cap) { chains.push_back(chain); chain.clear(); }
    }
    if (!chain.empty()) chains.push_back(chain);
  }
  for (const auto& ch : chains) {
    const size_t b = dion_workspace_bytes(ctx, ch[0]->m, ch[0]->n, ch[0]->r) * ch.size();
    if (b > need) need = b;
  }
  DION_TRY(ensure_ws(ctx, need));
  for (const auto& ch : chains) DION_TRY(step_batch(ctx, ch.data(), (int)ch.size(), lr, (cudaStream_t)cuda_stream));
  return DION_OK;
}

int dion_lazy_step(dion_ctx* ctx, const dion_matrix* a, float lr, int refresh, void* cuda_stream) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  DION_TRY(validate(a));
  if (a->transposed) return DION_ERR_INVALID;   // Algorithm 6 is built in the standard form only
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  DION_TRY(ensure_ws(ctx, dion_workspace_bytes(ctx, a->m, a->n, a->r)));
  return lazy_one(ctx, a, lr, refresh, (cudaStream_t)cuda_stream);
}

// ---- compressed data-parallel sync: the step in three calls --------------------------------

namespace {

int dp_check(dion_ctx* ctx, const dion_matrix* a, const void* p0, const void* p1, const int* flag) {
  if (ctx == nullptr || p0 == nullptr || p1 == nullptr || flag == nullptr) return DION_ERR_INVALID;
  DION_TRY(validate(a));
  if (a->transposed) return DION_ERR_INVALID;
  if (((uintptr_t)p0 & 15) || ((uintptr_t)p1 & 15) || ((uintptr_t)flag & 3)) return DION_ERR_ALIGN;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  return ensure_ws(ctx, dion_workspace_bytes(ctx, a->m, a->n, a->r));
}

GemmArgs dp_b_product(const dion_matrix* a, bool transposed_b, const float* rhs, float* out) {
  const i64 m = a->m, n = a->n, r = a->r;
  GemmArgs g = gemm_args();
  g.M = transposed_b ? n : m; g.N = r; g.K = transposed_b ? m : n;
  g.A = (const float*)a->M; g.a_si = transposed_b ? 1 : a->ldm; g.a_sk = transposed_b ? a->ldm : 1;
  g.A2 = a->G; g.a2_si = transposed_b ? 1 : a->ldg; g.a2_sk = transposed_b ? a->ldg : 1;
  g.a2_mode = (a->g_dtype == DION_BF16) ? ADD_BF16 : ADD_F32;
  g.B = rhs; g.b_sk = r; g.b_sn = 1;
  g.C = out; g.ldc = r; g.epi = EPI_STORE;
  return g;
}

// The pieces of a step on half pairs (step_on_half_pairs) as calls of their own.  P = (M + G) Q:
int half_project(StepCtx& s, const dion_matrix* a, float* P, int* flag) {
  const i64 m = a->m, n = a->n, r = a->r;
  DION_TRY(half_sum_chain(s, &a, n, true, true, flag));
  const __half* bh = reinterpret_cast<const __half*>(s.ws + s.L.Bp);
  const __half* qh = reinterpret_cast<const __half*>(s.ws + s.L.S16);
  GemmArgs p = gemm_args();
  p.M = m; p.N = r; p.K = n;
  p.ab16 = 1; p.f16 = 1;
  p.A = (const float*)bh; p.A16lo = bh + m * n; p.a_si = n; p.a_sk = 1;
  p.B = (const float*)qh; p.B16lo = qh + n * r; p.b_sk = r; p.b_sn = 1;
  p.alpha_dev = s.ws + s.L.lz + HS_P;
  p.C = P; p.ldc = r; p.epi = EPI_STORE;
  p.skip_flag = s.os + OS_P32;
  DION_TRY(launch_gemm(s, p, 0));
  s.no_split = n <= WIDE_P_WHOLE_K;
  const int rc = launch_gemm(s, wide_p(s, 0, a, false, P), 0);
  s.no_split = false;
  return rc;
}
// W = (M + G)^T U:
int half_factor(StepCtx& s, const dion_matrix* a, const float* U, float* W, const int* skip) {
  const i64 m = a->m, r = a->r;
  DION_TRY(half_sum_chain(s, &a, 0, false, true));
  DION_TRY(split_half_chain(s, &U, r, m, r, s.L.P1, HS_U_BITS, skip, -1));
  GemmArgs w;
  DION_TRY(r_pairs(s, 0, a, false, U, s.ws + s.L.P1, W, skip, &w, true));
  w.f16 = 1; w.wide_flag = s.os + OS_WIDE; w.alpha_dev = s.ws + s.L.lz + HS_R;
  return launch_gemm(s, w, 0);
}
// The error feedback, Q and the weight update (sums: see colnorm_launch; alpha: the update's factor).  M + G is not formed
// here: whether the error feedback's factors are half or bf16 pairs is decided by their own ranges.
int half_finish(StepCtx& s, const dion_matrix* a, const float* U, const float* W, const float* sums, float alpha, const int* flag) {
  dion_ctx* c = s.c;
  const i64 m = a->m, n = a->n, r = a->r;
  ChainPtrs t;
  t.p[0] = W; t.p[1] = U;
  ColnormPairs x = ColnormPairs();
  const i64 pieces = (((m > n) ? m : n) + RANGE_ROWS - 1) / RANGE_ROWS * ((r + 127) / 128);
  x.nrange = grid_for(c, 32 * pieces, 2);
  float* range = s.ws + s.L.part;
  launch_pdl(k_range_partial, dim3((unsigned)x.nrange, 2), dim3(256), 0, s.st, t, r, n, m, r, range, (i64)2 * x.nrange, (const int*)nullptr, (i64)0, s.os);
  DION_CHECK_LAUNCH(c);
  const i64 u_one = s.L.P0 + ((m > n) ? m : n) * r / 2;      // (behind Q's half array)
  x.kind = CN_HALF; x.qh = s.ws + s.L.P0; x.qscale = half_scale(n); x.hi = s.ws + s.L.S16; x.os = s.os; x.range = range;
  DION_TRY(colnorm(s, 0, W, n, r, (float*)a->Q, a->ldq, a->colnorm_out, flag, x, sums));
  DION_TRY(split_half_chain(s, &U, r, m, r, s.L.P1, HS_U_BITS, flag, u_one));
  GemmArgs e;
  DION_TRY(ef_update(s, 0, a, U, r, W, r, s.ws + s.L.P1, s.ws + s.L.S16, nullptr, flag, true, true, &e));
  if (e.ab16) { e.f16 = 1; e.wide_flag = s.os + OS_WIDE; e.alpha_dev = s.ws + s.L.lz + HS_EF; }
  DION_TRY(launch_gemm(s, e, 0));
  const bool rounded = x_single_pass(s, a, U, r, (const float*)a->Q, a->ldq) && x_half(a);
  return x_update(s, 0, a, U, r, (const float*)a->Q, a->ldq, s.ws + (rounded ? u_one : s.L.P1), s.ws + s.L.P0, alpha, flag, nullptr, nullptr, rounded,
                  rounded ? ldexpf(1.f, HS_U_BITS) : 0.f, 0.f);
}

}  // namespace

int dion_dp_project(dion_ctx* ctx, const dion_matrix* a, float* P, int* dp_flag, void* cuda_stream) {
  DION_TRY(dp_check(ctx, a, P, P, dp_flag));
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  if (step_on_half_pairs(s, a->m, a->n, a->r, (a->m < a->n) ? a->m : a->n)) return half_project(s, a, P, dp_flag);
  DION_TRY(clear_slots(s, dp_flag));
  GemmArgs p = dp_b_product(a, false, (const float*)a->Q, P);
  p.b_sk = a->ldq;
  p.precise = (resolve_orth(ctx, a->r, (a->m < a->n) ? a->m : a->n) == DION_ORTH_SHIFTED3) ? 1 : 0;
  return launch_gemm(s, p, 0);
}

int dion_dp_factor(dion_ctx* ctx, const dion_matrix* a, float* PU, float* W, int* dp_flag, void* cuda_stream) {
  DION_TRY(dp_check(ctx, a, PU, W, dp_flag));
  if (ctx->cfg.orth == DION_ORTH_RCQR) return DION_ERR_UNSUPPORTED;
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  const i64 m = a->m, n = a->n, r = a->r;
  dim3 grid((unsigned)grid_for(ctx, (m * r + 3) / 4), 1);
  const i64 pin_off = panel_offset(s, r, (m < n) ? m : n);
  launch_pdl(k_copy_block, grid, dim3(256), 0, st, PU, r, s.ws + pin_off, r, m, r, nullptr, 0, (const int*)nullptr, (int*)nullptr, s.os);
  DION_CHECK_LAUNCH(ctx);
  i64 U_off = 0;
  s.in_orth = true;
  const int rc = orthonormalize(s, m, r, (m < n) ? m : n, pin_off, &U_off);
  s.in_orth = false;
  DION_TRY(rc);
  launch_pdl(k_copy_block, grid, dim3(256), 0, st, s.ws + U_off, r, PU, r, m, r, nullptr, 0, (const int*)s.flag, dp_flag, (int*)nullptr);      // (a breakdown cancels dion_dp_finish)
  DION_CHECK_LAUNCH(ctx);
  if (step_on_half_pairs(s, m, n, r, (m < n) ? m : n)) return half_factor(s, a, PU, W, nullptr);
  if (r_on_pairs(s, m, n, r)) {       // as dion_step: W on the bf16 pairs of M + G and U
    DION_TRY(form_sum(s, 0, a, true));
    return r_pairs(s, 0, a, false, PU, s.ws + s.L.P1, W, nullptr);
  }
  return launch_gemm(s, dp_b_product(a, true, PU, W), 0);
}

int dion_dp_finish(dion_ctx* ctx, const dion_matrix* a, const float* U, const float* W, const int* dp_flag,
                   float lr, void* cuda_stream) {
  DION_TRY(dp_check(ctx, a, U, W, dp_flag));
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  const i64 m = a->m, n = a->n, r = a->r;
  const float alpha = lr * sqrtf((float)((double)m / (double)n));
  if (step_on_half_pairs(s, m, n, r, (m < n) ? m : n)) {
    DION_TRY(half_finish(s, a, U, W, nullptr, alpha, dp_flag));
  } else {
    DION_TRY(clear_slots(s));
    // M <- (M + G) - (1 - mu) U W^T, with this rank's M and G (as in dion_step)
    DION_TRY(ef_update(s, 0, a, U, r, W, r, s.ws + s.L.P1, s.ws + s.L.S16, nullptr, dp_flag));
    DION_TRY(colnorm(s, 0, W, n, r, (float*)a->Q, a->ldq, a->colnorm_out, dp_flag));
    // X <- X - lr sqrt(m/n) U Q^T, as in dion_step (rounded copies in the two panel buffers of the scratch)
    DION_TRY(x_update(s, 0, a, U, r, (const float*)a->Q, a->ldq, s.ws + s.L.P1, s.ws + s.L.R, alpha, dp_flag));
  }
  return DION_OK;
}

// ---- 1D-sharded Dion (Algorithm 3): the per-rank pieces between its collectives -------------------

namespace {

int shard_check(dion_ctx* ctx, const dion_matrix* a, int64_t n_total, const void* p0, const void* p1, const int* flag) {
  if (ctx == nullptr || p0 == nullptr || p1 == nullptr || flag == nullptr) return DION_ERR_INVALID;
  DION_TRY(validate(a, true));
  if (a->transposed || n_total < a->n || a->r > n_total) return DION_ERR_INVALID;
  if (((uintptr_t)p0 & 15) || ((uintptr_t)p1 & 15) || ((uintptr_t)flag & 3)) return DION_ERR_ALIGN;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  return ensure_ws(ctx, (size_t)make_layout(ctx, a->m, a->n, a->r).total * sizeof(float));
}

}  // namespace

int dion_shard_project(dion_ctx* ctx, const dion_matrix* a, int64_t n_total, float* P, int* flag, void* cuda_stream) {
  DION_TRY(shard_check(ctx, a, n_total, P, P, flag));
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  if (step_on_half_pairs(s, a->m, a->n, a->r, (a->m < n_total) ? a->m : n_total)) return half_project(s, a, P, flag);
  DION_TRY(clear_slots(s, flag));
  GemmArgs p = dp_b_product(a, false, (const float*)a->Q, P);
  p.b_sk = a->ldq;
  p.precise = (resolve_orth(ctx, a->r, (a->m < n_total) ? a->m : n_total) == DION_ORTH_SHIFTED3) ? 1 : 0;
  return launch_gemm(s, p, 0);
}

int dion_orthonormalize(dion_ctx* ctx, int64_t m, int64_t r, int64_t n_total, float* PU, int* flag, void* cuda_stream) {
  if (ctx == nullptr || PU == nullptr || flag == nullptr) return DION_ERR_INVALID;
  if (m < 1 || n_total < 1 || r < 1 || r > m || r > n_total) return DION_ERR_SHAPE;
  if (((uintptr_t)PU & 15) || ((uintptr_t)flag & 3)) return DION_ERR_ALIGN;
  if (ctx->cfg.orth == DION_ORTH_RCQR) return DION_ERR_UNSUPPORTED;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  dion_matrix shape;
  memset(&shape, 0, sizeof(shape));
  shape.m = m; shape.n = n_total; shape.r = r;
  DION_TRY(ensure_ws(ctx, (size_t)make_layout(ctx, m, n_total, r).total * sizeof(float)));
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, &shape, 1, st, &s));
  const i64 sd = (m < n_total) ? m : n_total;
  const i64 pin_off = panel_offset(s, r, sd);
  dim3 grid((unsigned)grid_for(ctx, (m * r + 3) / 4), 1);
  launch_pdl(k_copy_block, grid, dim3(256), 0, st, (const float*)PU, r, s.ws + pin_off, r, m, r, nullptr, 0, (const int*)nullptr, (int*)nullptr, s.os);
  DION_CHECK_LAUNCH(ctx);
  i64 U_off = 0;
  s.in_orth = true;
  const int rc = orthonormalize(s, m, r, sd, pin_off, &U_off);
  s.in_orth = false;
  DION_TRY(rc);
  launch_pdl(k_copy_block, grid, dim3(256), 0, st, (const float*)(s.ws + U_off), r, PU, r, m, r, nullptr, 0, (const int*)s.flag, flag, (int*)nullptr);
  DION_CHECK_LAUNCH(ctx);
  return DION_OK;
}

int dion_shard_factor(dion_ctx* ctx, const dion_matrix* a, int64_t n_total, const float* U, float* W, float* colsumsq,
                      const int* flag, void* cuda_stream) {
  DION_TRY(shard_check(ctx, a, n_total, U, W, flag));
  if (colsumsq == nullptr) return DION_ERR_INVALID;
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  DION_TRY(clear_slots(s));
  if (step_on_half_pairs(s, a->m, a->n, a->r, (a->m < n_total) ? a->m : n_total)) {
    DION_TRY(half_factor(s, a, U, W, flag));
  } else if (r_on_pairs(s, a->m, a->n, a->r)) {       // as dion_step: W on the bf16 pairs of M + G and U
    DION_TRY(form_sum(s, 0, a, true));
    DION_TRY(r_pairs(s, 0, a, false, U, s.ws + s.L.P1, W, flag));
  } else {
    GemmArgs w = dp_b_product(a, true, U, W);
    w.skip_flag = flag;
    DION_TRY(launch_gemm(s, w, 0));
  }
  int chunks; i64 per;
  colnorm_chunks(ctx, s.L, a->n, a->r, &chunks, &per);
  float* part = s.W(0, s.L.cn_part);
  const dim3 grid((unsigned)((a->r + 127) / 128), (unsigned)chunks);
  if (a->r % 4 == 0) {
    launch_pdl(k_colsumsq_partial<true>, grid, dim3(CN_THREADS), 0, st, (const float*)W, a->r, a->n, a->r, per, part, (float*)nullptr, flag, (i64)0);
    DION_CHECK_LAUNCH(ctx);
    launch_pdl(k_colsumsq_finish<true>, dim3(grid.x), dim3(CN_THREADS), 0, st, (const float*)part, chunks, a->r, colsumsq, flag);
  } else {
    launch_pdl(k_colsumsq_partial<false>, grid, dim3(CN_THREADS), 0, st, (const float*)W, a->r, a->n, a->r, per, part, (float*)nullptr, flag, (i64)0);
    DION_CHECK_LAUNCH(ctx);
    launch_pdl(k_colsumsq_finish<false>, dim3(grid.x), dim3(CN_THREADS), 0, st, (const float*)part, chunks, a->r, colsumsq, flag);
  }
  DION_CHECK_LAUNCH(ctx);
  return DION_OK;
}

int dion_shard_finish(dion_ctx* ctx, const dion_matrix* a, int64_t n_total, const float* U, const float* W,
                      const float* colsumsq, const int* flag, float lr, void* cuda_stream) {
  DION_TRY(shard_check(ctx, a, n_total, U, W, flag));
  if (colsumsq == nullptr) return DION_ERR_INVALID;
  StepCtx s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DION_TRY(begin_step(ctx, a, 1, st, &s));
  const i64 m = a->m, n = a->n, r = a->r;
  const float alpha = lr * sqrtf((float)((double)m / (double)n_total));
  if (step_on_half_pairs(s, m, n, r, (m < n_total) ? m : n_total)) {
    DION_TRY(half_finish(s, a, U, W, colsumsq, alpha, flag));
  } else {
    DION_TRY(clear_slots(s));
    // M <- (M + G) - (1 - mu) U W^T on the shard's columns; Q <- W / (sqrt(colsumsq) + eps) with the all-reduced squared norms
    DION_TRY(ef_update(s, 0, a, U, r, W, r, s.ws + s.L.P1, s.ws + s.L.S16, nullptr, flag));
    DION_TRY(colnorm(s, 0, W, n, r, (float*)a->Q, a->ldq, a->colnorm_out, flag, ColnormPairs(), colsumsq));
    // X <- X - lr sqrt(m / n_total) U Q^T on the shard's columns
    DION_TRY(x_update(s, 0, a, U, r, (const float*)a->Q, a->ldq, s.ws + s.L.P1, s.ws + s.L.R, alpha, flag));
  }
  return DION_OK;
}

int dion_get_status(dion_ctx* ctx, void* cuda_stream, int* device_status, int* steps_skipped) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int host[2] = {0, 0};
  if (cudaMemcpyAsync(host, ctx->dev_ints, sizeof(host), cudaMemcpyDeviceToHost, st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaMemsetAsync(ctx->dev_ints, 0, sizeof(host), st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DION_ERR_CUDA;
  if (device_status != nullptr) *device_status = host[0];
  if (steps_skipped != nullptr) *steps_skipped = host[1];
  return DION_OK;
}

int dion_profile_enable(dion_ctx* ctx, int on) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  ctx->prof_on = (on != 0);
  if (on) { ctx->prof_recs.clear(); ctx->prof_used = 0; }
  return DION_OK;
}

int dion_profile_read(dion_ctx* ctx, float* ms, int64_t* launches) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  float acc[DION_NUM_PHASES] = {0};
  int64_t nl[DION_NUM_PHASES] = {0};
  int rc = DION_OK;
  for (const auto& rec : ctx->prof_recs) {
    float t = 0.f;
    if (cudaEventSynchronize(rec.e1) != cudaSuccess || cudaEventElapsedTime(&t, rec.e0, rec.e1) != cudaSuccess) {
      rc = DION_ERR_CUDA;
      break;
    }
    acc[rec.phase] += t;
    nl[rec.phase] += rec.launches;
  }
  ctx->prof_recs.clear();
  ctx->prof_used = 0;
  for (int i = 0; i < DION_NUM_PHASES; ++i) {
    if (ms != nullptr) ms[i] = acc[i];
    if (launches != nullptr) launches[i] = nl[i];
  }
  return rc;
}

int dion_get_orth_rounds(dion_ctx* ctx, void* cuda_stream, int64_t* rounds) {
  if (ctx == nullptr || rounds == nullptr) return DION_ERR_INVALID;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int host = 0;
  if (cudaMemcpyAsync(&host, ctx->dev_ints + 2, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaMemsetAsync(ctx->dev_ints + 2, 0, sizeof(int), st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DION_ERR_CUDA;
  *rounds = host;
  return DION_OK;
}

int dion_get_fallbacks(dion_ctx* ctx, void* cuda_stream, int64_t* fallbacks) {
  if (ctx == nullptr || fallbacks == nullptr) return DION_ERR_INVALID;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int host = 0;
  if (cudaMemcpyAsync(&host, ctx->dev_ints + 3, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaMemsetAsync(ctx->dev_ints + 3, 0, sizeof(int), st) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DION_ERR_CUDA;
  *fallbacks = host;
  return DION_OK;
}

int64_t dion_launch_count(const dion_ctx* ctx) { return ctx == nullptr ? 0 : ctx->launches; }

void dion_destroy(dion_ctx* ctx) {
  if (ctx == nullptr) return;
  cudaSetDevice(ctx->cfg.device);
  cudaDeviceSynchronize();
  graphs_clear(ctx);
  if (ctx->graph_scalars != nullptr) cudaFree(ctx->graph_scalars);
  if (ctx->cap != nullptr) cudaStreamDestroy(ctx->cap);
  if (ctx->ws != nullptr) cudaFree(ctx->ws);
  if (ctx->dev_ints != nullptr) cudaFree(ctx->dev_ints);
  for (cudaEvent_t e : ctx->prof_pool) cudaEventDestroy(e);
  for (int i = 0; i < 32; ++i)
    if (ctx->side_ev[i] != nullptr) cudaEventDestroy(ctx->side_ev[i]);
  if (ctx->side != nullptr) cudaStreamDestroy(ctx->side);
  delete ctx;
}

const char* dion_strerror(int code) {
  switch (code) {
    case DION_OK: return "ok";
    case DION_ERR_INVALID: return "invalid argument";
    case DION_ERR_SHAPE: return "bad shape, rank or leading dimension";
    case DION_ERR_ALIGN: return "misaligned pointer";
    case DION_ERR_ALIAS: return "arrays overlap";
    case DION_ERR_NOMEM: return "out of device memory";
    case DION_ERR_CUDA: return "CUDA error or no sm_100 device";
    case DION_ERR_UNSUPPORTED: return "shape not supported by the requested engine";
    case DION_ERR_TOO_LARGE: return "shape needs more scratch than the built-in array of dion_step_noalloc holds";
    default: return "unknown error";
  }
}

}  // extern "C"

// ---------------------------------------------------------------------------
// dion_step_noalloc: the same step with its scratch in a built-in device array.
// ---------------------------------------------------------------------------

namespace {

// 24 MiB and the factorization's counters and maxima, resident on every device that loads the library
constexpr size_t NOALLOC_SCRATCH_BYTES = ((size_t)24 << 20) + 256 + 16 * 1024;
constexpr size_t NOALLOC_INT_BYTES = 256;                   // status word, counters and one step slot
constexpr size_t NOALLOC_CTL_BYTES = 16 * 1024;             // progress counters of the factorization
constexpr int NOALLOC_MAX_DEVICES = 64;

// Scratch of dion_step_noalloc.  In host code this name is only a handle for
// cudaGetSymbolAddress; the device address is looked up once per device below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

struct NoallocDevice {
  std::atomic<bool> ready;
  unsigned char* base;
  int sm_count;
};
NoallocDevice g_noalloc_dev[NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mutex;

template <typename K>
bool touch_kernel(K kernel) {
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) { cudaGetLastError(); return false; }
  return true;
}

// With lazy module loading a kernel's code is loaded at its first use, which may allocate device memory.
// Asking for the attributes of every kernel the launch chain can reach loads them all at set-up (the
// tensor-core variants and the reduction of their splits are covered by configure_kernels).
bool preload_kernels() {
  bool ok = true;
  ok = ok && touch_kernel(k_gemm_simt<128, 128, 8, 8, 8, 1, NoTabs>) && touch_kernel(k_gemm_simt<64, 64, 16, 4, 4, 2, NoTabs>) &&
       touch_kernel(k_gemm_simt<128, 32, 16, 4, 4, 2, NoTabs>) && touch_kernel(k_gemm_simt<128, 128, 8, 8, 8, 1, GemmSecond>) &&
       touch_kernel(k_gemm_simt<64, 64, 16, 4, 4, 2, GemmSecond>) && touch_kernel(k_gemm_simt<128, 32, 16, 4, 4, 2, GemmSecond>);
  ok = ok && touch_kernel(k_splitk_reduce) && touch_kernel(k_round_begin) && touch_kernel(k_chol_flow<true>);
  ok = ok && touch_kernel(k_chol_flow<false>) && touch_kernel(k_round_end) && touch_kernel(k_tiny_cholqr2);
  ok = ok && touch_kernel(k_probe_fused<true>) && touch_kernel(k_probe_fused<false>) && touch_kernel(k_probe_y) && touch_kernel(k_probe_y4) && touch_kernel(k_probe_w) && touch_kernel(k_probe_w4) && touch_kernel(k_probe_decide) && touch_kernel(k_reset_rounds);
  ok = ok && touch_kernel(k_orth_finish) && touch_kernel(k_cgs_fallback) && touch_kernel(k_copy_block);
  ok = ok && touch_kernel(k_colsumsq_partial<true>) && touch_kernel(k_colsumsq_partial<false>) &&
       touch_kernel(k_colnorm_apply<true, false>) && touch_kernel(k_colnorm_apply<false, false>) && touch_kernel(k_copy_panel);
  ok = ok && touch_kernel(k_hh_reflector);
  ok = ok && touch_kernel(k_hh_apply) && touch_kernel(k_set_identity) && touch_kernel(k_sign_fix);
  ok = ok && touch_kernel(k_form_b16<true>) && touch_kernel(k_form_b16<false>) && touch_kernel(k_form_b32<true>);
  ok = ok && touch_kernel(k_form_b32<false>) && touch_kernel(k_to_bf16) && touch_kernel(k_round_tf32);
  ok = ok && touch_kernel(k_split_bf16) && touch_kernel(k_round_f16);
  return ok;
}

// First use on the current device: resolve the array's device address and read the
// device attributes.  No allocation; must not run inside a stream capture.
int noalloc_setup(int device, NoallocDevice** out) {
  if (device < 0 || device >= NOALLOC_MAX_DEVICES) return DION_ERR_INVALID;
  NoallocDevice* d = &g_noalloc_dev[device];
  if (!d->ready.load(std::memory_order_acquire)) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (d->ready.load(std::memory_order_relaxed)) { *out = d; return DION_OK; }
    int major = 0, sms = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
      cudaGetLastError();
      return DION_ERR_CUDA;
    }
    if (major != 10) return DION_ERR_CUDA;
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || ptr == nullptr) {
      cudaGetLastError();
      return DION_ERR_CUDA;
    }
    if (configure_kernels() != DION_OK || !preload_kernels()) return DION_ERR_CUDA;
    d->base = (unsigned char*)ptr;
    d->sm_count = sms;
    d->ready.store(true, std::memory_order_release);
  }
  *out = d;
  return DION_OK;
}

}  // namespace

extern "C" int dion_step_noalloc(const dion_matrix* a, float lr, float mu, float eps, void* cuda_stream) {
  DION_TRY(validate(a));
  if (!(mu >= 0.f && mu <= 1.f) || !(eps >= 0.f)) return DION_ERR_INVALID;
  int device = -1;
  if (cudaGetDevice(&device) != cudaSuccess) { cudaGetLastError(); return DION_ERR_CUDA; }
  NoallocDevice* nd = nullptr;
  DION_TRY(noalloc_setup(device, &nd));

  // A context that lives on the host stack for this call only and points at the
  // built-in array: the launch chain is the one dion_step runs.
  dion_ctx c;
  dion_default_config(&c.cfg);
  c.cfg.mu = mu;
  c.cfg.eps = eps;
  c.cfg.device = device;
  c.sm_count = nd->sm_count;
  c.dev_ints = (int*)nd->base;
  c.flow_ctl = (int*)(nd->base + NOALLOC_INT_BYTES);
  c.flow_ctl_cap = NOALLOC_CTL_BYTES / sizeof(int);
  c.ws = (float*)(nd->base + NOALLOC_INT_BYTES + NOALLOC_CTL_BYTES);
  c.ws_bytes = NOALLOC_SCRATCH_BYTES - NOALLOC_INT_BYTES - NOALLOC_CTL_BYTES;
  c.flag_cursor = 0;
  c.launches = 0;
  c.prof_on = false;
  c.prof_used = 0;
  c.form_sum = false;
  const size_t need = (size_t)make_layout(&c, a->m, a->n, a->r).total * sizeof(float);
  if (need > c.ws_bytes) return DION_ERR_TOO_LARGE;
  // The array keeps what the previous call left: clear the status word and counters.
  // (The step's own slot is cleared by the launch chain.)
  if (cudaMemsetAsync(c.dev_ints, 0, 8 * sizeof(int), (cudaStream_t)cuda_stream) != cudaSuccess) return DION_ERR_CUDA;
  return step_one(&c, a, lr, (cudaStream_t)cuda_stream);
}

extern "C" size_t dion_noalloc_scratch_limit(void) { return NOALLOC_SCRATCH_BYTES - NOALLOC_INT_BYTES - NOALLOC_CTL_BYTES; }

// ---------------------------------------------------------------------------
// Internal test hook (dion_internal.h)
// ---------------------------------------------------------------------------
// Test hook: the orthogonality estimate of the most recent step's CholeskyQR2 check (first matrix of the chain).
extern "C" int dion_debug_orth_measure(dion_ctx* ctx, void* cuda_stream, float* estimate) {
  if (ctx == nullptr || estimate == nullptr) return DION_ERR_INVALID;
  if (cudaSetDevice(ctx->cfg.device) != cudaSuccess) return DION_ERR_CUDA;
  const int slot = (ctx->flag_cursor + MAX_FLAG_SLOTS - 1) % MAX_FLAG_SLOTS;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (cudaMemcpyAsync(estimate, ctx->dev_ints + 8 + (i64)slot * OS_SLOT_INTS + OS_MAXDEV, sizeof(float), cudaMemcpyDeviceToHost, st) !=
          cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DION_ERR_CUDA;
  return DION_OK;
}

// Test hook: row chunks of `rows` rows in a step on (m, n, r), and the chunks that its scratch holds.
extern "C" int dion_debug_chunks(int64_t m, int64_t n, int64_t r, int64_t rows, int sm_count, int64_t out[4]) {
  if (out == nullptr || m < 1 || n < 1 || r < 1 || rows < 1 || sm_count < 1) return DION_ERR_INVALID;
  dion_ctx c;
  dion_default_config(&c.cfg);
  c.sm_count = sm_count;
  const Layout L = make_layout(&c, m, n, r);
  int chunks; i64 per;
  colnorm_chunks(&c, L, rows, r, &chunks, &per);
  out[0] = chunks * per >= rows ? chunks : -1;
  out[1] = (L.d - L.cn_part - (L.XP < L.Dinv ? NEAR_MAX_BLOCKS : 0)) / r;
  probe_chunks(L, rows, &chunks, &per);
  out[2] = chunks * per >= rows ? chunks : -1;
  out[3] = (L.probe_sums - L.probe_part) / (r * NPROBE);
  return DION_OK;
}

extern "C" int dion_debug_flow_lose(dion_ctx* ctx, int cta, int threads) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  ctx->flow_lose_cta = cta;
  ctx->flow_lose = threads;
  graphs_clear(ctx);
  return DION_OK;
}

extern "C" int dion_debug_chain_batch(dion_ctx* ctx, int on) {
  if (ctx == nullptr) return DION_ERR_INVALID;
  ctx->chain_batch = on != 0;
  graphs_clear(ctx);
  return DION_OK;
}

extern "C" int dion_debug_gemm(int engine, int precision, const dion_debug_gemm_args* a, float* part,
                               int64_t part_floats, int* status, void* cuda_stream) {
  if (a == nullptr || status == nullptr) return DION_ERR_INVALID;
  int device = 0, sms = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return DION_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return DION_ERR_CUDA;
  if (configure_kernels() != DION_OK) return DION_ERR_CUDA;
  GemmArgs g = gemm_args();
  g.M = a->M; g.N = a->N; g.K = a->K;
  g.A = a->A; g.a_si = a->a_si; g.a_sk = a->a_sk;
  g.A2 = a->A2; g.a2_si = a->a2_si; g.a2_sk = a->a2_sk; g.a2_mode = a->a2_mode;
  g.B = a->B; g.b_sk = a->b_sk; g.b_sn = a->b_sn;
  g.C = a->C; g.ldc = a->ldc; g.epi = a->epi;
  g.C2 = a->C2; g.ldc2 = a->ldc2; g.c2_mode = a->c2_mode;
  g.alpha = a->alpha; g.tri = a->tri; g.klimit = a->klimit; g.precise = a->precise; g.ab16 = a->ab16; g.tf32x1 = a->tf32x1; g.f16 = a->f16;
  g.A16lo = a->A16lo; g.B16lo = a->B16lo;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (engine == DION_ENGINE_TENSOR) {
    const int rc = umma_try_launch(g, precision, sms, part, part_floats, status, st, a->variant);
    if (rc > 0) return DION_OK;
    return rc < 0 ? rc : DION_ERR_UNSUPPORTED;
  }
  dion_ctx c;
  dion_default_config(&c.cfg);
  c.sm_count = sms; c.launches = 0; c.prof_on = false; c.prof_used = 0;
  return launch_gemm_simt(&c, g, st, part, part_floats, false);
}
