// Internal declarations shared by the CUDA sources of the (T) library.
//
// Work decomposition (both precisions):
//   * occupied triplets i >= j >= k, all-equal triplets dropped (their sum is
//     exactly zero, Eq. 1), each with weight 2 - d_ij - d_jk;
//   * the virtual range [0, v) cut into tiles of edge NT; an "orbit" is a tile
//     triple P >= Q >= R.  The points (a, b, c) with a in P, b in Q, c in R and
//     a >= b >= c are the canonical points; W at the six permutations of each
//     canonical point lies in the six permuted tile blocks (P,Q,R), (P,R,Q),
//     (Q,P,R), (Q,R,P), (R,P,Q), (R,Q,P) of the same orbit, so one orbit holds
//     everything the energy bracket of Eq. 1 needs;
//   * a work item is (triplet, chunk of consecutive orbits); each item writes
//     one FP64 partial, so the result does not depend on which CTA ran it.
//
// Every kernel takes a batch of up to MAX_BATCH independent jobs by value;
// the global item range is the concatenation of the jobs' item ranges.  A
// job's result depends only on its own items, so it is the same alone or in
// any batch.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include <vector>

namespace tc {

constexpr int MAX_BATCH = 32;

struct Dims {
  int o, v;
  int nt;              // tile edge
  int ntiles;          // ceil(v / nt)
  int n_trip;          // triplets processed (all i >= j >= k without i == j == k, or a subset)
  int n_orb;           // tile triples P >= Q >= R
  int orb_per_item;
  int items_per_trip;
  long long n_items;
};

struct Inputs {        // device pointers, layouts as in include/tc.h
  const double *eps, *t1, *t2, *ovvv, *ovoo, *ovov;
};

struct Work {
  const int4 *trip;    // (i, j, k, weight)
  const int4 *orb;     // (P, Q, R, 0) tile indices
  double *partial;     // [n_items][2]: the item's E_(T) part and its E[5]_ST (V r3(W)/D) part
  unsigned int *counter;
  int *err;            // device error flag (0 = fine); err[1]: the FP64 tensor-core path's input flag
};

// The six permutations of three positions, in the order
// (abc), (acb), (bac), (bca), (cab), (cba); entries 0, 3, 4 are even.
__host__ __device__ constexpr int perm3(int s, int pos) {
  return (s == 0) ? pos
       : (s == 1) ? (pos == 0 ? 0 : (pos == 1 ? 2 : 1))
       : (s == 2) ? (pos == 0 ? 1 : (pos == 1 ? 0 : 2))
       : (s == 3) ? (pos == 0 ? 1 : (pos == 1 ? 2 : 0))
       : (s == 4) ? (pos == 0 ? 2 : (pos == 1 ? 0 : 1))
       :            (pos == 0 ? 2 : (pos == 1 ? 1 : 0));
}
__host__ __device__ constexpr bool perm3_even(int s) { return s == 0 || s == 3 || s == 4; }

// ---------------------------------------------------------------- FP64 path, DMMA kernel
struct FpJob {
  Dims d;
  Inputs in;
  Work w;
  long long item0;     // first global item of this job in the launch
  long long item_base; // the job's own index of that item (a launch may run a slice of a job)
  const int *list;     // optional: the job's items are those of these triplets (their partials' places unchanged)
};
struct FpBatch {
  int njobs;
  long long total_items;
  unsigned int *counter;   // global work counter of the launch (zeroed before it)
  FpJob job[MAX_BATCH];
};
int fp64_tile();
size_t fp64_smem_bytes();
[[nodiscard]] cudaError_t fp64_blocks_per_sm(int *n);
[[nodiscard]] cudaError_t launch_fp64(const FpBatch &b, int grid, cudaStream_t st);
// Kernel-node parameters of one FP64 launch (for CUDA graphs); args[0] must
// point to b while the parameters are used.
void fp64_node_params(const FpBatch &b, int grid, void **args, cudaKernelNodeParams *p);

// ---------------------------------------------------------------- split path
// Geometry of one job's split path (tc_split.cu): W-term GEMMs with 128-row M
// tiles over the v^2 virtual pairs, K blocks of 16, N chunks over v.
struct SplitGeom {
  int o, v, S;
  int mt;                // M tiles: ceil(v^2 / 128)
  int kbv, kbo;          // 16-wide blocks over a virtual / an occupied index (kbv sets the N padding)
  int hv, ho;            // 8-wide K halves over a virtual / an occupied index
  int nch, nc;           // N chunks and their width (multiple of 16, <= 256; <= 224 at s = 4)
  int vc;                // innermost extent of the W buffer and FP32 copies (v rounded up to 4)
  int nb;                // triplets per block (capacity of the W buffer)
};
// Byte offsets of the operand images, FP32 copies and W buffer inside a
// job's split workspace.
struct SplitLayout {
  SplitGeom g;
  size_t pa, pa2, hc, hc2, tb, hb, t1f, epsf, ovovf, y;
  size_t total;
};
struct WtJob {           // one job's block of triplets in a W-term launch
  SplitGeom g;
  const int4 *trip;      // the job's triplet table
  int t0, nt;            // triplets [t0, t0 + nt) of the table
  const unsigned char *pa, *pa2, *hc, *hc2, *tb, *hb;
  float *y;              // W buffer [nt][a][b][vc]: W_abc = F(i,j,k)[ab,c] + F(i,k,j)[ac,b] + F(j,k,i)[bc,a]
  int gsel;              // which F this launch forms: 0 F(i,j,k) (stores), 1 F(i,k,j), 2 F(j,k,i) (add)
  long long item0;       // first global item of this job in the launch (set by the launcher)
};
struct WtBatch {
  int njobs;
  int stages, nprod;     // set by the launcher
  size_t slot;           // set by the launcher: stage stride in shared memory
  long long total_items;
  int *err;
  WtJob job[MAX_BATCH];
};
struct EnJob {           // one job's block of triplets in an energy launch
  CUtensorMap ymap;      // 4-D map of the W buffer: (c, b, a, triplet)
  CUtensorMap gmap;      // 5-D map of the FP32 (p u|q w) in both orders
  CUtensorMap tmap;      // 2-D map of the FP32 t1
  Dims d;
  SplitGeom g;
  const int4 *trip, *orb;
  const double *eps;
  const float *t1f;      // t1 [o][vc]
  const float *epsf;     // eps as float pairs: [0, o+v) hi, [o+v, 2(o+v)) lo
  const float *ovovf;    // [2][o][v][o][vc]: (p u|q w) at [0][p][u][q][w] and [1][q][w][p][u]
  const float *y;
  double *partial;       // [n_items][2], slot t * items_per_trip + chunk
  int t0, nt;
  long long item0;
};
struct EnBatch {
  int njobs;
  long long total_items;
  int *err;
  EnJob job[MAX_BATCH];
};
int split_tile();
// Orbits per energy work item of the split path: about 8 items per SM of a
// 152-SM GPU in each energy launch, so the per-item reduction is amortised.
int split_orb_per_item(int o, int v, int S);
SplitGeom split_geom(int o, int v, int S);
SplitLayout split_layout(int o, int v, int S);
// Operand images and FP32 copies of a job: launch_split_prep builds all of
// them; launch_split_prep_common builds those of t1 and the orbital energies
// and launch_split_prep_range those read from t2, ovvv, ovoo and ovov rows
// whose first occupied index lies in [p0, p1) (what a triplet (i, j, k) with
// i >= j >= k reads lies in the rows p <= i).
[[nodiscard]] cudaError_t launch_split_prep(const SplitLayout &L, const Inputs &in, void *ws, cudaStream_t st);
[[nodiscard]] cudaError_t launch_split_prep_common(const SplitLayout &L, const Inputs &in, void *ws, cudaStream_t st);
[[nodiscard]] cudaError_t launch_split_prep_range(const SplitLayout &L, const Inputs &in, void *ws, cudaStream_t st,
                                                  int p0, int p1);
int split_prep_launches();
int split_prep_common_launches();
int split_prep_range_launches();
WtJob wt_job(const SplitLayout &L, const void *ws, const int4 *trip, int t0, int nt);
// Energy job of triplets [t0, t0 + nt); encodes its tensor map (driver entry point).
[[nodiscard]] cudaError_t en_job(EnJob *out, const Dims &d, const SplitLayout &L, const void *ws, const Inputs &in, const Work &w,
                   int t0, int nt);
// W-term launches per block of triplets: one per F, in the order gsel = 0, 1, 2.
constexpr int SPLIT_WT_LAUNCHES = 3;
// One block of triplets: the three W-term launches, then the energy launch,
// on st.  w0 / w1 (optional) are recorded around the W-term launches.
[[nodiscard]] cudaError_t launch_split_block(WtBatch &wb, EnBatch &eb, int S, int num_sms, cudaStream_t st,
                               cudaEvent_t w0 = nullptr, cudaEvent_t w1 = nullptr);
// Prepare the batches as launch_split_block would and fill the kernel-node
// parameters of its launches: wb[0] is filled by the caller and copied into
// wb[1], wb[2] (gsel 1, 2); wargs[f] / wp[f] belong to wb[f] (f < 3), eargs[0]
// / ep to eb.  The nodes must run in the order wp[0], wp[1], wp[2], ep.
[[nodiscard]] cudaError_t split_block_params(WtBatch *wb, EnBatch &eb, int S, int num_sms, void **wargs, void **eargs,
                               cudaKernelNodeParams *wp, cudaKernelNodeParams *ep);

// ---------------------------------------------------------------- FP64 path on the tensor cores (tc_rns.cu)
// Geometry of one job: 128-row M tiles over the v^2 virtual pairs, K halves of
// 8 over a virtual / an occupied index, N chunks over v.
struct RnsGeom {
  int o, v;
  int mt;                // M tiles: ceil(v^2 / 128)
  int hv, ho;            // K halves over a virtual / an occupied index (hv + ho is even)
  int nch, nc;           // N chunks and their width (multiple of 16, <= 208)
  int vc;                // innermost extent of the W buffer (v rounded up to 4)
  int nb;                // triplets per block (capacity of the W buffer)
};
// Byte offsets inside a job's workspace: operand images, W buffer, the scale
// search's norms, maxima and exponents, unit table, the items' margins over
// the weak triplets' bound and the list of weak triplets, mask of occupied pairs.
struct RnsLayout {
  RnsGeom g;
  size_t pa, pa2, hc, hc2, tb, hb, y, ra, rt, rb, rh, mx, nz, ex, unit, margin, weak, need;
  size_t total;
};
// Host tables of a triplet list.  A unit is one F GEMM of one triplet:
// (triplet index << 3) | (half of K << 2) | F number.  unit holds the storing
// launch's units (one per triplet), then the adding launch's; off[t] counts the
// latter before triplet t.  need: occupied pairs whose operands are read.
struct RnsTables {
  std::vector<int> unit, off;
  std::vector<unsigned char> need;
};
struct RnJob {           // one job's block of triplets in a GEMM launch
  RnsGeom g;
  const int4 *trip;      // the job's triplet table
  const int *unit;       // the block's units
  int t0, nu;            // first triplet of the block; number of units
  const unsigned char *pa, *pa2, *hc, *hc2, *tb, *hb;
  unsigned long long *y; // W buffer [triplet][a][b][vc], 64-bit fractions
  long long item0;       // first global item of this job in the launch (set by the launcher)
};
struct RnBatch {
  int njobs;
  int stages, hps, acc;  // set by the launcher: pipeline stages, K halves of a stage, TMEM columns between the two accumulators (the
                         // launch's widest N chunk: items of different jobs meet in the pipeline)
  size_t slot;           // set by the launcher: stage stride in shared memory
  long long total_items;
  int *err;
  const int *skip;       // optional device flag: not 0, the launch does nothing (inputs beyond the integer grid)
  RnJob job[MAX_BATCH];
};
struct RnEnJob {         // one job's block of triplets in an energy launch
  Dims d;
  int vc;
  const int4 *trip, *orb;
  const double *eps, *t1, *ovov;
  const long long *y;
  const int *ev, *uo, *sh;
  const double *nz;      // W's squared error (Scales::nz)
  double *partial;       // [n_items][2], slot t * items_per_trip + chunk
  double *margin;        // [n_items]: |E[4]_ST| of the item less the weak triplets' bound
  int t0, nt;
  long long item0;
};
struct RnEnBatch {
  int njobs;
  long long total_items;
  const int *skip;       // as RnBatch::skip
  RnEnJob job[MAX_BATCH];
};
constexpr int RNS_GEMM_LAUNCHES = 2;       // storing, then adding
// Smallest v of the residues: v = 8 is one whole DMMA tile but half an N = 16
// chunk and half a 128-row tile here.  Whole calls, residues against DMMA: v = 8
// o = 8 198 / 165 us, o = 16 538 / 438 us, o = 24 1056 / 1010 us; v = 9 o = 2
// 105 / 113 us, o = 8 199 / 308 us, o = 16 536 / 1308 us.
constexpr int RNS_MIN_V = 9;
// Whether the path covers the shape (K bound of the exact FP32 sums).
bool rns_supported(int o, int v);
RnsGeom rns_geom(int o, int v);
RnsLayout rns_layout(const Dims &d);
RnsTables rns_tables(int o, const int4 *trip, int n);
// Scales, operand images and unit table (all: every occupied pair's images,
// else those t.need marks).  *flag (device) is set to 1 when the inputs leave
// the range of the integer grid: the results are then not to be used.  t must
// stay alive until st reaches the copies' end.
[[nodiscard]] cudaError_t launch_rns_prep(const RnsLayout &L, const Inputs &in, void *ws, const RnsTables &t, bool all, int *flag,
                            cudaStream_t st);
int rns_prep_launches(int o, int v);
// Jobs of triplets [t0, t0 + nt) for the two GEMM launches and the energy launch.
void rns_block(const RnsLayout &L, void *ws, const Dims &d, const Inputs &in, const Work &w, const RnsTables &t, int t0,
               int nt, RnJob *j0, RnJob *j1, RnEnJob *en);
[[nodiscard]] cudaError_t launch_rns_block(RnBatch *gb, RnEnBatch &eb, int num_sms, cudaStream_t st, cudaEvent_t w0 = nullptr,
                             cudaEvent_t w1 = nullptr);
// As split_block_params: gp[0], gp[1], ep must run in this order.
[[nodiscard]] cudaError_t rns_block_params(RnBatch *gb, RnEnBatch &eb, int num_sms, void **gargs, void **eargs,
                             cudaKernelNodeParams *gp, cudaKernelNodeParams *ep);

// Fill in the fields by which the reduction lists the weak triplets: those whose
// W lies too far below the common grid's range.  The caller forms them again with
// the DMMA kernel (FpJob::list) and reduces them a second time (RedJob::list).
struct RedJob;
void rns_weak(const RnsLayout &L, void *ws, RedJob *j);

// ---------------------------------------------------------------- integrals from DF factors (tc_df.cu)
// (ia|bd), (ia|jl) and (ia|jb) from B[nq][o+v][o+v] (Eq. 6) as exact digit
// products on the tensor cores.  scratch: df_scratch_bytes(o, v, nq) device
// bytes.  *digits receives the number of base-256 digits the factors needed
// (at most 7); the call synchronises st once to read it.
size_t df_scratch_bytes(int o, int v, int nq);
[[nodiscard]] cudaError_t df_assemble(const double *B, int nq, int o, int v, double *ovvv, double *ovoo, double *ovov,
                        void *scratch, int num_sms, cudaStream_t st, int *digits);
// Device error flag of the assembly's kernels inside its scratch (0 = fine).
int *df_error_flag(void *scratch, int o, int v, int nq);

// ---------------------------------------------------------------- reduction
struct RedJob {
  int n_trip, items_per_trip, o;
  const int4 *trip;
  double *partial;       // [n_trip][items_per_trip][2]; each triplet's first pair is overwritten by its sums
  double *e_trip;        // [n_trip] weighted triplet contributions
  double *e_ijk;         // optional [o][o][o]
  double *out;           // [4]: E, sum |e|, E[5]_ST and the number of weak triplets
  const double *margin;  // optional [n_trip][items_per_trip]: a triplet of negative (or NaN) sum is weak
  int *weak_n, *weak;    // with margin: their number (zero before) and their indices, in any order
  const int *list;       // optional: only the partials of these nlist triplets are new; the others' are their sums
  int nlist;
};
struct RedBatch {
  int njobs;
  RedJob job[MAX_BATCH];
};
[[nodiscard]] cudaError_t launch_reduce(const RedBatch &b, cudaStream_t st);

}  // namespace tc
