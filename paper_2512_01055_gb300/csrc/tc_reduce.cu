// Final reduction: per-item FP64 partials -> weighted per-triplet energies (a
// warp per triplet) -> E_(T) (one CTA per job of the batch).  Both stages use
// Neumaier's compensated summation (Neumaier 1974) in a fixed order, so each job's result is bitwise
// reproducible and independent of the other jobs in the batch.
#include "tc_internal.cuh"

namespace tc {
namespace {

struct Comp { double s, c; };

__device__ __forceinline__ void neumaier_add(Comp &a, double x) {
  const double t = a.s + x;
  a.c += (fabs(a.s) >= fabs(x)) ? ((a.s - t) + x) : ((x - t) + a.s);
  a.s = t;
}

constexpr int RT = 256;

// The sum of two compensated sums.
__device__ __forceinline__ Comp combine(Comp a, const Comp &b) {
  neumaier_add(a, b.s);
  a.c += b.c;
  return a;
}

// The lanes' sums combined by a fixed tree; lane 0 holds the result.
__device__ __forceinline__ Comp warp_combine(Comp p) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    p = combine(p, Comp{__shfl_down_sync(0xffffffffu, p.s, off), __shfl_down_sync(0xffffffffu, p.c, off)});
  return p;
}

// One warp per triplet: lane q sums the item partials q, q + 32, ... in order,
// the lanes are combined by a fixed tree.  Writes the weighted contribution and
// leaves its (E, E[5]_ST) pair in the triplet's first partial slot, and lists
// the triplet where its margin is negative.  One CTA
// with a thread per triplet did this before: 1.6 ms of FP64 latency at o=12
// v=132 (352 triplets of 969 items).
__global__ void __launch_bounds__(RT) reduce_triplets(const __grid_constant__ RedBatch B) {
  const RedJob &J = B.job[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (RT / 32);
  const int n = J.list ? J.nlist : J.n_trip;
  for (int m = blockIdx.x * (RT / 32) + (threadIdx.x >> 5); m < n; m += nw) {
    const int t = J.list ? J.list[m] : m;
    Comp p{0.0, 0.0}, p5{0.0, 0.0};
    double margin = 0.0;
    double *pp = J.partial + 2LL * t * J.items_per_trip;
    for (int c = lane; c < J.items_per_trip; c += 32) {
      const double2 x = *(const double2 *)(pp + 2 * c);
      neumaier_add(p, x.x);
      neumaier_add(p5, x.y);
      if (J.margin) margin += J.margin[(long long)t * J.items_per_trip + c];
    }
    p = warp_combine(p);
    p5 = warp_combine(p5);
    if (J.margin) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) margin += __shfl_down_sync(0xffffffffu, margin, off);
      if (lane == 0 && !(margin >= 0.0)) J.weak[atomicAdd(J.weak_n, 1)] = t;
    }
    __syncwarp();                                           // every lane's reads are done
    if (lane == 0) {
      const int4 tr = J.trip[t];
      const double e = (double)tr.w * (p.s + p.c);          // weight 1 or 2: exact
      J.e_trip[t] = e;
      if (J.e_ijk) J.e_ijk[((long long)tr.x * J.o + tr.y) * J.o + tr.z] = e;
      *(double2 *)pp = make_double2(e, (double)tr.w * (p5.s + p5.c));
    }
  }
}

// One CTA per job: thread q sums triplets q, q + RT, ... in order; the lanes of
// a warp, then the warps, are combined by fixed trees.  Bound by the latency of
// dependent FP64 additions: thread 0 adding up to RT sums in a row took about
// 0.6 us a sum (whole split calls at o=6 v=36 182 us, with the trees 158 us; 0.11
// to 0.23 ms less at o=13 v=131 and o=12 v=132).
__global__ void __launch_bounds__(RT) reduce_jobs(const __grid_constant__ RedBatch B) {
  const RedJob &J = B.job[blockIdx.x];
  constexpr int NW = RT / 32;
  __shared__ Comp s4[NW], s5[NW];
  __shared__ double sa[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Comp a{0.0, 0.0}, a5{0.0, 0.0};
  double absum = 0.0;
  for (int t = threadIdx.x; t < J.n_trip; t += RT) {
    const double2 x = *(const double2 *)(J.partial + 2LL * t * J.items_per_trip);
    neumaier_add(a, x.x);
    neumaier_add(a5, x.y);
    absum += fabs(x.x);
  }
  a = warp_combine(a);
  a5 = warp_combine(a5);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) absum += __shfl_down_sync(0xffffffffu, absum, off);
  if (lane == 0) { s4[warp] = a; s5[warp] = a5; sa[warp] = absum; }
  __syncthreads();
  if (warp == 0) {
    a = lane < NW ? s4[lane] : Comp{0.0, 0.0};
    a5 = lane < NW ? s5[lane] : Comp{0.0, 0.0};
    absum = lane < NW ? sa[lane] : 0.0;
    a = warp_combine(a);
    a5 = warp_combine(a5);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) absum += __shfl_down_sync(0xffffffffu, absum, off);
    if (lane == 0) {
      J.out[0] = a.s + a.c;
      J.out[1] = absum;
      J.out[2] = a5.s + a5.c;
      J.out[3] = J.margin ? (double)*J.weak_n : 0.0;
    }
  }
}

}  // namespace

cudaError_t launch_reduce(const RedBatch &b, cudaStream_t st) {
  if (b.njobs <= 0) return cudaSuccess;
  int most = 0;
  for (int j = 0; j < b.njobs; ++j) {
    const int n = b.job[j].list ? b.job[j].nlist : b.job[j].n_trip;
    most = n > most ? n : most;
  }
  if (most > 0) {
    const int blocks = (most + RT / 32 - 1) / (RT / 32);
    reduce_triplets<<<dim3(blocks < 1024 ? blocks : 1024, b.njobs), RT, 0, st>>>(b);
  }
  reduce_jobs<<<b.njobs, RT, 0, st>>>(b);
  return cudaGetLastError();
}

}  // namespace tc
