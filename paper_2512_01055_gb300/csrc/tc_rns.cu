// FP64 path on the BF16 tensor cores: W (Eqs. 2, 5) as exact integer products
// in a residue number system, V (Eq. 3), D (Fig. 4 sign) and the bracket of
// Eq. 1 in FP64.
//
// GB300's FP64 pipe does about 1 TFLOP/s, its BF16 tensor cores 2400.  So the
// operands are scaled by powers of two and rounded once to integers (about 60
// bits below their row's norm bound), and every integer is held as its
// residues modulo RL pairwise coprime moduli of at most 257: small integers of
// magnitude <= 128, which BF16 holds exactly, whose products sum exactly in
// FP32 while K <= 1024 (128^2 * 1024 = 2^24).  One BF16 GEMM per modulus gives
// the product's residue, and the Chinese remainder theorem the integer itself
// (the second Ozaki scheme: Ozaki, Uchino, Imamura, arXiv 2504.08009; RL = 15
// products, where multiplying digits of the same operands takes 28 to 36).
// The only roundings of W are those of its operands to the integer grid and of
// the integer to its leading 64 bits.
//
// Fractions instead of integers.  With P the product of the moduli,
// x / P mod 1 = sum_l (x q_l mod m_l) / m_l mod 1, q_l = (P / m_l)^-1 mod m_l,
// so x's leading 64 bits are a 64-bit sum of (residue x constant) that wraps
// by itself.  The constant I_l ~ 2^64 k_l / m_l would cost its rounding error
// times the residue; the multiplier k_l is free (the operand images of one
// side absorb q_l / k_l mod m_l), and k_l = (2^64)^-1 mod m_l makes
// I_l = (2^64 k_l - 1) / m_l, i.e. an error of 1/m_l: the sum of 15 terms is
// right to about one unit in the last of 64 places.
//
// Scales.  W_ijk^abc is a sum of products with one fixed-point grid,
// 2^-(e_a + e_b + e_c + u_i + u_j + u_k + SS): an exponent >= 0 per virtual and
// per occupied orbital from the norms of integrals and amplitudes together, and
// a global shift from the largest scaled norms.  The exponents raise no row by
// more than 2 bits over the largest of its array: they refine the grid of weak
// orbitals and hardly coarsen that of the others.  The contributions of all six
// permutations are integers on one grid: they are added by 64-bit integer
// reductions in L2, which are exact and free of order.
//
// W as three GEMMs per triplet (F(p,q,r) of tc_split.cu, the same operand
// segments):  W_abc = F(i,j,k)[ab,c] + F(i,k,j)[ac,b] + F(j,k,i)[bc,a].
// Triplets with two equal indices need half of that: for i = j,
// F(i,k,j) = F(j,k,i) and F(i,i,k)[ab,c] = H[ab,c] + H[ba,c] with half the K
// extent, so U_abc = H[ab,c] + F(i,k,i)[ac,b] is formed and
// W_abc = U_abc + U_bac; for j = k, U_abc = F(i,j,j)[ab,c] + H[bc,a] and
// W_abc = U_abc + U_acb.  The energy kernel does that (exact) addition.
//
// GEMM kernel.  A work item is (128-row M tile, triplet and F, N chunk of at
// most 208 columns); it runs the RL products one after another, each over the
// whole K into one of two TMEM accumulators, while the drain warps reduce the
// previous one modulo m_l and add it to 64-bit sums.  Two registers per
// element hold 160 columns of the tile; the sums of the columns beyond live in
// the TMEM columns the accumulators leave free.
//
// Energy kernel.  Per tile orbit (edge 8) it loads the six W blocks as
// integers and evaluates the canonical points in FP64: the brackets of Eq. 1
// are differences of W, formed exactly in integers before conversion.
//
// Weak triplets.  The grid is common to all triplets, so W of one whose
// amplitudes or integrals are far below the others' keeps fewer bits, where FP64
// accumulation keeps them relative to each product.  The rounding error of a
// triplet's W follows from the norms of its rows.  The energy kernel sums, beside
// E[4]_ST, what E[4]_ST would be if W were 2^49 times that error everywhere, and
// the DMMA kernel forms the triplets below that again.
#include <algorithm>
#include <type_traits>

#include "tc_internal.cuh"
#include "tc_ptx.cuh"

namespace tc {
namespace {

constexpr int RL = 15;                       // moduli
// In pairs for the drain, the power of two last and alone.  The first of a pair
// packs its residue into a byte and is at most 253: with 255 the rounding of
// c * fl(1/255) gives +128 for sums c from -8454907 down (K above 512, residues
// of one sign), which a byte holds as -128.
constexpr int MODULI[RL] = {253, 257, 251, 255, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 256};
constexpr bool packed_fit() {
  for (int l = 0; l + 1 < RL; l += 2)
    if (MODULI[l] > 253) return false;
  return true;
}
static_assert(packed_fit(), "the first modulus of a pair packs into a byte");
constexpr int KMAX = 1024;                   // largest K whose residue products sum exactly in FP32
// |sum of three F| <= 3 * 2^(BITS_A + BITS_B + 2) < P / 2 = 2^117.16
constexpr int BITS_A = 57, BITS_B = 56;
constexpr int MROWS = 128;
constexpr int A_HALF = MROWS * 16;           // bytes of one A half (8 K values)
constexpr int HPS_MAX = 16;                  // most K halves of a pipeline stage
constexpr int NCMAX = 208;                   // widest N chunk
constexpr int REG_UNITS = 10;                // most units of 8 columns of a drain thread whose sums live in registers
constexpr int TM_COLS = NCMAX / 2 - 8 * REG_UNITS;   // columns whose sums live in TMEM
constexpr int TM_BASE = 512 - 4 * TM_COLS;   // first TMEM column of those sums (two halves, two words)
constexpr int MAX_STAGES = 10;
constexpr int NPROD = 3;
constexpr int THREADS = 384;                 // warps 0, 2, 3: copies; 1: MMA; 4 .. 11: drain
constexpr int DRAIN_WARPS = 8;
constexpr int SMEM_DYN_MAX = 232448 - 2048;
constexpr int NT = 8;                        // tile edge of the energy orbits
constexpr int NT2 = NT * NT, NT3 = NT2 * NT;
constexpr int EN_THREADS = 128, EN_CTAS = 5;   // per CTA, CTAs per SM
// A triplet's W has to be 2^49 times its error in the root mean square.  The bound
// of the error takes every row at its largest, 1 to 2 bits over what it is: with
// factors of 2^-9 to 1 per orbital, triplets at that edge among them, energies are
// as far from 80-bit references as the DMMA kernel's (at most 1.0e-15 and 9.7e-16
// of |E[4]| + |V r3(W) / D|), whose W is right to 2^-51.2 (K = 132) to 2^-50.4
// (K = 400).  On data of uniform size W is above 2^52 times the bound (50 shapes
// from o=2 v=9 to o=2 v=504 and o=6 v=290).  The bracket sum n4 of independent W
// of variance 1 has mean 72.
constexpr double WEAK_N4 = 72.0 * 0x1p98;

constexpr int ERR_TIMEOUT_FULL = 11, ERR_TIMEOUT_EMPTY = 12, ERR_TIMEOUT_ACCFULL = 13,
              ERR_TIMEOUT_ACCEMPTY = 14, ERR_TIMEOUT_TEARDOWN = 15;

// ---------------------------------------------------------------- constants of the residue system

constexpr int inv_mod(int a, int m) {
  int r = 1;
  for (int x = 1; x < m; ++x)
    if ((long long)(a % m) * x % m == 1) r = x;
  return r;
}
constexpr int pow2_mod(int e, int m) {
  int r = 1 % m;
  for (int i = 0; i < e; ++i) r = 2 * r % m;
  return r;
}
struct RnsConst {
  unsigned long long I[RL];        // (2^64 k_l - 1) / m_l (m_l = 256: 2^56)
  unsigned long long Ip[RL / 2];   // the same for the product of a pair
  unsigned long long off, offp;    // 0x4B400000 * (sum I_l), * (sum Ip + I of the last): the exponent bits that
                                   // magic-number integers leave in the sums
  float inv[RL], neg[RL];          // 1 / m_l, -m_l
  unsigned ca[RL][3], cb[RL][3];   // 2^(20 i) mod m_l, and times q_l / k_l mod m_l
  unsigned c16[RL];                // 2^16 mod m_l
  unsigned ha[RL], hb[RL];         // -(the images' bias 2^58, times the same) mod m_l
};
constexpr RnsConst make_const() {
  RnsConst c{};
  for (int l = 0; l < RL; ++l) {
    const int m = MODULI[l];
    int q = 1;                                     // P / m_l mod m_l
    for (int j = 0; j < RL; ++j)
      if (j != l) q = q * (MODULI[j] % m) % m;
    q = inv_mod(q, m);
    const int t64 = pow2_mod(64, m);
    const int k = t64 != 0 ? inv_mod(t64, m) : 1;  // 2^64 k = 1 mod m (m = 256: k = 1, no remainder)
    // I = (2^64 k - d) / m by long division over 64 zero bits
    unsigned long long quo = 0, rem = (unsigned long long)k;
    for (int b = 0; b < 64; ++b) {
      rem *= 2;
      quo *= 2;
      if (rem >= (unsigned long long)m) { quo += rem / m; rem %= m; }
    }
    c.I[l] = quo;
    c.off += 0x4B400000ULL * quo;
    if (l % 2 == 0 && l + 1 < RL) {                // K = (2^64)^-1 mod m m' by CRT from k mod m and k' mod m'
      const int m2 = MODULI[l + 1], M = m * m2, k2 = inv_mod(pow2_mod(64, m2), m2);
      unsigned long long K = (unsigned long long)((long long)k * m2 % M * inv_mod(m2, m) % M +
                                                  (long long)k2 * m % M * inv_mod(m, m2) % M) % (unsigned long long)M;
      unsigned long long qp = 0;
      for (int b = 0; b < 64; ++b) {
        K *= 2;
        qp *= 2;
        if (K >= (unsigned long long)M) { qp += K / M; K %= M; }
      }
      c.Ip[l / 2] = qp;
      c.offp += 0x4B400000ULL * qp;
    } else if (l + 1 == RL) {
      c.offp += 0x4B400000ULL * quo;
    }
    c.inv[l] = 1.0f / (float)m;
    c.neg[l] = -(float)m;
    const int g = q * inv_mod(k, m) % m;
    for (int i = 0; i < 3; ++i) {
      c.ca[l][i] = (unsigned)pow2_mod(20 * i, m);
      c.cb[l][i] = (unsigned)(g * pow2_mod(20 * i, m) % m);
    }
    c.c16[l] = (unsigned)pow2_mod(16, m);
    const int bias = pow2_mod(58, m);
    c.ha[l] = (unsigned)((m - bias) % m);
    c.hb[l] = (unsigned)((m - g * bias % m) % m);
  }
  return c;
}
__constant__ RnsConst RC = make_const();

// P / 2^64 and its square, as doubles (the value of a unit of W's fraction).
constexpr double p_scaled() {
  // the product of the moduli in two exact halves: 8 and 7 of them below 2^64
  unsigned long long lo = 1, hi = 1;
  for (int l = 0; l < 8; ++l) lo *= (unsigned long long)MODULI[l];
  for (int l = 8; l < RL; ++l) hi *= (unsigned long long)MODULI[l];
  return ((double)lo * 0x1p-64) * (double)hi;
}
constexpr double C_P = p_scaled();

// ---------------------------------------------------------------- scales

// Arrays of the scale search inside a job's scratch: squared norms of the
// operand rows, their maxima per array and orbital as IEEE bits, exponents.
// Arrays: 0 ovvv[p][x][y][:], 1 t2[p][:][x][y] (hole), 2 t2[r][q][z][:], 3 ovoo[r][z][q][:].
struct Scales {
  double *ra, *rt, *rb, *rh;       // [o][v][v], [o][v][v], [o][o][v], [o][v][o]
  unsigned long long *nv, *no;     // [4][v], [4][o]: largest squared norm of the array's rows with that orbital
  int *dv, *du;                    // [v], [o]: exponents that suit every array's largest rows, one orbital at a time
  int *fv, *fu;                    // [v], [o]: share of them, in 256ths, that suits every row
  int *ev, *uo;                    // [v], [o]: the exponents taken
  int *sh;                         // [5]: shifts of the four operands and SS; sh[5]: 1 if any of dv, du is not 0
  unsigned long long *pm, *qm;     // with exponents, [2][o]: largest scaled squared norm of arrays 0, 1 by p; [2][o][o]: of
                                   // arrays 2, 3 by (r, q)
  double *nz;                      // squared error of W in units of its fraction: [0] of any triplet without exponents;
                                   // with them [1 + p] and [1 + o + r o + q], summed over a triplet's p and (r, q)
  int *flag;                       // 1: inputs out of the range the integer grid covers
};

// 0 for a zero of either sign.
__device__ __forceinline__ unsigned magnitude(double x) {
  return (unsigned)__double2hiint(x) << 1 | (unsigned)__double2loint(x);
}

// Squared norms of the operand rows, one warp per row:
//   [0, n0)   ovvv[p][x][y][:]    (n0 = o v v, length v)
//   [.., n1)  t2[r][q][z][:]      (o o v, length v)
//   [.., n2)  ovoo[r][z][q][:]    (o v o, length o)
//   then, one thread per column, t2[p][:][x][y] (o v v, length o)
// The maxima per orbital are collected in shared memory first (whole calls at
// o=6 v=36 270 us; 283 us with a look at the global maxima for every row).  The
// FP64 pipe bounds it at o=20 v=200, so zeros are told by their bits (FP64
// comparisons: 0.5 ms more).  A row whose squares all underflow gets the smallest
// denormal instead of the 0 of a row of zeros: an array of such rows is out of
// the grid's range.
__global__ void rns_norms(Inputs in, int o, int v, Scales s) {
  const long long n0 = (long long)o * v * v, n1 = n0 + (long long)o * o * v, n2 = n1 + (long long)o * v * o;
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  extern __shared__ unsigned long long top[];              // [4][v] and [4][o], as s.nv and s.no
  unsigned long long *const tv = top, *const to = top + 4 * v;
  for (int x = threadIdx.x; x < 4 * (v + o); x += blockDim.x) top[x] = 0;
  __syncthreads();
  auto up = [](double a, unsigned long long *m0, unsigned long long *m1, unsigned long long *m2) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    unsigned long long *const m[3] = {m0, m1, m2};
#pragma unroll
    for (int i = 0; i < 3; ++i)                            // most rows raise no maximum
      if (b > *(volatile unsigned long long *)m[i]) atomicMax(m[i], b);
  };
  for (long long w = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < n2; w += warps) {
    const double *src;
    int len;
    if (w < n0)      { src = in.ovvv + w * v; len = v; }
    else if (w < n1) { src = in.t2 + (w - n0) * v; len = v; }
    else             { src = in.ovoo + (w - n1) * o; len = o; }
    double a = 0.0;
    unsigned any = 0;                                      // by bits: a comparison would take the FP64 pipe, which bounds this
    for (int k = lane; k < len; k += 32) {
      const double t = src[k];
      any |= magnitude(t);
      a = fma(t, t, a);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    any = __any_sync(0xffffffffu, any != 0);
    if (any && magnitude(a) == 0) a = __longlong_as_double(1);
    if (lane == 0) {                                       // row numbers fit 32 bits (o, v <= 504)
      if (w < n0) {
        const unsigned e = (unsigned)w;
        s.ra[w] = a;
        up(a, to + e / v / v, tv + e / v % v, tv + e % v);
      } else if (w < n1) {
        const unsigned e = (unsigned)(w - n0);
        s.rb[e] = a;
        up(a, to + 2 * o + e / v / o, to + 2 * o + e / v % o, tv + 2 * v + e % v);
      } else {
        const unsigned e = (unsigned)(w - n1);
        s.rh[e] = a;
        up(a, to + 3 * o + e / o / v, to + 3 * o + e % o, tv + 3 * v + e / o % v);
      }
    }
  }
  const long long vv = (long long)v * v;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n0; e += (long long)gridDim.x * blockDim.x) {
    const long long p = e / vv, xy = e - p * vv;
    double a = 0.0;
    unsigned any = 0;
    for (int l = 0; l < o; ++l) {
      const double t = in.t2[(p * o + l) * vv + xy];
      any |= magnitude(t);
      a = fma(t, t, a);
    }
    if (any && magnitude(a) == 0) a = __longlong_as_double(1);
    s.rt[e] = a;
    up(a, to + o + p, tv + v + (unsigned)xy / v, tv + v + (unsigned)xy % v);
  }
  __syncthreads();
  for (int x = threadIdx.x; x < 4 * (v + o); x += blockDim.x) {
    unsigned long long *const m = x < 4 * v ? s.nv + x : s.no + (x - 4 * v);
    if (top[x] > *(volatile unsigned long long *)m) atomicMax(m, top[x]);
  }
}

// Exponents.  A row of array k may be scaled up by its slack, the powers of two
// between its norm and the array's largest (from binary exponents alone, so
// scaling an input array by a power of two changes none of them).  d of an
// orbital is the least slack of the rows that hold it, over all four arrays: 0
// where any array has a row of full size.  A row holds three orbitals, so the
// sum of their d may exceed its slack; each orbital then takes the share (slack +
// SPARE) / sum of its d, the smallest over its rows, which keeps every row within
// 2^SPARE of the array's largest.  Where all arrays carry one factor per orbital,
// the shares stay 1 and the exponents take it out (SPARE = 0: some row's scatter
// halves them).  An exponent from the integrals alone scales amplitudes up with
// it: W lost all digits when one orbital's ovvv was 2^-24 of the others'.
constexpr int D_MAX = 16, SPARE = 2;
constexpr int NO_ROW = 1 << 20;                           // slack of a row of zeros

// Slack of a squared norm (IEEE bits) against the array's largest.
__device__ __forceinline__ int slack(unsigned long long bits, int emax) {
  return bits == 0 ? NO_ROW : max(emax - ((int)(bits >> 52) - 1023), 0) / 2;
}
__device__ __forceinline__ int expo(unsigned long long bits) { return (int)(bits >> 52) - 1023; }

// Each array's largest squared norm (IEEE bits), to every thread of the CTA.
__device__ void array_max(int v, const Scales &s, unsigned long long (&mb)[4]) {
  __shared__ unsigned long long m[4];
  if (threadIdx.x < 4) m[threadIdx.x] = 0;
  __syncthreads();
  for (int k = 0; k < 4; ++k)
    for (int x = threadIdx.x; x < v; x += blockDim.x) {
      const unsigned long long b = __ldcg(s.nv + (size_t)k * v + x);
      if (b > *(volatile unsigned long long *)(m + k)) atomicMax(m + k, b);
    }
  __syncthreads();
  for (int k = 0; k < 4; ++k) mb[k] = m[k];
  __syncthreads();
}

// d of every orbital, shares of 256 / 256, by one CTA.
__device__ void wanted(int o, int v, const Scales &s) {
  unsigned long long mb[4];
  array_max(v, s, mb);
  if (threadIdx.x == 0) s.sh[5] = 0;
  __syncthreads();
  for (int x = threadIdx.x; x < v + o; x += blockDim.x) {
    const bool vir = x < v;
    int d = NO_ROW;
    for (int k = 0; k < 4; ++k)
      d = min(d, slack(__ldcg(vir ? s.nv + (size_t)k * v + x : s.no + (size_t)k * o + (x - v)), expo(mb[k])));
    d = d == NO_ROW ? 0 : min(d, D_MAX);
    (vir ? s.dv[x] : s.du[x - v]) = d;
    (vir ? s.fv[x] : s.fu[x - v]) = 256;
    if (d) s.sh[5] = 1;
  }
}

// Shares: every row's slack against the sum of its orbitals' d.
__device__ void shares(int o, int v, const Scales &s) {
  if (__ldcg(s.sh + 5) == 0) return;
  unsigned long long mb[4];
  array_max(v, s, mb);
  const long long vv = (long long)v * v, n0 = (long long)o * vv, n1 = (long long)o * o * v;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, st = (long long)gridDim.x * blockDim.x;
  auto row = [&](double n, int k, const int *d0, const int *d1, const int *d2, int *f0, int *f1, int *f2) {
    const int sum = __ldcg(d0) + __ldcg(d1) + __ldcg(d2);
    const int sl = slack((unsigned long long)__double_as_longlong(n), expo(mb[k])) + SPARE;
    if (sl >= sum) return;
    const int f = 256 * sl / sum;
    int *const ff[3] = {f0, f1, f2};
    for (int i = 0; i < 3; ++i)
      if (f < *(volatile int *)ff[i]) atomicMin(ff[i], f);
  };
  for (long long e = t; e < n0; e += st) {
    const int p = (int)(e / vv), x = (int)(e % vv / v), y = (int)(e % v);
    row(s.ra[e], 0, s.du + p, s.dv + x, s.dv + y, s.fu + p, s.fv + x, s.fv + y);
    row(s.rt[e], 1, s.du + p, s.dv + x, s.dv + y, s.fu + p, s.fv + x, s.fv + y);
  }
  for (long long e = t; e < n1; e += st) {
    const int z = (int)(e % v), q = (int)(e / v % o), r = (int)(e / v / o);
    row(s.rb[e], 2, s.du + r, s.du + q, s.dv + z, s.fu + r, s.fu + q, s.fv + z);
    const int q2 = (int)(e % o), z2 = (int)(e / o % v), r2 = (int)(e / o / v);
    row(s.rh[e], 3, s.du + r2, s.du + q2, s.dv + z2, s.fu + r2, s.fu + q2, s.fv + z2);
  }
}

__device__ __forceinline__ int taken(const int *d, const int *f, int x) { return __ldcg(d + x) * __ldcg(f + x) >> 8; }
__device__ __forceinline__ double pow4(int e) { return __longlong_as_double((long long)(1023 + 2 * e) << 52); }   // |e| <= 500

// Largest scaled squared norms by p (arrays 0, 1; a warp takes the rows of one
// (p, x)) and by (r, q) (arrays 2, 3; a warp per pair).
__device__ void scaled_max(int o, int v, const Scales &s) {
  if (__ldcg(s.sh + 5) == 0) return;
  const int lane = threadIdx.x & 31, w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int warps = gridDim.x * (blockDim.x >> 5);
  auto bits = [](double n, int e) { return (unsigned long long)__double_as_longlong(n * pow4(e)); };
  auto top = [](unsigned long long b) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, off));
    return b;
  };
  for (int w = w0; w < o * v; w += warps) {
    const int p = w / v, e0 = taken(s.du, s.fu, p) + taken(s.dv, s.fv, w % v);
    unsigned long long b0 = 0, b1 = 0;
    for (int y = lane; y < v; y += 32) {
      const int e = e0 + taken(s.dv, s.fv, y);
      b0 = max(b0, bits(s.ra[(long long)w * v + y], e));
      b1 = max(b1, bits(s.rt[(long long)w * v + y], e));
    }
    b0 = top(b0);
    b1 = top(b1);
    if (lane == 0) {
      if (b0 > *(volatile unsigned long long *)(s.pm + p)) atomicMax(s.pm + p, b0);
      if (b1 > *(volatile unsigned long long *)(s.pm + o + p)) atomicMax(s.pm + o + p, b1);
    }
  }
  for (int w = w0; w < o * o; w += warps) {
    const int r = w / o, q = w % o, e0 = taken(s.du, s.fu, r) + taken(s.du, s.fu, q);
    unsigned long long b2 = 0, b3 = 0;
    for (int z = lane; z < v; z += 32) {
      const int e = e0 + taken(s.dv, s.fv, z);
      b2 = max(b2, bits(s.rb[(long long)w * v + z], e));
      b3 = max(b3, bits(s.rh[((long long)r * v + z) * o + q], e));
    }
    b2 = top(b2);
    b3 = top(b3);
    if (lane == 0) {
      s.qm[w] = b2;
      s.qm[o * o + w] = b3;
    }
  }
}

// The exponents taken.
__device__ void take_exps(int o, int v, const Scales &s) {
  for (int x = threadIdx.x; x < v; x += blockDim.x) s.ev[x] = taken(s.dv, s.fv, x);
  for (int p = threadIdx.x; p < o; p += blockDim.x) s.uo[p] = taken(s.du, s.fu, p);
}

// Each array's largest scaled squared norm (IEEE bits), to every thread of the CTA.
__device__ void array_scaled_max(int o, int v, const Scales &s, unsigned long long (&mb)[4]) {
  if (__ldcg(s.sh + 5) == 0) {
    array_max(v, s, mb);
    return;
  }
  __shared__ unsigned long long m[4];
  if (threadIdx.x < 4) m[threadIdx.x] = 0;
  __syncthreads();
  for (int x = threadIdx.x; x < 2 * (o + o * o); x += blockDim.x) {
    const unsigned long long b = __ldcg(x < 2 * o ? s.pm + x : s.qm + (x - 2 * o));
    unsigned long long *const k = m + (x < 2 * o ? x / o : 2 + (x - 2 * o) / (o * o));
    if (b > *(volatile unsigned long long *)k) atomicMax(k, b);
  }
  __syncthreads();
  for (int k = 0; k < 4; ++k) mb[k] = m[k];
  __syncthreads();
}

// Shifts of the four operands (one CTA).  A row of norm n is scaled to at
// most 2^BITS: i = ceil(log2 of the largest norm).  Particle and hole products
// share the grid (sa + sb = sah + sbh = SS); the pair with room to spare is
// scaled down.  Arrays of zeros take shift 0; inputs whose norms leave
// [2^-100, 2^100] or are not finite set the flag.
__device__ void shifts(const Scales &s, const unsigned long long (&mb)[4]) {
  int i[4];
  bool any[4];
  if (threadIdx.x != 0) return;
  for (int k = 0; k < 4; ++k) {
    any[k] = mb[k] != 0;
    const int e = any[k] ? expo(mb[k]) : 0;
    if (any[k] && (e < -200 || e > 200)) *s.flag = 1;
    i[k] = (e + 202) / 2 - 100;                    // ceil((e + 1) / 2)
  }
  const bool part = any[0] && any[2], hole = any[1] && any[3];
  int sa = BITS_A - i[0], sb = BITS_B - i[2], sah = BITS_A - i[1], sbh = BITS_B - i[3];
  if (part && hole) {
    const int d = (sa + sb) - (sah + sbh);
    if (d > 0) { sa -= d / 2; sb -= d - d / 2; }
    else { sah -= (-d) / 2; sbh -= (-d) - (-d) / 2; }
  } else if (hole) {
    sa = sah; sb = sbh;                            // one particle operand is all zeros
  } else {
    sah = sa; sbh = sb;
  }
  // a zero operand's partner may hold any values: its rows stay within the same bound
  s.sh[0] = any[0] ? min(sa, BITS_A - i[0]) : sa;
  s.sh[1] = any[1] ? min(sah, BITS_A - i[1]) : sah;
  s.sh[2] = any[2] ? min(sb, BITS_B - i[2]) : sb;
  s.sh[3] = any[3] ? min(sbh, BITS_B - i[3]) : sbh;
  s.sh[4] = sa + sb;
}

// W's squared error, from the rounding of the operands to the grid: an element of
// a row is off by a variance of 1/12, a product by (|a|^2 + |b|^2) / 12 in units
// of the grid, C_P of which make a unit of W's fraction; 1 more for each of the
// three F's own fraction (one CTA).
__device__ void noise(int o, const Scales &s, const unsigned long long (&mb)[4]) {
  auto scaled = [&](unsigned long long b, int k) {
    return __longlong_as_double((long long)b) * pow4(s.sh[k]) * (1.0 / (12.0 * C_P * C_P));
  };
  if (threadIdx.x == 0) {
    double n = 0.0;
    for (int k = 0; k < 4; ++k) n += scaled(mb[k], k);
    s.nz[0] = 6.0 * n + 3.0;
  }
  if (s.sh[5] == 0) return;
  for (int p = threadIdx.x; p < o; p += blockDim.x)
    s.nz[1 + p] = 2.0 * (scaled(__ldcg(s.pm + p), 0) + scaled(__ldcg(s.pm + o + p), 1));
  for (int w = threadIdx.x; w < o * o; w += blockDim.x)
    s.nz[1 + o + w] = scaled(__ldcg(s.qm + w), 2) + scaled(__ldcg(s.qm + o * o + w), 3);
}

// The last step, by one CTA: exponents, shifts, errors.
__device__ void finish_scales(int o, int v, const Scales &s) {
  unsigned long long mb[4];
  take_exps(o, v, s);
  array_scaled_max(o, v, s, mb);
  shifts(s, mb);
  __syncthreads();
  noise(o, s, mb);
}

__global__ void rns_wanted(int o, int v, Scales s) { wanted(o, v, s); }
__global__ void rns_shares(int o, int v, Scales s) { shares(o, v, s); }
__global__ void rns_scaled_max(int o, int v, Scales s) { scaled_max(o, v, s); }
__global__ void rns_scales(int o, int v, Scales s) { finish_scales(o, v, s); }

// All four steps by one CTA, for jobs where their launches take longer than
// their work: up to SCALES_ONE rows of ovvv.
// (Preparation, one launch against four: o=6 v=36 40 / 50 us, o=9 v=77 156 / 166,
// o=8 v=104 218 / 230; where there are exponents 68 / 58, 258 / 173 and 428 / 241.)
constexpr long long SCALES_ONE = 1 << 16;
__global__ void __launch_bounds__(1024) rns_scales_one(int o, int v, Scales s) {
  wanted(o, v, s);
  __syncthreads();
  shares(o, v, s);
  __syncthreads();
  scaled_max(o, v, s);
  __syncthreads();
  finish_scales(o, v, s);
}

// ---------------------------------------------------------------- operand images

// The operands of tc_split.cu in the same K-major layout, with the RL residues
// of the scaled integer in place of the slices, modulus-major: a half is rows x
// 16 bytes, [p][m tile][modulus][half] (A) and [r][q][N chunk][modulus][half] (B).

__device__ __forceinline__ unsigned long long pack2(float x) {
  const unsigned long long b = __float_as_uint(x);
  return b << 32 | b;
}

// 8 values times 2^ex rounded to integers, biased to be positive, in three limbs of 20 bits.
struct Limbs {
  unsigned u[8][3];
};
__device__ __forceinline__ Limbs limbs(const double (&x)[8], int ex) {
  const double f = __longlong_as_double((long long)(1023 + ex) << 52);
  Limbs r;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned long long b = (unsigned long long)(__double2ll_rn(x[k] * f) + (1LL << 58));
    r.u[k][0] = (unsigned)b & 0xFFFFF;
    r.u[k][1] = (unsigned)(b >> 20) & 0xFFFFF;
    r.u[k][2] = (unsigned)(b >> 40);
  }
  return r;
}

// The residues modulo m_l, at most 128 in magnitude, as 8 BF16: the limbs
// folded below 2^22 in integers, then t - m round(t / m) in packed FP32.
__device__ __forceinline__ uint4 residues8(const Limbs &x, int l, const unsigned (*c)[3], unsigned h) {
  const unsigned c0 = c[l][0], c1 = c[l][1], c2 = c[l][2], c16 = RC.c16[l];
  const unsigned long long inv = pack2(RC.inv[l]), neg = pack2(RC.neg[l]);
  unsigned w[8];
#pragma unroll
  for (int k = 0; k < 8; k += 2) {
    unsigned t[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      t[e] = x.u[k + e][0] * c0 + x.u[k + e][1] * c1 + x.u[k + e][2] * c2 + h;       // < 2^30
      t[e] = ((t[e] & 0xFFFF) + (t[e] >> 16) * c16) | 0x4B000000;                    // 2^23 + (t < 2^22)
    }
    asm("{\n .reg .b64 c, k;\n mov.b64 c, {%2, %3};\n add.rn.f32x2 c, c, %6;\n fma.rn.f32x2 k, c, %4, %7;\n"
        " add.rn.f32x2 k, k, %8;\n fma.rn.f32x2 c, k, %5, c;\n mov.b64 {%0, %1}, c;\n}\n"
        : "=r"(w[k]), "=r"(w[k + 1])
        : "r"(t[0]), "r"(t[1]), "l"(inv), "l"(neg), "l"(0xCB000000CB000000ULL), "l"(0x4B4000004B400000ULL),
          "l"(0xCB400000CB400000ULL));
  }
  uint4 q;                                              // the leading half of each float is its BF16
  q.x = __byte_perm(w[0], w[1], 0x7632);
  q.y = __byte_perm(w[2], w[3], 0x7632);
  q.z = __byte_perm(w[4], w[5], 0x7632);
  q.w = __byte_perm(w[6], w[7], 0x7632);
  return q;
}

// A images, both orders of the virtual pair at once.  vv: (p x|y f) with K f =
// ovvv[p][x][y][f] goes to row (x, y) of out and row (y, x) of outT; else
// t_pl^xy with K l = t2[p][l][x][y], likewise (hc2 and its transpose hc).  A warp takes 8 x by 4 y, so its
// stores cover 64 and 128 contiguous bytes; a CTA's warps take consecutive K
// halves of the same pairs.  The rows behind the last pair of the last M tile
// are zeroed by the trailing warps.  Making each residue once instead of once
// per image, with three limbs and packed FP32 for the reduction, took the
// preparation of o=20 v=200 from 3.8 to 2.8 ms (9.6 GB of images).
// need (may be NULL): only occupied indices p with need[p (o + 1)].
__device__ void rns_image_a(bool vv, const double *__restrict__ src, RnsGeom G, Scales s,
                            const unsigned char *__restrict__ need, unsigned char *__restrict__ out,
                            unsigned char *__restrict__ outT) {
  const int o = G.o, v = G.v, nh = vv ? G.hv : G.ho, kmax = vv ? v : o;
  const int nx = (v + 7) / 8, ny = (v + 3) / 4;
  const int lane = threadIdx.x & 31;
  const long long per_p = (long long)nx * ny * nh, warps = (long long)gridDim.x * (blockDim.x >> 5);
  const int shift = s.sh[vv ? 0 : 1];
  const long long rows = (long long)v * v;
  const int tail = (int)(G.mt * (long long)MROWS - rows);
  const long long tails = tail ? (long long)o * RL * nh * ((tail + 31) / 32) : 0;
  auto at = [&](unsigned char *b, long long p, long long row, int l, int h) {
    return (uint4 *)(b + (((p * G.mt + row / MROWS) * RL + l) * nh + h) * A_HALF + row % MROWS * 16);
  };
  for (long long w = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < o * per_p + tails; w += warps) {
    if (w >= o * per_p) {
      long long e = w - o * per_p;
      const int part = (int)(e % ((tail + 31) / 32));
      e /= (tail + 31) / 32;
      const int h = (int)(e % nh), l = (int)(e / nh % RL);
      const long long p = e / nh / RL;
      if (part * 32 + lane < tail) {
        *at(out, p, rows + part * 32 + lane, l, h) = make_uint4(0, 0, 0, 0);
        *at(outT, p, rows + part * 32 + lane, l, h) = make_uint4(0, 0, 0, 0);
      }
      continue;
    }
    const int p = (int)(w / per_p);
    if (need && !need[(long long)p * (o + 1)]) continue;
    const long long e = w - p * per_p;
    const int h = (int)(e % nh), px = (int)(e / nh / ny), py = (int)(e / nh % ny);
    const int x = px * 8 + (lane & 7), y = py * 4 + (lane >> 3);
    if (x >= v || y >= v) continue;
    double val[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = h * 8 + u;
      val[u] = k >= kmax ? 0.0
             : vv ? src[(((long long)p * v + x) * v + y) * v + k] : src[(((long long)p * o + k) * v + x) * v + y];
    }
    const Limbs lb = limbs(val, shift + s.ev[x] + s.ev[y] + s.uo[p]);
    uint4 *d = at(out, p, (long long)x * v + y, 0, h), *dT = at(outT, p, (long long)y * v + x, 0, h);
    const size_t step = (size_t)nh * A_HALF / sizeof(uint4);
#pragma unroll 1
    for (int l = 0; l < RL; ++l) {
      const uint4 q = residues8(lb, l, RC.ca, RC.ha[l]);
      d[l * step] = q;
      dT[l * step] = q;
    }
  }
}

// B images: row z, K f: t_rq^zf = t2[r][q][z][f] (vv), or K l: -(r z|q l) =
// -ovoo[r][z][q][l]; rows or K values outside are zero.  One thread per (K
// half, row).  need (may be NULL): only occupied pairs with need[r o + q].
__device__ void rns_image_b(bool vv, const double *__restrict__ src, RnsGeom G, Scales s,
                            const unsigned char *__restrict__ need, unsigned char *__restrict__ out) {
  const int o = G.o, v = G.v, rows = G.nc, nh = vv ? G.hv : G.ho, kmax = vv ? v : o;
  const size_t half_bytes = (size_t)rows * 16;
  const long long total = (long long)o * o * G.nch * nh * rows;
  const int shift = s.sh[vv ? 2 : 3];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e % rows), h = (int)(e / rows % nh);
    const long long rest = e / rows / nh;
    const int nci = (int)(rest % G.nch), qq = (int)(rest / G.nch % o), rr = (int)(rest / G.nch / o);
    if (need && !need[rr * o + qq]) continue;
    const int z = nci * rows + r;
    double val[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = h * 8 + u;
      val[u] = z >= v || k >= kmax ? 0.0
             : vv ? src[(((long long)rr * o + qq) * v + z) * v + k] : -src[(((long long)rr * v + z) * o + qq) * o + k];
    }
    const Limbs lb = limbs(val, shift + (z < v ? s.ev[z] : 0) + s.uo[rr] + s.uo[qq]);
    uint4 *d = (uint4 *)(out + ((rest * RL) * nh + h) * half_bytes + (size_t)r * 16);
    const size_t step = (size_t)nh * half_bytes / sizeof(uint4);
#pragma unroll 1
    for (int l = 0; l < RL; ++l) d[l * step] = residues8(lb, l, RC.cb, RC.hb[l]);
  }
}

// All images in one launch, one task per blockIdx.y.
__global__ void rns_images(RnsLayout L, Inputs in, Scales s, const unsigned char *__restrict__ need,
                           unsigned char *__restrict__ b) {
  switch (blockIdx.y) {
    case 0: rns_image_a(true, in.ovvv, L.g, s, need, b + L.pa, b + L.pa2); break;
    case 1: rns_image_b(true, in.t2, L.g, s, need, b + L.tb); break;
    case 2: rns_image_a(false, in.t2, L.g, s, need, b + L.hc2, b + L.hc); break;
    case 3: rns_image_b(false, in.ovoo, L.g, s, need, b + L.hb); break;
  }
}

// ---------------------------------------------------------------- GEMM kernel

__device__ __forceinline__ void mma_bf16(uint32_t dcol, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               :: "r"(dcol), "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_ld8u(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr) : "memory");
}
// Wait for this thread's TMEM loads; naming the loaded registers keeps their uses behind it.
__device__ __forceinline__ void tmem_wait_ld8(float (&v)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])
               :: "memory");
}
__device__ __forceinline__ void tmem_wait_ld8u(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
               :: "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void prod_bar() { asm volatile("bar.sync 2, %0;" :: "n"(NPROD * 32) : "memory"); }

// Item q of a job -> (M tile, unit of the block, N chunk), M-tile-major.  A
// unit is one F of one triplet: the triplet's index (bits 3 and up), whether it
// runs half of the K segments (bit 2), F number (bits 0, 1).
struct RnItem {
  int m, tl, f, half, nci;
  int p, q, r;
};
__device__ __forceinline__ RnItem rn_decode(const RnJob &J, long long x) {
  RnItem t;
  t.nci = (int)(x % J.g.nch);
  x /= J.g.nch;
  const int u = J.unit[x % J.nu];
  t.m = (int)(x / J.nu);
  t.tl = (u >> 3) - J.t0;
  t.half = (u >> 2) & 1;
  t.f = u & 3;
  const int4 tr = J.trip[J.t0 + t.tl];
  t.p = t.f == 2 ? tr.y : tr.x;
  t.q = t.f == 0 ? tr.y : tr.z;
  t.r = t.f == 0 ? tr.z : (t.f == 1 ? tr.y : tr.x);
  return t;
}

// The residue modulo m of an FP32 accumulator value c (an exact integer) is
// t = c - m round(c / m), exact; adding 1.5 * 2^23 puts an integer into the low
// bits of its float (the exponent bits this leaves are taken out once at the
// end).  Packed FP32 instructions, two columns at a time.
struct ModConst {
  unsigned long long inv, neg;     // (1/m, 1/m), (-m, -m)
  unsigned long long m1, m2;       // pairs: (m of this modulus, twice), (m of its partner, twice)
  uint32_t ilo, ihi;               // I_l, or Ip
};
constexpr unsigned long long MAG2 = 0x4B4000004B400000ULL, NMAG2 = 0xCB400000CB400000ULL;
// t + mag of two columns (mag: MAG2, or with 128 added: the low byte is t + 128)
__device__ __forceinline__ void residues(float c0, float c1, const ModConst &m, unsigned long long mag, uint32_t &u0,
                                         uint32_t &u1) {
  asm("{\n .reg .b64 c, k, t;\n mov.b64 c, {%2, %3};\n fma.rn.f32x2 k, c, %4, %6;\n add.rn.f32x2 k, k, %7;\n"
      " fma.rn.f32x2 t, k, %5, c;\n add.rn.f32x2 t, t, %8;\n mov.b64 {%0, %1}, t;\n}\n"
      : "=r"(u0), "=r"(u1)
      : "f"(c0), "f"(c1), "l"(m.inv), "l"(m.neg), "l"(MAG2), "l"(NMAG2), "l"(mag));
}
// Second modulus of a pair: b0, b1 hold 2^23 + 128 + t of the first; u = t m2 +
// t' m1 is the pair's residue in units of 1 / (m1 m2), below 2^17.
__device__ __forceinline__ void residues_pair(float c0, float c1, uint32_t b0, uint32_t b1, const ModConst &m,
                                              uint32_t &u0, uint32_t &u1) {
  asm("{\n .reg .b64 c, k, t, b;\n mov.b64 c, {%2, %3};\n mov.b64 b, {%4, %5};\n fma.rn.f32x2 k, c, %6, %8;\n"
      " add.rn.f32x2 k, k, %9;\n add.rn.f32x2 b, b, %10;\n fma.rn.f32x2 t, k, %7, c;\n fma.rn.f32x2 b, b, %11, %8;\n"
      " fma.rn.f32x2 t, t, %12, b;\n mov.b64 {%0, %1}, t;\n}\n"
      : "=r"(u0), "=r"(u1)
      : "f"(c0), "f"(c1), "r"(b0), "r"(b1), "l"(m.inv), "l"(m.neg), "l"(MAG2), "l"(NMAG2), "l"(0xCB000080CB000080ULL),
        "l"(m.m1), "l"(m.m2));
}
// acc += u I (mod 2^64)
__device__ __forceinline__ void add_frac(unsigned long long &acc, uint32_t u, const ModConst &m) {
  asm("{\n .reg .b32 lo, hi;\n mad.wide.u32 %0, %1, %2, %0;\n mov.b64 {lo, hi}, %0;\n mad.lo.u32 hi, %1, %3, hi;\n"
      " mov.b64 %0, {lo, hi};\n}\n"
      : "+l"(acc) : "r"(u), "r"(m.ilo), "r"(m.ihi));
}

// One finished product of an item: the tile row's columns are reduced modulo
// m_l and added to the 64-bit sums.  The 64-bit multiply-add is the dear part
// (8.4 of 12.7 clocks a column and warp), so moduli go in pairs: the first
// (MODE 0) only packs its residues into bytes, the second (MODE 1) forms the
// pair's 17-bit residue and adds that; MODE 2 is a modulus alone.  Columns
// whose sums live in TMEM always take that form.  UN, the units of 8 columns in
// registers, is fixed at compile time and columns behind the chunk are reduced
// along: a test around every unit costs more (18.5 clocks a column and modulus
// instead of 11.7).
template <int MODE, int UN>
__device__ __forceinline__ void drain_product(int l, int my, uint32_t tacc, uint32_t tmp,
                                              unsigned long long (&part)[8 * UN], uint32_t (&pk)[2 * UN]) {
  ModConst mc;
  mc.inv = pack2(RC.inv[l]);
  mc.neg = pack2(RC.neg[l]);
  if (MODE == 1) {
    mc.m1 = pack2(-RC.neg[l]);                             // t times the partner's modulus: this one
    mc.m2 = pack2(-RC.neg[l - 1]);
  }
  const unsigned long long I = MODE == 1 ? RC.Ip[l >> 1] : RC.I[l];
  mc.ilo = (uint32_t)I;
  mc.ihi = (uint32_t)(I >> 32);
  float c[2][8];
  tmem_ld8(tacc, c[0]);
  tmem_wait_ld8(c[0]);
#pragma unroll
  for (int u = 0; u < UN; ++u) {
    {
      if (u + 1 < UN) tmem_ld8(tacc + 8 * (u + 1), c[(u + 1) & 1]);
      const float (&x)[8] = c[u & 1];
      if (MODE == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t r[4];
          residues(x[4 * h], x[4 * h + 1], mc, MAG2 + 0x0000008000000080ULL, r[0], r[1]);
          residues(x[4 * h + 2], x[4 * h + 3], mc, MAG2 + 0x0000008000000080ULL, r[2], r[3]);
          pk[2 * u + h] = __byte_perm(__byte_perm(r[0], r[1], 0x0040), __byte_perm(r[2], r[3], 0x0040), 0x5410);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          uint32_t u0, u1;
          if (MODE == 1) {
            const uint32_t b = pk[2 * u + e / 4];
            residues_pair(x[e], x[e + 1], __byte_perm(b, 0x4B000000, 0x7650 + (e & 2)), __byte_perm(b, 0x4B000000, 0x7651 + (e & 2)),
                          mc, u0, u1);
          } else {
            residues(x[e], x[e + 1], mc, MAG2, u0, u1);
          }
          add_frac(part[8 * u + e], u0, mc);
          add_frac(part[8 * u + e + 1], u1, mc);
        }
      }
      if (u + 1 < UN) tmem_wait_ld8(c[(u + 1) & 1]);
    }
  }
  if (UN == REG_UNITS && my > UN) {
    ModConst ms = mc;
    ms.ilo = (uint32_t)RC.I[l];
    ms.ihi = (uint32_t)(RC.I[l] >> 32);
#pragma unroll 1
    for (int u = UN; u < my; ++u) {
      const uint32_t ts = tmp + 16 * (uint32_t)(u - UN);
      float x[8];
      uint32_t plo[8] = {}, phi[8] = {};
      tmem_ld8(tacc + 8 * u, x);
      if (l > 0) {
        tmem_ld8u(ts, plo);
        tmem_ld8u(ts + 8, phi);
      }
      tmem_wait_ld8u(plo, phi);
      tmem_wait_ld8(x);
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        uint32_t r[2];
        residues(x[e], x[e + 1], ms, MAG2, r[0], r[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          unsigned long long p = (unsigned long long)phi[e + h] << 32 | plo[e + h];
          add_frac(p, r[h], ms);
          plo[e + h] = (uint32_t)p;
          phi[e + h] = (uint32_t)(p >> 32);
        }
      }
      tmem_st8(ts, plo);
      tmem_st8(ts + 8, phi);
      tmem_wait_st();
    }
  }
}

template <int UN>
__global__ void __launch_bounds__(THREADS, 1)
rns_gemm_kernel(const __grid_constant__ RnBatch B) {
  if (B.skip && *B.skip) return;                   // the results would not be used
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *sm = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES], empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t accfull_bar[2], accempty_bar[2], teardown_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;
  __shared__ long long last_seq[NPROD][MAX_STAGES];   // per producer: its latest copy into each stage

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < NPROD * MAX_STAGES) last_seq[tid / MAX_STAGES][tid % MAX_STAGES] = -1;
  if (tid == 0) {
    for (int s = 0; s < B.stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int k = 0; k < 2; ++k) { mbar_init(&accfull_bar[k], 1); mbar_init(&accempty_bar[k], DRAIN_WARPS); }
    mbar_init(&teardown_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&tmem_base_sh)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = tmem_base_sh;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // Register split of the launch's 168 a thread: 3 x 168 = 40 + 232 + 232.
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp != 1) {
      // ---------------------------------------------------------- bulk-copy producers
      // Every producer walks the same sequence of stages; producer pw fills
      // the stages whose sequence number is pw modulo NPROD.  Addresses are
      // warp-uniform and one elected lane issues (a pair of copies takes 61
      // clocks to issue, 179 from a lane picked by its number).
      const int pw = warp == 0 ? 0 : warp - 1;
      const uint32_t el = elect_one();
      int stage = 0, rr = 0, jc = 0;
      uint32_t phase = 0;
      long long seq = 0;
      bool ok = true;
      for (long long gi = blockIdx.x; ok && gi < B.total_items; gi += gridDim.x) {
        while (jc + 1 < B.njobs && gi >= B.job[jc + 1].item0) ++jc;
        const RnJob &J = B.job[jc];
        const RnItem it = rn_decode(J, gi - J.item0);
        const int hv = J.g.hv, ho = J.g.ho, nc16 = J.g.nc * 16;
        const size_t tA = (size_t)J.g.mt * RL * A_HALF, tB = (size_t)J.g.nch * RL * nc16;
        // K segments: their operands' halves of modulus 0.  A half-K unit runs
        // the first and the last.
        const unsigned char *a[4], *b[4];
        int end[4];
        a[0] = J.pa + (it.p * tA + (size_t)it.m * RL * A_HALF) * hv;
        a[1] = J.pa2 + (it.q * tA + (size_t)it.m * RL * A_HALF) * hv;
        a[2] = J.hc2 + (it.p * tA + (size_t)it.m * RL * A_HALF) * ho;
        a[3] = J.hc + (it.q * tA + (size_t)it.m * RL * A_HALF) * ho;
        const size_t rq = (size_t)it.r * J.g.o + it.q, rp = (size_t)it.r * J.g.o + it.p, ch = (size_t)it.nci * RL * nc16;
        b[0] = J.tb + (rq * tB + ch) * hv;
        b[1] = J.tb + (rp * tB + ch) * hv;
        b[2] = J.hb + (rq * tB + ch) * ho;
        b[3] = J.hb + (rp * tB + ch) * ho;
        end[0] = hv;
        end[1] = hv + (it.half ? 0 : hv);
        end[2] = end[1] + (it.half ? 0 : ho);
        end[3] = end[2] + ho;
        const int H = end[3];
        for (int l = 0; ok && l < RL; ++l) {
          for (int h0 = 0; h0 < H; h0 += B.hps, ++seq) {
            const bool mine = rr == pw;
            if (++rr == NPROD) rr = 0;
            if (mine) {
              const bool got = mbar_wait(&empty_bar[stage], phase ^ 1u, &abort_flag, B.err, ERR_TIMEOUT_EMPTY);
              if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
              const int h1 = min(H, h0 + B.hps);
              unsigned char *sA = sm + (size_t)stage * B.slot, *sB = sA + B.hps * A_HALF;
              if (el) {
                last_seq[pw][stage] = seq;
                mbar_expect_tx(&full_bar[stage], (uint32_t)(h1 - h0) * (uint32_t)(A_HALF + nc16));
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                  const int g0 = g ? end[g - 1] : 0, s0 = max(h0, g0), s1 = min(h1, end[g]);
                  if (s1 > s0) {
                    const uint32_t n = (uint32_t)(s1 - s0);
                    bulk_load(sA + (s0 - h0) * A_HALF, a[g] + (size_t)(s0 - g0) * A_HALF, n * A_HALF, &full_bar[stage]);
                    bulk_load(sB + (s0 - h0) * nc16, b[g] + (size_t)(s0 - g0) * nc16, n * nc16, &full_bar[stage]);
                  }
                }
              }
              __syncwarp();
            }
            if (++stage == B.stages) { stage = 0; phase ^= 1u; }
          }
#pragma unroll
          for (int g = 0; g < 4; ++g) {                    // the next modulus
            const int nh = g < 2 ? hv : ho;
            a[g] += (size_t)nh * A_HALF;
            b[g] += (size_t)nh * nc16;
          }
        }
      }
      // every issued copy has landed before the CTA may exit (bounded wait)
      prod_bar();
      if (pw == 0 && lane == 0) {
        for (int s = 0; s < B.stages; ++s) {
          long long last = -1;
          for (int q = 0; q < NPROD; ++q) last = max(last, last_seq[q][s]);
          if (last < 0) continue;
          const uint32_t par = (uint32_t)((last / B.stages) & 1);
          const uint32_t ad = smem_u32(&full_bar[s]);
          for (long long i2 = 0; i2 < WAIT_LIMIT && !mbar_try(ad, par); ++i2) {
            if ((i2 & 255) == 255) __nanosleep(128);
            if (i2 == WAIT_LIMIT - 1) atomicCAS(B.err, 0, ERR_TIMEOUT_TEARDOWN);
          }
        }
      }
      __syncwarp();
    } else {
      // ---------------------------------------------------------- MMA issuer (see tc_split.cu)
      const uint32_t el = elect_one();
      const uint32_t sbase = smem_u32(sm), slot = (uint32_t)B.slot;
      int stage = 0, jc = 0;
      uint32_t phase = 0, cnt = 0;
      bool ok = true;
      for (long long gi = blockIdx.x; ok && gi < B.total_items; gi += gridDim.x) {
        while (jc + 1 < B.njobs && gi >= B.job[jc + 1].item0) ++jc;
        const RnJob &J = B.job[jc];
        const int half = (J.unit[(gi - J.item0) / J.g.nch % J.nu] >> 2) & 1;
        const uint32_t nc = (uint32_t)J.g.nc;
        const int H = half ? J.g.hv + J.g.ho : 2 * (J.g.hv + J.g.ho);
        const uint32_t id = idesc(128, (int)nc);
        const uint64_t da0 = sdesc(0, A_HALF), db0 = sdesc(0, nc * 16) + (uint32_t)((B.hps * A_HALF) >> 4);
        for (int l = 0; ok && l < RL; ++l, ++cnt) {
          const uint32_t buf = cnt & 1u;
          if (!mbar_wait(&accempty_bar[buf], ((cnt >> 1) & 1u) ^ 1u, &abort_flag, B.err, ERR_TIMEOUT_ACCEMPTY)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d = tbase + buf * (uint32_t)B.acc;
          for (int h0 = 0; h0 < H; h0 += B.hps) {
            if (!mbar_try(smem_u32(&full_bar[stage]), phase) &&
                !mbar_wait(&full_bar[stage], phase, &abort_flag, B.err, ERR_TIMEOUT_FULL)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t at = (sbase + (uint32_t)stage * slot) >> 4;
            const uint64_t da = da0 + at, db = db0 + at;
            if (el) {
              // the stage's K blocks in straight runs of 4, 2 and 1 (a test
              // around every MMA would cost half an MMA's time each)
              constexpr uint32_t SA = 2 * A_HALF >> 4;
              const uint32_t SB = 2 * nc;
              int n = min(B.hps, H - h0) / 2;
              uint64_t xa = da, xb = db;
              uint32_t acc = h0 > 0 ? 1u : 0u;
              for (; n >= 4; n -= 4, xa += 4 * SA, xb += 4 * SB, acc = 1u) {
                mma_bf16(d, xa, xb, id, acc);
                mma_bf16(d, xa + SA, xb + SB, id, 1u);
                mma_bf16(d, xa + 2 * SA, xb + 2 * SB, id, 1u);
                mma_bf16(d, xa + 3 * SA, xb + 3 * SB, id, 1u);
              }
              if (n & 2) {
                mma_bf16(d, xa, xb, id, acc);
                mma_bf16(d, xa + SA, xb + SB, id, 1u);
                xa += 2 * SA;
                xb += 2 * SB;
                acc = 1u;
              }
              if (n & 1) mma_bf16(d, xa, xb, id, acc);
              mma_commit(&empty_bar[stage]);
            }
            if (++stage == B.stages) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          if (el) mma_commit(&accfull_bar[buf]);
        }
      }
      if (el) {
        mma_commit(&teardown_bar);
        const uint32_t a = smem_u32(&teardown_bar);
        for (long long it = 0; it < WAIT_LIMIT && !mbar_try(a, 0); ++it) {
          if ((it & 255) == 255) __nanosleep(128);
          if (it == WAIT_LIMIT - 1) atomicCAS(B.err, 0, ERR_TIMEOUT_TEARDOWN);
        }
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    // ------------------------------------------------------------ drain: residues -> 64-bit sums -> Y
    const int quarter = warp & 3;                   // TMEM lane quarter this warp may access
    const int hsel = (warp - 4) >> 2;               // which half of the columns
    const int lrow = 32 * quarter + lane;
    const uint32_t trow = tbase + ((uint32_t)(32 * quarter) << 16);
    const uint32_t tmp = trow + TM_BASE + (uint32_t)(hsel * 2 * TM_COLS);   // this thread's sums in TMEM
    uint32_t cnt = 0;
    bool ok = true, dep_done = false;
    int jc = 0;
    for (long long gi = blockIdx.x; ok && gi < B.total_items; gi += gridDim.x) {
      while (jc + 1 < B.njobs && gi >= B.job[jc + 1].item0) ++jc;
      const RnJob &J = B.job[jc];
      const int nc = J.g.nc, my = nc / 16;            // units of 8 columns of this thread
      const uint32_t c0 = (uint32_t)(hsel * (nc / 2));
      unsigned long long part[8 * UN];
#pragma unroll
      for (int e = 0; e < 8 * UN; ++e) part[e] = 0;
      uint32_t pk[2 * UN] = {};
      // wait for product l, reduce it, hand its accumulator back
      auto product = [&](auto mode, int l) {
        const uint32_t buf = cnt & 1u;
        const bool got = mbar_wait(&accfull_bar[buf], (cnt >> 1) & 1u, &abort_flag, B.err, ERR_TIMEOUT_ACCFULL);
        if (!__all_sync(0xffffffffu, got)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        drain_product<decltype(mode)::value, UN>(l, my, trow + buf * (uint32_t)B.acc + c0, tmp, part, pk);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty_bar[buf]);
        ++cnt;
        return true;
      };
#pragma unroll 1
      for (int l = 0; ok && l + 1 < RL; l += 2)
        ok = product(std::integral_constant<int, 0>{}, l) && product(std::integral_constant<int, 1>{}, l + 1);
      if (ok) ok = product(std::integral_constant<int, 2>{}, RL - 1);
      if (!ok) break;
      // The sums go into the job's buffer Y[triplet][a][b][c] (64-bit
      // fractions): F(i,j,k) stores its rows (a, b), the launch after it adds
      // F(i,k,j) (rows (a, c)) and F(j,k,i) (rows (b, c)) by reductions in L2.
      const RnItem it = rn_decode(J, gi - J.item0);
      const int vo = J.g.v, vc = J.g.vc;
      const int row = it.m * MROWS + lrow;
      if (!dep_done) { asm volatile("griddepcontrol.wait;" ::: "memory"); dep_done = true; }
      unsigned long long *Y = J.y + (size_t)it.tl * vo * vo * vc;
      const int zb = it.nci * nc + (int)c0;
      const bool in = row < vo * vo;
      const int p = in ? row / vo : 0, c = in ? row - p * vo : 0;
      const size_t st = it.f == 0 ? 1 : (it.f == 1 ? (size_t)vc : (size_t)vo * vc);
      unsigned long long *dst = Y + (it.f == 0 ? (size_t)row * vc : (it.f == 1 ? (size_t)p * vo * vc + c : (size_t)p * vc + c)) +
                                (size_t)zb * st;
      auto put = [&](int u, const unsigned long long *s8) {
        if (!in) return;
        if (it.f == 0) {
#pragma unroll
          for (int e = 0; e < 8; e += 2)
            if (zb + 8 * u + e < vc) *(ulonglong2 *)(dst + 8 * u + e) = make_ulonglong2(s8[e], s8[e + 1]);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (zb + 8 * u + e < vo) atomicAdd(dst + (size_t)(8 * u + e) * st, s8[e]);
        }
      };
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        if (u < my) {
          unsigned long long s8[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) s8[e] = part[8 * u + e] - RC.offp;
          put(u, s8);
        }
      }
#pragma unroll 1
      for (int u = UN; u < my; ++u) {
        const uint32_t ts = tmp + 16 * (uint32_t)(u - UN);
        uint32_t plo[8], phi[8];
        tmem_ld8u(ts, plo);
        tmem_ld8u(ts + 8, phi);
        tmem_wait_ld8u(plo, phi);
        unsigned long long s8[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) s8[e] = (((unsigned long long)phi[e] << 32) | plo[e]) - RC.off;
        put(u, s8);
      }
      __syncwarp();
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "r"(512));
  }
}

// ---------------------------------------------------------------- energy kernel

constexpr int WX = 73, WY = 9;               // W block index = x WX + y WY + z (8-byte words)
constexpr int WBLK = 7 * WX + 7 * WY + 8;

// |x| as a float (its leading 20 bits; beyond the float range 0 or infinity),
// without the FP64 pipe.
__device__ __forceinline__ float abs_float(double x) {
  const int h = (__double2hiint(x) & 0x7FFFFFFF) - (896 << 20);
  return __int_as_float(min(max(h, 0), 255 << 20) << 3);
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }   // |e| <= 126

// A 128-bit integer as a double (rounded once).
__device__ __forceinline__ double u128_double(unsigned __int128 x) {
  unsigned long long h = (unsigned long long)(x >> 64);
  const unsigned long long l = (unsigned long long)x;
  if (h == 0) return (double)l;
  const int z = __clzll((long long)h);
  if (z) h = h << z | l >> (64 - z);
  const double d = (double)(h | ((l << z) != 0));          // the low bits as a sticky bit
  return __hiloint2double(__double2hiint(d) + ((64 - z) << 20), __double2loint(d));
}

// One CTA per item (triplet, chunk of consecutive orbits).  The FP64 pipe (two
// lanes per SM and clock) bounds it, so the work per point is arranged for few
// FP64 operations.  With x_n the W values of the even and y_n of the odd
// permutations of a point, se and so their sums and d = se - so, the bracket of
// Eq. 1 is br = 3 x_n - se + 2 d and 3 y_n - so - 2 d: integers, exact while
// |W| < 2^59 units (14 standard deviations on data of uniform size; larger
// values take the same formulas in FP64), converted once each.  Then
// sum_s w_s br_s = (sum_s br_s^2) / 3 - 6 d^2, formed in 128-bit integers (the
// integer pipes have room beside the FP64 pipe); 34 FP64 operations a point and the
// division by D, which is left to the compiler: an own reciprocal of three
// operations made o=12 v=132 1.4 % faster and was right to the last place only.
// The weak triplets' bound, the sum of |1/D| (times WEAK_N4 and W's squared error
// at the end), is summed in FP32.
// Five small CTAs on an SM keep the pipe fed while one of them loads.
// Orbits with equal tiles list their canonical points (36 x 8 of 512 points for
// two equal tiles, 120 for three), so no warp runs for points outside them.
__global__ void __launch_bounds__(EN_THREADS, EN_CTAS)
rns_energy_kernel(const __grid_constant__ RnEnBatch B) {
  if (B.skip && *B.skip) return;
  __shared__ long long Wb[6 * WBLK];
  __shared__ double Gs[18 * NT2], Ts[9 * NT], Eab[NT2];   // Eab: e_i + e_j + e_k - e_a - e_b
  __shared__ double s_red[EN_THREADS / 32][2];
  __shared__ float s_abs[EN_THREADS / 32];
  __shared__ unsigned short tab2[36], tab3[120];   // points a >= b (a 8 + b) and a >= b >= c (a 64 + b 8 + c)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < NT3; e += EN_THREADS) {
    const int a = e / NT2, b = e / NT % NT, c = e % NT;
    if (a >= b && c == 0) tab2[a * (a + 1) / 2 + b] = (unsigned short)(e / NT);
    if (a >= b && b >= c) tab3[a * (a + 1) * (a + 2) / 6 + b * (b + 1) / 2 + c] = (unsigned short)e;
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  bool dep_done = false;
  int jc = 0;
  for (long long gi = blockIdx.x; gi < B.total_items; gi += gridDim.x) {
    while (jc + 1 < B.njobs && gi >= B.job[jc + 1].item0) ++jc;
    const RnEnJob &J = B.job[jc];
    const Dims &d = J.d;
    const int o = d.o, v = d.v, vc = J.vc;
    const long long q0 = gi - J.item0;
    const int tl = (int)(q0 / d.items_per_trip), chunk = (int)(q0 % d.items_per_trip);
    const int4 tr = J.trip[J.t0 + tl];
    const int occ[3] = {tr.x, tr.y, tr.z};
    const bool eq01 = tr.x == tr.y, eq12 = tr.y == tr.z;
    const double eijk = J.eps[occ[0]] + J.eps[occ[1]] + J.eps[occ[2]];
    const int sexp = J.uo[occ[0]] + J.uo[occ[1]] + J.uo[occ[2]] + J.sh[4];
    const long long *Y = J.y + (size_t)tl * v * v * vc;
    // the sums in units of the grid 2^-S of the orbits so far (S: sprev)
    double acc4 = 0.0, acc5 = 0.0;
    float accr = 0.f;                              // sum of |1/D|
    int sprev = 0;
    const int ob0 = chunk * d.orb_per_item, ob1 = min(d.n_orb, ob0 + d.orb_per_item);
    for (int ob = ob0; ob < ob1; ++ob) {
      const int4 og = J.orb[ob];
      const int t3[3] = {og.x, og.y, og.z};
      __syncthreads();                             // the previous orbit's reads are done
      // G_pq^uw = (p u|q w), occupied pairs (j,k), (i,k), (i,j) x ordered tile
      // position pairs (0,1) (1,0) (0,2) (2,0) (1,2) (2,1), and t1 rows
      for (int e = tid; e < 18 * NT2; e += EN_THREADS) {
        const int t = e / NT2, lu = e / NT % NT, lw = e % NT, op = t / 6, tp = t % 6;
        const int u = tp < 4 ? (tp & 1 ? (tp == 1 ? 1 : 2) : 0) : (tp == 4 ? 1 : 2);
        const int w = tp < 2 ? (tp == 0 ? 1 : 0) : tp == 2 ? 2 : tp == 3 ? 0 : (tp == 4 ? 2 : 1);
        const int p = op == 0 ? occ[1] : occ[0], q = op == 2 ? occ[1] : occ[2];
        const int gu = t3[u] * NT + lu, gw = t3[w] * NT + lw;
        Gs[e] = gu < v && gw < v ? __ldg(J.ovov + (((long long)p * v + gu) * o + q) * v + gw) : 0.0;
      }
      if (tid < NT2) {
        const int ga = t3[0] * NT + tid / NT, gb = t3[1] * NT + tid % NT;
        if (ga < v && gb < v) Eab[tid] = eijk - (__ldg(J.eps + o + ga) + __ldg(J.eps + o + gb));
      }
      if (tid < 9 * NT) {
        const int op = tid / (3 * NT), g = t3[tid / NT % 3] * NT + tid % NT;
        Ts[tid] = g < v ? __ldg(J.t1 + occ[op] * v + g) : 0.0;
      }
      if (!dep_done) { asm volatile("griddepcontrol.wait;" ::: "memory"); dep_done = true; }
      int blk[6];                                  // distinct block of each permutation of the tiles
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        blk[s] = s;
        for (int s2 = 0; s2 < s; ++s2)
          if (blk[s] == s && t3[perm3(s2, 0)] == t3[perm3(s, 0)] && t3[perm3(s2, 1)] == t3[perm3(s, 1)] &&
              t3[perm3(s2, 2)] == t3[perm3(s, 2)])
            blk[s] = s2;
      }
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        if (blk[s] != s) continue;
        const int x0 = t3[perm3(s, 0)] * NT, y0 = t3[perm3(s, 1)] * NT, z0 = t3[perm3(s, 2)] * NT;
#pragma unroll
        for (int k = 0; k < NT3 / EN_THREADS; ++k) {
          const int e = tid + k * EN_THREADS, x = e / NT2, y = e / NT % NT, z = e % NT;
          const bool in = x0 + x < v && y0 + y < v && z0 + z < v;
          Wb[s * WBLK + x * WX + y * WY + z] =
              in ? __ldcs(Y + ((long long)(x0 + x) * v + (y0 + y)) * vc + z0 + z) : 0;
        }
      }
      __syncthreads();
      // the orbit's exponent at its first point; points off it are brought to it
      const int S0 = sexp + __ldg(J.ev + t3[0] * NT) + __ldg(J.ev + t3[1] * NT) + __ldg(J.ev + t3[2] * NT);
      if (ob == ob0) {
        sprev = S0;
      } else if (S0 != sprev) {
        const double f = __longlong_as_double((long long)(1023 + S0 - sprev) << 52);
        acc5 *= f;
        acc4 = acc4 * f * f;
        accr *= pow2f(S0 - sprev) * pow2f(S0 - sprev);
        sprev = S0;
      }
      const bool eqP = t3[0] == t3[1], eqR = t3[1] == t3[2];
      const int npts = eqP ? (eqR ? 120 : 36 * NT) : (eqR ? NT * 36 : NT3);
#pragma unroll 1
      for (int n = tid; n < npts; n += EN_THREADS) {
        const int e = eqP ? (eqR ? tab3[n] : tab2[n / NT] * NT + n % NT) : (eqR ? n / 36 * NT2 + tab2[n % 36] : n);
        const int l3[3] = {e / NT2, e / NT % NT, e % NT};
        const int ga = t3[0] * NT + l3[0], gb = t3[1] * NT + l3[1], gc = t3[2] * NT + l3[2];
        if (ga >= v || gb >= v || gc >= v) continue;
        long long w[6];
#pragma unroll
        for (int s = 0; s < 6; ++s)
          w[s] = Wb[blk[s] * WBLK + l3[perm3(s, 0)] * WX + l3[perm3(s, 1)] * WY + l3[perm3(s, 2)]];
        if (eq01) {                                // W_xyz = U_xyz + U_yxz
          w[0] = w[2] = w[0] + w[2];
          w[1] = w[4] = w[1] + w[4];
          w[3] = w[5] = w[3] + w[5];
        } else if (eq12) {                         // W_xyz = U_xyz + U_xzy
          w[0] = w[1] = w[0] + w[1];
          w[2] = w[3] = w[2] + w[3];
          w[4] = w[5] = w[4] + w[5];
        }
        double br[6], n4;                          // n4 = 3 sum_s w_s br_s
        unsigned long long big = 0;
#pragma unroll
        for (int s = 0; s < 6; ++s) big |= (unsigned long long)(w[s] + (1LL << 59)) >> 60;
        if (big == 0) {
          const long long se = w[0] + w[3] + w[4], so = w[1] + w[2] + w[5], dl = se - so;
          const long long be = 2 * dl - se, bo = -2 * dl - so;
          unsigned __int128 q = 0;
#pragma unroll
          for (int s = 0; s < 6; ++s) {
            const long long b = 3 * w[s] + (perm3_even(s) ? be : bo);
            br[s] = (double)b;
            const unsigned long long x = (unsigned long long)(b < 0 ? -b : b);
            q += (unsigned __int128)x * x;
          }
          const unsigned long long x = (unsigned long long)(dl < 0 ? -dl : dl);
          n4 = u128_double(q - (unsigned __int128)x * x * 18);
        } else {
          double f[6];
#pragma unroll
          for (int s = 0; s < 6; ++s) f[s] = (double)w[s];
          const double se = f[0] + f[3] + f[4], so = f[1] + f[2] + f[5];
          n4 = 0.0;
#pragma unroll
          for (int s = 0; s < 6; ++s) {
            br[s] = 3.0 * f[s] + (perm3_even(s) ? se - 2.0 * so : so - 2.0 * se);
            n4 = fma(3.0 * f[s], br[s], n4);
          }
        }
        auto T = [&](int op, int pos) { return Ts[(op * 3 + pos) * NT + l3[pos]]; };
        auto G = [&](int op, int u, int x) {       // G of op at positions (u, x) of the point
          const int tp = u == 0 ? (x == 1 ? 0 : 2) : u == 1 ? (x == 0 ? 1 : 4) : (x == 0 ? 3 : 5);
          return Gs[(op * 6 + tp) * NT2 + l3[u] * NT + l3[x]];
        };
        // V at the six permutations of the point (Eq. 3) times the brackets
        double n5 = 0.0;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
          const int p0 = perm3(s, 0), p1 = perm3(s, 1), p2 = perm3(s, 2);
          const double vs = fma(T(0, p0), G(0, p1, p2), fma(T(1, p1), G(1, p0, p2), T(2, p2) * G(2, p0, p1)));
          n5 = s == 0 ? vs * br[0] : fma(vs, br[s], n5);
        }
        double r = 1.0 / (Eab[l3[0] * NT + l3[1]] - __ldg(J.eps + o + gc));
        if (ga == gb || gb == gc) r *= ga == gc ? 1.0 / 6.0 : 0.5;   // the point's share of the bracket sums
        const int dS = S0 - sexp - __ldg(J.ev + ga) - __ldg(J.ev + gb) - __ldg(J.ev + gc);
        if (dS != 0) {
          const double f = __longlong_as_double((long long)(1023 + dS) << 52);
          n4 = n4 * f * f;
          n5 *= f;
          accr = fmaf(abs_float(r), pow2f(dS) * pow2f(dS), accr);
        } else {
          accr += abs_float(r);
        }
        acc5 = fma(n5, r, acc5);
        acc4 = fma(n4, r, acc4);
      }
    }
    // the item's partial, in a fixed order
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc4 += __shfl_down_sync(0xffffffffu, acc4, off);
      acc5 += __shfl_down_sync(0xffffffffu, acc5, off);
      accr += __shfl_down_sync(0xffffffffu, accr, off);
    }
    if (lane == 0) { s_red[warp][0] = acc4; s_red[warp][1] = acc5; s_abs[warp] = accr; }
    __syncthreads();
    if (tid == 0) {
      double e4 = 0.0, e5 = 0.0, er = 0.0;
      for (int k = 0; k < EN_THREADS / 32; ++k) { e4 += s_red[k][0]; e5 += s_red[k][1]; er += s_abs[k]; }
      const double f = __longlong_as_double((long long)(1023 - sprev) << 52);
      double nz = J.nz[0];
      if (J.sh[5]) {
        const double *np = J.nz + 1, *nq = np + o;
        auto pair = [&](int r, int q) { return nq[r * o + q] + nq[q * o + r]; };
        nz = 3.0 + (np[occ[0]] + np[occ[1]] + np[occ[2]]) +
             (pair(occ[0], occ[1]) + pair(occ[0], occ[2]) + pair(occ[1], occ[2]));
      }
      er = (fabs(e4) - WEAK_N4 * nz * er) * f * (C_P * C_P / 3.0) * f;
      e4 = e4 * f * (C_P * C_P / 3.0) * f;
      e5 = e5 * f * C_P;
      const long long idx = (long long)(J.t0 + tl) * d.items_per_trip + chunk;
      J.partial[2 * idx] = e4 + e5;
      J.partial[2 * idx + 1] = e5;
      J.margin[idx] = er;
    }
  }
}

// ---------------------------------------------------------------- host side

Scales scales_at(const RnsLayout &L, void *ws, int *flag) {
  char *b = (char *)ws;
  Scales s{};
  s.ra = (double *)(b + L.ra);
  s.rt = (double *)(b + L.rt);
  s.rb = (double *)(b + L.rb);
  s.rh = (double *)(b + L.rh);
  const int v = L.g.v, o = L.g.o;
  s.nv = (unsigned long long *)(b + L.mx);
  s.no = s.nv + 4 * v;
  s.ev = (int *)(b + L.ex);
  s.uo = s.ev + v;
  s.dv = s.uo + o;
  s.du = s.dv + v;
  s.fv = s.du + o;
  s.fu = s.fv + v;
  s.sh = s.fu + o;
  s.pm = s.no + 4 * o + 1;                               // behind the number of weak triplets
  s.qm = s.pm + 2 * o;
  s.nz = (double *)(b + L.nz);
  s.flag = flag;
  return s;
}

constexpr int PREP_BLOCKS = 152 * 16, PREP_THREADS = 256;

size_t rn_slot(int hps, int ncmax) { return (size_t)hps * (A_HALF + (size_t)ncmax * 16); }

using RnKernel = void (*)(RnBatch);

// The GEMM kernel instance for a widest N chunk of ncmax columns: the columns of
// the next instance are reduced along (W at o=6 v=64 379 us on <5>, 365 on a <4>;
// v=96 1061 on <7>, 1037 on a <6>; eight instances compile in 11 s, five in 8).
RnKernel rn_kernel(int ncmax) {
  const int u = ncmax / 16;
  return u <= 3 ? rns_gemm_kernel<3> : u <= 5 ? rns_gemm_kernel<5> : u <= 7 ? rns_gemm_kernel<7>
       : u <= 9 ? rns_gemm_kernel<9> : rns_gemm_kernel<REG_UNITS>;
}

// Item offsets, shared-memory plan, grids and kernel instance of a GEMM batch and an energy batch.
cudaError_t prepare(RnBatch *gb, RnEnBatch &eb, int num_sms, int *ggrid, int *egrid, size_t *smem, RnKernel *fn) {
  int ncmax = 16;
  for (int f = 0; f < RNS_GEMM_LAUNCHES; ++f) {
    RnBatch &b = gb[f];
    if (b.njobs < 1 || b.njobs > MAX_BATCH || eb.njobs != b.njobs) return cudaErrorInvalidValue;
    long long total = 0;
    for (int j = 0; j < b.njobs; ++j) {
      RnJob &J = b.job[j];
      if (J.g.nc > NCMAX || 16 * (J.g.hv + J.g.ho) > KMAX) return cudaErrorInvalidValue;
      J.item0 = total;
      total += (long long)J.g.mt * J.nu * J.g.nch;
      ncmax = std::max(ncmax, J.g.nc);
    }
    b.total_items = total;
    ggrid[f] = (int)std::max<long long>(1, std::min<long long>(num_sms, total));
  }
  // The longest stages of which NPROD fit (fewer, longer copies and fewer
  // barriers a product: 16 halves instead of 8 save 5 %, o=12 v=132)
  int hps = HPS_MAX;
  while (hps > 2 && NPROD * rn_slot(hps, ncmax) > (size_t)SMEM_DYN_MAX - 1024) hps -= 2;
  const size_t slot = rn_slot(hps, ncmax);
  const int stages = (int)std::min<size_t>(MAX_STAGES, ((size_t)SMEM_DYN_MAX - 1024) / slot);
  if (stages < NPROD) return cudaErrorInvalidValue;
  for (int f = 0; f < RNS_GEMM_LAUNCHES; ++f) {
    gb[f].stages = stages;
    gb[f].hps = hps;
    gb[f].acc = ncmax;
    gb[f].slot = slot;
  }
  *smem = 1024 + (size_t)stages * slot;
  long long total = 0;
  for (int j = 0; j < eb.njobs; ++j) {
    eb.job[j].item0 = total;
    total += (long long)eb.job[j].nt * eb.job[j].d.items_per_trip;
  }
  eb.total_items = total;
  *egrid = (int)std::max<long long>(1, std::min<long long>((long long)EN_CTAS * num_sms, total));
  *fn = rn_kernel(ncmax);
  // The limit is the process's, not the launch's: always the same value, as another
  // thread may be between this and its launch.
  return cudaFuncSetAttribute(*fn, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_DYN_MAX);
}

}  // namespace

bool rns_supported(int o, int v) {
  const RnsGeom g = rns_geom(o, v);
  return o >= 2 && v >= RNS_MIN_V && 16 * (g.hv + g.ho) <= KMAX;
}

RnsGeom rns_geom(int o, int v) {
  RnsGeom g{};
  g.o = o;
  g.v = v;
  g.mt = (int)(((long long)v * v + MROWS - 1) / MROWS);
  g.hv = (v + 7) / 8;
  g.ho = (o + 7) / 8;
  g.ho += (g.hv + g.ho) & 1;                     // half of the K segments is a whole number of K blocks
  const int vp = (v + 15) / 16 * 16;
  g.nch = (vp + NCMAX - 1) / NCMAX;
  g.nc = ((vp + g.nch - 1) / g.nch + 15) / 16 * 16;
  g.vc = (v + 3) / 4 * 4;
  // Triplets per block: about 32 items per SM of a 152-SM GPU in the first of
  // its two GEMM launches, at most 256 and at most a 4 GB W buffer.
  const long long per_trip = (long long)g.mt * g.nch;
  long long nb = (32LL * 152 + per_trip - 1) / per_trip;
  nb = std::min<long long>(nb, (4LL << 30) / ((long long)v * v * g.vc * 8));
  nb = std::max<long long>(1, std::min<long long>(256, nb));
  const long long ntrip = std::max<long long>(1, (long long)o * (o + 1) * (o + 2) / 6 - o);
  g.nb = (int)std::min(nb, ntrip);
  return g;
}

RnsLayout rns_layout(const Dims &d) {
  const int o = d.o, v = d.v;
  RnsLayout L{};
  const RnsGeom g = rns_geom(o, v);
  L.g = g;
  const size_t a_v = (size_t)o * g.mt * g.hv * RL * A_HALF, a_o = (size_t)o * g.mt * g.ho * RL * A_HALF;
  const size_t b_v = (size_t)o * o * g.nch * g.hv * RL * g.nc * 16, b_o = (size_t)o * o * g.nch * g.ho * RL * g.nc * 16;
  const size_t O = o, V = v;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t r = off; off = (off + bytes + 255) & ~(size_t)255; return r; };
  L.pa = take(a_v);
  L.pa2 = take(a_v);
  L.hc = take(a_o);
  L.hc2 = take(a_o);
  L.tb = take(b_v);
  L.hb = take(b_o);
  L.y = take((size_t)g.nb * V * V * g.vc * 8);
  L.ra = take(O * V * V * 8);
  L.rt = take(O * V * V * 8);
  L.rb = take(O * O * V * 8);
  L.rh = take(O * V * O * 8);
  L.mx = take((4 * (V + O) + 1 + 2 * O + 2 * O * O) * 8);
  L.nz = take((1 + O + O * O) * 8);
  L.ex = take((3 * (V + O) + 8) * 4);
  L.unit = take((size_t)3 * std::max(1, d.n_trip) * 4);
  L.margin = take((size_t)std::max<long long>(1, d.n_items) * 8);
  L.weak = take((size_t)std::max(1, d.n_trip) * 4);
  L.need = take(O * O);
  L.total = off;
  return L;
}

RnsTables rns_tables(int o, const int4 *trip, int n) {
  RnsTables t;
  t.off.assign((size_t)n + 1, 0);
  t.unit.resize((size_t)n);
  std::vector<int> add;
  t.need.assign((size_t)o * o, 0);
  for (int m = 0; m < n; ++m) {
    const int i = trip[m].x, j = trip[m].y, k = trip[m].z;
    t.unit[(size_t)m] = (m << 3) | (i == j ? 4 : 0);
    if (j != k) add.push_back((m << 3) | 1);
    if (i != j) add.push_back((m << 3) | (j == k ? 4 : 0) | 2);
    t.off[(size_t)m + 1] = (int)add.size();
    const int x[3] = {i, j, k};
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) t.need[(size_t)x[a] * o + x[b]] = 1;
  }
  t.unit.insert(t.unit.end(), add.begin(), add.end());
  return t;
}

int rns_prep_launches(int o, int v) { return (long long)o * v * v <= SCALES_ONE ? 3 : 6; }

cudaError_t launch_rns_prep(const RnsLayout &L, const Inputs &in, void *ws, const RnsTables &t, bool all, int *flag,
                            cudaStream_t st) {
  const RnsGeom &g = L.g;
  char *b = (char *)ws;
  const Scales s = scales_at(L, ws, flag);
  cudaError_t e = cudaMemcpyAsync(b + L.unit, t.unit.data(), t.unit.size() * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && !all) e = cudaMemcpyAsync(b + L.need, t.need.data(), t.need.size(), cudaMemcpyHostToDevice, st);
  // the maxima per array and orbital, the number of weak triplets, the scaled maxima by p
  if (e == cudaSuccess) e = cudaMemsetAsync(b + L.mx, 0, (4 * ((size_t)g.v + g.o) + 1 + 2 * (size_t)g.o) * 8, st);
  if (e != cudaSuccess) return e;
  const unsigned char *need = all ? nullptr : (const unsigned char *)(b + L.need);
  rns_norms<<<PREP_BLOCKS, PREP_THREADS, 4 * ((size_t)g.v + g.o) * 8, st>>>(in, g.o, g.v, s);
  if ((long long)g.o * g.v * g.v <= SCALES_ONE) {
    rns_scales_one<<<1, 1024, 0, st>>>(g.o, g.v, s);
  } else {
    rns_wanted<<<1, 512, 0, st>>>(g.o, g.v, s);
    rns_shares<<<152 * 2, 256, 0, st>>>(g.o, g.v, s);
    rns_scaled_max<<<152 * 2, 256, 0, st>>>(g.o, g.v, s);
    rns_scales<<<1, 512, 0, st>>>(g.o, g.v, s);
  }
  unsigned char *ub = (unsigned char *)b;
  const long long work = (long long)g.o * ((g.v + 7) / 8) * ((g.v + 3) / 4) * g.hv;   // warps of the largest task
  const int blocks = (int)std::max<long long>(1, std::min<long long>(PREP_BLOCKS, (work + 7) / 8));
  rns_images<<<dim3(blocks, 4), PREP_THREADS, 0, st>>>(L, in, s, need, ub);
  return cudaGetLastError();
}

void rns_block(const RnsLayout &L, void *ws, const Dims &d, const Inputs &in, const Work &w, const RnsTables &t, int t0,
               int nt, RnJob *j0, RnJob *j1, RnEnJob *en) {
  unsigned char *b = (unsigned char *)ws;
  const Scales s = scales_at(L, ws, nullptr);
  RnJob J{};
  J.g = L.g;
  J.trip = w.trip;
  J.t0 = t0;
  J.pa = b + L.pa;
  J.pa2 = b + L.pa2;
  J.hc = b + L.hc;
  J.hc2 = b + L.hc2;
  J.tb = b + L.tb;
  J.hb = b + L.hb;
  J.y = (unsigned long long *)(b + L.y);
  const int *unit = (const int *)(b + L.unit);
  *j0 = J;
  j0->unit = unit + t0;
  j0->nu = nt;
  *j1 = J;
  j1->unit = unit + (t.off.size() - 1) + t.off[(size_t)t0];
  j1->nu = t.off[(size_t)t0 + nt] - t.off[(size_t)t0];
  RnEnJob &E = *en;
  E = RnEnJob{};
  E.d = d;
  E.vc = L.g.vc;
  E.trip = w.trip;
  E.orb = w.orb;
  E.eps = in.eps;
  E.t1 = in.t1;
  E.ovov = in.ovov;
  E.y = (const long long *)(b + L.y);
  E.ev = s.ev;
  E.uo = s.uo;
  E.sh = s.sh;
  E.nz = s.nz;
  E.partial = w.partial;
  E.margin = (double *)(b + L.margin);
  E.t0 = t0;
  E.nt = nt;
}

void rns_weak(const RnsLayout &L, void *ws, RedJob *j) {
  char *b = (char *)ws;
  j->margin = (const double *)(b + L.margin);
  j->weak_n = (int *)(b + L.mx + 4 * ((size_t)L.g.v + L.g.o) * 8);
  j->weak = (int *)(b + L.weak);
}

cudaError_t rns_block_params(RnBatch *gb, RnEnBatch &eb, int num_sms, void **gargs, void **eargs,
                             cudaKernelNodeParams *gp, cudaKernelNodeParams *ep) {
  int ggrid[RNS_GEMM_LAUNCHES], egrid = 1;
  size_t smem = 0;
  RnKernel fn = nullptr;
  const cudaError_t e = prepare(gb, eb, num_sms, ggrid, &egrid, &smem, &fn);
  if (e != cudaSuccess) return e;
  for (int f = 0; f < RNS_GEMM_LAUNCHES; ++f) {
    gargs[f] = (void *)&gb[f];
    gp[f] = cudaKernelNodeParams{};
    gp[f].func = (void *)fn;
    gp[f].gridDim = dim3(ggrid[f]);
    gp[f].blockDim = dim3(THREADS);
    gp[f].sharedMemBytes = (unsigned)smem;
    gp[f].kernelParams = &gargs[f];
  }
  eargs[0] = (void *)&eb;
  *ep = cudaKernelNodeParams{};
  ep->func = (void *)rns_energy_kernel;
  ep->gridDim = dim3(egrid);
  ep->blockDim = dim3(EN_THREADS);
  ep->kernelParams = eargs;
  return cudaSuccess;
}

cudaError_t launch_rns_block(RnBatch *gb, RnEnBatch &eb, int num_sms, cudaStream_t st, cudaEvent_t w0, cudaEvent_t w1) {
  int ggrid[RNS_GEMM_LAUNCHES], egrid = 1;
  size_t smem = 0;
  RnKernel fn = nullptr;
  cudaError_t e = prepare(gb, eb, num_sms, ggrid, &egrid, &smem, &fn);
  if (e != cudaSuccess) return e;
  if (w0 && (e = cudaEventRecord(w0, st)) != cudaSuccess) return e;
  // programmatic launches, as launch_split_block: each kernel waits for its
  // predecessor only before it touches Y
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  for (int f = 0; f < RNS_GEMM_LAUNCHES; ++f) {
    cfg.gridDim = dim3(ggrid[f]);
    if ((e = cudaLaunchKernelEx(&cfg, fn, gb[f])) != cudaSuccess) return e;
  }
  if (w1 && (e = cudaEventRecord(w1, st)) != cudaSuccess) return e;
  cfg.gridDim = dim3(egrid);
  cfg.blockDim = dim3(EN_THREADS);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, rns_energy_kernel, eb);
}

}  // namespace tc
