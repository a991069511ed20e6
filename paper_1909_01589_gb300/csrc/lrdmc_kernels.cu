// CUDA kernels (sm_103a) of the LRDMC hot path.
//
// One warp owns one walker at a time. Shared memory holds the walker's
// positions, inverse Slater matrices, lattice rotation, the P jump rates of
// its cached evaluation, per-electron work vectors and (double-float mode)
// the electron-pair and electron-nucleus caches of the evaluation; the MO
// coefficients are staged once per block. The lanes split the P lattice
// moves of an evaluation, the electrons of the local energy, the orbitals
// and matrix entries of the Sherman-Morrison update, and the rows of the
// Gauss-Jordan inverse. The evaluation runs in IEEE double, in double-float
// on the FP32 pipe, or in single precision (the kernels' template argument
// carries the arithmetic and whether the neural pair term is set); inverses,
// updates, weights and reconfiguration stay in IEEE double. Kernels:
//   k_init      start configurations -> inverses, first rotation
//   k_eval_all  evaluate every walker (after a change of lattice)
//   k_interval  one interval tau of continuous-time projection per walker,
//               walkers fetched dynamically by the warps (ragged jump counts)
//   k_comb_sums, k_comb_parents  reconfiguration: running weight sums, comb
//               parents, trace entry, order of the next interval
//   k_evaluate  stateless evaluation of given configurations (and the
//               variant with static scratch, k_evaluate_static)
//   k_base_terms  gradients and local energies without the neural term
// The population is double-buffered: k_interval gathers the record of
// parent[s] from the source buffer, so reconfiguration needs no copy pass.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <mutex>

#include "lrdmc_internal.h"
#include "lean64.cuh"

// This file is compiled several times, so that the kernel variants build in
// parallel: part 0 holds the kernels without variants and every host entry,
// parts 1.. instantiate the variants listed at the end of the file.
#ifndef LRDMC_PART
#define LRDMC_PART 0
#endif

namespace lrdmc {

#define FULL_MASK 0xffffffffu

// ----------------------------------------------------------------------------
// Counter-based random numbers: Philox4x64-10 (Salmon, Moraes, Dror, Shaw,
// SC'11), key (seed, 0), counter (slot, interval, iteration, tag).
// ----------------------------------------------------------------------------
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1)
{
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
    uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
    uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B97F4A7C15ull;
    k1 += 0xBB67AE8584CAA73Bull;
  }
}

__device__ __forceinline__ double to_u01(uint64_t bits)
{
  return ((double)(bits >> 12) + 0.5) * 0x1.0p-52;
}

__device__ __forceinline__ void draw_uniforms(uint64_t seed, uint64_t slot, uint64_t k, uint64_t m,
                                              uint64_t tag, double u[4])
{
  uint64_t c[4] = {slot, k, m, tag};
  philox4x64_10(c, seed, 0ull);
#pragma unroll
  for (int j = 0; j < 4; ++j) u[j] = to_u01(c[j]);
}

// The same uniform ((bits >> 12) + 1/2) 2^-52 = N 2^-53, N = 2 (bits >> 12)
// + 1 < 2^53, as a double-float built with integer operations only (no FP64
// pipe): the 24 bits below N's leading bit give hi exactly, the remaining
// low bits (at most 29) give lo, so the relative error is below 2^-47 for
// every uniform, however small.
__device__ __forceinline__ df df_u01(uint64_t bits)
{
  const uint64_t N = ((bits >> 12) << 1) | 1ull;
  const int sh = (63 - __clzll((long long)N)) - 23;  // shift that leaves 24 bits
  const uint64_t top = sh >= 0 ? (N >> sh) : (N << (-sh));
  const uint64_t rem = sh > 0 ? (N - (top << sh)) : 0ull;
  const float hi = (float)(uint32_t)top * __int_as_float((127 + sh - 53) << 23);
  const float lo = (float)(uint32_t)rem * 0x1.0p-53f;
  return fast_two_sum(hi, lo);
}

// A single-precision uniform from the top 24 bits, in (0, 1).
__device__ __forceinline__ float f_u01(uint64_t bits)
{
  return ((float)(uint32_t)(bits >> 40) + 0.5f) * 0x1.0p-24f;
}

__device__ __forceinline__ uint64_t shfl_u64(uint64_t v, int src)
{
  uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)v, src), hi = __shfl_sync(0xffffffffu, (uint32_t)(v >> 32), src);
  return ((uint64_t)hi << 32) | lo;
}

// Uniformly random rotation (Shoemake's unit quaternion from three uniforms).
static __device__ void rotation_matrix(double u1, double u2, double u3, double* R)
{
  double s1 = sqrt(1.0 - u1), s2 = sqrt(u1);
  double sa, ca, sb, cb;
  sincospi(2.0 * u2, &sa, &ca);
  sincospi(2.0 * u3, &sb, &cb);
  double x = s1 * sa, y = s1 * ca, z = s2 * sb, w = s2 * cb;
  R[0] = 1.0 - 2.0 * (y * y + z * z); R[1] = 2.0 * (x * y - z * w);       R[2] = 2.0 * (x * z + y * w);
  R[3] = 2.0 * (x * y + z * w);       R[4] = 1.0 - 2.0 * (x * x + z * z); R[5] = 2.0 * (y * z - x * w);
  R[6] = 2.0 * (x * z - y * w);       R[7] = 2.0 * (y * z + x * w);       R[8] = 1.0 - 2.0 * (x * x + y * y);
}

// The same rotation from the three uniforms of bits[0..2], with the work
// spread over the warp: lanes 0-3 evaluate sqrt(1-u1), sqrt(u1),
// sincospi(2 u2) and sincospi(2 u3), lanes 0-8 then form one entry of R
// each. IEEE double (the same operations as rotation_matrix), for the FP64
// mode; the others draw ahead. All lanes must call it; R goes to shared memory.
__device__ __forceinline__ void rotation_matrix_warp(const uint64_t* bits, double* R, int lane)
{
  double x, y, z, w;
  {
    double a = 0.0, c = 0.0;
    const double u1 = to_u01(bits[0]);
    if (lane == 0) a = sqrt(1.0 - u1);
    else if (lane == 1) a = sqrt(u1);
    else if (lane == 2) sincospi(2.0 * to_u01(bits[1]), &a, &c);
    else if (lane == 3) sincospi(2.0 * to_u01(bits[2]), &a, &c);
    double s1 = __shfl_sync(FULL_MASK, a, 0), s2 = __shfl_sync(FULL_MASK, a, 1);
    double sa = __shfl_sync(FULL_MASK, a, 2), ca = __shfl_sync(FULL_MASK, c, 2);
    double sb = __shfl_sync(FULL_MASK, a, 3), cb = __shfl_sync(FULL_MASK, c, 3);
    x = s1 * sa; y = s1 * ca; z = s2 * sb; w = s2 * cb;
  }
  double v = 0.0;
  switch (lane) {
    case 0: v = 1.0 - 2.0 * (y * y + z * z); break;
    case 1: v = 2.0 * (x * y - z * w); break;
    case 2: v = 2.0 * (x * z + y * w); break;
    case 3: v = 2.0 * (x * y + z * w); break;
    case 4: v = 1.0 - 2.0 * (x * x + z * z); break;
    case 5: v = 2.0 * (y * z - x * w); break;
    case 6: v = 2.0 * (x * z - y * w); break;
    case 7: v = 2.0 * (y * z + x * w); break;
    case 8: v = 1.0 - 2.0 * (x * x + y * y); break;
    default: break;
  }
  if (lane < 9) R[lane] = v;
}

// ----------------------------------------------------------------------------
// Warp helpers.
// ----------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

// Chunked inclusive scan of T[0..P): chunks of 32 in order, a Hillis-Steele
// scan inside each chunk plus the running total of the previous chunks.
// Returns the total (identical in every lane). When pick != nullptr, *pick
// receives the smallest c with target < C_c (or -1), and *last the largest c
// with T_c > 0 (or -1).
static __device__ double warp_scan(const double* T, int P, int lane, double target, int* pick, int* last)
{
  double carry = 0.0;
  int p = -1, lp = -1;
  for (int base = 0; base < P; base += 32) {
    int c = base + lane;
    double t = (c < P) ? T[c] : 0.0;
    double v = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      double y = __shfl_up_sync(FULL_MASK, v, o);
      if (lane >= o) v += y;
    }
    double C = carry + v;
    if (pick) {
      unsigned hit = __ballot_sync(FULL_MASK, (c < P) && (target < C));
      if (p < 0 && hit) p = base + __ffs(hit) - 1;
      unsigned pos = __ballot_sync(FULL_MASK, (c < P) && (t > 0.0));
      if (pos) lp = base + 31 - __clz(pos);
    }
    carry = __shfl_sync(FULL_MASK, C, 31);
  }
  if (pick) { *pick = p; *last = lp; }
  return carry;
}

// ----------------------------------------------------------------------------
// Atomic orbitals: chi = S(d) R(|d|), d = r - R_centre, S a real solid
// harmonic of degree l, R Slater r^m exp(-zeta r) or a Gaussian contraction.
// ----------------------------------------------------------------------------
__device__ __forceinline__ double int_pow(double r, int m)
{
  double p = 1.0;
  for (int j = 0; j < m; ++j) p *= r;
  return p;
}

// Radial value R, R'/r and R''. e is exp(-zeta r) for Slater shells.
__device__ __forceinline__ void radial(const ShellDev& sh, double r, double e, double& R, double& R1,
                                       double& R2, bool der)
{
  if (sh.kind == 0) {
    double pw = (sh.m_int >= 0) ? int_pow(r, sh.m_int) : pow(r, sh.m);
    R = pw * e;
    if (der) {
      double t = sh.m / r - sh.zeta;
      R1 = t * R / r;
      R2 = (t * t - sh.m / (r * r)) * R;
    }
  } else {
    double r2 = r * r;
    R = 0.0; R1 = 0.0; R2 = 0.0;
    for (int p = 0; p < sh.n_prim; ++p) {
      double al = sh.alpha[p];
      double g = sh.coef[p] * exp(-al * r2);
      R += g;
      if (der) {
        R1 += -2.0 * al * g;
        R2 += (4.0 * al * al * r2 - 2.0 * al) * g;
      }
    }
  }
}

// Solid harmonics of degree l at d and their gradients.
__device__ __forceinline__ int solid(int l, const double d[3], double S[5], double gS[5][3], bool der)
{
  if (l == 0) {
    S[0] = 1.0;
    if (der) { gS[0][0] = gS[0][1] = gS[0][2] = 0.0; }
    return 1;
  }
  if (l == 1) {
    S[0] = d[0]; S[1] = d[1]; S[2] = d[2];
    if (der) {
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int k = 0; k < 3; ++k) gS[f][k] = (f == k) ? 1.0 : 0.0;
    }
    return 3;
  }
  S[0] = d[0] * d[1];
  S[1] = d[1] * d[2];
  S[2] = d[2] * d[0];
  S[3] = d[0] * d[0] - d[1] * d[1];
  S[4] = 2.0 * d[2] * d[2] - d[0] * d[0] - d[1] * d[1];
  if (der) {
    gS[0][0] = d[1];        gS[0][1] = d[0];        gS[0][2] = 0.0;
    gS[1][0] = 0.0;         gS[1][1] = d[2];        gS[1][2] = d[1];
    gS[2][0] = d[2];        gS[2][1] = 0.0;         gS[2][2] = d[0];
    gS[3][0] = 2.0 * d[0];  gS[3][1] = -2.0 * d[1]; gS[3][2] = 0.0;
    gS[4][0] = -2.0 * d[0]; gS[4][1] = -2.0 * d[1]; gS[4][2] = 4.0 * d[2];
  }
  return 5;
}

// A float's value as a double, in integer operations (a conversion holds the
// FP64 pipe for 64 cycles); a zero or a denormal becomes about 1e-38.
__device__ __forceinline__ double widen(float f)
{
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// sqrt(x) in three operations of the FP64 pipe, which takes 64 cycles for
// each, against about nine: Karp and Markstein's iteration (ACM TOMS 23
// (1997)) in double-float on the FP32 pipe (to 2^-45), the last step in
// double. Outside [2^-95, 2^80] (and for zero, NaN) CUDA's.
__device__ __forceinline__ double sqrt64(double x)
{
  const unsigned h = (unsigned)__double2hiint(x);
  if (h - 0x3a000000u >= 0x0af00000u) return sqrt(x);
  const df a = dl_from_double(x);
  const float y = rsqrt_ftz(a.hi), s = __fmul_rn(a.hi, y), hy = __fmul_rn(0.5f, y);
  const float ds = __fmul_rn(__fadd_rn(__fmaf_rn(-s, s, a.hi), a.lo), hy);
  const double g = widen(s) + widen(ds);
  return fma(fma(-g, g, x), widen(hy), g);
}

// Shells [q0, q1) of the basis at d = p - R_centre of electron position p:
// v . chi, and with der its gradient and Laplacian, added to the sums.
template <bool DER>
__device__ __forceinline__ void ao_dot(const SysDev& S, const double* v, const double* p, int q0, int q1, double& val,
                                       double g[3], double& lap)
{
  int prev_c = -1;
  double d[3] = {0, 0, 0}, r = 0.0, e = 0.0;
#pragma unroll 1
  for (int q = q0; q < q1; ++q) {
    const ShellDev& sh = S.sh[q];
    if (sh.center != prev_c) {
      prev_c = sh.center;
#pragma unroll
      for (int k = 0; k < 3; ++k) d[k] = p[k] - S.nuc[prev_c][k];
      r = sqrt64(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    }
    if (sh.kind == 0 && (q == q0 || !sh.same_exp)) e = exp(-sh.zeta * r);
    double R, R1, R2, Sv[5], gS[5][3];
    radial(sh, r, e, R, R1, R2, DER);
    const int nf = solid(sh.l, d, Sv, gS, DER);
    if (!DER) {
      double part = 0.0;
      for (int f = 0; f < nf; ++f) part += v[sh.ao_offset + f] * Sv[f];
      val += part * R;
      continue;
    }
    // with P = sum_f v_f S_f: grad = R grad P + (R'/r) P d
    double P = 0.0;
    for (int f = 0; f < nf; ++f) {
      const double c = v[sh.ao_offset + f], cR = c * R;
      P += c * Sv[f];
      if (sh.l > 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] += cR * gS[f][k];
    }
    const double W = P * R1;
#pragma unroll
    for (int k = 0; k < 3; ++k) g[k] += W * d[k];
    lap += P * (R2 + 2.0 * (sh.l + 1) * R1);
  }
}

// chi_mu(p) of shell q into out[n_ao].
static __device__ void shell_values(const SysDev& S, int q, const double* p, double* out)
{
  const ShellDev& sh = S.sh[q];
  const double d[3] = {p[0] - S.nuc[sh.center][0], p[1] - S.nuc[sh.center][1], p[2] - S.nuc[sh.center][2]};
  const double r = sqrt64(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const double e = sh.kind == 0 ? exp(-sh.zeta * r) : 0.0;
  double R, R1, R2, Sv[5], gS[5][3];
  radial(sh, r, e, R, R1, R2, false);
  const int nf = solid(sh.l, d, Sv, gS, false);
  for (int f = 0; f < nf; ++f) out[sh.ao_offset + f] = Sv[f] * R;
}

// ----------------------------------------------------------------------------
// Jastrow factor.
// ----------------------------------------------------------------------------
__device__ __forceinline__ int spin_of(const SysDev& S, int i) { return i < S.n_up ? 0 : 1; }

// Neural pair term, tabulated: the cell of r (uniform in sqrt(r) on
// [0, r_cut)) holds r_k, 1/w_k and c_0..c_5; g = sum_q c_q t^q with
// t = (r - r_k)/w_k (Horner), 0 from r_cut on. The cell index is taken in
// single precision: next to a cell edge either neighbour's polynomial
// agrees with the other to second order at the edge, so the choice is
// immaterial.
__device__ __forceinline__ int nj_ch_ee(const SysDev& S, int i, int j) { return spin_of(S, i) == spin_of(S, j) ? 0 : 1; }

__device__ __forceinline__ const double* nj_cell(const SysDev& S, int c, double r)
{
  int k = (int)(sqrtf((float)r) * S.nj_scale_f[c]);
  k = min(max(k, 0), S.nj_cells - 1);
  return S.nj_tab + ((size_t)c * S.nj_cells + k) * 8;
}

__device__ __forceinline__ double nj_value(const SysDev& S, int c, double r)
{
  if (!(r < S.nj_rcut[c])) return 0.0;
  const double* e = nj_cell(S, c, r);
  const double t = (r - __ldg(e)) * __ldg(e + 1);
  double v = __ldg(e + 7);
#pragma unroll
  for (int q = 6; q >= 2; --q) v = fma(v, t, __ldg(e + q));
  return v;
}

__device__ __forceinline__ void nj_value3(const SysDev& S, int c, double r, double& g, double& g1, double& g2)
{
  g = 0.0; g1 = 0.0; g2 = 0.0;
  if (!(r < S.nj_rcut[c])) return;
  const double* e = nj_cell(S, c, r);
  const double iw = __ldg(e + 1), t = (r - __ldg(e)) * iw;
  const double c0 = __ldg(e + 2), c1 = __ldg(e + 3), c2 = __ldg(e + 4), c3 = __ldg(e + 5), c4 = __ldg(e + 6),
               c5 = __ldg(e + 7);
  g = c0 + t * (c1 + t * (c2 + t * (c3 + t * (c4 + t * c5))));
  const double d1 = c1 + t * (2.0 * c2 + t * (3.0 * c3 + t * (4.0 * c4 + t * 5.0 * c5)));
  const double d2 = 2.0 * c2 + t * (6.0 * c3 + t * (12.0 * c4 + t * 20.0 * c5));
  g1 = d1 * iw;
  g2 = d2 * iw * iw;
}

// ----------------------------------------------------------------------------
// Per-warp shared-memory views.
// ----------------------------------------------------------------------------
struct WarpMem {
  double* x;    // [N][3]
  double* A;    // inverse up [nu][nu] then down [nd][nd]
  double* R;    // [9]
  double* T;    // [P_max]
  double* dr;   // [kDrawAhead][kDrawWords] draws made ahead (double-float and mixed modes)
  double* sm;   // [4 + n_ao + 3 nu] Sherman-Morrison scratch of the double-float mode
  // the evaluation's state; scr is scratch over the same storage (the
  // inverse and the other modes' Sherman-Morrison updates, which run while
  // no evaluation's state is needed)
  double* v;    // [N][n_ao]
  double* Ssum; // [N]
  df* xd;       // [N][3]      double-float copies for the FP32-pipe evaluations
  df* vd;       // [N][n_ao]   (aliases v)
  df* Sd;       // [N]         (aliases Ssum) Jastrow sums; double-float mode: the e-e sums
  df* Sn;       // [N]         double-float mode: the e-n sums (and the neural term)
  df* y;        // [N][3]      double-float mode: positions on the rotated axes, scaled
  df* Rd;       // [12]
  df* pfx;      // [32]        double-float mode: running sums of the rates
  df* enc;      // [N][n_nuc][7] electron-nucleus cache: d, |d|^2, e_k . d
  df* pc;       // [n_pc] squared distances of the electron pairs, scaled
  double* scr;
  int n_pc;     // pairs in the cache (0: no cache)
};

__device__ __forceinline__ WarpMem warp_mem(const Layout& Lo, const SysDev& S, double* base)
{
  WarpMem m;
  m.x = base;
  m.A = m.x + 3 * Lo.N;
  m.R = m.A + Lo.nu * Lo.nu + Lo.nd * Lo.nd;
  m.T = m.R + 12;
  m.dr = m.T + Lo.P_max;
  m.sm = m.dr + Lo.n_draw;
  m.scr = m.sm + 4 + S.n_ao + 3 * Lo.nu;
  m.v = m.scr;
  m.Ssum = m.v + Lo.N * S.n_ao;
  // the FP64 evaluation uses v and Ssum, the FP32-pipe evaluations their
  // double-float images vd and Sd: one precision runs per launch, so they
  // share the storage
  m.vd = reinterpret_cast<df*>(m.v);
  m.Sd = reinterpret_cast<df*>(m.Ssum);
  m.Sn = m.Sd + Lo.N;
  m.xd = m.Sn + Lo.N;
  m.y = m.xd + 3 * Lo.N;
  m.Rd = m.y + 3 * Lo.N;
  m.pfx = m.Rd + 12;
  m.enc = m.pfx + 32;
  m.pc = m.enc + (Lo.enc ? kEncWords * Lo.N * S.n_nuc : 0);
  m.n_pc = Lo.n_pc;
  return m;
}

// Block-shared tables: the MO coefficients and the masks of the non-zero ones.
struct BlockMem {
  double* C;
  unsigned long long* col;  // [n_mo] non-zero rows of a column of C
  unsigned* row;            // [n_ao] non-zero columns of a row
};

__device__ __forceinline__ BlockMem block_mem(const SysDev& S, double* smem)
{
  BlockMem b;
  b.C = smem;
  b.col = reinterpret_cast<unsigned long long*>(smem + mask_offset(S));
  b.row = reinterpret_cast<unsigned*>(smem + mask_offset(S) + S.n_mo);
  return b;
}

// sum_m C[mu][m] A[m n + l] and sum_mu C[mu][m] chi[mu] over the non-zero
// coefficients only, in order (a zero's product would add nothing): an FP64
// multiply-add holds its sub-partition's pipe for 64 cycles, and an atom's C
// has few non-zeros (18 of 324 for Kr).
__device__ __forceinline__ double project_ao(const SysDev& S, const BlockMem& bm, const double* A, int mu, int l, int n)
{
  double acc = 0.0;
#pragma unroll 1
  for (unsigned k = bm.row[mu] & (n < 32 ? (1u << n) - 1u : 0xffffffffu); k; k &= k - 1) {
    const int m = __ffs(k) - 1;
    acc += bm.C[mu * S.n_mo + m] * A[m * n + l];
  }
  return acc;
}

__device__ __forceinline__ double orbital_value(const SysDev& S, const BlockMem& bm, const double* chi, int m)
{
  double a = 0.0;
#pragma unroll 1
  for (unsigned long long k = bm.col[m]; k; k &= k - 1) {
    const int mu = __ffsll((long long)k) - 1;
    a += bm.C[mu * S.n_mo + m] * chi[mu];
  }
  return a;
}

// ----------------------------------------------------------------------------
// Inverse Slater matrices of both spin blocks by Gauss-Jordan elimination
// with partial pivoting (warp-cooperative), A[l][m] = phi_m(r_l), the inverse
// stored as Ainv[m][l]; false for a singular matrix (below). With resid
// (nullable), first the residual of the inverses the blocks hold (the
// Sherman-Morrison-updated ones): max |sum_m A[l][m] Ainv[m][q] - delta_lq|,
// where A is the Slater matrix at the current positions; *resid becomes the
// larger of itself and that residual (the same value in every lane).
//
// Bound by the FP64 pipe, which takes 64 cycles per warp instruction whatever
// its lane count, so the work is dealt to all lanes: basis values by
// (electron, shell), matrix entries one per lane, and the elimination in
// place on n x n entries (the identity's columns of the augmented form are
// produced where its pivot columns vanish, with the same operations). Pivots
// are compared as integers, off that pipe.
// ----------------------------------------------------------------------------
static __device__ bool warp_inverses(const SysDev& S, const double* sC, const double* sx, double* Ainv0,
                                                double* scr, int lane, double* resid = nullptr)
{
  const BlockMem bm = block_mem(S, const_cast<double*>(sC));
  double* chi = scr;                                    // [N][n_ao]
  double* M = chi + S.N * S.n_ao;                       // [n][n]
  double* fc = M + S.n_up * S.n_up;                     // [n] the pivot column
  int* perm = reinterpret_cast<int*>(fc + S.n_up);      // [n] row of the original matrix
#pragma unroll 1
  for (int u = lane; u < S.N * S.n_shell; u += 32) {
    const int i = u / S.n_shell, q = u - i * S.n_shell;
    shell_values(S, q, &sx[3 * i], &chi[i * S.n_ao]);
  }
  __syncwarp();
  bool ok = true;
#pragma unroll 1
  for (int spin = 0; spin < 2 && ok; ++spin) {
    const int n = spin == 0 ? S.n_up : S.n_dn, off = spin == 0 ? 0 : S.n_up;
    double* Ainv = spin ? Ainv0 + S.n_up * S.n_up : Ainv0;
    if (n == 0) break;
    // entry idx = lane, lane + 32, ... as (row, column): advanced without divisions
    const int dr = 32 / n, dc = 32 - dr * n, r0 = lane / n, c0 = lane - r0 * n;
#define LRDMC_ENTRIES(r, c) \
    for (int idx = lane, r = r0, c = c0; idx < n * n; idx += 32, r += dr, c += dc, c >= n ? (c -= n, ++r) : 0)
#pragma unroll 1
    LRDMC_ENTRIES(l, m) M[idx] = orbital_value(S, bm, &chi[(off + l) * S.n_ao], m);
    if (lane < n) perm[lane] = lane;
    __syncwarp();
    if (resid) {
      double res = 0.0;
#pragma unroll 1
      LRDMC_ENTRIES(l, q) {
        double a = (l == q) ? -1.0 : 0.0;
#pragma unroll 1
        for (int m = 0; m < n; ++m) a += M[l * n + m] * Ainv[m * n + q];
        res = fmax(res, fabs(a));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) res = fmax(res, __shfl_xor_sync(FULL_MASK, res, o));
      *resid = fmax(*resid, res);
    }
    // Singular Slater matrix: two equal-spin electrons on one point (the
    // determinant vanishes by antisymmetry; elimination would leave a residual
    // row of rounding size, not an exact zero), or a pivot that is zero or not
    // finite. No relative pivot threshold is applied: the orbitals of a heavy
    // atom span many orders of magnitude (a 1s value at a valence electron),
    // so pivots far below the largest entry of their column are legitimate,
    // and rounding noise amplified by that scale spread cannot be told apart
    // from a small genuine pivot.
    int coincide = 0;
#pragma unroll 1
    LRDMC_ENTRIES(l, q) {
      const double* a = &sx[3 * (off + l)];
      const double* b = &sx[3 * (off + q)];
      coincide |= l < q && a[0] == b[0] && a[1] == b[1] && a[2] == b[2];
    }
    if (__any_sync(FULL_MASK, coincide)) return false;
#pragma unroll 1
    for (int col = 0; col < n && ok; ++col) {
      // pivot row: largest |M[r][col]| for r >= col (n <= 32: one row per
      // lane), lowest r on ties, NaN passed over; the bits of non-negative
      // doubles order as the doubles
      long long best = -1;
      int br = col;
      if (lane >= col && lane < n) {
        const long long a = __double_as_longlong(M[lane * n + col]) & 0x7fffffffffffffffll;
        if (a <= 0x7ff0000000000000ll) { best = a; br = lane; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(FULL_MASK, best, o);
        const int orr = __shfl_xor_sync(FULL_MASK, br, o);
        if (ob > best || (ob == best && orr < br)) { best = ob; br = orr; }
      }
      if (best <= 0 || best >= 0x7ff0000000000000ll) { ok = false; break; }
      if (br != col) {
        if (lane < n) {
          const double t = M[col * n + lane];
          M[col * n + lane] = M[br * n + lane];
          M[br * n + lane] = t;
        }
        if (lane == 0) {
          const int t = perm[col];
          perm[col] = perm[br];
          perm[br] = t;
        }
        __syncwarp();
      }
      const double inv = 1.0 / M[col * n + col];
      if (lane < n) fc[lane] = M[lane * n + col];
      __syncwarp();
      if (lane < n) M[col * n + lane] = lane == col ? inv : M[col * n + lane] * inv;
      __syncwarp();
#pragma unroll 1
      LRDMC_ENTRIES(r, c) {
        const double f = fc[r];
        if (r != col && f != 0.0) M[idx] = fma(-f, M[col * n + c], c == col ? 0.0 : M[idx]);
      }
      __syncwarp();
    }
    if (ok) {
#pragma unroll 1
      LRDMC_ENTRIES(m, c) Ainv[m * n + perm[c]] = M[idx];
    }
    __syncwarp();
#undef LRDMC_ENTRIES
  }
  return ok;
}

// ----------------------------------------------------------------------------
// One evaluation of all P lattice moves out of the walker's configuration
// (Eq. 1 lattice, fixed-node rates) and of its continuous local energy.
// On return sT holds T_c, b and el are warp-uniform. ratio_out (global,
// nullable) receives psi_G(x')/psi_G(x) for every move.
//
// Bound by the FP64 pipe: an instruction holds it for 64 cycles whatever its
// lane count. So the local energy is dealt to all lanes (el_L parts per
// electron, combined by shuffles), a lane evaluates the two moves +-h e_k,
// square roots take three operations of that pipe, and the e-e Pade sum is one
// running fraction, c r/(1 + b r) = c/b - (c/b)/(1 + b r), whose constant
// cancels (three operations per partner instead of nine; for b below 1/4,
// where that form would lose digits, and above 2^20 term by term). Distances
// come from the differences of positions: D + h^2 +- 2 h (y_ik - y_jk), as in
// eval64.cuh, is as fast to 1 % (Ne, 1021 walkers, 4 intervals: 7.45 ms
// against 7.54, 10.34 before this form), but its absolute error of 2^-53 h^2
// costs a move that lands close to the partner the digits this mode stands for.
// ----------------------------------------------------------------------------
// den's power of two out of num/den (exact)
__device__ __forceinline__ void pow2_rescale64(double& num, double& den)
{
  const int e = (__double2hiint(den) >> 20) & 0x7ff;
  const double s = __hiloint2double((2046 - min(e, 2045)) << 20, 0);
  num *= s;
  den *= s;
}

template <bool NJ>
__device__ void warp_eval(const SysDev& S, const double* sC, const LatDev& L, const WarpMem& wm,
                          int lane, double* ratio_out, double& b, double& el, double* grad_out = nullptr,
                          bool moves = true)
{
  const int N = S.N, nao = S.n_ao, nu = S.n_up, E = S.el_E, Lp = S.el_L;
  const BlockMem bm = block_mem(S, const_cast<double*>(sC));
  double* see_i = wm.Ssum;                               // [N] e-e sums: of c q, or c r q (below b = 1/4)
  double* sen_i = reinterpret_cast<double*>(wm.Sn);      // [N] e-n sums and the neural terms
  const bool recip = S.ee_recip != 0;
  // projected inverse columns: v[i][mu] = sum_m C[mu][m] Ainv_sigma[m][l_i]
#pragma unroll 1
  for (int idx = lane; idx < N * nao; idx += 32) {
    int i = idx / nao, mu = idx % nao;
    int spin = i < nu ? 0 : 1, l = i < nu ? i : i - nu, n = spin ? S.n_dn : nu;
    const double* A = spin ? wm.A + nu * nu : wm.A;
    wm.v[idx] = project_ao(S, bm, A, mu, l, n);
  }
  __syncwarp();
  // local energy: E electrons at a time, Lp lanes (parts) each
  double total = 0.0;
  const int part = lane / E;
#pragma unroll 1
  for (int i0 = 0; i0 < N; i0 += E) {
    const int i = i0 + lane - part * E;
    const bool act = part < Lp && i < N;
    double gD[3] = {0.0, 0.0, 0.0}, gJ[3] = {0.0, 0.0, 0.0}, see = 0.0, sen = 0.0;
    if (act) {
      const double* ri = &wm.x[3 * i];
      double val = 0.0, lap = 0.0, V = 0.0;
#pragma unroll 1
      for (int gi = part; gi < S.n_grp64; gi += Lp)
        ao_dot<true>(S, &wm.v[i * nao], ri, S.grp64_first[gi], S.grp64_first[gi + 1], val, gD, lap);
      const int si = spin_of(S, i);
#pragma unroll 1
      for (int t = part; t < N - 1; t += Lp) {
        const int j = t < i ? t : t + 1;
        const double d0 = ri[0] - wm.x[3 * j], d1 = ri[1] - wm.x[3 * j + 1], d2 = ri[2] - wm.x[3 * j + 2];
        const double r = sqrt64(d0 * d0 + d1 * d1 + d2 * d2);
        const double c = (spin_of(S, j) == si) ? S.c_par : S.c_anti;
        // 1/(1 + b r) and 1/r from one division (a pair on one point: 1 and
        // infinity, so that its Jastrow sum, and with it the moves, stay finite)
        const double u = fma(S.b_ee, r, 1.0), w = 1.0 / (r * u), inv = __double2hiint(r) ? w * r : 1.0, ir = w * u;
        const double cq = c * inv;
        see += recip ? cq : cq * r;
        double u1 = cq * inv, u2 = -2.0 * S.b_ee * u1 * inv;
        if (NJ) {
          double g, g1, g2;
          nj_value3(S, nj_ch_ee(S, i, j), r, g, g1, g2);
          u1 += g1; u2 += g2; sen += g;
        }
        const double a = u1 * ir;
        gJ[0] += a * d0; gJ[1] += a * d1; gJ[2] += a * d2;
        lap += u2 + 2.0 * a;
        if (j > i && S.ee_on) V += ir;
      }
#pragma unroll 1
      for (int I = part; I < S.n_nuc; I += Lp) {
        const double d0 = ri[0] - S.nuc[I][0], d1 = ri[1] - S.nuc[I][1], d2 = ri[2] - S.nuc[I][2];
        const double r = sqrt64(d0 * d0 + d1 * d1 + d2 * d2);
        const double b1 = S.en_b1[I], ir = 1.0 / r;
        double u1 = 0.0, u2 = 0.0;
        if (b1 != 0.0) {
          const double inv = 1.0 / (1.0 + S.en_b2 * r);
          u1 = -b1 * inv * inv;
          u2 = -2.0 * S.en_b2 * u1 * inv;
          sen -= b1 * r * inv;
        }
        if (NJ) {
          double g, g1, g2;
          nj_value3(S, 2 + S.nj_species[I], r, g, g1, g2);
          u1 += g1; u2 += g2; sen += g;
        }
        const double a = u1 * ir;
        gJ[0] += a * d0; gJ[1] += a * d1; gJ[2] += a * d2;
        lap += u2 + 2.0 * a;
        V -= S.Z[I] * ir;
      }
      total += V - 0.5 * lap;
    }
    // combine the parts of each electron (lane part * E + i)
    if (Lp > 1) {
#pragma unroll 1
      for (int o = S.el_top; o > 0; o >>= 1) {
        const bool take = part < o && part + o < Lp;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          double t = __shfl_down_sync(FULL_MASK, gD[k], o * E);
          if (take) gD[k] += t;
          t = __shfl_down_sync(FULL_MASK, gJ[k], o * E);
          if (take) gJ[k] += t;
        }
        double t = __shfl_down_sync(FULL_MASK, see, o * E);
        if (take) see += t;
        t = __shfl_down_sync(FULL_MASK, sen, o * E);
        if (take) sen += t;
      }
    }
    if (part == 0 && act) {
      see_i[i] = see;
      sen_i[i] = sen;
      double quad = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        quad += gJ[k] * (gJ[k] + 2.0 * gD[k]);
        if (grad_out) grad_out[3 * i + k] = gD[k] + gJ[k];
      }
      total -= 0.5 * quad;
    }
  }
  el = warp_sum(total) + S.V_nn;
  __syncwarp();
  if (!moves) {
    b = 0.0;
    return;
  }
  // the moves: lanes over (electron, grid, axis), both directions each
  const int G = L.G, units = 3 * G * N;
#pragma unroll 1
  for (int u = lane; u < units; u += 32) {
    const int i = u / (3 * G), rem = u - i * 3 * G, g = rem / 3, k = rem - 3 * g;
    const double h = g ? L.ap : L.a, h2 = h * h;
    const double* ri = &wm.x[3 * i];
    const double he[3] = {h * wm.R[k], h * wm.R[3 + k], h * wm.R[6 + k]};
    double rdet[2], jn[2] = {0.0, 0.0}, mid[2] = {INFINITY, INFINITY};
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {
      const double p[3] = {m ? ri[0] - he[0] : ri[0] + he[0], m ? ri[1] - he[1] : ri[1] + he[1],
                           m ? ri[2] - he[2] : ri[2] + he[2]};
      double none[3], lap, acc = 0.0, jm = 0.0;
      ao_dot<false>(S, &wm.v[i * nao], p, 0, S.n_shell, acc, none, lap);
      if (m) rdet[1] = acc;
      else rdet[0] = acc;
#pragma unroll 1
      for (int I = 0; I < S.n_nuc; ++I) {
        if (!NJ && S.en_b1[I] == 0.0) continue;
        const double d0 = p[0] - S.nuc[I][0], d1 = p[1] - S.nuc[I][1], d2 = p[2] - S.nuc[I][2];
        const double r = sqrt64(d0 * d0 + d1 * d1 + d2 * d2);
        if (S.en_b1[I] != 0.0) jm -= S.en_b1[I] * r / (1.0 + S.en_b2 * r);
        if (NJ) jm += nj_value(S, 2 + S.nj_species[I], r);
      }
      if (m) jn[1] = jm;
      else jn[0] = jm;
    }
    if (G == 2) {
      // |d +- h e/2|^2 of the nearest heavy nucleus
#pragma unroll 1
      for (int I = 0; I < S.n_nuc; ++I) {
        if (!S.heavy[I]) continue;
        const double d0 = ri[0] - S.nuc[I][0], d1 = ri[1] - S.nuc[I][1], d2 = ri[2] - S.nuc[I][2];
        const double q = d0 * d0 + d1 * d1 + d2 * d2 + 0.25 * h2, w = d0 * he[0] + d1 * he[1] + d2 * he[2];
        mid[0] = fmin(mid[0], q + w);
        mid[1] = fmin(mid[1], q - w);
      }
    }
    double jee[2] = {0.0, 0.0};
    const int si = spin_of(S, i);
#pragma unroll 1
    for (int sp = 0; sp < 2; ++sp) {
      const int j0 = sp ? nu : 0, j1 = sp ? N : nu;
      const double c = sp == si ? S.c_par : S.c_anti;
      double num[2] = {0.0, 0.0}, den[2] = {1.0, 1.0};
#pragma unroll 1
      for (int j = j0; j < j1; ++j) {
        if (j == i) continue;
        const double d0 = ri[0] - wm.x[3 * j], d1 = ri[1] - wm.x[3 * j + 1], d2 = ri[2] - wm.x[3 * j + 2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          // from the differences: D + h^2 +- 2 h p loses a move that lands close to the partner
          const double w0 = m ? d0 - he[0] : d0 + he[0], w1 = m ? d1 - he[1] : d1 + he[1],
                       w2 = m ? d2 - he[2] : d2 + he[2];
          const double r = sqrt64(fma(w0, w0, fma(w1, w1, w2 * w2))), q = fma(S.b_ee, r, 1.0);
          if (recip) {
            num[m] = fma(num[m], q, den[m]);
            den[m] *= q;
          } else {
            num[m] += r / q;
          }
          if (NJ) jn[m] += nj_value(S, nj_ch_ee(S, i, j), r);
        }
        if (recip && ((j - j0) & 15) == 15) {
          pow2_rescale64(num[0], den[0]);
          pow2_rescale64(num[1], den[1]);
        }
      }
#pragma unroll
      for (int m = 0; m < 2; ++m) jee[m] += c * (recip ? num[m] / den[m] : num[m]);
    }
    const int c0 = (i * G + g) * 6 + 2 * k;
    const double fac = recip ? -1.0 / S.b_ee : 1.0, inv2 = g ? L.inv2ap2 : L.inv2a2;
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {
      const double dJ = fac * ((m ? jee[1] : jee[0]) - see_i[i]) + ((m ? jn[1] : jn[0]) - sen_i[i]);
      const double rho = (m ? rdet[1] : rdet[0]) * exp(dJ);
      double w = 1.0;
      if (G == 2) {
        const double q = L.p_coef * (m ? mid[1] : mid[0]);
        const double pm = L.pkind == 0 ? exp(-q) : 1.0 / (1.0 + q);
        w = g ? 1.0 - pm : pm;
      }
      const double T = rho > 0.0 ? w * inv2 * rho : 0.0;
      wm.T[c0 + m] = T;
      if (ratio_out) ratio_out[c0 + m] = rho;
    }
  }
  __syncwarp();
  b = warp_scan(wm.T, 6 * G * N, lane, 0.0, nullptr, nullptr);
}

// ----------------------------------------------------------------------------
// The lattice moves of the mixed mode (LRDMC_PRECISION_FP32) in single
// precision. They read the leading floats of the evaluation's double-float
// state in shared memory (positions, rotation, projected inverse columns,
// Jastrow sums); rates are stored as double-floats with a zero low part.
// ----------------------------------------------------------------------------
__device__ __forceinline__ float dot3(float a0, float a1, float a2)
{
  return a0 * a0 + a1 * a1 + a2 * a2;
}

// Slater radial part r^m e^(-zeta r) (e given) or a Gaussian contraction.
__device__ __forceinline__ float radial_value_m(const ShellDev& sh, const DfShell& dsh, float r, float r2, float e)
{
  if (sh.kind == 0) {
    if (sh.m_int >= 0) {
      float pw = 1.0f;
      for (int j = 0; j < sh.m_int; ++j) pw = pw * r;
      return pw * e;
    }
    float lr = logf(r);
    return expf(dsh.m.hi * lr) * e;
  }
  float acc = 0.0f;
  for (int p = 0; p < sh.n_prim; ++p)
    acc = acc + dsh.coef[p].hi * expf(-(dsh.alpha[p].hi * r2));
  return acc;
}

__device__ __forceinline__ int solid_m(int l, const float d[3], float Sv[5])
{
  if (l == 0) {
    Sv[0] = 1.0f;
    return 1;
  }
  if (l == 1) {
    Sv[0] = d[0]; Sv[1] = d[1]; Sv[2] = d[2];
    return 3;
  }
  float xx = d[0] * d[0], yy = d[1] * d[1], zz = d[2] * d[2];
  Sv[0] = d[0] * d[1];
  Sv[1] = d[1] * d[2];
  Sv[2] = d[2] * d[0];
  Sv[3] = xx - yy;
  Sv[4] = zz + zz - (xx + yy);
  return 5;
}

// Per nucleus I (one distance each): the determinant ratio
// sum_mu v[mu] chi_mu(p) over the shells centred on I, and the e-n Jastrow
// -sum_I b1_I r/(1 + b2 r).
// The neural pair term (the double-float copy of the table): the cell at r.
__device__ __forceinline__ const df* nj_cell_m(const SysDev& S, int c, float rf)
{
  int k = (int)(sqrtf(rf) * S.nj_scale_f[c]);
  k = min(max(k, 0), S.nj_cells - 1);
  return S.nj_tab_df + ((size_t)c * S.nj_cells + k) * 8;
}

__device__ __forceinline__ void nj_load(const df* e, df E[8])
{
  const float4* q = reinterpret_cast<const float4*>(e);
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float4 v = __ldg(q + h);
    E[2 * h] = df_make(v.x, v.y);
    E[2 * h + 1] = df_make(v.z, v.w);
  }
}

__device__ __forceinline__ float nj_value_m(const SysDev& S, int c, float r)
{
  if (!(r < S.nj_rcut_f[c])) return 0.0f;
  df E[8];
  nj_load(nj_cell_m(S, c, r), E);
  const float t = (r - E[0].hi) * E[1].hi;
  float v = E[7].hi;
#pragma unroll
  for (int q = 6; q >= 2; --q) v = v * t + E[q].hi;
  return v;
}

// One nucleus's part of a lattice move: the e-n Jastrow terms (Pade and,
// when set, neural) into jen and the basis functions centred on it,
// contracted with the projected inverse column v, into rdet. d = r' - R_I,
// r2 = |d|^2.
template <bool NJ>
__device__ __forceinline__ void nucleus_term_m(const SysDev& S, const df* v, int I, const float d[3], float r2,
                                               float& rdet, float& jen)
{
  float r = sqrtf(r2);
  if (S.en_b1[I] != 0.0)
    jen = jen - S.D.en_b1[I].hi * r / (S.D.en_b2.hi * r + 1.0f);
  if (NJ) jen = jen + nj_value_m(S, 2 + S.nj_species[I], r);
  float e = 0.0f;
  for (int q = S.nuc_shell_begin[I]; q < S.nuc_shell_begin[I + 1]; ++q) {
    const ShellDev& sh = S.sh[q];
    const DfShell& dsh = S.D.sh[q];
    if (sh.kind == 0 && !sh.same_exp) e = expf(-(dsh.zeta.hi * r));
    float Rv = radial_value_m(sh, dsh, r, r2, e);
    float part;
    if (sh.l == 0) {
      part = v[sh.ao_offset].hi;
    } else {
      float Sv[5];
      int nf = solid_m(sh.l, d, Sv);
      part = 0.0f;
      for (int f = 0; f < nf; ++f) part = part + v[sh.ao_offset + f].hi * Sv[f];
    }
    rdet = rdet + part * Rv;
  }
}

template <bool NJ>
__device__ void nucleus_terms_m(const SysDev& S, const df* v, const float p[3], float& rdet, float& jen)
{
  rdet = 0.0f;
  jen = 0.0f;
  for (int I = 0; I < S.n_nuc; ++I) {
    const float d[3] = {p[0] - S.D.nuc[I][0].hi, p[1] - S.D.nuc[I][1].hi, p[2] - S.D.nuc[I][2].hi};
    nucleus_term_m<NJ>(S, v, I, d, dot3(d[0], d[1], d[2]), rdet, jen);
  }
}

// num and den times the power of two that brings den (positive, normal,
// below 2^127) into [1, 2): exact, so num/den keeps its value bit for bit.
__device__ __forceinline__ void pow2_rescale(float& num, float& den)
{
  const float s = __int_as_float((254 - ((__float_as_int(den) >> 23) & 0xff)) << 23);
  num *= s;
  den *= s;
}

// sum_{j != i} u_ee(|p - r_j|): the Pade terms c r/(1 + b r) (all of one
// sign) are summed as one running fraction num/den, so one division serves
// all partners. Every 16 partners pow2_rescale brings den back into [1, 2):
// the product of the (1 + b r) would otherwise leave the float exponent
// range (about 3.4e38), as 47 partners a few bohr away do; 16 factors fit
// while their geometric mean stays below 200.
template <bool NJ>
__device__ float jastrow_ee_m(const SysDev& S, const df* xd, int i, const float p[3])
{
  float num = 0.0f, den = 1.0f, nn = 0.0f;
  const int si = spin_of(S, i);
  const float b = S.D.b_ee.hi, cp = S.D.c_par.hi, ca = S.D.c_anti.hi;
  for (int j = 0; j < S.N; ++j) {
    if (j == i) continue;
    const float r = sqrtf(dot3(p[0] - xd[3 * j].hi, p[1] - xd[3 * j + 1].hi, p[2] - xd[3 * j + 2].hi));
    const float c = (spin_of(S, j) == si) ? cp : ca;
    const float dj = b * r + 1.0f;
    num = num * dj + c * r * den;
    den = den * dj;
    if (NJ) nn = nn + nj_value_m(S, nj_ch_ee(S, i, j), r);
    if ((j & 15) == 15) pow2_rescale(num, den);
  }
  return num / den + nn;
}

__device__ __forceinline__ float p_weight_m(const SysDev& S, const LatDev& L, const float m[3])
{
  float best = INFINITY;
  for (int I = 0; I < S.n_nuc; ++I) {
    if (!S.heavy[I]) continue;
    const float d2s = dot3(m[0] - S.D.nuc[I][0].hi, m[1] - S.D.nuc[I][1].hi, m[2] - S.D.nuc[I][2].hi);
    if (d2s < best) best = d2s;
  }
  if (L.pkind == 0) return expf(-(best * L.p_coef_df.hi));
  return 1.0f / (L.p_coef_df.hi * best + 1.0f);
}

// Chunked inclusive scan of the rates (as warp_scan) in single precision.
static __device__ float warp_scan_m(const df* T, int P, int lane, float target, int* pick, int* last)
{
  float carry = 0.0f;
  int p = -1, lp = -1;
  for (int base = 0; base < P; base += 32) {
    int c = base + lane;
    float t = (c < P) ? T[c].hi : 0.0f;
    float v = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      float y = __shfl_up_sync(FULL_MASK, v, o);
      if (lane >= o) v = v + y;
    }
    float C = carry + v;
    if (pick) {
      unsigned hit = __ballot_sync(FULL_MASK, (c < P) && target < C);
      if (p < 0 && hit) p = base + __ffs(hit) - 1;
      unsigned pos = __ballot_sync(FULL_MASK, (c < P) && t > 0.0f);
      if (pos) lp = base + 31 - __clz(pos);
    }
    carry = __shfl_sync(FULL_MASK, C, 31);
  }
  if (pick) { *pick = p; *last = lp; }
  return carry;
}

// One lattice move c of an evaluation (Eq. 1 lattice, fixed-node rate): the
// determinant and Jastrow ratios at the displaced position, p at the bond
// midpoint on the double grid, the rate T_c into Td[c]. Reads the
// evaluation's shared-memory state (projected inverse columns, positions,
// rotation and the Jastrow sums Sd of its local-energy pass).
template <bool NJ>
__device__ __forceinline__ void candidate_m(const SysDev& S, const LatDev& L, const WarpMem& wm, int c, df* Td,
                                            double* ratio_out)
{
  const int nao = S.n_ao;
  const int G = L.G, per_e = 6 * G;
  {
    const int i = c / per_e, rem = c - i * per_e, g = rem / 6, k = (rem % 6) >> 1;
    float h = g ? L.ap_df.hi : L.a_df.hi;
    if (c & 1) h = -h;
    const float e0 = wm.Rd[k].hi, e1 = wm.Rd[3 + k].hi, e2 = wm.Rd[6 + k].hi;
    float rdet, jen, jee, pm = 1.0f;
    const float ri[3] = {wm.xd[3 * i].hi, wm.xd[3 * i + 1].hi, wm.xd[3 * i + 2].hi};
    const float p[3] = {ri[0] + h * e0, ri[1] + h * e1, ri[2] + h * e2};
    nucleus_terms_m<NJ>(S, &wm.vd[i * nao], p, rdet, jen);
    jee = jastrow_ee_m<NJ>(S, wm.xd, i, p);
    if (G == 2) {
      const float hh = 0.5f * h;
      const float mid[3] = {ri[0] + hh * e0, ri[1] + hh * e1, ri[2] + hh * e2};
      pm = p_weight_m(S, L, mid);
    }
    float dJ = jee + jen - wm.Sd[i].hi;
    float rho = rdet * expf(dJ);
    float w = 1.0f;
    if (G == 2) w = g ? -pm + 1.0f : pm;
    float T = 0.0f;
    if (rho > 0.0f) T = w * (g ? L.inv2ap2_df.hi : L.inv2a2_df.hi) * rho;
    Td[c] = df_make(T, 0.0f);
    if (ratio_out) ratio_out[c] = (double)rho;
  }
}

}  // namespace lrdmc
#include "eval64.cuh"
namespace lrdmc {

// The mixed mode's evaluation: projected columns, local energy and Jastrow
// sums as in the double-float mode, the moves in single precision (they read
// the double-float values' leading floats).
template <bool NJ>
__device__ __forceinline__ double prelude32(const SysDev& S, const double* sC, const WarpMem& wm, const Lean& lt,
                                            int lane, int moved)
{
  const double el = prelude64<NJ, true, false>(S, sC, wm, lt, lane, moved);
  total_jastrow64(S, wm, lane);
  return el;
}

template <bool NJ>
__device__ void warp_eval32(const SysDev& S, double* sC, const LatDev& L, const WarpMem& wm, int lane,
                            double* ratio_out, double& b, double& el)
{
  el = prelude32<NJ>(S, sC, wm, lean_mem(S, sC), lane, -1);
  const int P = 6 * L.G * S.N;
  df* Td = reinterpret_cast<df*>(wm.T);  // rates stored as double-floats
  for (int c = lane; c < P; c += 32) candidate_m<NJ>(S, L, wm, c, Td, ratio_out);
  __syncwarp();
  b = (double)warp_scan_m(Td, P, lane, 0.0f, nullptr, nullptr);
}

template <int PREC, bool NJ, bool NC>
__device__ __forceinline__ void warp_eval_any(const SysDev& S, double* sC, const LatDev& L, const WarpMem& wm,
                                              int lane, double* ratio_out, double& b, double& el,
                                              const float4* gt = nullptr)
{
  if (PREC == LRDMC_PRECISION_DF64) {
    warp_eval64<NJ, NC>(S, sC, L, wm, lane, ratio_out, b, el, gt);
  } else if (PREC == LRDMC_PRECISION_FP32) {
    warp_eval32<NJ>(S, sC, L, wm, lane, ratio_out, b, el);
  } else {
    warp_eval<NJ>(S, sC, L, wm, lane, ratio_out, b, el);
  }
}

// ----------------------------------------------------------------------------
// Sherman-Morrison update for electron i moving to p (warp-cooperative):
// y_n = sum_m phi_m(p) Ainv[m][n], ratio = y_l,
// Ainv[m][n] -= Ainv[m][l] (y_n - delta_nl) / ratio.
// ----------------------------------------------------------------------------
// The FP64 mode's update.
static __device__ bool warp_sm_update(const SysDev& S, const double* sC, const WarpMem& wm, int i,
                                                 const double* p, int lane)
{
  const int nu = S.n_up;
  const int spin = i < nu ? 0 : 1, l = i < nu ? i : i - nu, n = spin ? S.n_dn : nu;
  double* A = spin ? wm.A + nu * nu : wm.A;
  const BlockMem bm = block_mem(S, const_cast<double*>(sC));
  double* chi = wm.scr;            // [n_ao]
  double* phi = chi + S.n_ao;      // [n]
  double* y = phi + n;             // [n]
  double* col = y + n;             // [n]
#pragma unroll 1
  for (int q = lane; q < S.n_shell; q += 32) shell_values(S, q, p, chi);
  __syncwarp();
  for (int m = lane; m < n; m += 32) {
    phi[m] = orbital_value(S, bm, chi, m);
  }
  __syncwarp();
  for (int q = lane; q < n; q += 32) {
    double a = 0.0;
    for (int m = 0; m < n; ++m) a += phi[m] * A[m * n + q];
    y[q] = a;
    col[q] = A[q * n + l];
  }
  __syncwarp();
  double ratio = y[l];
  if (ratio == 0.0) return false;
  double inv = 1.0 / ratio;
  for (int idx = lane; idx < n * n; idx += 32) {
    int m = idx / n, q = idx % n;
    A[idx] -= col[m] * ((y[q] - (q == l ? 1.0 : 0.0)) * inv);
  }
  __syncwarp();
  return true;
}

// ----------------------------------------------------------------------------
// Record load / store.
// ----------------------------------------------------------------------------
__device__ __forceinline__ void load_record(const Layout& Lo, const double* rec, const WarpMem& wm,
                                            int lane, double& b, double& el)
{
  for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = rec[Lo.off_x + j];
  for (int j = lane; j < Lo.nu * Lo.nu + Lo.nd * Lo.nd; j += 32) wm.A[j] = rec[Lo.off_au + j];
  for (int j = lane; j < 9; j += 32) wm.R[j] = rec[Lo.off_R + j];
  for (int j = lane; j < Lo.P_max; j += 32) wm.T[j] = rec[Lo.off_T + j];
  b = rec[Lo.off_b];
  el = rec[Lo.off_el];
  __syncwarp();
}

__device__ __forceinline__ void store_record(const Layout& Lo, double* rec, const WarpMem& wm,
                                             int lane, double b, double el)
{
  __syncwarp();
  for (int j = lane; j < 3 * Lo.N; j += 32) rec[Lo.off_x + j] = wm.x[j];
  for (int j = lane; j < Lo.nu * Lo.nu + Lo.nd * Lo.nd; j += 32) rec[Lo.off_au + j] = wm.A[j];
  for (int j = lane; j < 9; j += 32) rec[Lo.off_R + j] = wm.R[j];
  for (int j = lane; j < Lo.P_max; j += 32) rec[Lo.off_T + j] = wm.T[j];
  if (lane == 0) {
    rec[Lo.off_b] = b;
    rec[Lo.off_el] = el;
  }
}

template <bool LEAN = false>
__device__ __forceinline__ void stage_coefficients(const SysDev& S, double* sC)
{
  if (LEAN) lean_stage(S, sC);
  BlockMem bm = block_mem(S, sC);
  for (int j = threadIdx.x; j < S.n_ao * S.n_mo; j += blockDim.x) sC[j] = S.C[j];
  for (int j = threadIdx.x; j < S.n_mo; j += blockDim.x) bm.col[j] = S.col_mask[j];
  for (int j = threadIdx.x; j < S.n_ao; j += blockDim.x) bm.row[j] = S.row_mask[j];
  __syncthreads();
}

// ----------------------------------------------------------------------------
// Kernels.
// ----------------------------------------------------------------------------
#if LRDMC_PART == 0
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_init(const __grid_constant__ SysDev S, const Layout Lo, const PopDev P, const double* x0)
{
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  stage_coefficients(S, sC);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int s = blockIdx.x * kWarpsPerBlock + wib;
  if (s >= P.W) return;
  WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
  for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = x0[(size_t)s * 3 * Lo.N + j];
  for (int j = lane; j < Lo.P_max; j += 32) wm.T[j] = 0.0;
  __syncwarp();
  bool ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane);
  if (!ok && lane == 0) atomicOr(P.err, kErrSingular);
  if (lane == 0) {
    double u[4];
    draw_uniforms(P.seed, (uint64_t)s, kIntervalInit, 0, kTagRot, u);
    rotation_matrix(u[0], u[1], u[2], wm.R);
    P.parent[s] = s;
    P.order[s] = s;
  }
  store_record(Lo, P.rec_src + (size_t)s * Lo.rec, wm, lane, NAN, NAN);
}

#endif  // LRDMC_PART == 0

template <int PREC>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_eval_all(const __grid_constant__ SysDev S, const Layout Lo, const LatDev L, const PopDev P)
{
  constexpr int PR = PREC & 3;         // the arithmetic (LRDMC_PRECISION_*)
  constexpr bool NJ = (PREC & 8) != 0;  // the neural pair term is set
  constexpr bool NC = (PREC & 4) != 0;  // the layout has no evaluation caches
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  stage_coefficients<(PREC & 3) != LRDMC_PRECISION_FP64>(S, sC);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int s = blockIdx.x * kWarpsPerBlock + wib;
  if (s >= P.W) return;
  WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
  double* rec = P.rec_src + (size_t)s * Lo.rec;
  double b, el;
  load_record(Lo, rec, wm, lane, b, el);
  warp_eval_any<PR, NJ, NC>(S, sC, L, wm, lane, nullptr, b, el, P.gt);
  if (!isfinite(el) || !isfinite(b)) {
    if (lane == 0) atomicOr(P.err, kErrNonFinite);
  }
  store_record(Lo, rec, wm, lane, b, el);
}

// ----------------------------------------------------------------------------
// Tail helpers of the interval kernel. Walkers make Poisson-distributed
// numbers of jumps, so at the end of an interval most warps of a block have
// no walker left while a few still run one. A warp whose fetch finds the
// queue empty attaches to a warp of its block that still runs a walker and,
// in every evaluation that warp publishes (projected columns, caches, local
// energy and Jastrow sums ready), takes chunks of 32 of its lattice moves.
// Owner and helpers run the same inlined move code (one loop of the kernel
// serves both roles), so a rate has the same bits whoever computes it and
// no second copy of the move code competes for the instruction cache. Every
// wait is bounded (kTeamSpin polls with a short sleep); one that runs out
// sets kErrTimeout in the error word and gives up, reported to the host as
// LRDMC_ERR_TIMEOUT, never a hang.
// ----------------------------------------------------------------------------
constexpr int kMaxIntervalWarps = 16;
struct TeamSlot {
  int attach;  // bit 31: closed to helpers; bits 0-30: helpers attached
  int pub;     // published evaluation (generation << 4 | participants), or kTeamRelease
  int next;    // next chunk of moves of the published evaluation
  int done;    // helpers finished with the published evaluation
  int gen;     // the owner's generation counter
  int pad[3];
};
constexpr int kTeamClosed = (int)0x80000000;
constexpr int kTeamRelease = -1;
constexpr int kTeamSpin = 1 << 22;

__device__ __forceinline__ int ld_vol(const int* p) { return *(const volatile int*)p; }

// Owner, after the evaluation's first part: the number of helpers taking
// part (0: alone; a helper that attaches later joins at the next one).
__device__ __forceinline__ int team_publish(TeamSlot* t, int lane)
{
  int nh = 0;
  if (lane == 0) {
    nh = ld_vol(&t->attach);
    nh = nh < 0 ? 0 : (nh > 15 ? 15 : nh);
  }
  nh = __shfl_sync(FULL_MASK, nh, 0);
  if (nh == 0) return 0;
  __threadfence_block();  // this lane's writes of the evaluation state
  __syncwarp();
  if (lane == 0) {
    const int g = t->gen + 1;
    t->gen = g;
    t->next = 0;
    t->done = 0;
    __threadfence_block();
    atomicExch(&t->pub, (g << 4) | nh);
  }
  __syncwarp();
  return nh;
}

// The moves of an evaluation in chunks of 32: alone (t == nullptr) in
// order, or taken in turn from t->next by the owner and its helpers.
// A unit is one move, in the double-float mode the two moves along one axis.
template <bool DF, bool NJ, bool NC>
__device__ __forceinline__ void chunked_moves(const SysDev& S, const LatDev& L, const WarpMem& wm, const Lean& lt,
                                              TeamSlot* t, int units, int lane, const float4* gt)
{
  df* Td = reinterpret_cast<df*>(wm.T);
  // in a team chunks of 16 where whole ones would not go round: 3 % faster
  // than 32 for Ne (60 units); 32 for Kr (216), 40.5 ms to 39.3 for 4096
  // walkers, since a half chunk costs as many issue slots as a whole one
  const int cs = t && units <= 32 * ((ld_vol(&t->pub) & 15) + 1) ? 16 : 32;
#pragma unroll 1
  for (int c0 = 0;; c0 += 32) {
    if (t) {
      int c = 0;
      if (lane == 0) c = atomicAdd(&t->next, cs);
      c0 = __shfl_sync(FULL_MASK, c, 0);
    }
    if (c0 >= units) break;
    if (lane < cs && c0 + lane < units) {
      if (DF) moves64<NJ, NC>(S, L, wm, lt, c0 + lane, Td, nullptr, gt);
      else candidate_m<NJ>(S, L, wm, c0 + lane, Td, nullptr);
    }
  }
  if (t) __threadfence_block();
  __syncwarp();
}

// Owner: wait until the nh helpers of the published evaluation are done.
__device__ __forceinline__ void team_wait_helpers(TeamSlot* t, int nh, int lane, int* err)
{
  if (lane == 0) {
    int it = 0;
    while (ld_vol(&t->done) < nh && ++it < kTeamSpin) __nanosleep(32);
    if (it >= kTeamSpin) atomicOr(err, kErrTimeout);
    __threadfence_block();
  }
  __syncwarp();
}

// Owner, when its walker's interval is over: close the slot and release
// the helpers attached to it.
__device__ __forceinline__ void team_close(TeamSlot* t, int lane)
{
  if (lane == 0) {
    atomicOr(&t->attach, kTeamClosed);
    atomicExch(&t->pub, kTeamRelease);
  }
  __syncwarp();
}

__device__ __forceinline__ void team_open(TeamSlot* t, int lane)
{
  if (lane == 0) {
    t->pub = 0;
    __threadfence_block();
    atomicExch(&t->attach, 0);
  }
  __syncwarp();
}

// Helper: attach to the open slot of the block with the fewest helpers;
// returns the owner's warp (or -1: no warp of the block runs a walker) and
// the helper's index among that owner's helpers.
__device__ __forceinline__ int team_attach(TeamSlot* slots, int nw, int wib, int lane, int& kidx)
{
  int o = -1, kk = 0;
  if (lane == 0) {
    for (int tries = 0; tries < 64 && o < 0; ++tries) {
      int best = -1, bc = 0x7fffffff;
      for (int q = 0; q < nw; ++q) {
        const int a = ld_vol(&slots[q].attach);
        if (q == wib || a < 0) continue;  // itself, or closed (bit 31)
        if (a < bc) { bc = a; best = q; }
      }
      if (best < 0) break;
      if (atomicCAS(&slots[best].attach, bc, bc + 1) == bc) { o = best; kk = bc; }
    }
  }
  kidx = __shfl_sync(FULL_MASK, kk, 0);
  return __shfl_sync(FULL_MASK, o, 0);
}

// Helper: wait for an evaluation of its owner it takes part in (returns
// its generation), a release (-1) or a timeout (-2, reported).
__device__ __forceinline__ int team_wait_publication(TeamSlot* t, int kidx, int last, int lane, int* err)
{
  int g = 0;
  if (lane == 0) {
    int it = 0;
    for (;;) {
      const int pub = ld_vol(&t->pub);
      if (pub == kTeamRelease) { g = -1; break; }
      if ((pub >> 4) > last && kidx < (pub & 15)) { g = pub >> 4; break; }
      if (++it >= kTeamSpin) { g = -2; atomicOr(err, kErrTimeout); break; }
      __nanosleep(64);
    }
    __threadfence_block();
  }
  g = __shfl_sync(FULL_MASK, g, 0);
  __syncwarp();  // orders lane 0's observation before every lane's reads
  return g;
}

static __shared__ TeamSlot g_team[kMaxIntervalWarps];

// Per-warp state of the interval loop that the move code does not need: it
// lives in shared memory (written by lane 0, read by the whole warp after a
// __syncwarp), so that the registers of the move code are the same as in a
// loop without helpers.
struct WarpState {
  double tau_left, logw, b, el;
  unsigned long long m;
  df bdf;
  int s, jumps, finish;
  int fresh;  // no evaluation of this walker by this warp yet
  int owner, kidx, last;
};
static __shared__ WarpState g_ws[kMaxIntervalWarps];

// The interval loop of the FP32-pipe evaluations (double-float and FP32):
// each warp is an owner while it runs a walker (the same steps, draws and
// arithmetic as the loop of the FP64 mode below), then a helper of the
// warps of its block that still run one.
template <int PR, bool NJ, bool NC>
__device__ __forceinline__ void interval_team(const SysDev& S, const Layout& Lo, const LatDev& L, const PopDev& P,
                                              double* sC, uint64_t k, bool recompute, int lane, int wib)
{
  const int P_moves = S.N * 6 * L.G;
  constexpr bool kDf = PR == LRDMC_PRECISION_DF64;
  const int units = kDf ? P_moves / 2 : P_moves;
  const Lean lt = lean_mem(S, sC);
  TeamSlot* mine = &g_team[wib];
  WarpState& st = g_ws[wib];
  enum { kNeed, kOwner, kSearch, kHelper, kDone };
  int mode = kNeed;
  for (;;) {
    if (mode == kNeed) {
      int idx = 0;
      if (lane == 0) idx = atomicAdd(P.counter, 1);
      idx = __shfl_sync(FULL_MASK, idx, 0);
      if (idx >= P.W) {
        // out of walkers: a kernel launched after this one with programmatic
        // stream serialization (the pipelined batch) may start on the SMs
        // this block frees
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        mode = P.helpers ? kSearch : kDone;
      } else {
        if (P.helpers) team_open(mine, lane);
        const int s = bounded(P.order[idx], P.W, P.err);
        const WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
        double b, el;
        load_record(Lo, P.rec_src + (size_t)bounded(P.parent[s], P.W, P.err) * Lo.rec, wm, lane, b, el);
        if (recompute) {
          double rs = 0.0;
          bool ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane, &rs);
          if (!ok && lane == 0) atomicOr(P.err, kErrSingular);
          if (lane == 0 && isfinite(rs)) atomicMax(P.resid, (unsigned long long)__double_as_longlong(rs));
        }
        // the running sums of the cached rates, for the first heat bath
        if (kDf) rate_scan64(reinterpret_cast<const df*>(wm.T), P_moves, lane, wm.pfx);
        if (lane == 0) {
          st.s = s;
          st.b = b;
          st.el = el;
          st.bdf = kDf ? dl_from_double(b) : df_from_double(b);
          st.fresh = 1;
          st.tau_left = P.tau;
          st.logw = 0.0;
          st.jumps = 0;
          st.m = 0;
          st.finish = 0;
        }
        __syncwarp();
        mode = kOwner;
      }
    }
    if (mode == kDone) break;
    int target = wib, nh = 0;
    if (mode == kOwner) {
      const WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
      const double b = st.b, el = st.el, tau_left = st.tau_left;
      const df bdf = st.bdf;
      bool over = st.finish != 0;
      double t = 0.0, logw = st.logw;
      const int it = (int)(st.m % kDrawAhead);
      const df* draws = reinterpret_cast<const df*>(wm.dr + it * kDrawWords);
      if (!over) {
        if (it == 0) {
          if (kDf) draw_ahead64(P.seed, (uint64_t)st.s, k, (uint64_t)st.m, wm.dr, lane, S, lt);
          else draw_ahead32(P.seed, (uint64_t)st.s, k, (uint64_t)st.m, wm.dr, lane);
        }
        const df nl = draws[9];
        if (kDf) t = b > 0.0 ? df_to_double(dl_mul(nl, dl_norm(dl_rcp(bdf)))) : INFINITY;
        else t = b > 0.0 ? (double)(nl.hi / bdf.hi) : INFINITY;
        if (t >= tau_left) {
          logw -= tau_left * (el - P.e_trial);
          over = true;
        }
      }
      int i = 0, pick = -1;
      if (!over) {
        logw -= t * (el - P.e_trial);
        // heat bath over the cached rates
        if (kDf) {
          pick = heat_bath64(reinterpret_cast<const df*>(wm.T), P_moves, lane, wm.pfx,
                             dl_norm(dl_mul(draws[10], bdf)));
        } else {
          int lastc;
          warp_scan_m(reinterpret_cast<const df*>(wm.T), P_moves, lane, draws[10].hi * bdf.hi, &pick,
                             &lastc);
          if (pick < 0) pick = lastc;
        }
        if (pick < 0) {  // no allowed move: cannot happen with b > 0
          if (lane == 0) atomicOr(P.err, kErrNonFinite);
          over = true;
        }
      }
      if (!over) {
        const int per_e = 6 * L.G;
        i = pick / per_e;
        const int rem = pick - i * per_e, g = rem / 6, kx = (rem % 6) >> 1;
        const double sign = (pick & 1) ? -1.0 : 1.0, h = g ? L.ap : L.a;
        // both arithmetics keep the update in IEEE double
        const bool sm_ok = sm_update64(S, sC, wm, lt, i, sign * h, kx, lane);
        if (!sm_ok) {
          if (lane == 0) atomicOr(P.err, kErrSingular);
          over = true;
        }
      }
      if (over) {
        if (P.helpers) team_close(mine, lane);
        store_record(Lo, P.rec_dst + (size_t)st.s * Lo.rec, wm, lane, b, el);
        if (lane == 0) {
          const int s = st.s;
          P.logw[s] = logw;
          P.wgt[s] = exp(logw);
          P.el_end[s] = el;
          P.jumps[s] = st.jumps;
        }
        __syncwarp();
        mode = kNeed;
        continue;
      }
      if (lane == 0) {
        st.logw = logw;
        st.tau_left = tau_left - t;
      }
      if (lane < 3) wm.x[3 * i + lane] = wm.sm[lane];
      __syncwarp();
      if (lane < 9) wm.R[lane] = wm.dr[it * kDrawWords + lane];
      __syncwarp();
      double eln;
      if (kDf) eln = prelude64<NJ, NC>(S, sC, wm, lt, lane, st.fresh ? -1 : i);
      else eln = prelude32<NJ>(S, sC, wm, lt, lane, st.fresh ? -1 : i);
      if (lane == 0) {
        st.el = eln;
        st.fresh = 0;
      }
      if (P.helpers) nh = team_publish(mine, lane);
    } else {
      if (mode == kSearch) {
        int kidx;
        const int o = team_attach(g_team, blockDim.x >> 5, wib, lane, kidx);
        if (o < 0) {
          mode = kDone;
          continue;
        }
        if (lane == 0) {
          st.owner = bounded(o, blockDim.x >> 5, P.err);
          st.kidx = kidx;
          st.last = 0;
        }
        __syncwarp();
        mode = kHelper;
      }
      const int gw = team_wait_publication(&g_team[st.owner], st.kidx, st.last, lane, P.err);
      if (gw == -2) {
        mode = kDone;
        continue;
      }
      if (gw == -1) {
        mode = kSearch;
        continue;
      }
      if (lane == 0) st.last = gw;
      target = st.owner;
    }
    // the moves of the target walker's evaluation: one copy of the move
    // code for the owner alone, the owner with helpers, and the helpers
    {
      const WarpMem twm = warp_mem(Lo, S, sC + Lo.head + target * Lo.smem_warp);
      chunked_moves<kDf, NJ, NC>(S, L, twm, lt, (mode == kHelper || nh > 0) ? &g_team[target] : nullptr, units, lane,
                                 P.gt);
    }
    if (mode == kHelper) {
      if (lane == 0) atomicAdd(&g_team[target].done, 1);
      __syncwarp();
      continue;
    }
    if (nh > 0) team_wait_helpers(mine, nh, lane, P.err);
    const WarpMem own = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
    const df* Td = reinterpret_cast<const df*>(own.T);
    df bnew;
    if (kDf) bnew = rate_scan64(Td, P_moves, lane, own.pfx);
    else bnew = df_make(warp_scan_m(Td, P_moves, lane, 0.0f, nullptr, nullptr), 0.0f);
    const double b = df_to_double(bnew);
    if (lane == 0) {
      st.bdf = bnew;
      st.b = b;
      st.jumps = st.jumps + 1;
      int fin = 0;
      if (!isfinite(st.el) || !isfinite(b)) {
        atomicOr(P.err, kErrNonFinite);
        fin = 1;
      }
      if (st.m + 1 >= (unsigned long long)kMaxItersPerInterval) {
        atomicOr(P.err, kErrIters);
        fin = 1;
      }
      st.finish = fin;
      st.m = st.m + 1;
    }
    __syncwarp();
  }
}

// One interval of length tau for every walker slot (continuous-time
// projection of the cited LRDMC method): wait for an exponential time of
// rate b_x, decrease log w by (E_L - E_T) times the time spent, and at the
// end of the wait jump to move c with probability T_c / b_x.
#ifndef LRDMC_INTERVAL_MIN_BLOCKS
#define LRDMC_INTERVAL_MIN_BLOCKS 1
#endif
template <int PREC>
__global__ void __launch_bounds__(kMaxIntervalWarps * 32, LRDMC_INTERVAL_MIN_BLOCKS)
k_interval(const __grid_constant__ SysDev S, const Layout Lo, const LatDev L, const PopDev P)
{
  constexpr int PR = PREC & 3;         // the arithmetic (LRDMC_PRECISION_*)
  constexpr bool NJ = (PREC & 8) != 0;  // the neural pair term is set
  constexpr bool NC = (PREC & 4) != 0;  // the layout has no evaluation caches
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  // interval k from the device counter (advanced by k_comb_parents); the inverse
  // Slater matrices are recomputed at the start of every recompute_every-th
  // interval
  const uint64_t k = *P.kdev;
  const bool recompute = k > 0 && P.recompute_every > 0 && k % (uint64_t)P.recompute_every == 0;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (PR != LRDMC_PRECISION_FP64 && lane == 0) {
    g_team[wib].attach = kTeamClosed;
    g_team[wib].pub = 0;
    g_team[wib].next = 0;
    g_team[wib].done = 0;
    g_team[wib].gen = 0;
  }
  stage_coefficients<(PREC & 3) != LRDMC_PRECISION_FP64>(S, sC);  // ends with __syncthreads
  if constexpr (PR != LRDMC_PRECISION_FP64) {
    if (PR == LRDMC_PRECISION_DF64) interval_team<PR, NJ, NC>(S, Lo, L, P, sC, k, recompute, lane, wib);
    else interval_team<PR, NJ, true>(S, Lo, L, P, sC, k, recompute, lane, wib);
  } else {
    // the FP64 mode: every warp alone
    WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
    const int P_moves = S.N * 6 * L.G;
    for (;;) {
      int idx = 0;
      if (lane == 0) idx = atomicAdd(P.counter, 1);
      idx = __shfl_sync(FULL_MASK, idx, 0);
      if (idx >= P.W) {
        // out of walkers: a kernel launched after this one with programmatic
        // stream serialization (the pipelined batch) may start on the SMs
        // this block frees
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        break;
      }
      const int s = bounded(P.order[idx], P.W, P.err);
      const int src = bounded(P.parent[s], P.W, P.err);
      double b, el;
      load_record(Lo, P.rec_src + (size_t)src * Lo.rec, wm, lane, b, el);
      if (recompute) {
        double rs = 0.0;
        bool ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane, &rs);
        if (!ok && lane == 0) atomicOr(P.err, kErrSingular);
        if (lane == 0 && isfinite(rs)) atomicMax(P.resid, (unsigned long long)__double_as_longlong(rs));
      }
      double tau_left = P.tau, logw = 0.0;
      int jumps = 0;
      for (uint64_t m = 0;; ++m) {
        // both draws of this iteration at once: even lanes compute the
        // (waiting time, heat bath) block, odd lanes the rotation block
        uint64_t cb[4] = {(uint64_t)s, k, m, (lane & 1) ? kTagRot : kTagTimeHB};
        philox4x64_10(cb, P.seed, 0ull);
        uint64_t b0[4], b1[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          b0[j] = shfl_u64(cb[j], 0);
          b1[j] = shfl_u64(cb[j], 1);
        }
        const double t = b > 0.0 ? -log(to_u01(b0[0])) / b : INFINITY;
        if (t >= tau_left) {
          logw -= tau_left * (el - P.e_trial);
          break;
        }
        logw -= t * (el - P.e_trial);
        tau_left -= t;
        // heat bath over the cached rates
        int pick, last;
        warp_scan(wm.T, P_moves, lane, to_u01(b0[1]) * b, &pick, &last);
        if (pick < 0) pick = last;
        if (pick < 0) {  // no allowed move: cannot happen with b > 0
          if (lane == 0) atomicOr(P.err, kErrNonFinite);
          break;
        }
        const int per_e = 6 * L.G;
        const int i = pick / per_e, rem = pick - i * per_e, g = rem / 6, kx = (rem % 6) >> 1;
        const double sign = (pick & 1) ? -1.0 : 1.0, h = g ? L.ap : L.a;
        double pnew[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) pnew[d] = wm.x[3 * i + d] + sign * h * wm.R[3 * d + kx];
        const bool sm_ok = warp_sm_update(S, sC, wm, i, pnew, lane);
        if (!sm_ok) {
          if (lane == 0) atomicOr(P.err, kErrSingular);
          break;
        }
        if (lane < 3) wm.x[3 * i + lane] = pnew[lane];
        __syncwarp();
        rotation_matrix_warp(b1, wm.R, lane);
        __syncwarp();
        warp_eval_any<PR, NJ, NC>(S, sC, L, wm, lane, nullptr, b, el);
        ++jumps;
        if (!isfinite(el) || !isfinite(b)) {
          if (lane == 0) atomicOr(P.err, kErrNonFinite);
          break;
        }
        if (m + 1 >= (uint64_t)kMaxItersPerInterval) {
          if (lane == 0) atomicOr(P.err, kErrIters);
          break;
        }
      }
      store_record(Lo, P.rec_dst + (size_t)s * Lo.rec, wm, lane, b, el);
      if (lane == 0) {
        P.logw[s] = logw;
        P.wgt[s] = exp(logw);
        P.el_end[s] = el;
        P.jumps[s] = jumps;
      }
      __syncwarp();
    }
    // Launched early behind another system's interval kernel (pipelined
    // batch): this grid does not read that kernel's results, but it finishes
    // only after that kernel has, so that work after the chain in the stream
    // sees every kernel of the chain complete. Without a prerequisite grid
    // the wait returns at once.
  }
  if (threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

#if LRDMC_PART == 0
// Reconfiguration at the end of interval k, spread over G blocks of
// kCombThreads threads; block g owns the R = ceil(W/G) slots from g R. Its
// FP64 work (running sums, comb targets and comparisons) used to run on one
// SM, whose FP64 pipe took 38 us for 4096 walkers. Two kernels:
//   k_comb_sums     per block: running weight sums of its slots from the
//                   block's start (P.cum) and the block's totals (weights,
//                   w E_L, jumps)
//   k_comb_parents  per block: the block offsets off[g] (the same sequential
//                   sum in every block), the comb parents of its slots, and
//                   the next interval's processing order of its slots; the
//                   last block to finish writes the trace entry and clears
//                   the counters.
// Running sums: within a block, lane i of the first kCombLanes lanes sums
// its consecutive slots from zero (l_i(s)), and O_0 = 0, O_{i+1} = O_i +
// l_i(last slot of i) sequentially; c(s) = O_i + l_i(s). Over the blocks
// off[0] = 0, off[g+1] = off[g] + c(last slot of g), and C_s = off[g] +
// c(s). Each boundary repeats the rounding of the sum that ends the previous
// part, so C is non-decreasing (rounding is monotone, weights are >= 0) and
// slot t's parent is well defined: the smallest s with
// (t + xi) C_{W-1} / W < C_s, else W - 1. The sequential parts are kept
// short (FP64 additions have a long latency on this GPU): kCombLanes lanes
// per block, a few dozen blocks.
//
// Processing order of the next interval, longest expected first: a slot's
// number of jumps is about tau times the total rate b of the walker it
// receives. Each block sorts its slots by that b (64 buckets over the
// block's range, descending), and the blocks' sorted lists are dealt round
// robin into P.order: the r-th slot of every block comes before the
// (r+1)-th of any. The blocks are samples of the population, so this is
// close to a global sort, with no pass over the whole population. The order
// affects no result, only the tail of the next interval.
constexpr int kCombLanes = 16;

__device__ __forceinline__ int comb_slots(int W, int G) { return (W + G - 1) / G; }

__global__ void __launch_bounds__(kCombThreads) k_comb_sums(const PopDev P)
{
  // the parents kernel is launched behind this one with programmatic stream
  // serialization; its blocks may take their SMs now and wait for this grid
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NW = kCombThreads / 32;
  __shared__ double s_e[NW], s_tot[kCombLanes];
  __shared__ long long s_j[NW];
  const int W = P.W, G = gridDim.x, g = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int R = comb_slots(W, G);
  const int b0 = min(W, g * R), b1 = min(W, b0 + R);
  // the block's totals other than the weights: every thread
  double swe = 0.0;
  long long sj = 0;
  for (int s = b0 + t; s < b1; s += kCombThreads) {
    swe += P.wgt[s] * P.el_end[s];
    sj += P.jumps[s];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    swe += __shfl_xor_sync(FULL_MASK, swe, o);
    sj += __shfl_xor_sync(FULL_MASK, sj, o);
  }
  if (lane == 0) { s_e[wid] = swe; s_j[wid] = sj; }
  // the running sums: the first kCombLanes lanes, each a run of slots
  const int per = (b1 - b0 + kCombLanes - 1) / kCombLanes;
  const int lo = min(b1, b0 + t * per), hi = min(b1, lo + per);
  if (t < kCombLanes) {
    double l = 0.0;
    for (int s = lo; s < hi; ++s) l += P.wgt[s];
    s_tot[t] = l;
  }
  __syncthreads();
  if (t == 0) {
    double o = 0.0;
    for (int i = 0; i < kCombLanes; ++i) {
      const double ti = s_tot[i];
      s_tot[i] = o;
      o += ti;
    }
    P.part[g].w = o;  // = c(last slot of the block): the last lane with slots ends there
  }
  if (t == 32) {  // fixed-order sums of the warps' totals
    double es = 0.0;
    long long js = 0;
    for (int q = 0; q < NW; ++q) {
      es += s_e[q];
      js += s_j[q];
    }
    P.part[g].swe = es;
    P.part[g].jumps = js;
  }
  __syncthreads();
  if (t < kCombLanes) {
    const double O = s_tot[t];
    double c = 0.0;
    for (int s = lo; s < hi; ++s) {
      c += P.wgt[s];
      P.cum[s] = O + c;
    }
  }
}

// Running sum C_s of the comb: from shared memory when the population's sums
// were staged there, else off[block of s] + P.cum[s] (the same number).
__device__ __forceinline__ double comb_C(const double* s_cum, const double* s_off, const double* cum, int R, int s,
                                        bool in_smem)
{
  return in_smem ? s_cum[s] : s_off[s / R] + __ldcg(cum + s);
}

// Adds one to the shared counter of bucket q for every lane of the warp
// (lanes with q < 0 take no part) and returns this lane's old count plus
// its rank among the lanes with the same q: one shared-memory atomic per
// distinct bucket of the warp instead of one per lane.
__device__ __forceinline__ int bucket_take(int* cnt, int q, int lane)
{
  const unsigned peers = __match_any_sync(FULL_MASK, q);
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (lane == leader && q >= 0) base = atomicAdd(&cnt[q], __popc(peers));
  base = __shfl_sync(FULL_MASK, base, leader);
  return base + __popc(peers & ((1u << lane) - 1u));
}

// Position in P.order of the r-th slot (in the block's sorted order) of
// block g: the blocks hold R slots but for a shorter last non-empty block
// (Rl slots) and empty ones after it (Gn non-empty blocks); the first Rl
// ranks of all Gn blocks come first, round robin, then the further ranks of
// the Gn - 1 full blocks. A bijection of the slots onto 0..W-1.
__device__ __forceinline__ int comb_order_pos(int g, int r, int Gn, int Rl)
{
  return r < Rl ? r * Gn + g : Rl * Gn + (r - Rl) * (Gn - 1) + g;
}

__global__ void __launch_bounds__(kCombThreads) k_comb_parents(const PopDev P, const double* rec_next,
                                                              int rec_stride, int off_b)
{
  extern __shared__ double s_cum[];  // the running sums C_s (W <= kReconfigSmemW)
  __shared__ double s_off[kMaxCombBlocks + 1];
  __shared__ double s_pw[kMaxCombBlocks];
  __shared__ float s_lo[kCombThreads / 32], s_hi[kCombThreads / 32];
  __shared__ int s_cnt[64];
  __shared__ int s_last;
  const int W = P.W, G = gridDim.x, g = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int R = comb_slots(W, G);
  const bool in_smem = W <= kReconfigSmemW;
  // everything below reads the sums kernel's results
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint64_t k = *P.kdev;
  if (t < 64) s_cnt[t] = 0;
  for (int h = t; h < G; h += kCombThreads) s_pw[h] = __ldcg(&P.part[h].w);
  __syncthreads();
  if (t == 0) {
    double o = 0.0;
    for (int h = 0; h < G; ++h) {
      s_off[h] = o;
      o += s_pw[h];
    }
    s_off[G] = o;
  }
  __syncthreads();
  if (in_smem) {
    constexpr int U = 8;
    for (int s0 = 0; s0 < W; s0 += U * kCombThreads) {
      double v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = s0 + u * kCombThreads + t;
        v[u] = s < W ? __ldcg(P.cum + s) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = s0 + u * kCombThreads + t;
        if (s < W) s_cum[s] = s_off[s / R] + v[u];
      }
    }
    __syncthreads();
  }
  const double total = s_off[G];
  double uu[4];
  draw_uniforms(P.seed, kSlotGlobal, k, 0, kTagComb, uu);
  const double xi = uu[0];
  // t -> (t + xi) total / W; for W a power of two the product with 1/W is
  // the same number as the quotient (an exact scaling)
  const bool w_pow2 = (W & (W - 1)) == 0;
  const double inv_w = 1.0 / (double)W;
  const int b0 = min(W, g * R), b1 = min(W, b0 + R);
  const int chunk = (b1 - b0 + kCombThreads - 1) / kCombThreads;
  const int lo = min(b1, b0 + t * chunk), hi = min(b1, lo + chunk);
  // The targets grow with the slot, so the parents do too: a thread searches
  // for its first slot's parent, then steps forward from the previous one
  // (up to 8 steps, else a search over the rest), with the same comparisons.
  // The rate b of each slot's parent goes to the slot's bq byte's place in
  // shared memory (as a float, in the dynamic area after the sums).
  float* s_b = reinterpret_cast<float*>(s_cum + (in_smem ? W : 0));
  int a = 0;
  float bmin = INFINITY, bmax = -INFINITY;
  for (int tt = lo; tt < hi; ++tt) {
    const double num = ((double)tt + xi) * total;
    const double target = w_pow2 ? num * inv_w : num / (double)W;
    int steps = 0;
    while (tt > lo && steps < 8 && a < W - 1 && !(target < comb_C(s_cum, s_off, P.cum, R, a, in_smem))) {
      ++a;
      ++steps;
    }
    if (tt == lo || (steps == 8 && a < W - 1 && !(target < comb_C(s_cum, s_off, P.cum, R, a, in_smem)))) {
      int bnd = W - 1;
      while (a < bnd) {
        const int mid = (a + bnd) >> 1;
        if (target < comb_C(s_cum, s_off, P.cum, R, mid, in_smem)) bnd = mid; else a = mid + 1;
      }
    }
    a = bounded(a, W, P.err);
    P.parent[tt] = a;
    const float bt = (float)rec_next[(size_t)a * rec_stride + off_b];
    s_b[bounded(tt - b0, R, P.err)] = bt;
    bmin = fminf(bmin, bt);
    bmax = fmaxf(bmax, bt);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    bmin = fminf(bmin, __shfl_xor_sync(FULL_MASK, bmin, o));
    bmax = fmaxf(bmax, __shfl_xor_sync(FULL_MASK, bmax, o));
  }
  if (lane == 0) { s_lo[wid] = bmin; s_hi[wid] = bmax; }
  __syncthreads();
  // the block's slots by bucket of b, descending: counts, bases, positions
  float gmin = INFINITY, gmax = -INFINITY;
  for (int q = 0; q < kCombThreads / 32; ++q) {
    gmin = fminf(gmin, s_lo[q]);
    gmax = fmaxf(gmax, s_hi[q]);
  }
  const float scale = (gmax > gmin) ? 64.0f / (gmax - gmin) : 0.0f;
  const int n = b1 - b0;
  const int rounds = (n + kCombThreads - 1) / kCombThreads;  // warp-uniform
  for (int i = 0; i < rounds; ++i) {
    const int j = i * kCombThreads + t;
    int q = -1;
    if (j < n) {
      q = (int)((s_b[j] - gmin) * scale);
      q = 63 - min(63, max(0, q));
    }
    bucket_take(s_cnt, q, lane);
  }
  __syncthreads();
  if (t < 32) {  // exclusive scan of the 64 bucket counts (two per lane)
    const int c0 = s_cnt[2 * t], c1 = s_cnt[2 * t + 1];
    int incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL_MASK, incl, o);
      if (lane >= o) incl += y;
    }
    const int ex = incl - c0 - c1;
    s_cnt[2 * t] = ex;
    s_cnt[2 * t + 1] = ex + c0;
  }
  __syncthreads();
  const int Gn = (W + R - 1) / R;  // blocks with slots
  const int Rl = W - (Gn - 1) * R;  // slots of the last of them
  for (int i = 0; i < rounds; ++i) {
    const int j = i * kCombThreads + t;
    int q = -1;
    if (j < n) {
      q = (int)((s_b[j] - gmin) * scale);
      q = 63 - min(63, max(0, q));
    }
    const int r = bucket_take(s_cnt, q, lane);
    if (j < n) P.order[bounded(comb_order_pos(g, r, Gn, Rl), W, P.err)] = b0 + j;
  }
  // the last block to finish writes the trace entry
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(P.ticket, 1) == G - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (t < 32) {  // fixed-order sums over the blocks' totals
    double swe = 0.0;
    long long sj = 0;
    for (int h = t; h < G; h += 32) {
      swe += __ldcg(&P.part[h].swe);
      sj += __ldcg(&P.part[h].jumps);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      swe += __shfl_xor_sync(FULL_MASK, swe, o);
      sj += __shfl_xor_sync(FULL_MASK, sj, o);
    }
    if (t == 0) {
      const uint64_t kt = bounded(k, P.trace_cap, P.err);  // the trace slot
      P.trace[kt] = swe / total;
      P.trace[P.trace_cap + kt] = total / (double)W;
      P.trace[2 * P.trace_cap + kt] = (double)sj / (double)W;
      // the Sherman-Morrison residual measured at this interval's recompute
      // (-1: no recompute at this interval), then cleared for the next one
      const bool recomputed = k > 0 && P.recompute_every > 0 && k % (uint64_t)P.recompute_every == 0;
      P.trace[3 * P.trace_cap + kt] = recomputed ? __longlong_as_double((long long)*P.resid) : -1.0;
      *P.resid = 0ull;
      *P.moves += (unsigned long long)sj;
      *P.counter = 0;
      *P.ticket = 0;
      // every block has read k before taking its ticket: advance it
      *P.kdev = k + 1;
    }
  }
}
#endif  // LRDMC_PART == 0

// The FP64 mode's stateless evaluation of configuration c (one warp):
// inverses from x, then one evaluation of every lattice move and of the
// local energy. Returns false, with no output written, for a singular Slater
// matrix.
template <bool NJ>
__device__ __forceinline__ bool evaluate_config64(const SysDev& S, const Layout& Lo, const LatDev& L, const double* sC,
                                                  int c, int lane, int wib, const double* x, const double* rot,
                                                  double* ratio, double* T, double* b_out, double* el_out)
{
  WarpMem wm = warp_mem(Lo, S, const_cast<double*>(sC) + Lo.head + wib * Lo.smem_warp);
  for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = x[(size_t)c * 3 * Lo.N + j];
  for (int j = lane; j < 9; j += 32) wm.R[j] = rot[(size_t)c * 9 + j];
  __syncwarp();
  bool ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane);
  if (!ok) return false;
  const int P = S.N * 6 * L.G;
  double b, el;
  warp_eval<NJ>(S, sC, L, wm, lane, ratio ? ratio + (size_t)c * P : nullptr, b, el);
  if (T)
    for (int j = lane; j < P; j += 32) T[(size_t)c * P + j] = wm.T[j];
  if (lane == 0) {
    if (b_out) b_out[c] = b;
    if (el_out) el_out[c] = el;
  }
  return true;
}

// Warps and configurations of an evaluation block, at most.
constexpr int kMaxEvalWarps = 8, kMaxEvalConfigs = 8;

// The stateless evaluations of a block: r configurations, one warp each for
// the inverses, the local energy and the Jastrow sums, then every warp of the
// block takes chunks of all their moves. Bound, like the projection, by the
// latency of dependent chains: shared memory holds 4 warps' worth of Kr
// configurations per SM side by side, and a call with fewer configurations
// than SMs has one each, so the moves (about half of the work) get the warps
// that have no configuration of their own; and warps that pass through the
// same code together share its instruction fetches. 16384 Kr: 7.10 to 4.64
// ms; 37 H2O: 105 to 90 us. report: a singular configuration.
template <int PREC, class Report>
__device__ __forceinline__ void evaluate_block(const SysDev& S, const Layout& Lo, const LatDev& L, double* sC, int n,
                                               int r, const double* x, const double* rot, double* ratio, double* T,
                                               double* b_out, double* el_out, Report report)
{
  constexpr int PR = PREC & 3;         // the arithmetic (LRDMC_PRECISION_*)
  constexpr bool NJ = (PREC & 8) != 0;  // the neural pair term is set
  constexpr bool NC = (PREC & 4) != 0;  // the layout has no evaluation caches
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int c = blockIdx.x * r + wib;
  if constexpr (PR == LRDMC_PRECISION_FP64) {
    if (wib < r && c < n && !evaluate_config64<NJ>(S, Lo, L, sC, c, lane, wib, x, rot, ratio, T, b_out, el_out) &&
        lane == 0)
      report();
  } else {
    __shared__ int s_ok[kMaxEvalConfigs];
    const Lean lt = lean_mem(S, sC);
    const int P = S.N * 6 * L.G, units = PR == LRDMC_PRECISION_DF64 ? P / 2 : P;
    double el = 0.0;
    bool ok = false;
    if (wib < r) {
      if (c < n) {
        const WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
        for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = x[(size_t)c * 3 * Lo.N + j];
        for (int j = lane; j < 9; j += 32) wm.R[j] = rot[(size_t)c * 9 + j];
        __syncwarp();
        ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane);
        if (!ok && lane == 0) report();
        if (ok) {
          if (PR == LRDMC_PRECISION_DF64) el = prelude64<NJ, NC>(S, sC, wm, lt, lane, -1);
          else el = prelude32<NJ>(S, sC, wm, lt, lane, -1);
        }
      }
      if (lane == 0) s_ok[wib] = ok;
    }
    __syncthreads();
    // chunks of 32 units, of 16 where whole ones would leave warps idle
    const int nw = blockDim.x >> 5, cs = r * ((units + 31) / 32) < nw ? 16 : 32, nch = (units + cs - 1) / cs;
#pragma unroll 1
    for (int ch = wib; ch < r * nch; ch += nw) {
      const int q = ch / nch, u = (ch - q * nch) * cs + lane, cq = blockIdx.x * r + q;
      if (!s_ok[q] || lane >= cs || u >= units) continue;
      const WarpMem wm = warp_mem(Lo, S, sC + Lo.head + q * Lo.smem_warp);
      df* Td = reinterpret_cast<df*>(wm.T);
      double* ro = ratio ? ratio + (size_t)cq * P : nullptr;
      if (PR == LRDMC_PRECISION_DF64) moves64<NJ, NC>(S, L, wm, lt, u, Td, ro, nullptr);
      else candidate_m<NJ>(S, L, wm, u, Td, ro);
    }
    __syncthreads();
    if (ok) {
      const WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
      const df* Td = reinterpret_cast<const df*>(wm.T);
      const double b = PR == LRDMC_PRECISION_DF64
                           ? df_to_double(rate_scan64(Td, P, lane, wm.pfx))
                           : (double)warp_scan_m(Td, P, lane, 0.0f, nullptr, nullptr);
      if (T)
        for (int j = lane; j < P; j += 32) T[(size_t)c * P + j] = df_to_double(Td[j]);
      if (lane == 0) {
        if (b_out) b_out[c] = b;
        if (el_out) el_out[c] = el;
      }
    }
  }
}

// Stateless evaluation of given configurations.
template <int PREC>
__global__ void __launch_bounds__(kMaxEvalWarps * 32, 2)
k_evaluate(const __grid_constant__ SysDev S, const Layout Lo, const LatDev L, int n, int r,
           const double* x, const double* rot, double* ratio, double* T, double* b_out,
           double* el_out, int* err)
{
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  stage_coefficients<(PREC & 3) != LRDMC_PRECISION_FP64>(S, sC);
  evaluate_block<PREC>(S, Lo, L, sC, n, r, x, rot, ratio, T, b_out, el_out, [&] { atomicOr(err, kErrSingular); });
}

// ----------------------------------------------------------------------------
// Host launchers.
// ----------------------------------------------------------------------------
#if LRDMC_PART == 0
static df split_ld(long double x)
{
  float h = (float)x;
  float l = (float)(x - (long double)h);
  return df_make(h, l);
}

void fill_df_constants(SysDev& S)
{
  DfSys& D = S.D;
  for (int I = 0; I < S.n_nuc; ++I) {
    for (int k = 0; k < 3; ++k) D.nuc[I][k] = split_ld(S.nuc[I][k]);
    D.Z[I] = split_ld(S.Z[I]);
    D.en_b1[I] = split_ld(S.en_b1[I]);
  }
  D.b_ee = split_ld(S.b_ee);
  D.c_par = split_ld(S.c_par);
  D.c_anti = split_ld(S.c_anti);
  D.en_b2 = split_ld(S.en_b2);
  for (int q = 0; q < S.n_shell; ++q) {
    D.sh[q].m = split_ld(S.sh[q].m);
    D.sh[q].zeta = split_ld(S.sh[q].zeta);
    for (int p = 0; p < kMaxPrim; ++p) {
      D.sh[q].alpha[p] = split_ld(S.sh[q].alpha[p]);
      D.sh[q].coef[p] = split_ld(S.sh[q].coef[p]);
    }
  }
  // e-e part: the reciprocal form needs b away from zero (its terms c/b q
  // would lose log2(c/b) bits) and positive (1 + b r > 0), and b^2 r^2 and the
  // FP64 mode's products of up to 31 (1 + b r) within range; the general form
  // takes lengths as they are
  S.ee_recip = S.b_ee >= 0.25 && S.b_ee <= 0x1p20 ? 1 : 0;
  const double bs = S.ee_recip ? S.b_ee : 1.0;
  D.ee_scale = split_ld(bs);
  D.ee_scale2 = split_ld((long double)bs * bs);
  D.ee_iscale = split_ld(1.0L / bs);
  D.ee_factor = split_ld(S.ee_recip ? -1.0L / bs : 1.0L);
  // from long double arithmetic
  const long double ln2 = logl(2.0L);
  const df c = split_ld(ln2 / kExpEntries);
  D.lexp.c_hi = c.hi;
  D.lexp.c_lo = c.lo;
  D.lexp.inv = (float)(kExpEntries / ln2);
  long double f = 1.0L;
  for (int k = 0; k < 18; ++k) {
    if (k > 0) f *= (long double)k;
    D.inv_fact[k] = split_ld(1.0L / f);
  }
  D.half_pi = split_ld(2.0L * atanl(1.0L));
}

// The radial table pays from three primitives on (about 75 instructions per
// pair of distances against 55 per primitive); a shell whose exponents span so
// much that it would take over kMaxCells cells (0.8 MB) is summed directly.
constexpr int kMaxCells = 16384;
static uint32_t cell_key(float y)
{
  uint32_t u;
  memcpy(&u, &y, 4);
  return u >> 15;
}

void plan_radial_table(SysDev& S)
{
  S.gt_total = 0;
  for (int q = 0; q < S.n_shell; ++q) {
    ShellDev& sh = S.sh[q];
    sh.gt_cells = 0;
    if (sh.kind != 1 || sh.n_prim < 3) continue;
    double lo = sh.alpha[0], hi = sh.alpha[0];
    bool fine = true;
    for (int p = 0; p < sh.n_prim; ++p) {
      lo = std::min(lo, sh.alpha[p]);
      hi = std::max(hi, sh.alpha[p]);
      fine = fine && std::isfinite(sh.alpha[p]) && std::isfinite(sh.coef[p]);
    }
    if (!fine || !(lo > 1e-6) || !(hi < 1e12)) continue;
    sh.gt_beta = (float)exp2(floor(-log2(hi)));
    sh.gt_key0 = (int)cell_key(sh.gt_beta);
    const int n = (int)cell_key((float)(87.0 / lo + sh.gt_beta)) - sh.gt_key0 + 1;
    if (n > kMaxCells) continue;
    sh.gt_base = S.gt_total;
    sh.gt_cells = n;
    S.gt_total += n;
  }
}

// One cell per thread: the Taylor coefficients of sum_p c_p e^(-alpha_p x) at
// the cell's centre to degree 9 in u, the last two economised onto the lower
// ones by Chebyshev polynomials (the remainder is 2^-15 of the degree-8 term).
__global__ void __launch_bounds__(128) k_radial_table(const __grid_constant__ SysDev S, float4* tab)
{
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= S.gt_total) return;
  int q = 0;
  while (S.sh[q].gt_cells == 0 || id < S.sh[q].gt_base || id >= S.sh[q].gt_base + S.sh[q].gt_cells) ++q;
  const ShellDev& sh = S.sh[q];
  const unsigned key = (unsigned)(sh.gt_key0 + id - sh.gt_base);
  const double y0 = __uint_as_float(key << 15), w = (double)__uint_as_float((key + 1) << 15) - y0;
  const double x = y0 + 0.5 * w - (double)sh.gt_beta;
  double c[10];
  for (int j = 0; j < 10; ++j) c[j] = 0.0;
  for (int p = 0; p < sh.n_prim; ++p) {
    const double al = sh.alpha[p], z = al * x, r = fma(al, x, -z);
    double t = sh.coef[p] * exp(-z);
    t -= t * r;
    for (int j = 0; j < 10; ++j) {
      c[j] += t;
      t *= -al * w / (j + 1);
    }
  }
  c[7] += 0.5625 * c[9];
  c[5] -= 0.10546875 * c[9];
  c[3] += 0.00732421875 * c[9];
  c[1] -= 0.0001373291015625 * c[9];
  c[6] += 0.5 * c[8];
  c[4] -= 0.078125 * c[8];
  c[2] += 0.00390625 * c[8];
  c[0] -= 0.000030517578125 * c[8];
  df d[4];
  for (int j = 0; j < 4; ++j) d[j] = df_from_double(c[j]);
  tab[3 * (size_t)id] = make_float4(d[0].hi, d[0].lo, d[1].hi, d[1].lo);
  tab[3 * (size_t)id + 1] = make_float4(d[2].hi, d[2].lo, d[3].hi, d[3].lo);
  tab[3 * (size_t)id + 2] = make_float4((float)c[4], (float)c[5], (float)c[6], (float)c[7]);
}

cudaError_t launch_radial_table(const SysDev& S, float4* tab, cudaStream_t st)
{
  k_radial_table<<<(S.gt_total + 127) / 128, 128, 0, st>>>(S, tab);
  return cudaGetLastError();
}

void fill_lattice_df(LatDev& L)
{
  L.a_df = split_ld(L.a);
  L.ap_df = split_ld(L.ap);
  L.inv2a2_df = split_ld(L.inv2a2);
  L.inv2ap2_df = split_ld(L.inv2ap2);
  L.p_coef_df = split_ld(L.p_coef);
}

static_assert(sizeof(SysDev) + sizeof(Layout) + sizeof(LatDev) + sizeof(PopDev) + 64 < 32764,
              "kernel parameters exceed the 32 KB limit");

Layout make_layout(const SysDev& S, bool caches)
{
  Layout Lo;
  Lo.N = S.N;
  Lo.nu = S.n_up;
  Lo.nd = S.n_dn;
  Lo.P_max = 12 * S.N;
  Lo.off_x = 0;
  Lo.off_au = 3 * S.N;
  Lo.off_ad = Lo.off_au + S.n_up * S.n_up;
  Lo.off_R = Lo.off_ad + S.n_dn * S.n_dn;
  Lo.off_T = Lo.off_R + 9;
  Lo.off_b = Lo.off_T + Lo.P_max;
  Lo.off_el = Lo.off_b + 1;
  Lo.rec = (Lo.off_el + 1 + 3) & ~3;
  const int n = S.n_up;
  Lo.n_draw = kDrawAhead * kDrawWords;
  Lo.n_scr = n * n + S.N * S.n_ao + n + (n + 1) / 2;         // inverses: basis values, matrix, pivot column, order
  Lo.n_scr = std::max(Lo.n_scr, S.n_ao + 3 * n + n * n);     // Sherman-Morrison (FP64 or FP32 mode)
  // The caches of the double-float evaluation (omitted when caches is false):
  // the electron-nucleus cache (7 df per electron and nucleus), and one
  // squared distance per electron pair; up to 40 electrons. Beyond, what they
  // save and the warps per SM that they cost about cancel: per walker and
  // jump, 2048 walkers, without and with them, 42 electrons on 4 centres 0.43
  // and 0.49 us, 48 on 8 centres 0.67 and 0.64, 54 on one 0.43 and 0.43; the
  // mixed mode, which shares the layout and reads no cache, 0.47 and 0.59, 0.75
  // and 0.74, 0.50 and 0.59.
  Lo.n_pc = (caches && S.N <= 40) ? S.N * (S.N - 1) / 2 : 0;
  Lo.enc = caches && S.N <= 40 ? 1 : 0;
  const int state = S.N * S.n_ao + 2 * S.N + 6 * S.N + 12 + 32 + (Lo.enc ? kEncWords * S.N * S.n_nuc : 0) + Lo.n_pc;
  Lo.smem_warp = 3 * S.N + S.n_up * S.n_up + S.n_dn * S.n_dn + 12 + Lo.P_max + Lo.n_draw + 4 + S.n_ao + 3 * n +
                 std::max(Lo.n_scr, state);
  Lo.smem_warp = (Lo.smem_warp + 1) & ~1;
  Lo.head = lean_offset(S) + kExpEntries + 2 * S.n_prim + (int)(sizeof(LShell) / sizeof(double)) * S.n_shell;
  Lo.smem_block_bytes = (int)sizeof(double) * (Lo.head + kWarpsPerBlock * Lo.smem_warp);
  return Lo;
}

int accept_smem_bytes(const SysDev& S, bool caches)
{
  const int n = S.n_up;
  const int scr = std::max(2 * n * n + n * S.n_ao, S.n_ao + 3 * n + n * n);
  int warp = 3 * S.N + S.n_up * S.n_up + S.n_dn * S.n_dn + 12 + 12 * S.N + S.N * S.n_ao + S.N + (3 * S.N + 12) + scr;
  if (caches) warp += (S.N <= 24 ? S.N * (S.N - 1) / 2 * (S.N <= 12 ? 8 : 4) : 0) + 8 * S.N * S.n_nuc;
  warp = (warp + 1) & ~1;
  // the head stands for coefficients in three arithmetics and a 64-entry table
  const int nc = S.n_ao * S.n_mo, head = (2 * nc + (nc + 1) / 2 + 64 + 1) & ~1;
  return (int)sizeof(double) * (head + kWarpsPerBlock * warp);
}
#endif  // LRDMC_PART == 0

// Without the attribute a block's dynamic and static shared memory together
// are limited to 48 KB (the interval kernel's static part is below 2 KB).
static cudaError_t set_smem(const void* fn, int bytes)
{
  if (bytes > 44 * 1024) return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return cudaSuccess;
}

#if LRDMC_PART == 0
cudaError_t launch_init(const SysDev& S, const Layout& Lo, const PopDev& P, const double* x0,
                        cudaStream_t st)
{
  cudaError_t e = set_smem((const void*)k_init, Lo.smem_block_bytes);
  if (e != cudaSuccess) return e;
  int blocks = (P.W + kWarpsPerBlock - 1) / kWarpsPerBlock;
  k_init<<<blocks, kWarpsPerBlock * 32, Lo.smem_block_bytes, st>>>(S, Lo, P, x0);
  return cudaGetLastError();
}

#endif  // LRDMC_PART == 0

// Kernel variant of a system: the arithmetic in bits 0-1 of the template
// argument, bit 2 for a double-float system whose layout has no evaluation
// caches, the neural pair term in bit 3 (kernels without a feature carry
// none of its code).
constexpr int kNoCacheBit = 4;
constexpr int kNjBit = 8;

#define LRDMC_DISPATCH_NJ(S, BASE, ...)                                            \
  do {                                                                             \
    if ((S).nj_on != 0) { constexpr int V = (BASE) | kNjBit; __VA_ARGS__; }        \
    else { constexpr int V = (BASE); __VA_ARGS__; }                                \
  } while (0)

#define LRDMC_DISPATCH(S, Lo, ...)                                                 \
  do {                                                                             \
    if ((S).precision == LRDMC_PRECISION_DF64) {                                   \
      if ((Lo).enc) LRDMC_DISPATCH_NJ(S, LRDMC_PRECISION_DF64, __VA_ARGS__);       \
      else LRDMC_DISPATCH_NJ(S, LRDMC_PRECISION_DF64 | kNoCacheBit, __VA_ARGS__);  \
    } else if ((S).precision == LRDMC_PRECISION_FP32) {                            \
      LRDMC_DISPATCH_NJ(S, LRDMC_PRECISION_FP32, __VA_ARGS__);                     \
    } else {                                                                       \
      LRDMC_DISPATCH_NJ(S, LRDMC_PRECISION_FP64, __VA_ARGS__);                     \
    }                                                                              \
  } while (0)

template <int PREC>
cudaError_t launch_eval_all_t(const SysDev& S, const Layout& Lo, const LatDev& L, const PopDev& P,
                                     cudaStream_t st)
{
  cudaError_t e = set_smem((const void*)k_eval_all<PREC>, Lo.smem_block_bytes);
  if (e != cudaSuccess) return e;
  int blocks = (P.W + kWarpsPerBlock - 1) / kWarpsPerBlock;
  k_eval_all<PREC><<<blocks, kWarpsPerBlock * 32, Lo.smem_block_bytes, st>>>(S, Lo, L, P);
  return cudaGetLastError();
}

static int sm_count_current()
{
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                cudaSuccess)
    return 152;
  return n;
}

static int interval_smem(const Layout& Lo, int w) { return (int)sizeof(double) * (Lo.head + w * Lo.smem_warp); }

// Persistent grid of the interval kernel: as many blocks as fit on the GPU
// at once (occupancy for this system's shared memory), at most one warp per
// walker.
template <int PREC>
cudaError_t interval_occupancy(const Layout& Lo, int w, int* blocks)
{
  int per_sm = 0;
  cudaError_t e = set_smem((const void*)k_interval<PREC>, interval_smem(Lo, w));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_interval<PREC>, w * 32, interval_smem(Lo, w));
  *blocks = (per_sm < 1 ? 1 : per_sm) * sm_count_current();
  return e;
}

template <int PREC>
cudaError_t launch_interval_t(const SysDev& S, const Layout& Lo, const LatDev& L, const PopDev& P,
                                     int blocks, int carveout, bool pdl, cudaStream_t st)
{
  static int cached_blocks = -1, cached_smem = -1;
  const int w = interval_warps(Lo, P.W);
  const int smem = interval_smem(Lo, w);
  cudaError_t e = set_smem((const void*)k_interval<PREC>, smem);
  if (e != cudaSuccess) return e;
  if (blocks <= 0) {
    if (cached_smem != smem) {
      e = interval_occupancy<PREC>(Lo, w, &cached_blocks);
      if (e != cudaSuccess) return e;
      cached_smem = smem;
    }
    blocks = cached_blocks;
  }
  const int need = (P.W + w - 1) / w;
  if (blocks > need) blocks = need;
  if (carveout < 0 && !pdl) {
    k_interval<PREC><<<blocks, w * 32, smem, st>>>(S, Lo, L, P);
    return cudaGetLastError();
  }
  // the same launch with launch attributes: a preferred shared-memory
  // carveout for this launch only (kernels of different systems sharing the
  // SMs then ask for the same L1/shared split), and programmatic stream
  // serialization (this kernel may start once every block of the previous
  // kernel in the stream has run out of walkers)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(w * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (carveout >= 0) {
    attr[na].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[na].val.sharedMemCarveout = (unsigned)carveout;
    ++na;
  }
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, k_interval<PREC>, S, Lo, L, P);
}

// Configurations r and warps of an evaluation block. Four and four where three
// such blocks fit an SM. A larger system gets as many as let two blocks of
// eight warps share an SM (one's inverses and local energies run beside the
// other's moves). Fewer configurations than fill the SMs are spread over
// them.
struct EvalShape {
  int r, warps;
};

template <int PREC>
static EvalShape eval_shape(const Layout& Lo, int n)
{
  EvalShape e = {kWarpsPerBlock, kWarpsPerBlock};
  if ((PREC & 3) == LRDMC_PRECISION_FP64) return e;
  const int sm = 228 * 1024, reserved = 1024 + 64;  // of an SM; the runtime's and the static part of a block
  if (3 * (Lo.smem_block_bytes + reserved) > sm) {
    e.warps = kMaxEvalWarps;
    int r = std::min(kMaxEvalConfigs, (int)((sm / 2 - reserved) / sizeof(double) - Lo.head) / Lo.smem_warp);
    if (r >= 2) e.r = r;
  }
  const int per_sm = std::max(1, (n + sm_count_current() - 1) / sm_count_current());
  if (per_sm < e.r) e = {per_sm, kMaxEvalWarps};
  return e;
}

template <int PREC>
cudaError_t launch_evaluate_t(const SysDev& S, const Layout& Lo, const LatDev& L, int n, const double* x,
                                     const double* rot, double* ratio, double* T, double* b, double* el, int* err,
                                     cudaStream_t st)
{
  const EvalShape sh = eval_shape<PREC>(Lo, n);
  const int blocks = (n + sh.r - 1) / sh.r, smem = interval_smem(Lo, sh.r);
  // the largest size always: calls of other sizes may run in other threads
  cudaError_t e = set_smem((const void*)k_evaluate<PREC>, kMaxSmemBlock);
  if (e != cudaSuccess) return e;
  k_evaluate<PREC><<<blocks, sh.warps * 32, smem, st>>>(S, Lo, L, n, sh.r, x, rot, ratio, T, b, el, err);
  return cudaGetLastError();
}

template <int PREC>
__global__ void __launch_bounds__(kMaxEvalWarps * 32, 2)
k_evaluate_static(const __grid_constant__ SysDev S, const Layout Lo, const LatDev L, int n, int r,
                  const double* x, const double* rot, double* ratio, double* T, double* b_out,
                  double* el_out, int* scratch)
{
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  stage_coefficients<(PREC & 3) != LRDMC_PRECISION_FP64>(S, sC);
  // word 64 + c: status of configuration c; word 0: OR of all statuses
  evaluate_block<PREC>(S, Lo, L, sC, n, r, x, rot, ratio, T, b_out, el_out, [&] {
    scratch[64 + blockIdx.x * r + (threadIdx.x >> 5)] = kErrSingular;
    atomicOr(&scratch[0], kErrSingular);
  });
}

template <int PREC>
cudaError_t launch_evaluate_static_t(const SysDev& S, const Layout& Lo, const LatDev& L, int n, const double* x,
                                     const double* rot, double* ratio, double* T, double* b, double* el,
                                     int* scratch, cudaStream_t st)
{
  const EvalShape sh = eval_shape<PREC>(Lo, n);
  const int blocks = (n + sh.r - 1) / sh.r, smem = interval_smem(Lo, sh.r);
  // the largest size always: calls of other sizes may run in other threads
  cudaError_t e = set_smem((const void*)k_evaluate_static<PREC>, kMaxSmemBlock);
  if (e != cudaSuccess) return e;
  if (blocks > 0)
    k_evaluate_static<PREC><<<blocks, sh.warps * 32, smem, st>>>(S, Lo, L, n, sh.r, x, rot, ratio, T, b, el, scratch);
  return cudaGetLastError();
}

// The variants and the part that compiles each.
#define LRDMC_VARIANT(KEYWORD, V)                                                                                  \
  KEYWORD template cudaError_t launch_eval_all_t<V>(const SysDev&, const Layout&, const LatDev&, const PopDev&,    \
                                                    cudaStream_t);                                                 \
  KEYWORD template cudaError_t interval_occupancy<V>(const Layout&, int, int*);                                    \
  KEYWORD template cudaError_t launch_interval_t<V>(const SysDev&, const Layout&, const LatDev&, const PopDev&,    \
                                                    int, int, bool, cudaStream_t);                                 \
  KEYWORD template cudaError_t launch_evaluate_t<V>(const SysDev&, const Layout&, const LatDev&, int,              \
                                                    const double*, const double*, double*, double*, double*,       \
                                                    double*, int*, cudaStream_t);                                  \
  KEYWORD template cudaError_t launch_evaluate_static_t<V>(const SysDev&, const Layout&, const LatDev&, int,       \
                                                           const double*, const double*, double*, double*,         \
                                                           double*, double*, int*, cudaStream_t);
#if LRDMC_PART == 0
LRDMC_VARIANT(extern, LRDMC_PRECISION_DF64)
LRDMC_VARIANT(extern, LRDMC_PRECISION_DF64 | kNjBit)
LRDMC_VARIANT(extern, LRDMC_PRECISION_DF64 | kNoCacheBit)
LRDMC_VARIANT(extern, LRDMC_PRECISION_DF64 | kNoCacheBit | kNjBit)
LRDMC_VARIANT(extern, LRDMC_PRECISION_FP32)
LRDMC_VARIANT(extern, LRDMC_PRECISION_FP32 | kNjBit)
LRDMC_VARIANT(extern, LRDMC_PRECISION_FP64)
LRDMC_VARIANT(extern, LRDMC_PRECISION_FP64 | kNjBit)
#elif LRDMC_PART == 1
LRDMC_VARIANT(, LRDMC_PRECISION_DF64)
#elif LRDMC_PART == 2
LRDMC_VARIANT(, LRDMC_PRECISION_DF64 | kNjBit)
#elif LRDMC_PART == 3
LRDMC_VARIANT(, LRDMC_PRECISION_DF64 | kNoCacheBit)
#elif LRDMC_PART == 4
LRDMC_VARIANT(, LRDMC_PRECISION_DF64 | kNoCacheBit | kNjBit)
#elif LRDMC_PART == 5
LRDMC_VARIANT(, LRDMC_PRECISION_FP32)
LRDMC_VARIANT(, LRDMC_PRECISION_FP32 | kNjBit)
#elif LRDMC_PART == 6
LRDMC_VARIANT(, LRDMC_PRECISION_FP64)
LRDMC_VARIANT(, LRDMC_PRECISION_FP64 | kNjBit)
#endif

#if LRDMC_PART == 0
cudaError_t launch_eval_all(const SysDev& S, const Layout& Lo, const LatDev& L, const PopDev& P,
                            cudaStream_t st)
{
  LRDMC_DISPATCH(S, Lo, return launch_eval_all_t<V>(S, Lo, L, P, st));
  return cudaErrorInvalidValue;
}

// Warps per block of the interval kernel: enough that one block per SM holds
// the population (so that the warps of an SM can help one another at the end
// of an interval), at least the other kernels' four, at most 16 and what the
// shared memory holds.
int interval_warps(const Layout& Lo, int W)
{
  const int sms = sm_count_current();
  int w = std::min(kMaxIntervalWarps, std::max(kWarpsPerBlock, (W + sms - 1) / sms));
  while (w > kWarpsPerBlock && (int)sizeof(double) * (Lo.head + w * Lo.smem_warp) > kMaxSmemBlock) --w;
  return w;
}

int interval_default_blocks(const SysDev& S, const Layout& Lo, int W)
{
  int b = 0;
  const int w = interval_warps(Lo, W);
  LRDMC_DISPATCH(S, Lo, interval_occupancy<V>(Lo, w, &b));
  return b;
}

cudaError_t launch_interval(const SysDev& S, const Layout& Lo, const LatDev& L, const PopDev& P, int blocks,
                            cudaStream_t st, int carveout, bool pdl)
{
  LRDMC_DISPATCH(S, Lo, return launch_interval_t<V>(S, Lo, L, P, blocks, carveout, pdl, st));
  return cudaErrorInvalidValue;
}

int comb_blocks(int W)
{
  // at least 256 slots per block (short sequential sums over the blocks),
  // at most kMaxCombBlocks blocks
  const int R = std::max(kCombThreads, (W + kMaxCombBlocks - 1) / kMaxCombBlocks);
  return std::max(1, (W + R - 1) / R);
}

cudaError_t launch_reconfig(const PopDev& P, const Layout& Lo, cudaStream_t st)
{
  const int G = comb_blocks(P.W);
  const int R = (P.W + G - 1) / G;
  // the running sums (up to kReconfigSmemW walkers), then a float per slot
  // of the block
  const int smem = (P.W <= kReconfigSmemW ? (int)sizeof(double) * P.W : 0) + (int)sizeof(float) * R;
  // the attribute always takes the largest size, so systems of different
  // populations (and batches captured in one graph) never lower it
  cudaError_t e = set_smem((const void*)k_comb_parents, kCombSmemMax);
  if (e != cudaSuccess) return e;
  if (smem > kCombSmemMax) return cudaErrorInvalidValue;
  k_comb_sums<<<G, kCombThreads, 0, st>>>(P);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kCombThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_comb_parents, P, (const double*)P.rec_dst, Lo.rec, Lo.off_b);
}

// Base terms of the neural objective: grad_i log|psi_G| and E_L of every
// configuration in IEEE double, one warp per configuration (the caller
// passes the system with the neural term switched off).
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_base_terms(const __grid_constant__ SysDev S, const Layout Lo, int n, const double* x, double* grad,
             double* e, int* err)
{
  extern __shared__ __align__(16) double smem[];
  double* sC = smem;
  stage_coefficients(S, sC);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int s = blockIdx.x * kWarpsPerBlock + wib;
  if (s >= n) return;
  WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
  for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = x[(size_t)s * 3 * Lo.N + j];
  __syncwarp();
  bool ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane);
  if (!ok) {
    if (lane == 0) atomicOr(err, kErrSingular);
    for (int j = lane; j < 3 * Lo.N; j += 32) grad[(size_t)s * 3 * Lo.N + j] = NAN;
    if (lane == 0) e[s] = NAN;
    return;
  }
  LatDev L{};
  L.G = 1;
  double b, el;
  warp_eval<false>(S, sC, L, wm, lane, nullptr, b, el, grad + (size_t)s * 3 * Lo.N, false);
  if (lane == 0) e[s] = el;
}

cudaError_t launch_base_terms(const SysDev& S, const Layout& Lo, int n, const double* x, double* grad,
                              double* e_out, int* err, cudaStream_t st)
{
  if (n <= 0) return cudaSuccess;
  cudaError_t e = set_smem((const void*)k_base_terms, Lo.smem_block_bytes);
  if (e != cudaSuccess) return e;
  const int blocks = (n + kWarpsPerBlock - 1) / kWarpsPerBlock;
  k_base_terms<<<blocks, kWarpsPerBlock * 32, Lo.smem_block_bytes, st>>>(S, Lo, n, x, grad, e_out, err);
  return cudaGetLastError();
}

cudaError_t launch_evaluate(const SysDev& S, const Layout& Lo, const LatDev& L, int n,
                            const double* x, const double* rot, double* ratio, double* T,
                            double* b, double* el, int* err, cudaStream_t st)
{
  LRDMC_DISPATCH(S, Lo, return launch_evaluate_t<V>(S, Lo, L, n, x, rot, ratio, T, b, el, err, st));
  return cudaErrorInvalidValue;
}

// ----------------------------------------------------------------------------
// Tensor-core form of the orbital contraction (tcgen05, FP32 mode).
//
// The literal contraction of the displaced positions' basis values with the
// MO coefficients, phi_m(r'_c) = sum_mu chi_mu(r'_c) C[mu][m], as a GEMM on
// the fifth-generation tensor cores: one CTA of four warps evaluates four
// configurations in lock step; per round every lane computes the basis
// values of one lattice move (FP32) and writes them, split into bfloat16
// high and low parts, as one row of a 128-row A tile in shared memory;
// thread 0 issues D = A_hi B_hi + A_hi B_lo + A_lo B_hi (B = C^T split the
// same way; three bf16 products carry about 16 significant bits) into a
// 128 x 32 FP32 accumulator in tensor memory; each warp reads its 32 rows
// back (tcgen05.ld) and finishes its moves: the determinant ratio
// sum_m phi_m Ainv[m][l_i] (FP32), the Jastrow ratio and the rate, as the
// FP32 mode's projected form does. Shared-memory operands use the
// canonical K-major layout without swizzle: 8 x 16-byte core matrices,
// adjacent in K at LBO = 128 bytes, 8-row groups at SBO = 16 Kp bytes.
// Every wait on the MMA's mbarrier is bounded; a wait that runs out sets
// kErrTimeout, waits once more (bounded) and frees the tensor memory.
// ----------------------------------------------------------------------------
constexpr int kTcRows = 128;    // A tile rows: 4 warps x 32 moves
constexpr int kTcN = 32;        // accumulator columns (orbitals, padded)
constexpr int kTcCols = 32;     // tensor-memory columns allocated
constexpr int kTcSpin = 1 << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t tc_desc(const void* base, uint32_t lbo, uint32_t sbo)
{
  uint64_t d = (uint64_t)((smem_u32(base) & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of sm_100-class tensor cores; no swizzle, base offset 0
  return d;
}

// kind::f16 instruction descriptor: D F32, A and B BF16, both K-major, N, M.
__host__ __device__ constexpr uint32_t tc_idesc_bf16(int M, int N)
{
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, int accumulate)
{
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* mbar)
{
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               :: "r"(smem_u32(mbar)) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, int count)
{
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(mbar)), "r"(count) : "memory");
}

// Non-blocking test of the phase with the given parity.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* mbar, uint32_t parity)
{
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(smem_u32(mbar)), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait for the phase of the MMA barrier (kTcSpin polls, a short
// sleep between them: well under a second); false when it ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* mbar, uint32_t parity)
{
  for (int it = 0; it < kTcSpin; ++it) {
    if (mbar_test_wait(mbar, parity)) return true;
    __nanosleep(20);
  }
  return false;
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float* v)
{
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// x as bfloat16 high part plus the bfloat16 of the remainder (round to
// nearest even both times): x - hi - lo is about 2^-17 |x|.
__device__ __forceinline__ void bf16_split(float x, uint16_t& hi, uint16_t& lo)
{
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
  hi = __bfloat16_as_ushort(h);
  lo = __bfloat16_as_ushort(l);
}

// Byte offset of element (row, k) in a K-major tile without swizzle.
__device__ __forceinline__ uint32_t tc_off(int row, int k, int Kp)
{
  return (uint32_t)((row >> 3) * (Kp * 16) + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Writes one row of the A tiles, value by value in K order.
struct TcRowWriter {
  char* hi;
  char* lo;
  int row, Kp, k;
  __device__ __forceinline__ void put(float v)
  {
    uint16_t h, l;
    bf16_split(v, h, l);
    const uint32_t o = tc_off(row, k, Kp);
    *reinterpret_cast<uint16_t*>(hi + o) = h;
    *reinterpret_cast<uint16_t*>(lo + o) = l;
    ++k;
  }
  // zeros up to Kp (the padding of K, or a whole inactive row)
  __device__ __forceinline__ void finish()
  {
    while (k < Kp) put(0.0f);
  }
};

// Basis values chi_mu(p) of every AO (FP32, in AO order) into the row
// writer, and the electron-nucleus Jastrow terms into jen.
template <bool NJ>
__device__ __forceinline__ void tc_basis_row(const SysDev& S, const float p[3], TcRowWriter& w, float& jen)
{
  jen = 0.0f;
  for (int I = 0; I < S.n_nuc; ++I) {
    const float d[3] = {p[0] - S.D.nuc[I][0].hi, p[1] - S.D.nuc[I][1].hi, p[2] - S.D.nuc[I][2].hi};
    const float r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const float r = sqrtf(r2);
    if (S.en_b1[I] != 0.0) jen -= S.D.en_b1[I].hi * r / (S.D.en_b2.hi * r + 1.0f);
    if (NJ) jen += nj_value_m(S, 2 + S.nj_species[I], r);
    float e = 0.0f;
    for (int q = S.nuc_shell_begin[I]; q < S.nuc_shell_begin[I + 1]; ++q) {
      const ShellDev& sh = S.sh[q];
      const DfShell& dsh = S.D.sh[q];
      if (sh.kind == 0 && !sh.same_exp) e = expf(-dsh.zeta.hi * r);
      const float Rv = radial_value_m(sh, dsh, r, r2, e);
      float Sv[5];
      const int nf = solid_m(sh.l, d, Sv);
      w.k = sh.ao_offset;
      for (int f = 0; f < nf; ++f) w.put(Sv[f] * Rv);
    }
  }
}

template <int PREC>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
k_evaluate_tc(const __grid_constant__ SysDev S, const Layout Lo, const LatDev L, int n, const double* x,
              const double* rot, double* ratio, double* T, double* b_out, double* el_out, int* err, int Kp,
              int tile_off)
{
  constexpr bool NJ = (PREC & 8) != 0;
  extern __shared__ __align__(16) double smem[];
  __shared__ __align__(8) uint64_t s_mbar;
  __shared__ uint32_t s_tmem;
  __shared__ int s_bad;
  double* sC = smem;
  const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  char* tiles = reinterpret_cast<char*>(smem) + tile_off;
  const int tileA = kTcRows * Kp * 2, tileB = kTcN * Kp * 2;
  char* Ah = tiles;
  char* Al = Ah + tileA;
  char* Bh = Al + tileA;
  char* Bl = Bh + tileB;
  stage_coefficients<true>(S, sC);
  // B = C^T (orbital m, AO k), split into bfloat16 high and low parts
  for (int idx = tid; idx < kTcN * Kp; idx += blockDim.x) {
    const int m = idx / Kp, k = idx - m * Kp;
    const float v = (m < S.n_mo && k < S.n_ao) ? (float)S.C[k * S.n_mo + m] : 0.0f;
    uint16_t h, l;
    bf16_split(v, h, l);
    const uint32_t o = tc_off(m, k, Kp);
    *reinterpret_cast<uint16_t*>(Bh + o) = h;
    *reinterpret_cast<uint16_t*>(Bl + o) = l;
  }
  if (wib == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&s_tmem)), "r"(kTcCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&s_mbar, 1);
    s_bad = 0;
  }
  fence_async_shared();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  // this warp's configuration: inverses, then the local energy and the
  // Jastrow sums of the FP32 evaluation
  const int c = blockIdx.x * kWarpsPerBlock + wib;
  WarpMem wm = warp_mem(Lo, S, sC + Lo.head + wib * Lo.smem_warp);
  bool ok = c < n;
  double b = 0.0, el = 0.0;
  df bdf;
  if (ok) {
    for (int j = lane; j < 3 * Lo.N; j += 32) wm.x[j] = x[(size_t)c * 3 * Lo.N + j];
    for (int j = lane; j < 9; j += 32) wm.R[j] = rot[(size_t)c * 9 + j];
    __syncwarp();
    ok = warp_inverses(S, sC, wm.x, wm.A, wm.scr, lane);
    if (!ok && lane == 0) atomicOr(err, kErrSingular);
    if (ok) el = prelude32<NJ>(S, sC, wm, lean_mem(S, sC), lane, -1);
  }
  const int N = S.N, G = L.G, per_e = 6 * G, P = N * per_e;
  const int rounds = (P + 31) / 32;
  df* Td = reinterpret_cast<df*>(wm.T);
  const uint32_t idesc = tc_idesc_bf16(kTcRows, kTcN);
  uint32_t phase = 0;
  for (int rd = 0; rd < rounds; ++rd) {
    const int cand = rd * 32 + lane;
    const bool act = ok && cand < P;
    TcRowWriter w;
    w.hi = Ah;
    w.lo = Al;
    w.row = wib * 32 + lane;
    w.Kp = Kp;
    w.k = 0;
    float jsum = 0.0f, pm = 1.0f;
    int i = 0, g = 0;
    if (act) {
      i = cand / per_e;
      const int rem = cand - i * per_e, k = (rem % 6) >> 1;
      g = rem / 6;
      float h = g ? L.ap_df.hi : L.a_df.hi;
      if (cand & 1) h = -h;
      const float e0 = wm.Rd[k].hi, e1 = wm.Rd[3 + k].hi, e2 = wm.Rd[6 + k].hi;
      const float ri[3] = {wm.xd[3 * i].hi, wm.xd[3 * i + 1].hi, wm.xd[3 * i + 2].hi};
      const float p[3] = {ri[0] + h * e0, ri[1] + h * e1, ri[2] + h * e2};
      float jen;
      tc_basis_row<NJ>(S, p, w, jen);
      jsum = jastrow_ee_m<NJ>(S, wm.xd, i, p) + jen;
      if (G == 2) {
        const float hh = 0.5f * h;
        const float mid[3] = {ri[0] + hh * e0, ri[1] + hh * e1, ri[2] + hh * e2};
        pm = p_weight_m(S, L, mid);
      }
    }
    w.finish();
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      for (int kk = 0; kk < Kp / 16; ++kk) {
        const uint32_t off = (uint32_t)kk * 256;
        const uint64_t ah = tc_desc(Ah + off, 128, Kp * 16), al = tc_desc(Al + off, 128, Kp * 16);
        const uint64_t bh = tc_desc(Bh + off, 128, Kp * 16), bl = tc_desc(Bl + off, 128, Kp * 16);
        tc_mma(tmem, ah, bh, idesc, kk > 0);
        tc_mma(tmem, ah, bl, idesc, 1);
        tc_mma(tmem, al, bh, idesc, 1);
      }
      tc_commit(&s_mbar);
    }
    if (!mbar_wait_bounded(&s_mbar, phase)) s_bad = 1;
    phase ^= 1u;
    __syncthreads();
    if (s_bad) break;
    tc_fence_after();
    float phi[32];
    tc_ld32(tmem + ((uint32_t)(wib * 32) << 16), phi);
    if (act) {
      const int nu = S.n_up, spin = i < nu ? 0 : 1, l = i < nu ? i : i - nu, ns = spin ? S.n_dn : nu;
      const double* Am = spin ? wm.A + nu * nu : wm.A;
      float rdet = 0.0f;
#pragma unroll
      for (int m = 0; m < kTcN; ++m)
        if (m < ns) rdet += phi[m] * (float)Am[m * ns + l];
      const float rho = rdet * expf(jsum - wm.Sd[i].hi);
      float wgt = 1.0f;
      if (G == 2) wgt = g ? 1.0f - pm : pm;
      float Tc = 0.0f;
      if (rho > 0.0f) Tc = wgt * (g ? L.inv2ap2_df.hi : L.inv2a2_df.hi) * rho;
      Td[cand] = df_make(Tc, 0.0f);
      if (ratio) ratio[(size_t)c * P + cand] = (double)rho;
    }
    tc_fence_before();
    __syncthreads();  // every lane has read the accumulator and the A tiles are free
  }
  if (s_bad) {
    // the MMA barrier did not complete in time: report, wait once more for
    // the tensor core to finish with this CTA's memory, then free it
    if (tid == 0) {
      atomicOr(err, kErrTimeout);
      mbar_wait_bounded(&s_mbar, phase ^ 1u);
    }
    __syncthreads();
  } else if (ok) {
    __syncwarp();
    const float btot = warp_scan_m(Td, P, lane, 0.0f, nullptr, nullptr);
    b = (double)btot;
    if (T)
      for (int j = lane; j < P; j += 32) T[(size_t)c * P + j] = (double)Td[j].hi;
    if (lane == 0) {
      if (b_out) b_out[c] = b;
      if (el_out) el_out[c] = el;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (wib == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTcCols) : "memory");
  }
}

// Shared memory of the tensor-core evaluation: the evaluation's own layout,
// then (128-byte aligned) the A and B tiles in both parts.
static int tc_tile_offset(const Layout& Lo) { return (Lo.smem_block_bytes + 127) & ~127; }
static int tc_smem_bytes(const Layout& Lo, int Kp) { return tc_tile_offset(Lo) + 2 * (kTcRows + kTcN) * Kp * 2; }

// The same beside the acceptance layout (its caches where they fit): what
// decides whether a system can use the tensor-core evaluation.
int evaluate_tc_smem_bytes(const SysDev& S, const Layout& Lo)
{
  const int Kp = (S.n_ao + 15) & ~15;
  Layout La = Lo;
  La.smem_block_bytes = accept_smem_bytes(S, true);
  if (La.smem_block_bytes > kMaxSmemBlock) La.smem_block_bytes = accept_smem_bytes(S, false);
  return std::max(tc_smem_bytes(Lo, Kp), tc_smem_bytes(La, Kp));
}

cudaError_t launch_evaluate_tc(const SysDev& S, const Layout& Lo, const LatDev& L, int n, const double* x,
                               const double* rot, double* ratio, double* T, double* b, double* el, int* err,
                               cudaStream_t st)
{
  if (n <= 0) return cudaSuccess;
  const int Kp = (S.n_ao + 15) & ~15;
  const int bytes = tc_smem_bytes(Lo, Kp);
  const int blocks = (n + kWarpsPerBlock - 1) / kWarpsPerBlock;
  cudaError_t e;
  if (S.nj_on) {
    e = set_smem((const void*)k_evaluate_tc<LRDMC_PRECISION_FP32 | kNjBit>, bytes);
    if (e != cudaSuccess) return e;
    k_evaluate_tc<LRDMC_PRECISION_FP32 | kNjBit><<<blocks, kWarpsPerBlock * 32, bytes, st>>>(
        S, Lo, L, n, x, rot, ratio, T, b, el, err, Kp, tc_tile_offset(Lo));
  } else {
    e = set_smem((const void*)k_evaluate_tc<LRDMC_PRECISION_FP32>, bytes);
    if (e != cudaSuccess) return e;
    k_evaluate_tc<LRDMC_PRECISION_FP32><<<blocks, kWarpsPerBlock * 32, bytes, st>>>(
        S, Lo, L, n, x, rot, ratio, T, b, el, err, Kp, tc_tile_offset(Lo));
  }
  return cudaGetLastError();
}


// ----------------------------------------------------------------------------
// Evaluation that allocates nothing (lrdmc_evaluate_static).
//
// Some callers cannot allocate device memory at the moment they evaluate:
// code that runs inside another framework's fixed memory budget (a caching
// allocator that has reserved the device), processes that forbid any
// allocation after start-up, or callers that must not synchronise the
// device the way cudaMalloc and cudaFree can. This variant of k_evaluate
// keeps its scratch - a summary status word and one status word per
// configuration - in the file-scope device array below instead of memory
// from cudaMalloc. Every GPU that loads the library holds the array
// (64 + LRDMC_STATIC_EVAL_MAX ints, 1 MiB) until the process exits. All
// calls share it: calls that overlap on the GPU race on it.
// ----------------------------------------------------------------------------
static __device__ __align__(256) int g_eval_scratch[64 + LRDMC_STATIC_EVAL_MAX];

// Device address of g_eval_scratch, looked up once per device with that
// device current (host code must not pass the symbol itself: in host code
// it names a host-side stand-in, not device memory).
static int* g_eval_scratch_ptr[64];
static std::mutex g_eval_scratch_mu;

static cudaError_t eval_scratch_address(int** out)
{
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_eval_scratch_mu);
  if (!g_eval_scratch_ptr[dev]) {
    int* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_eval_scratch);
    if (e != cudaSuccess) return e;
    g_eval_scratch_ptr[dev] = p;
  }
  *out = g_eval_scratch_ptr[dev];
  return cudaSuccess;
}

cudaError_t launch_evaluate_static(const SysDev& S, const Layout& Lo, const LatDev& L, int n,
                                   const double* x, const double* rot, double* ratio, double* T,
                                   double* b, double* el, int* summary, int* first_bad, cudaStream_t st)
{
  if (first_bad) *first_bad = -1;
  if (n < 0 || n > LRDMC_STATIC_EVAL_MAX) return cudaErrorInvalidValue;
  int* scratch = nullptr;
  cudaError_t e = eval_scratch_address(&scratch);
  if (e != cudaSuccess) return e;
  // the summary word and the statuses of this call start at zero
  e = cudaMemsetAsync(scratch, 0, sizeof(int) * (64 + (size_t)n), st);
  if (e != cudaSuccess) return e;
  LRDMC_DISPATCH(S, Lo, e = launch_evaluate_static_t<V>(S, Lo, L, n, x, rot, ratio, T, b, el, scratch, st));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(summary, scratch, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess || *summary == 0 || !first_bad) return e;
  // a configuration failed: find the first one from the per-configuration
  // words, in chunks through a fixed host buffer (no allocation)
  int chunk[1024];
  for (int c0 = 0; c0 < n; c0 += 1024) {
    const int m = n - c0 < 1024 ? n - c0 : 1024;
    e = cudaMemcpyAsync(chunk, scratch + 64 + c0, sizeof(int) * (size_t)m, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    for (int j = 0; j < m; ++j)
      if (chunk[j] != 0) {
        *first_bad = c0 + j;
        return cudaSuccess;
      }
  }
  return cudaSuccess;
}

#endif  // LRDMC_PART == 0

}  // namespace lrdmc
