// The evaluation of the double-float mode (LRDMC_PRECISION_DF64): all
// lattice moves out of a configuration (Eq. 1 lattice, fixed-node rates) and
// its local energy, one warp per walker, in lean double-float arithmetic on
// the FP32 pipe (lean64.cuh). The mixed mode shares the local energy and the
// Sherman-Morrison update.
//
// What bounds it: issue slots and the latency of dependent chains (an FP32
// instruction 4-5 cycles, a shared-memory read about 30; an FP64
// instruction holds its sub-partition's pipe for 64 cycles whatever its lane
// count, so conversions are integer code). So the design removes
// instructions:
//   * a lane evaluates the two moves +-h e_k of one electron, grid and axis
//     together: they share D + h^2, 2 h P_k, the angular parts and every
//     table read, and their two chains interleave;
//   * distances come from one cached D = |r_i - r_j|^2 per pair and the
//     positions on the rotated axes y = R^T r: |r_i +- h e_k - r_j|^2 = D +
//     h^2 +- 2h (y_ik - y_jk). Lengths of the e-e part are scaled by b in
//     the form below, so that the square root is b r itself;
//   * the e-e Pade sum needs one reciprocal per partner: c r/(1 + b r) =
//     c/b - (c/b)/(1 + b r), whose constant cancels in the Jastrow
//     difference (for b below 1/4, where that form would lose digits or
//     divide by zero, and above 2^20, where its lengths could leave the float
//     range, the product form c r q);
//   * after a jump only what moved is formed again: the projected columns of
//     one spin, one electron's position and its N - 1 distances.
// Near a node the projected columns are large and the basis sums cancel, so
// the radial parts and their sums are renormalised at every step (1 to 3 % of
// a projection's time): error of the ratios against 64 bits, in the 2-norm
// over 8 samples of 150 configurations (Kr 30; geometric mean), He 5.8e-15, Ne
// 8e-14, H2O 1.7e-13, Ar 1.3e-13, Kr 1.6e-13, where products and sums left
// unnormalised gave 7.9e-15, 1.3e-13, 2.6e-13, 1.8e-13 and 2.3e-13.
#pragma once
#include "lean64.cuh"

namespace lrdmc {

// A shell as the evaluation reads it from shared memory (16-byte reads).
struct LShell {
  int kind, l, m_int, ao;      // kind 0 Slater, 1 Gaussian contraction
  int prim, n_prim, same_exp, center;
  float zeta_hi, zeta_lo, m_hi, m_lo;
  int gt_base, gt_cells, gt_key0;
  float gt_beta;
};

static __device__ const __align__(16) float2 g_exp_tab[kExpEntries] = {
#include "exp_table.inc"
};

// Block-shared tables of the double-float evaluation.
struct Lean {
  const float2* tab;   // 2^(j/1024)
  const LShell* sh;    // [n_shell]
  const float4* prim;  // [n_prim] alpha (hi, lo), coefficient (hi, lo)
};

__device__ __forceinline__ Lean lean_mem(const SysDev& S, double* head)
{
  Lean m;
  double* p = head + lean_offset(S);
  m.tab = reinterpret_cast<const float2*>(p);
  p += kExpEntries;
  m.prim = reinterpret_cast<const float4*>(p);
  p += 2 * S.n_prim;
  m.sh = reinterpret_cast<const LShell*>(p);
  return m;
}

// Fills the tables (every thread of the block; the caller synchronises).
__device__ __forceinline__ void lean_stage(const SysDev& S, double* head)
{
  const Lean m = lean_mem(S, head);
  float4* tab = reinterpret_cast<float4*>(const_cast<float2*>(m.tab));
#pragma unroll 1
  for (int j = threadIdx.x; j < kExpEntries / 2; j += blockDim.x)
    tab[j] = __ldg(reinterpret_cast<const float4*>(g_exp_tab) + j);
#pragma unroll 1
  for (int q = threadIdx.x; q < S.n_shell; q += blockDim.x) {
    LShell* o = const_cast<LShell*>(m.sh) + q;
    const ShellDev& sh = S.sh[q];
    const DfShell& d = S.D.sh[q];
    o->kind = sh.kind; o->l = sh.l; o->m_int = sh.m_int; o->ao = sh.ao_offset;
    o->prim = sh.prim_begin; o->n_prim = sh.n_prim; o->same_exp = sh.same_exp; o->center = sh.center;
    o->gt_base = sh.gt_base; o->gt_cells = sh.gt_cells; o->gt_key0 = sh.gt_key0; o->gt_beta = sh.gt_beta;
    o->zeta_hi = d.zeta.hi; o->zeta_lo = d.zeta.lo; o->m_hi = d.m.hi; o->m_lo = d.m.lo;
    float4* pr = const_cast<float4*>(m.prim) + sh.prim_begin;
#pragma unroll 1
    for (int p = 0; p < sh.n_prim; ++p)
      pr[p] = make_float4(d.alpha[p].hi, d.alpha[p].lo, d.coef[p].hi, d.coef[p].lo);
  }
}

__device__ __forceinline__ dl dl_at(float4 v, int half) { return half ? df_make(v.z, v.w) : df_make(v.x, v.y); }

__device__ __forceinline__ dl dl_shfl_down(dl v, int o)
{
  return df_make(__shfl_down_sync(FULL_MASK, v.hi, o), __shfl_down_sync(FULL_MASK, v.lo, o));
}

__device__ __forceinline__ dl dl_warp_sum(dl v)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = dl_add_n(v, df_make(__shfl_xor_sync(FULL_MASK, v.hi, o), __shfl_xor_sync(FULL_MASK, v.lo, o)));
  return v;
}

// Pair (i, j), i != j, in the distance cache: the pairs of spin-up electrons
// (lower triangle), of spin-down electrons, then up x down.
__device__ __forceinline__ int pair_q(const SysDev& S, int i, int j)
{
  const int nu = S.n_up, nd = S.n_dn, a = min(i, j), b = max(i, j), tu = nu * (nu - 1) / 2;
  if (b < nu) return b * (b - 1) / 2 + a;
  if (a >= nu) return tu + (b - nu) * (b - nu - 1) / 2 + (a - nu);
  return tu + nd * (nd - 1) / 2 + a * nd + (b - nu);
}

// r^m = e^(m log r) (out of line: one copy of code that few systems run)
static __device__ __noinline__ dl real_power(dl m, dl r, const LeanExp K, const float2* tab)
{
  return dl_norm(dl_exp(dl_norm(dl_mul(m, dl_log(dl_norm(r), K, tab))), K, tab));
}

// r^m for a Slater shell: a small whole power, or e^(m log r)
__device__ __forceinline__ dl slater_power(const LShell& sh, dl r, const SysDev& S, const Lean& t)
{
  if (sh.m_int == 1) return r;
  if (sh.m_int >= 0) {
    dl p = df_make(1.0f, 0.0f);
#pragma unroll 1
    for (int j = 0; j < sh.m_int; ++j) p = dl_mul(p, r);
    return dl_norm(p);
  }
  return real_power(df_make(sh.m_hi, sh.m_lo), r, S.D.lexp, t.tab);
}

// The five degree-2 solid harmonics of two points contracted with v.
__device__ __forceinline__ dl2 solid2_dot2(const df* v, const dl2 d[3])
{
  const dl2 xx = dl2_sqr(d[0]), yy = dl2_sqr(d[1]), zz = dl2_sqr(d[2]);
  dl2 s = dl2_add(dl2_mul(dl2_all(v[0]), dl2_mul(d[0], d[1])), dl2_mul(dl2_all(v[1]), dl2_mul(d[1], d[2])));
  s = dl2_add(s, dl2_mul(dl2_all(v[2]), dl2_mul(d[2], d[0])));
  s = dl2_add(s, dl2_mul(dl2_all(v[3]), dl2_norm(dl2_sub(xx, yy))));
  return dl2_add_n(s, dl2_mul(dl2_all(v[4]), dl2_norm(dl2_sub(dl2_add(zz, zz), dl2_add(xx, yy)))));
}

__device__ __forceinline__ dl2 slater_power2(const LShell& sh, dl2 r, const SysDev& S, const Lean& t)
{
  if (sh.m_int == 1) return r;
  if (sh.m_int >= 0) {
    dl2 p = dl2_all(df_make(1.0f, 0.0f));
#pragma unroll 1
    for (int j = 0; j < sh.m_int; ++j) p = dl2_mul(p, r);
    return dl2_norm(p);
  }
  dl a, b;
  dl2_split(r, a, b);
  const dl m = df_make(sh.m_hi, sh.m_lo);
  a = real_power(m, a, S.D.lexp, t.tab);
  b = real_power(m, b, S.D.lexp, t.tab);
  return dl2_pack(a, b);
}

__device__ __forceinline__ dl dl_dot3(const df* a, const dl b[3])
{
  return dl_add_n(dl_add(dl_mul(a[0], b[0]), dl_mul(a[1], b[1])), dl_mul(a[2], b[2]));
}

// Electron-nucleus geometry of electron i and nucleus I from the positions:
// d = r_i - R_I and D = |d|^2.
__device__ __forceinline__ void en_geometry(const SysDev& S, const WarpMem& wm, int i, int I, dl d[3], dl& D)
{
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = dl_sub_n(wm.xd[3 * i + k], S.D.nuc[I][k]);
  D = dl_add_n(dl_add_n(dl_norm(dl_sqr(d[0])), dl_norm(dl_sqr(d[1]))), dl_norm(dl_sqr(d[2])));
}

__device__ __forceinline__ dl axis_dot(const WarpMem& wm, int k, const dl d[3])
{
  return dl_add_n(dl_add(dl_mul(wm.Rd[k], d[0]), dl_mul(wm.Rd[3 + k], d[1])), dl_mul(wm.Rd[6 + k], d[2]));
}

// b^2 |r_i - r_j|^2 from the positions (b: the scale of the e-e part, ee_scale)
__device__ __forceinline__ dl pair_d2(const SysDev& S, const WarpMem& wm, int i, int j, dl d[3])
{
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = dl_sub_n(wm.xd[3 * i + k], wm.xd[3 * j + k]);
  const dl D = dl_add(dl_add(dl_sqr(d[0]), dl_sqr(d[1])), dl_sqr(d[2]));
  return dl_norm(dl_mul(dl_norm(D), S.D.ee_scale2));
}

// The neural pair term at r: the cell's quintic (cubic to quintic terms in
// single precision, see nj_value_m), and its derivatives.
__device__ __forceinline__ dl nj_value64(const SysDev& S, int c, dl r)
{
  const float rf = r.hi;
  if (!(rf < S.nj_rcut_f[c])) return df_make(0.0f, 0.0f);
  df E[8];
  nj_load(nj_cell_m(S, c, rf), E);
  const dl t = dl_mul(dl_sub_n(r, E[0]), E[1]);
  const float hi = fmaf(fmaf(E[7].hi, t.hi, E[6].hi), t.hi, E[5].hi);
  dl v = dl_add(E[4], dl_mul_f(t, hi));
  v = dl_add_n(dl_mul(v, t), E[3]);
  return dl_add_n(dl_mul(v, t), E[2]);
}

__device__ __forceinline__ void nj_value3_64(const SysDev& S, int c, dl r0, dl& g, dl& g1, dl& g2)
{
  g = g1 = g2 = df_make(0.0f, 0.0f);
  const df r = dl_norm(r0);
  if (!(r.hi < S.nj_rcut_f[c])) return;
  df E[8];
  nj_load(nj_cell_m(S, c, r.hi), E);
  const df iw = E[1], t = df_mul(df_sub(r, E[0]), iw);
  df v = E[7], d1 = df_mul_f(E[7], 5.0f), d2 = df_mul_f(E[7], 20.0f);
#pragma unroll
  for (int q = 6; q >= 2; --q) v = df_add(df_mul(v, t), E[q]);
  g = v;
#pragma unroll
  for (int q = 6; q >= 4; --q) d1 = df_add(df_mul(d1, t), df_mul_f(E[q], (float)(q - 2)));
  d1 = df_add(df_mul(d1, t), E[3]);
#pragma unroll
  for (int q = 6; q >= 4; --q) d2 = df_add(df_mul(d2, t), df_mul_f(E[q], (float)((q - 2) * (q - 3))));
  g1 = df_mul(d1, iw);
  g2 = df_mul(d2, df_sqr(iw));
}

// ----------------------------------------------------------------------------
// Local energy of the configuration, and per electron the e-e and e-n
// Jastrow sums that the moves compare with. Electrons are taken el_E at a
// time with el_L lanes ("parts") each; a part sums over its own shell units,
// partners and nuclei. Every part's share of the terms that enter linearly
// (Laplacians, potential) goes straight into the warp's total; the gradients
// and Jastrow sums are combined over the parts by a shuffle tree.
// ----------------------------------------------------------------------------
template <bool NJ>
__device__ __forceinline__ double local_energy64(const SysDev& S, const WarpMem& wm, const Lean& lt, int lane)
{
  const int N = S.N, nao = S.n_ao, E = S.el_E, L = S.el_L;
  const int part = lane / E;
  const dl zero = df_make(0.0f, 0.0f);
  const bool recip = S.ee_recip != 0;
  dl total = zero;
#pragma unroll 1
  for (int i0 = 0; i0 < N; i0 += E) {
    const int i = i0 + lane - part * E;
    const bool act = part < L && i < N;
    dl gD[3] = {zero, zero, zero}, gJ[3] = {zero, zero, zero}, see = zero, sen = zero;
    if (act) {
      const df* v = &wm.vd[i * nao];
      // basis: per shell P = sum_f v_f S_f and grad P, then gD += R grad P +
      // (R'/r) P d and lap += P (R'' + 2 (l + 1) R'/r)
      dl lap = zero;
      int pc = -1;
      dl d[3], r2 = zero, r = zero, ir = zero, e = zero;
#pragma unroll 1
      for (int gi = part; gi < S.n_grp64; gi += L)
#pragma unroll 1
        for (int q = S.grp64_first[gi]; q < S.grp64_first[gi + 1]; ++q) {
          const LShell sh = lt.sh[q];
          if (sh.center != pc) {
            pc = sh.center;
            en_geometry(S, wm, i, pc, d, r2);
            r = dl_norm(dl_sqrt_acc(r2));
            ir = dl_norm(dl_rcp(r));
          }
          dl R, R1, R2;
          if (sh.kind == 0) {
            const dl zeta = df_make(sh.zeta_hi, sh.zeta_lo);
            if (q == S.grp64_first[gi] || !sh.same_exp) e = dl_exp(dl_neg(dl_norm(dl_mul(zeta, r))), S.D.lexp, lt.tab);
            R = sh.m_int == 0 ? dl_norm(e) : dl_mul_n(slater_power(sh, r, S, lt), e);
            const dl m = df_make(sh.m_hi, sh.m_lo);
            const dl mir = dl_mul(m, ir);
            const dl t = dl_sub_n(mir, zeta);
            R1 = dl_mul_n(dl_mul_n(t, ir), R);
            R2 = dl_mul_n(dl_sub_n(dl_sqr(t), dl_mul(mir, ir)), R);
          } else {
            dl A0 = zero, A1 = zero, A2 = zero;
#pragma unroll 1
            for (int p = 0; p < sh.n_prim; ++p) {
              const float4 pr = lt.prim[sh.prim + p];
              const dl al = dl_at(pr, 0);
              // R'/r = -2 sum a g, R'' = 4 sum a g (a r^2 - 1/2)
              const dl t = dl_norm(dl_mul(al, r2));
              const dl g = dl_mul_n(dl_at(pr, 1), dl_norm(dl_exp(dl_neg(t), S.D.lexp, lt.tab)));
              const dl ag = dl_mul_n(al, g);
              A0 = dl_add_n(A0, g);
              A1 = dl_add_n(A1, ag);
              A2 = dl_add_n(A2, dl_mul_n(dl_norm(dl_add_f(t, -0.5f)), ag));
            }
            R = A0;
            R1 = dl_scale(A1, -2.0f);
            R2 = dl_scale(A2, 4.0f);
          }
          dl P, g[3];
          if (sh.l == 0) {
            P = v[sh.ao];
          } else if (sh.l == 1) {
            P = dl_dot3(&v[sh.ao], d);
#pragma unroll
            for (int k = 0; k < 3; ++k) g[k] = v[sh.ao + k];
          } else {
            // gradient of the quadratic form; P = d . grad P / 2
            const df* w = &v[sh.ao];
            const dl w34 = dl_scale(dl_sub_n(w[3], w[4]), 2.0f), w43 = dl_scale(dl_add_n(w[3], w[4]), -2.0f);
            g[0] = dl_add_n(dl_add(dl_mul(w[0], d[1]), dl_mul(w[2], d[2])), dl_mul(w34, d[0]));
            g[1] = dl_add_n(dl_add(dl_mul(w[0], d[0]), dl_mul(w[1], d[2])), dl_mul(w43, d[1]));
            g[2] = dl_add_n(dl_add(dl_mul(w[1], d[1]), dl_mul(w[2], d[0])), dl_scale(dl_mul(w[4], d[2]), 4.0f));
            P = dl_scale(dl_dot3(g, d), 0.5f);
          }
          const dl W = dl_mul_n(P, R1);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            gD[k] = dl_add(gD[k], dl_mul(W, d[k]));
            if (sh.l > 0) gD[k] = dl_add(gD[k], dl_mul(R, g[k]));
          }
          lap = dl_add(lap, dl_mul(P, dl_add_n(R2, dl_mul_f(R1, 2.0f * (sh.l + 1)))));
        }
      // e-e pairs, the N - 1 partners dealt to the parts. With s = b r (r in
      // the general form), q = 1/(1 + b r): u'/r = c q^2 / r, u'' + 2 u'/r =
      // 2 c q^2 (1/r - b q)
      dl lap2 = zero, pot = zero, snj = zero;
      const int si = spin_of(S, i);
#pragma unroll 1
      for (int t = part; t < N - 1; t += L) {
        const int j = t < i ? t : t + 1;
        dl dd[3], D;
        D = pair_d2(S, wm, i, j, dd);
        const dl s = dl_norm(dl_sqrt_acc(D)), is = dl_inv_distance(D, s);
        const dl c = spin_of(S, j) == si ? S.D.c_par : S.D.c_anti;
        dl q, qs;
        if (recip) {
          q = dl_norm(dl_rcp(dl_one_plus(s)));
          qs = q;
          see = dl_add(see, dl_mul(c, q));
        } else {
          q = dl_rcp(dl_norm(dl_add_f(dl_mul(S.D.b_ee, s), 1.0f)));
          qs = dl_mul(S.D.b_ee, q);
          see = dl_add(see, dl_mul(c, dl_mul(s, q)));
        }
        const dl cq2 = dl_mul_n(c, dl_norm(dl_sqr(q)));
        dl a1 = dl_mul_n(cq2, is);
        lap2 = dl_add(lap2, dl_mul(cq2, dl_sub_n(is, qs)));
        if (NJ) {
          dl gv, g1, g2;
          const dl r = dl_mul(s, S.D.ee_iscale);
          nj_value3_64(S, nj_ch_ee(S, i, j), r, gv, g1, g2);
          const dl g1r = dl_mul(g1, dl_mul(is, S.D.ee_scale));
          snj = dl_add(snj, gv);
          lap = dl_add(lap, dl_add(g2, dl_scale(g1r, 2.0f)));
          a1 = dl_add_n(a1, dl_mul(g1r, S.D.ee_iscale));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) gJ[k] = dl_add(gJ[k], dl_mul(a1, dd[k]));
        if (j > i) pot = dl_add(pot, is);
      }
      sen = snj;
      lap = dl_add(lap, dl_scale(dl_mul(dl_norm(lap2), S.D.ee_scale), 2.0f));
#pragma unroll
      for (int k = 0; k < 3; ++k) gJ[k] = dl_mul(dl_norm(gJ[k]), S.D.ee_scale);
      dl lin = S.ee_on ? dl_mul(dl_norm(pot), S.D.ee_scale) : zero;
      // e-n terms
#pragma unroll 1
      for (int I = part; I < S.n_nuc; I += L) {
        dl dd[3], D;
        en_geometry(S, wm, i, I, dd, D);
        const dl rr = dl_norm(dl_sqrt_acc(D));
        const dl is = dl_inv_distance(D, rr);
        const dl b1 = S.D.en_b1[I], b2 = S.D.en_b2;
        const dl q = dl_norm(dl_rcp(dl_norm(dl_add_f(dl_mul(b2, rr), 1.0f))));
        const dl bq2 = dl_mul_n(b1, dl_norm(dl_sqr(q)));
        dl a1 = dl_neg(dl_mul_n(bq2, is));
        lap = dl_sub(lap, dl_scale(dl_mul(bq2, dl_sub_n(is, dl_mul(b2, q))), 2.0f));
        sen = dl_sub(sen, dl_mul(dl_mul(b1, rr), q));
        if (NJ) {
          dl gv, g1, g2;
          nj_value3_64(S, 2 + S.nj_species[I], rr, gv, g1, g2);
          const dl g1r = dl_mul(g1, is);
          sen = dl_add(sen, gv);
          lap = dl_add(lap, dl_add(g2, dl_scale(g1r, 2.0f)));
          a1 = dl_add_n(a1, g1r);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) gJ[k] = dl_add(gJ[k], dl_mul(a1, dd[k]));
        lin = dl_sub(lin, dl_mul(S.D.Z[I], is));
      }
      total = dl_add_n(total, dl_sub(lin, dl_scale(lap, 0.5f)));
    }
    // combine the parts of each electron (lane part * E + i)
    if (L > 1) {
#pragma unroll 1
      for (int o = S.el_top; o > 0; o >>= 1) {
        const bool take = part < o && part + o < L;
        const int sh = o * E;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          dl t = dl_shfl_down(gD[k], sh);
          if (take) gD[k] = dl_add(gD[k], t);
          t = dl_shfl_down(gJ[k], sh);
          if (take) gJ[k] = dl_add(gJ[k], t);
        }
        dl t = dl_shfl_down(see, sh);
        if (take) see = dl_add(see, t);
        t = dl_shfl_down(sen, sh);
        if (take) sen = dl_add(sen, t);
      }
    }
    if (part == 0 && act) {
      wm.Sd[i] = dl_norm(see);
      wm.Sn[i] = dl_norm(sen);
      dl quad = zero;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const dl j = dl_norm(gJ[k]);
        quad = dl_add(quad, dl_mul(j, dl_add_n(j, dl_scale(gD[k], 2.0f))));
      }
      total = dl_sub_n(total, dl_scale(quad, 0.5f));
    }
  }
  return df_to_double(dl_warp_sum(total)) + S.V_nn;
}

// ----------------------------------------------------------------------------
// The first part of an evaluation: projected inverse columns, positions and
// rotation, distances, then the local energy and the Jastrow sums. moved < 0:
// everything; else electron `moved` jumped since the warp's last evaluation
// of this walker, whose other spin's columns, positions and distances stand.
// ----------------------------------------------------------------------------
// MOVES = false leaves out what only the double-float moves read.
template <bool NJ, bool NC, bool MOVES = true>
__device__ __forceinline__ double prelude64(const SysDev& S, const double* sC, const WarpMem& wm, const Lean& lt,
                                            int lane, int moved)
{
  const int N = S.N, nao = S.n_ao, nu = S.n_up, nd = S.n_dn;
  const BlockMem bm = block_mem(S, const_cast<double*>(sC));
  int lo = 0, hi = N;
  if (moved >= 0) {
    lo = moved < nu ? 0 : nu;
    hi = moved < nu ? nu : N;
  }
#pragma unroll 1
  for (int idx = lo * nao + lane; idx < hi * nao; idx += 32) {
    const int i = idx / nao, mu = idx - i * nao;
    const int l = i < nu ? i : i - nu, n = i < nu ? nu : nd;
    const double* Am = i < nu ? wm.A : wm.A + nu * nu;
    wm.vd[idx] = dl_from_double(project_ao(S, bm, Am, mu, l, n));
  }
  if (moved < 0) {
#pragma unroll 1
    for (int j = lane; j < 3 * N; j += 32) wm.xd[j] = dl_from_double(wm.x[j]);
  } else if (lane < 3) {
    wm.xd[3 * moved + lane] = dl_from_double(wm.x[3 * moved + lane]);
  }
  if (lane < 9) wm.Rd[lane] = dl_from_double(wm.R[lane]);
  __syncwarp();
#pragma unroll 1
  for (int j = lane; MOVES && j < 3 * N; j += 32) {
    const int i = j / 3, k = j - 3 * i;
    const dl x[3] = {wm.xd[3 * i], wm.xd[3 * i + 1], wm.xd[3 * i + 2]};
    wm.y[j] = dl_norm(dl_mul(axis_dot(wm, k, x), S.D.ee_scale));
  }
  if (MOVES && !NC) {
#pragma unroll 1
    for (int q = lane; q < N * S.n_nuc; q += 32) {
      const int i = q / S.n_nuc, I = q - i * S.n_nuc;
      dl d[3], D;
      en_geometry(S, wm, i, I, d, D);
      df* e = &wm.enc[kEncWords * q];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        e[k] = d[k];
        e[4 + k] = axis_dot(wm, k, d);
      }
      e[3] = D;
    }
    {
      dl d[3];
      if (moved < 0) {
        const int tu = nu * (nu - 1) / 2, td = nd * (nd - 1) / 2;
#pragma unroll 1
        for (int q = lane; q < wm.n_pc; q += 32) {
          int i, j;
          if (q < tu + td) {
            const int p = q < tu ? q : q - tu;
            // the row a of the triangle with a (a - 1)/2 <= p
            int a = (int)(0.5f * (1.0f + sqrtf(1.0f + 8.0f * (float)p)));
            if (a * (a - 1) / 2 > p) --a;
            if (a * (a + 1) / 2 <= p) ++a;
            i = a;
            j = p - a * (a - 1) / 2;
            if (q >= tu) { i += nu; j += nu; }
          } else {
            const int p = q - tu - td;
            i = p / nd;
            j = nu + p - i * nd;
          }
          wm.pc[q] = pair_d2(S, wm, i, j, d);
        }
      } else {
#pragma unroll 1
        for (int t = lane; t < N - 1; t += 32) {
          const int j = t < moved ? t : t + 1;
          wm.pc[pair_q(S, moved, j)] = pair_d2(S, wm, moved, j, d);
        }
      }
    }
  }
  __syncwarp();
  const double el = local_energy64<NJ>(S, wm, lt, lane);
  __syncwarp();
  return el;
}

// The neural pair term at two distances.
__device__ __forceinline__ dl2 nj_value64_2(const SysDev& S, int c, dl2 r)
{
  dl a, b;
  dl2_split(r, a, b);
  return dl2_pack(nj_value64(S, c, a), nj_value64(S, c, b));
}

// A contracted Gaussian's radial part at two squared distances from its
// table: cells of 1/256 octave of y = x + beta (beta about one over the
// largest exponent: uniform cells near the nucleus, relative ones beyond),
// the degree-7 polynomial of the cell in u = (y - centre)/width, its first
// four coefficients as double-floats, the others single (their terms stay
// below 2e-6 of the value while the exponent is below 40); 0 beyond the last
// cell, where every primitive's exponent is below -87. About 75 instructions
// for the two distances whatever the contraction length, against about 55
// per primitive: 64 k cycles of a water walker-move's 116 k went to its 30
// primitives.
__device__ __forceinline__ dl2 radial_table2(const LShell& sh, const float4* gt, dl2 x)
{
  const dl2 y = dl2_two_sum(x.hi, f2_all(sh.gt_beta));
  const f2 ylo = f2_add(y.lo, x.lo);
  float yh[2], ctr[2], iw[2];
  f2_split(y.hi, yh[0], yh[1]);
  // x may be a rounding residue below zero: the first cell begins at beta
#pragma unroll
  for (int m = 0; m < 2; ++m) yh[m] = fmax_nan(yh[m], sh.gt_beta);
  const f2 yhi = f2_make(yh[0], yh[1]);
  float4 c[2][3];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const unsigned key = __float_as_uint(yh[m]) >> 15;
    const unsigned cell = key - (unsigned)sh.gt_key0;
    ctr[m] = __uint_as_float((key << 15) | 0x4000u);
    iw[m] = __uint_as_float((262u - (key >> 8)) << 23);
    if (cell < (unsigned)sh.gt_cells) {
      const float4* p = gt + 3 * (size_t)(sh.gt_base + (int)cell);
#pragma unroll
      for (int q = 0; q < 3; ++q) c[m][q] = __ldg(p + q);
    } else {
#pragma unroll
      for (int q = 0; q < 3; ++q) c[m][q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      ctr[m] = yh[m];
      iw[m] = 0.0f;
    }
  }
  const f2 w = f2_make(iw[0], iw[1]);
  const dl2 u = dl2_make(f2_mul(f2_sub(yhi, f2_make(ctr[0], ctr[1])), w), f2_mul(ylo, w));
#define LRDMC_C(q, f) f2_make(c[0][q].f, c[1][q].f)
  f2 t = f2_fma(u.hi, LRDMC_C(2, w), LRDMC_C(2, z));
  t = f2_fma(u.hi, t, LRDMC_C(2, y));
  t = f2_fma(u.hi, t, LRDMC_C(2, x));
  dl2 v = dl2_fast_two_sum(LRDMC_C(1, z), f2_fma(u.hi, t, LRDMC_C(1, w)));
  v = dl2_add(dl2_make(LRDMC_C(1, x), LRDMC_C(1, y)), dl2_mul(u, v));
  v = dl2_add(dl2_make(LRDMC_C(0, z), LRDMC_C(0, w)), dl2_mul(u, v));
  v = dl2_add(dl2_make(LRDMC_C(0, x), LRDMC_C(0, y)), dl2_mul(u, v));
#undef LRDMC_C
  return v;
}

// One partner of the e-e sums of the moves +-h e_k: Dh = b^2 (D + h^2), p =
// 2 b^2 h (y_ik - y_jk)/b, b the scale; acc receives q (r q in the general form).
template <bool NJ>
__device__ __forceinline__ void ee_partner64(const SysDev& S, dl Dh, dl p, int ch, dl2& acc, dl2& nj)
{
  const dl2 s = dl2_sqrt(dl2_norm(dl2_add_big(dl2_all(Dh), dl2_pm(p))));
  if (S.ee_recip) {
    // q <= 1 <= acc: the sum starts from one
    acc = dl2_add_big(acc, dl2_rcp(dl2_one_plus(s)));
  } else {
    const dl2 q = dl2_rcp(dl2_norm(dl2_add_f(dl2_mul(dl2_all(S.D.b_ee), s), f2_all(1.0f))));
    acc = dl2_add(acc, dl2_mul(s, q));
  }
  if (NJ) nj = dl2_add(nj, nj_value64_2(S, ch, dl2_mul(s, dl2_all(S.D.ee_iscale))));
}

// The two lattice moves +-h e_k of unit u = (electron, grid, axis): rates
// into Td, ratios into ratio_out (nullable). gt: the radial table, or null
// (the stateless evaluations, which keep no device memory for a system).
template <bool NJ, bool NC>
__device__ __forceinline__ void moves64(const SysDev& S, const LatDev& L, const WarpMem& wm, const Lean& lt, int u,
                                        df* Td, double* ratio_out, const float4* gt)
{
  const int G = L.G, i = u / (3 * G), rem = u - i * 3 * G, g = rem / 3, k = rem - 3 * g;
  const int nu = S.n_up;
  const df* v = &wm.vd[i * S.n_ao];
  const dl h = g ? L.ap_df : L.a_df;
  const f2 one = f2_all(1.0f);
  dl2 rdet = dl2_zero(), jn = dl2_zero();
  dl mid[2];
  mid[0] = mid[1] = df_make(INFINITY, 0.0f);
  {
    const dl h2 = dl_sqr(h);
    const dl he[3] = {dl_mul(h, wm.Rd[k]), dl_mul(h, wm.Rd[3 + k]), dl_mul(h, wm.Rd[6 + k])};
#pragma unroll 1
    for (int I = 0; I < S.n_nuc; ++I) {
      dl d[3], D, hp;
      if (NC) {
        en_geometry(S, wm, i, I, d, D);
        hp = dl_mul(h, axis_dot(wm, k, d));
      } else {
        const df* e = &wm.enc[kEncWords * (i * S.n_nuc + I)];
#pragma unroll
        for (int q = 0; q < 3; ++q) d[q] = e[q];
        D = e[3];
        hp = dl_mul(h, e[4 + k]);
      }
      // |d +- h e|^2 = D + h^2 +- 2 h p (D + h^2 >= 2 h |p|); the bond's
      // midpoint D + h^2/4 +- h p
      const dl Dh = dl_add_n(D, h2);
      if (G == 2 && S.heavy[I]) {
        dl t[2];
        dl2_split(dl2_norm(dl2_add_big(dl2_all(dl_add_n(D, dl_scale(h2, 0.25f))), dl2_pm(hp))), t[0], t[1]);
#pragma unroll
        for (int m = 0; m < 2; ++m)
          if (t[m].hi < mid[m].hi || (t[m].hi == mid[m].hi && t[m].lo < mid[m].lo)) mid[m] = t[m];
      }
      const dl2 r2 = dl2_norm(dl2_add_big(dl2_all(Dh), dl2_pm(dl_scale(hp, 2.0f))));
      const dl2 r = dl2_norm(dl2_sqrt_acc(r2));
      dl2 e = dl2_zero();
      if (S.en_b1[I] != 0.0) {
        const dl2 q = dl2_rcp(dl2_norm(dl2_add_f(dl2_mul(dl2_all(S.D.en_b2), r), one)));
        jn = dl2_sub(jn, dl2_mul(dl2_mul(dl2_all(S.D.en_b1[I]), r), q));
      }
      if (NJ) jn = dl2_add(jn, nj_value64_2(S, 2 + S.nj_species[I], r));
#pragma unroll 1
      for (int q = S.nuc_shell_begin[I]; q < S.nuc_shell_begin[I + 1]; ++q) {
        const LShell sh = lt.sh[q];
        dl2 R;
        if (sh.kind == 0) {
          if (!sh.same_exp)
            e = dl2_exp(dl2_norm(dl2_mul(dl2_all(df_make(-sh.zeta_hi, -sh.zeta_lo)), r)), S.D.lexp, lt.tab);
          R = sh.m_int == 0 ? e : dl2_mul(slater_power2(sh, r, S, lt), e);
        } else if (gt && sh.gt_cells) {
          R = radial_table2(sh, gt, r2);
        } else {
          R = dl2_zero();
#pragma unroll 1
          for (int p = 0; p < sh.n_prim; ++p) {
            const float4 pr = lt.prim[sh.prim + p];
            const dl2 al = dl2_all(df_make(-pr.x, -pr.y)), co = dl2_all(df_make(pr.z, pr.w));
            R = dl2_add_n(R, dl2_mul_n(co, dl2_norm(dl2_exp(dl2_norm(dl2_mul(al, r2)), S.D.lexp, lt.tab))));
          }
        }
        dl2 P;
        if (sh.l == 0) {
          P = dl2_all(v[sh.ao]);
        } else if (sh.l == 1) {
          P = dl2_add_n(dl2_all(dl_dot3(&v[sh.ao], d)), dl2_pm(dl_dot3(&v[sh.ao], he)));
        } else {
          dl2 dm[3];
#pragma unroll
          for (int t = 0; t < 3; ++t) dm[t] = dl2_add_n(dl2_all(d[t]), dl2_pm(he[t]));
          P = solid2_dot2(&v[sh.ao], dm);
        }
        rdet = dl2_add_n(rdet, dl2_mul(P, dl2_norm(R)));
      }
    }
  }
  // e-e part: partners of the same spin, then of the other
  dl2 jee, nj = dl2_zero();
  {
    const dl hb = dl_norm(dl_mul(h, S.D.ee_scale)), h2b = dl_norm(dl_sqr(hb)), hb2 = dl_scale(hb, 2.0f);
    const dl yi = wm.y[3 * i + k];
    const bool up = i < nu;
    const dl2 start = dl2_all(df_make(S.ee_recip ? 1.0f : 0.0f, 0.0f));
    const int n_same = up ? nu : S.n_dn, off_same = up ? 0 : nu, l = i - off_same;
    const int tri = up ? 0 : nu * (nu - 1) / 2;
    dl2 acc = start;
    int qq = tri + l * (l - 1) / 2;
    dl dd[3];
#pragma unroll 1
    for (int t = 0; t < n_same - 1; ++t) {
      const int jl = t < l ? t : t + 1, j = off_same + jl;
      dl D;
      if (!NC) {
        if (t >= l) qq = tri + jl * (jl - 1) / 2 + l;
        D = wm.pc[qq];
        ++qq;
      } else {
        D = pair_d2(S, wm, i, j, dd);
      }
      const dl p = dl_mul(hb2, dl_sub(yi, wm.y[3 * j + k]));
      ee_partner64<NJ>(S, dl_add(D, h2b), p, 0, acc, nj);
    }
    jee = dl2_mul(dl2_all(S.D.c_par), dl2_norm(dl2_add_f(acc, f2_neg(start.hi))));
    acc = start;
    const int n_opp = up ? S.n_dn : nu, off_opp = up ? nu : 0;
    const int opp = nu * (nu - 1) / 2 + S.n_dn * (S.n_dn - 1) / 2;
    int qo = up ? opp + l * S.n_dn : opp + l;
    const int dq = up ? 1 : S.n_dn;
#pragma unroll 1
    for (int t = 0; t < n_opp; ++t) {
      const int j = off_opp + t;
      dl D;
      if (!NC) {
        D = wm.pc[qo];
        qo += dq;
      } else {
        D = pair_d2(S, wm, i, j, dd);
      }
      const dl p = dl_mul(hb2, dl_sub(yi, wm.y[3 * j + k]));
      ee_partner64<NJ>(S, dl_add(D, h2b), p, 1, acc, nj);
    }
    jee = dl2_add(jee, dl2_mul(dl2_all(S.D.c_anti), dl2_norm(dl2_add_f(acc, f2_neg(start.hi)))));
  }
  const int c0 = (i * G + g) * 6 + 2 * k;
  // e^(Delta J): J = J_ee(-1/b sum c q, or 1/b sum c s q) + J_en (+ neural)
  dl2 dJ = dl2_mul(dl2_sub_n(jee, dl2_all(wm.Sd[i])), dl2_all(S.D.ee_factor));
  dl2 jx = dl2_sub(jn, dl2_all(wm.Sn[i]));
  if (NJ) jx = dl2_add(jx, nj);
  dJ = dl2_add_n(dJ, jx);
  const dl2 rho = dl2_norm(dl2_mul(dl2_norm(rdet), dl2_exp(dJ, S.D.lexp, lt.tab)));
  dl2 T = dl2_mul(rho, dl2_all(g ? L.inv2ap2_df : L.inv2a2_df));
  if (G == 2) {
    const dl2 x = dl2_mul(dl2_pack(mid[0], mid[1]), dl2_all(L.p_coef_df));
    dl2 w = L.pkind == 0 ? dl2_exp(dl2_neg(dl2_norm(x)), S.D.lexp, lt.tab) : dl2_rcp(dl2_norm(dl2_add_f(x, one)));
    if (g) w = dl2_add_f(dl2_neg(w), one);
    T = dl2_mul(T, dl2_norm(w));
  }
  T = dl2_norm(T);
  dl t[2], ro[2];
  dl2_split(T, t[0], t[1]);
  dl2_split(rho, ro[0], ro[1]);
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    // a move across a node is not allowed
    if (!(ro[m].hi > 0.0f)) t[m] = df_make(0.0f, 0.0f);
    Td[c0 + m] = t[m];
    if (ratio_out) ratio_out[c0 + m] = df_to_double(ro[m]);
  }
}

// ----------------------------------------------------------------------------
// Cumulative rates: every lane sums a run of ceil(P/32) consecutive moves,
// one scan over the lanes gives the running sums at the ends of the runs
// (into pfx, read by the next heat bath); returns the total rate.
// ----------------------------------------------------------------------------
__device__ __forceinline__ dl rate_scan64(const df* T, int P, int lane, df* pfx)
{
  const int run = (P + 31) >> 5, c0 = lane * run;
  dl v = df_make(0.0f, 0.0f);
#pragma unroll 1
  for (int q = 0; q < run; ++q)
    if (c0 + q < P) v = dl_add_n(v, T[c0 + q]);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const dl y = df_make(__shfl_up_sync(FULL_MASK, v.hi, o), __shfl_up_sync(FULL_MASK, v.lo, o));
    if (lane >= o) v = dl_add_n(v, y);
  }
  pfx[lane] = v;
  __syncwarp();
  return df_make(__shfl_sync(FULL_MASK, v.hi, 31), __shfl_sync(FULL_MASK, v.lo, 31));
}

__device__ __forceinline__ bool dl_lt(dl a, dl b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }

// Heat bath: the first move whose cumulative rate exceeds target; where
// rounding at the end of a run or of the list leaves none, the last move
// with a positive rate before that end (-1: no positive rate at all).
__device__ __forceinline__ int heat_bath64(const df* T, int P, int lane, const df* pfx, dl target)
{
  const int run = (P + 31) >> 5;
  const unsigned hit = __ballot_sync(FULL_MASK, dl_lt(target, pfx[lane]));
  const int L = hit ? __ffs(hit) - 1 : 31;
  const int c0 = L * run, c1 = min(P, c0 + run);
  dl C = L > 0 ? pfx[L - 1] : df_make(0.0f, 0.0f);
#pragma unroll 1
  for (int c = c0; c < c1; ++c) {
    C = dl_add_n(C, T[c]);
    if (dl_lt(target, C)) return c;
  }
#pragma unroll 1
  for (int c = c1 - 1; c >= 0; --c)
    if (T[c].hi > 0.0f) return c;
  return -1;
}

// The random numbers of iterations m0 .. m0 + kDrawAhead - 1 of a walker's
// interval, one iteration per lane: lanes 0-15 the waiting time's -log u and
// the heat bath's uniform, lanes 16-31 the rotation (Shoemake's quaternion
// from three uniforms). Per iteration dr holds R[9], then the two
// double-floats. A walker makes about ten jumps per interval, so one pass
// replaces ten in which 30 lanes idled (10 k of 78 k cycles per Ne move).
__device__ __forceinline__ void draw_ahead64(uint64_t seed, uint64_t slot, uint64_t k, uint64_t m0, double* dr,
                                             int lane, const SysDev& S, const Lean& lt)
{
  static_assert(kDrawAhead == 16, "half a warp per tag");
  uint64_t c[4] = {slot, k, m0 + (lane & 15), lane < 16 ? kTagTimeHB : kTagRot};
  philox4x64_10(c, seed, 0ull);
  double* o = dr + (lane & 15) * kDrawWords;
  __syncwarp();
  if (lane < 16) {
    df* od = reinterpret_cast<df*>(o);
    od[9] = dl_neg(dl_log(df_u01(c[0]), S.D.lexp, lt.tab));
    od[10] = df_u01(c[1]);
  } else {
    const dl u = df_u01(c[0]);
    const dl s1 = dl_norm(dl_sqrt_acc(dl_norm(dl_add_f(dl_neg(u), 1.0f)))), s2 = dl_norm(dl_sqrt_acc(u));
    dl q[4];  // x, y, z, w
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      dl a, b;
      dl_sincospi(dl_scale(df_u01(h ? c[2] : c[1]), 2.0f), S.D.inv_fact, S.D.half_pi, &a, &b);
      const dl sh = h ? s2 : s1;
      a = dl_mul(sh, dl_norm(a));
      b = dl_mul(sh, dl_norm(b));
      if (h) { q[2] = a; q[3] = b; }
      else { q[0] = a; q[1] = b; }
    }
    // R00 = 1 - 2(yy + zz)  R01 = 2(xy - zw)  R02 = 2(xz + yw)
    // R10 = 2(xy + zw)  R11 = 1 - 2(xx + zz)  R12 = 2(yz - xw)
    // R20 = 2(xz - yw)  R21 = 2(yz + xw)  R22 = 1 - 2(xx + yy)
    const dl xx = dl_sqr(q[0]), yy = dl_sqr(q[1]), zz = dl_sqr(q[2]);
    const dl xy = dl_mul(q[0], q[1]), xz = dl_mul(q[0], q[2]), yz = dl_mul(q[1], q[2]);
    const dl xw = dl_mul(q[0], q[3]), yw = dl_mul(q[1], q[3]), zw = dl_mul(q[2], q[3]);
    auto off = [](dl a, dl b) { return df_to_double(dl_scale(dl_add_n(a, b), 2.0f)); };
    auto diag = [](dl a, dl b) { return df_to_double(dl_norm(dl_add_f(dl_scale(dl_add_n(a, b), -2.0f), 1.0f))); };
    o[0] = diag(yy, zz);
    o[1] = off(xy, dl_neg(zw));
    o[2] = off(xz, yw);
    o[3] = off(xy, zw);
    o[4] = diag(xx, zz);
    o[5] = off(yz, dl_neg(xw));
    o[6] = off(xz, dl_neg(yw));
    o[7] = off(yz, xw);
    o[8] = diag(xx, yy);
  }
  __syncwarp();
}

// The same for the mixed mode, whose waiting times, uniforms and rotations
// are single precision (Ne 4096, 20 intervals: 13.44 to 12.66 ms).
__device__ __forceinline__ void draw_ahead32(uint64_t seed, uint64_t slot, uint64_t k, uint64_t m0, double* dr,
                                             int lane)
{
  uint64_t c[4] = {slot, k, m0 + (lane & 15), lane < 16 ? kTagTimeHB : kTagRot};
  philox4x64_10(c, seed, 0ull);
  double* o = dr + (lane & 15) * kDrawWords;
  __syncwarp();
  if (lane < 16) {
    df* od = reinterpret_cast<df*>(o);
    od[9] = df_make(-logf(f_u01(c[0])), 0.0f);
    od[10] = df_make(f_u01(c[1]), 0.0f);
  } else {
    const float s1 = sqrtf(1.0f - f_u01(c[0])), s2 = sqrtf(f_u01(c[0]));
    float sa, ca, sb, cb;
    sincospif(2.0f * f_u01(c[1]), &sa, &ca);
    sincospif(2.0f * f_u01(c[2]), &sb, &cb);
    const float qx = s1 * sa, qy = s1 * ca, qz = s2 * sb, qw = s2 * cb;
    // a b + s c d, the second product rounded
    auto e = [](float a, float b, float s, float c, float d) { return __fmaf_rn(a, b, s * __fmul_rn(c, d)); };
    o[0] = (double)(1.0f - 2.0f * e(qy, qy, 1.0f, qz, qz));
    o[1] = (double)(2.0f * e(qx, qy, -1.0f, qz, qw));
    o[2] = (double)(2.0f * e(qx, qz, 1.0f, qy, qw));
    o[3] = (double)(2.0f * e(qx, qy, 1.0f, qz, qw));
    o[4] = (double)(1.0f - 2.0f * e(qx, qx, 1.0f, qz, qz));
    o[5] = (double)(2.0f * e(qy, qz, -1.0f, qx, qw));
    o[6] = (double)(2.0f * e(qx, qz, -1.0f, qy, qw));
    o[7] = (double)(2.0f * e(qy, qz, 1.0f, qx, qw));
    o[8] = (double)(1.0f - 2.0f * e(qx, qx, 1.0f, qy, qy));
  }
  __syncwarp();
}

// Sherman-Morrison update for electron i jumping by sign h along axis kx, in
// IEEE double (near a node the update amplifies rounding by the condition
// number of the Slater matrix: a double-float update parts trajectories from
// the FP64 reference), with the orbitals' basis values in double-float, one
// lane per shell. The new position is left in sm[0..2]. Its own scratch, so
// that the projected columns of the other spin stand.
__device__ __forceinline__ bool sm_update64(const SysDev& S, const double* sC, const WarpMem& wm, const Lean& lt,
                                            int i, double step, int kx, int lane)
{
  const int nu = S.n_up, nao = S.n_ao;
  const int spin = i < nu ? 0 : 1, l = i < nu ? i : i - nu, n = spin ? S.n_dn : nu;
  const BlockMem bm = block_mem(S, const_cast<double*>(sC));
  double* A = spin ? wm.A + nu * nu : wm.A;
  double* pn = wm.sm;          // [4]
  double* chi = pn + 4;        // [n_ao] (double-float, then double)
  double* phi = chi + nao;     // [n]
  double* y = phi + n;         // [n]
  double* col = y + n;         // [n]
  if (lane < 3) pn[lane] = wm.x[3 * i + lane] + step * wm.R[3 * lane + kx];
  __syncwarp();
  const dl pd[3] = {dl_from_double(pn[0]), dl_from_double(pn[1]), dl_from_double(pn[2])};
  df* cd = reinterpret_cast<df*>(chi);
#pragma unroll 1
  for (int q = lane; q < S.n_shell; q += 32) {
    const LShell sh = lt.sh[q];
    dl d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = dl_sub_n(pd[k], S.D.nuc[sh.center][k]);
    const dl r2 = dl_norm(dl_add(dl_add(dl_sqr(d[0]), dl_sqr(d[1])), dl_sqr(d[2])));
    dl R;
    if (sh.kind == 0) {
      const dl r = dl_norm(dl_sqrt_acc(r2));
      R = dl_exp(dl_norm(dl_mul(df_make(-sh.zeta_hi, -sh.zeta_lo), r)), S.D.lexp, lt.tab);
      if (sh.m_int != 0) R = dl_mul(slater_power(sh, r, S, lt), R);
    } else {
      R = df_make(0.0f, 0.0f);
#pragma unroll 1
      for (int p = 0; p < sh.n_prim; ++p) {
        const float4 pr = lt.prim[sh.prim + p];
        R = dl_add(R, dl_mul(df_make(pr.z, pr.w),
                             dl_exp(dl_norm(dl_mul(df_make(-pr.x, -pr.y), r2)), S.D.lexp, lt.tab)));
      }
    }
    R = dl_norm(R);
    df* o = cd + sh.ao;
    if (sh.l == 0) {
      o[0] = R;
    } else if (sh.l == 1) {
#pragma unroll
      for (int k = 0; k < 3; ++k) o[k] = dl_mul(d[k], R);
    } else {
      const dl xx = dl_sqr(d[0]), yy = dl_sqr(d[1]), zz = dl_sqr(d[2]);
      o[0] = dl_mul(dl_mul(d[0], d[1]), R);
      o[1] = dl_mul(dl_mul(d[1], d[2]), R);
      o[2] = dl_mul(dl_mul(d[2], d[0]), R);
      o[3] = dl_mul(dl_sub_n(xx, yy), R);
      o[4] = dl_mul(dl_sub_n(dl_add(zz, zz), dl_add(xx, yy)), R);
    }
  }
  __syncwarp();
#pragma unroll 1
  for (int mu = lane; mu < nao; mu += 32) chi[mu] = df_to_double(cd[mu]);
  __syncwarp();
#pragma unroll 1
  for (int m = lane; m < n; m += 32) {
    phi[m] = orbital_value(S, bm, chi, m);
  }
  __syncwarp();
#pragma unroll 1
  for (int q = lane; q < n; q += 32) {
    double a = 0.0;
#pragma unroll 1
    for (int m = 0; m < n; ++m) a += phi[m] * A[m * n + q];
    y[q] = a;
    col[q] = A[q * n + l];
  }
  __syncwarp();
  const double ratio = y[l];
  if (ratio == 0.0) return false;
  const double inv = 1.0 / ratio;
  __syncwarp();
#pragma unroll 1
  for (int q = lane; q < n; q += 32) y[q] = (y[q] - (q == l ? 1.0 : 0.0)) * inv;
  __syncwarp();
#pragma unroll 1
  for (int idx = lane; idx < n * n; idx += 32) {
    const int m = idx / n, q = idx - m * n;
    A[idx] -= col[m] * y[q];
  }
  __syncwarp();
  return true;
}

// The Jastrow exponent of every electron's pairs and nuclei (the sums that
// single-precision moves compare with), in place of the e-e sums.
__device__ __forceinline__ void total_jastrow64(const SysDev& S, const WarpMem& wm, int lane)
{
#pragma unroll 1
  for (int i = lane; i < S.N; i += 32) {
    const int n_same = (i < S.n_up ? S.n_up : S.n_dn) - 1, n_opp = i < S.n_up ? S.n_dn : S.n_up;
    dl s = wm.Sd[i];
    if (S.ee_recip)  // sum c r/(1 + b r) = 1/b (sum c - sum c q)
      s = dl_sub_n(s, dl_add_n(dl_mul_f(S.D.c_par, (float)n_same), dl_mul_f(S.D.c_anti, (float)n_opp)));
    wm.Sd[i] = dl_add_n(dl_mul(s, S.D.ee_factor), wm.Sn[i]);
  }
  __syncwarp();
}

// One whole evaluation (stateless evaluation, change of lattice).
template <bool NJ, bool NC>
__device__ void warp_eval64(const SysDev& S, double* sC, const LatDev& L, const WarpMem& wm, int lane,
                            double* ratio_out, double& b, double& el, const float4* gt)
{
  const Lean lt = lean_mem(S, sC);
  el = prelude64<NJ, NC>(S, sC, wm, lt, lane, -1);
  const int units = 3 * L.G * S.N;
  df* Td = reinterpret_cast<df*>(wm.T);
#pragma unroll 1
  for (int u = lane; u < units; u += 32) moves64<NJ, NC>(S, L, wm, lt, u, Td, ratio_out, gt);
  __syncwarp();
  b = df_to_double(rate_scan64(Td, 2 * units, lane, wm.pfx));
}

}  // namespace lrdmc
