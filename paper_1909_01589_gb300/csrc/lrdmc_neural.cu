// Neural pair term of the Jastrow factor: the host-side table that the
// projection interpolates, and the training kernels of the variance
// objective (forward with radial derivatives, per-configuration assembly,
// backward to the parameters).
//
// The term (declared in include/lrdmc.h): g_c(r) = m(r, c) s(r / r_cut_c),
// m = w3 . silu(W2 silu(W1 z + b1) + b2) + b3, z = [r^2/(r^2 + ell_k^2),
// one-hot(c)], s(t) = 1 - 10t^3 + 15t^4 - 6t^5. Radial derivatives are
// carried forward through the layers as chains (value, d/dr, d2/dr2):
// a linear layer maps each chain by the same matrix (the bias only the
// value), an activation maps (z, z', z'') to (silu z, silu'(z) z',
// silu''(z) z'^2 + silu'(z) z'').
//
// Training arithmetic is FP32 with the parameters staged in shared memory
// (bfloat16-rounded when the spec asks for it). A block takes 32 pairs at a
// time; their chains are the 96 rows of small matrix products with W2, which
// the threads compute in register tiles (below).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "lrdmc_internal.h"
#include "lean64.cuh"

namespace lrdmc {

// ----------------------------------------------------------------------------
// Host: parameters, rounding and the interpolation table.
// ----------------------------------------------------------------------------
int nj_n_params(int n_feat, int n_ch, int hidden)
{
  const int D = n_feat + n_ch, H = hidden;
  return H * D + H + H * H + H + H + 1;
}

float nj_bf16(float x)
{
  // round to nearest bfloat16, ties to even, on the float32 bit pattern
  uint32_t u;
  memcpy(&u, &x, 4);
  u = (u + 0x7FFFu + ((u >> 16) & 1u)) & 0xFFFF0000u;
  float y;
  memcpy(&y, &u, 4);
  return y;
}

namespace {

struct HostNet {
  int F, C, H, D;
  std::vector<double> ell2, rcut, W1, b1, W2, b2, w3;
  double b3;
};

HostNet host_net(const lrdmc_nj_spec& sp, const float* params)
{
  HostNet n;
  n.F = sp.n_feat; n.C = sp.n_ch; n.H = sp.hidden; n.D = n.F + n.C;
  for (int f = 0; f < n.F; ++f) n.ell2.push_back(sp.ell[f] * sp.ell[f]);
  for (int c = 0; c < n.C; ++c) n.rcut.push_back(sp.r_cut[c]);
  auto val = [&](int idx) { return (double)(sp.bf16 ? nj_bf16(params[idx]) : params[idx]); };
  int o = 0;
  const int H = n.H, D = n.D;
  for (int q = 0; q < H * D; ++q) n.W1.push_back(val(o++));
  for (int q = 0; q < H; ++q) n.b1.push_back(val(o++));
  for (int q = 0; q < H * H; ++q) n.W2.push_back(val(o++));
  for (int q = 0; q < H; ++q) n.b2.push_back(val(o++));
  for (int q = 0; q < H; ++q) n.w3.push_back(val(o++));
  n.b3 = val(o++);
  return n;
}

void silu_chain_d(double z, double z1, double z2, double& a, double& a1, double& a2)
{
  const double sg = 1.0 / (1.0 + exp(-z));
  const double d1 = sg * (1.0 + z * (1.0 - sg));
  const double d2 = sg * (1.0 - sg) * (2.0 + z * (1.0 - 2.0 * sg));
  a = z * sg;
  a1 = d1 * z1;
  a2 = d2 * z1 * z1 + d1 * z2;
}

// g_c(r), g', g'' in IEEE double
void host_radial(const HostNet& n, int c, double r, double& g, double& g1, double& g2)
{
  const double rc = n.rcut[c];
  g = g1 = g2 = 0.0;
  if (!(r < rc)) return;
  std::vector<double> x0(n.D, 0.0), x1(n.D, 0.0), x2(n.D, 0.0);
  for (int f = 0; f < n.F; ++f) {
    const double l2 = n.ell2[f], den = r * r + l2;
    x0[f] = r * r / den;
    x1[f] = 2.0 * r * l2 / (den * den);
    x2[f] = 2.0 * l2 * (l2 - 3.0 * r * r) / (den * den * den);
  }
  x0[n.F + c] = 1.0;
  std::vector<double> h(n.H), h1(n.H), h2(n.H), k(n.H), k1(n.H), k2(n.H);
  for (int u = 0; u < n.H; ++u) {
    double z = n.b1[u], z1 = 0.0, z2 = 0.0;
    for (int f = 0; f < n.D; ++f) {
      const double w = n.W1[u * n.D + f];
      z += w * x0[f]; z1 += w * x1[f]; z2 += w * x2[f];
    }
    silu_chain_d(z, z1, z2, h[u], h1[u], h2[u]);
  }
  for (int u = 0; u < n.H; ++u) {
    double z = n.b2[u], z1 = 0.0, z2 = 0.0;
    for (int v = 0; v < n.H; ++v) {
      const double w = n.W2[u * n.H + v];
      z += w * h[v]; z1 += w * h1[v]; z2 += w * h2[v];
    }
    silu_chain_d(z, z1, z2, k[u], k1[u], k2[u]);
  }
  double m = n.b3, m1 = 0.0, m2 = 0.0;
  for (int u = 0; u < n.H; ++u) { m += n.w3[u] * k[u]; m1 += n.w3[u] * k1[u]; m2 += n.w3[u] * k2[u]; }
  const double t = r / rc;
  const double s = 1.0 - t * t * t * (10.0 - t * (15.0 - 6.0 * t));
  const double s1 = -30.0 * t * t * (1.0 - t) * (1.0 - t) / rc;
  const double s2 = -60.0 * t * (1.0 - t) * (1.0 - 2.0 * t) / (rc * rc);
  g = m * s;
  g1 = m1 * s + m * s1;
  g2 = m2 * s + 2.0 * m1 * s1 + m * s2;
}

}  // namespace

// Per channel and cell k: r_k, 1/w_k and the coefficients c_0..c_5 (in
// t = (r - r_k)/w_k) of the quintic that matches (g, w g', w^2 g'') at both
// ends of the cell. With D = p1 - p0:
//   c0 = p0, c1 = d0, c2 = s0/2,
//   c3 = 10 D - 6 d0 - 4 d1 - (3 s0 - s1)/2,
//   c4 = -15 D + 8 d0 + 7 d1 + (3 s0 - 2 s1)/2,
//   c5 = 6 D - 3 d0 - 3 d1 - (s0 - s1)/2.
void nj_build_table(const lrdmc_nj_spec& sp, const float* params, std::vector<double>& tab)
{
  const HostNet net = host_net(sp, params);
  const int n = sp.n_cells;
  tab.assign((size_t)sp.n_ch * n * 8, 0.0);
  std::vector<double> G(n + 1), G1(n + 1), G2(n + 1), R(n + 1);
  for (int c = 0; c < sp.n_ch; ++c) {
    const double rc = sp.r_cut[c];
    for (int k = 0; k <= n; ++k) {
      const double q = (double)k / n;
      R[k] = rc * q * q;
      host_radial(net, c, R[k], G[k], G1[k], G2[k]);
    }
    for (int k = 0; k < n; ++k) {
      const double w = R[k + 1] - R[k];
      const double p0 = G[k], d0 = w * G1[k], s0 = w * w * G2[k];
      const double p1 = G[k + 1], d1 = w * G1[k + 1], s1 = w * w * G2[k + 1];
      const double D = p1 - p0;
      double* e = &tab[((size_t)c * n + k) * 8];
      e[0] = R[k];
      e[1] = 1.0 / w;
      e[2] = p0;
      e[3] = d0;
      e[4] = 0.5 * s0;
      e[5] = 10.0 * D - 6.0 * d0 - 4.0 * d1 - 0.5 * (3.0 * s0 - s1);
      e[6] = -15.0 * D + 8.0 * d0 + 7.0 * d1 + 0.5 * (3.0 * s0 - 2.0 * s1);
      e[7] = 6.0 * D - 3.0 * d0 - 3.0 * d1 - 0.5 * (s0 - s1);
    }
  }
}

// ----------------------------------------------------------------------------
// Device: training kernels.
// ----------------------------------------------------------------------------
constexpr int kNjH = LRDMC_NJ_HIDDEN;
constexpr int kNjMaxF = LRDMC_NJ_MAX_FEAT;
constexpr int kNjThreads = 128;
constexpr int kNjTile = 32;    // pairs per tile
constexpr int kNjSuper = 128;  // pairs whose geometry is formed at once, one per thread
constexpr int kNjLd = kNjH + 4;  // row stride of the chain matrices (floats; 16-byte aligned, staggered over the banks)
static_assert(kNjH == 64, "16 unit groups of four");

// Shared memory of a block: the parameters (float, bf16-rounded if asked) as
// W1T [D][H], b1, W2T [H][H] (transposed), b2, w3, b3; the pair table; of 128
// pairs the radius, unit vector and channel; of the tile's 32 pairs the
// features with their radial derivatives; the layer-1 activations A [chain][pair][H].
// The backward pass adds W2 [H][H], the upstream derivatives, the layer-2
// derivatives Z [chain][pair][H] and a layer-1 gradient slice per warp.
//
// Thread (pg, ug) of a tile owns pairs 4 pg .. 4 pg + 3 and units 4 ug .. 4 ug +
// 3: per step of a product it reads 12 chain values and 4 weights (16-byte
// loads, most of them broadcast) for 48 multiply-adds, so the FP32 pipe binds
// (with one warp per pair a lane read three words for six multiply-adds, and
// 128 weight gradients per lane spilled).
struct NjSmem {
  float* W1T; float* b1; float* W2T; float* b2; float* w3; float* b3;
  int* pairs;      // [n_pairs]: i | j << 8 | channel << 16 (j = nucleus for e-n)
  float4* geo;     // [128] r, e
  int* ch;         // [128]
  float4* feat;    // [32][F] f, f', f''
  float* A;        // [96][kNjLd]
  float* sum;      // [96] output-layer sums
  float* W2;       // backward: [H][H]
  float4* up;      // [128] upstream derivatives of m, m', m''
  float* Z;        // [96][kNjLd]
  float* acc1;     // [4][D][H]
};

__host__ __device__ inline int nj_smem_floats(int F, int C, int n_pairs, bool backward)
{
  const int D = F + C, H = kNjH;
  int n = D * H + H + H * H + 2 * H + 4;
  n += (n_pairs + 3) & ~3;
  n += 4 * kNjSuper + kNjSuper + 4 * kNjTile * F + 3 * kNjTile * (kNjLd + 1);
  if (backward) n += H * H + 4 * kNjSuper + 3 * kNjTile * kNjLd + 4 * D * H;
  return n;
}

__device__ inline NjSmem nj_stage(const NjGeom& G, const NjNetDev& N, const float* params, float* sm, bool backward)
{
  NjSmem m;
  const int D = N.D, H = kNjH, np = G.n_pairs;
  m.W1T = sm;
  m.b1 = m.W1T + D * H;
  m.W2T = m.b1 + H;
  m.b2 = m.W2T + H * H;
  m.w3 = m.b2 + H;
  m.b3 = m.w3 + H;
  m.pairs = reinterpret_cast<int*>(m.b3 + 4);
  m.geo = reinterpret_cast<float4*>(m.pairs + ((np + 3) & ~3));
  m.ch = reinterpret_cast<int*>(m.geo + kNjSuper);
  m.feat = reinterpret_cast<float4*>(m.ch + kNjSuper);
  m.A = reinterpret_cast<float*>(m.feat + kNjTile * N.F);
  m.sum = m.A + 3 * kNjTile * kNjLd;
  m.W2 = m.sum + 3 * kNjTile;
  m.up = reinterpret_cast<float4*>(m.W2 + H * H);
  m.Z = reinterpret_cast<float*>(m.up + kNjSuper);
  m.acc1 = m.Z + 3 * kNjTile * kNjLd;
  auto rd = [&](int idx) { float v = params[idx]; return N.bf16 ? __bfloat162float(__float2bfloat16_rn(v)) : v; };
  const int oW1 = 0, ob1 = H * D, oW2 = ob1 + H, ob2 = oW2 + H * H, ow3 = ob2 + H, ob3 = ow3 + H;
  for (int q = threadIdx.x; q < H * D; q += blockDim.x) {
    const int u = q / D, f = q % D;
    m.W1T[f * H + u] = rd(oW1 + q);
  }
  for (int q = threadIdx.x; q < H * H; q += blockDim.x) {
    const int u = q / H, v = q % H;
    const float w = rd(oW2 + q);
    if (backward) m.W2[q] = w;
    m.W2T[v * H + u] = w;
  }
  for (int q = threadIdx.x; q < H; q += blockDim.x) {
    m.b1[q] = rd(ob1 + q);
    m.b2[q] = rd(ob2 + q);
    m.w3[q] = rd(ow3 + q);
  }
  if (threadIdx.x == 0) m.b3[0] = rd(ob3);
  if (backward)
    for (int q = threadIdx.x; q < 4 * D * H; q += blockDim.x) m.acc1[q] = 0.0f;
  // pair table: electron pairs i < j, then electron-nucleus pairs i-major
  const int N_e = G.N, n_ee = N_e * (N_e - 1) / 2;
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    int i, j, c;
    if (q < n_ee) {
      // invert q = i N - i (i + 1)/2 + (j - i - 1)
      i = 0;
      int base = 0;
      while (base + (N_e - 1 - i) <= q) { base += N_e - 1 - i; ++i; }
      j = i + 1 + (q - base);
      c = ((i < G.n_up) == (j < G.n_up)) ? 0 : 1;
    } else {
      const int r = q - n_ee;
      i = r / G.n_nuc;
      j = r % G.n_nuc;
      c = 2 + G.species[j];
    }
    m.pairs[q] = i | (j << 8) | (c << 16);
  }
  __syncthreads();
  return m;
}

__device__ __forceinline__ void silu3(float z, float& a, float& d1, float& d2, float& d3)
{
  const float sg = 1.0f / (1.0f + expf(-z));
  const float sp = sg * (1.0f - sg);       // sigma'
  const float u = 1.0f - 2.0f * sg;
  a = z * sg;
  d1 = sg * (1.0f + z * (1.0f - sg));     // silu'
  d2 = sp * (2.0f + z * u);               // silu''
  d3 = sp * (u * (3.0f + z * u) - 2.0f * z * sp);  // third derivative
}

// Distance and unit vector of d = a - b (both double): in double-float
// arithmetic, rounded to single (as the FP64 form to within its rounding;
// FP64 instructions hold their pipe for 64 cycles each); not a number where
// the two coincide.
__device__ __forceinline__ float4 unit_vector(const double* a, const double* b)
{
  dl d[3];
  for (int k = 0; k < 3; ++k) d[k] = dl_sub_n(dl_from_double(a[k]), dl_from_double(b[k]));
  const dl r2 = dl_norm(dl_add(dl_add(dl_sqr(d[0]), dl_sqr(d[1])), dl_sqr(d[2])));
  const dl r = dl_norm(dl_sqrt_acc(r2)), ir = dl_inv_distance(r2, r);
  return make_float4(r.hi, dl_norm(dl_mul(d[0], ir)).hi, dl_norm(dl_mul(d[1], ir)).hi, dl_norm(dl_mul(d[2], ir)).hi);
}

// Cut-off factor s(r/r_c) and its radial derivatives.
__device__ __forceinline__ void cutoff(float r, float rc, float& s, float& s1, float& s2)
{
  const float t = r / rc;
  if (t >= 1.0f) { s = 0.0f; s1 = 0.0f; s2 = 0.0f; return; }
  s = 1.0f - t * t * t * (10.0f - t * (15.0f - 6.0f * t));
  s1 = -30.0f * t * t * (1.0f - t) * (1.0f - t) / rc;
  s2 = -60.0f * t * (1.0f - t) * (1.0f - 2.0f * t) / (rc * rc);
}

// Features of the tile's pairs and their radial derivatives (radial part
// only; the channel code is constant).
__device__ __forceinline__ void tile_features(const NjNetDev& N, const NjSmem& m, int sub)
{
  for (int t = threadIdx.x; t < kNjTile * N.F; t += kNjThreads) {
    const int p = t / N.F, f = t - p * N.F;
    const float r = m.geo[sub * kNjTile + p].x;
    const float l2 = N.ell2[f], r2 = r * r, den = r2 + l2, id = 1.0f / den;
    m.feat[t] = make_float4(r2 * id, 2.0f * r * l2 * id * id, 2.0f * l2 * (l2 - 3.0f * r2) * id * id * id, 0.0f);
  }
}

// c[0..3] += a b over four units
__device__ __forceinline__ void fma4(float c[4], float a, const float4& b)
{
  c[0] = fmaf(a, b.x, c[0]);
  c[1] = fmaf(a, b.y, c[1]);
  c[2] = fmaf(a, b.z, c[2]);
  c[3] = fmaf(a, b.w, c[3]);
}

// Layer-1 pre-activation chains z[chain][pair][unit] of the thread's tile.
__device__ __forceinline__ void layer1(const NjNetDev& N, const NjSmem& m, int sub, int pg, int ug, float z[3][4][4])
{
  const float4 b = *reinterpret_cast<const float4*>(m.b1 + 4 * ug);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int c = m.ch[sub * kNjTile + 4 * pg + p];
    const float4 w = *reinterpret_cast<const float4*>(m.W1T + (N.F + c) * kNjH + 4 * ug);
    z[0][p][0] = b.x + w.x; z[0][p][1] = b.y + w.y; z[0][p][2] = b.z + w.z; z[0][p][3] = b.w + w.w;
#pragma unroll
    for (int u = 0; u < 4; ++u) z[1][p][u] = z[2][p][u] = 0.0f;
  }
#pragma unroll 1
  for (int f = 0; f < N.F; ++f) {
    const float4 w = *reinterpret_cast<const float4*>(m.W1T + f * kNjH + 4 * ug);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float4 ft = m.feat[(4 * pg + p) * N.F + f];
      fma4(z[0][p], ft.x, w);
      fma4(z[1][p], ft.y, w);
      fma4(z[2][p], ft.z, w);
    }
  }
}

// y[chain][pair][unit] += sum_k X[chain][pair][k] W[k][unit] over the 64 k.
__device__ __forceinline__ void row_product(const float* X, const float* W, int pg, int ug, float y[3][4][4])
{
#pragma unroll 1
  for (int k = 0; k < kNjH; k += 4) {
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const float4*>(W + (k + q) * kNjH + 4 * ug);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float4 x = *reinterpret_cast<const float4*>(X + (c * kNjTile + 4 * pg + p) * kNjLd + k);
        fma4(y[c][p], x.x, w[0]);
        fma4(y[c][p], x.y, w[1]);
        fma4(y[c][p], x.z, w[2]);
        fma4(y[c][p], x.w, w[3]);
      }
  }
}

// Activations of the tile's pre-activation chains into A (all three chains).
__device__ __forceinline__ void activate(float* A, int pg, int ug, float z[3][4][4])
{
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    float v[3][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float d1, d2, d3;
      silu3(z[0][p][u], v[0][u], d1, d2, d3);
      v[1][u] = d1 * z[1][p][u];
      v[2][u] = fmaf(d1, z[2][p][u], __fmul_rn(__fmul_rn(d2, z[1][p][u]), z[1][p][u]));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
      *reinterpret_cast<float4*>(A + (c * kNjTile + 4 * pg + p) * kNjLd + 4 * ug) =
          make_float4(v[c][0], v[c][1], v[c][2], v[c][3]);
  }
}

// Both layers' pre-activations of the tile: A filled, y the layer-2 chains.
// Two barriers: the features before, A after.
__device__ __forceinline__ void tile_forward(const NjNetDev& N, const NjSmem& m, int sub, int pg, int ug,
                                             float y[3][4][4])
{
  tile_features(N, m, sub);
  __syncthreads();
  layer1(N, m, sub, pg, ug, y);
  activate(m.A, pg, ug, y);
  const float4 b = *reinterpret_cast<const float4*>(m.b2 + 4 * ug);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    y[0][p][0] = b.x; y[0][p][1] = b.y; y[0][p][2] = b.z; y[0][p][3] = b.w;
#pragma unroll
    for (int u = 0; u < 4; ++u) y[1][p][u] = y[2][p][u] = 0.0f;
  }
  __syncthreads();
  row_product(m.A, m.W2T, pg, ug, y);
}

__device__ __forceinline__ float warp_sum_f(float v)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Geometry of this thread's pair of the super-tile; pairs beyond the total
// repeat the last one (their results are not used).
__device__ __forceinline__ void super_geometry(const NjGeom& G, const NjSmem& m, const double* x, long long p,
                                               size_t& cfg, int& code)
{
  cfg = (size_t)(p / G.n_pairs);
  code = m.pairs[(int)(p - (long long)cfg * G.n_pairs)];
  const int i = code & 0xFF, j = (code >> 8) & 0xFF, c = code >> 16;
  const double* xi = x + (cfg * G.N + i) * 3;
  m.geo[threadIdx.x] = unit_vector(xi, c >= 2 ? G.nuc[j] : x + (cfg * G.N + j) * 3);
  m.ch[threadIdx.x] = c;
}

// g, g', g'' of every pair of every configuration.
__global__ void __launch_bounds__(kNjThreads, 2)
k_nj_pairs_fwd(const __grid_constant__ NjGeom G, const __grid_constant__ NjNetDev N, const float* params, int n,
               const double* x, float* pair_out)
{
  extern __shared__ float4 nj_smem4[];
  const NjSmem m = nj_stage(G, N, params, reinterpret_cast<float*>(nj_smem4), false);
  const int pg = threadIdx.x >> 4, ug = threadIdx.x & 15;
  const long long total = (long long)n * G.n_pairs;
  const float b3 = m.b3[0];
  for (long long base = (long long)blockIdx.x * kNjSuper; base < total; base += (long long)gridDim.x * kNjSuper) {
    __syncthreads();  // the previous super-tile is done with geo, ch and A
    size_t cfg;
    int code;
    super_geometry(G, m, x, min(base + threadIdx.x, total - 1), cfg, code);
    __syncthreads();
#pragma unroll 1
    for (int sub = 0; sub < kNjSuper / kNjTile && base + sub * kNjTile < total; ++sub) {
      float y[3][4][4];
      tile_forward(N, m, sub, pg, ug, y);
      __syncthreads();  // A is read; it takes the layer-2 activation chains now
      activate(m.A, pg, ug, y);
      __syncthreads();
      // output layer, one row (chain, pair) per thread: p_l = w_l k_l + w_{l+32}
      // k_{l+32}, summed as the tree l, l ^ 16, l ^ 8, .., l ^ 1
      if (threadIdx.x < 3 * kNjTile) {
        const float* k = m.A + threadIdx.x * kNjLd;
        float v[8][4];
        // the four residues of l modulo 4, each of its eight l
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 a = *reinterpret_cast<const float4*>(k + 4 * q), b = *reinterpret_cast<const float4*>(k + 4 * q + 32);
          const float4 wa = *reinterpret_cast<const float4*>(m.w3 + 4 * q),
                       wb = *reinterpret_cast<const float4*>(m.w3 + 4 * q + 32);
          v[q][0] = fmaf(wb.x, b.x, wa.x * a.x);
          v[q][1] = fmaf(wb.y, b.y, wa.y * a.y);
          v[q][2] = fmaf(wb.z, b.z, wa.z * a.z);
          v[q][3] = fmaf(wb.w, b.w, wa.w * a.w);
        }
        float t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          t[u] = ((v[0][u] + v[4][u]) + (v[2][u] + v[6][u])) + ((v[1][u] + v[5][u]) + (v[3][u] + v[7][u]));
        const float mv = (t[0] + t[2]) + (t[1] + t[3]);
        m.sum[threadIdx.x] = mv;
      }
      __syncthreads();
      const int t = sub * kNjTile + threadIdx.x;
      if (threadIdx.x < kNjTile && base + t < total) {
        const float mv = m.sum[threadIdx.x] + b3, m1 = m.sum[kNjTile + threadIdx.x], m2 = m.sum[2 * kNjTile + threadIdx.x];
        float s, s1, s2;
        cutoff(m.geo[t].x, N.rcut[m.ch[t]], s, s1, s2);
        float* out = pair_out + (size_t)(base + t) * 3;
        out[0] = mv * s;
        out[1] = fmaf(mv, s1, __fmul_rn(m1, s));
        out[2] = fmaf(mv, s2, fmaf(2.0f * m1, s1, __fmul_rn(m2, s)));
      }
    }
  }
}

// Per configuration (one warp): G_i, L_i, J, E_L and q = a + G, in fixed
// summation order.
__global__ void __launch_bounds__(128)
k_nj_assemble(const __grid_constant__ NjGeom G, int n, const double* x, const double* grad_base,
              const double* e_base, const float* pair_out, float* el_out, float* j_out, float* q_out)
{
  const int lane = threadIdx.x & 31;
  const long long cfg = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (cfg >= n) return;
  const int N_e = G.N, n_ee = N_e * (N_e - 1) / 2;
  const float* po = pair_out + (size_t)cfg * G.n_pairs * 3;
  const double* xc = x + (size_t)cfg * N_e * 3;
  float part = 0.0f, jsum = 0.0f;
  for (int q = lane; q < G.n_pairs; q += 32) jsum += po[3 * q];
  for (int i = lane; i < N_e; i += 32) {
    float Gi[3] = {0.0f, 0.0f, 0.0f}, Li = 0.0f;
    for (int j = 0; j < N_e; ++j) {
      if (j == i) continue;
      const int a = min(i, j), b = max(i, j);
      const int q = a * N_e - a * (a + 1) / 2 + (b - a - 1);
      const float4 e = unit_vector(&xc[3 * i], &xc[3 * j]);
      const float g1 = po[3 * q + 1], g2 = po[3 * q + 2];
      Gi[0] += g1 * e.y; Gi[1] += g1 * e.z; Gi[2] += g1 * e.w;
      Li += g2 + 2.0f * g1 / e.x;
    }
    for (int I = 0; I < G.n_nuc; ++I) {
      const int q = n_ee + i * G.n_nuc + I;
      const float4 e = unit_vector(&xc[3 * i], G.nuc[I]);
      const float g1 = po[3 * q + 1], g2 = po[3 * q + 2];
      Gi[0] += g1 * e.y; Gi[1] += g1 * e.z; Gi[2] += g1 * e.w;
      Li += g2 + 2.0f * g1 / e.x;
    }
    const double* a = grad_base + ((size_t)cfg * N_e + i) * 3;
    float dot = 0.0f, gg = 0.0f;
    for (int k = 0; k < 3; ++k) {
      const float ak = (float)a[k];
      dot += ak * Gi[k];
      gg += Gi[k] * Gi[k];
      q_out[((size_t)cfg * N_e + i) * 3 + k] = ak + Gi[k];
    }
    part += 2.0f * dot + gg + Li;
  }
  part = warp_sum_f(part);
  jsum = warp_sum_f(jsum);
  if (lane == 0) {
    el_out[cfg] = (float)(e_base[cfg] - 0.5 * (double)part);
    j_out[cfg] = jsum;
  }
}

// Backward: per pair, the upstream derivatives with respect to g, g', g''
// from d_el and d_j of its configuration, then reverse through the cut-off,
// the output layer and both activations (the derivative chains included):
// per tile three products, W2 times the layer-1 chains (recomputed), W2^T
// times the layer-2 derivatives, and the weight gradient, of which a thread
// keeps 4 x 8 entries in registers over all its block's tiles. Every sum runs
// in a fixed order, so the gradient is the same bits from run to run; each
// block writes its sums to partials [blockIdx.x][n_params] for
// k_nj_grad_reduce.
__global__ void __launch_bounds__(kNjThreads, 2)
k_nj_pairs_bwd(const __grid_constant__ NjGeom G, const __grid_constant__ NjNetDev N, const float* params, int n,
               const double* x, const float* qv, const float* d_el, const float* d_j, float* partials)
{
  extern __shared__ float4 nj_smem4[];
  const NjSmem m = nj_stage(G, N, params, reinterpret_cast<float*>(nj_smem4), true);
  const int pg = threadIdx.x >> 4, ug = threadIdx.x & 15, lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int D = N.D, F = N.F, H = kNjH;
  const int oW1 = 0, ob1 = H * D, oW2 = ob1 + H, ob2 = oW2 + H * H, ow3 = ob2 + H, ob3 = ow3 + H, np = ob3 + 1;
  float gW2[4][8], gb2[4] = {0.0f, 0.0f, 0.0f, 0.0f}, gw3[4] = {0.0f, 0.0f, 0.0f, 0.0f}, gb3 = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) gW2[a][b] = 0.0f;
  const float4 w34 = *reinterpret_cast<const float4*>(m.w3 + 4 * ug);
  const float w3[4] = {w34.x, w34.y, w34.z, w34.w};
  float* my1 = m.acc1 + wib * D * H;
  const long long total = (long long)n * G.n_pairs;
  for (long long base = (long long)blockIdx.x * kNjSuper; base < total; base += (long long)gridDim.x * kNjSuper) {
    __syncthreads();
    {
      // upstream derivatives of this thread's pair (0 beyond the total)
      const bool in = base + threadIdx.x < total;
      size_t cfg;
      int code;
      super_geometry(G, m, x, min(base + threadIdx.x, total - 1), cfg, code);
      const int i = code & 0xFF, j = (code >> 8) & 0xFF, c = code >> 16;
      const float4 e = m.geo[threadIdx.x];
      const float de = in ? d_el[cfg] : 0.0f, dj = in ? d_j[cfg] : 0.0f;
      const float* qi = qv + (cfg * G.N + i) * 3;
      float dg1, dg2;
      if (c >= 2) {
        const float qe = qi[0] * e.y + qi[1] * e.z + qi[2] * e.w;
        dg1 = de * (-qe - 1.0f / e.x);
        dg2 = -0.5f * de;
      } else {
        const float* qj = qv + (cfg * G.N + j) * 3;
        const float qe = (qi[0] - qj[0]) * e.y + (qi[1] - qj[1]) * e.z + (qi[2] - qj[2]) * e.w;
        dg1 = de * (-qe - 2.0f / e.x);
        dg2 = -de;
      }
      float s, s1, s2;
      cutoff(e.x, N.rcut[c], s, s1, s2);
      m.up[threadIdx.x] = in ? make_float4(dj * s + dg1 * s1 + dg2 * s2, dg1 * s + 2.0f * dg2 * s1, dg2 * s, 0.0f)
                             : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncthreads();
#pragma unroll 1
    for (int sub = 0; sub < kNjSuper / kNjTile && base + sub * kNjTile < total; ++sub) {
      float y[3][4][4];
      tile_forward(N, m, sub, pg, ug, y);
      // output layer and layer-2 activation; the derivatives of the layer-2
      // chains into Z
      float tb2[4] = {0.0f, 0.0f, 0.0f, 0.0f}, tw3[4] = {0.0f, 0.0f, 0.0f, 0.0f}, tb3 = 0.0f;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float4 d = m.up[sub * kNjTile + 4 * pg + p];
        if (ug == 0) tb3 += d.x;
        float v[3][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float y1 = y[1][p][u], y2 = y[2][p][u];
          float a, d1, d2, d3;
          silu3(y[0][p][u], a, d1, d2, d3);
          const float k1 = d1 * y1, k2 = d2 * y1 * y1 + d1 * y2;
          tw3[u] += d.x * a + d.y * k1 + d.z * k2;
          const float dh = w3[u] * d.x, dh1 = w3[u] * d.y, dh2 = w3[u] * d.z;
          v[0][u] = dh * d1 + dh1 * d2 * y1 + dh2 * (d3 * y1 * y1 + d2 * y2);
          v[1][u] = dh1 * d1 + 2.0f * dh2 * d2 * y1;
          v[2][u] = dh2 * d1;
          tb2[u] += v[0][u];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
          *reinterpret_cast<float4*>(m.Z + (c * kNjTile + 4 * pg + p) * kNjLd + 4 * ug) =
              make_float4(v[c][0], v[c][1], v[c][2], v[c][3]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        gb2[u] += tb2[u];
        gw3[u] += tw3[u];
      }
      gb3 += tb3;
      __syncthreads();
      // weight gradient: units 4 ug .., inputs 8 pg ..; the tile's sum is
      // formed first (a pair's three chains, which largely cancel, together)
      {
        float gt[4][8];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) gt[a][b] = 0.0f;
#pragma unroll 1
        for (int p = 0; p < kNjTile; ++p)
#pragma unroll
          for (int c = 2; c >= 0; --c) {
            const int r = c * kNjTile + p;
            const float4 z = *reinterpret_cast<const float4*>(m.Z + r * kNjLd + 4 * ug);
            const float4 a0 = *reinterpret_cast<const float4*>(m.A + r * kNjLd + 8 * pg);
            const float4 a1 = *reinterpret_cast<const float4*>(m.A + r * kNjLd + 8 * pg + 4);
            fma4(gt[0], z.x, a0); fma4(gt[0] + 4, z.x, a1);
            fma4(gt[1], z.y, a0); fma4(gt[1] + 4, z.y, a1);
            fma4(gt[2], z.z, a0); fma4(gt[2] + 4, z.z, a1);
            fma4(gt[3], z.w, a0); fma4(gt[3] + 4, z.w, a1);
          }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) gW2[a][b] += gt[a][b];
      }
      // derivatives of the layer-1 activations, W2^T dz, then through silu
      float da[3][4][4];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int u = 0; u < 4; ++u) da[c][p][u] = 0.0f;
      row_product(m.Z, m.W2, pg, ug, da);
      layer1(N, m, sub, pg, ug, y);
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float z1 = y[1][p][u], z2 = y[2][p][u];
          float a, d1, d2, d3;
          silu3(y[0][p][u], a, d1, d2, d3);
          const float e0 = da[0][p][u], e1 = da[1][p][u], e2 = da[2][p][u];
          da[0][p][u] = e0 * d1 + e1 * d2 * z1 + e2 * (d3 * z1 * z1 + d2 * z2);
          da[1][p][u] = e1 * d1 + 2.0f * e2 * d2 * z1;
          da[2][p][u] = e2 * d1;
        }
      // layer-1 gradient: the warp's two pair groups added, then into its slice
#pragma unroll 1
      for (int f = 0; f < F; ++f) {
        float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float4 ft = m.feat[(4 * pg + p) * F + f];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            g[u] += da[0][p][u] * ft.x + da[1][p][u] * ft.y + da[2][p][u] * ft.z;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) g[u] += __shfl_xor_sync(0xffffffffu, g[u], 16);
        if (lane < 16) {
          float4* o = reinterpret_cast<float4*>(my1 + f * H + 4 * ug);
          float4 t = *o;
          t.x += g[0]; t.y += g[1]; t.z += g[2]; t.w += g[3];
          *o = t;
        }
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if ((lane >> 4) == h) {
            float4* o = reinterpret_cast<float4*>(my1 + (F + m.ch[sub * kNjTile + 4 * pg + p]) * H + 4 * ug);
            float4 t = *o;
            t.x += da[0][p][0]; t.y += da[0][p][1]; t.z += da[0][p][2]; t.w += da[0][p][3];
            *o = t;
          }
          __syncwarp();
        }
      __syncthreads();  // the features and Z are free again
    }
  }
  // block totals: the weight gradient is the threads' own; the others are
  // added over the pair groups (layers 2 and 3) or warps (layer 1) in order
  float* out = partials + (size_t)blockIdx.x * np;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) out[oW2 + (4 * ug + a) * H + 8 * pg + b] = gW2[a][b];
  __syncthreads();
  float* red = m.A;  // [8][2][H], then [8]
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    red[(pg * 2) * H + 4 * ug + u] = gb2[u];
    red[(pg * 2 + 1) * H + 4 * ug + u] = gw3[u];
  }
  if (ug == 0) red[16 * H + pg] = gb3;
  __syncthreads();
  for (int t = threadIdx.x; t < H; t += blockDim.x) {
    float a = 0.0f, b = 0.0f;
    for (int g = 0; g < 8; ++g) {
      a += red[(g * 2) * H + t];
      b += red[(g * 2 + 1) * H + t];
    }
    out[ob2 + t] = a;
    out[ow3 + t] = b;
    float c1 = 0.0f;
    for (int f = 0; f < D; ++f) {
      float w = 0.0f;
      for (int g = 0; g < 4; ++g) w += m.acc1[(g * D + f) * H + t];
      out[oW1 + t * D + f] = w;
      if (f >= F) c1 += w;  // every pair has one channel
    }
    out[ob1 + t] = c1;
  }
  if (threadIdx.x == 0) {
    float a = 0.0f;
    for (int g = 0; g < 8; ++g) a += red[16 * H + g];
    out[ob3] = a;
  }
}

// grad[t] = sum over the backward blocks of partials[b][t], in block order,
// compensated (the blocks' sums cancel).
__global__ void k_nj_grad_reduce(const float* partials, int blocks, int np, float* grad)
{
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= np) return;
  dl a = df_make(0.0f, 0.0f);
#pragma unroll 8
  for (int b = 0; b < blocks; ++b) a = dl_add_f(a, partials[(size_t)b * np + t]);
  grad[t] = a.hi + a.lo;
}

static int nj_smem_bytes(const NjGeom& G, const NjNetDev& N, bool backward)
{
  return (int)sizeof(float) * nj_smem_floats(N.F, N.C, G.n_pairs, backward);
}

static int nj_grid(const void* fn, int smem)
{
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kNjThreads, smem);
  return sms * (per > 0 ? per : 1);
}

cudaError_t launch_nj_forward(const NjGeom& G, const NjNetDev& N, const float* params, int n, const double* x,
                              const double* grad_base, const double* e_base, float* el, float* j, float* q,
                              float* pair_out, cudaStream_t st)
{
  if (n <= 0) return cudaSuccess;
  const int smem = nj_smem_bytes(G, N, false);
  cudaError_t e = cudaFuncSetAttribute((const void*)k_nj_pairs_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const long long total = (long long)n * G.n_pairs;
  long long blocks = nj_grid((const void*)k_nj_pairs_fwd, smem);
  blocks = std::min(blocks, (total + kNjSuper - 1) / kNjSuper);
  k_nj_pairs_fwd<<<(int)blocks, kNjThreads, smem, st>>>(G, N, params, n, x, pair_out);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_nj_assemble<<<(n + 3) / 4, 128, 0, st>>>(G, n, x, grad_base, e_base, pair_out, el, j, q);
  return cudaGetLastError();
}

int nj_backward_max_blocks(const NjGeom& G, const NjNetDev& N)
{
  const int smem = nj_smem_bytes(G, N, true);
  if (cudaFuncSetAttribute((const void*)k_nj_pairs_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return -1;
  return nj_grid((const void*)k_nj_pairs_bwd, smem);
}

cudaError_t launch_nj_backward(const NjGeom& G, const NjNetDev& N, const float* params, int n, const double* x,
                               const float* q, const float* d_el, const float* d_j, float* grad, float* partials,
                               int max_blocks, cudaStream_t st)
{
  const int np = nj_n_params(N.F, N.C, kNjH);
  if (n <= 0) return cudaMemsetAsync(grad, 0, sizeof(float) * np, st);
  const int smem = nj_smem_bytes(G, N, true);
  cudaError_t e = cudaFuncSetAttribute((const void*)k_nj_pairs_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem);
  if (e != cudaSuccess) return e;
  const long long total = (long long)n * G.n_pairs;
  long long blocks = std::min((long long)max_blocks, (total + kNjSuper - 1) / kNjSuper);
  k_nj_pairs_bwd<<<(int)blocks, kNjThreads, smem, st>>>(G, N, params, n, x, q, d_el, d_j, partials);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_nj_grad_reduce<<<(np + 255) / 256, 256, 0, st>>>(partials, (int)blocks, np, grad);
  return cudaGetLastError();
}

}  // namespace lrdmc
