// Assembly of the Burton-Miller collocation operators L and R (paper Sec. 4, Eq. 6; the two
// combined matrices are built directly in one pass, Sec. 4.1).
//
//   L_ij = 1/2 d_ij - int_j [dG/dn_y + beta d2G/dn_x dn_y] dS_y
//   R_ij = -int_j [G + beta dG/dn_x] dS_y - (beta/2) d_ij,     G = e^{ikr}/(4 pi r), beta = i/k
//
// Four kernels:
//   k_geometry           per element: centroid (as a float hi/lo pair), normal, area, the 7
//                        quadrature points as offsets from the centroid with their weights, and
//                        the FP64 copies used by the near-pair kernels.
//   k_assemble_regular   every pair (i, j) that shares no vertex, in FP32: one thread per source
//                        column j holding that element's rule in registers, collocation rows
//                        staged through shared memory and read as broadcasts, coalesced row
//                        stores of L and R. Pairs that share a vertex are skipped.
//   k_assemble_adjacent  vertex-sharing pairs (j != i), 16 lanes per pair over the subdivided
//                        rule: d = x - y formed in float-float arithmetic (where it cancels)
//                        from per-pair FP64 differences, everything after it in FP32 with
//                        compensated sums.
//   k_assemble_self      the self pair, one warp per element: the vertices relative to the
//                        centroid in FP64, the edge geometry and the angular integrals in FP32
//                        with cancellation-free forms.
//
// With d = x - y, r = |d|, rho = k r, q = (d.n_x)(d.n_y)/r^2 the integrands reduce to
//   dG/dn_y + beta H = G/r^2 [ (d.n_y - b/k) + i (a/k - rho d.n_y) ],
//       a = (rho^2 - 3) q + n_x.n_y,   b = rho (3 q - n_x.n_y),
//   G + beta dG/dn_x = G [ 1 - d.n_x / r - i d.n_x / (k r^2) ].
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <array>
#include <cmath>
#include <cstdlib>
#include <vector>

#include "internal.h"
#include "pairs.cuh"

namespace natbem {

// ------------------------------------------------------------------------ rule tables
// 7-point degree-5 triangle rule (Radon 1948): centroid weight 9/40, then the orbits of
// (a, a, 1-2a) with a = (6 -+ sqrt 15)/21 and weights (155 -+ sqrt 15)/1200.
__constant__ double c_rule7[7][4];          // barycentric l0, l1, l2 and weight (sum 1)
constexpr int kMaxAdjPts = 7 * 64;          // 4^3 sub-triangles
constexpr int kMaxSelfPts = 64;
__device__ double4 g_adj_rule[kMaxAdjPts];  // parent barycentrics and weight (sum 1)
__device__ float4 g_adj_ab[kMaxAdjPts];     // barycentrics l1, l2 as FP32 (hi, lo) pairs
__device__ float g_adj_w[kMaxAdjPts];       // the weight in FP32
__device__ float2 g_glf[kMaxSelfPts];       // Gauss-Legendre nodes / weights on [-1, 1]
__constant__ int c_adj_npts;
__constant__ int c_self_pts;

namespace {

void rule7_host(double out[7][4]) {
  const double s = std::sqrt(15.0);
  const double a = (6.0 - s) / 21.0, wa = (155.0 - s) / 1200.0;
  const double b = (6.0 + s) / 21.0, wb = (155.0 + s) / 1200.0;
  const double t[7][4] = {{1.0 / 3, 1.0 / 3, 1.0 / 3, 9.0 / 40},
                          {a, a, 1 - 2 * a, wa},
                          {a, 1 - 2 * a, a, wa},
                          {1 - 2 * a, a, a, wa},
                          {b, b, 1 - 2 * b, wb},
                          {b, 1 - 2 * b, b, wb},
                          {1 - 2 * b, b, b, wb}};
  for (int i = 0; i < 7; ++i)
    for (int c = 0; c < 4; ++c) out[i][c] = t[i][c];
}

// The 4^levels congruent sub-triangles of the reference triangle, as barycentric corners.
void split(const double tri[3][3], int levels, std::vector<std::array<double, 9>>& out) {
  if (levels == 0) {
    std::array<double, 9> t;
    for (int v = 0; v < 3; ++v)
      for (int c = 0; c < 3; ++c) t[3 * v + c] = tri[v][c];
    out.push_back(t);
    return;
  }
  double m[3][3];  // midpoints of edges (0,1), (1,2), (2,0)
  for (int c = 0; c < 3; ++c) {
    m[0][c] = 0.5 * (tri[0][c] + tri[1][c]);
    m[1][c] = 0.5 * (tri[1][c] + tri[2][c]);
    m[2][c] = 0.5 * (tri[2][c] + tri[0][c]);
  }
  const double* corner[4][3] = {{tri[0], m[0], m[2]}, {m[0], tri[1], m[1]},
                                {m[2], m[1], tri[2]}, {m[0], m[1], m[2]}};
  for (int s = 0; s < 4; ++s) {
    double sub[3][3];
    for (int v = 0; v < 3; ++v)
      for (int c = 0; c < 3; ++c) sub[v][c] = corner[s][v][c];
    split(sub, levels - 1, out);
  }
}

void gauss_legendre_host(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  const double pi = 3.14159265358979323846;
  for (int i = 0; i < n; ++i) {
    double z = std::cos(pi * (i + 0.75) / (n + 0.5)), d = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int m = 2; m <= n; ++m) {
        double p2 = ((2 * m - 1) * z * p1 - (m - 1) * p0) / m;
        p0 = p1;
        p1 = p2;
      }
      if (n == 1) p0 = 1.0;
      d = n * (z * p1 - p0) / (z * z - 1.0);
      double step = p1 / d;
      z -= step;
      if (std::fabs(step) < 1e-16) break;
    }
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * d * d);
  }
}

}  // namespace

nat_bem_status upload_rules(int adj_levels, int self_pts) {
  double r7[7][4];
  rule7_host(r7);
  NB_TRY_CUDA(cudaMemcpyToSymbol(c_rule7, r7, sizeof(r7)));
  // vertex-sharing pairs: the 7-point rule on each of the 4^levels sub-triangles
  const double ref[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
  std::vector<std::array<double, 9>> subs;
  split(ref, adj_levels, subs);
  std::vector<double4> pts;
  const double wsub = 1.0 / (double)subs.size();
  for (const auto& t : subs)
    for (int q = 0; q < 7; ++q) {
      double l[3];
      for (int c = 0; c < 3; ++c) l[c] = r7[q][0] * t[c] + r7[q][1] * t[3 + c] + r7[q][2] * t[6 + c];
      pts.push_back(make_double4(l[0], l[1], l[2], r7[q][3] * wsub));
    }
  int np = (int)pts.size();
  NB_TRY_CUDA(cudaMemcpyToSymbol(g_adj_rule, pts.data(), np * sizeof(double4)));
  std::vector<float4> ab(np);
  std::vector<float> wf(np);
  for (int i = 0; i < np; ++i) {
    const float ah = (float)pts[i].y, bh = (float)pts[i].z;
    ab[i] = make_float4(ah, (float)(pts[i].y - (double)ah), bh, (float)(pts[i].z - (double)bh));
    wf[i] = (float)pts[i].w;
  }
  NB_TRY_CUDA(cudaMemcpyToSymbol(g_adj_ab, ab.data(), np * sizeof(float4)));
  NB_TRY_CUDA(cudaMemcpyToSymbol(g_adj_w, wf.data(), np * sizeof(float)));
  NB_TRY_CUDA(cudaMemcpyToSymbol(c_adj_npts, &np, sizeof(int)));
  std::vector<double> gx, gw;
  gauss_legendre_host(self_pts, gx, gw);
  std::vector<float2> glf(self_pts);
  for (int i = 0; i < self_pts; ++i) glf[i] = make_float2((float)gx[i], (float)gw[i]);
  NB_TRY_CUDA(cudaMemcpyToSymbol(g_glf, glf.data(), self_pts * sizeof(float2)));
  NB_TRY_CUDA(cudaMemcpyToSymbol(c_self_pts, &self_pts, sizeof(int)));
  return NAT_BEM_OK;
}

// ------------------------------------------------------------------------- geometry
__global__ void k_geometry(const double* __restrict__ V, const int32_t* __restrict__ T, int n,
                           float4* c_hi, float4* c_lo, float4* nrm, float4* qp, int4* vid, float4* group,
                           double* tri, double* cen, double* nrm64, double* area) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x, t = min(at, n - 1);
  int ia = T[3 * t], ib = T[3 * t + 1], ic = T[3 * t + 2];
  double a[3], b[3], c[3];
  for (int d = 0; d < 3; ++d) {
    a[d] = V[3 * ia + d];
    b[d] = V[3 * ib + d];
    c[d] = V[3 * ic + d];
  }
  double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
  double e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
  double cr[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                  e1[0] * e2[1] - e1[1] * e2[0]};
  double len = sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
  double A = 0.5 * len;
  double nn[3] = {cr[0] / len, cr[1] / len, cr[2] / len};
  double cc[3];
  for (int d = 0; d < 3; ++d) cc[d] = (a[d] + b[d] + c[d]) / 3.0;
  {
    // the warp's elements: the middle of their centroids' box, its half diagonal and sqrt(6) of the
    // largest offset of a first-orbit point, (1 - 3a) of a vertex's; FP32 rounds the centre and points
    const float kFirst = 1.f - 3.f * (float)c_rule7[1][0];
    float most = 0.f, half2 = 0.f, far = 0.f, mid[3];
    for (int d = 0; d < 3; ++d) {
      float l = (float)cc[d], h = l;
      for (int o = 16; o > 0; o >>= 1) {
        l = fminf(l, __shfl_xor_sync(0xffffffffu, l, o));
        h = fmaxf(h, __shfl_xor_sync(0xffffffffu, h, o));
      }
      mid[d] = 0.5f * l + 0.5f * h;
      half2 += 0.25f * (h - l) * (h - l);
      far = fmaxf(far, fmaxf(fabsf(l), fabsf(h)));
    }
    for (int v = 0; v < 3; ++v) {
      const double* x = v == 0 ? a : v == 1 ? b : c;
      float q2 = 0.f;
      for (int d = 0; d < 3; ++d) q2 += (float)((x[d] - cc[d]) * (x[d] - cc[d]));
      most = fmaxf(most, q2);
    }
    for (int o = 16; o > 0; o >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
    const float rad = 1.001f * (sqrtf(half2) + 2.45f * kFirst * sqrtf(most)) + 1e-6f * far;
    if ((threadIdx.x & 31) == 0 && at < n) group[at >> 5] = make_float4(mid[0], mid[1], mid[2], rad * rad);
  }
  if (at >= n) return;
  float hi[3], lo[3];
  for (int d = 0; d < 3; ++d) {
    hi[d] = (float)cc[d];
    lo[d] = (float)(cc[d] - (double)hi[d]);
  }
  c_hi[t] = make_float4(hi[0], hi[1], hi[2], (float)A);
  c_lo[t] = make_float4(lo[0], lo[1], lo[2], 0.f);
  nrm[t] = make_float4((float)nn[0], (float)nn[1], (float)nn[2], 0.f);
  vid[t] = make_int4(ia, ib, ic, 0);
  const double inv4pi = 0.25 / 3.14159265358979323846;
  for (int q = 0; q < 7; ++q) {
    double y[3];
    for (int d = 0; d < 3; ++d)
      y[d] = c_rule7[q][0] * a[d] + c_rule7[q][1] * b[d] + c_rule7[q][2] * c[d] - cc[d];
    qp[7 * t + q] = make_float4((float)y[0], (float)y[1], (float)y[2],
                                (float)(c_rule7[q][3] * A * inv4pi));
  }
  for (int d = 0; d < 3; ++d) {
    tri[9 * t + d] = a[d];
    tri[9 * t + 3 + d] = b[d];
    tri[9 * t + 6 + d] = c[d];
    cen[3 * t + d] = cc[d];
    nrm64[3 * t + d] = nn[d];
  }
  area[t] = A;
}

// -------------------------------------------------------------- regular pairs (FP32)
namespace {

__device__ __forceinline__ bool shares_vertex(int4 a, int4 b) {
  return a.x == b.x || a.x == b.y || a.x == b.z || a.y == b.x || a.y == b.y || a.y == b.z ||
         a.z == b.x || a.z == b.y || a.z == b.z;
}

// complex value as two bf16 (real in the low half), round to nearest even
__device__ __forceinline__ uint32_t pack_bf16(float re, float im) {
  __nv_bfloat162 v = __floats2bfloat162_rn(re, im);
  return *reinterpret_cast<uint32_t*>(&v);
}

constexpr int kRegThreads = 256;  // source columns per block
constexpr int kRowStage = 64;     // collocation rows staged in shared memory at a time

// Entries (L, R) of a pair with centroid difference D, normals nj (source) and ni (collocation
// point) and the source's points q: d is formed for every point by itself.
__device__ __forceinline__ float4 regular_entry(float Dx, float Dy, float Dz, float3 nj, float3 ni,
                                                const float4* q, float k, float kinv) {
  const float dny = Dx * nj.x + Dy * nj.y + Dz * nj.z;  // quadrature offsets lie in the plane
  const float Dni = Dx * ni.x + Dy * ni.y + Dz * ni.z;
  const float nxny = ni.x * nj.x + ni.y * nj.y + ni.z * nj.z;
  float Lr = 0.f, Li = 0.f, Rr = 0.f, Ri = 0.f;
#pragma unroll
  for (int p = 0; p < 7; ++p) {
    const float dx = Dx - q[p].x, dy = Dy - q[p].y, dz = Dz - q[p].z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    const float dnx = Dni - fmaf(q[p].x, ni.x, fmaf(q[p].y, ni.y, q[p].z * ni.z));
    const float rho = k * r;
    const float nq = rintf(rho * kInvTwoPi);
    float th = fmaf(-nq, kTwoPiHi, rho);
    th = fmaf(-nq, kTwoPiLo, th);
    float sn, cs;
    __sincosf(th, &sn, &cs);
    const float gw = rinv * q[p].w;  // w A / (4 pi r)
    const float Gr = cs * gw, Gi = sn * gw;
    const float rinv2 = rinv * rinv;
    const float qq = dnx * dny * rinv2;
    const float a = fmaf(fmaf(rho, rho, -3.0f), qq, nxny);
    const float b = rho * fmaf(3.0f, qq, -nxny);
    const float lr = fmaf(-b, kinv, dny);
    const float li = fmaf(a, kinv, -rho * dny);
    const float Hr = Gr * rinv2, Hi = Gi * rinv2;
    Lr = fmaf(Hr, lr, fmaf(-Hi, li, Lr));
    Li = fmaf(Hr, li, fmaf(Hi, lr, Li));
    const float t1 = fmaf(-dnx, rinv, 1.0f);
    const float t2 = -dnx * rinv2 * kinv;
    Rr = fmaf(Gr, t1, fmaf(-Gi, t2, Rr));
    Ri = fmaf(Gr, t2, fmaf(Gi, t1, Ri));
  }
  return make_float4(-Lr, -Li, -Rr, -Ri);
}

}  // namespace

__global__ void __launch_bounds__(kRegThreads)
k_assemble_regular(const float4* __restrict__ c_hi, const float4* __restrict__ c_lo,
                   const float4* __restrict__ nrm, const float4* __restrict__ qp,
                   const int4* __restrict__ vid, int n, int ld, int rows_per_block, float k,
                   float2* __restrict__ L, float2* __restrict__ R, uint32_t* __restrict__ Lb) {
  __shared__ float4 s_hi[kRowStage], s_lo[kRowStage], s_n[kRowStage];
  __shared__ int4 s_v[kRowStage];
  const int j = blockIdx.x * kRegThreads + threadIdx.x;
  const bool col_ok = j < n, col_pad = j >= n && j < ld;
  // the source element's rule stays in registers for the whole row range
  float3 chi = make_float3(0.f, 0.f, 0.f), clo = chi, nj = chi;
  float4 q[7];
  int4 vj = make_int4(-1, -1, -1, 0);
  if (col_ok) {
    float4 t = c_hi[j];
    chi = make_float3(t.x, t.y, t.z);
    t = c_lo[j];
    clo = make_float3(t.x, t.y, t.z);
    t = nrm[j];
    nj = make_float3(t.x, t.y, t.z);
#pragma unroll
    for (int p = 0; p < 7; ++p) q[p] = qp[7 * j + p];
    vj = vid[j];
  } else {
#pragma unroll
    for (int p = 0; p < 7; ++p) q[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float kinv = 1.0f / k;
  const int i_begin = blockIdx.y * rows_per_block;
  const int i_end = min(n, i_begin + rows_per_block);
  for (int ib = i_begin; ib < i_end; ib += kRowStage) {
    const int cnt = min(kRowStage, i_end - ib);
    __syncthreads();
    if (threadIdx.x < cnt) {
      int i = ib + threadIdx.x;
      s_hi[threadIdx.x] = c_hi[i];
      s_lo[threadIdx.x] = c_lo[i];
      s_n[threadIdx.x] = nrm[i];
      s_v[threadIdx.x] = vid[i];
    }
    __syncthreads();
    for (int t = 0; t < cnt; ++t) {
      const int i = ib + t;
      const size_t off = (size_t)i * ld + j;
      if (col_pad) {
        L[off] = make_float2(0.f, 0.f);
        R[off] = make_float2(0.f, 0.f);
        if (Lb) Lb[off] = 0u;
        continue;
      }
      if (!col_ok) continue;
      const int4 vi = s_v[t];
      if (shares_vertex(vi, vj)) continue;  // self and vertex-sharing pairs: FP64 kernel
      const float4 xh = s_hi[t], xl = s_lo[t], ni4 = s_n[t];
      // centroid difference from the hi/lo pairs: exact-ish even for close elements
      const float Dx = (xh.x - chi.x) + (xl.x - clo.x);
      const float Dy = (xh.y - chi.y) + (xl.y - clo.y);
      const float Dz = (xh.z - chi.z) + (xl.z - clo.z);
      const float4 e = regular_entry(Dx, Dy, Dz, nj, make_float3(ni4.x, ni4.y, ni4.z), q, k, kinv);
      __stcs(L + off, make_float2(e.x, e.y));
      __stcs(R + off, make_float2(e.z, e.w));
      if (Lb) __stcs(Lb + off, pack_bf16(e.x, e.y));
    }
  }
}

// ---------------------------------------------------- regular pairs, paired FP32 (f32x2)
// The entries of k_assemble_regular for two adjacent source columns per thread, one in each half of
// paired FP32 operations (pairs.cuh). Bound by the FMA pipe (72% busy, and a paired operation takes
// it for two cycles: pairing saves issue slots only), so the form is chosen for its operation
// count, 28 paired operations a point:
//   - the outer points are c + s v_m with three directions v_m, so |d|^2 = |D|^2 + s^2 |v_m|^2 -
//     2 s D.v_m and d.n_x = D.n_x - s v_m.n_x cost three operations a point, not ten. That |d|^2
//     cancels where d is small against s v_m (two sheets at 0.02 of an element's size: rows 3e-4
//     off; nearer it can be negative), so the rows within sqrt(6) of the largest |s v_m| of a
//     column's centroid, one or two a column, are marked and formed again by regular_entry (2 us at
//     10240 triangles and at 1280; out to three times, 9 and 4 us; as a branch inside the loop,
//     which it broke up, 100 and 14). At sqrt(6) both forms round |d|^2 at about 3 x 2^-24;
//   - with u = d.n_x, v = d.n_y, t = 1/r, N = n_x.n_y and e = 3 u v t^2 - N the integrands are
//     G t^2 [ (v - r e) + i (k v (u - r) - e/k) ] and G [ (1 - u t) - i u t^2 / k ];
//   - the phase is reduced by the centroid's whole turns for all seven points (float-float, the
//     product k r unrounded), and both cross products have accumulators of their own.
// 10240 triangles: 1.198 -> 1.046 ms (49 operations a point and roundings on the rsqrt unit before);
// the error against FP64 entries is the same at k = 1 and a quarter less at k = 20. Four blocks per
// SM: three (more loads in flight) 1.128 ms, five and six (spilled column data) 1.051 and 1.083 ms.
namespace {
constexpr int kX2Threads = 128;  // 256 source columns per block, two per thread

struct RegPair {  // of one collocation row and two source columns
  u64 v3, mkv, N, Nk;  // 3 D.n_y, -k D.n_y, n_x.n_y, n_x.n_y / k
  u64 v, turn, turn_lo;  // D.n_y, minus the whole turns as a float-float
};
struct RegSums {  // sums of L = (Lr - Lb, La) and R = (Ra - Rb, Ri)
  u64 Lr, La, Lb, Ra, Rb, Ri;
};

// One point: r from r2, nu = -d.n_x, weight w A / 4 pi.
__device__ __forceinline__ void reg_point(const RegPair& c, u64 k2, u64 kinv2, u64 t, u64 r, u64 nu, u64 w, RegSums& o) {
  const u64 th = add2(fma2(k2, r, c.turn), c.turn_lo);
  float tha, thb, sa, ca, sb, cb;
  upk(th, tha, thb);
  __sincosf(tha, &sa, &ca);
  __sincosf(thb, &sb, &cb);
  const u64 gw = mul2(t, w);
  const u64 Gr = mul2(pk(ca, cb), gw), Gi = mul2(pk(sa, sb), gw);
  const u64 t2 = mul2(t, t);
  const u64 g = mul2(nu, t2), gk = mul2(g, kinv2);  // -u t^2, -u t^2 / k
  const u64 me = fma2(g, c.v3, c.N);                // -e
  const u64 lr = fma2(r, me, c.v);
  const u64 li = fma2(c.mkv, add2(nu, r), fma2(gk, c.v3, c.Nk));
  const u64 Hr = mul2(Gr, t2), Hi = mul2(Gi, t2);
  o.Lr = fma2(Hr, lr, o.Lr);
  o.Lb = fma2(Hi, li, o.Lb);
  o.La = fma2(Hi, lr, fma2(Hr, li, o.La));
  const u64 t1 = fma2(nu, t, bc(1.f));
  o.Ra = fma2(Gr, t1, o.Ra);
  o.Rb = fma2(Gi, gk, o.Rb);
  o.Ri = fma2(Gi, t1, fma2(Gr, gk, o.Ri));
}
}  // namespace

__global__ void __launch_bounds__(kX2Threads, 4)
k_assemble_regular_x2(const float4* __restrict__ c_hi, const float4* __restrict__ c_lo,
                      const float4* __restrict__ nrm, const float4* __restrict__ qp,
                      const int4* __restrict__ vid, int n, int ld, int rows_per_block, float k,
                      float2* __restrict__ L, float2* __restrict__ R, uint32_t* __restrict__ Lb) {
  // row records with every value in both halves of a pair: centroid high, low, normal
  __shared__ __align__(16) u64 s_row[kRowStage][10];
  __shared__ int4 s_v[kRowStage];
  __shared__ int s_top;
  const int j0 = (blockIdx.x * kX2Threads + threadIdx.x) * 2;  // columns j0, j0 + 1
  const bool ok0 = j0 < n, ok1 = j0 + 1 < n;
  const bool pad0 = !ok0 && j0 < ld, pad1 = !ok1 && j0 + 1 < ld;
  // column records as pairs (column j0 in the low half, j0 + 1 in the high half); va, vb: the first
  // orbit's offsets towards vertices 2 and 1 (the third is -(va + vb)); sq: the first orbit's |offset|^2
  u64 chx, chy, chz, clx, cly, clz, njx, njy, njz, vax, vay, vaz, vbx, vby, vbz, sq[3], qw[3];
  float near2 = 0.f;  // 6 max |offset|^2 of the two columns
  int4 v0 = make_int4(-1, -1, -1, 0), v1 = v0;
  float grid;
  {
    const int ja = ok0 ? j0 : 0, jb = ok1 ? j0 + 1 : ja;
    const float4 a = c_hi[ja], b = c_hi[jb];
    // High parts of the centroids on one grid, a 2^22nd of the largest coordinate among the
    // block's columns: the difference to a row within twice that is then exact, and what D loses to
    // rounding is known (a row farther out: rounded once, at 2^-24 of the difference).
    if (threadIdx.x == 0) s_top = 0;
    __syncthreads();
    atomicMax(&s_top, __float_as_int(fminf(1e37f, fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fabsf(a.z)),
                                                        fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fabsf(b.z))))));
    __syncthreads();
    grid = 3.f * __int_as_float((s_top & 0x7f800000) + 0x00800000);
    const float4 al = c_lo[ja], bl = c_lo[jb];
    const u64 g2 = bc(grid), hx = pk(a.x, b.x), hy = pk(a.y, b.y), hz = pk(a.z, b.z);
    chx = sub2(add2(hx, g2), g2), chy = sub2(add2(hy, g2), g2), chz = sub2(add2(hz, g2), g2);
    clx = add2(sub2(hx, chx), pk(al.x, bl.x));
    cly = add2(sub2(hy, chy), pk(al.y, bl.y));
    clz = add2(sub2(hz, chz), pk(al.z, bl.z));
    const float4 an = nrm[ja], bn = nrm[jb];
    njx = pk(an.x, bn.x), njy = pk(an.y, bn.y), njz = pk(an.z, bn.z);
    qw[0] = pk(qp[7 * (size_t)ja].w, qp[7 * (size_t)jb].w);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const float4 qa = qp[7 * (size_t)ja + 1 + p], qb = qp[7 * (size_t)jb + 1 + p];
      const u64 x = pk(qa.x, qb.x), y = pk(qa.y, qb.y), z = pk(qa.z, qb.z);
      sq[p] = fma2(x, x, fma2(y, y, mul2(z, z)));
      float sa, sb;
      upk(sq[p], sa, sb);
      near2 = fmaxf(near2, 6.f * fmaxf(sa, sb));
      if (p == 0) vax = x, vay = y, vaz = z, qw[1] = pk(qa.w, qb.w);
      if (p == 1) vbx = x, vby = y, vbz = z, qw[2] = pk(qp[7 * (size_t)ja + 4].w, qp[7 * (size_t)jb + 4].w);
    }
    if (ok0) v0 = vid[j0];
    if (ok1) v1 = vid[j0 + 1];
  }
  const float kinv = 1.0f / k;
  const u64 k2 = bc(k), kinv2 = bc(kinv);
  const int i_begin = blockIdx.y * rows_per_block;
  const int i_end = min(n, i_begin + rows_per_block);
  for (int ib = i_begin; ib < i_end; ib += kRowStage) {
    const int cnt = min(kRowStage, i_end - ib);
    __syncthreads();
    if (threadIdx.x < cnt) {
      const int i = ib + threadIdx.x;
      const float4 h = c_hi[i], l = c_lo[i], m = nrm[i];
      u64* o = s_row[threadIdx.x];
      const float hx = (h.x + grid) - grid, hy = (h.y + grid) - grid, hz = (h.z + grid) - grid;
      o[0] = bc(hx), o[1] = bc(hy), o[2] = bc(hz);
      o[3] = bc((h.x - hx) + l.x), o[4] = bc((h.y - hy) + l.y), o[5] = bc((h.z - hz) + l.z);
      o[6] = bc(m.x), o[7] = bc(m.y), o[8] = bc(m.z);
      s_v[threadIdx.x] = vid[i];
    }
    __syncthreads();
    for (int tb = 0; tb < cnt; tb += 32) {
    unsigned close = 0u;  // rows tb + 0..31 whose entries are formed again
    for (int t = tb; t < min(cnt, tb + 32); ++t) {
      const int i = ib + t;
      const size_t off = (size_t)i * ld + j0;
      if (pad0 || pad1) {  // zero the padding columns (ld > n)
        if (pad0) {
          L[off] = make_float2(0.f, 0.f);
          R[off] = make_float2(0.f, 0.f);
          if (Lb) Lb[off] = 0u;
        }
        if (pad1) {
          L[off + 1] = make_float2(0.f, 0.f);
          R[off + 1] = make_float2(0.f, 0.f);
          if (Lb) Lb[off + 1] = 0u;
        }
      }
      if (!ok0) continue;
      const int4 vi = s_v[t];
      const bool w0 = !shares_vertex(vi, v0), w1 = ok1 && !shares_vertex(vi, v1);
      if (!w0 && !w1) continue;
      const u64* x = s_row[t];
      const u64 nix = x[6], niy = x[7], niz = x[8];
      const u64 ax = sub2(x[0], chx), bx = sub2(x[3], clx), Dx = add2(ax, bx);
      const u64 ay = sub2(x[1], chy), by = sub2(x[4], cly), Dy = add2(ay, by);
      const u64 az = sub2(x[2], chz), bz = sub2(x[5], clz), Dz = add2(az, bz);
      // |D|^2 is shared by the seven points, so its error does not average out over them: formed
      // from the exact a and the small b, a.a + b.(a + D), without the rounding of D
      const u64 D2 = fma2(ax, ax, fma2(ay, ay, fma2(az, az,
                     fma2(bx, add2(ax, Dx), fma2(by, add2(ay, Dy), mul2(bz, add2(az, Dz)))))));
      {
        float da, db;
        upk(D2, da, db);
        if ((w0 && da < near2) || (w1 && db < near2)) close |= 1u << (t & 31);
      }
      const u64 nu = sub2(bc(0.f), fma2(Dx, nix, fma2(Dy, niy, mul2(Dz, niz))));  // -D.n_x
      RegPair c;
      c.v = fma2(Dx, njx, fma2(Dy, njy, mul2(Dz, njz)));  // d.n_y of every point
      c.N = fma2(nix, njx, fma2(niy, njy, mul2(niz, njz)));
      c.Nk = mul2(c.N, kinv2);
      c.v3 = mul2(c.v, bc(3.f));
      c.mkv = mul2(c.v, bc(-k));
      RegSums o;
      o.Lr = o.La = o.Lb = o.Ra = o.Rb = o.Ri = bc(0.f);
      {
        const u64 ri = rsqrt2(D2), r = mul2(D2, ri), turns = turns2(mul2(k2, r));
        c.turn = mul2(turns, bc(-kTwoPiHi));
        c.turn_lo = fma2(turns, bc(-kTwoPiLo), fma2(turns, bc(-kTwoPiHi), mul2(turns, bc(kTwoPiHi))));
        reg_point(c, k2, kinv2, ri, r, nu, qw[0], o);
      }
      u64 dm[3], nm[3];  // D.v_m and v_m.n_x
      dm[0] = fma2(Dx, vax, fma2(Dy, vay, mul2(Dz, vaz)));
      dm[1] = fma2(Dx, vbx, fma2(Dy, vby, mul2(Dz, vbz)));
      dm[2] = add2(dm[0], dm[1]);
      nm[0] = fma2(nix, vax, fma2(niy, vay, mul2(niz, vaz)));
      nm[1] = fma2(nix, vbx, fma2(niy, vby, mul2(niz, vbz)));
      nm[2] = add2(nm[0], nm[1]);
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int ob = 0; ob < 2; ++ob) {
          const float sc = (ob == 0 ? 1.f : kOrbit), sgn = q == 2 ? -sc : sc;
          const u64 base = ob == 0 ? add2(D2, sq[q]) : fma2(bc(kOrbit * kOrbit), sq[q], D2);
          const u64 r2 = fma2(bc(-2.f * sgn), dm[q], base);
          const u64 ri = rsqrt2(r2);
          reg_point(c, k2, kinv2, ri, mul2(r2, ri), fma2(bc(sgn), nm[q], nu), qw[1 + ob], o);
        }
      float lr0, lr1, li0, li1, rr0, rr1, ri0, ri1;
      upk(sub2(o.Lb, o.Lr), lr0, lr1);  // the entries are minus the integrals
      upk(o.La, li0, li1);
      upk(sub2(o.Rb, o.Ra), rr0, rr1);
      upk(o.Ri, ri0, ri1);
      if (w0 && w1) {
        __stcs(reinterpret_cast<float4*>(L + off), make_float4(lr0, -li0, lr1, -li1));
        __stcs(reinterpret_cast<float4*>(R + off), make_float4(rr0, -ri0, rr1, -ri1));
        if (Lb) __stcs(reinterpret_cast<uint2*>(Lb + off), make_uint2(pack_bf16(lr0, -li0), pack_bf16(lr1, -li1)));
      } else {
        if (w0) {
          __stcs(L + off, make_float2(lr0, -li0));
          __stcs(R + off, make_float2(rr0, -ri0));
          if (Lb) __stcs(Lb + off, pack_bf16(lr0, -li0));
        }
        if (w1) {
          __stcs(L + off + 1, make_float2(lr1, -li1));
          __stcs(R + off + 1, make_float2(rr1, -ri1));
          if (Lb) __stcs(Lb + off + 1, pack_bf16(lr1, -li1));
        }
      }
    }
    for (; close; close &= close - 1u) {
      const int t = tb + __ffs(close) - 1;
      const u64* x = s_row[t];
      float D[3][2], nj[3][2], ni[3], u;
      upk(add2(sub2(x[0], chx), sub2(x[3], clx)), D[0][0], D[0][1]);
      upk(add2(sub2(x[1], chy), sub2(x[4], cly)), D[1][0], D[1][1]);
      upk(add2(sub2(x[2], chz), sub2(x[5], clz)), D[2][0], D[2][1]);
      upk(njx, nj[0][0], nj[0][1]);
      upk(njy, nj[1][0], nj[1][1]);
      upk(njz, nj[2][0], nj[2][1]);
#pragma unroll
      for (int d = 0; d < 3; ++d) upk(x[6 + d], ni[d], u);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!(h ? ok1 : ok0) || shares_vertex(s_v[t], h ? v1 : v0)) continue;
        if (!(D[0][h] * D[0][h] + D[1][h] * D[1][h] + D[2][h] * D[2][h] < near2)) continue;
        const float4 e = regular_entry(D[0][h], D[1][h], D[2][h], make_float3(nj[0][h], nj[1][h], nj[2][h]),
                                       make_float3(ni[0], ni[1], ni[2]), qp + 7 * (size_t)(j0 + h), k, kinv);
        const size_t off = (size_t)(ib + t) * ld + j0 + h;
        L[off] = make_float2(e.x, e.y);
        R[off] = make_float2(e.z, e.w);
        if (Lb) Lb[off] = pack_bf16(e.x, e.y);
      }
    }
    }
  }
}

// ------------------------------------------------------------- near pairs and self terms
namespace {

// Compensated FP32 running sum (Kahan 1965): s - c is the exact sum to about twice FP32 precision.
__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// Knuth's TwoSum: s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Sum over the 16 lanes of a half warp of the compensated sums (s, c), as a double-float
// (hi, lo); every lane of the warp must call it.
__device__ __forceinline__ void half_warp_sum_df(float s, float c, float& hi, float& lo) {
  two_sum(s, -c, hi, lo);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    float t, e;
    two_sum(hi, h2, t, e);
    e += lo + l2;
    hi = t + e;
    lo = e - (hi - t);
  }
}

}  // namespace

// D - (a e + b f) for float-float D, e, f and barycentrics a = (ab.x, ab.y), b = (ab.z, ab.w):
// error-free products and sums (Dekker, Knuth) in round-to-nearest FP32 intrinsics (never
// contracted), rounded to FP32 once at the end.
__device__ __forceinline__ float ff_offset(float Dh, float Dl, float4 ab, float eh, float el, float fh, float fl) {
  const float p = __fmul_rn(ab.x, eh);
  const float pe = __fmaf_rn(ab.x, el, __fmaf_rn(ab.y, eh, __fmaf_rn(ab.x, eh, -p)));
  const float q = __fmul_rn(ab.z, fh);
  const float qe = __fmaf_rn(ab.z, fl, __fmaf_rn(ab.w, fh, __fmaf_rn(ab.z, fh, -q)));
  const float s = __fadd_rn(p, q);
  const float sb = __fsub_rn(s, p);
  const float se = __fadd_rn(__fadd_rn(__fsub_rn(p, __fsub_rn(s, sb)), __fsub_rn(q, sb)), __fadd_rn(pe, qe));
  const float d = __fsub_rn(Dh, s);
  const float db = __fsub_rn(d, Dh);
  const float de = __fadd_rn(__fsub_rn(Dh, __fsub_rn(d, db)), __fsub_rn(-s, db));
  return __fadd_rn(d, __fadd_rn(de, __fsub_rn(Dl, se)));
}

// Vertex-sharing pairs (i, j != i): the 7-point rule on the 4^levels sub-triangles of element j,
// 16 lanes per pair (two pairs per warp; 112 points at levels = 2 is seven per lane). The
// quadrature point and x_i are close compared with their distance from the origin, so
// d = x_i - y is formed from x_i - v0 and the edges of j (taken in FP64 from the FP64 vertices,
// once per pair) in float-float arithmetic (ff_offset, about 48 bits); d is then exact to FP32
// rounding. The normal components d.n_i and d.n_j come from per-pair FP64 dot products (they
// cancel for nearly coplanar neighbours). Everything after that (r, the phase, G and the
// hypersingular combination) runs on the FP32 pipe, which GB300 issues ~60x faster than FP64.
// Per-lane sums are compensated (Kahan) and the 16 lanes are added as double-float.
__global__ void __launch_bounds__(256)
k_assemble_adjacent(const int2* __restrict__ pairs, int64_t n_pairs, const double* __restrict__ tri,
                    const double* __restrict__ cen, const double* __restrict__ nrm64,
                    const double* __restrict__ area, int ld, float kf, float kinvf, float2* __restrict__ L,
                    float2* __restrict__ R, uint32_t* __restrict__ Lb) {
  const int64_t pr_idx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  const int l16 = threadIdx.x & 15;
  const bool valid = pr_idx < n_pairs;  // no early exit: the lane sums use full-warp shuffles
  int i = 0, j = 0;
  if (valid) {
    const int2 pr = pairs[pr_idx];
    i = pr.x;
    j = pr.y;
  }
  const double* t = tri + 9 * j;
  // D = x_i - v0 and the edges e1 = v1 - v0, e2 = v2 - v0 of triangle j as float-float pairs:
  // d = D - (l1 e1 + l2 e2) then keeps about 48 bits on the FP32 pipe (GB300's FP64 rate is
  // about 1/76 of its FP32 rate; this kernel was FP64-pipe-bound). The FP64 prologue is dealt
  // over the pair's 16 lanes (lane c < 9: component c % 3 of D, e1 or e2; lanes 9-14: the two
  // normals; lane 15: the area factor) and broadcast by shuffles.
  float vh = 0.f, vl = 0.f;
  double pi = 0.0, pj = 0.0;  // lanes 0..8: component c of D, e1 or e2 times n_i,c and n_j,c
  if (l16 < 9) {
    const int w = l16 / 3, c = l16 % 3;
    const double v = (w == 0 ? cen[3 * i + c] : t[3 * w + c]) - t[c];
    vh = (float)v;
    vl = (float)(v - (double)vh);
    pi = v * nrm64[3 * i + c];
    pj = v * nrm64[3 * j + c];
  } else if (l16 < 12) {
    vh = (float)nrm64[3 * i + (l16 - 9)];
  } else if (l16 < 15) {
    vh = (float)nrm64[3 * j + (l16 - 12)];
  } else {
    vh = (float)(area[j] * (0.25 / 3.14159265358979323846));
  }
  float Dh[3], Dl[3], e1h[3], e1l[3], e2h[3], e2l[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Dh[c] = __shfl_sync(0xffffffffu, vh, c, 16);
    Dl[c] = __shfl_sync(0xffffffffu, vl, c, 16);
    e1h[c] = __shfl_sync(0xffffffffu, vh, 3 + c, 16);
    e1l[c] = __shfl_sync(0xffffffffu, vl, 3 + c, 16);
    e2h[c] = __shfl_sync(0xffffffffu, vh, 6 + c, 16);
    e2l[c] = __shfl_sync(0xffffffffu, vl, 6 + c, 16);
  }
  const float ni0 = __shfl_sync(0xffffffffu, vh, 9, 16), ni1 = __shfl_sync(0xffffffffu, vh, 10, 16),
              ni2 = __shfl_sync(0xffffffffu, vh, 11, 16);
  const float nj0 = __shfl_sync(0xffffffffu, vh, 12, 16), nj1 = __shfl_sync(0xffffffffu, vh, 13, 16),
              nj2 = __shfl_sync(0xffffffffu, vh, 14, 16);
  const float scale = __shfl_sync(0xffffffffu, vh, 15, 16);
  // d.n_i and d.n_j are O(theta |d|) for nearly coplanar neighbours (theta the angle between
  // them): as FP32 dot products with FP32-rounded normals they carry an absolute error of about
  // 6e-8 |d|, which at low k (beta = i/k weights d.n_i in R) reached 2e-6 of an entry. So the
  // pair's D.n_i, e1.n_i, e2.n_i and D.n_j are FP64 dot products with the FP64 normals (summed
  // over the three lanes of each vector), and per point d.n_i = D.n_i - a e1.n_i - b e2.n_i has
  // no cancellation; d.n_j = D.n_j on the whole flat element j (its edges are normal to n_j).
  const int g3 = (l16 / 3) * 3;  // first lane of this lane's vector (lanes 9..15: unused values)
  const double si = __shfl_sync(0xffffffffu, pi, g3, 16) + __shfl_sync(0xffffffffu, pi, g3 + 1, 16) +
                    __shfl_sync(0xffffffffu, pi, g3 + 2, 16);
  const double sj = __shfl_sync(0xffffffffu, pj, g3, 16) + __shfl_sync(0xffffffffu, pj, g3 + 1, 16) +
                    __shfl_sync(0xffffffffu, pj, g3 + 2, 16);
  const float fi = (float)si, fj = (float)sj;
  const float Dni = __shfl_sync(0xffffffffu, fi, 0, 16), E1i = __shfl_sync(0xffffffffu, fi, 3, 16),
              E2i = __shfl_sync(0xffffffffu, fi, 6, 16);
  const float dny = __shfl_sync(0xffffffffu, fj, 0, 16);
  const float nxny = ni0 * nj0 + ni1 * nj1 + ni2 * nj2;
  float Lr = 0.f, Li = 0.f, Rr = 0.f, Ri = 0.f, cLr = 0.f, cLi = 0.f, cRr = 0.f, cRi = 0.f;
  const int np = valid ? c_adj_npts : 0;
  for (int p = l16; p < np; p += 16) {
    const float4 ab = g_adj_ab[p];
    const float d0 = ff_offset(Dh[0], Dl[0], ab, e1h[0], e1l[0], e2h[0], e2l[0]);
    const float d1 = ff_offset(Dh[1], Dl[1], ab, e1h[1], e1l[1], e2h[1], e2l[1]);
    const float d2 = ff_offset(Dh[2], Dl[2], ab, e1h[2], e1l[2], e2h[2], e2l[2]);
    const float r2 = fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
    const float rinv = rsqrtf(r2);
    const float r = r2 * rinv;
    const float dnx = fmaf(-ab.x, E1i, fmaf(-ab.z, E2i, Dni));
    const float rho = kf * r;
    const float nq = rintf(rho * kInvTwoPi);
    const float th = fmaf(-nq, kTwoPiLo, fmaf(-nq, kTwoPiHi, rho));
    float sn, cs;
    sincosf(th, &sn, &cs);
    const float gw = g_adj_w[p] * scale * rinv;
    const float Gr = cs * gw, Gi = sn * gw;
    const float rinv2 = rinv * rinv;
    const float qq = dnx * dny * rinv2;
    const float a = fmaf(fmaf(rho, rho, -3.0f), qq, nxny);
    const float b = rho * fmaf(3.0f, qq, -nxny);
    const float lr = fmaf(-b, kinvf, dny), li = fmaf(a, kinvf, -rho * dny);
    const float Hr = Gr * rinv2, Hi = Gi * rinv2;
    const float t1 = fmaf(-dnx, rinv, 1.0f), t2 = -dnx * rinv2 * kinvf;
    kahan_add(Lr, cLr, fmaf(Hr, lr, -Hi * li));
    kahan_add(Li, cLi, fmaf(Hr, li, Hi * lr));
    kahan_add(Rr, cRr, fmaf(Gr, t1, -Gi * t2));
    kahan_add(Ri, cRi, fmaf(Gr, t2, Gi * t1));
  }
  float hLr, lLr, hLi, lLi, hRr, lRr, hRi, lRi;
  half_warp_sum_df(Lr, cLr, hLr, lLr);
  half_warp_sum_df(Li, cLi, hLi, lLi);
  half_warp_sum_df(Rr, cRr, hRr, lRr);
  half_warp_sum_df(Ri, cRi, hRi, lRi);
  if (valid && l16 == 0) {
    const float2 lv = make_float2(-(hLr + lLr), -(hLi + lLi));
    const float2 rv = make_float2(-(hRr + lRr), -(hRi + lRi));
    L[(size_t)i * ld + j] = lv;
    R[(size_t)i * ld + j] = rv;
    if (Lb) Lb[(size_t)i * ld + j] = pack_bf16(lv.x, lv.y);
  }
}

// Self terms (flat element, collocation at the centroid), one warp per element (the vertices
// relative to the centroid in FP64, everything after them in FP32):
//   S = (1/4pi) sum_e int (e^{ikR} - 1)/(ik) dpsi,   FP = (1/4pi) sum_e int (ik - e^{ikR}/R) dpsi,
// with R = d_e / cos(psi) the distance from the centroid to edge e along the ray (radial part
// analytic, Hadamard finite part of the hypersingular term); L_ii = 1/2 - beta FP and
// R_ii = -S - beta/2 with beta = i/k.
__global__ void __launch_bounds__(256)
k_assemble_self(int n, const double* __restrict__ tri, const double* __restrict__ cen, int ld,
                float kf, float kinvf, float2* __restrict__ L, float2* __restrict__ R, uint32_t* __restrict__ Lb) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;  // whole warps
  const float inv4pi = (float)(0.25 / 3.14159265358979323846);
  const double* t = tri + 9 * i;
  const int ns = c_self_pts;
  // per edge e (lanes 0..2): the distance d_e from the centroid to the edge line and the
  // angles of the edge's end points seen from the centroid, measured from the perpendicular.
  // The end points relative to the centroid are formed in FP64 (the coordinates are far larger
  // than the element) and the rest in FP32 on those element-sized vectors.
  float de = 0.f, mid = 0.f, half = 0.f;
  if (lane < 3) {
    const double* P = t + 3 * lane;
    const double* Q = t + 3 * ((lane + 1) % 3);
    float p[3], q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double xc = cen[3 * i + c];
      p[c] = (float)(P[c] - xc);
      q[c] = (float)(Q[c] - xc);
    }
    float u0 = q[0] - p[0], u1 = q[1] - p[1], u2 = q[2] - p[2];
    const float ul = rsqrtf(fmaf(u0, u0, fmaf(u1, u1, u2 * u2)));
    u0 *= ul;
    u1 *= ul;
    u2 *= ul;
    // positions of P and Q along the edge line, relative to the foot of the perpendicular
    const float sP = fmaf(p[0], u0, fmaf(p[1], u1, p[2] * u2));
    const float sQ = fmaf(q[0], u0, fmaf(q[1], u1, q[2] * u2));
    const float f0 = fmaf(-sP, u0, p[0]), f1 = fmaf(-sP, u1, p[1]), f2 = fmaf(-sP, u2, p[2]);
    de = sqrtf(fmaf(f0, f0, fmaf(f1, f1, f2 * f2)));
    const float psiP = atan2f(sP, de), psiQ = atan2f(sQ, de);
    half = 0.5f * (psiQ - psiP);
    mid = 0.5f * (psiQ + psiP);
  }
  float dEf[3], mEf[3], hEf[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    dEf[e] = __shfl_sync(0xffffffffu, de, e);
    mEf[e] = __shfl_sync(0xffffffffu, mid, e);
    hEf[e] = __shfl_sync(0xffffffffu, half, e);
  }
  // The angular points in FP32 (GB300's FP64 rate is about 1/76 of its FP32 rate), with
  // cancellation-free forms: with x = kR and h = x/2, (e^{ikR} - 1)/(ik) = (sin x + 2i sin^2 h)/k,
  // cos x = cos^2 h - sin^2 h, and k - sin(kR)/R = k (1 - sinc x) from its Taylor series
  // sum_{n>=1} (-1)^(n+1) x^(2n) / (2n+1)! below x = 1.5 (six terms: below 2e-8 of the value)
  // and 1 - sin(x)/x above (where 1 - sinc x >= 0.33).
  float Sre = 0.f, Sim = 0.f, Fre = 0.f, Fim = 0.f;
  for (int p = lane; p < 3 * ns; p += 32) {
    const int e = p / ns, g = p - e * ns;
    const float dE = e == 0 ? dEf[0] : (e == 1 ? dEf[1] : dEf[2]);
    const float mE = e == 0 ? mEf[0] : (e == 1 ? mEf[1] : mEf[2]);
    const float hE = e == 0 ? hEf[0] : (e == 1 ? hEf[1] : hEf[2]);
    const float2 gl = g_glf[g];
    const float psi = fmaf(hE, gl.x, mE);
    const float cpsi = cosf(psi);
    const float Rr = dE / cpsi;
    const float invR = cpsi / dE;
    const float wq = hE * gl.y;
    const float x = kf * Rr;
    float s2, c2;
    sincosf(0.5f * x, &s2, &c2);
    const float sn = 2.0f * s2 * c2, omc = 2.0f * s2 * s2, cs = (c2 - s2) * (c2 + s2);
    float omsinc;  // 1 - sin(x)/x
    if (x < 1.5f) {
      const float x2 = x * x;
      omsinc = x2 * (1.0f / 6.0f -
                     x2 * (1.0f / 120.0f -
                           x2 * (1.0f / 5040.0f -
                                 x2 * (1.0f / 362880.0f - x2 * (1.0f / 39916800.0f - x2 * (1.0f / 6227020800.0f))))));
    } else {
      omsinc = 1.0f - sn / x;
    }
    Sre = fmaf(wq, sn * kinvf, Sre);
    Sim = fmaf(wq, omc * kinvf, Sim);
    Fre = fmaf(-wq, cs * invR, Fre);
    Fim = fmaf(wq, kf * omsinc, Fim);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Sre += __shfl_xor_sync(0xffffffffu, Sre, o);
    Sim += __shfl_xor_sync(0xffffffffu, Sim, o);
    Fre += __shfl_xor_sync(0xffffffffu, Fre, o);
    Fim += __shfl_xor_sync(0xffffffffu, Fim, o);
  }
  Sre *= inv4pi;
  Sim *= inv4pi;
  Fre *= inv4pi;
  Fim *= inv4pi;
  if (lane == 0) {
    const float2 lv = make_float2(fmaf(Fim, kinvf, 0.5f), -Fre * kinvf);
    L[(size_t)i * ld + i] = lv;
    R[(size_t)i * ld + i] = make_float2(-Sre, fmaf(-0.5f, kinvf, -Sim));
    if (Lb) Lb[(size_t)i * ld + i] = pack_bf16(lv.x, lv.y);
  }
}

// ----------------------------------------------------------------------- drivers
nat_bem_status geometry_build(nat_bem_op* op, const double* dV, const int32_t* dT, int64_t nv,
                              const std::vector<int2>& near_pairs, cudaStream_t s) {
  Geometry& g = op->geo;
  const int64_t n = g.n;  // elements
  (void)nv;
  NB_TRY(dev_alloc_n(&g.c_hi, n, s));
  NB_TRY(dev_alloc_n(&g.c_lo, n, s));
  NB_TRY(dev_alloc_n(&g.nrm, n, s));
  NB_TRY(dev_alloc_n(&g.qp, 7 * n, s));
  NB_TRY(dev_alloc_n(&g.vid, n, s));
  NB_TRY(dev_alloc_n(&g.group, (n + 31) / 32, s));
  NB_TRY(dev_alloc_n(&g.tri, 9 * n, s));
  NB_TRY(dev_alloc_n(&g.cen, 3 * n, s));
  NB_TRY(dev_alloc_n(&g.nrm64, 3 * n, s));
  NB_TRY(dev_alloc_n(&g.area, n, s));
  g.n_near = (int64_t)near_pairs.size();
  NB_TRY(dev_alloc_n(&g.near_pairs, g.n_near, s));
  NB_TRY_CUDA(cudaMemcpyAsync(g.near_pairs, near_pairs.data(), g.n_near * sizeof(int2),
                              cudaMemcpyHostToDevice, s));
  const int threads = 128;
  NB_LAUNCH("geometry", s, k_geometry<<<(unsigned)((n + threads - 1) / threads), threads, 0, s>>>(
      dV, dT, (int)n, g.c_hi, g.c_lo, g.nrm, g.qp, g.vid, g.group, g.tri, g.cen, g.nrm64, g.area));
  NB_CHECK_LAUNCH();
  return NAT_BEM_OK;
}

nat_bem_status assemble_operators(nat_bem_op* op, cudaStream_t s) {
  const Geometry& g = op->geo;
  const int n = (int)op->n, ld = (int)g.ld;
  // The near pairs write exactly the entries the regular kernel skips. The three kernels run in
  // order on the solve's stream: beside the FP32 regular kernel on a second stream the FP64
  // kernels saved ~0.3 ms per solve with one solve in flight and nothing with several, and
  // they slowed the regular kernel they shared the SMs with.
  {
    const int64_t threads = 256;
    const int64_t adj_blocks = (g.n_near * 16 + threads - 1) / threads;
    if (adj_blocks > 0)
      NB_LAUNCH("assemble_near", s, k_assemble_adjacent<<<(unsigned)adj_blocks, (unsigned)threads, 0, s>>>(
          g.near_pairs, g.n_near, g.tri, g.cen, g.nrm64, g.area, ld, (float)op->k, (float)(1.0 / op->k), op->L,
          op->R, bf16_target(op)));
    const int64_t self_blocks = ((int64_t)n * 32 + threads - 1) / threads;
    NB_LAUNCH("assemble_self", s, k_assemble_self<<<(unsigned)self_blocks, (unsigned)threads, 0, s>>>(
        n, g.tri, g.cen, ld, (float)op->k, (float)(1.0 / op->k), op->L, op->R, bf16_target(op)));
    NB_CHECK_LAUNCH();
  }
  // regular pairs: columns in blocks of 256 (two columns a thread in the paired form), rows
  // split in blocks of rows_per_block. Every entry is computed the same way whatever the split,
  // so the autotuner (rows per block 64, 32, 128 or 16, per size class) changes no result.
  const int col_blocks = (ld + kRegThreads - 1) / kRegThreads;
  static const bool scalar = std::getenv("NATBEM_ASSEMBLY_SCALAR") != nullptr;
  auto launch = [&](int rows_per_block) -> nat_bem_status {
    const int row_blocks = (n + rows_per_block - 1) / rows_per_block;
    dim3 grid(col_blocks, row_blocks);
    if (scalar)
      NB_LAUNCH("assemble_regular", s, k_assemble_regular<<<grid, kRegThreads, 0, s>>>(
          g.c_hi, g.c_lo, g.nrm, g.qp, g.vid, n, ld, rows_per_block, (float)op->k, op->L, op->R, bf16_target(op)));
    else
      NB_LAUNCH("assemble_regular", s, k_assemble_regular_x2<<<grid, kX2Threads, 0, s>>>(
          g.c_hi, g.c_lo, g.nrm, g.qp, g.vid, n, ld, rows_per_block, (float)op->k, op->L, op->R, bf16_target(op)));
    NB_CHECK_LAUNCH();
    return NAT_BEM_OK;
  };
  static const int kRows[4] = {64, 32, 128, 16};
  const int pick = autotune("assemble_rows", (n + 1023) / 1024, 4, [&](int c) { return launch(kRows[c]); }, s);
  NB_TRY(launch(kRows[pick]));
  return finish_low_copy(op, s);
}

// The row-scaled FP16 copy of L: one block per row finds the row's largest real or imaginary
// magnitude m = f 2^E (f in [0.5, 1)), takes s = 2^(15 - E) so that the scaled entries stay
// below 2^15 (FP16's largest finite value is 65504) and keep FP16's full 11 significant bits
// down to 2^-29 of m, writes half2(L_ij s) rounded to nearest, and 1/s (exact) as the row scale.
__global__ void __launch_bounds__(256) k_copy_fp16_rows(const float2* __restrict__ L, int ld,
                                                        uint32_t* __restrict__ Lh, float* __restrict__ row_scale) {
  __shared__ float red[8];
  const size_t row = blockIdx.x;
  const float2* src = L + row * ld;
  float m = 0.f;
  for (int j = threadIdx.x; j < ld; j += 256) {
    const float2 v = src[j];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) m = fmaxf(m, red[w]);
  int e = 0;
  if (m > 0.f) frexpf(m, &e);
  const float scale = m > 0.f ? ldexpf(1.0f, 15 - e) : 1.0f;
  for (int j = threadIdx.x; j < ld; j += 256) {
    const float2 v = src[j];
    __half2 h = __floats2half2_rn(v.x * scale, v.y * scale);
    Lh[row * ld + j] = *reinterpret_cast<uint32_t*>(&h);
  }
  if (threadIdx.x == 0) row_scale[row] = m > 0.f ? ldexpf(1.0f, e - 15) : 1.0f;
}

nat_bem_status finish_low_copy(nat_bem_op* op, cudaStream_t s) {
  op->split_of = -1;  // L and R changed: a three-way split is rebuilt before the next use
  if (!op->copy_fp16 || !op->Lb) return NAT_BEM_OK;
  NB_LAUNCH("copy_fp16", s, k_copy_fp16_rows<<<(unsigned)op->n, 256, 0, s>>>(op->L, (int)op->geo.ld, op->Lb,
                                                                              op->row_scale));
  NB_CHECK_LAUNCH();
  return NAT_BEM_OK;
}

}  // namespace natbem
