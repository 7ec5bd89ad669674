// Galerkin form of the Burton-Miller equation (paper Sec. 4, Eq. 6 tested with P1 hat functions;
// the element-to-element integration of Sec. 4.1): P1 Dirichlet data at the vertices, P0
// Neumann data per triangle,
//
//   L p = R g,  L = 1/2 M11 - K - beta H,  R = -V - beta K' - (beta/2) M10,
//   H_ij = int int G [k^2 (n_x . n_y) phi_j psi_i - curl phi_j . curl psi_i]   (Maue's form).
//
// Every entry is a sum over element pairs (tau test, sigma trial). The kernels compute, per
// pair, the 3 x 3 block of L and the 3 entries of R that the pair contributes (k_gal_regular for
// pairs sharing no vertex, 7 x 7 points; k_gal_singular for pairs sharing a vertex, an edge, or
// identical, a warp each over 4^4 Gauss points per region of the transformed 4-cube), into
// scratch arrays of pair blocks. The gathers then sum, for every vertex i and column (vertex j,
// or triangle s), the blocks of the triangles around i (and around j) in a fixed order, so the
// result does not depend on scheduling: k_gal_rowsum_L first sums each test triangle's row over
// the triangles around every column vertex (reading each pair block once; from planes over the
// trial triangle 338 us at 5120 triangles, from 72-byte blocks 556), k_gal_gather_L and
// k_gal_gather_R then sum over the triangles around each row vertex. FP32 arithmetic throughout: near the
// singularity x - y is formed from the transformed coordinates (a radius times a bounded
// vector), and for regular pairs from the centroid difference (hi/lo pairs) plus the points'
// offsets, so no cancellation occurs.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "internal.h"
#include "pairs.cuh"

namespace natbem {

namespace {
constexpr int kGalSing = 4;          // Gauss-Legendre points per dimension on singular pairs
constexpr int kGalVals = 12;         // per pair: L block (a, b) at 3a + b, then R entries (a)
constexpr double kGalScratch = 4e9;  // bytes of pair blocks per round of test triangles
constexpr float kInv4Pi = 0.0795774715459476679f;
constexpr float kFourPi = 12.5663706143591730f;

__constant__ float c_gal_b7[7][4];           // barycentric l0, l1, l2 and weight (sum 1)
__constant__ float c_gal_gl[kGalSing][2];    // Gauss-Legendre nodes and weights on [0, 1]

__device__ __forceinline__ uint32_t gal_pack_bf16(float re, float im) {
  __nv_bfloat162 v = __floats2bfloat162_rn(re, im);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Per-pair sums over x in tau, y in sigma, d = x - y, with F = G (1 - i k r) / r^2:
// gb[a][b] = sum w lam_a mu_b G, ky[a][b] = sum w lam_a mu_b F d.n_sigma, kx[a][b] = sum w lam_a mu_b F d.n_tau
// (complex, interleaved). dG/dn_y = F d.n_sigma and dG/dn_x = -F d.n_tau, and with the roles
// swapped d changes sign: the three sums give the blocks of both (tau, sigma) and (sigma, tau).
struct GalAcc {
  float gb[18], ky[18], kx[18];
};

__device__ __forceinline__ void gal_acc_zero(GalAcc& A) {
#pragma unroll
  for (int i = 0; i < 18; ++i) A.gb[i] = A.ky[i] = A.kx[i] = 0.f;
}

// w G and w F (w includes 1 / (4 pi)); turns: the phase's nearest number of turns, or a
// nearby point's.
__device__ __forceinline__ void gal_kernels(float rinv, float rho, float turns, float w, float2& G, float2& F) {
  float th = fmaf(-turns, kTwoPiHi, rho);
  th = fmaf(-turns, kTwoPiLo, th);
  float sn, cs;
  __sincosf(th, &sn, &cs);
  const float gw = rinv * w;
  G.x = cs * gw;
  G.y = sn * gw;
  const float r2inv = rinv * rinv;
  F.x = fmaf(rho, G.y, G.x) * r2inv;
  F.y = fmaf(-rho, G.x, G.y) * r2inv;
}
__device__ __forceinline__ float gal_turns(float rho) { return fmaf(rho, kInvTwoPi, kRound) - kRound; }

// The 12 values of (tau, sigma), or with kSwap of (sigma, tau): L block -Kb - beta H and R entries
// -Vb - beta Kp (beta = i / k), with H = k^2 (n_t . n_s) Gb - (curl_a^t . curl_b^s) G0,
// Vb[a] = sum_b Gb[a][b], G0 = sum Gb, Kp[a] the sum of dG/dn_x over the trial triangle.
template <bool kSwap>
__device__ __forceinline__ void gal_finish(const GalAcc& A, float k, float nn, const float (&cc)[9],
                                           float2 (&out)[kGalVals]) {
  const float kinv = 1.f / k, k2nn = k * k * nn;
  float g0r = 0.f, g0i = 0.f;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    g0r += A.gb[2 * i];
    g0i += A.gb[2 * i + 1];
  }
  const float* kb = kSwap ? A.kx : A.ky;  // dG/dn_y, up to the sign of d
  const float* kp = kSwap ? A.ky : A.kx;  // -dG/dn_x, likewise
  const float sg = kSwap ? -1.f : 1.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float vr = 0.f, vi = 0.f, pr = 0.f, pi = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int i = kSwap ? 3 * b + a : 3 * a + b;
      const float hr = k2nn * A.gb[2 * i] - cc[i] * g0r;
      const float hi = k2nn * A.gb[2 * i + 1] - cc[i] * g0i;
      // -Kb - (i/k) H = (-Kb_r + H_i / k, -Kb_i - H_r / k)
      out[3 * a + b] = make_float2(-sg * kb[2 * i] + hi * kinv, -sg * kb[2 * i + 1] - hr * kinv);
      vr += A.gb[2 * i];
      vi += A.gb[2 * i + 1];
      pr -= sg * kp[2 * i];
      pi -= sg * kp[2 * i + 1];
    }
    out[9 + a] = make_float2(-vr + pi * kinv, -vi - pr * kinv);
  }
}

// Pair blocks of a round: value i of pair (t, s), i < 9 the L block at 3a + b, then the R entries,
// in planes over s: partL[((t - t0) 9 + i) nt + s], partR[((t - t0) 3 + a) nt + s].
__device__ __forceinline__ float2* gal_plane(float2* partL, float2* partR, int nt, int tr, int i) {
  return i < 9 ? partL + ((size_t)tr * 9 + i) * nt : partR + ((size_t)tr * 3 + i - 9) * nt;
}
__device__ __forceinline__ void gal_store(float2* partL, float2* partR, int nt, int tr, int s,
                                          const float2 (&v)[kGalVals]) {
#pragma unroll
  for (int i = 0; i < kGalVals; ++i) gal_plane(partL, partR, nt, tr, i)[s] = v[i];
}
constexpr int kGalT = 8;  // test triangles of a block of k_gal_regular (a warp each)
}  // namespace

// Per element: the three P1 curls (P_{a+1} - P_{a+2}) / (2A); per quadrature point (7 per
// element): a point record for the field kernels (position hi/lo, normal, weight w A / (4 pi)).
__global__ void k_gal_geometry(const double* __restrict__ tri, const double* __restrict__ nrm64,
                               const double* __restrict__ area, int nt, float4* __restrict__ curl,
                               float4* __restrict__ p_hi, float4* __restrict__ p_lo, float4* __restrict__ p_n,
                               float4* __restrict__ p_q) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double* P = tri + 9 * (size_t)t;
  const double A = area[t];
  for (int a = 0; a < 3; ++a) {
    const double* p1 = P + 3 * ((a + 1) % 3);
    const double* p2 = P + 3 * ((a + 2) % 3);
    curl[3 * (size_t)t + a] = make_float4((float)((p1[0] - p2[0]) / (2 * A)), (float)((p1[1] - p2[1]) / (2 * A)),
                                          (float)((p1[2] - p2[2]) / (2 * A)), 0.f);
  }
  for (int q = 0; q < 7; ++q) {
    float hi[3], lo[3];
    for (int d = 0; d < 3; ++d) {
      const double y = (double)c_gal_b7[q][0] * P[d] + (double)c_gal_b7[q][1] * P[3 + d] + (double)c_gal_b7[q][2] * P[6 + d];
      hi[d] = (float)y;
      lo[d] = (float)(y - (double)hi[d]);
    }
    const size_t i = 7 * (size_t)t + q;
    p_hi[i] = make_float4(hi[0], hi[1], hi[2], 0.f);
    p_lo[i] = make_float4(lo[0], lo[1], lo[2], 0.f);
    p_n[i] = make_float4((float)nrm64[3 * t], (float)nrm64[3 * t + 1], (float)nrm64[3 * t + 2], 0.f);
    p_q[i] = make_float4(0.f, 0.f, 0.f, (float)((double)c_gal_b7[q][3] * A * 0.25 / 3.14159265358979323846));
  }
}

// Pairs sharing no vertex: a block has eight test triangles t, a warp each, and 32 triangles s, a
// lane each. A thread computes (t, s) and (s, t) together where both rows belong to the round: s > t
// then, and those with t0 <= s <= t are left out. For a flat sigma d.n_sigma depends on x alone, and
// d.n_tau on y alone, so both normal derivatives come from the sums of F. The blocks (s, t) go
// through shared memory, so both directions are stored in runs (256 and 64 bytes).
//
// Bound by the FMA pipe: about 2300 operations for the two blocks (2 x 2310 when every ordered pair
// was formed by itself, with the projections in the innermost loop); 5120 triangles: 2.71 ms
// before, 1.34 ms now (1.67 with the blocks (s, t) stored by each thread in 72-byte pieces).
__global__ void __launch_bounds__(kGalT * 32, 2)
k_gal_regular(const float4* __restrict__ c_hi, const float4* __restrict__ c_lo, const float4* __restrict__ nrm,
              const float4* __restrict__ qp, const int4* __restrict__ vid, const float4* __restrict__ curl,
              int nt, int t0, int t1, float k, float2* __restrict__ partL, float2* __restrict__ partR) {
  __shared__ float2 s_st[kGalVals][32][kGalT + 1];
  __shared__ unsigned s_ok[kGalT];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int tb = t0 + blockIdx.y * kGalT, sb0 = blockIdx.x * 32;
  if (sb0 >= t0 && sb0 + 31 <= tb) return;  // every pair of the tile is another tile's
  const int t = min(tb + w, t1 - 1), s = min(sb0 + lane, nt - 1);
  bool live = tb + w < t1 && sb0 + lane < nt && !(s >= t0 && s <= t);
  const int4 vt = vid[t], vs = vid[s];
  const int va[3] = {vt.x, vt.y, vt.z}, vb[3] = {vs.x, vs.y, vs.z};
  bool touch = false;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) touch |= va[a] == vb[b];
  live = live && !touch;  // k_gal_singular writes the pairs that touch
  const bool both = live && s >= t0 && s < t1;
  const unsigned oks = __ballot_sync(0xffffffffu, both);
  if (lane == 0) s_ok[w] = oks;
  if (live) {
  const float4 th = c_hi[t], tl = c_lo[t], sh = c_hi[s], sl = c_lo[s];
  const float Dx = (th.x - sh.x) + (tl.x - sl.x);
  const float Dy = (th.y - sh.y) + (tl.y - sl.y);
  const float Dz = (th.z - sh.z) + (tl.z - sl.z);
  const float4 nx = nrm[t], ny = nrm[s];
  const float Dny = fmaf(Dx, ny.x, fmaf(Dy, ny.y, Dz * ny.z)), Dnx = fmaf(Dx, nx.x, fmaf(Dy, nx.y, Dz * nx.z));
  // trial points: the centroid, then the first orbit's points towards vertices 0, 1, 2 and the
  // second orbit's at kOrbit times the same offsets
  float bx[3], by[3], bz[3], nb[3];
  float wc, wo[2];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const float4 q = qp[7 * (size_t)s + 3 - m];
    bx[m] = q.x;
    by[m] = q.y;
    bz[m] = q.z;
    nb[m] = fmaf(q.x, nx.x, fmaf(q.y, nx.y, q.z * nx.z));
    wo[0] = q.w;
  }
  wc = qp[7 * (size_t)s].w;
  wo[1] = qp[7 * (size_t)s + 4].w;
  GalAcc A;
  gal_acc_zero(A);
#pragma unroll 1
  for (int p = 0; p < 7; ++p) {
    const float4 qt = qp[7 * (size_t)t + p];
    const float wx = qt.w * kFourPi;  // w_p A_tau (the 1 / (4 pi) is in the trial weights)
    const float px = Dx + qt.x, py = Dy + qt.y, pz = Dz + qt.z;
    const float pny = Dny + fmaf(qt.x, ny.x, fmaf(qt.y, ny.y, qt.z * ny.z));
    // inner sums over the trial points per basis function b, of G, F and F d.n_tau. On an orbit
    // with barycentrics (e, e, 1 - 2e): sum_q mu_b(q) v_q = e S + (1 - 3e) v_b, S the orbit's sum
    // and v_b its point towards vertex b; the centroid counts a third on every b.
    float cm[6], sb[3][6];
    float turns;
    {
      const float r2 = fmaf(px, px, fmaf(py, py, pz * pz));
      const float rinv = rsqrtf(r2), rho = k * (r2 * rinv);
      turns = gal_turns(rho);
      float2 G, F;
      gal_kernels(rinv, rho, turns, wc, G, F);
      const float third = c_gal_b7[0][0];
      cm[0] = third * G.x;
      cm[1] = third * G.y;
      cm[2] = third * F.x;
      cm[3] = third * F.y;
      cm[4] = cm[2] * Dnx;
      cm[5] = cm[3] * Dnx;
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const float c = o == 0 ? -1.f : -kOrbit;
      const float e = c_gal_b7[1 + 3 * o][0], f = c_gal_b7[1 + 3 * o][2] - e;  // e and 1 - 3e
      float S[6];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const float dx = fmaf(c, bx[m], px), dy = fmaf(c, by[m], py), dz = fmaf(c, bz[m], pz);
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float rinv = rsqrtf(r2), rho = k * (r2 * rinv);
        float2 G, F;
        gal_kernels(rinv, rho, turns, wo[o], G, F);
        const float dnx = fmaf(c, nb[m], Dnx);
        const float v[6] = {G.x, G.y, F.x, F.y, F.x * dnx, F.y * dnx};
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          S[i] = m == 0 ? v[i] : S[i] + v[i];
          sb[m][i] = o == 0 ? f * v[i] : fmaf(f, v[i], sb[m][i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) cm[i] = fmaf(e, S[i], cm[i]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
#pragma unroll
      for (int i = 0; i < 6; ++i) sb[b][i] += cm[i];
      sb[b][2] *= pny;
      sb[b][3] *= pny;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float la = c_gal_b7[p][a] * wx;
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          A.gb[2 * (3 * a + b) + i] = fmaf(la, sb[b][i], A.gb[2 * (3 * a + b) + i]);
          A.ky[2 * (3 * a + b) + i] = fmaf(la, sb[b][2 + i], A.ky[2 * (3 * a + b) + i]);
          A.kx[2 * (3 * a + b) + i] = fmaf(la, sb[b][4 + i], A.kx[2 * (3 * a + b) + i]);
        }
    }
  }
  float cc[9];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float4 ca = curl[3 * (size_t)t + a];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float4 cb = curl[3 * (size_t)s + b];
      cc[3 * a + b] = ca.x * cb.x + ca.y * cb.y + ca.z * cb.z;
    }
  }
  const float nn = nx.x * ny.x + nx.y * ny.y + nx.z * ny.z;
  float2 out[kGalVals];
  gal_finish<false>(A, k, nn, cc, out);
  gal_store(partL, partR, nt, t - t0, s, out);
  if (both) {
    gal_finish<true>(A, k, nn, cc, out);
#pragma unroll
    for (int i = 0; i < kGalVals; ++i) s_st[i][lane][w] = out[i];
  }
  }
  __syncthreads();
  const int q = threadIdx.x % kGalT, e = threadIdx.x / kGalT;  // test triangle, s: 32 of them
  if (s_ok[q] >> e & 1u) {
#pragma unroll
    for (int i = 0; i < kGalVals; ++i) gal_plane(partL, partR, nt, sb0 + e - t0, i)[tb + q] = s_st[i][e][q];
  }
}

namespace {
// Barycentric coordinates placed at local vertices (i0, i1, i2).
__device__ __forceinline__ void gal_place(float (&l)[3], int i0, int i1, float v0, float v1, float v2) {
#pragma unroll
  for (int v = 0; v < 3; ++v) l[v] = v == i0 ? v0 : v == i1 ? v1 : v2;
}

__device__ __forceinline__ float3 f3sub(const double* a, const double* b) {
  return make_float3((float)(a[0] - b[0]), (float)(a[1] - b[1]), (float)(a[2] - b[2]));
}
}  // namespace

// Pairs sharing a vertex or an edge (the near-pair list), then the identical pairs: one warp
// per pair, the rule's points dealt over the lanes, a fixed shuffle tree, lane 0 writes. The rules
// for (t, s) and (s, t) are the same points with the roles swapped (regions, signs and the
// symmetric Gauss points trade places), so one warp forms both where both rows are in the round.
__global__ void __launch_bounds__(256)
k_gal_singular(const int2* __restrict__ near_pairs, int64_t n_near, const double* __restrict__ tri,
               const double* __restrict__ nrm64, const double* __restrict__ area, const int4* __restrict__ vid,
               const float4* __restrict__ curl, int nt, int t0, int t1, float k, float2* __restrict__ partL,
               float2* __restrict__ partR) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_near + nt) return;
  int t, s;
  if (w < n_near) {
    const int2 pr = near_pairs[w];
    t = pr.x;
    s = pr.y;
  } else {
    t = s = (int)(w - n_near);
  }
  if (t < t0 || t >= t1 || (s >= t0 && s < t)) return;
  const double* Pt = tri + 9 * (size_t)t;
  const double* Ps = tri + 9 * (size_t)s;
  const double At = area[t], As = area[s];
  const float3 nx = make_float3((float)nrm64[3 * t], (float)nrm64[3 * t + 1], (float)nrm64[3 * t + 2]);
  const float3 ny = make_float3((float)nrm64[3 * s], (float)nrm64[3 * s + 1], (float)nrm64[3 * s + 2]);
  const int4 vt4 = vid[t], vs4 = vid[s];
  const int vt[3] = {vt4.x, vt4.y, vt4.z}, vs[3] = {vs4.x, vs4.y, vs4.z};
  // shared vertices in the order (a over tau, b over sigma)
  int sh_a[2] = {0, 0}, sh_b[2] = {0, 0}, nsh = 0;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      if (vt[a] == vs[b] && nsh < 2) {
        sh_a[nsh] = a;
        sh_b[nsh] = b;
        ++nsh;
      }
  const int kind = t == s ? 3 : nsh;  // 1 vertex, 2 edge, 3 identical
  const int regions = kind == 1 ? 2 : 6;
  const int npts = regions * kGalSing * kGalSing * kGalSing * kGalSing;
  const float jac_area = (float)(4.0 * At * As) * kInv4Pi;
  GalAcc A;
  gal_acc_zero(A);
  // geometry of the rule in FP32 (differences of FP64 vertices)
  float3 e1, e2, e3, e4;
  int ia = 0, ib = 0, ic = 0, ja = 0, jb = 0, jc = 0;
  if (kind == 3) {
    e1 = f3sub(Pt + 3, Pt);      // B - A
    e2 = f3sub(Pt + 6, Pt + 3);  // C - B
    e3 = e4 = e1;
  } else if (kind == 2) {
    ia = sh_a[0];
    ib = sh_a[1];
    ja = sh_b[0];
    jb = sh_b[1];
    ic = 3 - ia - ib;
    jc = 3 - ja - jb;
    e1 = f3sub(Pt + 3 * ib, Pt + 3 * ia);  // Pb - Pa
    e2 = f3sub(Pt + 3 * ic, Pt + 3 * ia);  // Ct - Pa
    e3 = f3sub(Ps + 3 * jc, Pt + 3 * ia);  // Cs - Pa
    e4 = e1;
  } else {
    ia = sh_a[0];
    ja = sh_b[0];
    e1 = f3sub(Pt + 3 * ((ia + 1) % 3), Pt + 3 * ia);
    e2 = f3sub(Pt + 3 * ((ia + 2) % 3), Pt + 3 * ia);
    e3 = f3sub(Ps + 3 * ((ja + 1) % 3), Pt + 3 * ia);
    e4 = f3sub(Ps + 3 * ((ja + 2) % 3), Pt + 3 * ia);
  }
  for (int idx = lane; idx < npts; idx += 32) {
    const int region = idx >> 8, g = idx & 255;
    const float2 n0 = make_float2(c_gal_gl[g >> 6][0], c_gal_gl[g >> 6][1]);
    const float2 n1 = make_float2(c_gal_gl[(g >> 4) & 3][0], c_gal_gl[(g >> 4) & 3][1]);
    const float2 n2 = make_float2(c_gal_gl[(g >> 2) & 3][0], c_gal_gl[(g >> 2) & 3][1]);
    const float2 n3 = make_float2(c_gal_gl[g & 3][0], c_gal_gl[g & 3][1]);
    const float gw = n0.y * n1.y * n2.y * n3.y;
    float lam[3], mu[3], dx, dy, dz, jac;
    if (kind == 3) {
      // relative coordinate z on the hexagon T - T, sector `region`, Duffy (rho, w); x in the
      // homothetic triangle of scale 1 - rho by collapsed coordinates (a1, a1 a2)
      // hexagon vertices (1,0), (1,1), (0,1), (-1,0), (-1,-1), (0,-1), by selects (no local array)
      const int r1 = region == 5 ? 0 : region + 1;
      const float hx0 = region < 2 ? 1.f : (region == 2 || region == 5) ? 0.f : -1.f;
      const float hy0 = (region == 0 || region == 3) ? 0.f : region < 3 ? 1.f : -1.f;
      const float hx1 = r1 < 2 ? 1.f : (r1 == 2 || r1 == 5) ? 0.f : -1.f;
      const float hy1 = (r1 == 0 || r1 == 3) ? 0.f : r1 < 3 ? 1.f : -1.f;
      const float rho = n0.x, wv = n1.x, a1 = n2.x, a2 = n3.x;
      const float z1 = rho * fmaf(wv, hx1 - hx0, hx0);
      const float z2 = rho * fmaf(wv, hy1 - hy0, hy0);
      const float ca = fmaxf(0.f, -z2), cb = fmaxf(0.f, z2 - z1);
      const float scale = 1.f - rho;
      const float xs = ca + cb + scale * a1, xt = ca + scale * (a1 * a2);
      const float ys = xs + z1, yt = xt + z2;
      jac = rho * scale * scale * a1;
      dx = -(z1 * e1.x + z2 * e2.x);
      dy = -(z1 * e1.y + z2 * e2.y);
      dz = -(z1 * e1.z + z2 * e2.z);
      lam[0] = 1.f - xs;
      lam[1] = xs - xt;
      lam[2] = xt;
      mu[0] = 1.f - ys;
      mu[1] = ys - yt;
      mu[2] = yt;
    } else if (kind == 2) {
      // along the shared edge (xi on tau, xs on sigma = xi + delta) and towards the opposite
      // vertices (et, es); regions: sign of delta, then which of et, es, |delta| is largest
      const float tt = n0.x, u = n1.x, v = n2.x, wv = n3.x;
      const int sgn = region < 3 ? 1 : -1, reg = region % 3;
      const float et = reg == 0 ? tt : tt * u;
      const float es = reg == 0 ? tt * u : reg == 1 ? tt : tt * v;
      const float dd = reg == 2 ? tt : tt * v;
      const float delta = sgn > 0 ? dd : -dd;
      const float xi = sgn > 0 ? (1.f - dd) * wv : fmaf(1.f - dd, wv, dd);
      const float xs = xi + delta;
      jac = tt * tt * (1.f - dd) * (1.f - et) * (1.f - es);
      // d = -delta e + et (Ct - Et) - es (Cs - Es), Et - Pa = xi e, Es - Pa = xs e
      dx = -delta * e1.x + et * (e2.x - xi * e1.x) - es * (e3.x - xs * e1.x);
      dy = -delta * e1.y + et * (e2.y - xi * e1.y) - es * (e3.y - xs * e1.y);
      dz = -delta * e1.z + et * (e2.z - xi * e1.z) - es * (e3.z - xs * e1.z);
      gal_place(lam, ia, ib, (1.f - et) * (1.f - xi), (1.f - et) * xi, et);
      gal_place(mu, ja, jb, (1.f - es) * (1.f - xs), (1.f - es) * xs, es);
    } else {
      // polar coordinates about the shared vertex on both triangles, the smaller radius as a
      // fraction of the larger
      const float tt = n0.x, u = n1.x, thv = n2.x, ths = n3.x;
      const float rt = region == 0 ? tt : tt * u, rs = region == 0 ? tt * u : tt;
      jac = tt * tt * tt * u;
      const float etx = fmaf(thv, e2.x - e1.x, e1.x), ety = fmaf(thv, e2.y - e1.y, e1.y), etz = fmaf(thv, e2.z - e1.z, e1.z);
      const float esx = fmaf(ths, e4.x - e3.x, e3.x), esy = fmaf(ths, e4.y - e3.y, e3.y), esz = fmaf(ths, e4.z - e3.z, e3.z);
      dx = rt * etx - rs * esx;
      dy = rt * ety - rs * esy;
      dz = rt * etz - rs * esz;
      gal_place(lam, ia, (ia + 1) % 3, 1.f - rt, rt * (1.f - thv), rt * thv);
      gal_place(mu, ja, (ja + 1) % 3, 1.f - rs, rs * (1.f - ths), rs * ths);
    }
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float rinv = rsqrtf(r2), rho = k * (r2 * rinv);
    float2 G, F;
    gal_kernels(rinv, rho, gal_turns(rho), gw * jac * jac_area, G, F);
    const float dny = fmaf(dx, ny.x, fmaf(dy, ny.y, dz * ny.z)), dnx = fmaf(dx, nx.x, fmaf(dy, nx.y, dz * nx.z));
    const float v[6] = {G.x, G.y, F.x * dny, F.y * dny, F.x * dnx, F.y * dnx};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const float lm = lam[a] * mu[b];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          A.gb[2 * (3 * a + b) + i] = fmaf(lm, v[i], A.gb[2 * (3 * a + b) + i]);
          A.ky[2 * (3 * a + b) + i] = fmaf(lm, v[2 + i], A.ky[2 * (3 * a + b) + i]);
          A.kx[2 * (3 * a + b) + i] = fmaf(lm, v[4 + i], A.kx[2 * (3 * a + b) + i]);
        }
      }
  }
  // fixed-order reduction over the warp
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int i = 0; i < 18; ++i) {
      A.gb[i] += __shfl_xor_sync(0xffffffffu, A.gb[i], off);
      A.ky[i] += __shfl_xor_sync(0xffffffffu, A.ky[i], off);
      A.kx[i] += __shfl_xor_sync(0xffffffffu, A.kx[i], off);
    }
  }
  if (lane != 0) return;
  float cc[9];
  for (int a = 0; a < 3; ++a) {
    const float4 ca = curl[3 * (size_t)t + a];
    for (int b = 0; b < 3; ++b) {
      const float4 cb = curl[3 * (size_t)s + b];
      cc[3 * a + b] = ca.x * cb.x + ca.y * cb.y + ca.z * cb.z;
    }
  }
  float2 out[kGalVals];
  const float nn = nx.x * ny.x + nx.y * ny.y + nx.z * ny.z;
  gal_finish<false>(A, k, nn, cc, out);
  if (kind == 3) {
    // mass terms: 1/2 M11 (A / 12 (1 + delta_ab)) and -(beta / 2) M10 (A / 3), beta = i / k
    const float m = (float)(At / 24.0);
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) out[3 * a + b].x += a == b ? 2.f * m : m;
    for (int a = 0; a < 3; ++a) out[9 + a].y -= (float)(At / 6.0) / k;
  }
  gal_store(partL, partR, nt, t - t0, s, out);
  if (s > t && s < t1) {
    gal_finish<true>(A, k, nn, cc, out);
    gal_store(partL, partR, nt, s - t0, t, out);
  }
}

// First stage of the L gather, one block row per test triangle tau of the round: for every
// column vertex j and local test index a, P2[(tau - t0) 3 + a][j] = sum over the triangles sigma
// around j (local index b) of the pair blocks (tau, sigma)[a][b]. Each block reads its own row
// of pair blocks, so every pair block is read from memory once.
__global__ void __launch_bounds__(256)
k_gal_rowsum_L(const float2* __restrict__ partL, int nt, const int* __restrict__ adj_ptr,
               const int2* __restrict__ adj, int nv, int ldv, float2* __restrict__ P2) {
  const int tr = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nv) return;
  const float2* row = partL + (size_t)tr * 9 * nt;
  float2 acc[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  for (int v = adj_ptr[j]; v < adj_ptr[j + 1]; ++v) {
    const int2 sb = adj[v];
    const float2* blk = row + (size_t)sb.y * nt + sb.x;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float2 x = blk[(size_t)3 * a * nt];
      acc[a].x += x.x;
      acc[a].y += x.y;
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) P2[((size_t)tr * 3 + a) * ldv + j] = acc[a];
}

// L[i][j] (+)= sum over the triangles tau around i (local index a) in the round of
// P2[(tau - t0) 3 + a][j]; adjacency lists in increasing triangle order. Columns past nv are
// zero. With Lb, the BF16 copy is written too (on the last round).
__global__ void __launch_bounds__(256)
k_gal_gather_L(const float2* __restrict__ P2, int t0, int t1, const int* __restrict__ adj_ptr,
               const int2* __restrict__ adj, int nv, int ldv, int accumulate, float2* __restrict__ L,
               uint32_t* __restrict__ Lb) {
  const int i = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ldv) return;
  const size_t off = (size_t)i * ldv + j;
  float2 acc = accumulate ? L[off] : make_float2(0.f, 0.f);
  if (j < nv) {
    for (int u = adj_ptr[i]; u < adj_ptr[i + 1]; ++u) {
      const int2 ta = adj[u];
      if (ta.x < t0 || ta.x >= t1) continue;
      const float2 x = P2[((size_t)(ta.x - t0) * 3 + ta.y) * ldv + j];
      acc.x += x.x;
      acc.y += x.y;
    }
  }
  L[off] = acc;
  if (Lb) Lb[off] = gal_pack_bf16(acc.x, acc.y);
}

// R[i][s] (+)= sum over the triangles tau around i in the round of partR[(tau - t0) 3 + a][s].
__global__ void __launch_bounds__(256)
k_gal_gather_R(const float2* __restrict__ partR, int nt, int t0, int t1, const int* __restrict__ adj_ptr,
               const int2* __restrict__ adj, int ldr, int accumulate, float2* __restrict__ R) {
  const int i = blockIdx.y;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= ldr) return;
  const size_t off = (size_t)i * ldr + s;
  float2 acc = accumulate ? R[off] : make_float2(0.f, 0.f);
  if (s < nt) {
    for (int u = adj_ptr[i]; u < adj_ptr[i + 1]; ++u) {
      const int2 ta = adj[u];
      if (ta.x < t0 || ta.x >= t1) continue;
      const float2 x = partR[((size_t)(ta.x - t0) * 3 + ta.y) * nt + s];
      acc.x += x.x;
      acc.y += x.y;
    }
  }
  R[off] = acc;
}

// P1 data at the vertices and P0 data per triangle, expanded to the 7 points of every triangle:
// pq[r][7 t + q] = sum_b lam_qb p[r][vid_tb], gq[r][7 t + q] = g[r][t].
__global__ void k_gal_expand(const int4* __restrict__ vid, int nt, int nv, int nrhs, const float2* __restrict__ p,
                             const float2* __restrict__ g, float2* __restrict__ pq, float2* __restrict__ gq) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = 7 * (int64_t)nt;
  if (i >= per * nrhs) return;
  const int r = (int)(i / per);
  const int64_t e = i % per;
  const int t = (int)(e / 7), q = (int)(e % 7);
  const int4 v = vid[t];
  const float2* pr = p + (size_t)r * nv;
  const float2 a = pr[v.x], b = pr[v.y], c = pr[v.z];
  const float l0 = c_gal_b7[q][0], l1 = c_gal_b7[q][1], l2 = c_gal_b7[q][2];
  pq[i] = make_float2(l0 * a.x + l1 * b.x + l2 * c.x, l0 * a.y + l1 * b.y + l2 * c.y);
  gq[i] = g[(size_t)r * nt + t];
}

namespace {
nat_bem_status gal_upload_rules() {
  static bool done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && done[dev]) return NAT_BEM_OK;
  const double s15 = std::sqrt(15.0);
  const double a = (6.0 - s15) / 21.0, wa = (155.0 - s15) / 1200.0;
  const double b = (6.0 + s15) / 21.0, wb = (155.0 + s15) / 1200.0;
  const double r[7][4] = {{1.0 / 3, 1.0 / 3, 1.0 / 3, 9.0 / 40}, {a, a, 1 - 2 * a, wa}, {a, 1 - 2 * a, a, wa},
                          {1 - 2 * a, a, a, wa}, {b, b, 1 - 2 * b, wb}, {b, 1 - 2 * b, b, wb},
                          {1 - 2 * b, b, b, wb}};
  float rf[7][4];
  for (int i = 0; i < 7; ++i)
    for (int c = 0; c < 4; ++c) rf[i][c] = (float)r[i][c];
  NB_TRY_CUDA(cudaMemcpyToSymbol(c_gal_b7, rf, sizeof(rf)));
  // 4-point Gauss-Legendre on [0, 1] (nodes (1 -+ x) / 2, weights w / 2)
  const double x1 = std::sqrt(3.0 / 7.0 - 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double x2 = std::sqrt(3.0 / 7.0 + 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double w1 = (18.0 + std::sqrt(30.0)) / 36.0, w2 = (18.0 - std::sqrt(30.0)) / 36.0;
  const double gl[4][2] = {{0.5 * (1 - x2), 0.5 * w2}, {0.5 * (1 - x1), 0.5 * w1}, {0.5 * (1 + x1), 0.5 * w1},
                           {0.5 * (1 + x2), 0.5 * w2}};
  float glf[4][2];
  for (int i = 0; i < 4; ++i) {
    glf[i][0] = (float)gl[i][0];
    glf[i][1] = (float)gl[i][1];
  }
  NB_TRY_CUDA(cudaMemcpyToSymbol(c_gal_gl, glf, sizeof(glf)));
  if (dev >= 0 && dev < 64) done[dev] = true;
  return NAT_BEM_OK;
}
}  // namespace

nat_bem_status galerkin_geometry_build(nat_bem_op* op, const int32_t* T, int64_t nv, cudaStream_t s) {
  NB_TRY(gal_upload_rules());
  Geometry& g = op->geo;
  const int64_t nt = g.n;
  // vertex -> (triangle, local index) lists in increasing triangle order
  std::vector<int> ptr(nv + 1, 0);
  for (int64_t t = 0; t < nt; ++t)
    for (int a = 0; a < 3; ++a) ++ptr[T[3 * t + a] + 1];
  for (int64_t v = 0; v < nv; ++v) ptr[v + 1] += ptr[v];
  std::vector<int2> adj(3 * nt);
  std::vector<int> fill(ptr.begin(), ptr.end() - 1);
  for (int64_t t = 0; t < nt; ++t)
    for (int a = 0; a < 3; ++a) adj[fill[T[3 * t + a]]++] = make_int2((int)t, a);
  Galerkin& G = op->gal;
  NB_TRY(dev_alloc_n(&G.adj_ptr, (size_t)nv + 1, s));
  NB_TRY(dev_alloc_n(&G.adj, (size_t)3 * nt, s));
  NB_TRY(dev_alloc_n(&G.curl, (size_t)3 * nt, s));
  NB_TRY(dev_alloc_n(&G.pts.c_hi, (size_t)7 * nt, s));
  NB_TRY(dev_alloc_n(&G.pts.c_lo, (size_t)7 * nt, s));
  NB_TRY(dev_alloc_n(&G.pts.nrm, (size_t)7 * nt, s));
  NB_TRY(dev_alloc_n(&G.pts.qp, (size_t)7 * nt, s));
  G.pts.n = 7 * nt;
  NB_TRY_CUDA(cudaMemcpyAsync(G.adj_ptr, ptr.data(), (nv + 1) * sizeof(int), cudaMemcpyHostToDevice, s));
  NB_TRY_CUDA(cudaMemcpyAsync(G.adj, adj.data(), 3 * nt * sizeof(int2), cudaMemcpyHostToDevice, s));
  NB_TRY_CUDA(cudaStreamSynchronize(s));  // the host vectors go out of scope
  NB_LAUNCH("gal_geometry", s, k_gal_geometry<<<(unsigned)((nt + 127) / 128), 128, 0, s>>>(
      g.tri, g.nrm64, g.area, (int)nt, G.curl, G.pts.c_hi, G.pts.c_lo, G.pts.nrm, G.pts.qp));
  NB_CHECK_LAUNCH();
  return NAT_BEM_OK;
}

nat_bem_status galerkin_assemble_operators(nat_bem_op* op, cudaStream_t s) {
  NB_TRY(gal_upload_rules());
  const Geometry& g = op->geo;
  const Galerkin& G = op->gal;
  const int nt = (int)g.n, nv = (int)op->n, ldv = (int)g.ld, ldr = (int)op->ldr;
  const float k = (float)op->k;
  // rounds of test triangles: pair blocks (9 + 3 values) and first-stage row sums (3 ldv)
  const double per_row = (double)nt * kGalVals * sizeof(float2) + 3.0 * ldv * sizeof(float2);
  const int chunk = std::max(1, std::min(nt, std::max(512, (int)(kGalScratch / per_row))));
  float2 *partL = nullptr, *partR = nullptr, *P2 = nullptr;
  nat_bem_status st = dev_alloc_n(&partL, (size_t)chunk * nt * 9, s);
  if (st == NAT_BEM_OK) st = dev_alloc_n(&partR, (size_t)chunk * nt * 3, s);
  if (st == NAT_BEM_OK) st = dev_alloc_n(&P2, (size_t)chunk * 3 * ldv, s);
  for (int t0 = 0; t0 < nt && st == NAT_BEM_OK; t0 += chunk) {
    const int t1 = std::min(nt, t0 + chunk);
    const bool last = t1 == nt;
    NB_LAUNCH("gal_regular", s, k_gal_regular<<<dim3((unsigned)((nt + 31) / 32), (unsigned)((t1 - t0 + kGalT - 1) / kGalT)), kGalT * 32, 0, s>>>(
        g.c_hi, g.c_lo, g.nrm, g.qp, g.vid, G.curl, nt, t0, t1, k, partL, partR));
    const int64_t warps = g.n_near + nt;
    NB_LAUNCH("gal_singular", s, k_gal_singular<<<(unsigned)((warps * 32 + 255) / 256), 256, 0, s>>>(
        g.near_pairs, g.n_near, g.tri, g.nrm64, g.area, g.vid, G.curl, nt, t0, t1, k, partL, partR));
    NB_LAUNCH("gal_rowsum_L", s, k_gal_rowsum_L<<<dim3((unsigned)((nv + 255) / 256), (unsigned)(t1 - t0)), 256, 0, s>>>(
        partL, nt, G.adj_ptr, G.adj, nv, ldv, P2));
    NB_LAUNCH("gal_gather_L", s, k_gal_gather_L<<<dim3((unsigned)((ldv + 255) / 256), (unsigned)nv), 256, 0, s>>>(
        P2, t0, t1, G.adj_ptr, G.adj, nv, ldv, t0 > 0 ? 1 : 0, op->L, last ? bf16_target(op) : nullptr));
    NB_LAUNCH("gal_gather_R", s, k_gal_gather_R<<<dim3((unsigned)((ldr + 255) / 256), (unsigned)nv), 256, 0, s>>>(
        partR, nt, t0, t1, G.adj_ptr, G.adj, ldr, t0 > 0 ? 1 : 0, op->R));
    if (cudaGetLastError() != cudaSuccess) {
      set_error("Galerkin assembly: launch failed");
      st = NAT_BEM_ECUDA;
    }
  }
  dev_free(partL, s);
  dev_free(partR, s);
  dev_free(P2, s);
  if (st == NAT_BEM_OK) st = finish_low_copy(op, s);
  return st;
}

nat_bem_status galerkin_expand(const nat_bem_op* op, const float2* d_p, const float2* d_g, int nrhs,
                               float2** pq, float2** gq, cudaStream_t s) {
  const int64_t nt = op->geo.n, tot = 7 * nt * nrhs;
  *pq = *gq = nullptr;
  NB_TRY(dev_alloc_n(pq, (size_t)tot, s));
  nat_bem_status st = dev_alloc_n(gq, (size_t)tot, s);
  if (st != NAT_BEM_OK) {
    dev_free(*pq, s);
    *pq = nullptr;
    return st;
  }
  NB_LAUNCH("gal_expand", s, k_gal_expand<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(
      op->geo.vid, (int)nt, (int)op->n, nrhs, d_p, d_g, *pq, *gq));
  NB_CHECK_LAUNCH();
  return NAT_BEM_OK;
}

void galerkin_free(nat_bem_op* op, cudaStream_t s) {
  Galerkin& G = op->gal;
  void* ptrs[] = {G.adj_ptr, G.adj, G.curl, G.pts.c_hi, G.pts.c_lo, G.pts.nrm, G.pts.qp};
  for (void* p : ptrs) dev_free(p, s);
  G = Galerkin{};
}

}  // namespace natbem
