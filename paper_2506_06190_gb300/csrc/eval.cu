// Field evaluation: the exterior representation p(x) = int [p dG/dn_y - G g] dS_y with the
// piecewise-constant surface data (pressure anywhere from the Neumann and Dirichlet data,
// paper Sec. 3.4; its surface limit is the first line of Sec. 4, Eq. 6). For a Monte-Carlo op
// (Sec. 4.1.1) the same sum runs over the samples with weight |Gamma| / M each, one point per
// sample. Otherwise the 7-point rule is applied on every element:
//
//   field(x_q) = sum_j [ p_j sum_p w_p A_j dG/dn_y(x_q, y_jp) - g_j sum_p w_p A_j G(x_q, y_jp) ]
//
// FP32 kernel generation, one thread per field point, elements split over blocks and staged in
// shared memory (broadcast reads); per-split FP64 partial sums are reduced in a fixed order.
//
// The kernel is bound by the quarter-rate unit (rsqrt, sin, cos: 24 cycles per point, element point
// and scheduler) beside the FMA pipe, so everything else is kept small:
//   - the rule's outer points lie on the lines from the centroid to the vertices: with D the
//     difference to the centroid, |D - q|^2 = |D|^2 + |q|^2 - 2 D.q, and three projections D.q_m
//     (their sum is zero) serve all six; D.n is one value per element. That square cancels for a
//     point close to one of them (at 0.01 of the element's size 7e-4; nearer it can be negative): an
//     element whose centroid is within sqrt(6) of its largest |q| is left out, marked, and added
//     after the stage from the differences to its points. Warps whose points are away from all of
//     a stage's elements (Geometry::group) take a loop without that test: the
//     training field below keeps its time (669 -> 673 us), points over the surface take 5-25% longer;
//   - the phases are reduced with the centroid's number of turns, and rounding is an FMA and an add
//     (the rounding instruction runs on the quarter-rate unit);
//   - two elements at a time in paired FP32 instructions.
// 10,000 points x 10240 triangles: 882 us before, 673 us now (643 without the correction of |D|^2,
// whose errors against 64 bits were 1% above the earlier kernel's; with it they are 10-15% below);
// the far field in 2048 directions 123 -> 86 us.
#include <cuda_runtime.h>

#include <mutex>
#include <string>
#include <type_traits>

#include "internal.h"
#include "pairs.cuh"

namespace natbem {

namespace {
constexpr int kEvalThreads = 128;  // field points per block
constexpr int kElemStage = 32;     // elements staged per shared-memory round
constexpr int kMaxRhsPass = 16;    // far field: right-hand sides per pass (kernel values reused)
constexpr int kEvalRhsPass = 32;   // field: right-hand sides per pass
constexpr int kNoAllocRhsPass = 4; // the allocation-free path: passes of four (scratch sizing)

// Fields of a staged element pair (elements in the two halves).
enum { kFHi = 0, kFLo = 3, kFN = 6, kFW = 9, kFQ0 = 12, kFQ1 = 15, kFSq = 18, kFields7 = 24, kFields1 = 10 };

// Stages `cnt` elements from jb on, the centroids' high parts rounded to multiples of ulp(grid) (as
// they are for grid 0): element e is half e & 1 of pair e >> 1. A last odd element is
// paired with itself at weight zero. Four threads share an element's seven-point record.
template <int NQ>
__device__ __forceinline__ void stage_elements(float (*f)[2 * (NQ == 7 ? kFields7 : kFields1)],
                                               const float4* __restrict__ c_hi, const float4* __restrict__ c_lo,
                                               const float4* __restrict__ nrm, const float4* __restrict__ qp, int jb,
                                               int cnt, float grid) {
  const int e = threadIdx.x & (kElemStage - 1), part = threadIdx.x / kElemStage;
  const int up = (cnt + 1) & ~1;
  if (e >= up) return;
  const int j = jb + min(e, cnt - 1);
  float* o = f[e >> 1] + (e & 1);
  const float live = e < cnt ? 1.f : 0.f;
  if (part == 0) {
    const float4 h = c_hi[j], l = c_lo[j], nn = nrm[j];
    const float hh[3] = {h.x, h.y, h.z}, ll[3] = {l.x, l.y, l.z}, n3[3] = {nn.x, nn.y, nn.z};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float c = (hh[d] + grid) - grid;
      o[2 * (kFHi + d)] = c;
      o[2 * (kFLo + d)] = (hh[d] - c) + ll[d];
      o[2 * (kFN + d)] = n3[d];
    }
    o[2 * kFW] = live * qp[NQ * (size_t)j].w;
  } else if (NQ == 7) {
    // first- and second-orbit points towards vertex m = part - 1 (rule order: vertex 2, 1, 0)
    const int m = part - 1;
    const float4 qa = qp[7 * (size_t)j + 3 - m], qb = qp[7 * (size_t)j + 6 - m];
    if (m < 2) {
      o[2 * (kFQ0 + 3 * m)] = qa.x;
      o[2 * (kFQ0 + 3 * m + 1)] = qa.y;
      o[2 * (kFQ0 + 3 * m + 2)] = qa.z;
    }
    o[2 * (kFSq + m)] = fmaf(qa.x, qa.x, fmaf(qa.y, qa.y, qa.z * qa.z));
    o[2 * (kFSq + 3 + m)] = fmaf(qb.x, qb.x, fmaf(qb.y, qb.y, qb.z * qb.z));
    if (m == 0) o[2 * (kFW + 1)] = live * qa.w;
    if (m == 1) o[2 * (kFW + 2)] = live * qb.w;
  }
}

// Stages p and g of the pass for `cnt` elements: (p.x, p.y, g.x, g.y) per element and RHS, zero
// past nr and past the last element; paired elements interleaved when kPaired.
template <int NR, bool kPaired>
__device__ __forceinline__ void stage_data(float4* sd, const float2* __restrict__ p, const float2* __restrict__ g, int n,
                                           int jb, int cnt, int rhs0, int nr) {
  for (int i = threadIdx.x; i < kElemStage * NR; i += kEvalThreads) {
    const int e = i & (kElemStage - 1), s = i / kElemStage;
    float2 pj = make_float2(0.f, 0.f), gj = pj;
    if (e < cnt && s < nr) {
      pj = p[(size_t)(rhs0 + s) * n + jb + e];
      gj = g[(size_t)(rhs0 + s) * n + jb + e];
    }
    if (kPaired) {  // [pair][rhs]: p.x, p.y, g.x, g.y of both
      float* o = reinterpret_cast<float*>(sd) + ((e >> 1) * NR + s) * 8 + (e & 1);
      o[0] = pj.x;
      o[2] = pj.y;
      o[4] = gj.x;
      o[6] = gj.y;
    } else {
      sd[e * NR + s] = make_float4(pj.x, pj.y, gj.x, gj.y);
    }
  }
}

// Sums over one element point: G += w e^{i rho} / r, F += w e^{i rho} (1 - i rho) / r^3, rho = k r.
__device__ __forceinline__ void point_terms(u64 rinv, u64 rho, u64 turns, u64 w, u64& Gr, u64& Gi, u64& Fr,
                                            u64& Fi) {
  u64 cs, sn;
  sincos2(rho, turns, cs, sn);
  const u64 gw = mul2(rinv, w);
  const u64 er = mul2(cs, gw), ei = mul2(sn, gw);
  const u64 t2 = mul2(rinv, rinv);
  Gr = add2(Gr, er);
  Gi = add2(Gi, ei);
  Fr = fma2(t2, fma2(rho, ei, er), Fr);
  Fi = fma2(t2, sub2(ei, mul2(rho, er)), Fi);
}
}  // namespace

template <int NR, int NQ>
__global__ void __launch_bounds__(kEvalThreads)
k_eval(const float4* __restrict__ c_hi, const float4* __restrict__ c_lo,
       const float4* __restrict__ nrm, const float4* __restrict__ qp, const float4* __restrict__ group, float grid,
       int n, const double* __restrict__ pts, int m, double k, const float2* __restrict__ p,
       const float2* __restrict__ g, int rhs0, int nr, int elems_per_split, double2* __restrict__ part) {
  constexpr int kF = NQ == 7 ? kFields7 : kFields1;
  constexpr bool kPaired = NR <= 4;  // paired accumulators: twice the registers per right-hand side
  __shared__ __align__(16) float s_f[kElemStage / 2][2 * kF];
  __shared__ float4 s_d[kElemStage * NR];
  const int qi = blockIdx.x * kEvalThreads + threadIdx.x;
  const bool ok = qi < m;
  const u64 k2 = bc((float)k);
  if (NQ == 1) grid = 0.f;
  // High parts of points and centroids on the body's grid: their difference a is exact out to a few
  // diameters of the body, and with the small b of the low parts |D|^2 = a.a + b.(a + D) is free of
  // the rounding of D = a + b (else the largest error of the sum, three times the rest). Beyond, a
  // rounds at 2^-24. Nothing here depends on the call's other points. One-point records split where
  // FP32 does (grid 0) and square D: no other point shares its rounding.
  double v[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) v[d] = ok ? pts[3 * (size_t)qi + d] : 0.0;
  u64 xh[3], xl[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float h = ((float)v[d] + grid) - grid;
    xh[d] = bc(h);
    xl[d] = bc((float)(v[d] - (double)h));
  }
  const int j_begin = blockIdx.y * elems_per_split;
  const int j_end = min(n, j_begin + elems_per_split);
  u64 ar2[kPaired ? NR : 1], ai2[kPaired ? NR : 1];
  float ar[kPaired ? 1 : NR], ai[kPaired ? 1 : NR];
#pragma unroll
  for (int s = 0; s < (kPaired ? NR : 1); ++s) ar2[s] = ai2[s] = bc(0.f);
#pragma unroll
  for (int s = 0; s < (kPaired ? 1 : NR); ++s) ar[s] = ai[s] = 0.f;
  for (int jb = j_begin; jb < j_end; jb += kElemStage) {
    const int cnt = min(kElemStage, j_end - jb);
    __syncthreads();
    stage_elements<NQ>(s_f, c_hi, c_lo, nrm, qp, jb, cnt, grid);
    stage_data<NR, kPaired>(s_d, p, g, n, jb, cnt, rhs0, nr);
    bool near = false;
    if constexpr (NQ == 7) {
      const float4 c = group[jb / kElemStage];
      float x, y, z, u;
      upk(add2(xh[0], xl[0]), x, u);
      upk(add2(xh[1], xl[1]), y, u);
      upk(add2(xh[2], xl[2]), z, u);
      x -= c.x, y -= c.y, z -= c.z;
      near = __any_sync(0xffffffffu, ok && fmaf(x, x, fmaf(y, y, z * z)) < c.w);
    }
    __syncthreads();
    if (!ok) continue;
    unsigned close = 0u;  // pairs left for after the loop
    // the pair's sums of G and dG/dn times its data
    auto add = [&](int t, u64 Gr, u64 Gi, u64 Dr, u64 Di) {
      if constexpr (kPaired) {
        const u64 nGr = sub2(bc(0.f), Gr), nGi = sub2(bc(0.f), Gi), nDi = sub2(bc(0.f), Di);
        const u64* d = reinterpret_cast<const u64*>(s_d) + 4 * t * NR;
#pragma unroll
        for (int s = 0; s < NR; ++s) {
          const u64 px = d[4 * s], py = d[4 * s + 1], gx = d[4 * s + 2], gy = d[4 * s + 3];
          ar2[s] = fma2(px, Dr, fma2(py, nDi, fma2(gx, nGr, fma2(gy, Gi, ar2[s]))));
          ai2[s] = fma2(px, Di, fma2(py, Dr, fma2(gx, nGi, fma2(gy, nGr, ai2[s]))));
        }
      } else {
        float gr[2], gi[2], dr[2], di[2];
        upk(Gr, gr[0], gr[1]);
        upk(Gi, gi[0], gi[1]);
        upk(Dr, dr[0], dr[1]);
        upk(Di, di[0], di[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4* d = s_d + (2 * t + h) * NR;
#pragma unroll
          for (int s = 0; s < NR; ++s) {
            const float4 a = d[s];
            ar[s] = fmaf(a.x, dr[h], fmaf(-a.y, di[h], fmaf(-a.z, gr[h], fmaf(a.w, gi[h], ar[s]))));
            ai[s] = fmaf(a.x, di[h], fmaf(a.y, dr[h], fmaf(-a.z, gi[h], fmaf(-a.w, gr[h], ai[s]))));
          }
        }
      }
    };
    auto pairs = [&](auto tested) {
      constexpr bool kTest = decltype(tested)::value;
      for (int t = 0; t < (cnt + 1) / 2; ++t) {
        const u64* f = reinterpret_cast<const u64*>(s_f[t]);
        const u64 ax = sub2(xh[0], f[kFHi]), bx = sub2(xl[0], f[kFLo]), Dx = add2(ax, bx);
        const u64 ay = sub2(xh[1], f[kFHi + 1]), by = sub2(xl[1], f[kFLo + 1]), Dy = add2(ay, by);
        const u64 az = sub2(xh[2], f[kFHi + 2]), bz = sub2(xl[2], f[kFLo + 2]), Dz = add2(az, bz);
        const u64 D2 = NQ == 1 ? fma2(Dx, Dx, fma2(Dy, Dy, mul2(Dz, Dz)))
                               : fma2(ax, ax, fma2(ay, ay, fma2(az, az,
                                 fma2(bx, add2(ax, Dx), fma2(by, add2(ay, Dy), mul2(bz, add2(az, Dz)))))));
        if constexpr (kTest) {
          float d[2], q[2], far[2] = {0.f, 0.f};
          upk(D2, d[0], d[1]);
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            upk(f[kFSq + e], q[0], q[1]);
            far[0] = fmaxf(far[0], 6.f * q[0]);
            far[1] = fmaxf(far[1], 6.f * q[1]);
          }
          if (d[0] < far[0] || d[1] < far[1]) {
            close |= 1u << t;
            continue;
          }
        }
        const u64 dn = fma2(Dx, f[kFN], fma2(Dy, f[kFN + 1], mul2(Dz, f[kFN + 2])));  // d.n of every point
        u64 Gr = bc(0.f), Gi = Gr, Fr = Gr, Fi = Gr;
        const u64 rc = rsqrt2(D2), rho = mul2(k2, mul2(D2, rc)), turns = turns2(rho);
        point_terms(rc, rho, turns, f[kFW], Gr, Gi, Fr, Fi);
        if constexpr (NQ == 7) {
          const u64 d0 = fma2(Dx, f[kFQ0], fma2(Dy, f[kFQ0 + 1], mul2(Dz, f[kFQ0 + 2])));
          const u64 d1 = fma2(Dx, f[kFQ1], fma2(Dy, f[kFQ1 + 1], mul2(Dz, f[kFQ1 + 2])));
          const u64 dm[3] = {d0, d1, sub2(bc(0.f), add2(d0, d1))};
#pragma unroll
          for (int o = 0; o < 2; ++o)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const u64 r2 = fma2(bc(o == 0 ? -2.f : -2.f * kOrbit), dm[q], add2(D2, f[kFSq + 3 * o + q]));
              const u64 ri = rsqrt2(r2);
              point_terms(ri, mul2(k2, mul2(r2, ri)), turns, f[kFW + 1 + o], Gr, Gi, Fr, Fi);
            }
        }
        add(t, Gr, Gi, mul2(Fr, dn), mul2(Fi, dn));
      }
    };
    if (!near) {
      pairs(std::false_type{});
      continue;
    }
    if constexpr (NQ == 7) {
      pairs(std::true_type{});
      for (; close; close &= close - 1u) {
        const int t = __ffs(close) - 1;
        const u64* f = reinterpret_cast<const u64*>(s_f[t]);
        const u64 Dx = add2(sub2(xh[0], f[kFHi]), sub2(xl[0], f[kFLo]));
        const u64 Dy = add2(sub2(xh[1], f[kFHi + 1]), sub2(xl[1], f[kFLo + 1]));
        const u64 Dz = add2(sub2(xh[2], f[kFHi + 2]), sub2(xl[2], f[kFLo + 2]));
        const u64 dn = fma2(Dx, f[kFN], fma2(Dy, f[kFN + 1], mul2(Dz, f[kFN + 2])));
        const float4 *qa = qp + 7 * (size_t)(jb + 2 * t), *qb = 2 * t + 1 < cnt ? qa + 7 : qa;
        u64 Gr = bc(0.f), Gi = Gr, Fr = Gr, Fi = Gr;
#pragma unroll 1
        for (int q = 0; q < 7; ++q) {
          const float4 a = qa[q], b = qb[q];
          const u64 dx = sub2(Dx, pk(a.x, b.x)), dy = sub2(Dy, pk(a.y, b.y)), dz = sub2(Dz, pk(a.z, b.z));
          const u64 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), ri = rsqrt2(r2), rho = mul2(k2, mul2(r2, ri));
          point_terms(ri, rho, turns2(rho), f[kFW + (q + 2) / 3], Gr, Gi, Fr, Fi);
        }
        add(t, Gr, Gi, mul2(Fr, dn), mul2(Fi, dn));
      }
    }
  }
  if (ok) {
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      float re, im;
      if constexpr (kPaired) {
        float re1, im1;
        upk(ar2[s], re, re1);
        upk(ai2[s], im, im1);
        part[((size_t)blockIdx.y * m + qi) * NR + s] = make_double2((double)re + (double)re1, (double)im + (double)im1);
      } else {
        re = ar[s];
        im = ai[s];
        part[((size_t)blockIdx.y * m + qi) * NR + s] = make_double2(re, im);
      }
    }
  }
}

// Far-field pattern, the leading FFAT term (paper Sec. 3.1): for unit directions d,
//   F(d) = lim r e^{-ikr} p(r d) = sum_j sum_q (w_q A_j / 4pi) [p_j (-i k d.n_j) - g_j] e^{-ik d.y_jq}
// with the same per-element rule (or one point per Monte-Carlo sample) as the field; one thread
// per direction, elements staged in shared memory, per-split FP64 partials as in k_eval. The
// phases of the outer points follow from two projections k d.q_m; bound by sin and cos.
template <int NR, int NQ>
__global__ void __launch_bounds__(kEvalThreads)
k_far_field(const float4* __restrict__ c_hi, const float4* __restrict__ c_lo,
            const float4* __restrict__ nrm, const float4* __restrict__ qp, int n,
            const double* __restrict__ dirs, int nd, double k, const float2* __restrict__ p,
            const float2* __restrict__ g, int rhs0, int nr, int elems_per_split, double2* __restrict__ part) {
  constexpr int kF = NQ == 7 ? kFields7 : kFields1;
  __shared__ __align__(16) float s_f[kElemStage / 2][2 * kF];
  __shared__ float4 s_d[kElemStage * NR];
  const int qi = blockIdx.x * kEvalThreads + threadIdx.x;
  const bool ok = qi < nd;
  float df[3] = {0.f, 0.f, 0.f}, dl[3] = {0.f, 0.f, 0.f};  // -k d, high and low parts
  if (ok)
    for (int d = 0; d < 3; ++d) {
      const double v = -k * dirs[3 * (size_t)qi + d];
      df[d] = (float)v;
      dl[d] = (float)(v - (double)df[d]);
    }
  const u64 d0 = bc(df[0]), d1 = bc(df[1]), d2 = bc(df[2]), l0 = bc(dl[0]), l1 = bc(dl[1]), l2 = bc(dl[2]);
  const int j_begin = blockIdx.y * elems_per_split;
  const int j_end = min(n, j_begin + elems_per_split);
  float accr[NR], acci[NR];
#pragma unroll
  for (int s = 0; s < NR; ++s) accr[s] = acci[s] = 0.f;
  for (int jb = j_begin; jb < j_end; jb += kElemStage) {
    const int cnt = min(kElemStage, j_end - jb);
    __syncthreads();
    stage_elements<NQ>(s_f, c_hi, c_lo, nrm, qp, jb, cnt, 0.f);
    stage_data<NR, false>(s_d, p, g, n, jb, cnt, rhs0, nr);
    __syncthreads();
    if (!ok) continue;
    for (int t = 0; t < (cnt + 1) / 2; ++t) {
      const u64* f = reinterpret_cast<const u64*>(s_f[t]);
      const u64 ph = add2(fma2(d0, f[kFHi], fma2(d1, f[kFHi + 1], mul2(d2, f[kFHi + 2]))),
                          fma2(d0, f[kFLo], fma2(d1, f[kFLo + 1], fma2(d2, f[kFLo + 2],
                               fma2(l0, f[kFHi], fma2(l1, f[kFHi + 1], mul2(l2, f[kFHi + 2])))))));
      const u64 mkdn2 = fma2(d0, f[kFN], fma2(d1, f[kFN + 1], mul2(d2, f[kFN + 2])));
      const u64 turns = turns2(ph);
      u64 cs, sn;
      sincos2(ph, turns, cs, sn);
      u64 Er = mul2(f[kFW], cs), Ei = mul2(f[kFW], sn);  // sum_q (w A / 4pi) e^{-ik d.y}
      if constexpr (NQ == 7) {
        const u64 a0 = fma2(d0, f[kFQ0], fma2(d1, f[kFQ0 + 1], mul2(d2, f[kFQ0 + 2])));
        const u64 a1 = fma2(d0, f[kFQ1], fma2(d1, f[kFQ1 + 1], mul2(d2, f[kFQ1 + 2])));
        const u64 am[3] = {a0, a1, sub2(bc(0.f), add2(a0, a1))};
#pragma unroll
        for (int o = 0; o < 2; ++o)
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            sincos2(fma2(bc(o == 0 ? 1.f : kOrbit), am[q], ph), turns, cs, sn);
            Er = fma2(f[kFW + 1 + o], cs, Er);
            Ei = fma2(f[kFW + 1 + o], sn, Ei);
          }
      }
      float er[2], ei[2], mkdn[2];
      upk(Er, er[0], er[1]);
      upk(Ei, ei[0], ei[1]);
      upk(mkdn2, mkdn[0], mkdn[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int s = 0; s < NR; ++s) {
          const float4 d = s_d[(2 * t + h) * NR + s];
          // a = p (-i k d.n) - g
          const float ar = fmaf(-mkdn[h], d.y, -d.z), ai = fmaf(mkdn[h], d.x, -d.w);
          accr[s] += ar * er[h] - ai * ei[h];
          acci[s] += ar * ei[h] + ai * er[h];
        }
    }
  }
  if (ok) {
#pragma unroll
    for (int s = 0; s < NR; ++s)
      part[((size_t)blockIdx.y * nd + qi) * NR + s] = make_double2(accr[s], acci[s]);
  }
}

// Training-sample coordinates (paper Sec. 3.4): theta = pi u0, phi = 2 pi u1,
// r = r_lo + (r_hi - r_lo) u2 about the centre; writes (theta, phi, r) and the Cartesian point.
__global__ void k_sample_points(const double* __restrict__ u, int64_t n, double cx, double cy, double cz,
                                double r_lo, double r_hi, double* __restrict__ coords,
                                double* __restrict__ pts) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double th = 3.14159265358979323846 * u[3 * i];
  const double ph = 6.28318530717958647692 * u[3 * i + 1];
  const double r = r_lo + (r_hi - r_lo) * u[3 * i + 2];
  double st, ct, sp, cp;
  sincos(th, &st, &ct);
  sincos(ph, &sp, &cp);
  coords[3 * i] = th;
  coords[3 * i + 1] = ph;
  coords[3 * i + 2] = r;
  pts[3 * i] = cx + r * st * cp;
  pts[3 * i + 1] = cy + r * st * sp;
  pts[3 * i + 2] = cz + r * ct;
}

// |p| of complex64 values
__global__ void k_abs(const float2* __restrict__ v, int64_t count, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) out[i] = hypotf(v[i].x, v[i].y);
}

// out[q, rhs0 + s] = sum over splits of the partials, complex64, column-major (m x nrhs). Bound by
// the latency of its FP64 chain: eight threads an output, each every eighth split, added in order
// (one thread took 12-22 us, a tenth of a small field's time).
__global__ void __launch_bounds__(256)
k_eval_reduce(const double2* __restrict__ part, int m, int splits, int nr, int stride, int rhs0,
              float2* __restrict__ out) {
  __shared__ double2 sh[8][32];
  const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const bool ok = i < (int64_t)m * nr;
  const int qi = ok ? (int)(i / nr) : 0, s = ok ? (int)(i % nr) : 0;
  double re = 0.0, im = 0.0;
#pragma unroll 4
  for (int t = threadIdx.y; t < splits; t += 8) {
    const double2 v = part[((size_t)t * m + qi) * stride + s];
    re += v.x;
    im += v.y;
  }
  sh[threadIdx.y][threadIdx.x] = make_double2(re, im);
  __syncthreads();
  if (threadIdx.y != 0 || !ok) return;
#pragma unroll
  for (int y = 1; y < 8; ++y) {
    re += sh[y][threadIdx.x].x;
    im += sh[y][threadIdx.x].y;
  }
  out[(size_t)(rhs0 + s) * m + qi] = make_float2((float)re, (float)im);
}

// Pass width for nr right-hand sides: the smallest of 1, 2, 4, 8, 16 that holds them. Each
// (point, element) kernel value is computed once per pass and applied to every RHS of it.
static int pass_width(int nr) { return nr <= 1 ? 1 : nr <= 2 ? 2 : nr <= 4 ? 4 : nr <= 8 ? 8 : 16; }
// The field kernel also takes passes of 32 RHS (64 accumulators a thread, 168 registers): each
// kernel value is then evaluated twice at 64 RHS instead of four times. A pass of 64 spills.
static int eval_pass_width(int nr) { return nr <= 16 ? pass_width(nr) : 32; }

// One k_eval launch for nr right-hand sides: seven quadrature points per element, or one
// sample point per Monte-Carlo sample (weight w / (4 pi) at offset 0). Partials are strided by
// pass_width(nr).
template <int NQ>
static void eval_launch_nq(int nr, dim3 grid, cudaStream_t s, const Geometry& g, int n,
                           const double* d_pts, int m, double k, const float2* d_p,
                           const float2* d_g, int r0, int per, double2* part) {
  switch (eval_pass_width(nr)) {
    case 1: k_eval<1, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
    case 2: k_eval<2, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
    case 4: k_eval<4, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
    case 8: k_eval<8, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
    case 16: k_eval<16, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
    default: k_eval<32, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, g.group, g.grid, n, d_pts, m, k, d_p, d_g, r0, nr, per, part); break;
  }
}

// The element records a field kernel sums over: seven points per element, or one point per
// record (Monte-Carlo samples; the quadrature points of a Galerkin op's elements, with the P1
// pressure and the P0 Neumann data expanded to them).
struct EvalSource {
  const Geometry* g;
  int n;
  bool one_point;
};

static void eval_launch(const EvalSource& src, double k, int nr, dim3 grid, cudaStream_t s, const double* d_pts,
                        int m, const float2* d_p, const float2* d_g, int r0, int per, double2* part) {
  if (src.one_point)
    eval_launch_nq<1>(nr, grid, s, *src.g, src.n, d_pts, m, k, d_p, d_g, r0, per, part);
  else
    eval_launch_nq<7>(nr, grid, s, *src.g, src.n, d_pts, m, k, d_p, d_g, r0, per, part);
}

static EvalSource eval_source(const nat_bem_op* op) {
  if (op->galerkin) return EvalSource{&op->gal.pts, (int)op->gal.pts.n, true};
  return EvalSource{&op->geo, (int)op->n, op->mc};
}

static nat_bem_status eval_core(const nat_bem_op* op, const double* d_pts, int64_t m,
                                const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                                cudaStream_t s);

nat_bem_status eval_impl(const nat_bem_op* op, const double* d_pts, int64_t m,
                         const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                         cudaStream_t s) {
  if (m == 0) return NAT_BEM_OK;
  if (!op->galerkin) return eval_core(op, d_pts, m, d_p, d_g, nrhs, d_out, s);
  float2 *pq = nullptr, *gq = nullptr;
  NB_TRY(galerkin_expand(op, d_p, d_g, nrhs, &pq, &gq, s));
  nat_bem_status st = eval_core(op, d_pts, m, pq, gq, nrhs, d_out, s);
  dev_free(pq, s);
  dev_free(gq, s);
  return st;
}

static nat_bem_status eval_core(const nat_bem_op* op, const double* d_pts, int64_t m,
                                const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                                cudaStream_t s) {
  const EvalSource src = eval_source(op);
  const int n = src.n;
  const int pblocks = (int)((m + kEvalThreads - 1) / kEvalThreads);
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // split the elements so that the grid holds about `bps` blocks per SM; the autotuner picks
  // bps among 4 (the default), 2, 8 and 16 per size class (elements, points, RHS pass)
  auto split_of = [&](int bps, int* per_out) {
    int splits = (bps * sms + pblocks - 1) / pblocks;
    splits = max(1, min(splits, (n + kElemStage - 1) / kElemStage));
    int per = (n + splits - 1) / splits;
    per = (per + kElemStage - 1) / kElemStage * kElemStage;
    *per_out = per;
    return (n + per - 1) / per;
  };
  static const int kBps[4] = {4, 2, 8, 16};
  int max_splits = 1, per = 0;
  for (int c = 0; c < 4; ++c) max_splits = max(max_splits, split_of(kBps[c], &per));
  double2* part = nullptr;
  NB_TRY(dev_alloc_n(&part, (size_t)max_splits * m * eval_pass_width(min(kEvalRhsPass, nrhs)), s));
  auto run = [&](int bps, int r0, int nr) -> nat_bem_status {
    int per_c = 0;
    const int splits = split_of(bps, &per_c);
    dim3 grid(pblocks, splits);
    NB_LAUNCH("eval", s, eval_launch(src, op->k, nr, grid, s, d_pts, (int)m, d_p, d_g, r0, per_c, part));
    NB_CHECK_LAUNCH();
    const int64_t tot = m * nr;
    NB_LAUNCH("eval_reduce", s, k_eval_reduce<<<(unsigned)((tot + 31) / 32), dim3(32, 8), 0, s>>>(part, (int)m, splits, nr, eval_pass_width(nr), r0, d_out));
    NB_CHECK_LAUNCH();
    return NAT_BEM_OK;
  };
  const int nr0 = min(kEvalRhsPass, nrhs);
  const int64_t cls = ((int64_t)((n + 1023) / 1024) << 32) | ((int64_t)((m + 255) / 256) << 8) |
                      ((int64_t)eval_pass_width(nr0) << 1) | (src.one_point ? 1 : 0);
  const int pick = autotune("eval_bps", cls, 4, [&](int c) { return run(kBps[c], 0, nr0); }, s);
  nat_bem_status st = NAT_BEM_OK;
  for (int r0 = 0; r0 < nrhs && st == NAT_BEM_OK; r0 += kEvalRhsPass)
    st = run(kBps[pick], r0, min(kEvalRhsPass, nrhs - r0));
  dev_free(part, s);
  return st;
}

template <int NQ>
static void far_launch_nq(int nr, dim3 grid, cudaStream_t s, const Geometry& g, int n,
                          const double* d_dirs, int nd, double k, const float2* d_p,
                          const float2* d_g, int r0, int per, double2* part) {
  switch (pass_width(nr)) {
    case 1: k_far_field<1, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, n, d_dirs, nd, k, d_p, d_g, r0, nr, per, part); break;
    case 2: k_far_field<2, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, n, d_dirs, nd, k, d_p, d_g, r0, nr, per, part); break;
    case 4: k_far_field<4, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, n, d_dirs, nd, k, d_p, d_g, r0, nr, per, part); break;
    case 8: k_far_field<8, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, n, d_dirs, nd, k, d_p, d_g, r0, nr, per, part); break;
    default: k_far_field<16, NQ><<<grid, kEvalThreads, 0, s>>>(g.c_hi, g.c_lo, g.nrm, g.qp, n, d_dirs, nd, k, d_p, d_g, r0, nr, per, part); break;
  }
}

static nat_bem_status far_field_core(const nat_bem_op* op, const double* d_dirs, int64_t nd,
                                     const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                                     cudaStream_t s);

nat_bem_status far_field_impl(const nat_bem_op* op, const double* d_dirs, int64_t nd,
                              const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                              cudaStream_t s) {
  if (nd == 0) return NAT_BEM_OK;
  if (!op->galerkin) return far_field_core(op, d_dirs, nd, d_p, d_g, nrhs, d_out, s);
  float2 *pq = nullptr, *gq = nullptr;
  NB_TRY(galerkin_expand(op, d_p, d_g, nrhs, &pq, &gq, s));
  nat_bem_status st = far_field_core(op, d_dirs, nd, pq, gq, nrhs, d_out, s);
  dev_free(pq, s);
  dev_free(gq, s);
  return st;
}

static nat_bem_status far_field_core(const nat_bem_op* op, const double* d_dirs, int64_t nd,
                                     const float2* d_p, const float2* d_g, int nrhs, float2* d_out,
                                     cudaStream_t s) {
  const EvalSource src = eval_source(op);
  const int n = src.n;
  const int pblocks = (int)((nd + kEvalThreads - 1) / kEvalThreads);
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int splits = (4 * sms + pblocks - 1) / pblocks;
  splits = max(1, min(splits, (n + kElemStage - 1) / kElemStage));
  int per = (n + splits - 1) / splits;
  per = (per + kElemStage - 1) / kElemStage * kElemStage;
  splits = (n + per - 1) / per;
  double2* part = nullptr;
  NB_TRY(dev_alloc_n(&part, (size_t)splits * nd * pass_width(min(kMaxRhsPass, nrhs)), s));
  for (int r0 = 0; r0 < nrhs; r0 += kMaxRhsPass) {
    const int nr = min(kMaxRhsPass, nrhs - r0);
    dim3 grid(pblocks, splits);
    if (src.one_point)
      NB_LAUNCH("far_field", s, far_launch_nq<1>(nr, grid, s, *src.g, n, d_dirs, (int)nd, op->k, d_p, d_g, r0, per, part));
    else
      NB_LAUNCH("far_field", s, far_launch_nq<7>(nr, grid, s, *src.g, n, d_dirs, (int)nd, op->k, d_p, d_g, r0, per, part));
    NB_CHECK_LAUNCH();
    const int64_t tot = nd * nr;
    NB_LAUNCH("eval_reduce", s, k_eval_reduce<<<(unsigned)((tot + 31) / 32), dim3(32, 8), 0, s>>>(part, (int)nd, splits, nr, pass_width(nr), r0, d_out));
    NB_CHECK_LAUNCH();
  }
  dev_free(part, s);
  return NAT_BEM_OK;
}

nat_bem_status sample_field_impl(const nat_bem_op* op, const double* d_u, int64_t n, const double* center,
                                 double r_lo, double r_hi, const float2* d_p, const float2* d_g, int nrhs,
                                 double* d_coords, float* d_amp, cudaStream_t s) {
  if (n == 0) return NAT_BEM_OK;
  double* pts = nullptr;
  float2* field = nullptr;
  NB_TRY(dev_alloc_n(&pts, (size_t)(3 * n), s));
  nat_bem_status st = dev_alloc_n(&field, (size_t)n * nrhs, s);
  if (st != NAT_BEM_OK) {
    dev_free(pts, s);
    return st;
  }
  NB_LAUNCH("sample_points", s, k_sample_points<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
      d_u, n, center[0], center[1], center[2], r_lo, r_hi, d_coords, pts));
  st = eval_impl(op, pts, n, d_p, d_g, nrhs, field, s);
  if (st == NAT_BEM_OK) {
    const int64_t tot = n * nrhs;
    NB_LAUNCH("sample_abs", s, k_abs<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(field, tot, d_amp));
    if (cudaGetLastError() != cudaSuccess) {
      set_error("sample_field: launch failed");
      st = NAT_BEM_ECUDA;
    }
  }
  dev_free(pts, s);
  dev_free(field, s);
  return st;
}


// ------------------------------------------------------------- allocation-free variant
// Field evaluation for callers that must not allocate device memory: code running where
// cudaMalloc is off limits (inside another allocator's callback, under a memory budget that
// a framework enforces, or in a process whose device memory is owned by someone else). The
// per-split partial sums that eval_impl takes from the memory pool live instead in this fixed
// array, which every GPU that loads the library holds until the process exits.
constexpr size_t kNoAllocScratch = (size_t)1 << 18;  // double2 entries: 4 MiB
static __device__ __align__(256) double2 g_eval_scratch[kNoAllocScratch];
constexpr int64_t kNoAllocMaxPoints = (int64_t)(kNoAllocScratch / kNoAllocRhsPass);  // 65,536

namespace {
std::mutex g_scratch_mu;
void* g_scratch_ptr[64] = {};
}  // namespace

// Device address of g_eval_scratch on the current device, looked up once per device (host
// code cannot use the symbol itself: on the host it names a stand-in, not device memory). The
// address is kept for the life of the process, so the library must not be used across a
// cudaDeviceReset (which would also invalidate every op).
static nat_bem_status scratch_address(double2** out) {
  int dev = 0;
  NB_TRY_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("device ordinal out of range");
    return NAT_BEM_ECUDA;
  }
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_eval_scratch);
    if (e != cudaSuccess || !p) {
      set_error(std::string("cudaGetSymbolAddress(g_eval_scratch) failed: ") + cudaGetErrorString(e));
      return NAT_BEM_ECUDA;
    }
    g_scratch_ptr[dev] = p;
  }
  *out = static_cast<double2*>(g_scratch_ptr[dev]);
  return NAT_BEM_OK;
}

static nat_bem_status eval_noalloc_impl(const nat_bem_op* op, const double* d_pts, int64_t m,
                                        const float2* d_p, const float2* d_g, int nrhs,
                                        float2* d_out, cudaStream_t s) {
  double2* part = nullptr;
  NB_TRY(scratch_address(&part));
  const int n = (int)op->n;
  const int pblocks = (int)((m + kEvalThreads - 1) / kEvalThreads);
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // as many element splits as eval_impl would take, capped by the scratch size
  int splits = (4 * sms + pblocks - 1) / pblocks;
  splits = max(1, min(splits, (n + kElemStage - 1) / kElemStage));
  const int cap = (int)(kNoAllocScratch / ((size_t)m * kNoAllocRhsPass));
  splits = max(1, min(splits, cap));
  int per = (n + splits - 1) / splits;
  per = (per + kElemStage - 1) / kElemStage * kElemStage;
  splits = (n + per - 1) / per;
  for (int r0 = 0; r0 < nrhs; r0 += kNoAllocRhsPass) {
    const int nr = min(kNoAllocRhsPass, nrhs - r0);
    dim3 grid(pblocks, splits);
    NB_LAUNCH("eval", s, eval_launch(eval_source(op), op->k, nr, grid, s, d_pts, (int)m, d_p, d_g, r0, per, part));
    NB_CHECK_LAUNCH();
    const int64_t tot = m * nr;
    NB_LAUNCH("eval_reduce", s, k_eval_reduce<<<(unsigned)((tot + 31) / 32), dim3(32, 8), 0, s>>>(part, (int)m, splits, nr, eval_pass_width(nr), r0, d_out));
    NB_CHECK_LAUNCH();
  }
  return NAT_BEM_OK;
}

}  // namespace natbem

extern "C" nat_bem_status nat_bem_eval_noalloc(const nat_bem_op* op, const double* pts, int64_t m,
                                               const float* p, const float* neumann, int32_t nrhs,
                                               float* field_out, void* cuda_stream) {
  using namespace natbem;
  try {
    clear_error();
    if (!op || m < 0 || nrhs < 1 || (m > 0 && (!pts || !p || !neumann || !field_out))) {
      set_error("nat_bem_eval_noalloc: bad arguments (op NULL, m < 0, nrhs < 1 or NULL arrays)");
      return NAT_BEM_EINVAL;
    }
    if (m > kNoAllocMaxPoints) {
      set_error("nat_bem_eval_noalloc: m = " + std::to_string(m) + " exceeds the maximum of " +
                std::to_string(kNoAllocMaxPoints) + " points per call (split the points)");
      return NAT_BEM_EINVAL;
    }
    if (op->galerkin) {
      set_error("nat_bem_eval_noalloc: Galerkin ops need scratch for the P1 expansion: use nat_bem_eval");
      return NAT_BEM_EINVAL;
    }
    if (m == 0) return NAT_BEM_OK;
    if (!is_device_pointer(pts) || !is_device_pointer(p) || !is_device_pointer(neumann) ||
        !is_device_pointer(field_out)) {
      set_error("nat_bem_eval_noalloc: pts, p, neumann and field_out must be device pointers");
      return NAT_BEM_EINVAL;
    }
    return eval_noalloc_impl(op, pts, m, reinterpret_cast<const float2*>(p),
                             reinterpret_cast<const float2*>(neumann), nrhs,
                             reinterpret_cast<float2*>(field_out), (cudaStream_t)cuda_stream);
  } catch (...) {
    set_error("internal error in nat_bem_eval_noalloc");
    return NAT_BEM_ECUDA;
  }
}
