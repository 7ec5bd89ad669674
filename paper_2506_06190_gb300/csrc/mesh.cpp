// Host-side mesh checks and the list of element pairs integrated in FP64 (self pairs and
// pairs that share a vertex). The boundary integral equation of Sec. 4, Eq. 6 needs a closed
// surface with outward normals; this file rejects anything else before device work starts.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "internal.h"

namespace natbem {

namespace {

struct V3 {
  double x, y, z;
};
V3 vget(const double* V, int32_t i) { return {V[3 * i], V[3 * i + 1], V[3 * i + 2]}; }
V3 vsub(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
V3 vcross(V3 a, V3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
double vdot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

}  // namespace

float split_grid(const double* lo, const double* hi) {
  double reach = 0.0;
  for (int d = 0; d < 3; ++d)
    reach = std::max(reach, std::max(std::fabs(lo[d]), std::fabs(hi[d])) + 4.0 * (hi[d] - lo[d]));
  int e = 0;
  std::frexp(std::min(std::max(reach, 1e-36), 1e36), &e);  // reach < 2^e
  return std::ldexp(3.f, e);
}

nat_bem_status validate_mesh_host(const double* V, int64_t nv, const int32_t* T, int64_t nt, float* grid) {
  if (nv <= 0 || nt <= 0) {
    set_error("mesh: need nv > 0 and nt > 0");
    return NAT_BEM_EINVAL;
  }
  if (nt > (int64_t)1 << 30 || nv > (int64_t)1 << 30) {
    set_error("mesh: too many vertices or triangles");
    return NAT_BEM_EINVAL;
  }
  for (int64_t i = 0; i < 3 * nv; ++i)
    if (!std::isfinite(V[i])) {
      set_error("mesh: non-finite vertex coordinate at vertex " + std::to_string(i / 3));
      return NAT_BEM_EINVAL;
    }
  for (int64_t i = 0; i < 3 * nt; ++i)
    if (T[i] < 0 || T[i] >= nv) {
      set_error("mesh: vertex index out of range in triangle " + std::to_string(i / 3));
      return NAT_BEM_EINVAL;
    }
  double vol6 = 0.0;
  for (int64_t t = 0; t < nt; ++t) {
    const int32_t* f = T + 3 * t;
    V3 a = vget(V, f[0]), b = vget(V, f[1]), c = vget(V, f[2]);
    V3 cr = vcross(vsub(b, a), vsub(c, a));
    if (!(vdot(cr, cr) > 0.0)) {
      set_error("mesh: zero-area triangle " + std::to_string(t));
      return NAT_BEM_EINVAL;
    }
    vol6 += vdot(a, vcross(b, c));
  }
  // every directed edge exactly once, and its reverse exactly once (closed, consistently
  // oriented, two triangles per edge): the edges leaving each vertex, sorted by their ends. (A hash
  // map of the edges took 3 ms of a 10,000-triangle assembly; this takes 0.2.)
  std::vector<int32_t> first(nv + 1, 0);
  for (int64_t i = 0; i < 3 * nt; ++i) first[T[i] + 1]++;
  for (int64_t v = 0; v < nv; ++v) first[v + 1] += first[v];
  std::vector<int32_t> to(3 * nt), fill(first.begin(), first.end() - 1);
  for (int64_t t = 0; t < nt; ++t)
    for (int e = 0; e < 3; ++e) to[fill[T[3 * t + e]]++] = T[3 * t + (e + 1) % 3];
  for (int64_t v = 0; v < nv; ++v) {
    int32_t *lo = &to[0] + first[v], *hi = &to[0] + first[v + 1];
    if (hi - lo <= 16) {
      for (int32_t* p = lo; p < hi; ++p)  // insertion sort of a few ends
        for (int32_t* q = p; q > lo && q[-1] > q[0]; --q) std::swap(q[-1], q[0]);
    } else {
      std::sort(lo, hi);
    }
    for (int32_t* p = lo; p + 1 < hi; ++p)
      if (p[0] == p[1]) {
        set_error("mesh: directed edge used twice (inconsistent orientation or non-manifold) "
                  "at vertex " + std::to_string(v));
        return NAT_BEM_EINVAL;
      }
  }
  for (int64_t v = 0; v < nv; ++v)
    for (int32_t q = first[v]; q < first[v + 1]; ++q)
      if (!std::binary_search(to.begin() + first[to[q]], to.begin() + first[to[q] + 1], (int32_t)v)) {
        set_error("mesh: not closed (an edge has a single triangle)");
        return NAT_BEM_EINVAL;
      }
  if (!(vol6 > 0.0)) {
    set_error("mesh: enclosed volume is not positive (inward winding)");
    return NAT_BEM_EINVAL;
  }
  if (!grid) return NAT_BEM_OK;
  double lo[3] = {HUGE_VAL, HUGE_VAL, HUGE_VAL}, hi[3] = {-HUGE_VAL, -HUGE_VAL, -HUGE_VAL};
  for (int64_t v = 0; v < nv; ++v)
    if (first[v + 1] > first[v])  // the triangles' vertices
      for (int d = 0; d < 3; ++d) {
        lo[d] = std::min(lo[d], V[3 * v + d]);
        hi[d] = std::max(hi[d], V[3 * v + d]);
      }
  *grid = split_grid(lo, hi);
  return NAT_BEM_OK;
}

void build_near_pairs(const int32_t* T, int64_t nv, int64_t nt, std::vector<int2>& pairs) {
  // vertex -> incident triangles (CSR)
  std::vector<int32_t> deg(nv + 1, 0);
  for (int64_t i = 0; i < 3 * nt; ++i) deg[T[i] + 1]++;
  for (int64_t v = 0; v < nv; ++v) deg[v + 1] += deg[v];
  std::vector<int32_t> inc(3 * nt), fill(deg.begin(), deg.end() - 1);
  for (int64_t t = 0; t < nt; ++t)
    for (int e = 0; e < 3; ++e) inc[fill[T[3 * t + e]]++] = (int32_t)t;
  pairs.clear();
  pairs.reserve((size_t)nt * 14);
  for (int64_t t = 0; t < nt; ++t) {
    // the three vertices' triangle lists are increasing: their union by merging
    const int32_t* p[3];
    const int32_t* end[3];
    for (int e = 0; e < 3; ++e) {
      const int32_t v = T[3 * t + e];
      p[e] = &inc[0] + deg[v];
      end[e] = &inc[0] + deg[v + 1];
    }
    for (;;) {
      int32_t j = INT32_MAX;
      for (int e = 0; e < 3; ++e)
        if (p[e] < end[e] && *p[e] < j) j = *p[e];
      if (j == INT32_MAX) break;
      for (int e = 0; e < 3; ++e)
        while (p[e] < end[e] && *p[e] == j) ++p[e];
      if (j != t) pairs.push_back(make_int2((int)t, j));  // the self pair has its own kernel
    }
  }
}

}  // namespace natbem
