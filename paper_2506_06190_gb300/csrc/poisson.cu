// Poisson-disk surface sampling for the Monte-Carlo BEM (paper Sec. 4.2: samples that cover the
// surface evenly, drawn in parallel on the GPU after Bowers et al. 2010).
//
//   candidates  per draw (u0, u1, u2): the triangle whose cumulative-area interval holds
//               u0 * A, the point with barycentric (1 - sqrt(u1), sqrt(u1)(1 - u2), sqrt(u1) u2);
//               pushed onto its grid cell's list (cell size h = r / sqrt(3): one sample per cell)
//   27 phases   (i, j, k) mod 3; every cell of a phase accepts its lowest-index candidate with
//               no accepted sample closer than r in the 5 x 5 x 5 cells around it. Cells of one
//               phase are three or more cells apart, so a phase runs its cells in parallel and
//               the result equals the sequential definition, whatever the list order.
//
// The phases are a chain of 27 dependent steps of a few hundred cells each: latency, not work.
// They run in one cooperative launch (k_ps_run), a warp per cell. A warp fetches what does not
// depend on other cells (its candidates, the occupied neighbour cells of earlier phases) before
// it waits for the earlier phases' cells to be counted done, so a step costs one counter round
// trip, one load of the neighbours' samples and the tests. Those run in FP32 on coordinates
// scaled by 1/r and carried as hi/lo pairs; a distance too near r for that is tested again in
// FP64, so every decision is the FP64 one (an FP64 warp instruction takes about 76 cycles, and
// a cell needs a hundred). The samples' order and copies follow in the same launch.
// FP64 with explicit round-to-nearest intrinsics (no contraction), so candidate positions and
// the distance tests are the same on every machine.
//
// 32,768 draws on 10240 triangles: 27 launches of 27 us (725 us) before, one of 100 us now; a whole
// call 1000 -> 273 us (areas, checks and compaction moved to the device, one allocation).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"

namespace natbem {

namespace {
constexpr int64_t kPsMaxCells = (int64_t)1 << 28;

__device__ __forceinline__ double dm(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double da(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double ds(double a, double b) { return __dsub_rn(a, b); }
}  // namespace

struct PsGrid {
  double lox, loy, loz, h;
  int nx, ny, nz;
};

__device__ __forceinline__ int ps_clamp(int v, int n) { return v < 0 ? 0 : v >= n ? n - 1 : v; }

constexpr int kPsStripes = 8;

// Device scalars of a call.
struct PsInfo {
  unsigned long long lo[3], hi[3];  // bounding box (order-preserving bits)
  int bad_index;                    // a triangle index is out of range
  int bad_tri;                      // first degenerate triangle (nt: none)
  int nan_box;                      // the first vertex holds a NaN
  int n_occ;                        // occupied cells
  int phase_n[27], phase_fill[27];  // occupied cells per phase; scattered so far
  unsigned bar;                     // grid barrier arrivals
  int err;                          // a bounded wait gave up
  int count;                        // accepted samples
  unsigned beat;                    // batches of candidates looked at in long lists
  unsigned done[kPsStripes][32];    // cells decided, counted on several cache lines
};

// Bits of a double in an order-preserving unsigned form.
__device__ __forceinline__ unsigned long long ps_order(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u >> 63) ? ~u : u | 0x8000000000000000ull;
}

// Twice the area vector of triangle t; returns its area.
__device__ __forceinline__ double ps_area(const double* __restrict__ V, const int32_t* __restrict__ T, int t,
                                          double (&cr)[3]) {
  const double* a = V + 3 * (size_t)T[3 * (size_t)t];
  const double* b = V + 3 * (size_t)T[3 * (size_t)t + 1];
  const double* c = V + 3 * (size_t)T[3 * (size_t)t + 2];
  const double e1[3] = {ds(b[0], a[0]), ds(b[1], a[1]), ds(b[2], a[2])};
  const double e2[3] = {ds(c[0], a[0]), ds(c[1], a[1]), ds(c[2], a[2])};
  cr[0] = ds(dm(e1[1], e2[2]), dm(e1[2], e2[1]));
  cr[1] = ds(dm(e1[2], e2[0]), dm(e1[0], e2[2]));
  cr[2] = ds(dm(e1[0], e2[1]), dm(e1[1], e2[0]));
  return dm(0.5, __dsqrt_rn(da(da(dm(cr[0], cr[0]), dm(cr[1], cr[1])), dm(cr[2], cr[2]))));
}

__global__ void k_ps_init(PsInfo* __restrict__ info, int nt) {
  for (int i = threadIdx.x; i < (int)(sizeof(PsInfo) / 4); i += blockDim.x) reinterpret_cast<int*>(info)[i] = 0;
  __syncthreads();
  if (threadIdx.x < 3) info->lo[threadIdx.x] = ~0ull;
  if (threadIdx.x == 0) info->bad_tri = nt;
}

// Areas of the triangles, the vertices' bounding box, and the mesh checks.
__global__ void __launch_bounds__(256) k_ps_mesh(const double* __restrict__ V, int64_t nv, const int32_t* __restrict__ T,
                                                 int nt, double* __restrict__ area, PsInfo* __restrict__ info) {
  __shared__ unsigned long long s_lo[3], s_hi[3];
  if (threadIdx.x < 3) {
    s_lo[threadIdx.x] = ~0ull;
    s_hi[threadIdx.x] = 0ull;
  }
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t t = first; t < nt; t += stride) {
    const int a = T[3 * t], b = T[3 * t + 1], c = T[3 * t + 2];
    if (a < 0 || a >= nv || b < 0 || b >= nv || c < 0 || c >= nv) {
      info->bad_index = 1;
      continue;
    }
    double cr[3];
    const double A = ps_area(V, T, (int)t, cr);
    area[t] = A;
    if (!(A > 0.0) || !isfinite(A)) atomicMin(&info->bad_tri, (int)t);
  }
  unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
  for (int64_t v = first; v < nv; v += stride)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double x = V[3 * v + d];
      if (x != x) {  // only a NaN in the first vertex enters the box
        if (v == 0) info->nan_box = 1;
        continue;
      }
      lo[d] = min(lo[d], ps_order(x));
      hi[d] = max(hi[d], ps_order(x));
    }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
      hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
    }
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&s_lo[d], lo[d]);
      atomicMax(&s_hi[d], hi[d]);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    atomicMin(&info->lo[threadIdx.x], s_lo[threadIdx.x]);
    atomicMax(&info->hi[threadIdx.x], s_hi[threadIdx.x]);
  }
}

// Candidate i: its triangle, position and scaled coordinates, and the push onto its cell's list.
__global__ void __launch_bounds__(256) k_ps_candidates(const double* __restrict__ V, const int32_t* __restrict__ T,
                                                       const double* __restrict__ cum, int nt,
                                                       const double* __restrict__ u, int m, PsGrid g, double rinv,
                                                       double* __restrict__ x, int* __restrict__ tri,
                                                       float4* __restrict__ hi4, float4* __restrict__ lo4,
                                                       int* __restrict__ head, int* __restrict__ next,
                                                       int* __restrict__ occ, PsInfo* __restrict__ info) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const double u0 = u[3 * (size_t)i], u1 = u[3 * (size_t)i + 1], u2 = u[3 * (size_t)i + 2];
  // first triangle with cumulative area > u0 * A
  const double v = dm(u0, cum[nt - 1]);
  int lo = 0, hi = nt;  // answer in [lo, hi]
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (cum[mid] > v) hi = mid;
    else lo = mid + 1;
  }
  const int t = min(lo, nt - 1);
  const double* a = V + 3 * (size_t)T[3 * (size_t)t];
  const double* b = V + 3 * (size_t)T[3 * (size_t)t + 1];
  const double* c = V + 3 * (size_t)T[3 * (size_t)t + 2];
  const double s = __dsqrt_rn(u1);
  const double b0 = ds(1.0, s), b1 = dm(s, ds(1.0, u2)), b2 = dm(s, u2);
  const double org[3] = {g.lox, g.loy, g.loz};
  double p[3];
  float h[3], l[3];
  bool far = false;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    p[d] = da(da(dm(b0, a[d]), dm(b1, b[d])), dm(b2, c[d]));
    x[3 * (size_t)i + d] = p[d];
    const double q = dm(ds(p[d], org[d]), rinv);
    h[d] = (float)q;
    l[d] = (float)ds(q, (double)h[d]);
    far = far || !(fabsf(h[d]) < 134217728.f);  // beyond the pairs' accuracy: always tested in FP64
  }
  if (far) h[0] = nanf("");
  tri[i] = t;
  hi4[i] = make_float4(h[0], h[1], h[2], 0.f);
  lo4[i] = make_float4(l[0], l[1], l[2], 0.f);
  const int ci = ps_clamp((int)floor(__ddiv_rn(ds(p[0], g.lox), g.h)), g.nx);
  const int cj = ps_clamp((int)floor(__ddiv_rn(ds(p[1], g.loy), g.h)), g.ny);
  const int ck = ps_clamp((int)floor(__ddiv_rn(ds(p[2], g.loz), g.h)), g.nz);
  const int cell = (ci * g.ny + cj) * g.nz + ck;  // at most 2^28 cells
  const int prev = atomicExch(&head[cell], i);
  next[i] = prev;
  if (prev < 0) {  // first candidate of the cell: list the cell once
    occ[atomicAdd(&info->n_occ, 1)] = cell;
    atomicAdd(&info->phase_n[(ci % 3) * 9 + (cj % 3) * 3 + ck % 3], 1);
  }
}

// Eight warps of a block decide cells; a ninth polls the counters for all of them (a poll per
// warp, 1216 on one address, took 9 us a phase).
constexpr int kPsWorkers = 8;
constexpr int kPsThreads = kPsWorkers * 32 + 32;
// A scaled squared distance outside 1 +- this is decided in FP32: coordinates below 2^27 as hi/lo
// pairs carry 2^-21 or better, a difference rounds at 2^-24, so d^2 is off by less than 4e-6.
constexpr float kPsUnsure = 2e-5f;

__device__ __forceinline__ unsigned ps_load(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ps_peek(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ps_count(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
// Whether two seconds have passed since t0 (0: from now on).
__device__ __forceinline__ bool ps_late(uint64_t& t0) {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  if (t0 == 0) t0 = t;
  return t - t0 > 2000000000ull;
}
// One thread: waits until *p >= target, at most two seconds (then the error word is set).
__device__ __forceinline__ bool ps_wait(const unsigned* p, unsigned target, int* err) {
  uint64_t t0 = 0;
  for (unsigned it = 1;; ++it) {
    if (ps_load(p) >= target) return true;
    if ((it & 255u) == 0u && ps_late(t0)) {
      atomicOr(err, 1);
      return false;
    }
  }
}

// The phases, and the accepted samples in increasing index (cooperative launch: warps wait on
// cells that other warps decide). slot: two float4 per candidate, the sample of the cell whose
// list starts at that candidate (scaled hi with the index in w, or -1; scaled lo). flag: accepted
// candidates. part: accepted per block. Samples go to idx and, when at most cap, pts and nrm.
__global__ void __launch_bounds__(kPsThreads)
k_ps_run(PsGrid g, double r2, const double* __restrict__ V, const int32_t* __restrict__ T, const double* __restrict__ x,
         const int* __restrict__ tri, const float4* __restrict__ hi4, const float4* __restrict__ lo4, int m,
         const int* __restrict__ head, const int* __restrict__ next, const int* __restrict__ occ,
         int* __restrict__ list, float4* __restrict__ slot, unsigned char* __restrict__ flag, int* __restrict__ part,
         int64_t cap, int64_t* __restrict__ idx, double* __restrict__ pts, double* __restrict__ nrm,
         PsInfo* __restrict__ info) {
  __shared__ int s_off[28], s_nb[kPsWorkers][128], s_warp[kPsThreads / 32];
  __shared__ int s_base;
  __shared__ volatile int s_bad, s_done;  // given up; cells known to be decided
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int G = gridDim.x;
  const int n = info->n_occ;
  if (tid == 0) {
    s_bad = 0;
    s_done = 0;
    int t = 0;
    for (int p = 0; p < 27; ++p) {
      s_off[p] = t;
      t += info->phase_n[p];
    }
    s_off[27] = t;
  }
  __syncthreads();
  auto phase_of = [&](int cell) {
    const int k = cell % g.nz, q = cell / g.nz;
    return (q / g.ny % 3) * 9 + (q % g.ny % 3) * 3 + k % 3;
  };
  auto barrier = [&](unsigned target) {
    __syncthreads();
    if (tid == 0) {
      ps_count(&info->bar);
      if (!ps_wait(&info->bar, target, &info->err)) s_bad = 1;
    }
    __syncthreads();
    return s_bad == 0;
  };
  // cells in phase order
  for (int i = blockIdx.x * kPsThreads + tid; i < n; i += G * kPsThreads) {
    const int cell = occ[i], p = phase_of(cell);
    list[s_off[p] + atomicAdd(&info->phase_fill[p], 1)] = cell;
  }
  if (!barrier((unsigned)G)) return;
  if (w == kPsWorkers) {
    // the counters' sum for the block's warps, until every cell is decided; gives up when for two
    // seconds no cell was decided and no long list advanced
    uint64_t t0 = 0;
    unsigned seen = 0u, last = 0u, still = 0u;
    for (unsigned it = 1; s_done < n && !s_bad; ++it) {
      // An acquiring load empties the SM's L1, which a warp on a long list walks from (172 ns a
      // candidate, 64 without): after a while without news the polls are relaxed ones, and a fence
      // acquires what they find.
      const bool quiet = still >= 64u;
      unsigned v = lane >= kPsStripes ? 0u : quiet ? ps_peek(&info->done[lane][0]) : ps_load(&info->done[lane][0]);
      v = __reduce_add_sync(0xffffffffu, v);
      if (quiet && v != last) __threadfence();
      still = v == last ? still + 1u : 0u;
      last = v;
      if (lane == 0) {
        __threadfence_block();
        s_done = (int)v;
        if ((it & 255u) == 0u) {
          const unsigned now = v + ps_peek(&info->beat);
          if (now != seen) t0 = 0;
          seen = now;
          if (ps_late(t0)) {
            atomicOr(&info->err, 1);
            s_bad = 1;
          }
        }
      }
      __syncwarp();
    }
  }
  int phase = 0;
  for (int i = blockIdx.x + G * w; w < kPsWorkers && i < n; i += G * kPsWorkers) {  // a phase's cells on different SMs
    const int cell = __ldcg(list + i);
    while (i >= s_off[phase + 1]) ++phase;
    const int cz = cell % g.nz, cy = cell / g.nz % g.ny, cx = cell / g.nz / g.ny;
    // occupied neighbour cells of earlier phases
    int nb = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = lane + 32 * q;
      int h = -1;
      if (t < 125) {
        const int a = cx + t / 25 - 2, b = cy + (t / 5) % 5 - 2, c = cz + t % 5 - 2;
        if (a >= 0 && a < g.nx && b >= 0 && b < g.ny && c >= 0 && c < g.nz &&
            (a % 3) * 9 + (b % 3) * 3 + c % 3 < phase)
          h = head[(a * g.ny + b) * g.nz + c];
      }
      const unsigned got = __ballot_sync(0xffffffffu, h >= 0);
      if (h >= 0) s_nb[w][nb + __popc(got & ((1u << lane) - 1u))] = h;
      nb += __popc(got);
    }
    // up to 32 candidates, one a lane
    const int first = head[cell];
    int nxt = first, mine = -1, cnt = 0;
    for (; cnt < 32 && nxt >= 0; ++cnt) {
      if (lane == cnt) mine = nxt;
      nxt = next[nxt];
    }
    float4 mh = make_float4(0.f, 0.f, 0.f, 0.f), ml = mh;
    if (mine >= 0) {
      mh = hi4[mine];
      ml = lo4[mine];
    }
    __syncwarp();
    while (s_done < s_off[phase] && !s_bad) {
    }
    __threadfence_block();
    __syncwarp();
    if (s_bad) break;
    // the neighbours' samples, up to four a lane
    float4 sh[4], sl[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sh[q].w = __int_as_float(-1);
      if (lane + 32 * q < nb) {
        const float4* sp = slot + 2 * (size_t)s_nb[w][lane + 32 * q];
        sh[q] = __ldcg(sp);
        sl[q] = __ldcg(sp + 1);
      }
    }
    int best = -1;
    float4 bh = mh, bl = ml;
    for (unsigned batch = 1; cnt > 0; ++batch) {
      if ((batch & 31u) == 0u && lane == 0) ps_count(&info->beat);
      // the candidates below the best one yet, in list order
      unsigned todo = __ballot_sync(0xffffffffu, mine >= 0 && (best < 0 || mine < best));
      while (todo) {
        const int c = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int ci = __shfl_sync(0xffffffffu, mine, c);
        const float hx = __shfl_sync(0xffffffffu, mh.x, c), hy = __shfl_sync(0xffffffffu, mh.y, c),
                    hz = __shfl_sync(0xffffffffu, mh.z, c);
        const float lx = __shfl_sync(0xffffffffu, ml.x, c), ly = __shfl_sync(0xffffffffu, ml.y, c),
                    lz = __shfl_sync(0xffffffffu, ml.z, c);
        bool near = false, unsure = false;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (__float_as_int(sh[q].w) >= 0) {
            const float dx = (hx - sh[q].x) + (lx - sl[q].x), dy = (hy - sh[q].y) + (ly - sl[q].y),
                        dz = (hz - sh[q].z) + (lz - sl[q].z);
            const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (d2 < 1.f - kPsUnsure) near = true;
            else if (!(d2 > 1.f + kPsUnsure)) unsure = true;
          }
        if (__any_sync(0xffffffffu, near)) continue;
        if (__any_sync(0xffffffffu, unsure)) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int si = __float_as_int(sh[q].w);
            if (si >= 0) {
              const double *xi = x + 3 * (size_t)ci, *xs = x + 3 * (size_t)si;
              const double dx = ds(xi[0], xs[0]), dy = ds(xi[1], xs[1]), dz = ds(xi[2], xs[2]);
              if (da(da(dm(dx, dx), dm(dy, dy)), dm(dz, dz)) < r2) near = true;
            }
          }
          if (__any_sync(0xffffffffu, near)) continue;
        }
        best = ci;
        bh = make_float4(hx, hy, hz, __int_as_float(ci));
        bl = make_float4(lx, ly, lz, 0.f);
        todo &= __ballot_sync(0xffffffffu, mine < best);
      }
      mine = -1;  // the next 32 of a longer list
      for (cnt = 0; cnt < 32 && nxt >= 0; ++cnt) {
        if (lane == cnt) mine = nxt;
        nxt = next[nxt];
      }
      if (mine >= 0 && (best < 0 || mine < best)) {
        mh = hi4[mine];
        ml = lo4[mine];
      }
    }
    if (lane == 0) {
      if (best >= 0) {
        __stcg(slot + 2 * (size_t)first, bh);
        __stcg(slot + 2 * (size_t)first + 1, bl);
        flag[best] = 1;
      }
      ps_count(&info->done[blockIdx.x % kPsStripes][0]);
    }
  }
  // accepted candidates in increasing index: a contiguous range per block
  __syncthreads();
  if (s_bad) return;
  const int64_t per = ((int64_t)m + G - 1) / G, q0 = min((int64_t)m, blockIdx.x * per), q1 = min((int64_t)m, q0 + per);
  int mineN = 0;
  for (int64_t q = q0 + tid; q < q1; q += kPsThreads) mineN += __ldcg(flag + q);
  mineN = __reduce_add_sync(0xffffffffu, mineN);
  if (lane == 0) s_warp[w] = mineN;
  __syncthreads();
  if (tid == 0) {
    int t = 0;
    for (int q = 0; q < kPsThreads / 32; ++q) t += s_warp[q];
    __stcg(part + blockIdx.x, t);
  }
  if (!barrier(2u * (unsigned)G)) return;
  if (w == 0) {
    int before = 0, all = 0;
    for (int q = lane; q < G; q += 32) {
      const int c = __ldcg(part + q);
      all += c;
      if (q < (int)blockIdx.x) before += c;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    all = __reduce_add_sync(0xffffffffu, all);
    if (lane == 0) {
      s_base = before;
      s_off[0] = all;
      if (blockIdx.x == 0) info->count = all;
    }
  }
  __syncthreads();
  const bool fits = s_off[0] <= cap;
  int base = s_base;
  for (int64_t r = q0; r < q1; r += kPsThreads) {  // uniform over the block
    const int64_t q = r + tid;
    const bool take = q < q1 && __ldcg(flag + q);
    const unsigned got = __ballot_sync(0xffffffffu, take);
    __syncthreads();
    if (lane == 0) s_warp[w] = __popc(got);
    __syncthreads();
    int at = base, tot = 0;
    for (int o = 0; o < kPsThreads / 32; ++o) {
      at += o < w ? s_warp[o] : 0;
      tot += s_warp[o];
    }
    at += __popc(got & ((1u << lane) - 1u));
    base += tot;
    if (take && at < cap) idx[at] = q;
    if (take && fits) {
      double cr[3];
      const double twoA = dm(2.0, ps_area(V, T, tri[q], cr));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        pts[3 * (size_t)at + d] = x[3 * (size_t)q + d];
        nrm[3 * (size_t)at + d] = __ddiv_rn(cr[d], twoA);
      }
    }
  }
}

}  // namespace natbem

using namespace natbem;

extern "C" nat_bem_status nat_bem_poisson_sample(const double* verts, int64_t nv, const int32_t* tris, int64_t nt,
                                                 double radius, const double* u, int64_t m, int64_t cap,
                                                 int64_t* idx_out, double* pts_out, double* normals_out,
                                                 int64_t* count, void* cuda_stream) {
  try {
    clear_error();
    if (!verts || !tris || !u || !count || nv <= 0 || nt <= 0 || m < 0 || cap < 0 ||
        m > ((int64_t)1 << 31) - 1 || nt > ((int64_t)1 << 31) - 1 || !(radius > 0.0) || !std::isfinite(radius) ||
        (cap > 0 && (!pts_out || !normals_out))) {
      set_error("nat_bem_poisson_sample: bad arguments");
      return NAT_BEM_EINVAL;
    }
    *count = 0;
    if (m == 0) return NAT_BEM_OK;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // mesh and draws on the device, then one block of scratch for the whole call
    const double *dV = nullptr, *du = nullptr;
    const int32_t* dT = nullptr;
    double *tV = nullptr, *tu = nullptr;
    int32_t* tT = nullptr;
    char *mesh = nullptr, *scratch = nullptr;
    auto cleanup = [&]() {
      void* ptrs[] = {tV, tT, tu, mesh, scratch};
      for (void* p : ptrs)
        if (p) dev_free(p, s);
    };
    auto failed = [&](nat_bem_status st) {
      cleanup();
      return st;
    };
    auto cuda_failed = [&](cudaError_t e) {
      set_error(std::string("nat_bem_poisson_sample: ") + cudaGetErrorString(e));
      return failed(NAT_BEM_ECUDA);
    };
    nat_bem_status st = to_device(verts, (size_t)(3 * nv), s, &dV, &tV);
    if (st == NAT_BEM_OK) st = to_device(tris, (size_t)(3 * nt), s, &dT, &tT);
    if (st == NAT_BEM_OK) st = to_device(u, (size_t)(3 * m), s, &du, &tu);
    // areas, then their running sums; scalars
    const size_t info_at = ((size_t)nt * sizeof(double) + 255) / 256 * 256;
    if (st == NAT_BEM_OK) st = dev_alloc_n(&mesh, info_at + sizeof(PsInfo), s);
    if (st != NAT_BEM_OK) return failed(st);
    double* dcum = reinterpret_cast<double*>(mesh);
    PsInfo* info = reinterpret_cast<PsInfo*>(mesh + info_at);
    NB_LAUNCH("ps_init", s, k_ps_init<<<1, 128, 0, s>>>(info, (int)nt));
    NB_LAUNCH("ps_mesh", s, k_ps_mesh<<<(unsigned)std::min<int64_t>((std::max(nt, nv) + 255) / 256, 608), 256, 0, s>>>(
        dV, nv, dT, (int)nt, dcum, info));
    std::vector<char> back(info_at + sizeof(PsInfo));
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(back.data(), mesh, back.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_failed(e);
    PsInfo h;
    std::memcpy(&h, back.data() + info_at, sizeof(h));
    if (h.bad_index) {
      set_error("nat_bem_poisson_sample: triangle index out of range");
      return failed(NAT_BEM_EINVAL);
    }
    if (h.bad_tri < nt) {
      set_error("nat_bem_poisson_sample: degenerate or non-finite triangle " + std::to_string(h.bad_tri));
      return failed(NAT_BEM_EINVAL);
    }
    // cumulative areas: sequential FP64 sums by definition, so on the host (10 us at 10240)
    double* cum = reinterpret_cast<double*>(back.data());
    double acc = 0.0;
    for (int64_t t = 0; t < nt; ++t) {
      acc = acc + cum[t];
      cum[t] = acc;
    }
    double lo[3], hi[3];
    for (int d = 0; d < 3; ++d) {
      auto value = [](unsigned long long o) {
        const unsigned long long b = (o >> 63) ? o & 0x7fffffffffffffffull : ~o;
        double v;
        std::memcpy(&v, &b, 8);
        return v;
      };
      lo[d] = value(h.lo[d]);
      hi[d] = value(h.hi[d]);
    }
    PsGrid g;
    g.lox = lo[0];
    g.loy = lo[1];
    g.loz = lo[2];
    g.h = radius / std::sqrt(3.0);
    double fd[3];
    for (int d = 0; d < 3; ++d) fd[d] = std::floor((hi[d] - lo[d]) / g.h) + 1.0;
    if (h.nan_box || !(fd[0] * fd[1] * fd[2] <= (double)kPsMaxCells)) {
      set_error("nat_bem_poisson_sample: radius too small for the mesh's extent (more than 2^28 grid cells)");
      return failed(NAT_BEM_EINVAL);
    }
    g.nx = (int)fd[0];
    g.ny = (int)fd[1];
    g.nz = (int)fd[2];
    const size_t cells = (size_t)g.nx * g.ny * g.nz;
    int dev = 0, sms = 0, per_sm = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ps_run, kPsThreads, 0);
    if (e != cudaSuccess || per_sm < 1) return cuda_failed(e == cudaSuccess ? cudaErrorLaunchOutOfResources : e);
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (m + 127) / 128));
    // scratch: head and slot start at -1, flag at 0
    const bool pdev = cap > 0 && is_device_pointer(pts_out), ndev = cap > 0 && is_device_pointer(normals_out);
    const size_t most = (size_t)std::min<int64_t>(cap, m);
    size_t size = 0;
    auto take = [&](size_t bytes) {
      const size_t at = size;
      size += (bytes + 255) / 256 * 256;
      return at;
    };
    const size_t M = (size_t)m;
    const size_t a_head = take(cells * 4), a_slot = take(M * 32), a_flag = take(M), a_x = take(M * 24),
                 a_hi = take(M * 16), a_lo = take(M * 16), a_tri = take(M * 4), a_next = take(M * 4),
                 a_occ = take(M * 4), a_list = take(M * 4), a_part = take((size_t)blocks * 4), a_idx = take(most * 8),
                 a_pts = take(pdev ? 0 : most * 24), a_nrm = take(ndev ? 0 : most * 24);
    if ((st = dev_alloc_n(&scratch, size, s)) != NAT_BEM_OK) return failed(st);
    auto at = [&](size_t off) { return static_cast<void*>(scratch + off); };
    double* dx = static_cast<double*>(at(a_x));
    int* tri = static_cast<int*>(at(a_tri));
    float4 *hi4 = static_cast<float4*>(at(a_hi)), *lo4 = static_cast<float4*>(at(a_lo));
    int *head = static_cast<int*>(at(a_head)), *next = static_cast<int*>(at(a_next)), *occ = static_cast<int*>(at(a_occ));
    int *list = static_cast<int*>(at(a_list)), *part = static_cast<int*>(at(a_part));
    float4* slot = static_cast<float4*>(at(a_slot));
    unsigned char* flag = static_cast<unsigned char*>(at(a_flag));
    int64_t* didx = static_cast<int64_t*>(at(a_idx));
    double* dp = pdev ? pts_out : static_cast<double*>(at(a_pts));
    double* dn = ndev ? normals_out : static_cast<double*>(at(a_nrm));
    e = cudaMemcpyAsync(dcum, cum, (size_t)nt * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(scratch, 0xff, a_flag, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, M, s);
    if (e != cudaSuccess) return cuda_failed(e);
    NB_LAUNCH("ps_candidates", s, k_ps_candidates<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(
        dV, dT, dcum, (int)nt, du, (int)m, g, 1.0 / radius, dx, tri, hi4, lo4, head, next, occ, info));
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_failed(e);
    double r2 = radius * radius;
    int mi = (int)m;
    const double* dVc = dV;
    const int32_t* dTc = dT;
    const double* dxc = dx;
    const int *tric = tri, *headc = head, *nextc = next, *occc = occ;
    const float4 *hic = hi4, *loc = lo4;
    void* args[] = {&g, &r2, &dVc, &dTc, &dxc, &tric, &hic, &loc, &mi, &headc, &nextc, &occc, &list, &slot, &flag,
                    &part, &cap, &didx, &dp, &dn, &info};
    NB_LAUNCH("ps_run", s, e = cudaLaunchCooperativeKernel((const void*)k_ps_run, dim3(blocks), dim3(kPsThreads), args, 0, s));
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, info, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_failed(e);
    if (h.err) {
      set_error("nat_bem_poisson_sample: no progress for two seconds");
      return failed(NAT_BEM_ETIMEOUT);
    }
    *count = h.count;
    const size_t k = (size_t)std::min<int64_t>(cap, h.count);
    if (idx_out && k > 0) e = cudaMemcpyAsync(idx_out, didx, k * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (h.count <= cap && k > 0) {
      if (e == cudaSuccess && !pdev) e = cudaMemcpyAsync(pts_out, dp, k * 24, cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess && !ndev) e = cudaMemcpyAsync(normals_out, dn, k * 24, cudaMemcpyDeviceToHost, s);
    }
    if (e == cudaSuccess && k > 0) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_failed(e);
    cleanup();
    if (h.count > cap) {
      set_error("nat_bem_poisson_sample: " + std::to_string(h.count) + " samples exceed cap " + std::to_string(cap));
      return NAT_BEM_EINVAL;
    }
    return NAT_BEM_OK;
  } catch (...) {
    set_error("internal error in nat_bem_poisson_sample");
    return NAT_BEM_ECUDA;
  }
}
