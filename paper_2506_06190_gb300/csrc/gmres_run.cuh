// A whole GMRES run for one right-hand side, or for several systems of one each (a batch of
// operators, each system on blocks of its own and as long as it needs), in one cooperative launch
// (included by gmres.cu).
//
// The two-launch iteration (matvec, k_arnoldi) is bound by latency below a few thousand rows:
// every iteration pays two kernel starts and drains, reloads the Krylov basis, and leaves HBM
// idle during Gram-Schmidt. Here one block per SM keeps its rows of everything for the run:
//   - block b owns the contiguous rows [b n / G, (b + 1) n / G) of L, w and the basis; the basis
//     vectors' rows stay in shared memory (the columns past the space read from global memory);
//   - its rows of the operator stream through rings of asynchronous copies in shared memory, one
//     ring per warp (a column range of some of the rows, with that range of x in registers). A
//     lane copies and reads back its own 16-byte units, so the rings need no barriers; a warp
//     refills a stage as soon as it has read it, across iterations too, so the next matvec's
//     first rows arrive while the Gram-Schmidt phases wait. (Bulk copies measured 29 bytes a
//     cycle and SM in 2.6 KB pieces from L2, whatever the number in flight.)
//   - odd iterations walk the rows backwards: what the L2 still holds of the previous sweep is
//     read first, so an operator up to a few times the L2 does not come from HBM every time;
//   - a matvec needs no barrier after it: the rows' sums feed the block's own partial dots. An
//     iteration has three grid barriers (x published, partials, totals);
//   - an FP64 warp instruction holds its scheduler's unit for about 76 cycles whatever its lanes
//     do, so the FP64 phases put real and imaginary parts in lanes of their own and spread over
//     warps of all four schedulers;
//   - every block forms the rotations itself from the same totals in the same order (its last
//     warp, during the next barrier), so all blocks agree on convergence without exchanging it.
// The arithmetic is that of the two-launch form: FP32 products with compensated FP32 sums, FP64
// Gram-Schmidt and rotations (FP32 basis for inner refinement solves), the same second-pass
// test, and sums in a fixed order. A block has more rows than the two-launch form's (64 to 168, there
// 17 to 80), so on the FP32 basis its sums over rows and over basis vectors are compensated: plain
// FP32 chains of up to 84 terms left ||w - V h||^2 two to five times further from FP64 sums than
// that form does, these are as good as FP64 sums of the FP32 vectors. They take 0.4% of a mixed
// solve (2490 rows: 19.57 -> 19.65 us an iteration).
//
// Measured (GB300, one solve in flight, microseconds per iteration, before -> now): see the
// dispatch in gmres_run.
#pragma once

namespace natbem {
namespace {

constexpr int kRunWarps = 16;                      // all of them in the matvec; the last two also
                                                   // decide and form the rotations
constexpr int kRunThreads = kRunWarps * 32;
constexpr int kRunUpd = kRunWarps - 2;             // warps of the row updates
constexpr int kRunRows = 3 * kRunUpd * 4;          // rows a block may own: three rounds of updates
constexpr int kRunMaxStages = 8;
constexpr int kRunSmem = 206 * 1024;               // dynamic; 19 KB static beside it
constexpr int kRunLsqCols = 16;                    // least-squares panel, in the rings' space

// 16-byte units of a row per lane: x stays in registers for the matvec (slots x 4 floats for
// complex64 entries, x 8 for 16-bit pairs)
template <int kFmt>
constexpr int kRunSlots = kFmt == 0 ? 10 : 6;

struct RunArgs {
  int blocks;        // blocks per system; block b works on system s0 + b / blocks
  int s0;            // first system of the launch
  const int* ns;     // rows of each system, or null: n
  int64_t astride;   // operators of a batch: elements of A from one to the next (0: one system)
  int64_t sstride;   // row scales likewise
  const void* A;     // operator: complex64, or packed 16-bit pairs
  const float* rs;   // row scales of the FP16 copy, or null
  double2 *pb, *hr;  // (m + 2) x G partials, m + 2 totals
  unsigned* bar;     // arrivals (monotonic over the run), blocks that left
  int* err;
  float2* pout;
  int accumulate;
  int cw;            // column ranges the warps split a row into (1..16, a power of two)
  int stages;        // ring stages per warp
  int seg;           // units of a column range (at most) = units of a stage
  int ring;          // bytes of the rings (and later of the least-squares panel)
  int vcols;         // basis vectors held in shared memory
};

// Shared-memory shape for n rows on G blocks; stages = 0 if it does not fit. A row is split into
// as few column ranges as keep x in registers and the warps busy: every (row, range) ends in a
// warp reduction.
inline RunArgs run_shape(int n, int ld, int G, int fmt, bool f32, int cols) {
  RunArgs r{};
  const int rows = (n + G - 1) / G;
  const int n16 = fmt == 0 ? ld / 2 : ld / 4;
  const int slots = fmt == 0 ? kRunSlots<0> : kRunSlots<1>;
  const int least = fmt == 0 ? 128 : 64;
  r.cw = 1;
  while (r.cw < kRunWarps && n16 / (2 * r.cw) >= least) r.cw *= 2;
  r.seg = ((n16 + 31) / 32 + r.cw - 1) / r.cw * 32;  // ranges of whole warp-wide pieces
  if (r.seg > 32 * slots || rows > kRunRows) return r;
  const int64_t esz = f32 ? 8 : 16;
  const int64_t stage = 16ll * r.seg * kRunWarps;  // one stage of every warp
  const int64_t fixed = esz * rows + 8ll * r.cw * rows + 256;
  const int64_t want = esz * rows * std::min(cols, 32);
  int64_t st = std::min<int64_t>(kRunMaxStages, (kRunSmem - fixed - want) / stage);
  st = std::max<int64_t>(st, 2);
  const int64_t ring = std::max<int64_t>(stage * st, 16ll * kRunLsqCols * cols);
  const int64_t left = kRunSmem - fixed - ring;
  if (left < esz * rows) return r;
  r.stages = (int)st;
  r.ring = (int)ring;
  r.vcols = (int)std::min<int64_t>(cols, left / (esz * rows));
  return r;
}

__device__ __forceinline__ void run_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Grid barrier on a monotonic count: arrive publishes the block's writes (ordered before it by
// a block barrier), wait returns once `target` arrivals are visible. Bounded by two seconds.
__device__ __forceinline__ void run_arrive(unsigned* count) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
}
__device__ __forceinline__ bool run_wait(const unsigned* count, unsigned target, int* err) {
  uint64_t t0 = 0;
  for (unsigned it = 1;; ++it) {
    unsigned cur;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(count) : "memory");
    if ((int)(cur - target) >= 0) return true;
    if ((it & 255u) == 0u) {
      uint64_t t;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      if (t - t0 > 2000000000ull) {
        atomicOr(err, 64);
        return false;
      }
    }
  }
}
// Waits until at most `left` of this thread's copy groups are in flight.
__device__ __forceinline__ void run_landed(int left) {
  switch (left) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
  }
}

// 1 / sqrt(x), x > 0: the hardware's FP64 seed (a few bits over 20) and two Newton steps, each
// doubling the correct bits. No conversions and no FP64 comparisons, which cost as much as FMAs.
__device__ __forceinline__ double run_rsqrt(double x) {
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) - 1u;
  if (e >= 0x7fdu) return 1.0 / sqrt(x);  // subnormal, infinite, NaN
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double r = fma(-x * y, y, 1.0);
    y = fma(0.5 * y, r, y);
  }
  return y;
}

// sum over the four lanes of a quad
__device__ __forceinline__ double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 1);
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 1);
}

template <bool kF32>
struct RunBasis {
  using V = double2;
  using S = double;
};
template <>
struct RunBasis<true> {
  using V = float2;
  using S = float;
};

template <class V, class S>
__device__ __forceinline__ V run_make(S x, S y) {
  V v;
  v.x = x;
  v.y = y;
  return v;
}

// A running sum of products a b + c d over rows or basis vectors: FP64 as it comes, FP32 compensated.
template <class S>
struct RunSum;
template <>
struct RunSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b, double c, double d) { s = fma(c, d, fma(a, b, s)); }
  __device__ __forceinline__ double get() const { return s; }
  __device__ __forceinline__ double quad() const { return quad_sum(s); }
};
template <>
struct RunSum<float> {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float a, float b, float c, float d) { kahan_add(s, e, fmaf(a, b, c * d)); }
  __device__ __forceinline__ float get() const { return s - e; }
  __device__ __forceinline__ double quad() const {  // over the quad's lanes, as a float pair
    float hi, lo;
    two_sum(s, -e, hi, lo);
#pragma unroll
    for (int o = 2; o > 0; o >>= 1)
      df_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o));
    return (double)hi + (double)lo;
  }
};

// One warp: column hc[0..j] of the Hessenberg matrix through the earlier rotations, into Hcol, for
// the least squares, by givens_warp's prefix scan; `top` is its last entry.
__device__ __forceinline__ void run_rotated(int j, const double2* hc, const double* cs, const double2* sn, double2 top,
                                            double2* Hcol, int lane) {
  const int S = (j + 31) / 32;
  const int i0 = min(j, lane * S), i1 = min(j, i0 + S);
  double2 A = make_double2(1.0, 0.0), B = make_double2(0.0, 0.0);
  for (int i = i0; i < i1; ++i) {
    const double2 ai = make_double2(-sn[i].x, sn[i].y);
    const double2 bi = make_double2(cs[i] * hc[i + 1].x, cs[i] * hc[i + 1].y);
    A = cmul(ai, A);
    B = cadd(cmul(ai, B), bi);
  }
  for (int o = 1; o < 32 && o * S < j; o <<= 1) {
    const double2 Ap = make_double2(__shfl_up_sync(0xffffffffu, A.x, o), __shfl_up_sync(0xffffffffu, A.y, o));
    const double2 Bp = make_double2(__shfl_up_sync(0xffffffffu, B.x, o), __shfl_up_sync(0xffffffffu, B.y, o));
    if (lane >= o) {
      B = cadd(cmul(A, Bp), B);
      A = cmul(A, Ap);
    }
  }
  double2 Ae = make_double2(__shfl_up_sync(0xffffffffu, A.x, 1), __shfl_up_sync(0xffffffffu, A.y, 1));
  double2 Be = make_double2(__shfl_up_sync(0xffffffffu, B.x, 1), __shfl_up_sync(0xffffffffu, B.y, 1));
  if (lane == 0) {
    Ae = make_double2(1.0, 0.0);
    Be = make_double2(0.0, 0.0);
  }
  double2 t = cadd(cmul(Ae, hc[0]), Be);
  for (int i = i0; i < i1; ++i) {
    const double2 h1 = hc[i + 1];
    Hcol[i] = cadd(make_double2(cs[i] * t.x, cs[i] * t.y), cmul(sn[i], h1));
    t = cadd(cmul(make_double2(-sn[i].x, sn[i].y), t), make_double2(cs[i] * h1.x, cs[i] * h1.y));
  }
  if (lane == 0) Hcol[j] = top;
}

// kFmt: 0 complex64, 1 packed BF16 pairs, 2 packed FP16 pairs with row scales.
template <int kFmt, bool kF32>
__global__ void __launch_bounds__(kRunThreads, 1) k_gmres_run(GArgs a, RunArgs p) {
  using V = typename RunBasis<kF32>::V;
  using S = typename RunBasis<kF32>::S;
  constexpr int kC = kRunThreads;
  constexpr int kN = kRunSlots<kFmt>;
  constexpr int kX = kFmt == 0 ? 1 : 2;  // float4 of x per unit
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double2 s_h[258], s_hc[258], s_sn[256], s_d[258];
  __shared__ double s_cs[256];
  __shared__ double s_inv, s_hn2, s_tot[2][4];
  __shared__ double2 s_t;
  __shared__ V s_hv[kF32 ? 258 : 1];  // h in the basis' precision
  __shared__ int s_again, s_done, s_abort;
  // this block's system and its arrays
  const int G = p.blocks, b = (int)blockIdx.x % G, sys = p.s0 + (int)blockIdx.x / G;
  const int n = p.ns ? p.ns[sys] : a.n;
  const size_t vstr = (size_t)a.nrhs * a.n;  // from one basis vector to the next
  {
    const size_t ns = (size_t)sys * a.n;
    a.b += ns;
    a.x += ns;
    a.V += ns;
    if (kF32) a.Vf += ns;
    p.pout += ns;
    a.xf += (size_t)sys * a.ld;
    a.H += (size_t)sys * a.m * (a.m + 1);
    a.gv += (size_t)sys * (a.m + 1);
    p.pb += (size_t)sys * (a.m + 2) * G;
    p.hr += (size_t)sys * (a.m + 2);
    p.bar += 2 * sys;
    a.bnorm += sys;
    a.hnorm += sys;
    a.res += sys;
    a.iters += sys;
    a.done += sys;
    if (a.skip) a.skip += sys;
    if (a.bscale) a.bscale += sys;
    if (kFmt == 2) p.rs += sys * p.sstride;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool decides = warp == kRunWarps - 1, chains = warp == kRunWarps - 2;
  // a warp's lanes in the Gram-Schmidt phases: four items, real and imaginary part, a quad each
  const int item = lane >> 3, l4 = lane & 3;
  const bool im = lane & 4;
  const int r0 = (int)((int64_t)b * n / G), rows = (int)((int64_t)(b + 1) * n / G) - r0;
  const int rmax = (n + G - 1) / G;
  const int n16 = a.ld / (kFmt == 0 ? 2 : 4);  // 16-byte units per operator row
  V* sV = reinterpret_cast<V*>(smem + p.ring);
  V* sw = sV + (size_t)rmax * p.vcols;
  float* part = reinterpret_cast<float*>(sw + rmax);  // [column range][row][re, im]
  V* gV = kF32 ? reinterpret_cast<V*>(a.Vf) : reinterpret_cast<V*>(a.V);

  // this warp's rows and columns of the operator
  const int cwi = warp & (p.cw - 1), rw = warp / p.cw, nrw = kRunWarps / p.cw;
  const int ra = rows * rw / nrw, rb = rows * (rw + 1) / nrw;
  const int n32 = (n16 + 31) / 32;
  const int u0 = n32 * cwi / p.cw * 32, len = min(n16, n32 * (cwi + 1) / p.cw * 32) - u0;
  const float4* st0 = reinterpret_cast<const float4*>(smem) + (size_t)warp * p.stages * p.seg;
  const uint32_t ring = sa_u32(st0 + lane);
  const float4* Ab = reinterpret_cast<const float4*>(p.A) + (size_t)sys * (p.astride / (kFmt == 0 ? 2 : 4)) +
                     (size_t)r0 * n16 + u0 + lane;

  if (tid == 0) {
    s_done = (a.skip && a.skip[0]) ? 1 : 0;
    s_abort = 0;
  }
  __syncthreads();

  // The warp's rows in order, then backwards, and so on: irow the next one to request.
  int irow = ra, istep = 1, slot = 0;
  auto issue = [&](int q) {  // request the next row's column range into stage q, one copy group
    const uint32_t dst = ring + (uint32_t)(q * p.seg) * 16u;
    const float4* src = Ab + (size_t)irow * n16;
#pragma unroll
    for (int e = 0; e < kN; ++e)
      if (lane + 32 * e < len)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512u * e), "l"(src + 32 * e) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    irow += istep;
    if (irow == rb || irow < ra) {
      irow -= istep;  // the turn: the next iteration starts with the row this one ended with
      istep = -istep;
    }
  };
  if (rb > ra)
    for (int q = 0; q < p.stages; ++q) {
      // the lanes past the end of a last, partial piece multiply these zeros
      if ((len & 31) && lane >= (len & 31))
        const_cast<float4*>(st0)[q * p.seg + (len & ~31) + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      issue(q);
    }

  unsigned target = 0;  // arrivals the next wait needs
  auto arrive = [&]() {  // thread 0, after a barrier of the writers
    if (tid == 0) run_arrive(p.bar);
  };
  auto wait = [&]() {
    target += (unsigned)G;
    if (tid == 0 && !run_wait(p.bar, target, p.err)) s_abort = 1;
    __syncthreads();
  };

  // v_0 = b / ||b||
  double res = 0.0, goal2 = 0.0;  // the deciding warp: residual estimate, (stopping residual)^2
  double2 gj = make_double2(0.0, 0.0);
  if (warp == 0) {
    double t = 0.0;
    for (int r = lane; r < rows; r += 32) t += cabs2(a.b[r0 + r]);
    t = warp_sum(t);
    if (lane == 0) {
      __stcg(p.pb + b, make_double2(t, 0.0));
      run_arrive(p.bar);
    }
  }
  wait();
  if (decides) {
    double t = 0.0;
    for (int q = lane; q < G; q += 32) t += __ldcg(p.pb + q).x;
    t = warp_sum(t);
    const double hn = sqrt(t);
    gj = make_double2(hn, 0.0);
    res = hn;
    const double goal = a.tol * (a.bscale ? a.bscale[0] : hn);
    goal2 = goal * goal;
    if (lane == 0) {
      s_inv = hn > 0.0 ? 1.0 / hn : 0.0;
      if (!(hn > 0.0)) s_done = 1;
      s_d[0] = make_double2(1.0, 0.0);
      if (b == 0) {
        a.bnorm[0] = hn;
        a.hnorm[0] = hn;
        a.res[0] = hn;
        a.gv[0] = gj;
      }
    }
  }
  __syncthreads();
  for (int r = tid; r < rows; r += kC) {
    const double2 bv = a.b[r0 + r];
    const double2 v = make_double2(bv.x * s_inv, bv.y * s_inv);
    const V vv = run_make<V, S>((S)v.x, (S)v.y);
    sV[r] = vv;
    gV[r0 + r] = vv;
    __stcg(a.xf + r0 + r, make_float2((float)v.x, (float)v.y));
  }
  __syncthreads();
  arrive();
  int j = 0;
  for (;; ++j) {
    // x = v_j from every block
    wait();
    if (s_abort || s_done || j >= a.maxit) break;
    {
      float4 xv[kN * kX];
      const float4* xg = reinterpret_cast<const float4*>(a.xf) + (size_t)u0 * kX;
#pragma unroll
      for (int q = 0; q < kN; ++q) {
        const int u = lane + 32 * q;
#pragma unroll
        for (int e = 0; e < kX; ++e) xv[kX * q + e] = u < len ? __ldcg(xg + kX * u + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      // the rows of w = L v_j, two at a time: compensated FP32 sums per lane
      const int rstep = (j & 1) ? -1 : 1;
      int row = (j & 1) ? rb - 1 : ra;
      for (int left = rb - ra; left > 0; left -= 2, row += 2 * rstep) {
        const bool two = left > 1;
        const int slot1 = slot + 1 == p.stages ? 0 : slot + 1;
        run_landed(p.stages - (two ? 2 : 1));
        const float4* m0 = st0 + slot * p.seg;
        const float4* m1 = st0 + (two ? slot1 : slot) * p.seg;
        float sr[2] = {0.f, 0.f}, cr[2] = {0.f, 0.f}, si[2] = {0.f, 0.f}, ci[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < kN; ++q) {
          const int u = lane + 32 * q;
          if (32 * q < len) {
            const float4 mm[2] = {m0[u], m1[u]};
            if constexpr (kFmt == 0) {
              const float4 v = xv[q];
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const float4 m = mm[r];
                const float pr = fmaf(m.x, v.x, fmaf(-m.y, v.y, fmaf(m.z, v.z, -m.w * v.w)));
                const float pi_ = fmaf(m.x, v.y, fmaf(m.y, v.x, fmaf(m.z, v.w, m.w * v.z)));
                kahan_add(sr[r], cr[r], pr);
                kahan_add(si[r], ci[r], pi_);
              }
            } else {
              const float4 x0 = xv[kX * q], x1 = xv[kX * q + kX - 1];
              const float xr[4] = {x0.x, x0.z, x1.x, x1.z}, xi[4] = {x0.y, x0.w, x1.y, x1.w};
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const float4 m = mm[r];
                const uint32_t w[4] = {__float_as_uint(m.x), __float_as_uint(m.y), __float_as_uint(m.z),
                                       __float_as_uint(m.w)};
                float pr = 0.f, pi_ = 0.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  float ar, ai;
                  if (kFmt == 1) {
                    ar = __uint_as_float(w[e] << 16);
                    ai = __uint_as_float(w[e] & 0xffff0000u);
                  } else {
                    const float2 hv = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
                    ar = hv.x;
                    ai = hv.y;
                  }
                  pr = fmaf(ar, xr[e], fmaf(-ai, xi[e], pr));
                  pi_ = fmaf(ar, xi[e], fmaf(ai, xr[e], pi_));
                }
                kahan_add(sr[r], cr[r], pr);
                kahan_add(si[r], ci[r], pi_);
              }
            }
          }
        }
        issue(slot);
        if (two) issue(slot1);
        slot = two ? slot1 : slot;  // the last stage read
        if (++slot == p.stages) slot = 0;
        // lane sums of (row, component): halves of the warp keep a row, quarters a component
        const float k0 = sr[0] - cr[0], k1 = si[0] - ci[0], k2 = sr[1] - cr[1], k3 = si[1] - ci[1];
        const bool hi = lane & 16, odd = lane & 8;
        const float s0 = __shfl_xor_sync(0xffffffffu, hi ? k0 : k2, 16);
        const float s1 = __shfl_xor_sync(0xffffffffu, hi ? k1 : k3, 16);
        const float e0 = (hi ? k2 : k0) + s0, e1 = (hi ? k3 : k1) + s1;
        float v = (odd ? e1 : e0) + __shfl_xor_sync(0xffffffffu, odd ? e0 : e1, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        if ((lane & 7) == 0 && (!hi || two)) part[2 * (cwi * rmax + row + (hi ? rstep : 0)) + (odd ? 1 : 0)] = v;
      }
    }
    __syncthreads();
    for (int e = tid; e < 2 * rows; e += kC) {
      float t = 0.f, tc = 0.f;  // up to 16 column ranges
      for (int q = 0; q < p.cw; ++q) kahan_add(t, tc, part[2 * (q * rmax) + e]);
      S v = (S)(t - tc);
      if (kFmt == 2) v *= (S)p.rs[r0 + (e >> 1)];  // a power of two: exact
      reinterpret_cast<S*>(sw)[e] = v;
    }
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      // partial dots conj(V_c) . w over the block's rows, c <= j, and ||w||^2
      const int np = j + 2;
      for (int c0 = warp * 4; c0 < np; c0 += kRunWarps * 4) {
        const int c = c0 + item;
        RunSum<S> sum;
        if (c < np) {
          const V* v = c > j ? sw : c < p.vcols ? sV + (size_t)c * rmax : gV + c * vstr + r0;
          for (int r = l4; r < rows; r += 4) {
            const V vv = v[r], ww = sw[r];
            sum.add(vv.x, im ? ww.y : ww.x, vv.y, im ? -ww.x : ww.y);
          }
        }
        const double acc = sum.quad();
        if (l4 == 0 && c < np) __stcg(reinterpret_cast<double*>(p.pb + (size_t)c * G + b) + (im ? 1 : 0), acc);
      }
      __syncthreads();
      arrive();
      wait();
      // totals: column c by four warps of block c mod G, blocks in a fixed order
      if (warp < 4)
        for (int c = b; c < np; c += G) {
          const double* src = reinterpret_cast<const double*>(p.pb + (size_t)c * G) + (lane >> 4);
          double t[4];
          const int q0 = warp * 16 + (lane & 15);
#pragma unroll
          for (int u = 0; u < 4; ++u) t[u] = q0 + 64 * u < G ? __ldcg(src + 2 * (q0 + 64 * u)) : 0.0;
          double sum = t[0];
          if (64 < G) sum += t[1];
          if (128 < G) sum += t[2];
          if (192 < G) sum += t[3];
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if ((lane & 15) == 0) s_tot[lane >> 4][warp] = sum;
          run_bar(2, 128);
          if (tid < 2)
            __stcg(reinterpret_cast<double*>(p.hr + c) + tid,
                   (s_tot[tid][0] + s_tot[tid][1]) + (s_tot[tid][2] + s_tot[tid][3]));
          run_bar(2, 128);
        }
      __syncthreads();
      arrive();
      wait();
      for (int c = tid; c < np; c += kC) {
        const double2 h = __ldcg(p.hr + c);
        s_h[c] = h;
        if (kF32) s_hv[c] = run_make<V, S>((S)h.x, (S)h.y);
      }
      __syncthreads();
      S tsum[3];  // V h, the quad's component on rows 4 warp + item, + 56, + 112
      if (decides) {
        // ||w - V h||^2 by Pythagoras
        double hh = 0.0;
        for (int c = lane; c <= j; c += 32) hh += cabs2(s_h[c]);
        hh = warp_sum(hh);
        const double wn2 = s_h[j + 1].x;
        const double hn2 = fmax(wn2 - hh, 0.0);
        if (lane == 0) {
          s_hn2 = hn2;
          s_inv = hn2 > 0.0 ? run_rsqrt(hn2) : 0.0;
          s_again = pass == 0 && !(hn2 > 1e-4 * wn2);
        }
      } else if (chains) {
        // the column's entry t_j that the next rotation meets: a rotation chain
        // t_{i+1} = -conj(s_i) t_i + c_i h_{i+1} is linear in h, so t_j is sum_i d_i h_i with d
        // kept up to date as the rotations are made
        double2 t = make_double2(0.0, 0.0);
        for (int c = lane; c <= j; c += 32) {
          const double2 col = pass == 0 ? s_h[c] : cadd(s_hc[c], s_h[c]);
          s_hc[c] = col;
          t = cadd(t, cmul(s_d[c], col));
        }
        t.x = warp_sum(t.x);
        t.y = warp_sum(t.y);
        if (lane == 0) s_t = t;
      } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int base = 4 * (warp + q * kRunUpd), row = base + item;
          S acc = 0;
          if (base < rows) {
            RunSum<S> sum;
            if (row < rows)
              for (int c = l4; c <= j; c += 4) {
                const V vv = c < p.vcols ? sV[(size_t)c * rmax + row] : gV[c * vstr + r0 + row];
                const V h = kF32 ? s_hv[c] : reinterpret_cast<const V*>(s_h)[c];
                sum.add(vv.x, im ? h.y : h.x, vv.y, im ? h.x : -h.y);
              }
            acc = quad_sum(sum.get());
          }
          tsum[q] = acc;
        }
      }
      __syncthreads();
      if (s_abort) break;
      const bool again = s_again;
      if (!decides && !chains) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int row = 4 * (warp + q * kRunUpd) + item;
          if (row < rows && l4 == 0) {
            S* we = reinterpret_cast<S*>(sw + row) + (im ? 1 : 0);
            const S w = *we - tsum[q];
            if (again) {
              *we = w;
            } else {
              const S v = w * (S)s_inv;
              if (j + 1 < p.vcols) reinterpret_cast<S*>(sV + (size_t)(j + 1) * rmax + row)[im ? 1 : 0] = v;
              reinterpret_cast<S*>(gV + (j + 1) * vstr + r0 + row)[im ? 1 : 0] = v;
              __stcg(reinterpret_cast<float*>(a.xf + r0 + row) + (im ? 1 : 0), (float)v);
            }
          }
        }
        if (!again) {
          run_bar(1, kRunUpd * 32);
          arrive();
        }
      } else if (decides && !again) {
        // the rotation that zeroes h_{j+1,j} = hn against t_j, while the blocks meet
        const double2 t = s_t;
        const double hn2 = s_hn2, q2 = cabs2(t), rho2 = q2 + hn2;
        // the estimate after this rotation is res hn / sqrt(|t_j|^2 + hn^2)
        if (lane == 0 && (hn2 == 0.0 || hn2 * (res * res) <= goal2 * rho2)) s_done = 1;
        const double hn = hn2 * s_inv;
        double c = 0.0, absS = 1.0;
        double2 sv = make_double2(1.0, 0.0), top = make_double2(hn, 0.0);
        if (q2 != 0.0) {
          const double ia = run_rsqrt(q2), ir = run_rsqrt(rho2);
          const double2 ph = make_double2(t.x * ia, t.y * ia);
          c = q2 * ia * ir;
          absS = hn * ir;
          sv = make_double2(ph.x * absS, ph.y * absS);
          top = make_double2(ph.x * (rho2 * ir), ph.y * (rho2 * ir));
        }
        res *= absS;
        const double2 ns = make_double2(-sv.x, sv.y);
        if (lane == 0) {
          s_cs[j] = c;
          s_sn[j] = sv;
          if (b == 0) {
            a.gv[j] = make_double2(c * gj.x, c * gj.y);
            a.res[0] = res;
            a.hnorm[0] = hn;
          }
        }
        if (b == j % G) {  // this block rotates the column once the run has ended
          double2* Hcol = a.H + (size_t)j * (a.m + 1);
          for (int i = lane; i <= j; i += 32) Hcol[i] = s_hc[i];
          if (lane == 0) Hcol[j + 1] = top;
        }
        gj = cmul(ns, gj);
        for (int i = lane; i <= j; i += 32) s_d[i] = cmul(s_d[i], ns);
        if (lane == 0) s_d[j + 1] = make_double2(c, 0.0);
        __syncwarp();
      }
      if (!again) break;
      __syncthreads();
    }
    // an abort leaves through the check after the next x: the one place where every warp of the
    // block reads the same flags
  }
  // the rows requested beyond the end have to land before their stages are reused
  run_landed(0);
  __syncthreads();
  if (s_abort) return;  // the host reads the error word
  // least squares: R y = g by every block, on rows scaled to a unit diagonal
  const int kd = j;
  if (b == 0 && tid == 0) {
    a.iters[0] = kd;
    a.done[0] = s_done;
    if (sys == p.s0) {
      a.scal[0] = kd;
      a.scal[1] = 1;
    }
  }
  if (warp == 0)
    for (int c = b; c < kd; c += G) {
      double2* Hcol = a.H + (size_t)c * (a.m + 1);
      for (int i = lane; i <= c + 1; i += 32) s_hc[i] = Hcol[i];
      __syncwarp();
      run_rotated(c, s_hc, s_cs, s_sn, s_hc[c + 1], Hcol, lane);
      __syncwarp();
    }
  __syncthreads();
  arrive();  // the rotated columns, and block 0's g
  wait();
  if (s_abort) return;
  const int ms = a.m + 1;
  for (int k = tid; k < kd; k += kC) {
    const double2 d = __ldcg(a.H + (size_t)k * ms + k);
    const double dd = cabs2(d);
    const double2 inv = dd > 0.0 ? make_double2(d.x / dd, -d.y / dd) : make_double2(0.0, 0.0);
    s_sn[k] = inv;
    s_hc[k] = cmul(__ldcg(a.gv + k), inv);
  }
  double2* pan = reinterpret_cast<double2*>(smem);  // kRunLsqCols x kd
  for (int i1 = kd; i1 > 0; i1 -= kRunLsqCols) {
    const int i0 = max(0, i1 - kRunLsqCols);
    __syncthreads();
    for (int q = warp; q < i1 - i0; q += kRunWarps)
      for (int k = lane; k < i0 + q; k += 32) pan[q * kd + k] = cmul(__ldcg(a.H + (size_t)(i0 + q) * ms + k), s_sn[k]);
    __syncthreads();
    if (warp == 0) {
      double2 g = i0 + lane < i1 ? s_hc[i0 + lane] : make_double2(0.0, 0.0);
      for (int q = i1 - i0 - 1; q > 0; --q) {
        const double2 y = make_double2(__shfl_sync(0xffffffffu, g.x, q), __shfl_sync(0xffffffffu, g.y, q));
        if (lane < q) {
          const double2 r = pan[q * kd + i0 + lane];
          g.x = fma(-r.x, y.x, fma(r.y, y.y, g.x));
          g.y = fma(-r.x, y.y, fma(-r.y, y.x, g.y));
        }
      }
      if (i0 + lane < i1) s_hc[i0 + lane] = g;
    }
    __syncthreads();
    for (int k = tid; k < i0; k += kC) {
      double2 g = s_hc[k];
      for (int q = 0; q < i1 - i0; ++q) {
        const double2 r = pan[q * kd + k], y = s_hc[i0 + q];
        g.x = fma(-r.x, y.x, fma(r.y, y.y, g.x));
        g.y = fma(-r.x, y.y, fma(-r.y, y.x, g.y));
      }
      s_hc[k] = g;
    }
  }
  __syncthreads();
  // x (+)= V y on the block's rows
  for (int base = 4 * warp; base < rows; base += 4 * kRunWarps) {
    const int row = base + item;
    RunSum<S> sum;
    if (row < rows)
      for (int c = l4; c < kd; c += 4) {
        const V vv = c < p.vcols ? sV[(size_t)c * rmax + row] : gV[c * vstr + r0 + row];
        const double2 y = s_hc[c];
        sum.add(vv.x, (S)(im ? y.y : y.x), vv.y, (S)(im ? y.x : -y.y));
      }
    const S acc = quad_sum(sum.get());
    if (row < rows && l4 == 0) {
      const size_t e = 2 * (size_t)(r0 + row) + (im ? 1 : 0);
      double* xe = reinterpret_cast<double*>(a.x) + e;
      const double x = (p.accumulate ? *xe : 0.0) + (double)acc;
      *xe = x;
      reinterpret_cast<float*>(p.pout)[e] = (float)x;
      reinterpret_cast<float*>(a.xf)[e] = (float)x;
    }
  }
  // the last block to leave readies the barrier for the next run
  if (tid == 0) {
    const unsigned t = atomicAdd(p.bar + 1, 1u);
    if (t == (unsigned)G - 1u) {
      p.bar[0] = 0u;
      p.bar[1] = 0u;
    }
  }
}

}  // namespace
}  // namespace natbem
