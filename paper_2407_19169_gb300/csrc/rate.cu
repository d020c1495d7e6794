// rate.cu — the CFL rate of a state that was written or projected: max over the cells of
// beta^x / hx (+ beta^y / hy) at the cell averages and, with the positivity limiter, at the limiter's
// points; the first step's dt comes from it (later steps take theirs inside the last stage).
//
// The maximum is formed in FP64 whatever the storage, and FP64 arithmetic is 1/63 of FP32's here, so
// every rate is first bracketed in FP32 (an upper and a lower bound that allow for the rounding of the
// coefficients, of the evaluation and of the flux functions). One kernel takes the largest lower bound of
// the mesh, a second evaluates in FP64 only cells whose upper bound reaches it: the result is the FP64
// maximum, from a few cells. Cells without higher modes take their average alone. What bounds it then
// is two FP32 passes over the points; before, each point cost an FP64 Legendre recurrence with
// divisions (writing and reading a 1024^2 Q2 solve with the limiter: 9.8 ms, now 0.5).
#include "dg_internal.h"
#include "stage1d.cuh"

namespace dgk {

// Cell average of variable v from either storage form.
static __device__ inline double rate_avg(const AuxGeom& g, const void* st, int v, long long c) {
  if (g.prec == PREC_F64) return ((const double*)st)[((long long)v * g.nm) * g.ncell + c];
  const F32Layout L{g.ncell, g.nv, g.nm};
  const float* b = (const float*)st;
  return (double)b[L.word(v, 0, c)] + (double)b[L.word(v, g.nm, c)];
}

// CFL rate of one state in FP64, beta^x / hx (+ beta^y / hy), with correctly rounded division and root.
template <int EQ, int DIM>
static __device__ __forceinline__ double rate_of(const AuxGeom& g, const double* ub, bool& phys) {
  double bx, by, invH;
  if constexpr (EQ == EQ_EULER) {
    const double inv = 1.0 / ub[0], vx = ub[1] * inv;
    double p, c;
    if constexpr (DIM == 1) {
      p = (g.gamma - 1.0) * (ub[2] - 0.5 * ub[1] * vx);
      c = sqrt(g.gamma * p * inv);
      by = 0.0;
      invH = ub[0] * (1.0 / (ub[2] + p));
    } else {
      const double vy = ub[2] * inv;
      p = (g.gamma - 1.0) * (ub[3] - 0.5 * (ub[1] * vx + ub[2] * vy));
      c = sqrt(g.gamma * p * inv);
      by = fabs(vy) + c;
      invH = ub[0] * (1.0 / (ub[3] + p));
    }
    bx = fabs(vx) + c;
    phys = pos_finite(ub[0]) && pos_finite(p) && !not_finite(bx) && (DIM == 1 || !not_finite(by)) && !not_finite(invH);
  } else {
    avg_params<EQ, DIM>(ub, g.gamma, g.gamma - 1.0, g.ax, g.ay, bx, by, invH, phys);
  }
  return bx / g.hx + (DIM == 2 ? by / g.hy : 0.0);
}

// P_l(x) by the three-term recurrence.
static __device__ inline double legendre(int l, double x) {
  double pm = 1.0, p = x;
  if (l == 0) return 1.0;
  for (int j = 1; j < l; ++j) {
    const double pn = ((2.0 * j + 1.0) * x * p - j * pm) / (j + 1.0);
    pm = p;
    p = pn;
  }
  return p;
}

// Bounds of the rate of an Euler state w (NV = 3 or 4) whose variables are off by at most d[v]. lo > 0
// and up finite only where the state is physical for any values within the bounds and FP32 can tell: the
// kinetic energy is formed as m (m / rho), which stays in range where the energy does (m^2 of densities
// of 1e-30 does not), and every quantity on the way has to be far above the smallest normal number, or
// the lost digits could pass for pressure. Otherwise lo = 0 and up = inf: the cell is evaluated. The
// factors 1 -+ 1e-5 cover the rounding of the operations below.
struct RateBounds {
  float lo, up;
};
template <int NV>
static __device__ __forceinline__ RateBounds rate_bounds(const float (&w)[NV], const float (&d)[NV], float gam,
                                                         float gm1, float ihx, float ihy) {
  constexpr float TINY = 1e-33f;
  const float rlo = w[0] - d[0], rup = w[0] + d[0];
  const float ilo = arcp(rup), iup = arcp(rlo);                   // bounds of 1 / rho
  float vlo = 0.f, vup = 0.f, klo = 0.f, kup = 0.f;
#pragma unroll
  for (int v = 1; v < NV - 1; ++v) {
    const float a = fmaxf(fabsf(w[v]) - d[v], 0.f), b = fabsf(w[v]) + d[v], ih = v == 1 ? ihx : ihy;
    vlo += a * ilo * ih;
    vup += b * iup * ih;
    klo += a * (a * ilo);
    kup += b * (b * iup);
  }
  const float sh = NV == 3 ? ihx : ihx + ihy, g2 = gam * gm1;
  const float elo = w[NV - 1] - d[NV - 1] - 0.50001f * kup;       // p / (gamma - 1)
  const float eup = w[NV - 1] + d[NV - 1] - 0.49999f * klo;
  const float slo = elo * ilo, sup = eup * iup;
  const float clo = asqrt(fmaxf(g2 * slo, 0.f)), cup = asqrt(fmaxf(g2 * sup, 0.f));
  RateBounds r;
  r.lo = 0.99999f * (vlo + clo * sh);
  r.up = 1.00001f * (vup + cup * sh);
  const bool known = rlo > TINY && rup < 1.f / TINY && elo > TINY && slo > TINY && g2 * slo > TINY &&
                     rlo * clo > TINY && ihx > TINY && (NV == 3 || ihy > TINY) && r.lo > TINY && r.up < 3e38f;
  if (!known) {
    r.lo = 0.f;
    r.up = INFINITY;
  }
  return r;
}

// The largest lower bound into sc->rate_floor (bits of a non-negative float), one atomic per warp.
static __device__ __forceinline__ void floor_end(DevScalars* sc, float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&sc->rate_floor, __float_as_uint(x));
}

// Block end: the block's maximum (a NaN is kept) and physicality into the solver's scalars.
static __device__ __forceinline__ void rate_end(DevScalars* sc, int slot, double r, bool ok) {
  __shared__ double red[32];
  r = warp_max(r);
  const unsigned bad = __ballot_sync(0xffffffffu, !ok);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = (red[w] > m || red[w] != red[w]) ? red[w] : m;
    atomic_max_nonneg(&sc->rate_bits[slot], m);
  }
  if (bad && (threadIdx.x & 31) == 0) atomicOr(&sc->err, ERRB_NONPHYS);
}

// Rate over the cell averages. BOUND: the first kernel, the lower bounds; else the evaluation.
template <int EQ, int DIM, bool BOUND>
__global__ void __launch_bounds__(256) rate_averages_kernel(const AuxGeom g, const void* st, DevScalars* sc, int slot) {
  constexpr int NV = NVars<EQ, DIM>::value;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  float floor_ = 0.f;
  const float gam = (float)g.gamma, gm1 = (float)(g.gamma - 1.0), ihx = (float)(1.0 / g.hx), ihy = (float)(1.0 / g.hy);
  auto bounds = [&](const double (&ub)[NV]) -> RateBounds {
    float w[NV], d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      w[v] = (float)ub[v];
      d[v] = 1e-6f * fabsf(w[v]);
    }
    return rate_bounds<NV>(w, d, gam, gm1, ihx, ihy);
  };
  if constexpr (BOUND) {
    for (long long c = i0; c < g.ncell; c += step) {
      double ub[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) ub[v] = rate_avg(g, st, v, c);
      floor_ = fmaxf(floor_, bounds(ub).lo);
    }
    floor_end(sc, floor_);
    return;
  }
  if constexpr (EQ == EQ_EULER) floor_ = __uint_as_float(sc->rate_floor);
  double r = 0.0;
  bool ok = true;
  for (long long c = i0; c < g.ncell; c += step) {
    double ub[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) ub[v] = rate_avg(g, st, v, c);
    if constexpr (EQ == EQ_EULER) {
      if (bounds(ub).up < floor_) continue;
    }
    bool phys;
    const double rc = rate_of<EQ, DIM>(g, ub, phys);
    r = (rc > r || rc != rc) ? rc : r;
    ok = ok && phys;
  }
  rate_end(sc, slot, r, ok);
}

// Rate over the averages and the positivity limiter's points (Euler).
template <int DIM, int K, int BASIS, class PR, bool BOUND>
__global__ void __launch_bounds__(256) rate_points_kernel(const AuxGeom g, const void* st, DevScalars* sc, int slot) {
  constexpr int NV = NVars<EQ_EULER, DIM>::value;
  constexpr int NM = DIM == 1 ? K + 1 : Modes<K, BASIS>::NM;
  using S1 = Stage1D<K, EQ_EULER, PrecF32M>;
  using S2 = Stage2D<K, EQ_EULER, BASIS, PrecF32M>;
  using ST = Store<PR, NV, NM>;
  using TS = typename PR::T;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  const float gam = (float)g.gamma, gm1 = (float)(g.gamma - 1.0), ihx = (float)(1.0 / g.hx), ihy = (float)(1.0 / g.hy);
  // values of the modes at the limiter's points
  constexpr int NP = DIM == 1 ? S1::NP_LIM : limiter_points(K), NQ = K + 1;
  __shared__ double phi[NP * NM];
  for (int e = threadIdx.x; e < NP * NM && !BOUND; e += blockDim.x) {
    const int i = e / NM, m = e % NM;
    if constexpr (DIM == 1) {
      const double x = i < NQ ? GaussRule<NQ>::x(i < NQ ? i : 0) : (i == NQ ? -1.0 : (i == NQ + 1 ? 1.0 : 0.0));
      phi[e] = legendre(m, x);
    } else {
      double x, y;
      if (i < NQ * NQ) {
        x = GaussRule<NQ>::x(i / NQ);
        y = GaussRule<NQ>::x(i % NQ);
      } else if (i < NQ * NQ + 4 * NQ) {
        const int d = (i - NQ * NQ) & 3;
        const double at = GaussRule<NQ>::x((i - NQ * NQ) >> 2);
        x = d == 0 ? -1.0 : (d == 1 ? 1.0 : at);
        y = d == 2 ? -1.0 : (d == 3 ? 1.0 : at);
      } else {
        const int j = i - NQ * NQ - 4 * NQ;
        const double at = GaussRule<NQ>::x(j >> 1);
        x = (j & 1) ? at : 0.0;
        y = (j & 1) ? 0.0 : at;
      }
      phi[e] = legendre(g.mp[m], x) * legendre(g.mq[m], y);
    }
  }
  // the bounds of all of a cell's rates; the evaluation's error per variable from the sum of the
  // coefficients' magnitudes (|P_l| <= 1)
  auto bounds = [&](long long c) -> RateBounds {
    TS u[NV][NM], lo[NV];
    ST::load(st, g.ncell, c, u, lo);
    float uf[NV][NM], d[NV], avg[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float s = 0.f;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        uf[v][m] = (float)u[v][m];
        s += fabsf(uf[v][m]);
      }
      avg[v] = uf[v][0];
      d[v] = 2e-6f * s;
    }
    RateBounds r = rate_bounds<NV>(avg, d, gam, gm1, ihx, ihy);
    auto point = [&](const float (&w)[NV]) {
      const RateBounds b = rate_bounds<NV>(w, d, gam, gm1, ihx, ihy);
      r.lo = fmaxf(r.lo, b.lo);
      r.up = fmaxf(r.up, b.up);
    };
    if constexpr (DIM == 2) {
      S2::template each_point<true>(uf, point);
    } else {
      sfor<S1::NP_LIM>([&](auto I_) {
        constexpr int i = decltype(I_)::value;
        float w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          float x = uf[v][0];
#pragma unroll
          for (int l = 1; l < NM; ++l) x += (float)S1::lim_coef(i, l) * uf[v][l];
          w[v] = x;
        }
        point(w);
      });
    }
    return r;
  };
  if constexpr (BOUND) {
    float lower = 0.f;
    for (long long c = i0; c < g.ncell; c += step) lower = fmaxf(lower, bounds(c).lo);
    floor_end(sc, lower);
    return;
  }
  __syncthreads();
  const float floor_ = __uint_as_float(sc->rate_floor);
  double r = 0.0;
  bool ok = true;
  for (long long c = i0; c < g.ncell; c += step) {
    if (bounds(c).up < floor_) continue;
    TS u[NV][NM], lo[NV];
    ST::load(st, g.ncell, c, u, lo);
    double ub[NV];
    bool varies = false;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      ub[v] = (double)u[v][0] + (double)lo[v];
#pragma unroll
      for (int m = 1; m < NM; ++m) varies = varies || u[v][m] != TS(0);
    }
    bool phys, pphys;
    double rc = rate_of<EQ_EULER, DIM>(g, ub, phys);
    r = (rc > r || rc != rc) ? rc : r;
    ok = ok && phys;
    if (!varies) continue;                    // every point value is the average
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
      double w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double x = ub[v];
#pragma unroll
        for (int m = 1; m < NM; ++m) x = fma(phi[i * NM + m], (double)u[v][m], x);
        w[v] = x;
      }
      rc = rate_of<EQ_EULER, DIM>(g, w, pphys);
      r = (rc > r || rc != rc) ? rc : r;
    }
  }
  rate_end(sc, slot, r, ok);
}

namespace {
// the two kernels of a configuration (scalar laws need no bounds)
struct RateKernels {
  void (*bound)(AuxGeom, const void*, DevScalars*, int);
  void (*evaluate)(AuxGeom, const void*, DevScalars*, int);
};
template <int DIM, int K, int BASIS, class PR>
RateKernels points_kernels() {
  return {&rate_points_kernel<DIM, K, BASIS, PR, true>, &rate_points_kernel<DIM, K, BASIS, PR, false>};
}
template <int DIM, int K, int BASIS>
RateKernels points_kernels(int prec) {
  return prec == PREC_F64 ? points_kernels<DIM, K, BASIS, PrecF64>() : points_kernels<DIM, K, BASIS, PrecF32M>();
}
template <int K>
RateKernels points_kernels(const AuxGeom& g) {
  if (g.dim == 1) return points_kernels<1, K, BASIS_Q>(g.prec);
  return g.basis == BASIS_Q ? points_kernels<2, K, BASIS_Q>(g.prec) : points_kernels<2, K, BASIS_P>(g.prec);
}
template <int EQ>
RateKernels averages_kernels(int dim) {
  if constexpr (EQ == EQ_EULER) {
    if (dim == 1) return {&rate_averages_kernel<EQ, 1, true>, &rate_averages_kernel<EQ, 1, false>};
    return {&rate_averages_kernel<EQ, 2, true>, &rate_averages_kernel<EQ, 2, false>};
  } else {
    if (dim == 1) return {nullptr, &rate_averages_kernel<EQ, 1, false>};
    return {nullptr, &rate_averages_kernel<EQ, 2, false>};
  }
}
RateKernels rate_kernels_of(const AuxGeom& g) {
  if (g.eq == EQ_EULER) {
    if (!g.pp) return averages_kernels<EQ_EULER>(g.dim);
    return g.k == 1 ? points_kernels<1>(g) : (g.k == 2 ? points_kernels<2>(g) : points_kernels<3>(g));
  }
  return g.eq == EQ_BURG ? averages_kernels<EQ_BURG>(g.dim) : averages_kernels<EQ_ADV>(g.dim);
}
}  // namespace

cudaError_t launch_rate(const AuxGeom& g, const void* state, DevScalars* sc, int slot, cudaStream_t s) {
  unsigned blocks = (unsigned)((g.ncell + 255) / 256);
  if (blocks > 1216) blocks = 1216;
  const RateKernels k = rate_kernels_of(g);
  if (k.bound) k.bound<<<blocks, 256, 0, s>>>(g, state, sc, slot);
  k.evaluate<<<blocks, 256, 0, s>>>(g, state, sc, slot);
  return cudaGetLastError();
}
int rate_launches(const AuxGeom& g) { return rate_kernels_of(g).bound ? 2 : 1; }

}  // namespace dgk
