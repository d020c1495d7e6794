// stage1d.cuh — 1D SSP-RK3 steps with the jump filter: whole steps (step1d_kernel, the batched kernels),
// and single stages for the variants that need the whole mesh between stages.
//
// Per cell K_j and stage (Section 2.1):
//   R^l = (2l+1)/h [ sum_q w_q f(u_h(xi_q)) P_l'(xi_q) - f^_{j+1/2} + (-1)^l f^_{j-1/2} ]   (Eq. scheme:DG)
//   u~ = c0 u^n + c1 (u^(s) + dt R)                                                          (Eq. rkdg1)
//   u^l <- exp(-sigma^l dt) u~^l,  sigma^l = beta/(h Hbar) max_v (J_0 + sum_{m=1..l} m(m+1) h^m J_m)
// the last line being Eqs. (para:damp2)-(para:damp21) with c_f^l = beta/(4 l(l+1)) (1/Hbar for
// Euler, Section 3.1) substituted, the max over components of Eq. (para:dampsystems1d), and
// J_m = |[d^m u]_{j-1/2}| + |[d^m u]_{j+1/2}| with physical derivatives (2/h)^m d^m/dxi^m, so that the
// weight of a reference derivative is m(m+1) 2^m.
//
// Parallel structure: one lane per cell; traces, face fluxes, end derivatives and face sums of jumps
// move between neighbouring cells through a link (WarpLink: shuffles; BlockLink: shuffles, and shared
// memory across the warps of a block). Each face flux and face jump is computed once, by the face's
// left cell. A stage needs two cells on each side. Outflow boundaries: lanes outside the mesh are ghost
// cells holding the constant state of the adjacent interior cell's average (for the fluxes that of the
// stage input, for the jumps that of u~).
#pragma once
#include "stage2d.cuh"

namespace dgk {

struct Stage1DArgs {
  const void* uin;
  const void* un;
  void* uout;
  int nx;
  long long ncell;
  double h;
  int bc;            // BC_PERIODIC or BC_OUTFLOW (both ends alike)
  double c0, c1;     // one stage's Shu-Osher coefficients (step1d_kernel: SO_C0, SO_C1 of each stage)
  int stage;
  int filter_on;      // FILT_OFF, FILT_JUMP or FILT_GLOBAL
  double gamma, ax, cfl;
  long long nwarps;  // strips of 28 output cells; step1d_kernel: tiles
  int positivity;    // Euler: Zhang-Shu limiter after the filter
  int hybrid;        // hybrid limiter (Algorithm 1): store u^DG, eta and the filter factors
  HybridOut hyb;
  OedgOut oe;        // OEDG damping (kernels instantiated with OE = true)
  DevScalars* sc;
  // mesh constants computed once on the host (stage1d_consts): 1/h in both arithmetic types, c0 as a
  // double-float
  double inv_h_d;
  float inv_h_f;
  float c0_hi, c0_lo;
};

// Fill the host-side constants of a Stage1DArgs from its h and c0 (no FP64 division on the GPU).
inline void stage1d_consts(Stage1DArgs& a) {
  a.inv_h_d = 1.0 / a.h;
  a.inv_h_f = (float)a.inv_h_d;
  a.c0_hi = (float)a.c0;
  a.c0_lo = (float)(a.c0 - (double)a.c0_hi);
}

// Cells of halo on each side of a whole step's tile (two per stage), and the most threads of its block.
constexpr int STEP_HALO = 6;
constexpr int STEP_THREADS = 256;

// Shu-Osher coefficients of the three stages.
__host__ __device__ constexpr double so_c0(int stage) { return stage == 0 ? 0.0 : (stage == 1 ? 0.75 : 1.0 / 3.0); }
__host__ __device__ constexpr double so_c1(int stage) { return stage == 0 ? 1.0 : (stage == 1 ? 0.25 : 2.0 / 3.0); }

// Values of P_l at the positivity limiter's points in 1D (degree K), [point][l]: the Gauss points, both
// ends and, for K = 3, the node 0 of the 3-point Gauss-Lobatto rule (Zhang and Shu's positivity of the
// averages uses the Lobatto nodes with 2N - 3 >= k; for K = 2 the node 0 is a Gauss node already).
__host__ __device__ constexpr int limiter_points1(int K) { return K + 3 + ((K >= 2 && K % 2 == 1) ? 1 : 0); }
template <int K>
__host__ __device__ constexpr double limiter_value1(int i, int l) {
  return i <= K ? GaussRule<K + 1>::P(l, i < K + 1 ? i : 0)
                : (i == K + 1 ? ((l & 1) ? -1.0 : 1.0) : (i == K + 2 ? 1.0 : GaussRule<1>::P(l, 0)));
}
template <int K, class T>
constexpr carr<T, limiter_points1(K) * (K + 1)> limiter_values1() {
  carr<T, limiter_points1(K) * (K + 1)> t{};
  for (int i = 0; i < limiter_points1(K); ++i)
    for (int l = 0; l <= K; ++l) t[i * (K + 1) + l] = (T)limiter_value1<K>(i, l);
  return t;
}
template <int K, class T>
__constant__ carr<T, limiter_points1(K) * (K + 1)> lim_table1 = limiter_values1<K, T>();

// Neighbour values of a warp's 32 cells. The end lanes get their own values.
template <class T>
struct WarpLink {
  template <int N>
  __device__ __forceinline__ void right(const T (&x)[N], T (&y)[N], int) {
#pragma unroll
    for (int n = 0; n < N; ++n) y[n] = __shfl_down_sync(0xffffffffu, x[n], 1);
  }
  template <int N>
  __device__ __forceinline__ void left(const T (&x)[N], T (&y)[N], int) {
#pragma unroll
    for (int n = 0; n < N; ++n) y[n] = __shfl_up_sync(0xffffffffu, x[n], 1);
  }
};
// Neighbour values of a block's cells. Each exchange of a stage has its own buffer (the last argument),
// so one barrier per exchange suffices: a buffer is written again only after the barriers of the
// others. Called by every thread of the block.
constexpr int LINK_BUFFERS = 6, LINK_WARPS = 8, LINK_WORDS = 12;
template <class T>
struct BlockLink {
  T (*sm)[LINK_WARPS][LINK_WORDS];
  int warp, nwarps;
  template <int N>
  __device__ __forceinline__ void right(const T (&x)[N], T (&y)[N], int buf) {
    static_assert(N <= LINK_WORDS, "exchange too wide");
    const int lane = threadIdx.x & 31;
    if (nwarps > 1) {
      if (lane == 0) {
#pragma unroll
        for (int n = 0; n < N; ++n) sm[buf][warp][n] = x[n];
      }
      __syncthreads();
    }
#pragma unroll
    for (int n = 0; n < N; ++n) y[n] = __shfl_down_sync(0xffffffffu, x[n], 1);
    if (lane == 31 && warp + 1 < nwarps) {
#pragma unroll
      for (int n = 0; n < N; ++n) y[n] = sm[buf][warp + 1][n];
    }
  }
  template <int N>
  __device__ __forceinline__ void left(const T (&x)[N], T (&y)[N], int buf) {
    static_assert(N <= LINK_WORDS, "exchange too wide");
    const int lane = threadIdx.x & 31;
    if (nwarps > 1) {
      if (lane == 31) {
#pragma unroll
        for (int n = 0; n < N; ++n) sm[buf][warp][n] = x[n];
      }
      __syncthreads();
    }
#pragma unroll
    for (int n = 0; n < N; ++n) y[n] = __shfl_up_sync(0xffffffffu, x[n], 1);
    if (lane == 0 && warp > 0) {
#pragma unroll
      for (int n = 0; n < N; ++n) y[n] = sm[buf][warp - 1][n];
    }
  }
};

// OE = true: the OEDG form of the damping (the kernel stores u~ unfiltered with the jump sums A_v(l)
// and the reductions of OedgOut; the OEDG filter kernel applies the damping).
// COH = true: state loads through L2 (Store), for the persistent batched kernel.
template <int K, int EQ, class PR, bool OE = false, bool COH = false>
struct Stage1D {
  using T = typename PR::T;
  static constexpr int NM = K + 1;
  static constexpr int NV = NVars<EQ, 1>::value;
  static constexpr int NQ = K + 1;
  using GR = GaussRule<NQ>;
  using ST = Store<PR, NV, NM, COH>;
  using S2 = Stage2D<K, EQ, BASIS_Q, PR>;   // its Gauss-node transforms
  // FP32 form, Euler (three variables): the double-float cell averages of variables 0 and 1 in one
  // register pair (packed FP32 instructions, bitwise the same results). Degrees 1 and 2 only
  // (4 M cells: k = 1 0.108 -> 0.105 ms per launch, k = 2 -1 %; k = 3 +0.4 %).
  static constexpr bool PACK_DF = PR::MIXED && NV == 3 && K <= 2;
  using TB = Tab2D<K, BASIS_Q>;        // the 1D mode l is the x-degree p of the tables

  // The coefficients of one stage: c1 dt / h, with its half as a double-float, and c0.
  struct Coef {
    T base, c0;
    df dcf, dc0;
  };
  static __device__ __forceinline__ Coef coef_of_stage(double c1dt, double inv_h, double c0, df dc0) {
    Coef k;
    const double b = c1dt * inv_h;
    k.base = (T)b;
    k.c0 = (T)c0;
    k.dcf = df_from_double(0.5 * b);
    k.dc0 = dc0;
    return k;
  }

  // Where a lane's cell lies: ghost lanes (outflow) are outside the mesh, and the two next to it take
  // the adjacent interior cell's average from the lane on their right or left.
  struct Place {
    long long cell;     // the cell whose words it reads
    bool ghost, take_right, take_left;
    bool edge;          // any lane of the warp or block is a ghost (uniform)
    bool own;           // an output cell
  };

  // One stage of one cell: u, lo from the stage input to the stage output (before the positivity
  // limiter), un, unlo = u^n. bx, phys: wave speed and physicality of the new average. Ghost lanes hold
  // a constant state before and after. GLOBAL: one of the variants with work between the stages
  // (hybrid limiter, OEDG), which records what its second kernel needs.
  template <bool RECORD, class Link>
  static __device__ __forceinline__ void cell_stage(const Stage1DArgs& a, const Coef& k, bool first, T dt, const Place& pl,
                                                    Link& link, T (&u)[NV][NM], T (&lo)[NV], const T (&un)[NV][NM],
                                                    const T (&unlo)[NV], T& bx, bool& phys, T& eta) {
    const T gam = (T)a.gamma, gm1 = (T)(a.gamma - 1.0), ax = (T)a.ax;
    T inv_h;
    if constexpr (PR::MIXED) inv_h = a.inv_h_f;
    else inv_h = a.inv_h_d;
    // traces at xi = -1 and +1, and twice the face fluxes: right face by this lane, left face from the
    // left lane
    T FR[NV], FL[NV];
    {
      T tl[NV], tr[NV], nb[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T e = u[v][0], o = u[v][1];
        if constexpr (K >= 2) e += u[v][2];
        if constexpr (K >= 3) o += u[v][3];
        tr[v] = e + o;
        tl[v] = e - o;
      }
      link.right(tl, nb, 0);
      llf1d_twice<EQ>(tr, nb, FR, gam, gm1, ax);
      link.left(FR, FL, 1);
    }
    // volume integral M[v][l] = sum_q w_q f(u(xi_q)) P_l'(xi_q)
    T M[NV][NM];
    {
      T f[NV][NQ];
#pragma unroll
      for (int v = 0; v < NV; ++v) S2::gauss_values(u[v], f[v]);
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        T w[NV], fq[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) w[v] = f[v][q];
        flux1d<EQ>(w, fq, gm1, ax);
#pragma unroll
        for (int v = 0; v < NV; ++v) f[v][q] = fq[v];
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) S2::template gauss_moments<1>(f[v], M[v]);
    }
    // u~ = u + c1 dt R + c0 (u^n - u): equal to c0 u^n + c1 (u + dt R) when c0 + c1 = 1, and it keeps
    // that identity exact whatever the rounding of c0 and c1. FP32 form: the cell average in
    // double-float, u0 + c0 (un0 - u0) + c1 dt/h (F_L - F_R), a cascaded sum whose face terms are formed
    // bitwise alike on both sides
    if constexpr (PR::MIXED) {
      if constexpr (PACK_DF) {
        // variables 0 and 1 in one register pair (each lane performs the scalar operations)
        const f2 uh{u[0][0], u[1][0]}, ul{lo[0], lo[1]};
        df2_acc m0{uh, ul};
        if (!first) {
          df2_acc d{f2{un[0][0], un[1][0]}, f2{unlo[0], unlo[1]}};
          d.add(df2{-uh, -ul});
          m0.add(df2_mul(k.dc0, d.result()));
        }
        m0.add_prod(k.dcf, f2{FL[0], FL[1]});
        m0.add_prod(k.dcf, -f2{FR[0], FR[1]});
        const df2 r0 = m0.result();
        u[0][0] = r0.hi.x;
        u[1][0] = r0.hi.y;
        lo[0] = r0.lo.x;
        lo[1] = r0.lo.y;
      }
#pragma unroll
      for (int v = PACK_DF ? 2 : 0; v < NV; ++v) {
        df_acc m0{u[v][0], lo[v]};
        if (!first) {
          df_acc d{un[v][0], unlo[v]};
          d.add(df{-u[v][0], -lo[v]});
          m0.add(df_mul(k.dc0, d.result()));
        }
        m0.add_prod(k.dcf, FL[v]);
        m0.add_prod(k.dcf, -FR[v]);
        const df r0 = m0.result();
        u[v][0] = r0.hi;
        lo[v] = r0.lo;
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T dif = FR[v] - FL[v], sum = FR[v] + FL[v];
#pragma unroll
      for (int l = PR::MIXED ? 1 : 0; l < NM; ++l) {
        // FP32: one face at a time, which cancels the volume term without rounding (the sum of the two
        // twice-fluxes would round at twice its size)
        T r;
        if constexpr (PR::MIXED) r = tfma((l & 1) ? T(-0.5) : T(0.5), FL[v], tfma(T(-0.5), FR[v], M[v][l]));
        else r = l == 0 ? tmul(T(-0.5), dif) : tfma(T(-0.5), (l & 1) ? sum : dif, M[v][l]);
        T val = tfma(tmul(k.base, T(2 * l + 1)), r, u[v][l]);
        if (!first) val = tfma(k.c0, tadd(un[v][l], -u[v][l]), val);
        u[v][l] = val;
      }
    }
    T by, invH;
    {
      T ub[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) ub[v] = u[v][0];
      avg_params<EQ, 1>(ub, gam, gm1, ax, ax, bx, by, invH, phys);
    }
    // ghost cells take the constant state of the adjacent interior cell's u~ average
    if (pl.edge) {
      T own[NV], r[NV], l[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) own[v] = u[v][0];
      link.right(own, r, 2);
      link.left(own, l, 3);
      if (pl.ghost) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          u[v][0] = pl.take_right ? r[v] : (pl.take_left ? l[v] : own[v]);
#pragma unroll
          for (int m = 1; m < NM; ++m) u[v][m] = T(0);
        }
      }
    }
    if (!a.filter_on) return;
    // Per variable, the jump of the r-th reference derivative at the right face, weighted and summed
    // over r = 0..l: each face's sums once, by its left cell, the left face's from the left lane.
    // P_l^{(r)}(-1) = (-1)^{l+r} P_l^{(r)}(+1)
    T best[NM];
#pragma unroll
    for (int l = 0; l < NM; ++l) best[l] = T(0);
    {
      T at[NV * NM], nb[NV * NM];                 // at xi = -1, here and in the right cell
      T dr[NV][NM];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        sfor<NM>([&](auto R_) {
          constexpr int r = decltype(R_)::value;
          // modes r, r+1 (and r+2, r+3 of K = 3): the parity of r is x, the other y
          constexpr double c0 = TB::DE[r * (K + 1) + r];
          T x = c0 == 1.0 ? u[v][r] : tmul(u[v][r], (T)c0);
          if constexpr (r + 2 <= K) x = tfma(u[v][r + 2 <= K ? r + 2 : 0], (T)TB::DE[(r + 2 <= K ? r + 2 : 0) * (K + 1) + r], x);
          if constexpr (r + 3 <= K) {
            const T y = tfma(u[v][3], (T)TB::DE[3 * (K + 1) + r], tmul(u[v][r + 1], (T)TB::DE[(r + 1) * (K + 1) + r]));
            dr[v][r] = tadd(x, y);
            at[v * NM + r] = tadd(x, -y);
          } else if constexpr (r + 1 <= K) {
            constexpr double c1 = TB::DE[(r + 1 <= K ? r + 1 : 0) * (K + 1) + r];
            dr[v][r] = tfma(u[v][r + 1 <= K ? r + 1 : 0], (T)c1, x);
            at[v * NM + r] = tfma(u[v][r + 1 <= K ? r + 1 : 0], -(T)c1, x);
          } else {
            dr[v][r] = at[v * NM + r] = x;
          }
        });
      }
      link.right(at, nb, 4);
      T face[NV * NM], lf[NV * NM];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T s = T(-0.0);
        sfor<NM>([&](auto R_) {
          constexpr int r = decltype(R_)::value;
          constexpr double w = jump_weight(r);
          const T j = fabs(tadd(nb[v * NM + r], -dr[v][r]));
          s = r == 0 ? j : tfma(j, (T)w, s);
          face[v * NM + r] = s;
        });
      }
      link.left(face, lf, 5);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int l = 1; l < NM; ++l) {
          const T run = lf[v * NM + l] + face[v * NM + l];
          best[l] = keep_max(best[l], run);
          if constexpr (OE) {
            // A_v(l) = beta / h (J_0 + sum_{m<=l} (2m+1)/m! h^m J_m) for the OEDG filter kernel
            if (pl.own) ((T*)a.oe.A)[(long long)(v * K + l - 1) * a.ncell + pl.cell] = bx * inv_h * run;
          }
        }
      }
      // Algorithm 1: eta = (|[rho]_{j-1/2}| + |[rho]_{j+1/2}|) / (2 h)
      if constexpr (RECORD) eta = (lf[0] + face[0]) * T(0.5) * inv_h;
    }
    if constexpr (!OE) {
      const T rate = -(bx * inv_h * invH) * dt;
      T facs[NM];
#pragma unroll
      for (int l = 1; l < NM; ++l) best[l] *= rate;
      exp_damp(best, facs);
      if (a.filter_on == FILT_GLOBAL) {
        // one coefficient for every mode, from the jumps of all derivative orders (Eq. para:damp)
#pragma unroll
        for (int l = 1; l < NM - 1; ++l) facs[l] = facs[NM - 1];
      }
      if constexpr (RECORD) {
        if (a.hybrid) {
          // u^DG is stored as it is; the blend kernel limits the troubled cells
          hybrid_record<T, K>(a.hyb, a.ncell, pl.cell, pl.own, eta, facs);
          return;
        }
      }
#pragma unroll
      for (int l = 1; l < NM; ++l)
#pragma unroll
        for (int v = 0; v < NV; ++v) u[v][l] *= facs[l];
    }
  }
  // weight of the r-th reference derivative's jump: the jump filter's r(r+1) 2^r (1 for r = 0), the
  // OEDG form's (2r+1)/r! 2^r
  static constexpr double jump_weight(int r) {
    return OE ? (2 * r + 1) / cfact(r) * (1 << r) : (r == 0 ? 1.0 : (double)(r * (r + 1) * (1 << r)));
  }

  // One stage of a 32-cell strip (28 output cells) of one instance, step size dtd (the hybrid limiter and
  // the OEDG form, neither of which runs with the positivity limiter). The output cells'
  // largest wave speed (the CFL rate times h) and physicality are folded into my_speed and my_ok.
  static __device__ void item(const Stage1DArgs& a, double dtd, long long strip, T& my_speed, bool& my_ok) {
    const int lane = threadIdx.x & 31;
    const Coef k = coef_of_stage(a.c1 * dtd, a.inv_h_d, a.c0, df{a.c0_hi, a.c0_lo});
    const Place pl = place(a, strip * STRIP_OUT - 2, lane, 32, 2);
    T u[NV][NM], lo[NV], un[NV][NM], unlo[NV];
    ST::load(a.uin, a.ncell, pl.cell, u, lo);
    if (a.stage > 0) ST::load(a.un, a.ncell, pl.cell, un, unlo);
    if (pl.ghost) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int l = 1; l < NM; ++l) u[v][l] = T(0);
    }
    WarpLink<T> link;
    T bx, eta = T(0);
    bool phys;
    cell_stage<true>(a, k, a.stage == 0, (T)dtd, pl, link, u, lo, un, unlo, bx, phys, eta);
    if (pl.own) {
      ST::store(a.uout, a.ncell, pl.cell, u, lo);
      if (!phys) my_ok = false;
      my_speed = nan_max(bx, my_speed);
    }
    if (a.hybrid) hybrid_max(a.hyb, pl.own ? eta : T(0));
    if constexpr (OE) {
      // u~ is stored as it is; the reductions for the OEDG coefficient
      double osum[NV];
      T omax[NV], omin[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        osum[v] = 0.0;
        omax[v] = -INFINITY;
        omin[v] = INFINITY;
        if (pl.own) {
          osum[v] = (double)u[v][0] + (double)lo[v];
          T w[NQ];
          S2::gauss_values(u[v], w);
#pragma unroll
          for (int g = 0; g < NQ; ++g) {
            omax[v] = fmax(omax[v], w[g]);
            omin[v] = fmin(omin[v], w[g]);
          }
        }
      }
      oedg_reduce<NV>(a.oe, osum, omax, omin);
    }
  }
  // Lane i of `lanes` cells from x0, with `halo` cells on each side that are not its output.
  static __device__ __forceinline__ Place place(const Stage1DArgs& a, long long x0, int i, int lanes, int halo) {
    const int nx = a.nx;
    const unsigned c = column_of(x0) + (unsigned)i;
    const bool per = a.bc == BC_PERIODIC, inside = column_inside(c, nx);
    Place p;
    p.cell = cell_column(c, nx, per);
    p.ghost = !per && !inside;
    p.take_right = c == COLUMN0 - 1;
    p.take_left = c == COLUMN0 + (unsigned)nx;
    p.edge = !per && (x0 < 0 || x0 + lanes > nx);
    p.own = i >= halo && i < lanes - halo && inside;
    return p;
  }

  static constexpr int NP_LIM = limiter_points1(K);
  static __device__ __forceinline__ double lim_coef(int i, int l) { return limiter_value1<K>(i, l); }

  // Zhang-Shu positivity-preserving limiter on one cell (after the filter, Section 3.2 of the paper):
  // density first (theta_1), then pressure (theta_2), at the Gauss points, both ends and, for k = 3,
  // the Lobatto node 0; averages untouched. Returns the largest wave speed over those points of
  // the limited cell (Zhang and Shu's positivity of the averages needs the CFL bound there). One pass
  // takes the smallest density and pressure and the rate; limit_cell runs for the few cells that fail.
  static __device__ __forceinline__ T limit_and_rate(T (&ut)[NV][NM], bool active, T gam, T gm1) {
    T ub[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) ub[v] = ut[v][0];
    const T pbar = pressure_of<NV>(ub, gm1);
    // admissibility margins, relative to the cell average in both precisions (as the oracle):
    // rho(x) >= 1e-3 rho_bar and p(x) >= min(1e-3 (rho_bar + |E_bar|), rho_bar, p_bar); the reasons are
    // those of the 2D limiter
    T eps_r = T(1e-3) * ub[0];
    T eps = T(1e-3) * (ub[0] + fabs(ub[NV - 1]));
    eps_r = ub[0] < eps_r ? ub[0] : eps_r;
    eps = ub[0] < eps ? ub[0] : eps;
    eps = pbar < eps ? pbar : eps;
    T rmin = ub[0], pmin = INFINITY, rate = T(0);
    sfor<NP_LIM>([&](auto I_) {
      constexpr int i = decltype(I_)::value;
      T w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T x = ut[v][0];
        sfor<NM>([&](auto L_) {
          constexpr int l = decltype(L_)::value;
          constexpr double c = limiter_value1<K>(i, l);
          if constexpr (l >= 1 && c != 0.0) x += (T)c * ut[v][l];
        });
        w[v] = x;
      }
      const T inv = arcp(w[0]);
      const T p = gm1 * (w[2] - T(0.5) * w[1] * (w[1] * inv));
      rmin = fmin(rmin, w[0]);
      pmin = fmin(pmin, p);
      rate = nan_max(fabs(w[1] * inv) + asqrt(gam * p * inv), rate);
    });
    const bool fails = active && eps > T(0) && eps_r > T(0) && (rmin < eps_r || pmin < eps);
    if (fails) {
      // a copy, so that only it lives in local memory for the call
      T cell[NV][NM];
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int l = 0; l < NM; ++l) cell[v][l] = ut[v][l];
      rate = limit_cell(cell, eps_r, eps, rmin, gam, gm1);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int l = 1; l < NM; ++l) ut[v][l] = cell[v][l];
    }
    return rate;
  }
  static __device__ __noinline__ T limit_cell(T (&ut)[NV][NM], T eps_r, T eps, T rmin, T gam, T gm1) {
    const carr<T, NP_LIM * NM>& C = lim_table1<K, T>;
    T ub[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) ub[v] = ut[v][0];
    if (rmin < eps_r) {
      const T th1 = (ub[0] - eps_r) / (ub[0] - rmin);
#pragma unroll
      for (int l = 1; l < NM; ++l) ut[0][l] *= th1;
    }
    auto value = [&](int i, T (&w)[NV]) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T x = ut[v][0];
#pragma unroll
        for (int l = 1; l < NM; ++l) x += C[i * NM + l] * ut[v][l];
        w[v] = x;
      }
    };
    T th2 = T(1);
#pragma unroll 1
    for (int i = 0; i < NP_LIM; ++i) {
      T w[NV];
      value(i, w);
      if (pressure_of<NV>(w, gm1) < eps) {
        const T t = pp_segment<NV>(ub, w, eps, gm1);
        th2 = t < th2 ? t : th2;
      }
    }
    if (th2 < T(1)) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int l = 1; l < NM; ++l) ut[v][l] *= th2;
    }
    T rate = T(0);
#pragma unroll 1
    for (int i = 0; i < NP_LIM; ++i) {
      T w[NV];
      value(i, w);
      const T inv = arcp(w[0]);
      const T p = gm1 * (w[2] - T(0.5) * w[1] * (w[1] * inv));
      rate = nan_max(fabs(w[1] * inv) + asqrt(gam * p * inv), rate);
    }
    return rate;
  }

  // Single-instance stage: one warp per strip, step control on the instance's DevScalars.
  static __device__ void run(const Stage1DArgs& a, unsigned char* smem) {
    const StageCtl ctl = stage_begin(a.sc, a.stage, a.cfl);
    if (!ctl.run) return;
    if constexpr (OE) {
      if (blockIdx.x == 0 && threadIdx.x == 0) a.oe.sc->active = 1u;
    }
    T* red = (T*)smem;
    const long long gw = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nwt = (long long)gridDim.x * (blockDim.x >> 5);
    T my_speed = T(0);
    bool my_ok = true;
    // a bounded grid: each warp takes strips gw, gw + nwt, ... so the per-block step control and
    // rate reduction are paid once per block, not once per 28 cells
    for (long long w = gw; w < a.nwarps; w += nwt) item(a, ctl.dt, w, my_speed, my_ok);
    stage_end(a.sc, a.stage, ctl, a.cfl, my_speed, a.inv_h_d, my_ok, red);
  }

  // The coefficients of stage `lane` (lanes 0..2) of a step of size dt.
  static __device__ __forceinline__ void step_coef(int lane, double dt, double inv_h_d, Coef* coef) {
    if (lane < 3) {
      const double c0 = lane == 0 ? so_c0(0) : (lane == 1 ? so_c0(1) : so_c0(2));
      const double c1 = lane == 0 ? so_c1(0) : (lane == 1 ? so_c1(1) : so_c1(2));
      const float h0 = lane == 0 ? (float)so_c0(0) : (lane == 1 ? (float)so_c0(1) : (float)so_c0(2));
      const float l0 = lane == 2 ? (float)(so_c0(2) - (double)(float)so_c0(2)) : 0.f;
      coef[lane] = coef_of_stage(c1 * dt, inv_h_d, c0, df{h0, l0});
    }
  }
  // The step of one tile from u^n in un, unlo (already read); stores it and folds its output cells in.
  static __device__ __forceinline__ void step_tile(const Stage1DArgs& a, const Coef* coef, T dt, const Place& pl,
                                                   BlockLink<T>& link, T (&un)[NV][NM], T (&unlo)[NV], T& my_speed,
                                                   bool& my_ok) {
    T u[NV][NM], lo[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      lo[v] = unlo[v];
#pragma unroll
      for (int l = 0; l < NM; ++l) {
        if (l > 0 && pl.ghost) un[v][l] = T(0);
        u[v][l] = un[v][l];
      }
    }
    T bx, rate = T(0), eta;
#pragma unroll 1
    for (int s = 0; s < 3; ++s) {
      bool phys;
      cell_stage<false>(a, coef[s], s == 0, dt, pl, link, u, lo, un, unlo, bx, phys, eta);
      if (pl.own && !phys) my_ok = false;
      if constexpr (EQ == EQ_EULER) {
        if (a.positivity) rate = limit_and_rate(u, !pl.ghost, (T)a.gamma, (T)(a.gamma - 1.0));
      }
    }
    if (pl.own) {
      ST::store(a.uout, a.ncell, pl.cell, u, lo);
      my_speed = nan_max(nan_max(bx, rate), my_speed);
    }
  }

  // A whole step. A block owns tiles of blockDim.x cells, of which all but STEP_HALO on each side are
  // its output: the three stages run on the block's registers, each using up two cells of halo. The
  // state is read and written once per step (one launch per stage moved it 8 times and paid three
  // launches), and the step control is paid once. Bound by instruction issue in the FP32 form and by the
  // FP64 pipe (64 cycles a warp instruction on a quarter of an SM) in FP64. Per step, before and after:
  // Burgers P2 200 cells FP64 27.7 -> 15.0 us, Euler P3 65536 cells FP64 230 -> 160, FP32 form 31.2 ->
  // 12.4, Euler P2 1 M cells FP32 form 156 -> 60, with the limiter 179 -> 69.
  static __device__ void run_step(const Stage1DArgs& a) {
    __shared__ T link_words[LINK_BUFFERS][LINK_WARPS][LINK_WORDS];
    __shared__ Coef coef[3];
    __shared__ T red[32];
    const int out = (int)blockDim.x - 2 * STEP_HALO;
    // the first tile's state is on its way while the step control is read
    long long tile = blockIdx.x;
    Place pl = place(a, tile * out - STEP_HALO, (int)threadIdx.x, (int)blockDim.x, STEP_HALO);
    T un[NV][NM], unlo[NV];
    ST::load(a.un, a.ncell, pl.cell, un, unlo);
    const StageCtl ctl = stage_begin(a.sc, 0, a.cfl,
                                     [&](int lane, const StageCtl& c) { step_coef(lane, c.dt, a.inv_h_d, coef); });
    if (!ctl.run) return;
    BlockLink<T> link{link_words, (int)(threadIdx.x >> 5), (int)(blockDim.x >> 5)};
    const T dt = (T)ctl.dt;
    T my_speed = T(0);
    bool my_ok = true;
    for (;;) {
      step_tile(a, coef, dt, pl, link, un, unlo, my_speed, my_ok);
      tile += gridDim.x;
      if (tile >= a.nwarps) break;
      pl = place(a, tile * out - STEP_HALO, (int)threadIdx.x, (int)blockDim.x, STEP_HALO);
      ST::load(a.un, a.ncell, pl.cell, un, unlo);
    }
    stage_end(a.sc, 2, ctl, a.cfl, my_speed, a.inv_h_d, my_ok, red);
  }
};

template <int K, int EQ, class PR, bool OE = false>
__global__ void __launch_bounds__(256) stage1d_kernel(const Stage1DArgs a) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  Stage1D<K, EQ, PR, OE>::run(a, dyn_smem);
}

template <int K, int EQ, class PR>
__global__ void __launch_bounds__(STEP_THREADS) step1d_kernel(const Stage1DArgs a) {
  Stage1D<K, EQ, PR>::run_step(a);
}

}  // namespace dgk
