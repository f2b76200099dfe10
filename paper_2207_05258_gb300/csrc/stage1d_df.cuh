// One stage of the 1D scheme on a tile for FP64 states (included by
// stage1d_impl.cuh; the structure of a stage is described in stage1d.cu).
//
// What bounds it: the FP64 pipe takes one warp instruction per 65 to 77
// cycles and sub-partition, and an all-FP64 stage needs about 830 per point
// (Euler; it ran the pipe at 86%). Here FP64 keeps what the result's last
// bits depend on (fluxes, the differences of F and U, the linear limited
// derivative, the Runge-Kutta update; scalar equations: the derivative flux),
// about 130 per point; the rest is taken in pairs of FP32 numbers
// (weno_df.cuh), about 7 000 other instructions per point, which issue next to
// the FP64 pipe. Interfaces and points whose correction is not small
// (a percent or so in flows with shocks) go on a list and are evaluated in
// FP64. Measured, 2048 Riemann problems (2.5 M points): 12.8 -> 3.40 ms per
// step (FP64 pipe 47% busy, issue slots 42%; stalls per issue: no instruction
// 0.7, fixed latency 1.8, shared memory 1.6, barriers 1.7, in the persistent
// run's 256-thread CTAs); Buckley-Leverett, 246 k points: 0.40 -> 0.14 ms (FP64
// pipe 72%). Error relative to the all-FP64 form: weno_df.cuh.
// The loops over fields stay rolled: unrolled, the straight code outruns the
// instruction caches (6.9 ms per step when the sides were unrolled too).
//
// Phases, with a barrier after each:
//   1 points      load with ghosts; F, h = f'(u) v in FP64; H^{+-} = dx h^{+-},
//                 dx v and the eigen-system's inputs as pairs
//   2 edges       differences of F and U (FP64, then pairs)
//   3 interfaces  c = f-hat - (F_i + F_{i+1})/2 and the limited derivative
//     and points  from pairs; the derivative flux
//   3b            the list, in FP64
//   4 points      flux differences, update, wave speed
// The tile shape (threads, points per thread) and the stage are run-time
// arguments: one copy of the code for all of them.

template <int EQ>
using Tile1D = LineTile<Dim1<EQ>::M, 0, EQ == HWENO_EULER>;

constexpr int kMaxTile1D = 508;

template <int EQ, int NT, int PPT>
struct Layout1D<EQ, double, NT, PPT> {
  static constexpr int P = NT * PPT - 4;
  static constexpr size_t bytes = Tile1D<EQ>::bytes(P + 4, P + 1);
};

// Phase 1, point g of the tile that starts at s (the pairs of H and dx N are
// left to the caller: N in v, h in h).
template <int EQ, class T>
__device__ __forceinline__ void load_point_df(const T& r, const Args1D& a, const double* U,
                                              const double* V, int n, int s, int g, double* v,
                                              double* h) {
  constexpr int M = Dim1<EQ>::M;
  int kind;
  const int src = map_1d(s - 2 + g, n, a.sp.bc[0], a.sp.bc[1], kind);
  HWENO_CHECK(kind == 2 || (src >= 0 && src < n), a.status);
  double u[M];
#pragma unroll
  for (int c = 0; c < M; ++c) {
    if (kind == 2) {
      u[c] = a.sp.inflow[c];
      v[c] = 0.0;
    } else {
      u[c] = U[(long long)c * n + src];
      v[c] = V[(long long)c * n + src];
      if (kind == 1) {  // one of the two changes sign
        const bool odd = refl_sign<EQ>(c) < 0.f;
        if (odd) u[c] = -u[c];
        else v[c] = -v[c];
      }
    }
    r.U(c, g) = u[c];
    r.N(c, g) = v[c];
  }
  if constexpr (EQ == HWENO_BURGERS) {
    r.F(0, g) = mul(mul(0.5, u[0]), u[0]);
    h[0] = mul(u[0], v[0]);
    r.h(0, g) = h[0];
  } else if constexpr (EQ == HWENO_BUCKLEY) {
    const double w = sub(1.0, u[0]), u4 = mul(4.0, u[0]);
    const double iD = recip_fp64(madd(w, w, mul(u4, u[0])));
    r.F(0, g) = mul(mul(u4, u[0]), iD);
    h[0] = mul(mul(mul(mul(2.0, u4), w), mul(iD, iD)), v[0]);
    r.h(0, g) = h[0];
  } else {
    const double gm1 = a.sp.wd[9] - 1.0;
    const double ir = recip_fp64(u[0]);
    const double vel = mul(u[1], ir);
    const double p = mul(gm1, madd(mul(-0.5, u[1]), vel, u[2]));
    const double Ep = add(u[2], p);
    const double dvel = mul(madd(-vel, v[0], v[1]), ir);
    const double dp = mul(gm1, madd(mul(mul(0.5, vel), vel), v[0], madd(-vel, v[1], v[2])));
    h[0] = v[1];
    h[1] = madd(v[1], vel, madd(u[1], dvel, dp));
    h[2] = madd(add(v[2], dp), vel, mul(Ep, dvel));
    r.F(1, g) = madd(u[1], vel, p);
    r.F(2, g) = mul(Ep, vel);
    r.h(1, g) = h[1];
    r.h(2, g) = h[2];
    point_eigen(r, g, u[0], ir, Ep, vel, 0.0);
  }
}

// Phase 4, component c of point j: the flux differences, and L^1, L^2, v~
// (MODE_RHS) or the Runge-Kutta combination; returns U of the stage output.
struct Update1D {
  double b, a0, k1, k2, idx, idx2;
  __device__ __forceinline__ Update1D(int mode, double dt, double idx_, double idx2_)
      : idx(idx_), idx2(idx2_) {
    b = mode == MODE_STAGE1 ? 1.0 : mode == MODE_STAGE2 ? 0.25 : 2.0 / 3.0;
    a0 = mode == MODE_STAGE2 ? 0.75 : 1.0 / 3.0;
    k1 = mul(-mul(b, dt), idx);
    k2 = mul(-mul(b, dt), idx2);
  }
  template <class T>
  __device__ __forceinline__ double operator()(const T& r, const Args1D& a, const StageIO& io,
                                               int mode, int c, int j, long long q) const {
    const int g = j + 2;
    const double dF = madd(0.5, sub(r.F(c, g + 1), r.F(c, g - 1)), sub(r.C(c, j + 1), r.C(c, j)));
    const double dD = sub(r.D(c, j + 1), r.D(c, j));
    const double vt = a.sp.limiter != 0 ? r.lim(c, j) : r.N(c, g);
    if (mode == MODE_RHS) {
      static_cast<double*>(a.L1)[q] = mul(-dF, idx);
      static_cast<double*>(a.L2)[q] = mul(-dD, idx2);
      if (a.Vlim) static_cast<double*>(a.Vlim)[q] = vt;
      return 0.0;
    }
    // b (x + dt L) first, then a x0 added in one operation: one rounding of
    // the full value
    double x, y;
    if (mode == MODE_STAGE1) {  // b = 1, a = 0
      x = madd(k1, dF, r.U(c, g));
      y = madd(k2, dD, vt);
      static_cast<double*>(io.Vt0out)[q] = vt;
    } else {
      x = madd(k1, dF, mul(b, r.U(c, g)));
      y = madd(k2, dD, mul(b, vt));
      x = madd(a0, static_cast<const double*>(io.U0)[q], x);
      y = madd(a0, static_cast<const double*>(io.Vt0)[q], y);
    }
    static_cast<double*>(io.Uout)[q] = x;
    static_cast<double*>(io.Vout)[q] = y;
    return x;
  }
};

// One stage (mode) on the tile of P points of instance k starting at s.
template <int EQ>
__device__ __forceinline__ void stage_tile_df(const Args1D& a, const StageIO& io, const int mode,
                                              const int P, const int k, const int s) {
  constexpr int M = Dim1<EQ>::M;
  extern __shared__ __align__(16) unsigned char smem1d[];
  const Tile1D<EQ> r{reinterpret_cast<double*>(smem1d), P + 4, P + 1, a.status, D2{}};
  __shared__ double s_dt;
  __shared__ unsigned s_top;
  __shared__ int s_nf, s_nl;  // items of the lists
  __shared__ unsigned short s_f[kMaxTile1D + 1], s_l[kMaxTile1D];
  const int nt = blockDim.x;

  const int n = a.inst_n[k];
  if (a.skip_done && !(a.t[k] < a.t_end)) return;
  const int np = min(P, n - s);
  HWENO_CHECK(s >= 0 && np >= 1 && P <= kMaxTile1D, a.status);
  const long long off = a.inst_off[k] * M;
  const double* geo = a.inst_geo + 3 * k;
  const double dx = geo[0], idx = geo[1], idx2 = geo[2];
  const double alpha = io.alpha_in[k];

  // time step: once per CTA (thread 0), read back after the barriers below
  if (threadIdx.x == 0) {
    double dt = 0.0;
    if (mode == MODE_STAGE1) {
      int lands = 0;
      dt = a.dt_in ? a.dt_in[k]
                   : time_step(a.sp, io.alpha_in[k], a.inst_hx[k], a.t[k], a.t_end, lands);
      if (s == 0) { a.dt[k] = dt; a.lands[k] = lands; }
    } else if (mode != MODE_RHS) {
      dt = a.dt[k];
    }
    s_dt = dt;
    s_top = 0u;
    s_nf = s_nl = 0;
  }

  // 1: points
  {
    const D2 alp = scale_pair(alpha), dxp = to_pair(dx);
    const double* U = static_cast<const double*>(io.U) + off;
    const double* V = static_cast<const double*>(io.V) + off;
    for (int g = threadIdx.x; g < np + 4; g += nt) {
      double v[M], h[M];
      load_point_df<EQ>(r, a, U, V, n, s, g, v, h);
      point_pairs(r, g, v, h, alp, dxp);
    }
    __syncthreads();
    // 2: edges
    for (int g = threadIdx.x; g < np + 3; g += nt) edge_pairs(r, g, 1, alp);
  }
  __syncthreads();

  // 3: interfaces x_{s+j-1/2}, j = 0..np (left point at loaded index j + 1),
  // and the limited derivatives of points j = 0..np-1 (loaded index j + 2)
  const bool limited = a.sp.limiter != 0;
  for (int j = threadIdx.x; j <= np; j += nt) {
    double x[M], d[M];
    if (!interface_line<D2, 0>(r, j + 1, 1, alpha, dx, a.sp, x, d))
      s_f[atomicAdd(&s_nf, 1)] = (unsigned short)j;
#pragma unroll
    for (int c = 0; c < M; ++c) {
      r.C(c, j) = x[c];
      r.D(c, j) = d[c];
    }
    if (j < np && limited) {
      if (!limiter_line<D2, 0>(r, j + 2, 1, dx, idx, a.sp, x))
        s_l[atomicAdd(&s_nl, 1)] = (unsigned short)j;
#pragma unroll
      for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
    }
  }
  __syncthreads();

  // 3b: the lists
  if (s_nf + s_nl > 0) {  // uniform
    listed_items<0>(r, s_f, s_nf, s_l, s_nl, [](int j, bool lim) { return lim ? j + 2 : j + 1; }, 1,
                    k + s / P, alpha, dx, idx, a.sp);
    __syncthreads();
  }

  // 4: points
  const Update1D update(mode, s_dt, idx, idx2);
  const bool want_alpha = mode != MODE_RHS && io.alpha_out != nullptr;  // uniform
  float top = 0.f;
  for (int j = threadIdx.x; j < np; j += nt) {
    const int g = j + 2;
    HWENO_CHECK(s + j < n, a.status);
    double un[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
      un[c] = update(r, a, io, mode, c, j, off + s + j + (long long)c * n);
      // kept for the wave speed below in a row that this phase does not read
      reinterpret_cast<double&>(r.H(0, c, g)) = un[c];
    }
    if (want_alpha) {
      const float f = rough_speed<EQ>(un, a.sp.wf[9]);
      reinterpret_cast<float&>(r.H(1, 0, g)) = f;
      top = fmaxf(top, f);  // a NaN is no bound
    }
  }
  // The wave speed of the stage output (stages 1 and 2; stage 3 as well when
  // the persistent run asks for the next step's alpha): the FP64 speed is
  // evaluated only where the FP32 one comes within 2^-9 of the tile's largest
  // (or is not usable), which cannot miss the maximum.
  if (want_alpha) {
    const unsigned tw = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, tw);
    __syncthreads();
    top = __uint_as_float(s_top) * (1.f - 0x1p-9f);
    double amax = 0.0;
    bool bad = false;
    for (int j = threadIdx.x; j < np; j += nt) {
      const int g = j + 2;
      if (reinterpret_cast<float&>(r.H(1, 0, g)) < top) continue;
      double u[M];
#pragma unroll
      for (int c = 0; c < M; ++c) u[c] = reinterpret_cast<double&>(r.H(0, c, g));
      const double sp = wave_speed<EQ>(u, a.sp.wd[9], a.sp.wd[10]);
      bad |= !(sp <= real_max<double>());
      amax = fmax(amax, sp);
    }
    if (bad) atomicOr(a.status, STATUS_NONFINITE);
    if (__any_sync(0xffffffffu, amax > 0.0)) {
      const unsigned long long m = warp_max_bits(amax);
      if ((threadIdx.x & 31) == 0) atomicMax(&io.alpha_out[k], m);
    }
  }
}

// ---------------------------------------------------------------------------
// The wide form of a stage (wide_items), for launches that leave SMs idle:
// WideRoles threads per point; outside the item phases the threads share the
// components of a point. Results are the bits of stage_tile_df. Measured: the
// tiled form leaves a stage of one small instance to four warps on one SM
// (FP32 chains at 0.3 instructions per cycle); Riemann problem N = 200, one
// step 92 -> 88 us; cluster steps: blast waves N = 800 83 -> 64 us per step,
// Burgers N = 400 17.5 -> 15 us.
// ---------------------------------------------------------------------------
constexpr int kWideMax = 124;   // points of a wide tile
constexpr int kFieldsMax = 60;  // ... with one role per field

// Roles, threads and shared memory of a wide tile of P points (Euler tiles of
// up to kFieldsMax points have a role per field).
template <int EQ>
constexpr bool wide_fields(int P) { return EQ == HWENO_EULER && P <= kFieldsMax; }
template <int EQ>
constexpr int wide_threads(int P) {
  return (wide_fields<EQ>(P) ? WideRoles<Dim1<EQ>::M, true>::count
                             : WideRoles<Dim1<EQ>::M, false, EQ != HWENO_EULER>::count) * (P + 4);
}
template <int EQ>
constexpr size_t wide_bytes(int P) {
  return Tile1D<EQ>::bytes(P + 4, P + 1) +
         sizeof(D2) * WideRoles<Dim1<EQ>::M, true>::rows * (P + 1);
}

// The tile [s, s + P) of instance k from wave speed alpha and time step dt;
// returns (valid in every thread) the largest wave speed of the output as
// bits, when want_alpha.
template <int EQ, bool FIELDS>
__device__ __forceinline__ unsigned long long stage_wide_df(const Args1D& a, const StageIO& io,
                                                            const int mode, const int P,
                                                            const int k, const int s,
                                                            const double alpha, const double dt,
                                                            const bool want_alpha) {
  constexpr int M = Dim1<EQ>::M;
  extern __shared__ __align__(16) unsigned char smem1d[];
  const Tile1D<EQ> r{reinterpret_cast<double*>(smem1d), P + 4, P + 1, a.status, D2{}};
  D2* const xch = reinterpret_cast<D2*>(smem1d + Tile1D<EQ>::bytes(P + 4, P + 1));
  __shared__ unsigned s_top;
  __shared__ unsigned long long s_amax;
  __shared__ ItemLists<kWideMax + 1> ls;
  const int role = threadIdx.x / (P + 4), j = threadIdx.x - role * (P + 4);

  const int n = a.inst_n[k], np = min(P, n - s);
  HWENO_CHECK(s >= 0 && np >= 1 && P <= kWideMax, a.status);
  const long long off = a.inst_off[k] * M;
  const double* geo = a.inst_geo + 3 * k;
  const double dx = geo[0], idx = geo[1], idx2 = geo[2];
  if (threadIdx.x == 0) {
    s_top = 0u;
    s_amax = 0ull;
    ls.nf = ls.nl = 0;
  }
  const D2 alp = scale_pair(alpha), dxp = to_pair(dx);

  // 1: points
  if (role == 0 && j < np + 4) {
    double v[M], h[M];
    load_point_df<EQ>(r, a, static_cast<const double*>(io.U) + off,
                      static_cast<const double*>(io.V) + off, n, s, j, v, h);
  }
  __syncthreads();
  // 2: pairs of points and of edges, a component per role
  if (role < M && j < np + 4) point_pair(r, role, j, r.N(role, j), r.h(role, j), alp, dxp);
  const int er = role - (M == 1 || FIELDS ? M : 0);
  if (er >= 0 && er < M && j < np + 3) edge_pair(r, er, j, 1, alp);
  __syncthreads();
  // 3: items
  wide_items<0, FIELDS, EQ != HWENO_EULER>(r, xch, role, j, j <= np, j + 1, j < np, j + 2, 1, alpha,
                                           dx, idx, a.sp, ls,
                                           [](int i, bool lim) { return lim ? i + 2 : i + 1; }, 0);
  __syncthreads();
  // 4: points, a component per role
  const Update1D update(mode, dt, idx, idx2);
  if (role < M && j < np) {
    HWENO_CHECK(s + j < n, a.status);
    reinterpret_cast<double&>(r.H(0, role, j + 2)) =
        update(r, a, io, mode, role, j, off + s + j + (long long)role * n);
  }
  if (!want_alpha) return 0ull;
  __syncthreads();
  // the wave speed of the stage output, as in stage_tile_df
  double u[M];
  float rough = 0.f;
  if (role == 0) {
    if (j < np) {
#pragma unroll
      for (int c = 0; c < M; ++c) u[c] = reinterpret_cast<double&>(r.H(0, c, j + 2));
      rough = rough_speed<EQ>(u, a.sp.wf[9]);
    }
    const unsigned tw = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(rough, 0.f)));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, tw);
  }
  __syncthreads();
  if (role == 0) {
    double amax = 0.0;
    if (j < np && !(rough < __uint_as_float(s_top) * (1.f - 0x1p-9f))) {
      amax = wave_speed<EQ>(u, a.sp.wd[9], a.sp.wd[10]);
      if (!(amax <= real_max<double>())) atomicOr(a.status, STATUS_NONFINITE);
      amax = fmax(0.0, amax);
    }
    if (__any_sync(0xffffffffu, amax > 0.0)) {
      const unsigned long long m = warp_max_bits(amax);
      if ((threadIdx.x & 31) == 0) atomicMax(&s_amax, m);
    }
  }
  __syncthreads();
  return s_amax;
}
