// The two sweeps of a 2D stage for FP64 states (included by stage2d.cu, which
// describes the sweeps): FP64 for what the result's last bits depend on,
// pairs of FP32 numbers for the corrections (line_df.cuh, weno_df.cuh), the
// items whose correction is not small listed and evaluated in FP64.
//
// What bounds them: an all-FP64 stage (x- and y-sweep) needs about 2 200 FP64
// instructions per point at 65 to 77 cycles per warp and sub-partition; here
// about 335 remain (FP64 pipe 46% and 53% busy on the double Mach grid), next
// to about 18 500 others, whose latency and fetch take the rest of the time
// (stalls per issue: fixed latency 1.7 and 1.9, shared memory 1.4 and 1.6, no
// instruction 1.0 and 0.4). Measured per step: double Mach 1920 x 480 13.2 ->
// 3.19 ms; 256^2 1.06 -> 0.34 ms; Burgers rhs 321 x 203, 96 -> 52 us. Error
// relative to the all-FP64 sweeps: weno_df.cuh.
//
// Tiles (128 threads; Shape2D for large grids): the x-sweep takes row segments
// of 124 points. The y-sweep takes blocks of 4 columns x 31 rows: 35 rows
// loaded for 31 (16 columns x 7 rows load 11 for 7, and the point phase is FP64
// work), while the 4 columns are one 32-byte sector of a row. Both give 128 interfaces, one per thread, and
// 51 to 55 KB of shared memory, four CTAs per SM.

// Large Euler grids take CTAs of 256 threads (252 points; 8 columns x 31 rows),
// two per SM: the warps of a sub-partition that belong to one CTA run the same
// code at about the same time and share its fetch (large_tiles).
constexpr int kThreadsF64 = 256;
template <int NT>
struct Shape2D {  // NT: 128, 256, or kWideThreads2D (tiles of 128)
  static constexpr bool WIDE = NT > kThreadsF64;
  static constexpr int T = NT == kThreadsF64 ? NT : kThreads2D;  // threads of a tile
  static constexpr int TX = T - 4;                               // x-sweep points
  static constexpr int C = T / 32, R = 31;                       // y-sweep columns, rows
  static constexpr int min_ctas = WIDE ? 1 : HWENO_MINB_2D_F64 * kThreads2D / T;
};

template <int EQ, int DIR>
using Tile2D = LineTile<Dim2<EQ>::M, DIR, EQ == HWENO_EULER, Dim2<EQ>::M, true>;

using Lists2D = ItemLists<kThreadsF64>;

// Phase 1, loaded point k: state u, the derivatives v along and w across the
// line; stores the flux, the two Jacobian-vector products and the pairs.
template <int EQ, int DIR, bool WIDE>
__device__ __forceinline__ void load_point_2d(const Tile2D<EQ, DIR>& r, int k, const double* u,
                                              const double* v, const double* w, double gm1,
                                              D2 alp, D2 hp) {
  constexpr int M = Dim2<EQ>::M;
  double F[M], h[M], E[M];
  Prim2<double> q{};
  if constexpr (EQ == HWENO_EULER) q = prim2_ir(u, gm1, recip_fp64(u[0]));
  flux2<EQ, DIR>(u, q, F);
  jvp2<EQ, DIR>(u, q, v, gm1, h);
  jvp2<EQ, DIR>(u, q, w, gm1, E);
#pragma unroll
  for (int c = 0; c < M; ++c) {
    r.U(c, k) = u[c];
    r.N(c, k) = v[c];
    if (EQ != HWENO_EULER || c > 0) {
      r.F(c, k) = F[c];
      r.h(c, k) = h[c];
    }
    r.extra(c, k) = E[c];
  }
  if constexpr (EQ == HWENO_EULER)
    point_eigen(r, k, u[0], q.ir, q.Ep, DIR == 0 ? q.u : q.v, DIR == 0 ? q.v : q.u);
  if constexpr (!WIDE) point_pairs(r, k, v, h, alp, hp);
}

// The wide form of the sweeps (wide_items), for grids with at most one tile
// per SM: four threads per point (roles), in phases 2 and 4 one component each.
// Measured, two steps: density wave 48^2 370 -> 274 us, 100 x 60 379 -> 286 us.
constexpr int kWideThreads2D = 4 * kThreads2D;
template <int EQ, int DIR>
constexpr size_t xch_bytes(int LI) {
  return sizeof(D2) * WideRoles<Dim2<EQ>::M, false>::rows * LI;
}

// Phase 3 of one thread: interface j (left point kf) and limiter point j
// (point kl), where there are such.
template <int EQ, int DIR>
__device__ __forceinline__ void items_2d(const Tile2D<EQ, DIR>& r, int j, bool has_f, int kf,
                                         bool has_l, int kl, int S, double alpha, double dx,
                                         double idx, const SchemeParams& sp, Lists2D& ls) {
  constexpr int M = Dim2<EQ>::M;
  double x[M];
  if (has_f) {
    double d[M];
    if (!interface_line<D2, DIR>(r, kf, S, alpha, dx, sp, x, d))
      ls.f[atomicAdd(&ls.nf, 1)] = (unsigned short)j;
#pragma unroll
    for (int c = 0; c < M; ++c) {
      r.C(c, j) = x[c];
      r.D(c, j) = d[c];
    }
  }
  if (has_l && sp.limiter != 0) {
    if (!limiter_line<D2, DIR>(r, kl, S, dx, idx, sp, x))
      ls.l[atomicAdd(&ls.nl, 1)] = (unsigned short)j;
#pragma unroll
    for (int c = 0; c < M; ++c) r.lim(c, j) = x[c];
  }
}

// The differences of a point k between interfaces ja and jb: of f-hat, of the
// derivative flux, and of the central flux of Eq. mixed (times 12).
template <int EQ, int DIR>
__device__ __forceinline__ void differences_2d(const Tile2D<EQ, DIR>& r, int c, int k, int S,
                                               int ja, int jb, double& dF, double& dD,
                                               double& dE) {
  dF = madd(0.5, sub(r.F(c, k + S), r.F(c, k - S)), sub(r.C(c, jb), r.C(c, ja)));
  dD = sub(r.D(c, jb), r.D(c, ja));
  dE = madd(8.0, sub(r.extra(c, k + S), r.extra(c, k - S)),
            sub(r.extra(c, k - 2 * S), r.extra(c, k + 2 * S)));
}

template <int EQ, int NT>
__global__ void __launch_bounds__(NT, Shape2D<NT>::min_ctas)
k_xsweep_2d_f64(const __grid_constant__ Args2D a, int mode) {
  constexpr int M = Dim2<EQ>::M, T = Shape2D<NT>::T;
  constexpr int TX = Shape2D<NT>::TX;
  constexpr bool WIDE = Shape2D<NT>::WIDE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Lists2D ls;
  if (a.skip_done && !(a.t[0] < a.t_end)) return;
  const int nx = a.nx;
  const long long N = (long long)nx * a.ny;
  // block -> (row segment, row): the full segments of every row first, the
  // ragged last segments (shorter work) at the end of the dispatch order
  int tile = blockIdx.x, row_ = blockIdx.y;
  {
    const int T = gridDim.x, F = T - 1;
    if (F > 0 && nx % TX != 0) {
      const long long b = (long long)blockIdx.y * T + blockIdx.x, full = (long long)a.ny * F;
      if (b < full) { tile = (int)(b % F); row_ = (int)(b / F); }
      else { tile = F; row_ = (int)(b - full); }
    }
  }
  const int i0 = tile * TX, np = min(TX, nx - i0);
  HWENO_CHECK(np >= 1 && row_ >= 0 && row_ < a.ny, a.status);
  const long long row = (long long)row_ * nx;
  const double dx = a.geod[0], idx = a.geod[1], idx2 = a.geod[2];
  const double alpha = a.alpha_in[0], gm1 = a.sp.wd[9] - 1.0;
  if (threadIdx.x == 0) {
    ls.nf = ls.nl = 0;
    if (mode == MODE_STAGE1 && blockIdx.x == 0 && blockIdx.y == 0) {
      int lands;
      const double dt = time_step2(a, lands);
      a.dt[0] = dt;
      a.lands[0] = lands;
    }
  }
  const D2 alp = scale_pair(alpha), hp = to_pair(dx);
  const Tile2D<EQ, 0> r{reinterpret_cast<double*>(smem_raw), TX + 4, TX + 1, a.status,
                        div(D2{1.f, 0.f}, alp)};

  // 1: points
  for (int g = threadIdx.x; g < np + 4; g += NT) {
    const Src s = map_x(i0 - 2 + g, nx, a.sp);
    HWENO_CHECK(s.kind == 2 || (s.idx >= 0 && s.idx < nx), a.status);
    double u[M], v[M], w[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
      if (s.kind == 2) {
        u[c] = imposed(a.sp, s, c);
        v[c] = w[c] = 0.0;
      } else {
        const long long q = c * N + row + s.idx;
        u[c] = static_cast<const double*>(a.U)[q];
        v[c] = static_cast<const double*>(a.V)[q];
        w[c] = static_cast<const double*>(a.W)[q];
        if (s.kind == 1) {
          if (refl2<EQ, 0>(c) < 0.f) { u[c] = -u[c]; w[c] = -w[c]; }
          else v[c] = -v[c];
        }
      }
    }
    load_point_2d<EQ, 0, WIDE>(r, g, u, v, w, gm1, alp, hp);
  }
  __syncthreads();
  const int role = threadIdx.x / T, j = threadIdx.x % T;
  auto at = [](int i, bool lim) { return lim ? i + 2 : i + 1; };
  if constexpr (WIDE) {
    // 2: pairs of points and edges
    if (role < M && j < np + 4) point_pair(r, role, j, r.N(role, j), r.h(role, j), alp, hp);
    if (role < M && j < np + 3) edge_pair(r, role, j, 1, alp);
    __syncthreads();
    // 3: interfaces and limiter
    wide_items<0, false>(r, reinterpret_cast<D2*>(smem_raw + Tile2D<EQ, 0>::bytes(r.L, r.LI)), role,
                         j, j <= np, j + 1, j < np, j + 2, 1, alpha, dx, idx, a.sp, ls, at, 0);
    __syncthreads();
  } else {
    // 2: edges
    for (int g = threadIdx.x; g < np + 3; g += NT) edge_pairs(r, g, 1, alp);
    __syncthreads();
    // 3: interfaces and limiter
    items_2d<EQ, 0>(r, j, j <= np, j + 1, j < np, j + 2, 1, alpha, dx, idx, a.sp, ls);
    __syncthreads();
    if (ls.nf + ls.nl > 0) {
      listed_items<0>(r, ls.f, ls.nf, ls.l, ls.nl, at, 1, tile + row_, alpha, dx, idx, a.sp);
      __syncthreads();
    }
  }
  // 4: the x parts
  if (j < np && role < M) {
    const int k = j + 2;
    HWENO_CHECK(i0 + j < nx, a.status);
    const long long q = row + i0 + j;
    double* LX = static_cast<double*>(a.LX);
    double* VT = static_cast<double*>(a.VT);
#pragma unroll
    for (int cc = 0; cc < (WIDE ? 1 : M); ++cc) {
      const int c = WIDE ? role : cc;
      double dF, dD, dE;
      differences_2d<EQ, 0>(r, c, k, 1, j, j + 1, dF, dD, dE);
      LX[c * N + q] = mul(-dF, idx);
      LX[(M + c) * N + q] = mul(-dD, idx2);
      LX[(2 * M + c) * N + q] = mul(dE, mul(idx, -1.0 / 12.0));
      VT[c * N + q] = a.sp.limiter ? r.lim(c, j) : r.N(c, k);
    }
  }
}

template <int EQ, int NT>
__global__ void __launch_bounds__(NT, Shape2D<NT>::min_ctas)
k_ysweep_2d_f64(const __grid_constant__ Args2D a, int mode) {
  constexpr int M = Dim2<EQ>::M, T = Shape2D<NT>::T;
  constexpr bool WIDE = Shape2D<NT>::WIDE;
  constexpr int C = Shape2D<NT>::C, R = Shape2D<NT>::R, L = (R + 4) * C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Lists2D ls;
  __shared__ unsigned s_top[2];
  if (a.skip_done && !(a.t[0] < a.t_end)) return;
  const int nx = a.nx, ny = a.ny;
  const long long N = (long long)nx * ny;
  const int i0 = blockIdx.x * C, j0 = blockIdx.y * R;
  const int ncol = min(C, nx - i0), nrow = min(R, ny - j0);
  HWENO_CHECK(ncol >= 1 && nrow >= 1, a.status);
  const double dy = a.geod[3], idy = a.geod[4], idy2 = a.geod[5];
  const double alpha = a.alpha_in[1], gm1 = a.sp.wd[9] - 1.0;
  if (threadIdx.x == 0) {
    ls.nf = ls.nl = 0;
    s_top[0] = s_top[1] = 0u;
  }
  // the stage's time step (stage 1: written by the x-sweep before it) and
  // boundary time
  const double dt = mode == MODE_RHS ? 0.0 : a.dt[0];
  const D2 alp = scale_pair(alpha), hp = to_pair(dy);
  const Tile2D<EQ, 1> r{reinterpret_cast<double*>(smem_raw), L, (R + 1) * C, a.status,
                        div(D2{1.f, 0.f}, alp)};

  // 1: points
  for (int k = threadIdx.x; k < L; k += NT) {
    const int rr = k / C, col = k % C, i = i0 + col;
    if (col >= ncol || rr >= nrow + 4) continue;
    const int jj = j0 - 2 + rr;
    Src s{jj, 0, 0};
    if (jj < 0 || jj >= ny)
      s = map_y(jj, ny, i, a.x0, a.dx, a.y0, a.dy, __dadd_rn(a.t[0], __dmul_rn(a.stage_c, dt)),
                a.sp);
    HWENO_CHECK(s.kind == 2 || (s.idx >= 0 && s.idx < ny && i < nx), a.status);
    double u[M], v[M], w[M];
#pragma unroll
    for (int c = 0; c < M; ++c) {
      if (s.kind == 2) {
        u[c] = imposed(a.sp, s, c);
        v[c] = w[c] = 0.0;
      } else {
        const long long q = c * N + (long long)s.idx * nx + i;
        u[c] = static_cast<const double*>(a.U)[q];
        v[c] = static_cast<const double*>(a.V)[q];
        w[c] = static_cast<const double*>(a.W)[q];
        if (s.kind == 1) {
          if (refl2<EQ, 1>(c) < 0.f) { u[c] = -u[c]; v[c] = -v[c]; }
          else w[c] = -w[c];
        }
      }
    }
    load_point_2d<EQ, 1, WIDE>(r, k, u, w, v, gm1, alp, hp);
  }
  __syncthreads();
  // 3: interfaces y_{j0+r-1/2}, r = 0..nrow (lower point in loaded row r + 1),
  // and the limiter of the points of row r (loaded row r + 2)
  const int role = threadIdx.x / T, j = threadIdx.x % T, rr = j / C;
  const bool in = j % C < ncol, has_f = in && rr <= nrow, mine = in && rr < nrow;
  auto at = [](int i, bool lim) { return lim ? i + 2 * C : i + C; };
  if constexpr (WIDE) {
    if (role < M)
      for (int k = j; k < L; k += T) {
        if (k % C >= ncol) continue;
        if (k / C < nrow + 4) point_pair(r, role, k, r.N(role, k), r.h(role, k), alp, hp);
        if (k / C < nrow + 3) edge_pair(r, role, k, C, alp);
      }
    __syncthreads();
    wide_items<1, false>(r, reinterpret_cast<D2*>(smem_raw + Tile2D<EQ, 1>::bytes(r.L, r.LI)), role,
                         j, has_f, j + C, mine, j + 2 * C, C, alpha, dy, idy, a.sp, ls, at, 0);
    __syncthreads();
  } else {
    for (int k = threadIdx.x; k < (R + 3) * C; k += NT)
      if (k % C < ncol && k / C < nrow + 3) edge_pairs(r, k, C, alp);
    __syncthreads();
    items_2d<EQ, 1>(r, j, has_f, j + C, mine, j + 2 * C, C, alpha, dy, idy, a.sp, ls);
    __syncthreads();
    if (ls.nf + ls.nl > 0) {
      listed_items<1>(r, ls.f, ls.nf, ls.l, ls.nl, at, C, blockIdx.x + blockIdx.y, alpha, dy, idy,
                      a.sp);
      __syncthreads();
    }
  }
  // 4: the y parts, the Runge-Kutta combination
  const int k = j + 2 * C;
  const bool want_alpha = mode == MODE_STAGE1 || mode == MODE_STAGE2;
  double un[M];
  float fx = 0.f, fy = 0.f;
  if (mine && role < M) {
    HWENO_CHECK(j0 + rr < ny && i0 + j % C < nx, a.status);
    const long long q = (long long)(j0 + rr) * nx + i0 + j % C;
    const double* LX = static_cast<const double*>(a.LX);
    const double* VT = static_cast<const double*>(a.VT);
    const double b = mode == MODE_STAGE1 ? 1.0 : mode == MODE_STAGE2 ? 0.25 : 2.0 / 3.0;
    const double a0 = mode == MODE_STAGE2 ? 0.75 : 1.0 / 3.0;
    const double bdt = mul(b, dt);
#pragma unroll
    for (int cc = 0; cc < (WIDE ? 1 : M); ++cc) {
      const int c = WIDE ? role : cc;
      const long long qc = c * N + q;
      double dG, dT, dX;
      differences_2d<EQ, 1>(r, c, k, C, j, j + C, dG, dT, dX);
      const double l1 = madd(-idy, dG, LX[qc]), l3 = madd(-idy2, dT, LX[(2 * M) * N + qc]);
      const double l2 = madd(mul(idy, -1.0 / 12.0), dX, LX[M * N + qc]);
      const double vt = VT[qc], wt = a.sp.limiter ? r.lim(c, j) : r.N(c, k);
      if (mode == MODE_RHS) {
        static_cast<double*>(a.L1)[qc] = l1;
        static_cast<double*>(a.L2)[qc] = l2;
        static_cast<double*>(a.L3)[qc] = l3;
        if (a.Wlim) static_cast<double*>(a.Wlim)[qc] = wt;
      } else {
        // b (x + dt L) first, then a x0 added in one operation: one rounding
        // of the full value
        double x = r.U(c, k), y = vt, z = wt;
        if (mode == MODE_STAGE1) {  // b = 1, a = 0
          x = madd(bdt, l1, x);
          y = madd(bdt, l2, y);
          z = madd(bdt, l3, z);
          static_cast<double*>(a.Wt0out)[qc] = wt;
        } else {
          x = madd(bdt, l1, mul(b, x));
          y = madd(bdt, l2, mul(b, y));
          z = madd(bdt, l3, mul(b, z));
          x = madd(a0, static_cast<const double*>(a.U0)[qc], x);
          y = madd(a0, static_cast<const double*>(a.Vt0)[qc], y);
          z = madd(a0, static_cast<const double*>(a.Wt0)[qc], z);
        }
        un[cc] = x;
        if constexpr (WIDE) reinterpret_cast<double&>(r.H(0, c, k)) = x;  // (not read in phase 4)
        static_cast<double*>(a.Uout)[qc] = x;
        static_cast<double*>(a.Vout)[qc] = y;
        static_cast<double*>(a.Wout)[qc] = z;
      }
    }
  }
  if constexpr (WIDE) {
    if (!want_alpha) return;
    __syncthreads();
    if (role > 0) {
      __syncthreads();  // (the one below)
      return;
    }
    if (mine)
#pragma unroll
      for (int c = 0; c < M; ++c) un[c] = reinterpret_cast<double&>(r.H(0, c, k));
  }
  if (mine && want_alpha) rough_speeds2<EQ>(un, a.sp.wf[9], fx, fy);
  // wave speeds of the new state: in FP64 only where the FP32 ones come
  // within 2^-9 of the tile's largest (or are not usable)
  if (want_alpha) {
    const unsigned tx = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fx, 0.f)));
    const unsigned ty = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fy, 0.f)));
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&s_top[0], tx);
      atomicMax(&s_top[1], ty);
    }
    __syncthreads();
    const float topx = __uint_as_float(s_top[0]) * (1.f - 0x1p-9f);
    const float topy = __uint_as_float(s_top[1]) * (1.f - 0x1p-9f);
    double ax = 0.0, ay = 0.0;
    if (mine && !(fx < topx && fy < topy)) {
      double sx, sy;
      speeds2<EQ>(un, a.sp.wd[9], sx, sy);
      if (!(sx <= real_max<double>()) || !(sy <= real_max<double>()))
        atomicOr(a.status, STATUS_NONFINITE);
      ax = fmax(ax, sx);
      ay = fmax(ay, sy);
    }
    if (__any_sync(0xffffffffu, ax > 0.0 || ay > 0.0)) {
      const unsigned long long mx = warp_max_bits(ax), my = warp_max_bits(ay);
      if ((threadIdx.x & 31) == 0) {
        atomicMax(&a.alpha_out[0], mx);
        atomicMax(&a.alpha_out[1], my);
      }
    }
  }
}

template <int EQ, int NT>
cudaError_t xsweep_f64(int mode, const Args2D& a, cudaStream_t s) {
  constexpr int TX = Shape2D<NT>::TX;
  constexpr size_t bytes = Tile2D<EQ, 0>::bytes(TX + 4, TX + 1) +
                           (Shape2D<NT>::WIDE ? xch_bytes<EQ, 0>(TX + 1) : 0);
  static unsigned configured = 0;  // devices whose limit is raised
  if (const cudaError_t e = ensure_smem_limit(k_xsweep_2d_f64<EQ, NT>, bytes, configured)) return e;
  const dim3 grid((a.nx + TX - 1) / TX, a.ny);
  k_xsweep_2d_f64<EQ, NT><<<grid, NT, bytes, s>>>(a, mode);
  return cudaGetLastError();
}

template <int EQ, int NT>
cudaError_t ysweep_f64(int mode, const Args2D& a, cudaStream_t s) {
  constexpr int C = Shape2D<NT>::C, R = Shape2D<NT>::R, LI = (R + 1) * C;
  constexpr size_t bytes = Tile2D<EQ, 1>::bytes((R + 4) * C, LI) +
                           (Shape2D<NT>::WIDE ? xch_bytes<EQ, 1>(LI) : 0);
  static unsigned configured = 0;  // devices whose limit is raised
  if (const cudaError_t e = ensure_smem_limit(k_ysweep_2d_f64<EQ, NT>, bytes, configured)) return e;
  const dim3 grid((a.nx + C - 1) / C, (a.ny + R - 1) / R);
  k_ysweep_2d_f64<EQ, NT><<<grid, NT, bytes, s>>>(a, mode);
  return cudaGetLastError();
}

// The wide form of a sweep while its tiles number at most one per SM. Euler
// takes CTAs of 256 threads from four waves (of two per SM) of them on, unless
// their wider tiles cover more than 5% more threads (a step with them always /
// never, ms: 256^2 0.348 / 0.335, 512^2 1.067 / 1.019 (x-sweep padded by 20%),
// 640^2 1.468 / 1.488, 1000 x 500 1.687 / 1.782, 1024^2 3.39 / 3.52); Burgers, with
// a quarter of the instructions to fetch, never (1024^2 0.894 / 0.839).
inline bool large_tiles(long long tiles, long long tiles256) {
  return tiles256 >= 4 * 2 * kSMs && 40 * tiles256 <= 21 * tiles;
}
template <int EQ>
cudaError_t xsweep_f64(int mode, const Args2D& a, cudaStream_t s) {
  auto tiles = [&](int TX) { return (long long)((a.nx + TX - 1) / TX) * a.ny; };
  const long long n = tiles(Shape2D<kThreads2D>::TX);
  if (n <= kSMs) return xsweep_f64<EQ, kWideThreads2D>(mode, a, s);
  if constexpr (EQ == HWENO_EULER)
    if (large_tiles(n, tiles(Shape2D<kThreadsF64>::TX)))
      return xsweep_f64<EQ, kThreadsF64>(mode, a, s);
  return xsweep_f64<EQ, kThreads2D>(mode, a, s);
}
template <int EQ>
cudaError_t ysweep_f64(int mode, const Args2D& a, cudaStream_t s) {
  constexpr int R = Shape2D<kThreads2D>::R;
  auto tiles = [&](int C) { return (long long)((a.nx + C - 1) / C) * ((a.ny + R - 1) / R); };
  const long long n = tiles(Shape2D<kThreads2D>::C);
  if (n <= kSMs) return ysweep_f64<EQ, kWideThreads2D>(mode, a, s);
  if constexpr (EQ == HWENO_EULER)
    if (large_tiles(n, tiles(Shape2D<kThreadsF64>::C)))
      return ysweep_f64<EQ, kThreadsF64>(mode, a, s);
  return ysweep_f64<EQ, kThreads2D>(mode, a, s);
}
