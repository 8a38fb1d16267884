// fdlb_kernels.cu -- sm_103a kernels of the IMEX finite-difference lattice
// Boltzmann step (Kis & Ambrus): one fused kernel per advected IMEX stage.
//
// Every stage kernel owns a tile of cells and all populations of those cells,
// and runs two passes:
//   pass 1  for each group of G populations: stage the advected array on the
//           tile plus its 5-cell MP-9 halo in shared memory (ghosts by index
//           clamp = outlet copies of the adjacent fluid node, Sec. IV), march
//           every tile line (MP-9 + MP limiter; 2-D in 64-bit fixed point,
//           fdlb_mp9i.cuh, 1-D in binary64, fdlb_mp9.cuh), form the flux
//           difference and the explicit part R_i of the stage (Eq. IMEX),
//           accumulate the moments of R_i per cell (Eq. Moments_discrete) and
//           park R_i and the running accumulators in the output arrays;
//   pass 2  per cell: n, u, T from the moments, the Hermite equilibrium
//           factors (Eq. gExpanded, recurrence form), and the closed-form
//           implicit BGK relaxation of every population (Sec. III).  Stages
//           3 and 4 leave D_i = R_i - F_eq(R_i) in the array D, which the
//           next kernel folds into A4 and A_fin in its pass 1, so that pass 2
//           rewrites the relaxed populations and D only.
// The flux itself never goes to global memory.
#include "fdlb_device.cuh"
#include "fdlb_mp9i.cuh"

namespace fdlb {
namespace {

// ---- pass 2 of a cell --------------------------------------------------------

// n, u, T of the moment sums, the equilibrium's factors, and row by row of
// their outer product (1-D: phi, then chi) D = R - F_eq(R) and the relaxed
// value R - kd D, the next row's values loaded before this row is computed:
//   stage 3   R3 -> F3 and D3 (in D, free until the final stage rewrites it;
//             stage 4 applies its terms to A4 and A_fin),
//   stage 4   R4 -> F4 (in A4) and D4 for the final stage,
//   final and preparation   F -> F2 and D of the new state.
// fac (2-D): QP + QC shared doubles of stride FS for this thread's y factors,
// picked by row at run time (one copy of the row body: code size).
template <int DIM, int QP, int QC, int STAGE, int FS>
__device__ __forceinline__ void relax_cell64(const DevParams& p, const Geo& geo, unsigned c,
                                             const Moments& m, double* fac) {
  const int64_t N = p.N;
  // (stages 3 and 4 relax in place: Rin and Fout are one array there)
  const double* const Rin =
      (const double*)(STAGE == kStage3 ? p.F3 : STAGE == kStage4 ? p.A4 : p.F);
  double* const Fout = (double*)(STAGE == kStage3 ? p.F3 : STAGE == kStage4 ? p.A4 : p.F2);
  double* const Dn = (double*)p.D;
  const StageCoef& sc = p.sc;
  const double kd = STAGE == kStage3 ? sc.a33e3 : STAGE == kStage4 ? sc.a44e4 : sc.c2m1;
  constexpr int W = QP > QC ? QP : QC;
  double cur[W], nxt[W];
#pragma unroll
  for (int j = 0; j < QP; ++j) cur[j] = (Rin + j * N)[c];
  double n, ux, uy, T;
  if (!moments_to_nut<DIM>(geo.invDK, m, n, ux, uy, T)) {
    atomicOr(p.status, 1u);
    if (geo.prob >= 0) atomicOr(&p.pstatus[geo.prob], 1u);
  }
  // populations p0 .. of a row: D = R - F_eq, F_eq = h f, one fused operation
  // except in 1-D where F2 needs F_eq itself (small_stage_kernel does the same)
  auto relax_row = [&](int p0, int nq, const double* h, double f) {
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (j < nq) {
        const int64_t o = (p0 + j) * N;
        const double R = cur[j];
        if constexpr (DIM == 1 && STAGE != kStage3 && STAGE != kStage4) {
          const double fe = __dmul_rn(h[j], f), D = __dsub_rn(R, fe);
          (Dn + o)[c] = D;
          (Fout + o)[c] = fma(sc.c2, D, fe);
        } else {
          const double D = fma(-h[j], f, R);
          (Dn + o)[c] = D;
          (Fout + o)[c] = fma(-kd, D, R);
        }
      }
  };
  auto load_row = [&](int p0, int nq) {
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (j < nq) nxt[j] = (Rin + (p0 + j) * N)[c];
  };
  auto take_row = [&]() {
#pragma unroll
    for (int j = 0; j < W; ++j) cur[j] = nxt[j];
  };
  double h[QP];
  axis_g<QP>(p.wHp, ux, T, h);
  if constexpr (DIM == 1) {
    load_row(QP, QC);
    relax_row(0, QP, h, n);
    take_row();
    const double nchi = geo.kchi * T * n;
    if constexpr (QC == QP) {
      relax_row(QP, QC, h, nchi);
    } else {
      double hc[QC];
      axis_g<QC>(p.wHc, ux, T, hc);
      relax_row(QP, QC, hc, nchi);
    }
  } else {
    const double kT = geo.kchi * T;
    {
      double gy[QP];
      axis_g<QP>(p.wHp, uy, T, gy);
#pragma unroll
      for (int j = 0; j < QP; ++j) fac[j * FS] = n * gy[j];
    }
    if constexpr (QC != QP) {
      double gy[QC];
      axis_g<QC>(p.wHc, uy, T, gy);
#pragma unroll
      for (int j = 0; j < QC; ++j) fac[(QP + j) * FS] = kT * n * gy[j];
    }
#pragma unroll 1
    for (int r = 0; r < QP; ++r) {
      if (r + 1 < QP) load_row((r + 1) * QP, QP);
      else load_row(QP * QP, QC);
      relax_row(r * QP, QP, h, fac[r * FS]);
      take_row();
    }
    double hc[QC];
    if constexpr (QC != QP) axis_g<QC>(p.wHc, ux, T, hc);
#pragma unroll 1
    for (int r = 0; r < QC; ++r) {
      if (r + 1 < QC) load_row(QP * QP + (r + 1) * QC, QC);
      if constexpr (QC == QP) relax_row(QP * QP + r * QC, QC, h, kT * fac[r * FS]);
      else relax_row(QP * QP + r * QC, QC, hc, fac[(QP + r) * FS]);
      take_row();
    }
  }
}

// ---- explicit part of one population of a cell -----------------------------

// The inputs of the update: stage 3 F and D; stage 4 A4, D (holding D3) and
// A_fin; final A_fin and D (holding D4).
struct UpdateIn {
  double a, d, b;
};
template <int STAGE>
__device__ __forceinline__ UpdateIn load_update(const DevParams& p, int64_t o, unsigned c) {
  UpdateIn u;
  u.a = ((const double*)(STAGE == kStage3 ? p.F : STAGE == kStage4 ? p.A4 : p.Af) + o)[c];
  u.d = ((const double*)p.D + o)[c];
  u.b = STAGE == kStage4 ? ((const double*)p.Af + o)[c] : 0.0;
  return u;
}
// R_i of the stage, and the running accumulators to memory.
// PARK: R too, for a second pass of the cell's owner; the final stage's R is the
// new state.
template <int STAGE, bool PARK = true>
__device__ __forceinline__ double store_update(const DevParams& p, int64_t o, unsigned c, bool valid,
                                               const UpdateIn& u, double X) {
  const StageCoef& sc = p.sc;
  double R;
  if constexpr (STAGE == kStage3) {
    R = fma(-sc.at32, X, fma(-sc.k3, u.d, u.a));
    const double a4 = fma(-sc.at42, X, fma(-sc.k4, u.d, u.a));
    const double af = fma(-sc.wt2, X, fma(-sc.kf, u.d, u.a));
    if (valid) {
      if (PARK) ((double*)p.F3 + o)[c] = R;
      ((double*)p.A4 + o)[c] = a4;
      ((double*)p.Af + o)[c] = af;
    }
  } else if constexpr (STAGE == kStage4) {
    R = fma(-sc.at43, X, fma(-sc.a43e3, u.d, u.a));
    const double af = fma(-sc.wt3, X, fma(-sc.w3e3, u.d, u.b));
    if (valid) {
      if (PARK) ((double*)p.A4 + o)[c] = R;
      ((double*)p.Af + o)[c] = af;
    }
  } else {  // kFinal: F^{n+1}
    R = fma(-sc.wt4, X, fma(-sc.w4e4, u.d, u.a));
    if (valid) ((double*)p.F + o)[c] = R;
  }
  return R;
}

// ---- 2-D ------------------------------------------------------------------------

// Moment sums of a cell over groups of 4 populations.  On the lattice of
// 8 x 8 momenta the groups run along kx, first all ky of kx = 0..3, then of
// kx = 4..7: row sums feed jy and the y part of e, and the four column sums
// feed n, jx and the x part of e once per half, 9 binary64 operations per
// group instead of 16.
constexpr int kG = 4;  // populations per group
template <int QP, int QC>
struct GroupMoments {
  static constexpr bool kHalves = QP == 8;
  static constexpr int P = Lat<2, QP, QC>::P;
  static constexpr int NG = (P + kG - 1) / kG;
  Moments m;
  double col[kHalves ? 4 : 1];
  // first population of the gi-th group
  __device__ static __forceinline__ int first(int gi) {
    if constexpr (kHalves) return gi < 8 ? gi * 8 : gi < 16 ? gi * 8 - 60 : gi * 4;
    else return gi * kG;
  }
  __device__ __forceinline__ void add(const DevParams& p, int g0, const double (&v)[kG]) {
    if constexpr (kHalves) {
      const double r = (v[0] + v[1]) + (v[2] + v[3]);
      if (g0 < 64) {
        m.jy = fma(p.py[g0], r, m.jy);
        m.e = fma(p.pp2[g0 >> 3], r, m.e);
#pragma unroll
        for (int g = 0; g < 4; ++g) col[g] += v[g];
      } else {
        m.e += r;
      }
    } else {
#pragma unroll
      for (int g = 0; g < kG; ++g)
        if (g0 + g < P) accumulate<2, QP, QC>(p, m, g0 + g, v[g]);
    }
  }
  // after group gi: fold the columns of a finished half
  __device__ __forceinline__ void fold(const DevParams& p, int gi) {
    if constexpr (kHalves) {
      if (gi == 7 || gi == 15) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int k = gi == 7 ? g : g + 4;
          m.n += col[g];
          m.jx = fma(p.pp[k], col[g], m.jx);
          m.e = fma(p.pp2[k], col[g], m.e);
          col[g] = 0.0;
        }
      }
    }
  }
};

// Named barriers of the two roles of a 2-D CTA.
__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Tile of 16 x 16 cells (or 16 x 8, on small grids); a marching thread for
// every 8-cell half line of a group's populations, an updating one for every
// cell.
template <int TY_>
struct Tile2 {
  static constexpr int TX = 16, TY = TY_, NM = 16 * TY, NU = 16 * TY, SEG = 8;
  static_assert(TY == 8 || TY == 16, "lines of one or two halves");
  static constexpr int SX = TX + 2 * H + 1, SY = TY + 2 * H;  // padded row pitch
};
template <int QP, int QC, int TY>
struct Smem2 {
  using T2 = Tile2<TY>;
  static constexpr int P = Lat<2, QP, QC>::P;
  double tile[2][kG][T2::SY][T2::SX];  // cells + halo
  // flux differences along x and y, in units of their half line's scale, whose
  // exponents are in ex and ey (0: binary64 bits)
  int64_t hx[2][kG][T2::TY][T2::TX + 1];
  int64_t hy[2][kG][T2::TX][T2::TY + 1];
  int ex[2][kG][T2::TY][T2::TX / T2::SEG];
  int ey[2][kG][T2::TX][T2::TY / T2::SEG];
  double fac[QP + (QC == QP ? 0 : QC)][T2::NU];
  AdvCoef coef[P];  // dt |p| / ds
  int cex[P];
  int next[2];  // the tile after this one, after the next one
};

// One fused stage.  Integer and binary64 work run side by side: 8 warps march
// (staging, scaling and the fixed-point MP-9 flux differences: integer pipes)
// one group of populations ahead of 8 warps that update (explicit parts,
// moments and, per tile, pass 2: binary64 pipe), through two buffers of flux
// differences.  Where a CTA has more than one tile, the march of the next one
// runs during pass 2; it takes the tiles from a counter, because those with
// lines that march in binary64 (fdlb_mp9i.cuh) cost more.
// Measured at 512 x 512 x 128 populations, a step: 9.93 ms with every tile
// marching in binary64 and every warp marching and updating in turn (that pipe
// 78 % busy); 3.36 ms for a smooth field, all in fixed point; 3.87 ms for four
// quadrants, where 6 % of the groups have a line in binary64.  What bounds it:
// about 700 instructions per population-cell and stage at half the issue rate,
// the integer pipe and the binary64 pipe each about half busy; 16 warps a CTA
// wait on the fixed latency of 64-bit integer chains.  A line in binary64 is a
// chain of 145 instructions of 64 cycles, about as long again as a group, and
// the last tiles with such lines run beside idle SMs.
template <int QP, int QC, int STAGE, int CTAS, int TY_>
__global__ void __launch_bounds__(Tile2<TY_>::NM + Tile2<TY_>::NU, CTAS)
    stage_kernel_2d(const __grid_constant__ DevParams p, int ntx, int ntiles) {
  using L = Lat<2, QP, QC>;
  using GM = GroupMoments<QP, QC>;
  using T2 = Tile2<TY_>;
  constexpr int TX = T2::TX, TY = T2::TY, NM = T2::NM, NU = T2::NU;
  constexpr int kMarchBar = 1, kFull = 2, kEmpty = 4;  // + buffer
  extern __shared__ __align__(16) unsigned char smraw[];
  auto& sm = *reinterpret_cast<Smem2<QP, QC, TY_>*>(smraw);
  const int64_t N = p.N;
  constexpr bool kMany = CTAS > 1;  // CTAs with more than one tile
  for (int pop = threadIdx.x; pop < L::P; pop += NM + NU)
    sm.coef[pop] = advection_coef(p.cx[pop], p.cy[pop], sm.cex[pop]);
  __syncthreads();

  if (threadIdx.x < NM) {
    // ---- march
    const int tid = threadIdx.x;
    const double* __restrict__ const adv =
        (const double*)(STAGE == kStage3 ? p.F2 : STAGE == kStage4 ? p.F3 : p.A4);
    // the thread's half line: population tg of the group; 16 x 16: one warp
    // takes the x lines of a population, the next its y lines; 16 x 8: half a
    // warp each (either way 16 lanes access 8-byte elements of distinct banks)
    constexpr int PT = NM / kG;  // threads of a population
    const int tg = tid / PT;
    const bool xline = tid % PT < PT / 2;
    const int ln = xline ? tid % TY : tid % TX;
    const int s0 = (xline ? tid / TY % 2 : TY == 16 ? tid / 16 % 2 : 0) * T2::SEG;
    // the thread's staged cells (staged_pos skips the corners): ghosts by
    // index clamp or wrap
    constexpr int NST = TY * (TX + 2 * H) + 2 * H * TX;
    constexpr int J = (NST + NM - 1) / NM;
    int soff[J], goff[J];
    bool has[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      int r, c;
      staged_pos(tid + j * NM, 2, TX, TY, r, c);
      has[j] = tid + j * NM < NST;
      soff[j] = r * T2::SX + c;
    }
    auto set_tile = [&](int t) {
      const int x0 = t % ntx * TX, y0 = t / ntx * TY;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        int r, c;
        staged_pos(tid + j * NM, 2, TX, TY, r, c);
        goff[j] = wrap_or_clamp(y0 - H + r, p.ny, p.bc) * p.nx + wrap_or_clamp(x0 - H + c, p.nx, p.bc);
      }
    };
    auto prefetch = [&](int b, int g0) {
#pragma unroll
      for (int g = 0; g < kG; ++g)
        if (g0 + g < L::P) {
          const double* __restrict__ src = adv + (g0 + g) * N;
#pragma unroll
          for (int j = 0; j < J; ++j)
            if (has[j]) cp_async(&sm.tile[b][g][0][0] + soff[j], src + (unsigned)goff[j]);
        }
      cp_async_commit();
    };
    int tile = blockIdx.x, gi = 0, nth = 0;
    bool more = true;
    set_tile(tile);
    prefetch(0, GM::first(0));
    for (int it = 0; more; ++it) {
      const int b = it & 1, g0 = GM::first(gi);
      // the next tile's number; the last of the launch's ntiles requests leaves
      // the counter as it was
      if (kMany && gi == 0 && tid == 0) {
        const unsigned k = atomicAdd(p.ticket, 1u);
        if (k == (unsigned)ntiles - 1) *p.ticket = 0;
        sm.next[nth & 1] = (int)(gridDim.x + k);
      }
      cp_async_wait_all();
      bar_sync(kMarchBar, NM);  // the group's tile is in; the previous march is done
      int ngi = gi + 1;
      if (ngi == GM::NG) {
        ngi = 0;
        tile = kMany ? sm.next[nth++ & 1] : ntiles;
        more = tile < ntiles;
        if (more) set_tile(tile);
      }
      if (more) prefetch(b ^ 1, GM::first(ngi));
      if (it >= 2) bar_sync(kEmpty + b, NM + NU);  // the update is done with this buffer
      const int pop = g0 + tg;
      const double pv = pop < L::P ? (xline ? p.px[pop] : p.py[pop]) : 0.0;
      const int sgn = pv >= 0.0 ? 1 : -1;
      const int first = sgn > 0 ? s0 : s0 + T2::SEG - 1;
      const int step = xline ? 1 : T2::SX;
      const double* line = xline ? &sm.tile[b][tg][ln + H][H] : &sm.tile[b][tg][H][ln + H];
      const double* up = line + (first - sgn) * step;
      int64_t* out = xline ? &sm.hx[b][tg][ln][first] : &sm.hy[b][tg][ln][first];
      if (pop < L::P) {
        // (a warp's lines, of one population, march either way as a whole)
        int emax;
        const bool fixed = __all_sync(0xffffffffu, scale_of_line<T2::SEG>(up, sgn * step, emax));
        (xline ? sm.ex[b][tg][ln] : sm.ey[b][tg][ln])[s0 / T2::SEG] = fixed ? emax : 0;
        if (fixed) mp9_march_delta<T2::SEG>(ScaledCells{up, emax}, sgn * step, out, sgn);
        else mp9_march_delta_fp64(up, sgn * step, out, sgn, T2::SEG);
      }
      bar_arrive(kFull + b, NM + NU);
      gi = ngi;
    }
  } else {
    // ---- update
    const int tid = threadIdx.x - NM;
    const int lx = tid % TX, ly = tid / TX;
    const Geo geo{p.nx, p.ny, 0, p.kchi, p.invDK, p.dtdx, p.dtdy, -1};
    int next = ntiles, nth = 0, it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile = next, ++nth) {
      const int x = tile % ntx * TX + lx, y = tile / ntx * TY + ly;
      const bool valid = x < p.nx && y < p.ny;
      // (a thread without a cell reads the first one and stores nothing)
      const unsigned c = valid ? (unsigned)y * p.nx + x : 0u;
      GM mom = {};
      UpdateIn in[kG];
      auto load = [&](int g0, UpdateIn (&u)[kG]) {
#pragma unroll
        for (int g = 0; g < kG; ++g)
          if (g0 + g < L::P) u[g] = load_update<STAGE>(p, (g0 + g) * N, c);
      };
      for (int gi = 0; gi < GM::NG; ++gi, ++it) {
        const int b = it & 1, g0 = GM::first(gi);
        load(g0, in);
        // the next group's inputs on their way to L2, a thread per tile row,
        // population and array: the registers to load them ahead are not there
        // (512 x 512: 3.42 -> 3.36 ms a step; grids of few tiles sit in L2)
        if (CTAS == 2 && TY == 16 && gi + 1 < GM::NG && tid < (STAGE == kStage4 ? 3 : 2) * 16 * kG) {
          const int row = tid % 16, pop = GM::first(gi + 1) + tid / 16 % kG, arr = tid / (16 * kG);
          const int xr = tile % ntx * TX, yr = tile / ntx * TY + row;
          if (pop < L::P && yr < p.ny) {
            const double* a = (const double*)(arr == 1 ? p.D : arr == 2 || STAGE == kFinal ? p.Af
                                                          : STAGE == kStage3 ? p.F : p.A4);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a + pop * N + (unsigned)(yr * p.nx + xr)));
          }
        }
        bar_sync(kFull + b, NM + NU);  // the group's flux differences are in
        if (kMany && gi == 0) next = sm.next[nth & 1];
        double R[kG];
#pragma unroll
        for (int g = 0; g < kG; ++g) {
          const int pop = g0 + g;
          R[g] = 0.0;
          if (pop < L::P) {
            // X = dt p . grad F
            const int64_t dx = sm.hx[b][g][ly][lx], dy = sm.hy[b][g][lx][ly];
            const int ex = sm.ex[b][g][ly][lx / T2::SEG], ey = sm.ey[b][g][lx][ly / T2::SEG];
            const int e = max(ex, ey);
            double X = q_to_double(advection_int(sm.coef[pop], sar64(dx, e - ex), sar64(dy, e - ey)), e + sm.cex[pop]);
            if (!ex || !ey) X = advection_fp64(p.cx[pop], p.cy[pop], dx, ex, dy, ey);
            R[g] = store_update<STAGE>(p, pop * N, c, valid, in[g], X);
          }
        }
        // (the march waits for it two groups on, if it gets there)
        if (gi + 2 < GM::NG || next < ntiles) bar_arrive(kEmpty + b, NM + NU);
        mom.add(p, g0, R);
        mom.fold(p, gi);
      }
      if (valid) relax_cell64<2, QP, QC, STAGE, NU>(p, geo, c, mom.m, &sm.fac[0][tid]);
    }
  }
}

// ---- 1-D ------------------------------------------------------------------------
//
// 1-D problems march in binary64 (fdlb_mp9.cuh): batches, single problems and
// the checkpointed runs of the adjoint agree bit for bit, and the adjoint
// recomputes the limiter's choices with the march's own comparisons.

// Tile shapes: cells, threads, populations per group and interfaces per march
// task (a tile of TX cells has TX + 1 interfaces).
template <int VAR>
struct Tile1;
template <>
struct Tile1<0> {
  static constexpr int TX = 127, NT = 128, G = 8, SEG = 8;
};
template <>
struct Tile1<1> {
  static constexpr int TX = 63, NT = 128, G = 16, SEG = 8;
};
template <>
struct Tile1<2> {
  static constexpr int TX = 255, NT = 128, G = 8, SEG = 16;
};
// single problems of middle length, so that their tiles still spread over the SMs
template <>
struct Tile1<4> {
  static constexpr int TX = 31, NT = 64, G = 16, SEG = 8;
};

// Shared memory of one tile: the advected populations of a group on tile +
// halo, and the interface values.
template <int VAR>
struct Smem1 {
  using C = Tile1<VAR>;
  double tile[C::G][C::TX + 2 * H];
  double hx[C::G][C::TX + 1];
};

// One tile (first cell x0 of the problem of geo) of one fused stage.  Ends
// with every thread past its last use of the shared memory, so a persistent
// CTA may start its next tile at once.
template <int QP, int QC, int STAGE, int VAR>
__device__ __forceinline__ void stage_tile_1d(const DevParams& p, const Geo& geo, int x0, Smem1<VAR>& sm) {
  using C = Tile1<VAR>;
  constexpr int P = QP + QC;
  constexpr int TX = C::TX, NT = C::NT, G = C::G, SEG = C::SEG, NSEG = (TX + 1) / SEG;
  constexpr int CPT = (TX + NT - 1) / NT;
  static_assert(NSEG * SEG == TX + 1 && G * NSEG == NT, "one march task per thread");
  const int tid = threadIdx.x;
  const int64_t N = p.N;
  // the thread's cells (a slot without one reads the problem's first cell and
  // stores nothing)
  int lxs[CPT];
  unsigned cell[CPT];
  bool valid[CPT];
  Moments mom[CPT];
#pragma unroll
  for (int k = 0; k < CPT; ++k) {
    const int ci = tid + k * NT;
    lxs[k] = ci < TX ? ci : 0;
    valid[k] = ci < TX && x0 + ci < geo.nx;
    cell[k] = (unsigned)geo.base + (valid[k] ? x0 + ci : 0);
    mom[k] = {};
  }
  const double* __restrict__ const adv =
      (const double*)(STAGE == kStage3 ? p.F2 : STAGE == kStage4 ? p.F3 : p.A4);
  const int tg = tid / NSEG;  // the march task's population in a group
  // the thread's staged cells: ghosts by index clamp or wrap
  constexpr int NST = TX + 2 * H;
  constexpr int J = (NST + NT - 1) / NT;
  int goff[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int e = tid + j * NT;
    goff[j] = e < NST ? wrap_or_clamp(x0 - H + e, geo.nx, p.bc) : -1;
  }
  // the group's advected populations, copied asynchronously; the next group's
  // copies run during this group's update
  auto prefetch = [&](int g0) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (g0 + g >= P) break;
      const double* __restrict__ src = adv + ((g0 + g) * N + geo.base);
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (goff[j] >= 0) cp_async(&sm.tile[g][tid + j * NT], src + (unsigned)goff[j]);
    }
    cp_async_commit();
  };
  prefetch(0);
  for (int g0 = 0; g0 < P; g0 += G) {
    cp_async_wait_all();
    __syncthreads();  // the group's tile is in; the previous update is done
    // every interface value once, marching upwind -> downwind
    if (g0 + tg < P) {
      const int sgn = p.px[g0 + tg] >= 0.0 ? 1 : -1;
      const MarchTask t = march_task(tid, 1, TX, 1, SEG, NST, sgn);
      mp9_march_fp64<SEG>(&sm.tile[tg][t.bc_], sgn, &sm.hx[tg][t.ofirst], sgn);
    }
    // the own cells' inputs, in flight across the barrier
    UpdateIn in[CPT][G];
#pragma unroll
    for (int k = 0; k < CPT; ++k)
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (g0 + g < P) in[k][g] = load_update<STAGE>(p, (g0 + g) * N, cell[k]);
    __syncthreads();  // the march is done with the tile
    if (g0 + G < P) prefetch(g0 + G);
#pragma unroll
    for (int k = 0; k < CPT; ++k)
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int pop = g0 + g;
        if (pop >= P) break;
        // X = dt p dF/dx (single problems use the host's dt p/dx, the same
        // product)
        const double cx = geo.prob < 0 ? p.cx[pop] : geo.dtdx * p.px[pop];
        const double X = cx * (sm.hx[g][lxs[k] + 1] - sm.hx[g][lxs[k]]);
        const double R = store_update<STAGE>(p, pop * N, cell[k], valid[k], in[k][g], X);
        accumulate<1, QP, QC>(p, mom[k], pop, R);
      }
  }
  __syncthreads();  // every thread past its last use of hx
#pragma unroll
  for (int k = 0; k < CPT; ++k)
    if (valid[k]) relax_cell64<1, QP, QC, STAGE, 1>(p, geo, cell[k], mom[k], nullptr);
}

// One tile per CTA, the grid covering one problem (at most 128 registers: 4
// CTAs per SM keep the binary64 pipe about 75 % busy).
template <int QP, int QC, int STAGE, int VAR>
__global__ void __launch_bounds__(Tile1<VAR>::NT, 4) stage_kernel(const __grid_constant__ DevParams p) {
  __shared__ Smem1<VAR> sm;
  const Geo geo{p.nx, p.ny, 0, p.kchi, p.invDK, p.dtdx, p.dtdy, -1};
  stage_tile_1d<QP, QC, STAGE, VAR>(p, geo, blockIdx.x * Tile1<VAR>::TX, sm);
}

// One stage (or, STAGE = kPrep, D and F2 of a state that was set) of a short
// 1-D problem: 8 threads a population, one interface each, and the 7 cells
// between them.  A warp's binary64 instruction takes 64 cycles whether 1 or 32
// of its lanes work, so a short problem's time is the number of binary64
// instructions on one thread's path; here that is one interface, one
// population's update, QP + QC steps of the moment sums (the three sums of
// the cells in the lanes of every warp, so that they need no second barrier)
// and one node's equilibrium, about 100, against about 400 for a thread that
// owns a cell.  Every value is formed by the operations of stage_tile_1d in
// their order, so the results are the same bits.
// Measured a step: 400 cells of 16 populations 16.4 us against 51 (tiles of 15
// cells), of 8 populations 13.3 against 33.  Its work per cell is larger, so
// it gives way to the tiles where the chip is full: at 65 536
// population-cells, 43.9 us (16) and 34.8 us (8) against 46.5 and 35.7.
constexpr int kSmallCells = 7;
constexpr int kSmallPopCells = 65536;
template <int QP, int QC>
constexpr int small_threads() { return ((QP + QC) * 8 + 31) / 32 * 32; }
template <int QP, int QC, int STAGE>
__global__ void __launch_bounds__(small_threads<QP, QC>())
    small_stage_kernel(const __grid_constant__ DevParams p) {
  constexpr int P = QP + QC;
  __shared__ double Rs[P][8];
  const int tid = threadIdx.x, lc = tid % 8, lane = tid % 32;
  const int pop = tid / 8 < P ? tid / 8 : P - 1;
  const int x = blockIdx.x * kSmallCells + lc;  // cell, and the interface left of it
  const bool valid = tid / 8 < P && lc < kSmallCells && x < p.nx;
  const unsigned c = x < p.nx ? x : p.nx - 1;
  const int64_t o = pop * p.N;
  // the node's column of the equilibrium table: node k of Q, or its mirror
  const int Q = pop < QP ? QP : QC, k = pop < QP ? pop : pop - QP;
  const bool mirror = k >= (Q + 1) / 2;
  constexpr int QM = QP > QC ? QP : QC;
  double w[QM];
#pragma unroll
  for (int l = 0; l < QM; ++l)
    w[l] = l < Q ? (pop < QP ? p.wHp : p.wHc)[l * kMaxQ + (mirror ? Q - 1 - k : k)] : 0.0;
  double R;
  if constexpr (STAGE == kPrep) {
    R = ((const double*)p.F + o)[c];
  } else {
    // the interface's window in march order, from its upwind cell
    const int sgn = p.px[pop] >= 0.0 ? 1 : -1;
    const int up = sgn > 0 ? x - 1 : x;
    const double* __restrict__ const adv =
        (const double*)(STAGE == kStage3 ? p.F2 : STAGE == kStage4 ? p.F3 : p.A4) + o;
    double v[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) v[j] = adv[(unsigned)wrap_or_clamp(up + sgn * (j - 4), p.nx, p.bc)];
    const UpdateIn in = load_update<STAGE>(p, o, c);
    double f;
    mp9_march_fp64<1>(v + 4, 1, &f, 1);
    const double X = p.cx[pop] * (__shfl_down_sync(0xffffffffu, f, 1) - f);
    R = store_update<STAGE, false>(p, o, c, valid, in, X);
  }
  Rs[pop][lc] = R;
  __syncthreads();
  // moment sums in population order: lanes 0-7 n, 8-15 j, 16-31 e
  const int role = lane / 8;
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const double cf = q >= QP || role == 0 ? 1.0 : role == 1 ? p.px[q] : p.p2[q];
    const double s = fma(cf, Rs[q][lc], acc);
    if (q < QP || role >= 2) acc = s;
  }
  Moments m;
  m.n = __shfl_sync(0xffffffffu, acc, lc);
  m.jx = __shfl_sync(0xffffffffu, acc, 8 + lc);
  m.jy = 0.0;
  m.e = __shfl_sync(0xffffffffu, acc, 16 + lc);
  double n, u, uy, T;
  if (!moments_to_nut<1>(p.invDK, m, n, u, uy, T) && valid && pop == 0) atomicOr(p.status, 1u);
  // the node's equilibrium (axis_g's operations)
  double a[QM];
  a[0] = 1.0;
  a[1] = u;
  const double tm1 = T - 1.0;
#pragma unroll
  for (int l = 2; l < QM; ++l) a[l] = fma(u, a[l - 1], ((double)(l - 1) * tm1) * a[l - 2]);
  double ev = w[0], od = 0.0;
#pragma unroll
  for (int l = 1; l < QM; ++l) {
    if (l & 1) od = fma(w[l], a[l], od);
    else ev = fma(w[l], a[l], ev);
  }
  const double g = mirror ? ev - od : ev + od;
  const double f = pop < QP ? n : p.kchi * T * n;
  const StageCoef& sc = p.sc;
  if constexpr (STAGE == kStage3 || STAGE == kStage4) {
    const double D = fma(-g, f, R);
    const double Fi = fma(STAGE == kStage3 ? -sc.a33e3 : -sc.a44e4, D, R);
    if (valid) {
      ((double*)p.D + o)[c] = D;
      ((double*)(STAGE == kStage3 ? p.F3 : p.A4) + o)[c] = Fi;
    }
  } else {
    const double fe = __dmul_rn(g, f), D = __dsub_rn(R, fe);
    if (valid) {
      ((double*)p.D + o)[c] = D;
      ((double*)p.F2 + o)[c] = fma(sc.c2, D, fe);
    }
  }
}

// Batches of 1-D problems: a persistent grid walks the tile work list of all
// problems (each tile within one problem, ghosts clamped at its own ends).
template <int QP, int QC, int STAGE, int VAR>
__global__ void __launch_bounds__(Tile1<VAR>::NT, 4) batch_stage_kernel(const __grid_constant__ DevParams p) {
  __shared__ Smem1<VAR> sm;
  for (int w = blockIdx.x; w < p.nwork; w += gridDim.x) {
    const WorkItem it = p.work[w];
    const BatchProblem& bp = p.probs[it.prob];
    const Geo geo{bp.nx, 1, bp.base, bp.kchi, bp.invDK, bp.dtdx, 0.0, it.prob};
    stage_tile_1d<QP, QC, STAGE, VAR>(p, geo, it.x0, sm);
  }
}

// Store the binary64 equilibrium of cell c as the state: binary64 values
// (FDLB_FP64), or binary32 pairs hi + lo with hi the rounded value and lo
// the rounded remainder (FDLB_MIXED).
template <typename S, int DIM, int QP, int QC>
__device__ __forceinline__ void store_state(const DevParams& p,
                                            const EqCellS<DIM, QP, QC, double>& eq, int64_t c) {
  using L = Lat<DIM, QP, QC>;
  const int64_t m = sizeof(S) == 8 ? c : mixed_cell(p, c);
#pragma unroll
  for (int pop = 0; pop < L::P; ++pop) {
    const double v = feq_of<DIM, QP, QC, double>(eq, pop);
    if constexpr (sizeof(S) == 8) {
      ((double*)p.F)[pop * p.N + c] = v;
    } else {
      split_pair(v, p.sh[pop * p.NS + m], p.sl[pop * p.NS + m]);
    }
  }
}

// problem of cell c (problems sorted by base)
__device__ __forceinline__ int find_problem(const DevParams& p, int64_t c) {
  int lo = 0, hi = p.nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (p.probs[mid].base <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// D and F2 of a state that was set (fdlb_init_riemann, fdlb_set_state), one
// cell per thread, by the final stage's operations in their order.
template <int DIM, int QP, int QC>
__global__ void __launch_bounds__(128) prep_kernel(const __grid_constant__ DevParams p) {
  __shared__ double fac[DIM == 2 ? QP + QC : 1][128];
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  Geo geo{p.nx, p.ny, 0, p.kchi, p.invDK, p.dtdx, p.dtdy, -1};
  if (p.nprob > 0) {
    geo.prob = find_problem(p, c);
    geo.kchi = p.probs[geo.prob].kchi;
    geo.invDK = p.probs[geo.prob].invDK;
  }
  Moments m = {};
  if constexpr (DIM == 2) {
    // in the final stage's order, so that a run set from its own populations
    // goes on with the same bits
    using GM = GroupMoments<QP, QC>;
    GM g = {};
#pragma unroll 2
    for (int gi = 0; gi < GM::NG; ++gi) {
      const int g0 = GM::first(gi);
      double v[kG];
#pragma unroll
      for (int j = 0; j < kG; ++j) v[j] = g0 + j < GM::P ? ((const double*)p.F + (g0 + j) * p.N)[c] : 0.0;
      g.add(p, g0, v);
      g.fold(p, gi);
    }
    m = g.m;
  } else {
    for (int pop = 0; pop < Lat<DIM, QP, QC>::P; ++pop)
      accumulate<DIM, QP, QC>(p, m, pop, ((const double*)p.F + pop * p.N)[c]);
  }
  relax_cell64<DIM, QP, QC, kPrep, 128>(p, geo, (unsigned)c, m, &fac[0][threadIdx.x]);
}

template <int QP, int QC, typename S>
__global__ void batch_init_kernel(const __grid_constant__ DevParams p) {
  using L = Lat<1, QP, QC>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const BatchProblem& bp = p.probs[find_problem(p, c)];
  const int x = (int)(c - bp.base);
  const int q = ((double)x + 0.5 >= bp.split) ? 1 : 0;
  const double rho = bp.st[q][0], ux = bp.st[q][1], P = bp.st[q][2];
  EqCell<1, QP, QC> eq64;
  make_eq_nut<1, QP, QC>(p, bp.kchi, rho, ux, 0.0, P / rho, eq64);
  EqCellS<1, QP, QC, double> eq;
  to_storage(eq64, eq);
  store_state<S>(p, eq, c);
}

// Piecewise-constant Riemann data -> discrete equilibrium (Sec. V).
struct RiemannArgs {
  double st[4][4];
  int nq;
  double sx, sy;  // membranes in cell units (split_in_cells)
};

// index of the state that cell (x, y) takes
template <int DIM>
__device__ __forceinline__ int riemann_side(const RiemannArgs& a, int x, int y) {
  const bool right = (double)x + 0.5 >= a.sx;
  if (DIM == 1) return right ? 1 : 0;
  const bool upper = (double)y + 0.5 >= a.sy;
  return upper ? (right ? 0 : 1) : (right ? 3 : 2);
}

template <int DIM, int QP, int QC, typename S>
__global__ void init_riemann_kernel(const __grid_constant__ DevParams p,
                                    const __grid_constant__ RiemannArgs a) {
  using L = Lat<DIM, QP, QC>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const int x = (int)(c % p.nx), y = (int)(c / p.nx);
  const int q = riemann_side<DIM>(a, x, y);
  const double rho = a.st[q][0];
  const double ux = a.st[q][1];
  const double uy = DIM == 2 ? a.st[q][2] : 0.0;
  const double P = a.st[q][DIM == 2 ? 3 : 2];
  EqCell<DIM, QP, QC> eq64;
  make_eq_nut<DIM, QP, QC>(p, p.kchi, rho, ux, uy, P / rho, eq64);
  EqCellS<DIM, QP, QC, double> eq;  // binary64 products, rounded once on store
  to_storage(eq64, eq);
  store_state<S>(p, eq, c);
}

// The same on large grids: the data hold 2 or 4 states, so each CTA forms their
// populations once and its threads copy them (a state's populations took one
// thread 250 to 800 binary64 operations for every cell: 5.3 of the 11.6 ms of
// setting 2048 x 2048 x 128 mixed populations).
template <int DIM, int QP, int QC, typename S>
__global__ void __launch_bounds__(256) fill_riemann_kernel(const __grid_constant__ DevParams p,
                                                           const __grid_constant__ RiemannArgs a) {
  using L = Lat<DIM, QP, QC>;
  __shared__ double val[sizeof(S) == 8 ? 4 : 1][L::P];
  __shared__ float2 pair[sizeof(S) == 8 ? 1 : 4][L::P];
  if (threadIdx.x < a.nq) {
    const int q = threadIdx.x;
    const double rho = a.st[q][0], P = a.st[q][DIM == 2 ? 3 : 2];
    EqCell<DIM, QP, QC> eq64;
    make_eq_nut<DIM, QP, QC>(p, p.kchi, rho, a.st[q][1], DIM == 2 ? a.st[q][2] : 0.0, P / rho, eq64);
    EqCellS<DIM, QP, QC, double> eq;
    to_storage(eq64, eq);
#pragma unroll
    for (int pop = 0; pop < L::P; ++pop) {
      const double v = feq_of<DIM, QP, QC, double>(eq, pop);
      if constexpr (sizeof(S) == 8) val[q][pop] = v;
      else split_pair(v, pair[q][pop].x, pair[q][pop].y);
    }
  }
  __syncthreads();
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < p.N; c += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(c % p.nx), y = (int)(c / p.nx);
    const int q = riemann_side<DIM>(a, x, y);
    const int64_t m = sizeof(S) == 8 ? c : mixed_cell(p, c);
#pragma unroll 8
    for (int pop = 0; pop < L::P; ++pop) {
      if constexpr (sizeof(S) == 8) {
        ((double*)p.F)[pop * p.N + m] = val[q][pop];
      } else {
        p.sh[pop * p.NS + m] = pair[q][pop].x;
        p.sl[pop * p.NS + m] = pair[q][pop].y;
      }
    }
  }
}

// Moments of a binary32-pair state: the binary64 sums of the high parts
// (mhi, kept by the stage kernels) plus binary64 sums of the low parts.
template <int DIM, int QP, int QC>
__global__ void mixed_moments_kernel(const __grid_constant__ DevParams p, double* __restrict__ n,
                                     double* __restrict__ ux, double* __restrict__ uy,
                                     double* __restrict__ T) {
  using L = Lat<DIM, QP, QC>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const int64_t i = mixed_cell(p, c);
  Moments m = {p.mhi[i], p.mhi[p.NS + i], p.mhi[2 * p.NS + i], p.mhi[3 * p.NS + i]};
  if constexpr (DIM == 2 && QP == 8) {
    // row and column sums (GroupMoments): 1.6 binary64 operations a population
    using GM = GroupMoments<QP, QC>;
    GM g = {};
#pragma unroll 2
    for (int gi = 0; gi < GM::NG; ++gi) {
      const int g0 = GM::first(gi);
      double v[kG];
#pragma unroll
      for (int j = 0; j < kG; ++j) v[j] = widen(p.sl[(g0 + j) * p.NS + i]);
      g.add(p, g0, v);
      g.fold(p, gi);
    }
    m = Moments{m.n + g.m.n, m.jx + g.m.jx, m.jy + g.m.jy, m.e + g.m.e};
  } else {
#pragma unroll 4
    for (int pop = 0; pop < L::P; ++pop) accumulate<DIM, QP, QC>(p, m, pop, widen(p.sl[pop * p.NS + i]));
  }
  double nn, vx, vy, TT;
  const double invDK = p.nprob > 0 ? p.probs[find_problem(p, c)].invDK : p.invDK;
  moments_to_nut<DIM>(invDK, m, nn, vx, vy, TT);
  n[c] = nn;
  ux[c] = vx;
  if (DIM == 2 && uy) uy[c] = vy;
  T[c] = TT;
}

template <int DIM, int QP, int QC>
__global__ void moments_kernel(const __grid_constant__ DevParams p, double* __restrict__ n,
                               double* __restrict__ ux, double* __restrict__ uy,
                               double* __restrict__ T) {
  using L = Lat<DIM, QP, QC>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  Moments m = {};
  const double* F = (const double*)p.F;
  for (int pop = 0; pop < L::P; ++pop) accumulate<DIM, QP, QC>(p, m, pop, F[pop * p.N + c]);
  double nn, vx, vy, TT;
  const double invDK = p.nprob > 0 ? p.probs[find_problem(p, c)].invDK : p.invDK;
  moments_to_nut<DIM>(invDK, m, nn, vx, vy, TT);
  n[c] = nn;
  ux[c] = vx;
  if (DIM == 2 && uy) uy[c] = vy;
  T[c] = TT;
}

// Transpose of the moment map (n, u, T)(F) of Eq. (Moments_discrete) at the
// current binary64 state: with n = sum phi, u = j/n, j = sum phi p and
// T = (e - n u^2)/((D+K) n), e = sum phi p^2 + sum chi,
//   dn/dphi_k = 1,  du_a/dphi_k = (p_a,k - u_a)/n,
//   dT/dphi_k = (|p_k - u|^2 - (D+K) T)/((D+K) n),  dT/dchi_q = 1/((D+K) n),
// so Fbar = J^T (nbar, ubar, Tbar) (absent adjoints are zero).  The state is
// read only when ubar or Tbar is given: n is linear in F.
template <int DIM, int QP, int QC>
__global__ void moments_adjoint_kernel(const __grid_constant__ DevParams p,
                                       const double* __restrict__ nbar,
                                       const double* __restrict__ uxbar,
                                       const double* __restrict__ uybar,
                                       const double* __restrict__ Tbar, double* __restrict__ Fbar) {
  using L = Lat<DIM, QP, QC>;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= p.N) return;
  const double nb = nbar ? nbar[c] : 0.0;
  const double uxb = uxbar ? uxbar[c] : 0.0;
  const double uyb = (DIM == 2 && uybar) ? uybar[c] : 0.0;
  const double Tb = Tbar ? Tbar[c] : 0.0;
  double nn = 1.0, vx = 0.0, vy = 0.0, TT = 0.0;
  if (uxbar || (DIM == 2 && uybar) || Tbar) {
    Moments m = {};
    const double* F = (const double*)p.F;
    for (int pop = 0; pop < L::P; ++pop) accumulate<DIM, QP, QC>(p, m, pop, F[pop * p.N + c]);
    moments_to_nut<DIM>(p.invDK, m, nn, vx, vy, TT);
  }
  const double inv_n = 1.0 / nn;
  const double tq = Tb * p.invDK * inv_n;  // Tbar / ((D+K) n)
  for (int pop = 0; pop < L::P; ++pop) {
    double v;
    if (pop < L::NPHI) {
      const double dx = p.px[pop] - vx, dy = DIM == 2 ? p.py[pop] - vy : 0.0;
      v = nb + (uxb * dx + uyb * dy) * inv_n + tq * (dx * dx + dy * dy - p.DK * TT);
    } else {
      v = tq;
    }
    Fbar[pop * p.N + c] = v;
  }
}

template <int DIM, int QP, int QC>
int launch_prep(const DevParams& p, cudaStream_t s) {
  prep_kernel<DIM, QP, QC><<<(unsigned)((p.N + 127) / 128), 128, 0, s>>>(p);
  return (int)cudaGetLastError();
}

template <int QP, int QC, int STAGE, int CTAS, int TY>
int launch_stage_2d_c(const DevParams& p, int ntx, int nsm, cudaStream_t s) {
  using T2 = Tile2<TY>;
  constexpr int bytes = (int)sizeof(Smem2<QP, QC, TY>);
  const cudaError_t e = cudaFuncSetAttribute(stage_kernel_2d<QP, QC, STAGE, CTAS, TY>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return (int)e;
  const int ntiles = ntx * ((p.ny + TY - 1) / TY);
  const int grid = ntiles < CTAS * nsm ? ntiles : CTAS * nsm;
  stage_kernel_2d<QP, QC, STAGE, CTAS, TY><<<grid, T2::NM + T2::NU, bytes, s>>>(p, ntx, ntiles);
  return (int)cudaGetLastError();
}

// Grids of no more tiles than SMs run one CTA per SM, whose threads then have
// 128 registers, on tiles of 16 x 8 cells while these too have an SM each (a
// stage's time is then one tile's); larger grids run two CTAs of 64 registers
// (some spills, twice the warps).  A stage of 96 x 70 cells, 30 tiles, smooth
// field | quadrants: 0.187 | 0.356 ms on two CTAs per SM, 0.153 | 0.348 on one,
// 0.110 | 0.254 on 16 x 8 tiles; of 512 x 512, 1024 tiles: 1.10 | 1.30 on one,
// 1.12 | 1.29 on two.
template <int QP, int QC, int STAGE>
int launch_stage_2d(const DevParams& p, cudaStream_t s) {
  const int ntx = (p.nx + 15) / 16;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return (int)e;
  if (ntx * ((p.ny + 7) / 8) <= nsm) return launch_stage_2d_c<QP, QC, STAGE, 1, 8>(p, ntx, nsm, s);
  if (ntx * ((p.ny + 15) / 16) <= nsm) return launch_stage_2d_c<QP, QC, STAGE, 1, 16>(p, ntx, nsm, s);
  return launch_stage_2d_c<QP, QC, STAGE, 2, 16>(p, ntx, nsm, s);
}

template <int QP, int QC, int VAR>
int launch_stage_1d(const DevParams& p, int stage, cudaStream_t s) {
  using C = Tile1<VAR>;
  const int grid = (p.nx + C::TX - 1) / C::TX;
  switch (stage) {
    case kStage3: stage_kernel<QP, QC, kStage3, VAR><<<grid, C::NT, 0, s>>>(p); break;
    case kStage4: stage_kernel<QP, QC, kStage4, VAR><<<grid, C::NT, 0, s>>>(p); break;
    default: stage_kernel<QP, QC, kFinal, VAR><<<grid, C::NT, 0, s>>>(p); break;
  }
  return (int)cudaGetLastError();
}

template <int QP, int QC>
int launch_small_1d(const DevParams& p, int stage, cudaStream_t s) {
  const int grid = (p.nx + kSmallCells - 1) / kSmallCells, nt = small_threads<QP, QC>();
  switch (stage) {
    case kPrep: small_stage_kernel<QP, QC, kPrep><<<grid, nt, 0, s>>>(p); break;
    case kStage3: small_stage_kernel<QP, QC, kStage3><<<grid, nt, 0, s>>>(p); break;
    case kStage4: small_stage_kernel<QP, QC, kStage4><<<grid, nt, 0, s>>>(p); break;
    default: small_stage_kernel<QP, QC, kFinal><<<grid, nt, 0, s>>>(p); break;
  }
  return (int)cudaGetLastError();
}

template <int DIM, int QP, int QC>
int launch_stage_fp64(const DevParams& p, int stage, cudaStream_t s) {
  if constexpr (DIM == 1) {
    if (p.nx <= kSmallPopCells / (QP + QC)) return launch_small_1d<QP, QC>(p, stage, s);
    if (stage == kPrep) return launch_prep<1, QP, QC>(p, s);
    // longer problems: the largest tile that still gives about one per SM
    if (p.nx >= 127 * 152) return launch_stage_1d<QP, QC, 0>(p, stage, s);
    if (p.nx >= 63 * 152) return launch_stage_1d<QP, QC, 1>(p, stage, s);
    return launch_stage_1d<QP, QC, 4>(p, stage, s);
  } else {
    if (stage == kPrep) return launch_prep<DIM, QP, QC>(p, s);
    return stage == kStage3   ? launch_stage_2d<QP, QC, kStage3>(p, s)
           : stage == kStage4 ? launch_stage_2d<QP, QC, kStage4>(p, s)
                              : launch_stage_2d<QP, QC, kFinal>(p, s);
  }
}

template <int DIM, int QP, int QC>
int launch_stage_t(const DevParams& p, int stage, cudaStream_t s) {
  // binary32 contexts run the kernels of fdlb_mixed.cu
  return p.precision == 1 ? launch_mixed_stage(p, stage, s)
                          : launch_stage_fp64<DIM, QP, QC>(p, stage, s);
}

template <int DIM, int QP, int QC>
int launch_init_t(const DevParams& p, const RiemannArgs& a, cudaStream_t s) {
  const int nt = 128;
  const int64_t nb = (p.N + nt - 1) / nt;
  // from 2^16 cells on a CTA's own table (8 us) costs less than a cell's factors
  if (p.N >= (1 << 16)) {
    if (p.precision == 1) fill_riemann_kernel<DIM, QP, QC, float><<<608, 256, 0, s>>>(p, a);
    else fill_riemann_kernel<DIM, QP, QC, double><<<608, 256, 0, s>>>(p, a);
  } else if (p.precision == 1) init_riemann_kernel<DIM, QP, QC, float><<<(unsigned)nb, nt, 0, s>>>(p, a);
  else init_riemann_kernel<DIM, QP, QC, double><<<(unsigned)nb, nt, 0, s>>>(p, a);
  return (int)cudaGetLastError();
}

template <int DIM, int QP, int QC>
int launch_moments_t(const DevParams& p, double* n, double* ux, double* uy, double* T,
                     cudaStream_t s) {
  const int nt = 128;
  const int64_t nb = (p.N + nt - 1) / nt;
  if (p.precision == 1) mixed_moments_kernel<DIM, QP, QC><<<(unsigned)nb, nt, 0, s>>>(p, n, ux, uy, T);
  else moments_kernel<DIM, QP, QC><<<(unsigned)nb, nt, 0, s>>>(p, n, ux, uy, T);
  return (int)cudaGetLastError();
}

template <int QP, int QC, int VAR>
int launch_batch_stage_v(const DevParams& p, int stage, cudaStream_t s) {
  using C = Tile1<VAR>;
  const int grid = p.bgrid < p.nwork ? p.bgrid : p.nwork;
  switch (stage) {
    case kPrep: return launch_prep<1, QP, QC>(p, s);
    case kStage3: batch_stage_kernel<QP, QC, kStage3, VAR><<<grid, C::NT, 0, s>>>(p); break;
    case kStage4: batch_stage_kernel<QP, QC, kStage4, VAR><<<grid, C::NT, 0, s>>>(p); break;
    default: batch_stage_kernel<QP, QC, kFinal, VAR><<<grid, C::NT, 0, s>>>(p); break;
  }
  return (int)cudaGetLastError();
}

template <int QP, int QC>
int launch_batch_stage_fp64(const DevParams& p, int stage, cudaStream_t s) {
  switch (p.variant) {
    case 1: return launch_batch_stage_v<QP, QC, 1>(p, stage, s);
    case 2: return launch_batch_stage_v<QP, QC, 2>(p, stage, s);
    default: return launch_batch_stage_v<QP, QC, 0>(p, stage, s);
  }
}

template <int QP, int QC>
int launch_batch_stage_t(const DevParams& p, int stage, cudaStream_t s) {
  return p.precision == 1 ? launch_mixed_batch_stage(p, stage, s)
                          : launch_batch_stage_fp64<QP, QC>(p, stage, s);
}

template <int QP, int QC>
int launch_batch_init_t(const DevParams& p, cudaStream_t s) {
  const int nt = 128;
  const int64_t nb = (p.N + nt - 1) / nt;
  if (p.precision == 1) batch_init_kernel<QP, QC, float><<<(unsigned)nb, nt, 0, s>>>(p);
  else batch_init_kernel<QP, QC, double><<<(unsigned)nb, nt, 0, s>>>(p);
  return (int)cudaGetLastError();
}

}  // namespace

bool supported_lattice(int d, int Qp, int Qc) {
#define X(D_, P_, C_) \
  if (d == D_ && Qp == P_ && Qc == C_) return true;
  FDLB_LATTICES(X)
#undef X
  return false;
}

int launch_stage(const DevParams& p, int stage, cudaStream_t s) {
  if (stage == kStateOut || stage == kStateIn) return launch_mixed_exchange(p, stage == kStateOut, s);
#define X(D_, P_, C_) \
  if (p.d == D_ && p.Qp == P_ && p.Qc == C_) return launch_stage_t<D_, P_, C_>(p, stage, s);
  FDLB_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

int launch_init_riemann(const DevParams& p, const double* states, int nq, double sx, double sy,
                        cudaStream_t s) {
  RiemannArgs a{};
  const int w = p.d + 2;
  for (int q = 0; q < nq && q < 4; ++q)
    for (int j = 0; j < w; ++j) a.st[q][j] = states[q * w + j];
  a.nq = nq;
  a.sx = sx;
  a.sy = sy;
#define X(D_, P_, C_) \
  if (p.d == D_ && p.Qp == P_ && p.Qc == C_) return launch_init_t<D_, P_, C_>(p, a, s);
  FDLB_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

int launch_moments(const DevParams& p, double* n, double* ux, double* uy, double* T,
                   cudaStream_t s) {
#define X(D_, P_, C_) \
  if (p.d == D_ && p.Qp == P_ && p.Qc == C_) return launch_moments_t<D_, P_, C_>(p, n, ux, uy, T, s);
  FDLB_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

int launch_moments_adjoint(const DevParams& p, const double* nbar, const double* uxbar,
                           const double* uybar, const double* Tbar, double* Fbar, cudaStream_t s) {
  const int nt = 128;
  const unsigned nb = (unsigned)((p.N + nt - 1) / nt);
#define X(D_, P_, C_)                                                                       \
  if (p.d == D_ && p.Qp == P_ && p.Qc == C_) {                                              \
    moments_adjoint_kernel<D_, P_, C_><<<nb, nt, 0, s>>>(p, nbar, uxbar, uybar, Tbar, Fbar); \
    return (int)cudaGetLastError();                                                         \
  }
  FDLB_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

int batch_tile_cells(int variant) {
  switch (variant) {
    case 1: return TileCfg<1, 1>::TX;
    case 2: return TileCfg<1, 2>::TX;
    default: return TileCfg<1, 0>::TX;
  }
}

int launch_batch_stage(const DevParams& p, int stage, cudaStream_t s) {
#define X(P_, C_) \
  if (p.Qp == P_ && p.Qc == C_) return launch_batch_stage_t<P_, C_>(p, stage, s);
  FDLB_BATCH_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

int launch_batch_init(const DevParams& p, cudaStream_t s) {
#define X(P_, C_) \
  if (p.Qp == P_ && p.Qc == C_) return launch_batch_init_t<P_, C_>(p, s);
  FDLB_BATCH_LATTICES(X)
#undef X
  return (int)cudaErrorInvalidValue;
}

}  // namespace fdlb
