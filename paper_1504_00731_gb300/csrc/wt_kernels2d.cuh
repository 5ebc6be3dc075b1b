// Kernel templates of the 2D Euler hot path (dimension by dimension, Sec. 4.3), instantiated
// once per arithmetic policy:
//   pack2d / unpack2d   caller's [4][ny][nx] state <-> padded planes with ghost rows/columns
//   alpha2d             alpha_s per direction and the 2D CFL quantity (warp-shuffle maxima)
//   stage2d             fused RHS + RK stage: a TX x TY tile plus its 3-cell halo staged row by
//                       row with bulk copies, the x sweep then the y sweep in shared memory,
//                       one output write per cell; at most 112 KB of shared memory per 256
//                       threads, so that 16 warps share an SM
#pragma once

#include <type_traits>

#include "wt_central.cuh"
#include "wt_device.cuh"
#include "wt_launch.h"

namespace wt {

template <int TX, int TY>
struct Tile2D {
  static_assert(TX % 2 == 0, "tile width must be even so that staged rows start 16-byte aligned");
  static constexpr int WX = TX + 2 * G;          // staged row length (even)
  static constexpr int RY = TY + 2 * G;          // staged rows
  static constexpr int NCELL = WX * RY;
  static constexpr int NIX = (TX + 1) * TY;      // x-interfaces of the tile
  static constexpr int NIY = TX * (TY + 1);      // y-interfaces
  static constexpr int NI = NIX > NIY ? NIX : NIY;
  static constexpr int NT = 256;
  static_assert(TX * TY <= NT, "one cell per thread in the flux difference and the stage update");
  // Buffers are reused across the sweeps: the physical flux buffer holds f for the x sweep,
  // then g for the y sweep; the reconstruction buffer holds F, then h of the same sweep; the
  // x sweep's flux difference stays in registers until the update; the eigenvector buffer
  // takes the block reductions at the end.
  static constexpr int kBar = 0;
  static constexpr int kUin = 2;                       // [4][RY][WX]
  static constexpr int kU = kUin + 4 * NCELL;          // velocity u per staged cell
  static constexpr int kV = kU + NCELL;
  static constexpr int kH = kV + NCELL;
  static constexpr int kSr = kH + NCELL;
  static constexpr int kFg = kSr + NCELL;              // [4][NCELL] f, then g
  static constexpr int kL = kFg + 4 * NCELL;           // [16][NI]; 8 * 32 + 32 for the reductions
  static constexpr int kRs = kL + 16 * NI;             // [4][NI]
  static constexpr int kF = kRs + 4 * NI;              // [4][NI] F, then h
  static constexpr int kTotal = kF + 4 * NI;
  static_assert(16 * NI >= 9 * 32, "reduction scratch inside the eigenvector buffer");
  static constexpr size_t bytes = sizeof(double) * kTotal;
  static constexpr int kCtas = 2;
  // two CTAs per SM: 228 KB of shared memory per SM, 1 KB of it reserved per CTA
  static_assert(2 * (bytes + 1024) <= 228 * 1024, "two tiles must fit on one SM");
};

// What the fast policy's kernel costs: 230 FP64 thread instructions per cell and stage on 1024 x 1024
// vortices (1245 with every interface projected), 53 % of the FP64 pipe's cycles at 16 warps per SM; 2048 x 2048 vortices 59.8 -> 17.4 ms for two steps, 120 x 360 Rayleigh-Taylor 22.3 -> 11.5
// ms for 40 (a fifth of its y interfaces are on fronts and take the FP64 path).
//
// Tile of the central screen (wt_central.cuh; the fast policy): no eigenvector or reconstruction
// buffers per interface; the differences along the sweep as FP32 pairs, f's also in FP64 for
// the central fluxes, in one buffer for both sweeps.
template <int TX, int TY>
struct Tile2DC {
  static constexpr int WX = TX + 2 * G;
  static constexpr int RY = TY + 2 * G;
  static constexpr int NCELL = WX * RY;
  static constexpr int NIX = (TX + 1) * TY;
  static constexpr int NIY = TX * (TY + 1);
  static constexpr int NI = NIX > NIY ? NIX : NIY;
  static constexpr int NT = TX * 8;
  static_assert(NIX <= NT && NIY <= NT, "one interface per thread");
  static constexpr int kCtas = 512 / NT;  // per SM
  static_assert(TX * TY <= NT, "one cell per thread in the flux difference and the stage update");
  static constexpr int NDX = (TX + 5) * TY, NDY = TX * (TY + 5);  // differences of a sweep
  static constexpr int ND = NDX > NDY ? NDX : NDY;
  static constexpr int FC = 64;  // listed interfaces taken at a time
  static constexpr int kBar = 0;
  static constexpr int kUin = 2;
  static constexpr int kU = kUin + 4 * NCELL;
  static constexpr int kV = kU + NCELL;
  static constexpr int kH = kV + NCELL;
  static constexpr int kFg = kH + NCELL;               // [4][NCELL] f, then g
  static constexpr int kDf = kFg + 4 * NCELL;          // [4][ND] differences of the sweep's flux
  static constexpr int kPair = kDf + 4 * ND;           // [8][ND] differences of flux and state, FP32 pairs
  static constexpr int kL = kPair;                     // FP64 path: [16][FC], then [4][FC], [4][FC]
  static constexpr int kRs = kL + 16 * FC;
  static constexpr int kF = kRs + 4 * FC;
  static_assert(24 * FC <= 8 * ND, "the FP64 path's buffers over the pairs");
  static constexpr int kHf = kPair + 8 * ND;           // [4][NI]
  static constexpr int kRed = kHf + 4 * NI;            // maxima of the speeds
  static constexpr int kList = kRed + 32 + 9 * (NT / 32) + (NT / 32) % 2;              // ints [NI]: listed interfaces (or cells, for the speeds)
  static constexpr int kItems = kList + (NI + 1) / 2;  // ints [4 * FC]: (field, slot) pairs of the FP64 path
  static constexpr int kCnt = kItems + 2 * FC;         // ints: listed, items
  static constexpr int kTotal = kCnt + 1;
  static constexpr size_t bytes = sizeof(double) * kTotal;
  static_assert(kCtas * (bytes + 1024) <= 228 * 1024, "512 threads' tiles must fit on one SM");
};
// Rows per tile: with 7 every interface of a sweep has its own thread (231 and 256 of 256, 119 and 128 of
// 128); with 8 a second pass over 8 and 32 of them costs as long as the first.
template <class MATH>
constexpr int kTileY = MATH::kCentral ? 7 : 8;
template <class MATH, int TX, int TY>
using KernelTile2D = std::conditional_t<MATH::kCentral, Tile2DC<TX, TY>, Tile2D<TX, TY>>;

// One sweep's interface fluxes by the central screen (as central_fluxes in 1D): DIR 0 the x sweep
// (interface i of row r at r (tcx + 1) + i), 1 the y sweep (interface j of column t at j tcx + t).
template <class MATH, int DIR, class TL, int TX>
__device__ __forceinline__ void central_sweep(const Stage2DArgs& a, const int tcx, const int tcy,
                                              const double (&alpha)[4], double* sm) {
  constexpr int WX = TL::WX, NCELL = TL::NCELL, NI = TL::NI, NT = TL::NT, ND = TL::ND, FC = TL::FC;
  constexpr int ST = DIR == 0 ? 1 : WX;   // cell stride along the sweep
  constexpr int SD = DIR == 0 ? 1 : TX;   // stride of the differences along the sweep
  constexpr int PD = DIR == 0 ? TX + 5 : TX;  // their row pitch
  constexpr int N1 = 1 + DIR, T1 = 2 - DIR;   // components: normal and tangential momentum
  const int tid = threadIdx.x;
  double* s_uin = sm + TL::kUin;
  double* s_n = sm + (DIR == 0 ? TL::kU : TL::kV);
  double* s_t = sm + (DIR == 0 ? TL::kV : TL::kU);
  double* s_H = sm + TL::kH;
  double* s_fg = sm + TL::kFg;
  double* s_df = sm + TL::kDf;
  float2* s_pair = reinterpret_cast<float2*>(sm + TL::kPair);
  double* s_h = sm + TL::kHf;
  int* s_list = reinterpret_cast<int*>(sm + TL::kList);
  int* s_nl = reinterpret_cast<int*>(sm + TL::kCnt);  // listed interfaces, items of the FP64 path
  int* s_item = reinterpret_cast<int*>(sm + TL::kItems);
  // components in the sweep's order (density, normal momentum, tangential momentum, energy)
  auto comp = [](int c) { return c == 1 ? N1 : (c == 2 ? T1 : c); };
  const int nper = DIR == 0 ? tcx + 1 : tcx;  // interfaces per row of the tile
  const int ni = DIR == 0 ? (tcx + 1) * tcy : tcx * (tcy + 1);
  // ---- D1
  const int drow = DIR == 0 ? tcx + 5 : tcx, dn = DIR == 0 ? drow * tcy : drow * (tcy + 5);
  for (int q = tid; q < dn; q += NT) {
    const int r = q / drow, col = q - r * drow;
    const int k = DIR == 0 ? (r + G) * WX + col : r * WX + col + G;
    const int p = r * PD + col;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double* x = s_fg + comp(c) * NCELL + k;
      const double df = __dsub_rn(x[ST], x[0]);
      s_df[c * ND + p] = df;
      s_pair[c * ND + p] = c == 2 ? f32_pair_nz(df) : f32_pair(df);
      const double* y = s_uin + comp(c) * NCELL + k;
      const double dy = __dsub_rn(y[ST], y[0]);
      s_pair[(4 + c) * ND + p] = c == 2 ? f32_pair_nz(dy) : f32_pair(dy);
    }
  }
  if (tid == 0) s_nl[0] = s_nl[1] = 0;
  __syncthreads();
  // ---- D2
  const float gm1 = f32_trunc(a.gamma - 1.0), eps = f32_trunc(a.eps), aR = f32_trunc(a.alpha_R);
  const bool screenable = screen_constants(eps, aR);
  for (int it = tid; it < ni; it += NT) {
    const int r = it / nper, i = it - r * nper;
    const int k0 = DIR == 0 ? (r + G) * WX + i : r * WX + i + G;  // first stencil cell
    const int p0 = r * PD + i;
    const int ka = k0 + 2 * ST, kb = ka + ST;
    const Roe32Shear o = roe32_2d(s_uin[ka], s_n[ka], s_t[ka], s_H[ka], s_uin[kb], s_n[kb], s_t[kb], s_H[kb], gm1);
    Proj32Shear pf, pu;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      float d[4][5];
      float4 h[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float2 q[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          q[k] = s_pair[(4 * x + c) * ND + p0 + k * SD];
          d[c][k] = q[k].x;
        }
        h[c] = high_differences(q);
      }
      project_stencil_2d(o, d, h, x ? pu : pf);
    }
    int verdicts = 0;  // three bits per field
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      float fa[9], fb[9], ea[5], eb[5];
      take_field_2d(s, o, pf, fa, ea);
      take_field_2d(s, o, pu, fb, eb);
      const float kap = (s == 0 || s == 3) ? 4.0f : 2.0f;
      const float thr = s == 2 ? fmul(o.r.thr, o.T) : o.r.thr;  // the shear field carries rho v
      const int v = prove_field(fa, fb, ea, eb, f32_trunc(alpha[s]), fmul(eps, kap * kap), aR, fmul(thr, kap));
      verdicts |= (o.r.ok && screenable ? v : 0) << (3 * s);
    }
    if (verdicts == kAllCentral2D) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double *f = s_fg + comp(c) * NCELL + k0, *d = s_df + c * ND + p0;
        s_h[comp(c) * NI + it] = central_value(f[2 * ST], f[3 * ST], d[0], d[SD], d[3 * SD], d[4 * SD]);
      }
    } else {
      s_list[atomicAdd(s_nl, 1)] = it | (verdicts << 16);
    }
  }
  __syncthreads();
  // ---- D3: the FP64 path of the listed interfaces
  const int nl = *s_nl;
  double* s_L = sm + TL::kL;
  double* s_rs = sm + TL::kRs;
  double* s_F = sm + TL::kF;
  for (int base = 0; base < nl; base += FC) {
    const int nc = min(nl - base, FC);
    for (int q = tid; q < nc; q += NT) {
      const int it = s_list[base + q] & 0xffff, verdicts = s_list[base + q] >> 16, r = it / nper, i = it - r * nper;
      const int k0 = DIR == 0 ? (r + G) * WX + i : r * WX + i + G, p0 = r * PD + i;
      const int ka = k0 + 2 * ST, kb = ka + ST;
      double L[16], rs[4];
      MATH::roe2d(DIR, MATH::sqrt_rho(s_uin[ka]), sm[TL::kU + ka], sm[TL::kV + ka], s_H[ka], MATH::sqrt_rho(s_uin[kb]),
                  sm[TL::kU + kb], sm[TL::kV + kb], s_H[kb], a.gamma, L, rs);
#pragma unroll
      for (int e = 0; e < 16; ++e) s_L[e * FC + q] = L[e];
#pragma unroll
      for (int e = 0; e < 4; ++e) s_rs[e * FC + q] = rs[e];
      int un = 0;
#pragma unroll
      for (int s = 0; s < 4; ++s) un |= ((verdicts >> (3 * s)) & 7) == 0 ? 1 << s : 0;
      if (un != 15) {  // the fields the screen has decided (decided_field)
        double C[4], A[4], B[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {  // in the sweep's order of components
          const double *f = s_fg + comp(c) * NCELL + k0, *v = s_uin + comp(c) * NCELL + k0, *x = s_df + c * ND + p0;
          C[c] = central_value(f[2 * ST], f[3 * ST], x[0], x[SD], x[3 * SD], x[4 * SD]);
          A[c] = fifth_difference(x[0], x[SD], x[2 * SD], x[3 * SD], x[4 * SD]);
          B[c] = fifth_difference_q(v[0], v[ST], v[2 * ST], v[3 * ST], v[4 * ST], v[5 * ST]);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if ((un >> s) & 1) continue;
          const double l[4] = {L[4 * s], L[4 * s + N1], L[4 * s + T1], L[4 * s + 3]};
          const double c = fma(l[3], C[3], fma(l[2], C[2], fma(l[1], C[1], l[0] * C[0])));
          const double p = fma(l[3], A[3], fma(l[2], A[2], fma(l[1], A[1], l[0] * A[0])));
          const double w = fma(l[3], B[3], fma(l[2], B[2], fma(l[1], B[1], l[0] * B[0])));
          s_F[s * FC + q] = decided_field((verdicts >> (3 * s)) & 7, c, p, w, alpha[s]);
        }
      }
      if (un != 0) {
        int at = atomicAdd(&s_nl[1], __popc(un));
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if ((un >> s) & 1) s_item[at++] = q | (s << 16);
      }
    }
    __syncthreads();
    const int nit = s_nl[1];
    for (int e = tid; e < nit; e += NT) {
      const int s = s_item[e] >> 16, q = s_item[e] & 0xffff;
      const int it = s_list[base + q] & 0xffff, r = it / nper, i = it - r * nper;
      const int k0 = DIR == 0 ? (r + G) * WX + i : r * WX + i + G;
      const double l[4] = {s_L[(4 * s) * FC + q], s_L[(4 * s + 1) * FC + q], s_L[(4 * s + 2) * FC + q],
                           s_L[(4 * s + 3) * FC + q]};
      const double al = s == 0 ? alpha[0] : (s == 1 ? alpha[1] : (s == 2 ? alpha[2] : alpha[3]));
      double vp[6], vm[6];
#pragma unroll
      for (int kk = 0; kk < 6; ++kk) {
        const int k = k0 + kk * ST;
        const double f[4] = {s_fg[k], s_fg[NCELL + k], s_fg[2 * NCELL + k], s_fg[3 * NCELL + k]};
        const double U[4] = {s_uin[k], s_uin[NCELL + k], s_uin[2 * NCELL + k], s_uin[3 * NCELL + k]};
        MATH::project4(DIR, l, f, U, al, vp[kk], vm[kk]);
      }
      double qm[6];
#pragma unroll
      for (int kk = 0; kk < 6; ++kk) qm[kk] = vm[5 - kk];
      s_F[s * FC + q] = MATH::weno(vp, a.eps, a.alpha_R) + MATH::weno(qm, a.eps, a.alpha_R);
    }
    __syncthreads();
    for (int q = tid; q < nc; q += NT) {
      const int it = s_list[base + q] & 0xffff;
      const double rs[4] = {s_rs[q], s_rs[FC + q], s_rs[2 * FC + q], s_rs[3 * FC + q]};
      const double F[4] = {s_F[q], s_F[FC + q], s_F[2 * FC + q], s_F[3 * FC + q]};
      double h[4];
      MATH::backproject2d(DIR, rs, F, h);
#pragma unroll
      for (int c = 0; c < 4; ++c) s_h[c * NI + it] = h[c];
    }
    if (tid == 0) s_nl[1] = 0;
    __syncthreads();
  }
}

__global__ void pack2d_kernel(const double* __restrict__ src, double* __restrict__ dst, long long nx, long long ny,
                              long long rowp, long long planep, int bxl, int bxh, int byl, int byh);
__global__ void unpack2d_kernel(const double* __restrict__ src, double* __restrict__ dst, long long nx, long long ny,
                                long long rowp, long long planep);

template <class MATH>
__global__ void __launch_bounds__(256) alpha2d_kernel(const double* __restrict__ u, long long nx, long long ny,
                                                      long long rowp, long long planep, double gamma, double dx,
                                                      double dy, Ctl* ctl, int slot) {
  __shared__ double red[9 * 32];
  unsigned long long v[8], q = 0ull;
#pragma unroll
  for (int s = 0; s < 8; ++s) v[s] = 0ull;
  const long long cells = nx * ny;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < cells;
       k += (long long)gridDim.x * blockDim.x) {
    const long long y = k / nx, x = k - y * nx;
    const long long idx = (y + G) * rowp + x + G;
    double U[4] = {u[idx], u[planep + idx], u[2 * planep + idx], u[3 * planep + idx]};
    double lx[4], ly[4], qq;
    MATH::euler2d_speeds(U, gamma, dx, dy, lx, ly, qq);
    if (!finite4(U)) flag_error(ctl, WT_ERR_NONPHYSICAL);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      key_max(v[s], lx[s]);
      key_max(v[4 + s], ly[s]);
    }
    key_max(q, qq);
  }
  block_max_atomic<8>(v, red, ctl->amax[slot]);
  unsigned long long qa[1] = {q};
  block_max_atomic<1>(qa, red + 8 * 32, &ctl->cfl2d[slot]);
}

template <class MATH, int STAGE, int TX, int TY>
__global__ void __launch_bounds__(KernelTile2D<MATH, TX, TY>::NT, KernelTile2D<MATH, TX, TY>::kCtas) stage2d_kernel(const Stage2DArgs a) {
  using TL = KernelTile2D<MATH, TX, TY>;
  constexpr bool CENTRAL = MATH::kCentral;
  constexpr int WX = TL::WX, RY = TL::RY, NCELL = TL::NCELL, NI = TL::NI, NT = TL::NT;
  extern __shared__ __align__(16) double sm[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + TL::kBar);
  double* s_uin = sm + TL::kUin;
  double* s_u = sm + TL::kU;
  double* s_v = sm + TL::kV;
  double* s_H = sm + TL::kH;
  double* s_fg = sm + TL::kFg;
  double *s_h, *s_red;
  if constexpr (CENTRAL) {
    s_h = sm + TL::kHf;
    s_red = sm + TL::kRed;
  } else {
    s_h = sm + TL::kF;
    s_red = sm + TL::kL;
  }

  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x;
  Ctl* ctl = a.ctl;
  const long long nx = a.nx, ny = a.ny;
  // (a grid dimension holds 65535 rows of tiles; the rest are on z)
  const long long x0 = (long long)blockIdx.x * TX, y0 = (blockIdx.y + (long long)blockIdx.z * gridDim.y) * TY;
  if (x0 >= nx || y0 >= ny) return;
  const int tcx = (int)((nx - x0 < TX) ? (nx - x0) : TX);
  const int tcy = (int)((ny - y0 < TY) ? (ny - y0) : TY);
  const bool first_tile = x0 == 0 && y0 == 0;

  double dt = 0.0;
  if (STAGE != STAGE_RHS) {
    if (STAGE == STAGE_RK1) {
      const bool act = (ctl->status == 0) && (ctl->t < ctl->t_final);
      if (!act) {
        if (first_tile && tid == 0) ctl->active = 0;
        return;
      }
    } else if (ctl->active == 0) {
      return;
    }
    if (first_tile && tid < 8) ctl->amax[(STAGE + 2) % 3][tid] = 0ull;
    if (first_tile && tid == 8) ctl->cfl2d[(STAGE + 2) % 3] = 0ull;
  }
  const int slot_in = (STAGE == STAGE_RHS) ? 0 : STAGE;
  double ax[4], ay[4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    ax[s] = bits_to_double(ctl->amax[slot_in][s]);
    ay[s] = bits_to_double(ctl->amax[slot_in][4 + s]);
  }
  if (STAGE == STAGE_RK1) {
    dt = ctl->dt_fixed > 0.0 ? ctl->dt_fixed : MATH::cfl_dt_2d(ctl->cfl, bits_to_double(ctl->cfl2d[0]));
    const double rem = ctl->t_final - ctl->t;
    if (rem < dt) dt = rem;
    if (first_tile && tid == 0) {
      ctl->dt = dt;
      ctl->active = 1;
    }
  } else if (STAGE != STAGE_RHS) {
    dt = ctl->dt;
  }

  // ---- A: stage rows y0-3 .. y0+tcy+2, columns x0-3 .. x0+tcx+2 of every plane (u^n of
  //      stages 2 and 3 is read in phase E, one load per cell)
  const int rows = tcy + 2 * G;
  const int len = (tcx + 2 * G + 1) & ~1;
  constexpr bool kNeedUn = (STAGE == STAGE_RK2 || STAGE == STAGE_RK3);
  if (tid == 0) mbar_init(bar, 1);
  __syncthreads();
  if (tid < 32) {
    const uint32_t bytes = (uint32_t)len * 8u;
    const int ncopy = 4 * rows;
    if (tid == 0) mbar_arrive_expect_tx(bar, bytes * (uint32_t)ncopy);
    __syncwarp();
    for (int k = tid; k < ncopy; k += 32) {
      const int c = k / rows, r = k - c * rows;
      bulk_g2s(s_uin + (c * RY + r) * WX, a.uin + c * a.planep + (y0 + r) * a.rowp + x0, bytes, bar);
    }
  }
  const bool ok = mbar_wait_bounded(bar, 0);
  if (__syncthreads_or(ok ? 0 : 1)) {
    if (tid == 0) flag_error(ctl, WT_ERR_TIMEOUT);
    mbar_wait_bounded(bar, 0);
    return;
  }

  // ---- B: per staged cell of the cross (interior rows with x-halo, interior columns with
  //      y-halo): velocities, H, sqrt(rho) and f; g follows once the x sweep is done with f
  for (int k = tid; k < NCELL; k += NT) {
    const int r = k / WX, col = k - r * WX;
    if (r >= rows || col >= tcx + 2 * G) continue;
    const bool xin = (col >= G && col < G + tcx), yin = (r >= G && r < G + tcy);
    if (!xin && !yin) continue;  // corner: not on any stencil
    double U[4] = {s_uin[k], s_uin[NCELL + k], s_uin[2 * NCELL + k], s_uin[3 * NCELL + k]};
    if (!finite4(U)) flag_error(ctl, WT_ERR_NONPHYSICAL);
    double f[4], u, v, H;
    if constexpr (CENTRAL) {
      MATH::euler2d_cell_flux(U, a.gamma, f, u, v, H);
    } else {
      double g[4], sr;
      MATH::euler2d_cell(U, a.gamma, f, g, u, v, H, sr);
      sm[TL::kSr + k] = sr;
    }
    s_u[k] = u;
    s_v[k] = v;
    s_H[k] = H;
    if (yin) {
#pragma unroll
      for (int c = 0; c < 4; ++c) s_fg[c * NCELL + k] = f[c];
    }
  }
  __syncthreads();

  if constexpr (CENTRAL) {
    central_sweep<MATH, 0, TL, TX>(a, tcx, tcy, ax, sm);
  } else {
    double *s_L = sm + TL::kL, *s_rs = sm + TL::kRs, *s_F = sm + TL::kF;
  // ---- x sweep.  Interface i of row r sits between cells (r+3, i+2) and (r+3, i+3).
  const int nix = (tcx + 1) * tcy;
  for (int it = tid; it < nix; it += NT) {
    const int r = it / (tcx + 1), i = it - r * (tcx + 1);
    const int ka = (r + G) * WX + i + 2, kb = ka + 1;
    double L[16], rs[4];
    MATH::roe2d(0, sm[TL::kSr + ka], s_u[ka], s_v[ka], s_H[ka], sm[TL::kSr + kb], s_u[kb], s_v[kb], s_H[kb], a.gamma, L, rs);
#pragma unroll
    for (int e = 0; e < 16; ++e) s_L[e * NI + it] = L[e];
#pragma unroll
    for (int e = 0; e < 4; ++e) s_rs[e * NI + it] = rs[e];
  }
  __syncthreads();
  for (int item = tid; item < 4 * nix; item += NT) {
    const int s = item / nix, it = item - s * nix;
    const int r = it / (tcx + 1), i = it - r * (tcx + 1);
    const double l[4] = {s_L[(4 * s) * NI + it], s_L[(4 * s + 1) * NI + it], s_L[(4 * s + 2) * NI + it],
                         s_L[(4 * s + 3) * NI + it]};
    const double al = s == 0 ? ax[0] : (s == 1 ? ax[1] : (s == 2 ? ax[2] : ax[3]));
    double vp[6], vm[6];
#pragma unroll
    for (int kk = 0; kk < 6; ++kk) {
      const int k = (r + G) * WX + i + kk;
      const double f[4] = {s_fg[k], s_fg[NCELL + k], s_fg[2 * NCELL + k], s_fg[3 * NCELL + k]};
      const double U[4] = {s_uin[k], s_uin[NCELL + k], s_uin[2 * NCELL + k], s_uin[3 * NCELL + k]};
      MATH::project4(0, l, f, U, al, vp[kk], vm[kk]);
    }
    double qm[6];
#pragma unroll
    for (int kk = 0; kk < 6; ++kk) qm[kk] = vm[5 - kk];
    s_F[s * NI + it] = MATH::weno(vp, a.eps, a.alpha_R) + MATH::weno(qm, a.eps, a.alpha_R);
  }
  __syncthreads();
  // back-projection in place (F -> h of the same interface), and g of the y-sweep cells into
  // the flux buffer, which the x sweep no longer reads
  for (int it = tid; it < nix; it += NT) {
    const double rs[4] = {s_rs[it], s_rs[NI + it], s_rs[2 * NI + it], s_rs[3 * NI + it]};
    const double F[4] = {s_F[it], s_F[NI + it], s_F[2 * NI + it], s_F[3 * NI + it]};
    double h[4];
    MATH::backproject2d(0, rs, F, h);
#pragma unroll
    for (int c = 0; c < 4; ++c) s_h[c * NI + it] = h[c];
  }
  }
  for (int q = tid; q < rows * tcx; q += NT) {
    const int r = q / tcx, k = r * WX + G + (q - r * tcx);
    const double U[4] = {s_uin[k], s_uin[NCELL + k], s_uin[2 * NCELL + k], s_uin[3 * NCELL + k]};
    double g[4];
    MATH::euler2d_gflux(U, s_u[k], s_v[k], a.gamma, g);
#pragma unroll
    for (int c = 0; c < 4; ++c) s_fg[c * NCELL + k] = g[c];
  }
  __syncthreads();
  // the x sweep's flux difference of this thread's cell (the cell of phase E), and the y
  // sweep's Roe averages
  double Lx[4] = {0.0, 0.0, 0.0, 0.0};
  if (tid < tcx * tcy) {
    const int r = tid / tcx, t = tid - r * tcx;
    const int it = r * (tcx + 1) + t;
#pragma unroll
    for (int c = 0; c < 4; ++c) Lx[c] = MATH::flux_diff(s_h[c * NI + it + 1], s_h[c * NI + it], a.dx, a.inv_dx);
  }

  if constexpr (CENTRAL) {
    central_sweep<MATH, 1, TL, TX>(a, tcx, tcy, ay, sm);
  } else {
    double *s_L = sm + TL::kL, *s_rs = sm + TL::kRs, *s_F = sm + TL::kF;
  // ---- y sweep.  Interface j of column t sits between cells (j+2, t+3) and (j+3, t+3).
  const int niy = tcx * (tcy + 1);
  for (int it = tid; it < niy; it += NT) {
    const int j = it / tcx, t = it - j * tcx;
    const int ka = (j + 2) * WX + t + G, kb = ka + WX;
    double L[16], rs[4];
    MATH::roe2d(1, sm[TL::kSr + ka], s_u[ka], s_v[ka], s_H[ka], sm[TL::kSr + kb], s_u[kb], s_v[kb], s_H[kb], a.gamma, L, rs);
#pragma unroll
    for (int e = 0; e < 16; ++e) s_L[e * NI + it] = L[e];
#pragma unroll
    for (int e = 0; e < 4; ++e) s_rs[e * NI + it] = rs[e];
  }
  __syncthreads();
  for (int item = tid; item < 4 * niy; item += NT) {
    const int s = item / niy, it = item - s * niy;
    const int j = it / tcx, t = it - j * tcx;
    const double l[4] = {s_L[(4 * s) * NI + it], s_L[(4 * s + 1) * NI + it], s_L[(4 * s + 2) * NI + it],
                         s_L[(4 * s + 3) * NI + it]};
    const double al = s == 0 ? ay[0] : (s == 1 ? ay[1] : (s == 2 ? ay[2] : ay[3]));
    double vp[6], vm[6];
#pragma unroll
    for (int kk = 0; kk < 6; ++kk) {
      const int k = (j + kk) * WX + t + G;
      const double f[4] = {s_fg[k], s_fg[NCELL + k], s_fg[2 * NCELL + k], s_fg[3 * NCELL + k]};
      const double U[4] = {s_uin[k], s_uin[NCELL + k], s_uin[2 * NCELL + k], s_uin[3 * NCELL + k]};
      MATH::project4(1, l, f, U, al, vp[kk], vm[kk]);
    }
    double qm[6];
#pragma unroll
    for (int kk = 0; kk < 6; ++kk) qm[kk] = vm[5 - kk];
    s_F[s * NI + it] = MATH::weno(vp, a.eps, a.alpha_R) + MATH::weno(qm, a.eps, a.alpha_R);
  }
  __syncthreads();
  for (int it = tid; it < niy; it += NT) {
    const double rs[4] = {s_rs[it], s_rs[NI + it], s_rs[2 * NI + it], s_rs[3 * NI + it]};
    const double F[4] = {s_F[it], s_F[NI + it], s_F[2 * NI + it], s_F[3 * NI + it]};
    double h[4];
    MATH::backproject2d(1, rs, F, h);
#pragma unroll
    for (int c = 0; c < 4; ++c) s_h[c * NI + it] = h[c];
  }
  __syncthreads();
  }

  // ---- E: L = Lx + Ly, RK combine, ghost images, wave speeds of the new state
  unsigned long long vmax[8], qmax = 0ull;
#pragma unroll
  for (int s = 0; s < 8; ++s) vmax[s] = 0ull;
  [[maybe_unused]] bool ok32 = false;
  [[maybe_unused]] float l32[7] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  [[maybe_unused]] const float g32 = f32_hi(a.gamma * (a.gamma - 1.0)), idx32 = f32_hi(a.inv_dx), idy32 = f32_hi(a.inv_dy);
  if (tid < tcx * tcy) {
    const int r = tid / tcx, t = tid - r * tcx;
    const long long x = x0 + t, y = y0 + r;
    const int kc = (r + G) * WX + t + G;
    double un4[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) un4[c] = kNeedUn ? a.un[c * a.planep + (y + G) * a.rowp + x + G] : 0.0;
    double uo[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double Ly = MATH::flux_diff(s_h[c * NI + (r + 1) * tcx + t], s_h[c * NI + r * tcx + t], a.dy, a.inv_dy);
      double L = MATH::add_sweeps(Lx[c], Ly);
      // gravity along -y (TEST 6, Sec. 4.3): -g rho on the y momentum, -g rho v on the energy
      if (c >= 2 && a.gravity != 0.0) L = MATH::add_source(L, a.gravity, s_uin[(c == 2 ? 0 : 2) * NCELL + kc]);
      if (STAGE == STAGE_RHS) {
        a.Lout[(c * ny + y) * nx + x] = L;
      } else {
        const double us = s_uin[c * NCELL + kc];
        const double un = kNeedUn ? un4[c] : us;
        uo[c] = MATH::template rk<(STAGE == STAGE_RHS ? 0 : STAGE)>(un, us, dt, L);
      }
    }
    if (STAGE != STAGE_RHS) {
      const long long row = (y + G) * a.rowp;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        double* o = a.uout + c * a.planep;
        const double val = uo[c];
        o[row + x + G] = val;
        // x ghosts of this row (reflective: x-momentum negated)
        const double vx = (c == 1) ? -val : val;
        if (x < G || x >= nx - G) {
          if (a.bcx_hi == WT_BC_PERIODIC && x < G) o[row + nx + x + G] = val;
          if (a.bcx_lo == WT_BC_PERIODIC && x >= nx - G) o[row + x - nx + G] = val;
          if (a.bcx_lo == WT_BC_OUTFLOW && x == 0) o[row] = o[row + 1] = o[row + 2] = val;
          if (a.bcx_hi == WT_BC_OUTFLOW && x == nx - 1) o[row + nx + 3] = o[row + nx + 4] = o[row + nx + 5] = val;
          if (a.bcx_lo == WT_BC_REFLECTIVE && x < G) o[row + 2 - x] = vx;
          if (a.bcx_hi == WT_BC_REFLECTIVE && x >= nx - G) o[row + 2 * nx + 2 - x] = vx;
        }
        // y ghosts of this column (reflective: y-momentum negated)
        const double vy = (c == 2) ? -val : val;
        const long long col = x + G;
        if (y < G || y >= ny - G) {
          if (a.bcy_hi == WT_BC_PERIODIC && y < G) o[(ny + y + G) * a.rowp + col] = val;
          if (a.bcy_lo == WT_BC_PERIODIC && y >= ny - G) o[(y - ny + G) * a.rowp + col] = val;
          if (a.bcy_lo == WT_BC_OUTFLOW && y == 0) o[col] = o[a.rowp + col] = o[2 * a.rowp + col] = val;
          if (a.bcy_hi == WT_BC_OUTFLOW && y == ny - 1)
            o[(ny + 3) * a.rowp + col] = o[(ny + 4) * a.rowp + col] = o[(ny + 5) * a.rowp + col] = val;
          if (a.bcy_lo == WT_BC_REFLECTIVE && y < G) o[(2 - y) * a.rowp + col] = vy;
          if (a.bcy_hi == WT_BC_REFLECTIVE && y >= ny - G) o[(2 * ny + 2 - y) * a.rowp + col] = vy;
        }
      }
      if (!finite4(uo))
        flag_error(ctl, WT_ERR_NONPHYSICAL);
      if constexpr (CENTRAL) {
        // the output back to the tile, for the FP64 speeds of the cells that can hold a maximum
#pragma unroll
        for (int c = 0; c < 4; ++c) s_uin[c * NCELL + kc] = uo[c];
        ok32 = euler2d_speeds_screen(uo, g32, idx32, idy32, l32);
      } else {
        double lx[4], ly[4], q;
        MATH::euler2d_speeds(uo, a.gamma, a.dx, a.dy, lx, ly, q);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          key_max(vmax[s], lx[s]);
          key_max(vmax[4 + s], ly[s]);
        }
        key_max(qmax, q);
      }
    }
  }
  if constexpr (CENTRAL && STAGE != STAGE_RHS) {
    // As in 1D (the stage tiles' kScreen): the FP64 speeds (two divisions, a square root) only of
    // the cells whose FP32 speeds come within twice their error of a tile maximum (2^-12 of the
    // larger acoustic speed, 2^-16 of |u| or |v|, 2^-12 of q), one cell per run of bitwise-equal
    // states, gathered from the tile into full warps: 45 FP64 instructions per cell are left
    // to a few cells.
    float* s_lm = reinterpret_cast<float*>(s_red);  // [7][8] warp maxima
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(s_red + 32);  // [warps][9]
    int* s_list = reinterpret_cast<int*>(sm + TL::kList);
    int* s_nl = reinterpret_cast<int*>(sm + TL::kCnt);
    const bool cell = tid < tcx * tcy;
#pragma unroll
    for (int f = 0; f < 7; ++f) {
      // (non-negative floats order like their bit patterns)
      const unsigned v = __reduce_max_sync(0xffffffffu, (cell && ok32) ? __float_as_uint(l32[f]) : 0u);
      if ((tid & 31) == 0) s_lm[f * 8 + (tid >> 5)] = __uint_as_float(v);
    }
    if (tid == 0) *s_nl = 0;
    __syncthreads();
    if (cell) {
      float tm[7];
#pragma unroll
      for (int f = 0; f < 7; ++f) {
        tm[f] = 0.0f;
#pragma unroll
        for (int w = 0; w < TL::NT / 32; ++w) tm[f] = fmaxf(tm[f], s_lm[f * 8 + w]);
      }
      const float sx = 0x1p-12f * fmaxf(tm[0], tm[2]), sy = 0x1p-12f * fmaxf(tm[3], tm[5]);
      bool take = !ok32 || l32[0] >= tm[0] - sx || l32[2] >= tm[2] - sx || l32[3] >= tm[3] - sy ||
                  l32[5] >= tm[5] - sy || l32[6] >= tm[6] * (1.0f - 0x1p-12f) ||
                  (l32[1] > 0.0f && l32[1] >= tm[1] * (1.0f - 0x1p-16f)) ||
                  (l32[4] > 0.0f && l32[4] >= tm[4] * (1.0f - 0x1p-16f));
      const int r = tid / tcx, t = tid - r * tcx, kc = (r + G) * WX + t + G;
      if (take && t > 0) {  // the same state as the left neighbour's: the same speeds
        bool dup = true;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          dup = dup && __double_as_longlong(s_uin[c * NCELL + kc]) == __double_as_longlong(s_uin[c * NCELL + kc - 1]);
        take = !dup;
      }
      if (take) s_list[atomicAdd(s_nl, 1)] = kc;
    }
    __syncthreads();
    const int nsp = *s_nl;
    {
      unsigned long long key[9] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
      if (tid < nsp) {  // (at most one cell per thread)
        const int kc = s_list[tid];
        const double U[4] = {s_uin[kc], s_uin[NCELL + kc], s_uin[2 * NCELL + kc], s_uin[3 * NCELL + kc]};
        double lx[4], ly[4], q;
        MATH::euler2d_speeds(U, a.gamma, a.dx, a.dy, lx, ly, q);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          key[s] = speed_key(lx[s]);
          key[4 + s] = speed_key(ly[s]);
        }
        key[8] = speed_key(q);
      }
      if ((tid & ~31) < nsp) {
#pragma unroll
        for (int f = 0; f < 9; ++f) {
          const unsigned long long m = warp_max_key_redux(key[f]);
          if ((tid & 31) == 0) s_key[9 * (tid >> 5) + f] = m;
        }
      }
    }
    __syncthreads();
    constexpr int nxt = (STAGE + 1) % 3;
    if (tid < 9) {
      unsigned long long m = 0ull;
      for (int w = 0; 32 * w < nsp; ++w) m = max(m, s_key[9 * w + tid]);
      atomicMax(tid < 8 ? &ctl->amax[nxt][tid] : &ctl->cfl2d[nxt], m);
    }
    if (STAGE == STAGE_RK3 && first_tile && tid == 0) {
      ctl->t = ctl->t + dt;
      ctl->steps = ctl->steps + 1;
    }
  } else if (STAGE != STAGE_RHS) {
    const int nxt = (STAGE + 1) % 3;
    block_max_atomic<8>(vmax, s_red, ctl->amax[nxt]);
    unsigned long long qa[1] = {qmax};
    block_max_atomic<1>(qa, s_red + 8 * 32, &ctl->cfl2d[nxt]);
    if (STAGE == STAGE_RK3 && first_tile && tid == 0) {
      ctl->t = ctl->t + dt;
      ctl->steps = ctl->steps + 1;
    }
  }
}

template <class MATH, int STAGE, int TX>
cudaError_t launch_stage2d_t(const Stage2DArgs& a, cudaStream_t st) {
  constexpr int TY = kTileY<MATH>;
  using TL = KernelTile2D<MATH, TX, TY>;
  auto kern = stage2d_kernel<MATH, STAGE, TX, TY>;  // prepare_stage2d_policy() raised its shared-memory limit
  const long long rows = (a.ny + TY - 1) / TY, ny = rows < 65535 ? rows : 65535;
  dim3 grid((unsigned)((a.nx + TX - 1) / TX), (unsigned)ny, (unsigned)((rows + ny - 1) / ny));
  return launch_pdl(kern, grid, dim3(TL::NT), TL::bytes, st, a);
}

template <class MATH, int TX>
cudaError_t prepare_stage2d_tile() {
  constexpr int TY = kTileY<MATH>;
  using TL = KernelTile2D<MATH, TX, TY>;
  cudaError_t e = cudaSuccess;
  // the tile's shared memory, and the largest carveout, so that kCtas CTAs fit on an SM
  const void* kerns[4] = {(const void*)stage2d_kernel<MATH, STAGE_RK1, TX, TY>,
                          (const void*)stage2d_kernel<MATH, STAGE_RK2, TX, TY>,
                          (const void*)stage2d_kernel<MATH, STAGE_RK3, TX, TY>,
                          (const void*)stage2d_kernel<MATH, STAGE_RHS, TX, TY>};
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
    e = cudaFuncSetAttribute(kerns[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TL::bytes);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kerns[i], cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  return e;
}

template <class MATH>
cudaError_t prepare_stage2d_policy() {
  cudaError_t e = prepare_stage2d_tile<MATH, 32>();
  if constexpr (MATH::kCentral) {
    if (e == cudaSuccess) e = prepare_stage2d_tile<MATH, 16>();
  }
  return e;
}

// Width of the tiles (central): 32 columns (two CTAs of 256 threads per SM) on large grids, whose halo is
// the smaller share; 16 (four of 128) where 32-column tiles make fewer than four waves of the
// GPU's 304 slots, since the tiles on a front cost several times the others and smaller ones
// spread them (120 x 360: 16.8 -> 13.6 ms for 40 steps; 2048 x 2048: 18.1 -> 19.3 ms for 2).
template <class MATH>
bool narrow_tiles(const Stage2DArgs& a) {
  return MATH::kCentral && ((a.nx + 31) / 32) * ((a.ny + kTileY<MATH> - 1) / kTileY<MATH>) < 4 * 304;
}

template <class MATH, int STAGE>
cudaError_t launch_stage2d_w(const Stage2DArgs& a, cudaStream_t st) {
  if constexpr (MATH::kCentral) {
    if (narrow_tiles<MATH>(a)) return launch_stage2d_t<MATH, STAGE, 16>(a, st);
  }
  return launch_stage2d_t<MATH, STAGE, 32>(a, st);
}

template <class MATH>
cudaError_t launch_stage2d_policy(int stage, const Stage2DArgs& a, cudaStream_t st) {
  switch (stage) {
    case STAGE_RK1: return launch_stage2d_w<MATH, STAGE_RK1>(a, st);
    case STAGE_RK2: return launch_stage2d_w<MATH, STAGE_RK2>(a, st);
    case STAGE_RK3: return launch_stage2d_w<MATH, STAGE_RK3>(a, st);
    case STAGE_RHS: return launch_stage2d_w<MATH, STAGE_RHS>(a, st);
  }
  return cudaErrorInvalidValue;
}

template <class MATH>
cudaError_t launch_alpha2d_policy(const double* u, long long nx, long long ny, long long rowp, long long planep,
                                  double gamma, double dx, double dy, Ctl* ctl, int slot, cudaStream_t st) {
  long long blocks = (nx * ny + 255) / 256;
  if (blocks > 1216) blocks = 1216;
  alpha2d_kernel<MATH><<<(unsigned)(blocks < 1 ? 1 : blocks), 256, 0, st>>>(u, nx, ny, rowp, planep, gamma, dx, dy,
                                                                          ctl, slot);
  return cudaGetLastError();
}

}  // namespace wt
