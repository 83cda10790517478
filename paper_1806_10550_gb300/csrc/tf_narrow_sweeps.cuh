// tf_narrow_sweeps.cuh -- line sweeps in blocks of 4, 8 or 16 lines.
//
// The twisted LU solves of tf_line_sweeps.cuh for films whose blocks of 32
// lines would leave SMs idle.  Such a block's tick is as long as its slowest
// role, and the recurrence is the longest: so every other role has warps of
// its own, and the warps are placed by the SM sub-partition (warp index mod
// 4) that they run on.
//   warp 0            the recurrences of both halves of every line (lane =
//                     half * NL + line)
//   loaders           every cp.async tile copy
//   the others        producers (band rows; update and reductions on the way
//                     back) and, in FP64, two more warps of the elimination
// FP64 on this chip is bound by instructions: a sub-partition takes 65 cycles
// for a warp's FP64 instruction, however many lanes it carries (one warp's
// dependent ones 71 to 87, four independent 263; with ten warps 19.5 cycles
// an instruction over the SM).  One warp for both halves spends half of what
// a warp per half does.  The elimination's twelve operations a cell are three
// warps': warp 0 forms the pivot, its inverse and g (five, the chain); warp 4,
// beside it on sub-partition 0 where no producer runs, d and the next cells'
// coefficients (four, while warp 0 inverts); and the right side (three) is
// carried on another sub-partition, a few cells behind.  1024^2, 8 lines a
// block: sweeps of 289/294 us; 317/322 with warp 0 doing nine (890 cycles a
// cell), 422/430 with a warp per half doing fifteen beside producers (1350).
// FP32: a tick is the recurrence's (52 cycles a cell) instead of the
// producers' copies and band rows; 1024^2 37/45 us against 42/53 with copying
// producers and 69/86 in blocks of 32.
#pragma once

#include "tf_line_sweeps.cuh"

namespace tf {

template <class LP, int NL> struct NarrowCfg {
  static_assert(NL == 4 || NL == 8 || NL == 16, "lines per block");
  static constexpr int C = kCX;                    // cells per chunk
  static constexpr int G = NL == 4 ? 2 : 4;        // cells whose band rows one producer thread builds
  static constexpr int NG = C / G;                 // groups of a chunk
  static constexpr int NP = 2 * NG * NL;           // producer threads: one per half, group and line
  static constexpr int PW = NP / 32;               // producer warps
  static constexpr bool Z = sizeof(LP) == 8;       // the right side's recurrence has a warp of its own
  // loader warps: the copies of an FP32 tick must be issued within its 1500
  // cycles (one warp took 1500 to 1950), an FP64 tick is ten times longer
  static constexpr int LW = Z ? (PW > 3 ? 2 : 1) : (PW > 3 ? 3 : 4);
  static constexpr int NLD = 32 * LW;              // loader threads
  static constexpr int NW = 1 + LW + PW + (Z ? 2 : 0);
  static constexpr int NT = 32 * NW;
  static constexpr int D = 4, R = 5;               // ring slots, forward and backward tiles
  static constexpr int XP = 36;                    // row pitch of the x sweep's tiles (whole 16-byte vectors)
  static constexpr int YP = NL == 4 ? 12 : NL + 12;  // row pitch of the y sweep's film tile
  static constexpr int FH = 3 * C * NL + NL;       // a half's factors of a chunk, padded: the halves on different banks
  static constexpr int SUB = 6;                    // cells between two hand-overs to the right side's warp
  static_assert(PW * 32 == NP && PW % 3 == 0 && C % SUB == 0, "whole warps, three of four sub-partitions");
  // Roles of the warps, and a warp's index within its role.  FP32: warp 0, the
  // producers, the loaders.  FP64: warps 0 and 4 (kCoef) on sub-partition 0,
  // producers from 1 on, then the loaders and the right side's warp, none of
  // them on sub-partition 0 but a loader, which has no arithmetic.
  enum Role { kChain, kProducer, kCoef, kRight, kLoader };
  __device__ static Role role(int w) {
    if (w == 0) return kChain;
    if (!Z) return w <= PW ? kProducer : kLoader;
    if (w == 4) return kCoef;
    if (w < 4 || (PW == 6 && w < 8)) return kProducer;
    return w == (PW == 6 ? 9 : 5) ? kRight : kLoader;
  }
  __device__ static int index(int w) {
    if (!Z) return w > PW ? w - 1 - PW : w - 1;
    if (role(w) == kLoader) return PW == 6 ? (w - 8) / 2 : 0;
    return w < 4 ? w - 1 : w - 2;  // producers
  }
};

template <class LP, int NL, int DIR> struct NarrowFwd {
  typedef NarrowCfg<LP, NL> Cf;
  // film tiles: x, rows j0-1..j0+NL of columns c0-4..c0+27; y, rows r0-2.. of columns i0-4..i0+NL+3
  LP ut[Cf::D][2][DIR == 0 ? (NL + 2) * Cf::XP : (Cf::C + 4) * Cf::YP];
  LP rt[Cf::D][2][DIR == 0 ? NL * Cf::XP : Cf::C * NL];  // right sides (x: [row][col], y: [row][col])
  LP band[2][6][Cf::C][2 * NL];                          // [stage][a..e, r][cell][half, line]
  // FP64, between the elimination's warps: beta and 1/mu of a chunk for the
  // right side; 1/mu and g of a cell; beta, c - a d'' and d - beta d' of the next
  LP bi[Cf::Z ? Cf::C : 1][2 * NL][2];
  LP ig[2 * NL][2], co[2 * NL][5];
};
template <class LP, int NL, int DIR> struct NarrowBwd {
  typedef NarrowCfg<LP, NL> Cf;
  LP ft[Cf::R][2][Cf::FH];                                  // factor tiles
  LP xb[2][2][Cf::C][DIR == 0 ? NL + 1 : NL];               // solved chunk [cell][line]
  double ukt[DIR == 0 ? 1 : Cf::R][2][DIR == 0 ? 1 : Cf::C][NL];  // u_k tiles for the update
};
template <class LP, int NL, int DIR> struct NarrowSmem {
  union U {
    NarrowFwd<LP, NL, DIR> f;
    NarrowBwd<LP, NL, DIR> b;
  } s;
  LUState<LP> seam[2 * NL];
  LP xs[NL][4];
  PartY part[NarrowCfg<LP, NL>::NW];
};

// Whether the inverse of a pivot shows that the pivot is zero or not finite
// (no FP64 operation).
__device__ __forceinline__ bool zero_or_nonfinite(double inv) {
  const unsigned hi = (unsigned)__double2hiint(inv) & 0x7fffffffu;
  return hi >= 0x7ff00000u || (hi | (unsigned)__double2loint(inv)) == 0u;
}

// R x W tile columns [col0, col0 + W) x rows [row0, row0 + R) of a row-major
// [ny][nx] array, indices reflected at the walls, by NTH threads: 16-byte
// vectors inside the grid on aligned rows, else elements, with a thread's
// column fixed.
template <int NTH, class T, int R, int W, int DP>
__device__ __forceinline__ void narrow_tile(T* dst, const T* __restrict__ src, int row0, int col0, int ny, int nx, int p) {
  constexpr int V = 16 / sizeof(T), CV = W / V;
  static_assert(W % V == 0 && DP % V == 0, "whole vectors");
  const bool cols = col0 >= 0 && col0 + W <= nx;
  if (cols && row0 >= 0 && row0 + R <= ny && nx % V == 0 &&
      (reinterpret_cast<uintptr_t>(src + col0) & 15) == 0) {
    const T* base = src + (size_t)row0 * nx + col0;
#pragma unroll
    for (int i = 0; i < (R * CV + NTH - 1) / NTH; ++i) {
      const int k = p + i * NTH, r = k / CV, c = (k - r * CV) * V;
      if (k < R * CV) __pipeline_memcpy_async(dst + r * DP + c, base + (size_t)r * nx + c, 16);
    }
    return;
  }
  constexpr int WP = W <= 16 ? 16 : 32, RG = NTH / WP;
  static_assert(W <= WP, "a row of lanes");
  const int c = p % WP;
  if (c >= W) return;
  const T* s = src + (cols ? col0 + c : reflect_index(col0 + c, nx));
#pragma unroll 4
  for (int r = p / WP; r < R; r += RG) {
    int j = row0 + r;
    if (j < 0 || j >= ny) j = reflect_index(j, ny);
    cpT(dst + r * DP + c, s + (size_t)j * nx);
  }
}
// Rows [0, nr) x columns [0, nc) (nr <= R, nc <= W) from base, row pitch nx.
template <int NTH, class T, int R, int W, int DP>
__device__ __forceinline__ void narrow_rows(T* dst, const T* __restrict__ base, int nr, int nc, int nx, int p) {
  constexpr int V = 16 / sizeof(T), CV = W / V;
  static_assert(W % V == 0 && DP % V == 0, "whole vectors");
  if (nc == W && nx % V == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < (R * CV + NTH - 1) / NTH; ++i) {
      const int k = p + i * NTH, r = k / CV, c = (k - r * CV) * V;
      if (r < nr) __pipeline_memcpy_async(dst + r * DP + c, base + (size_t)r * nx + c, 16);
    }
    return;
  }
  constexpr int WP = W <= 4 ? 4 : (W <= 8 ? 8 : (W <= 16 ? 16 : 32)), RG = NTH / WP;
  const int c = p % WP;
  if (c >= nc) return;
#pragma unroll 4
  for (int r = p / WP; r < nr; r += RG) cpT(dst + r * DP + c, base + (size_t)r * nx + c);
}

// A line system given by its matrix instead of a film (FP64): A^T x = r with A's
// diagonals in band[d * N + cell] (the coefficient of line cell t + d - 2 in row
// t) and x to `out`.
struct GivenBand {
  const double* band;
  const double* r;
  double* out;
  size_t N;
};

// DIR 0: the x sweep (lines are rows; w holds the right sides and receives
// the solution).  DIR 1: the y sweep (lines are columns; w is the right side,
// u_{k+1} = u_k + v goes to unew and v to vout when asked for).  DEV and GEN
// as for k_ysweep.
// GIVEN: the producers read the band of A^T from gb.
template <class Mode, int NL, int DIR, bool DEV, bool GEN, bool GIVEN = false>
__global__ void __launch_bounds__((NarrowCfg<typename Mode::LP, NL>::NT), Mode::kSweepBlocks)
    k_narrow_sweep(ModelK M, LineK<typename Mode::LP> Lp, const double* __restrict__ up,
                   const typename Mode::LP* __restrict__ ul, typename Mode::LP* w, typename Mode::LP* __restrict__ fac,
                   double* __restrict__ unp, double* __restrict__ vout, PartX* __restrict__ partx,
                   PartY* __restrict__ party, const LineK<typename Mode::LP>* __restrict__ Ld,
                   const double* const* __restrict__ uio, RunAhead ra, GivenBand gb = {}) {
  if (ra.over()) return;
  typedef typename Mode::LP LP;
  typedef NarrowCfg<LP, NL> Cf;
  constexpr int C = Cf::C, G = Cf::G, D = Cf::D, R = Cf::R, NP = Cf::NP;
  const LineK<LP>& L = DEV ? *Ld : Lp;
  const double* __restrict__ u = DEV && DIR == 1 ? uio[0] : up;
  double* __restrict__ unew = DEV && DIR == 1 ? const_cast<double*>(uio[1]) : unp;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  NarrowSmem<LP, NL, DIR>& S = *reinterpret_cast<NarrowSmem<LP, NL, DIR>*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const typename Cf::Role role = Cf::role(warp);
  const bool chain = role == Cf::kChain, loader = role == Cf::kLoader, producer = role == Cf::kProducer;
  const bool coef = role == Cf::kCoef, zwarp = role == Cf::kRight;
  const int p = Cf::index(warp) * 32 + lane;  // thread within the role
  const int nx = M.nx, ny = M.ny;
  const int n = DIR == 0 ? nx : ny, nlines = DIR == 0 ? ny : nx, line0 = blockIdx.x * NL;
  const int m = split_point(n);
  const bool twisted = m < n;
  const int nch0 = (m + C - 1) / C, nch1 = twisted ? (n - m + C - 1) / C : 0;
  const int nch = max(nch0, nch1);
  auto nchh = [&](int h) { return h ? nch1 : nch0; };
  auto c0_of = [&](int h, int q) { return h == 0 ? q * C : max(m, n - (q + 1) * C); };  // cells [c0, c1) of chunk q
  auto c1_of = [&](int h, int q) { return h == 0 ? min(m, (q + 1) * C) : n - q * C; };
  // the recurrences' lane: half and line
  const int ch = lane / NL, cl = lane % NL;
  const bool mine = lane < 2 * NL && line0 + cl < nlines && ch < 2;
  int bad = 0;

  // ---------------- forward ----------------
  auto issue_fwd = [&](int q) {
    if (GIVEN) return;
    const int slot = q % D;
    for (int h = 0; h < 2; ++h) {
      if (q >= nchh(h)) continue;
      const int c0 = c0_of(h, q), c1 = c1_of(h, q);
      if constexpr (DIR == 0) {
        narrow_tile<Cf::NLD, LP, NL + 2, C + 8, Cf::XP>(S.s.f.ut[slot][h], ul, line0 - 1, c0 - 4, ny, nx, p);
        narrow_rows<Cf::NLD, LP, NL, C, Cf::XP>(S.s.f.rt[slot][h], w + (size_t)line0 * nx + c0, min(NL, ny - line0),
                                                c1 - c0, nx, p);
      } else {
        narrow_tile<Cf::NLD, LP, C + 4, NL + 8, Cf::YP>(S.s.f.ut[slot][h], ul, c0 - 2, line0 - 4, ny, nx, p);
        narrow_rows<Cf::NLD, LP, C, NL, NL>(S.s.f.rt[slot][h], w + (size_t)c0 * nx + line0, c1 - c0,
                                            min(NL, nx - line0), nx, p);
      }
    }
    __pipeline_commit();
  };
  // band rows of cells ia .. ib-1 of one line and half
  auto produce = [&](int t) {
    const int h = p / (NP / 2), g = p / NL % Cf::NG, c = p % NL;
    if (t >= nchh(h) || line0 + c >= nlines) return;
    const int c0 = c0_of(h, t), c1 = c1_of(h, t), ia = c0 + G * g, ib = min(c1, ia + G), slot = t % D;
    if (ia >= ib) return;
    // in the solver's processing order, the second half's band reversed
    LP* P = &S.s.f.band[t & 1][0][h ? c1 - 1 - ia : ia - c0][h * NL + c];
    const int ks = h ? -2 * NL : 2 * NL;
    constexpr int kF = C * 2 * NL;
    if constexpr (GIVEN) {  // row t of A^T is column t of A; the loads of all G cells in flight together
      const size_t step = DIR == 0 ? 1 : (size_t)nx, line = DIR == 0 ? (size_t)(line0 + c) * nx : (size_t)(line0 + c);
      LP v[G][6];
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const int t0 = ia + i;
        if (t0 >= ib) continue;
#pragma unroll
        for (int d = 0; d < 5; ++d) {
          const int row = t0 + d - 2;
          v[i][d] = row >= 0 && row < n ? __ldg(gb.band + (size_t)(4 - d) * gb.N + line + (size_t)row * step) : LP(0);
        }
        v[i][5] = __ldg(gb.r + line + (size_t)t0 * step);
      }
#pragma unroll
      for (int i = 0; i < G; ++i) {
        if (ia + i >= ib) continue;
        LP* q = P + i * ks;
        for (int d = 0; d < 5; ++d) q[d * kF] = h ? v[i][4 - d] : v[i][d];
        q[5 * kF] = v[i][5];
      }
      return;
    }
    const LP* T = S.s.f.ut[slot][h] + (DIR == 0 ? (c + 1) * Cf::XP + ia - c0 + 4 : (ia - c0 + 2) * Cf::YP + c + 4);
    const LP* W = S.s.f.rt[slot][h] + (DIR == 0 ? c * Cf::XP + ia - c0 : (ia - c0) * NL + c);
    auto A = [&](int s, int dr, int dc) {
      return DIR == 0 ? T[dr * Cf::XP + s + dc] : T[(s + dr) * Cf::YP + dc];
    };
    auto out = [&](int s, LP a, LP b, LP cc, LP d, LP e) {
      LP* q = P + s * ks;
      q[0] = h ? e : a;
      q[kF] = h ? d : b;
      q[2 * kF] = cc;
      q[3 * kF] = h ? b : d;
      q[4 * kF] = h ? a : e;
      q[5 * kF] = W[DIR == 0 ? s : s * NL];
    };
    const bool edge = !(ia >= 2 && ia + G + 1 < n);
    if (GEN)
      band_rows<LP, G, DIR, true, false>(L, A, ia, ib, n, out);
    else if (!edge)
      band_rows<LP, G, DIR, false, true>(L, A, ia, ib, n, out);
    else
      band_rows<LP, G, DIR, true, true>(L, A, ia, ib, n, out);
  };
  LUState<LP> lu;
  lu.reset();
  constexpr int kF = C * 2 * NL;
  // Cell s of this lane's chunk in the band stage B (LUState::step's
  // operations), FP32.  beta and tc = c - a d'' of the next cell need only
  // values of the cells before this one: they are formed while this cell's
  // pivot is inverted, out of the chain.
  LP beta = LP(0), tc = LP(0);
  auto eliminate = [&](int s, bool next, const LP* B, LP* Q, LP& chk) {
    const LP* b = B + s * 2 * NL + lane;
    const LP be = beta, mu = tc - beta * lu.g1, dg = b[3 * kF] - beta * lu.d1;
    if (next) {
      beta = b[2 * NL + kF] - b[2 * NL] * lu.g1;
      tc = b[2 * NL + 2 * kF] - b[2 * NL] * lu.d1;
    }
    const LP inv = rcp3(mu), g = dg * inv, dl = b[4 * kF] * inv;
    const LP z = (b[5 * kF] - b[0] * lu.z2 - be * lu.z1) * inv;
    chk = fma(mu, inv, chk);
    lu.g2 = lu.g1;
    lu.d2 = lu.d1;
    lu.z2 = lu.z1;
    lu.g1 = g;
    lu.d1 = dl;
    lu.z1 = z;
    Q[s * NL] = g;
    Q[C * NL + s * NL] = dl;
    Q[2 * C * NL + s * NL] = z;
  };
  // The same in FP64, a chunk of len cells (0: none of this lane's): the three
  // warps meet at named barriers of 64 threads, 5 (1/mu and g of a cell: the
  // chain to the coefficients' warp), 6 (the next cell's coefficients: back) and
  // 1 .. 4 (a sub-chunk's beta and 1/mu: the chain to the right side).  All their
  // lanes go through every cell of the chunk, so that the barriers match; cells
  // at len and beyond are computed from what the band buffer holds and dropped.
  LP* const ig = S.s.f.ig[lane < 2 * NL ? lane : 0];
  LP* const co = S.s.f.co[lane < 2 * NL ? lane : 0];
  const int bl = lane < 2 * NL ? lane : 0;
  auto chain64 = [&](int len, LP* Q) {
    asm volatile("bar.sync 6, 64;" ::: "memory");
    LP be = co[0], t = co[1], dg = co[2], be1 = co[3], t1 = co[4], g = lu.g1;
#pragma unroll 1
    for (int s0 = 0; s0 < C; s0 += Cf::SUB) {
#pragma unroll
      for (int i = 0; i < Cf::SUB; ++i) {
        const int s = s0 + i;
        const LP mu = t - be * g, inv = rcp3(mu);
        if (s > 0) {
          asm volatile("bar.sync 6, 64;" ::: "memory");
          be1 = co[0];
          t1 = co[1];
          dg = co[2];
        }
        g = dg * inv;
        if (lane < 2 * NL) {
          ig[0] = inv;
          ig[1] = g;
          S.s.f.bi[s][lane][0] = be;
          S.s.f.bi[s][lane][1] = inv;
        }
        asm volatile("bar.arrive 5, 64;" ::: "memory");
        if (s < len) {
          Q[s * NL] = g;
          lu.g1 = g;
        }
        be = be1;
        t = t1;
      }
      asm volatile("bar.arrive %0, 64;" ::"r"(1 + s0 / Cf::SUB) : "memory");
    }
  };
  auto coef64 = [&](int len, const LP* B, LP* Q) {
    const LP* b = B + bl;
    LP be1;
    {
      const LP be0 = b[kF] - b[0] * lu.g2, t0 = b[2 * kF] - b[0] * lu.d2;
      const LP a1 = b[2 * NL], dg0 = b[3 * kF] - be0 * lu.d1;
      be1 = b[2 * NL + kF] - a1 * lu.g1;
      const LP t1 = b[2 * NL + 2 * kF] - a1 * lu.d1;
      if (lane < 2 * NL) {
        co[0] = be0;
        co[1] = t0;
        co[2] = dg0;
        co[3] = be1;
        co[4] = t1;
      }
    }
    asm volatile("bar.arrive 6, 64;" ::: "memory");
#pragma unroll 6
    for (int s = 0; s < C; ++s) {
      asm volatile("bar.sync 5, 64;" ::: "memory");
      const LP inv = ig[0], g = ig[1], dl = b[4 * kF] * inv;
      LP be2 = LP(0);
      if (s + 1 < C) {
        const LP dgn = b[2 * NL + 3 * kF] - be1 * dl;
        LP t2 = LP(0);
        if (s + 2 < C) {
          be2 = b[4 * NL + kF] - b[4 * NL] * g;
          t2 = b[4 * NL + 2 * kF] - b[4 * NL] * dl;
        }
        if (lane < 2 * NL) {
          co[0] = be2;
          co[1] = t2;
          co[2] = dgn;
        }
        asm volatile("bar.arrive 6, 64;" ::: "memory");
      }
      if (s < len) {
        Q[C * NL + s * NL] = dl;
        lu.g2 = lu.g1;
        lu.d2 = lu.d1;
        lu.g1 = g;
        lu.d1 = dl;
      }
      be1 = be2;
      b += 2 * NL;
    }
  };
  auto right64 = [&](int len, const LP* B, LP* Q) {
#pragma unroll 1
    for (int s0 = 0; s0 < C; s0 += Cf::SUB) {
      asm volatile("bar.sync %0, 64;" ::"r"(1 + s0 / Cf::SUB) : "memory");
#pragma unroll
      for (int i = 0; i < Cf::SUB; ++i) {
        const int s = s0 + i;
        const LP* b = B + s * 2 * NL + bl;
        const LP inv = S.s.f.bi[s][bl][1];
        const LP z = (b[5 * kF] - b[0] * lu.z2 - S.s.f.bi[s][bl][0] * lu.z1) * inv;
        if (s < len) {
          lu.z2 = lu.z1;
          lu.z1 = z;
          Q[2 * C * NL + s * NL] = z;
          if (zero_or_nonfinite(inv)) bad = 1;
        }
      }
    }
  };
  if (loader) {
    for (int q = 0; q < D - 1; ++q) issue_fwd(q);
    __pipeline_wait_prior(D - 2);
  }
  __syncthreads();
  for (int t = 0; t <= nch; ++t) {
    if (loader) {
      issue_fwd(t + D - 1);  // its slot was consumed last tick
      __pipeline_wait_prior(D - 2);  // chunk t + 1 landed
    } else if (producer) {
      if (t < nch) produce(t);
    } else if (t >= 1) {
      const int q = t - 1;
      const int len = mine && q < nchh(ch) ? c1_of(ch, q) - c0_of(ch, q) : 0;
      const LP* B = &S.s.f.band[q & 1][0][0][0];
      LP* Q = fac + fac_slab<C>(NL, blockIdx.x, ch & 1, q, nch) + cl;
      if constexpr (Cf::Z) {
        if (chain)
          chain64(len, Q);
        else if (coef)
          coef64(len, B, Q);
        else
          right64(len, B, Q);
      } else {
        LP chk = LP(0);
        if (len) {
          beta = B[kF + lane] - B[lane] * lu.g2;
          tc = B[2 * kF + lane] - B[lane] * lu.d2;
        }
        if (__all_sync(0xffffffffu, len == C || len == 0)) {
          if (len) {
#pragma unroll
            for (int s = 0; s < C; ++s) eliminate(s, s + 1 < C, B, Q, chk);
          }
        } else {
#pragma unroll 2
          for (int s = 0; s < C; ++s)
            if (s < len) eliminate(s, s + 1 < len, B, Q, chk);
        }
        if (!(chk == chk)) bad = 1;
      }
    }
    __syncthreads();
  }
  // ---------------- seam ----------------
  if ((Cf::Z ? coef : chain) && lane < 2 * NL) {
    LUState<LP>& o = S.seam[lane];
    o.g1 = lu.g1;
    o.d1 = lu.d1;
    o.g2 = lu.g2;
    o.d2 = lu.d2;
    if (!Cf::Z) {
      o.z1 = lu.z1;
      o.z2 = lu.z2;
    }
  }
  if (zwarp && lane < 2 * NL) {
    S.seam[lane].z1 = lu.z1;
    S.seam[lane].z2 = lu.z2;
  }
  __syncthreads();
  // ---------------- backward ----------------
  // ring of the factor and u_k tiles as in k_ysweep: tick t issues
  // {f(t+R-1), u(t+R-2)} and waits for the group of tick t+2-R
  auto issue_bwd = [&](int bq, int bu) {
    for (int h = 0; h < 2; ++h) {
      const int q = nchh(h) - 1 - bq;
      if (bq < nch && q >= 0)
        copy_span<Cf::NLD, LP, 3 * C * NL>(S.s.b.ft[bq % R][h], fac + fac_slab<C>(NL, blockIdx.x, h, q, nch), 3 * C * NL, p);
      if constexpr (DIR == 1 && !GIVEN) {
        const int v = nchh(h) - 1 - bu;
        if (bu >= 0 && bu < nch && v >= 0) {
          const int r0 = c0_of(h, v);
          narrow_rows<Cf::NLD, double, C, NL, NL>(&S.s.b.ukt[bu % R][h][0][0], u + (size_t)r0 * nx + line0,
                                                  c1_of(h, v) - r0, min(NL, nx - line0), nx, p);
        }
      }
    }
    __pipeline_commit();
  };
  if (loader) {
    for (int g = 0; g < R - 1; ++g) issue_bwd(g, g - 1);
    __pipeline_wait_prior(R - 2);
  }
  if (chain && twisted && lane < NL) {
    LP x[4] = {LP(0), LP(0), LP(0), LP(0)};
    if (!seam(S.seam[lane], S.seam[NL + lane], x) && line0 + lane < nlines) bad = 1;
    for (int q = 0; q < 4; ++q) S.xs[lane][q] = x[q];
  }
  __syncthreads();
  LP x1 = LP(0), x2 = LP(0);
  if (chain && twisted && mine) {
    x1 = S.xs[cl][ch ? 1 : 2];
    x2 = S.xs[cl][ch ? 0 : 3];
  }
  LP err = LP(0);
  int nonfinite = 0;
  for (int t = 0; t <= nch; ++t) {
    if (chain) {
      const int q = nchh(ch & 1) - 1 - t;
      const bool act = mine && t < nch && q >= 0;
      const int c0 = act ? c0_of(ch, q) : 0, len = act ? c1_of(ch, q) - c0 : 0;
      // processed cell s is chunk cell len-1-s (first half) or s
      const int rb = ch ? 0 : len - 1, rs = ch ? 1 : -1;
      const LP* F = S.s.b.ft[t % R][ch & 1] + (act ? len - 1 : 0) * NL + cl;  // slab cell len-1-s, factor f: F[(f * C - s) * NL]
      LP* X = &S.s.b.xb[t & 1][ch & 1][act ? rb : 0][cl];
      const int ks = rs * (DIR == 0 ? NL + 1 : NL);
      // kU cells' factors at a time into registers, ahead of the stores (which
      // the compiler cannot tell from the loads)
      constexpr int kU = 8;
      LP f[kU][3];
      auto one = [&](int s, const LP (&v)[3]) {
        const LP x = fma(-v[0], x1, fma(-v[1], x2, v[2]));
        x2 = x1;
        x1 = x;
        X[s * ks] = x;
      };
      if (__all_sync(0xffffffffu, !act || len == C)) {
        if (act) {
#pragma unroll
          for (int s0 = 0; s0 < C; s0 += kU) {
#pragma unroll
            for (int i = 0; i < kU; ++i)
#pragma unroll
              for (int k = 0; k < 3; ++k) f[i][k] = F[(k * C - s0 - i) * NL];
#pragma unroll
            for (int i = 0; i < kU; ++i) one(s0 + i, f[i]);
          }
        }
      } else {
#pragma unroll 1
        for (int s0 = 0; s0 < C; s0 += kU) {
#pragma unroll
          for (int i = 0; i < kU; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k)
              if (s0 + i < len) f[i][k] = F[(k * C - s0 - i) * NL];
#pragma unroll
          for (int i = 0; i < kU; ++i)
            if (s0 + i < len) one(s0 + i, f[i]);
        }
      }
    } else if (loader) {
      issue_bwd(t + R - 1, t + R - 2);
      __pipeline_wait_prior(R - 2);
    } else if (producer && t >= 1) {
      const int bq = t - 1;
      if constexpr (DIR == 0) {  // w of backward chunk t-1, coalesced along rows
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = nchh(h) - 1 - bq;
          if (q < 0) continue;
          const int c0 = c0_of(h, q), nc = c1_of(h, q) - c0;
          LP* dst;
          if constexpr (GIVEN) dst = gb.out + (size_t)line0 * nx + c0;
          else dst = w + (size_t)line0 * nx + c0;
          const LP* X = &S.s.b.xb[bq & 1][h][0][0];
#pragma unroll
          for (int i = 0; i < (NL * C + NP - 1) / NP; ++i) {
            const int k = p + i * NP, r = k / C, c = k - r * C;
            if (r < NL && line0 + r < ny && c < nc) dst[(size_t)r * nx + c] = X[c * (NL + 1) + r];
          }
        }
      } else {  // update, store, reduce
        constexpr int RG = NP / NL;
        const int c = p % NL, rg = p / NL, col = line0 + c;
        if (col < nx) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int q = nchh(h) - 1 - bq;
            if (q < 0) continue;
            const int r0 = c0_of(h, q), nr = c1_of(h, q) - r0;
#pragma unroll
            for (int i = 0; i < (C + RG - 1) / RG; ++i) {
              const int r = rg + RG * i;
              if (r >= nr) break;
              const LP x = S.s.b.xb[bq & 1][h][r][c];
              if constexpr (GIVEN) {
                gb.out[(size_t)(r0 + r) * nx + col] = x;
                continue;
              }
              const double uk = S.s.b.ukt[bq % R][h][r][c];
              const double un = uk + widen_exact(x);
              const size_t idx = (size_t)(r0 + r) * nx + col;
              unew[idx] = un;
              if (vout) vout[idx] = to_f64(x);
              const LP ru = rel_update(x, uk);
              if (!(ru <= err)) err = ru;
              if (!positive_finite_bits(un)) nonfinite = 1;
            }
          }
        }
      }
    }
    __syncthreads();
  }
  if constexpr (GIVEN) return;
  // ---------------- block reduction ----------------
  for (int o = 16; o > 0; o >>= 1) {
    const LP e2 = __shfl_xor_sync(0xffffffffu, err, o);
    if (!(e2 <= err)) err = e2;
    nonfinite |= __shfl_xor_sync(0xffffffffu, nonfinite, o);
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (lane == 0) {
    S.part[warp].err = (double)err;
    S.part[warp].nonfinite = nonfinite;
    S.part[warp].pivot = bad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    PartY a;
    a.err = 0.0;
    a.hmin = INFINITY;
    a.mass.lo = a.mass.hi = 0ull;
    a.nonfinite = a.pivot = 0;
    for (int k = 0; k < Cf::NW; ++k) {
      if (!(S.part[k].err <= a.err)) a.err = S.part[k].err;
      a.nonfinite |= S.part[k].nonfinite;
      a.pivot |= S.part[k].pivot;
    }
    if constexpr (DIR == 1) {
      party[blockIdx.x] = a;
    } else {
      partx[blockIdx.x].gnorm = 0.0;
      partx[blockIdx.x].pivot = a.pivot;
      partx[blockIdx.x].pad = 0;
    }
  }
}

}  // namespace tf
