// tf_mode.cuh -- launchers of one precision mode; included once by
// tf_mode_fp64.cu and once by tf_mode_f32b.cu.
#pragma once

#include <type_traits>
#include <vector>

#include "tf_internal.h"
#include "tf_rhs_packed.cuh"
#include "tf_ensemble_dev.cuh"

static_assert(tf::kRhsStripCols == tf::kSW && tf::kRhsStripWarps == tf::kSWarps, "residual strips of the launch grid");

namespace tf {

template <class Mode> struct Launch {
  typedef typename Mode::HP HP;
  typedef typename Mode::LP LP;
  static constexpr size_t smem_stencil = sizeof(StencilSmem<HP, 16, 16>);
  template <int T> static constexpr size_t smem_rhs = sizeof(RhsSmem<HP, T>);
  // k_rhs in the context's tiles
  template <int KIND> static cudaError_t launch_rhs(tf_ctx& c, const RhsK<HP>& K, const double* u, RunAhead ra) {
    const dim3 grid(c.grid_rx, c.grid_ry);
    if (c.rhs_tile == 16)
      k_rhs<Mode, KIND, 16><<<grid, 256, smem_rhs<16>, c.stream>>>(c.mk, K, u, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp, c.px, ra);
    else
      k_rhs<Mode, KIND, 32><<<grid, 256, smem_rhs<32>, c.stream>>>(c.mk, K, u, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp, c.px, ra);
    return cudaGetLastError();
  }
  template <int KIND> static cudaError_t prepare_rhs(const tf_ctx& c) {
    return c.rhs_tile == 16 ? allow(k_rhs<Mode, KIND, 16>, smem_rhs<16>) : allow(k_rhs<Mode, KIND, 32>, smem_rhs<32>);
  }
  static constexpr bool kF32B = std::is_same<Mode, ModeF32B>::value;
  // The kernel, threads and shared memory of a sweep (DIR 0: x, 1: y) in
  // blocks of nl lines, and its launch.  DEV, GEN: see k_ysweep.
  template <int NL, int DIR> static constexpr size_t smem_n = sizeof(NarrowSmem<LP, NL, DIR>);
  static constexpr size_t smem_x = sizeof(XSmem<LP>), smem_y = sizeof(YSmem<LP>);
  // whether any film runs in blocks of 32 lines (see sweep_lines and set_shapes in
  // tf_api.cu); a context in a block shape without a kernel is refused
  template <bool GEN> static constexpr bool kWide = !(kF32B && GEN);
  template <int NL, bool DEV, bool GEN>
  static cudaError_t narrow_x(tf_ctx& c, const LineK<LP>& L, const LP* ul, const LineK<LP>* Ld, cudaStream_t s) {
    k_narrow_sweep<Mode, NL, 0, DEV, GEN><<<c.grid_x, NarrowCfg<LP, NL>::NT, smem_n<NL, 0>, s>>>(
        c.mk, L, nullptr, ul, (LP*)c.w, (LP*)c.fac_x, nullptr, nullptr, c.px + c.n_rhs_parts, nullptr, Ld, nullptr, c.ahead);
    return cudaGetLastError();
  }
  template <int NL, bool DEV, bool GEN>
  static cudaError_t narrow_y(tf_ctx& c, const LineK<LP>& L, const double* u, const LP* ul, double* un, double* v,
                       const LineK<LP>* Ld, const double* const* uio, cudaStream_t s) {
    k_narrow_sweep<Mode, NL, 1, DEV, GEN><<<c.grid_y, NarrowCfg<LP, NL>::NT, smem_n<NL, 1>, s>>>(
        c.mk, L, u, ul, (LP*)c.w, (LP*)c.fac_y, un, v, nullptr, c.py, Ld, uio, c.ahead);
    return cudaGetLastError();
  }
  template <bool DEV, bool GEN>
  static cudaError_t launch_x(tf_ctx& c, const LineK<LP>& L, const LP* ul, const LineK<LP>* Ld, cudaStream_t s) {
    switch (c.nlx) {
      case 4: return narrow_x<4, DEV, GEN>(c, L, ul, Ld, s);
      case 8: return narrow_x<8, DEV, GEN>(c, L, ul, Ld, s);
      case 16: return narrow_x<16, DEV, GEN>(c, L, ul, Ld, s);
    }
    if constexpr (kWide<GEN>) {
      if (c.nlx == 32) {
        k_xsweep<Mode, DEV, GEN><<<c.grid_x, kSweepThreads, smem_x, s>>>(c.mk, L, ul, (LP*)c.w, (LP*)c.fac_x,
                                                                       c.px + c.n_rhs_parts, Ld, c.ahead);
        return cudaGetLastError();
      }
    }
    return cudaErrorInvalidValue;
  }
  template <bool DEV, bool GEN>
  static cudaError_t launch_y(tf_ctx& c, const LineK<LP>& L, const double* u, const LP* ul, double* un, double* v,
                       const LineK<LP>* Ld, const double* const* uio, cudaStream_t s) {
    switch (c.nly) {
      case 4: return narrow_y<4, DEV, GEN>(c, L, u, ul, un, v, Ld, uio, s);
      case 8: return narrow_y<8, DEV, GEN>(c, L, u, ul, un, v, Ld, uio, s);
      case 16: return narrow_y<16, DEV, GEN>(c, L, u, ul, un, v, Ld, uio, s);
    }
    if constexpr (kWide<GEN>) {
      if (c.nly == 32) {
        k_ysweep<Mode, DEV, GEN><<<c.grid_y, kSweepThreads, smem_y, s>>>(c.mk, L, u, ul, (const LP*)c.w, (LP*)c.fac_y,
                                                                       un, v, c.py, Ld, uio, c.ahead);
        return cudaGetLastError();
      }
    }
    return cudaErrorInvalidValue;
  }
  // Dynamic shared memory of a sweep kernel; two blocks share an SM only with
  // the largest shared carveout.
  template <class K> static cudaError_t allow(K k, size_t smem) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e ? e : cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  }
  template <int DIR, bool DEV, bool GEN> static cudaError_t prepare_sweep(int nl) {
    switch (nl) {
      case 4: return allow(k_narrow_sweep<Mode, 4, DIR, DEV, GEN>, smem_n<4, DIR>);
      case 8: return allow(k_narrow_sweep<Mode, 8, DIR, DEV, GEN>, smem_n<8, DIR>);
      case 16: return allow(k_narrow_sweep<Mode, 16, DIR, DEV, GEN>, smem_n<16, DIR>);
    }
    if constexpr (kWide<GEN>) {
      if (nl == 32) {
        if constexpr (DIR == 0) return allow(k_xsweep<Mode, DEV, GEN>, smem_x);
        else return allow(k_ysweep<Mode, DEV, GEN>, smem_y);
      }
    }
    return cudaErrorInvalidValue;
  }
  template <bool DEV, bool GEN> static cudaError_t prepare_sweeps(const tf_ctx& c) {
    const cudaError_t e = prepare_sweep<0, DEV, GEN>(c.nlx);
    return e ? e : prepare_sweep<1, DEV, GEN>(c.nly);
  }
  template <int NL> static cudaError_t prepare_solve_t() {
    cudaError_t e = allow(k_narrow_sweep<Mode, NL, 0, false, false, true>, smem_n<NL, 0>);
    return e ? e : allow(k_narrow_sweep<Mode, NL, 1, false, false, true>, smem_n<NL, 1>);
  }
  static StepK step(const tf_ctx& c, double dt) {
    StepK k;
    k.theta_dt = c.p.theta * dt;
    k.expl_dt = (1.0 - c.p.theta) * dt;
    return k;
  }

  // The attributes of the kernels that a context runs (a kernel's take about a
  // microsecond; the ensemble graphs' and the transposed solves' are set on
  // their first use).
  static cudaError_t prepare(tf_ctx& c) {
    cudaError_t e;
    if (!c.packed_rhs &&
        ((e = prepare_rhs<kRhsResidual>(c)) || (e = prepare_rhs<kRhsExplicit>(c)) || (e = prepare_rhs<kRhsBoth>(c))))
      return e;
    if constexpr (kF32B) {
      if (c.part) return part::prepare();
    }
    return prepare_shapes(c);
  }
  // Those of the sweeps in the context's present block shapes, once per shape: a
  // film alone runs in one, and setting up all of them added 8 us to a context's
  // creation (64^2, FP64: 233 us without, 241 with).
  static cudaError_t prepare_shapes(tf_ctx& c) {
    if (c.part) return cudaSuccess;
    const unsigned need = (unsigned)(c.nlx | c.nly << 8);  // 4, 8, 16 or 32 each: a bit
    if ((c.prepared & need) == need) return cudaSuccess;
    const cudaError_t e = power32(c) ? prepare_sweeps<false, false>(c) : prepare_sweeps<false, true>(c);
    if (!e) c.prepared |= need;
    return e;
  }

  static cudaError_t explicit_part_c(tf_ctx& c, const double* u_old, double dt) {
    c.expl_kernels = 1;
    if constexpr (kF32B) {
      if (c.packed_rhs) {
        k_rhs_strip<kRhsExplicit><<<c.grid_pkx, kST, 0, c.stream>>>(
            c.mk, strip_consts(c.mk, step(c, dt), true), u_old, (HP*)c.bn, nullptr, nullptr, nullptr, c.strip_n, c.strip_rows);
        return cudaGetLastError();
      }
    }
    return launch_rhs<kRhsExplicit>(c, rhs_consts<HP>(c.mk, step(c, dt), true), u_old, RunAhead{nullptr, 0});
  }
  // tf_residual: b^n, G, the partial results of its norm (c.px) and the film's
  // mass and least height (c.py).  On the strips unless the heights that they
  // take leave out the precursor's b, below which no film is: such a film would
  // run on both kernels.
  static cudaError_t report_c(tf_ctx& c, const double* u_old, const double* u_k, double dt, double* G, bool tiles,
                              ReportParts* parts) {
    const dim3 grid(c.grid_st_x, c.grid_st_y), block(16, 16);
    if constexpr (kF32B) {
      if (c.packed_rhs && u_old && !strip_range(c.mk, step(c, dt).expl_dt).has(c.p.b)) {
        k_stencil<Mode, 0><<<grid, block, smem_stencil, c.stream>>>(c.mk, rhs_consts<HP>(c.mk, step(c, dt), true), u_old,
                                                                    (HP*)c.bn, nullptr, nullptr);
        u_old = nullptr;
      }
    }
    if (u_old) {
      const cudaError_t e = explicit_part_c(c, u_old, dt);
      if (e) return e;
    }
    if constexpr (kF32B) {
      if (c.packed_rhs && !tiles) {
        const StripRange range = strip_range(c.mk, step(c, dt).theta_dt);
        if (range.has(c.p.b)) {
          *parts = ReportParts{c.grid_pkx, c.grid_pkx, true};
          k_rhs_strip<kRhsReport><<<c.grid_pkx, kST, 0, c.stream>>>(
              c.mk, strip_consts(c.mk, step(c, dt), false), u_k, (HP*)c.bn, nullptr, nullptr, c.px, c.strip_n, c.strip_rows,
              nullptr, nullptr, G, c.py, RunAhead{nullptr, 0}, range);
          return cudaGetLastError();
        }
      }
    }
    *parts = ReportParts{c.grid_st_x * c.grid_st_y, c.grid_stats, false};
    k_grid_stats<<<c.grid_stats, 256, 0, c.stream>>>(u_k, c.N, c.py);
    k_stencil<Mode, 1><<<grid, block, smem_stencil, c.stream>>>(c.mk, rhs_consts<HP>(c.mk, step(c, dt)), u_k, (HP*)c.bn,
                                                                G, c.px);
    return cudaGetLastError();
  }
  static cudaError_t rhs_c(tf_ctx& c, const double* u_k, double dt) {
    if constexpr (kF32B) {
      if (c.packed_rhs) {
        k_rhs_strip<kRhsResidual><<<c.grid_pkx, kST, 0, c.stream>>>(
            c.mk, strip_consts(c.mk, step(c, dt), false), u_k, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp, c.px, c.strip_n, c.strip_rows,
            nullptr, nullptr, nullptr, nullptr, c.ahead);
        return cudaGetLastError();
      }
    }
    return launch_rhs<kRhsResidual>(c, rhs_consts<HP>(c.mk, step(c, dt)), u_k, c.ahead);
  }
  // b^n of a step and the right side of its first iteration (u_0 = u^n)
  // from one D(u^n); results equal explicit_part_c then rhs_c.
  static cudaError_t explicit_rhs0_c(tf_ctx& c, const double* u_old, double dt) {
    c.expl_kernels = 1;
    if constexpr (kF32B) {
      if (c.packed_rhs) {
        k_rhs_strip<kRhsBoth><<<c.grid_pkx, kST, 0, c.stream>>>(
            c.mk, strip_consts(c.mk, step(c, dt), true), u_old, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp, c.px, c.strip_n, c.strip_rows);
        return cudaGetLastError();
      }
    }
    return launch_rhs<kRhsBoth>(c, rhs_consts<HP>(c.mk, step(c, dt), true), u_old, RunAhead{nullptr, 0});
  }
  // A^T x = r along every line of direction dir (FP64): x in `out`, factors in
  // fac (fac_slab of 16 lines a block at most).
  template <int NL, int DIR> static cudaError_t solve_t_nl(tf_ctx& c, const GivenBand& gb, double* fac, cudaStream_t s) {
    const int lines = DIR == 0 ? c.mk.ny : c.mk.nx;
    k_narrow_sweep<Mode, NL, DIR, false, false, true><<<(lines + NL - 1) / NL, NarrowCfg<LP, NL>::NT, smem_n<NL, DIR>, s>>>(
        c.mk, LineK<LP>(), nullptr, nullptr, nullptr, (LP*)fac, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
        RunAhead{nullptr, 0}, gb);
    return cudaGetLastError();
  }
  template <int DIR> static cudaError_t solve_t_dir(tf_ctx& c, const GivenBand& gb, double* fac, cudaStream_t s) {
    switch (DIR == 0 ? c.nlx : c.nly) {
      case 4: return solve_t_nl<4, DIR>(c, gb, fac, s);
      case 8: return solve_t_nl<8, DIR>(c, gb, fac, s);
      default: return solve_t_nl<16, DIR>(c, gb, fac, s);
    }
  }
  static cudaError_t solve_t_prepare() {
    if constexpr (kF32B) {
      return cudaErrorNotSupported;
    } else {
      cudaError_t e;
      if ((e = prepare_solve_t<4>()) || (e = prepare_solve_t<8>())) return e;
      return prepare_solve_t<16>();
    }
  }
  static cudaError_t solve_t_c(tf_ctx& c, int dir, const double* band, const double* r, double* out, double* fac, cudaStream_t s) {
    if constexpr (kF32B) {
      return cudaErrorNotSupported;
    } else {
      const GivenBand gb = {band, r, out, c.N};
      return dir == 0 ? solve_t_dir<0>(c, gb, fac, s) : solve_t_dir<1>(c, gb, fac, s);
    }
  }
  // film the sweeps stage: u_k itself in FP64, its FP32 copy (written by
  // k_rhs of the same iteration) in FP32-bulk
  static const LP* film_lp(const tf_ctx& c, const double* u_k) {
    return sizeof(LP) == sizeof(double) ? (const LP*)u_k : (const LP*)c.ulp;
  }
  static bool power32(const tf_ctx& c) { return c.mk.model == 0 && c.mk.n == 3 && c.mk.m == 2; }
  static cudaError_t xsweep_c(tf_ctx& c, double dt, const double* u_k) {
    if constexpr (kF32B) {
      if (c.part) return part::xsweep(c, dt);
    }
    const LineK<LP> L = line_consts<LP>(c.mk, step(c, dt));
    return power32(c) ? launch_x<false, false>(c, L, film_lp(c, u_k), nullptr, c.stream)
                      : launch_x<false, true>(c, L, film_lp(c, u_k), nullptr, c.stream);
  }
  static cudaError_t ysweep_c(tf_ctx& c, const double* u_k, double dt, double* u_next,
                              double* v_out) {
    if constexpr (kF32B) {
      if (c.part) return part::ysweep(c, u_k, dt, u_next, v_out);
    }
    const LineK<LP> L = line_consts<LP>(c.mk, step(c, dt));
    return power32(c) ? launch_y<false, false>(c, L, u_k, film_lp(c, u_k), u_next, v_out, nullptr, nullptr, c.stream)
                      : launch_y<false, true>(c, L, u_k, film_lp(c, u_k), u_next, v_out, nullptr, nullptr, c.stream);
  }
  // The whole run of an ensemble film as one graph (FP32-bulk, (3, 2) power
  // law, twisted sweeps): k_ens_begin, then WHILE (attempts) { explicit part
  // with the first residual, x sweep, y sweep, k_ens_iter (reductions and
  // the iteration's classification); WHILE (further iterations) { residual,
  // x sweep, y sweep, k_ens_iter }; copy of the result, film statistics,
  // k_ens_step (their reductions and the step controller) }.  The kernels
  // and their order are those of a tf_advance step, with their constants and
  // grids read from e.
  static cudaError_t ens_graph_c(tf_ctx& c, EnsDev* e, cudaGraphExec_t* out) {
    if constexpr (!kF32B) {
      return cudaErrorNotSupported;
    } else {
      if (!c.packed_rhs || c.part) return cudaErrorNotSupported;
      cudaStream_t s = nullptr;
      cudaGraph_t g = nullptr, B = nullptr, I = nullptr;
      cudaError_t err = prepare_sweeps<true, false>(c);
      if (err) return err;
      err = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
      if (err) return err;
      const cudaStreamCaptureMode md = cudaStreamCaptureModeRelaxed;
      const StripK rk0 = strip_consts(c.mk, step(c, 1.0), false);  // placeholders: read from e
      const LineK<LP> l0 = line_consts<LP>(c.mk, step(c, 1.0));
      cudaGraphConditionalHandle ho, hi;
      cudaGraphNode_t nb = nullptr, no = nullptr, nx = nullptr, ni = nullptr;
      size_t one = 1;
      auto fail = [&](cudaError_t x) {
        cudaStreamDestroy(s);
        if (g) cudaGraphDestroy(g);
        return x;
      };
      // one Newton iteration's sweeps and reductions
      auto sweeps = [&]() {
        if ((err = launch_x<true, false>(c, l0, (const LP*)c.ulp, &e->line, s))) return;
        if ((err = launch_y<true, false>(c, l0, nullptr, (const LP*)c.ulp, nullptr, nullptr, &e->line, &e->p.uk, s))) return;
        k_ens_iter<<<1, 256, 0, s>>>(c.px, c.n_rhs_parts + c.grid_x, c.py, c.grid_y, e, hi);
      };
      if ((err = cudaGraphCreate(&g, 0))) return fail(err);
      if ((err = cudaGraphConditionalHandleCreate(&ho, g, 0, cudaGraphCondAssignDefault))) return fail(err);
      // top level: the first attempt
      if ((err = cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, md))) return fail(err);
      k_ens_begin<<<1, 1, 0, s>>>(e, ho);
      if ((err = cudaStreamEndCapture(s, &g))) return fail(err);
      if ((err = cudaGraphGetNodes(g, &nb, &one)) || one != 1) return fail(err ? err : cudaErrorUnknown);
      cudaGraphNodeParams po = {};
      po.type = cudaGraphNodeTypeConditional;
      po.conditional.handle = ho;
      po.conditional.type = cudaGraphCondTypeWhile;
      po.conditional.size = 1;
      if ((err = cudaGraphAddNode(&no, g, &nb, nullptr, 1, &po))) return fail(err);
      B = po.conditional.phGraph_out[0];
      // attempt: the explicit part with the first iteration's residual, and
      // the first iteration
      if ((err = cudaGraphConditionalHandleCreate(&hi, B, 0, cudaGraphCondAssignDefault))) return fail(err);
      if ((err = cudaStreamBeginCaptureToGraph(s, B, nullptr, nullptr, 0, md))) return fail(err);
      k_rhs_strip<kRhsBoth, true><<<c.grid_pkx, kST, 0, s>>>(c.mk, rk0, nullptr, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp, c.px,
                                                             c.strip_n, c.strip_rows, &e->rk_both, &e->p.cur);
      sweeps();
      if (err) return fail(err);
      if ((err = cudaStreamEndCapture(s, &B))) return fail(err);
      {  // the last node of the chain: the one no other node depends on
        size_t nn = 0, ne = 0;
        if ((err = cudaGraphGetNodes(B, nullptr, &nn))) return fail(err);
        std::vector<cudaGraphNode_t> nodes(nn);
        if ((err = cudaGraphGetNodes(B, nodes.data(), &nn))) return fail(err);
        for (cudaGraphNode_t n : nodes) {
          if ((err = cudaGraphNodeGetDependentNodes(n, nullptr, nullptr, &ne))) return fail(err);
          if (ne == 0) nx = n;
        }
        if (!nx) return fail(cudaErrorUnknown);
      }
      cudaGraphNodeParams pi = {};
      pi.type = cudaGraphNodeTypeConditional;
      pi.conditional.handle = hi;
      pi.conditional.type = cudaGraphCondTypeWhile;
      pi.conditional.size = 1;
      if ((err = cudaGraphAddNode(&ni, B, &nx, nullptr, 1, &pi))) return fail(err);
      I = pi.conditional.phGraph_out[0];
      // the iterations after the first
      if ((err = cudaStreamBeginCaptureToGraph(s, I, nullptr, nullptr, 0, md))) return fail(err);
      k_rhs_strip<kRhsResidual, true><<<c.grid_pkx, kST, 0, s>>>(c.mk, rk0, nullptr, (HP*)c.bn, (LP*)c.w, (LP*)c.ulp,
                                                                 c.px, c.strip_n, c.strip_rows, &e->rk_res, &e->p.uk);
      sweeps();
      if (err) return fail(err);
      if ((err = cudaStreamEndCapture(s, &I))) return fail(err);
      // end of the attempt: the result into nxt, its statistics, the controller
      if ((err = cudaStreamBeginCaptureToGraph(s, B, &ni, nullptr, 1, md))) return fail(err);
      k_ens_copy<<<c.grid_stats < 1024 ? c.grid_stats : 1024, 256, 0, s>>>(e, c.N);
      k_grid_stats<<<c.grid_stats, 256, 0, s>>>(nullptr, c.N, c.py, &e->p.nxt);
      k_ens_step<<<1, 256, 0, s>>>(c.py, c.grid_stats, e, ho);
      if ((err = cudaStreamEndCapture(s, &B))) return fail(err);
      cudaGraphExec_t x = nullptr;  // *out only ever holds an instantiated graph
      if ((err = cudaGraphInstantiate(&x, g, 0))) return fail(err);
      *out = x;
      cudaGraphDestroy(g);
      cudaStreamDestroy(s);
      return cudaSuccess;
    }
  }
  static cudaError_t w_to_f64_c(tf_ctx& c, double* out) {
    if (sizeof(LP) == sizeof(double))
      return cudaMemcpyAsync(out, c.w, c.N * sizeof(double), cudaMemcpyDeviceToDevice, c.stream);
    k_to_f64<LP><<<1024, 256, 0, c.stream>>>((const LP*)c.w, out, c.N);
    return cudaGetLastError();
  }
};

template <class Mode> Ops make_ops() {
  typedef Launch<Mode> L;
  Ops o;
  o.hp_bytes = sizeof(typename Mode::HP);
  o.lp_bytes = sizeof(typename Mode::LP);
  o.prepare = &L::prepare;
  o.prepare_shapes = &L::prepare_shapes;
  o.explicit_part = &L::explicit_part_c;
  o.explicit_rhs0 = &L::explicit_rhs0_c;
  o.report = &L::report_c;
  o.rhs = &L::rhs_c;
  o.xsweep = &L::xsweep_c;
  o.ysweep = &L::ysweep_c;
  o.w_to_f64 = &L::w_to_f64_c;
  o.ens_graph = L::kF32B ? &L::ens_graph_c : nullptr;
  o.solve_t_prepare = L::kF32B ? nullptr : &L::solve_t_prepare;
  o.solve_t = L::kF32B ? nullptr : &L::solve_t_c;
  return o;
}

}  // namespace tf
