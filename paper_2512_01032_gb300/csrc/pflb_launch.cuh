// pflb_launch.cuh -- per-precision kernel launchers (included by one
// translation unit per storage type).
#pragma once
#include <cstring>
#include <type_traits>

#include "pflb_async.cuh"
#include "pflb_internal.h"
#include "pflb_kernels.cuh"
#include "pflb_phase.cuh"
#include "pflb_pipe.cuh"

namespace pflb {

template <class R>
static Model<R> make_model(const pflb_params &p) {
  const double T = 1.0 / 3.0;
  Model<R> m;
  m.sigma = (R)p.sigma;
  m.W = (R)p.W;
  m.M = (R)p.M;
  m.rho_L = (R)p.rho_L;
  m.rho_dif = (R)(p.rho_H - p.rho_L);
  m.tau_H = (R)(p.nu_H / T + 0.5);
  m.tau_L = (R)(p.nu_L / T + 0.5);
  m.Fx = (R)p.Fex[0];
  m.Fy = (R)p.Fex[1];
  m.Fz = (R)p.Fex[2];
  m.gamma = (R)p.gamma;
  m.phi_M = (R)p.phi_M;
  m.phi_m = (R)p.phi_m;
  m.inv_D = (R)(1.0 / p.D);
  m.eps = (R)p.eps;
  m.blend = (R)p.blend;
  m.band_lo = (R)p.band_lo;
  m.band_hi = (R)p.band_hi;
  m.F_tilde = (R)p.F_tilde;
  m.inv_F_width = (R)(1.0 / p.F_width);
  m.inv_tau_phi = (R)(1.0 / (p.M / T + 0.5));
  m.theta_coef = (R)(p.M / (T * p.W));
  m.mu_a = (R)(48.0 * p.sigma / p.W);
  m.mu_b = (R)(1.5 * p.sigma * p.W);
  m.two_over_W = (R)(2.0 / p.W);
  m.F_mode = p.F_mode;
  m.mobility_corr = p.mobility_corr;
  m.free_slip = p.free_slip;
  return m;
}

template <class S, class R>
static Args<S, R> make_args(const Lattice &L, int parity) {
  Args<S, R> a;
  a.nx = L.nx; a.ny = L.ny; a.nz = L.nz; a.lz = L.lz;
  a.N = (int)L.N;
  a.nw = L.nw;
  a.dx = fast_div((uint32_t)L.nx);
  a.dxy = fast_div((uint32_t)L.nx * (uint32_t)L.ny);
  a.plain = L.nx % 4 != 0;
  a.batch = L.in_batch;
  const int rd = parity;
  for (int i = 0; i < Q + 1; ++i) {
    const bool have = i < h_slots<S>();
    a.hin[i] = have ? (const S *)L.h[rd] + (size_t)i * L.N : nullptr;
    a.hout[i] = have ? (S *)L.h[rd ^ 1] + (size_t)i * L.N : nullptr;
  }
  for (int i = 0; i < Q; ++i) a.g[i] = (S *)L.g + (size_t)i * L.N;
  a.flags = L.flags;
  a.widx = L.widx;
  a.wmask = L.wmask;
  a.wcell = L.wcell;
  a.wgeo = (const R *)L.wgeo;
  a.wcut = L.wcut;
  a.sfrac = (const R *)L.sfrac;
  a.ghost = (R *)L.ghost;
  a.wp_rd = (const S *)L.wp[rd];
  a.wp_wr = (S *)L.wp[rd ^ 1];
  a.phi = (const R *)L.phi;
  a.phi_w = (R *)L.phi;
  a.m = make_model<R>(L.p);
  a.diag = nullptr;
  a.diag_zero = nullptr;
  for (int k = 0; k < 6; ++k) a.reg[k] = L.reg[k];
  a.reg_all = L.reg[0] <= 0 && L.reg[1] >= L.nx && L.reg[2] <= 0 && L.reg[3] >= L.ny &&
              L.reg[4] <= 0 && L.reg[5] >= L.nz;
  a.out = nullptr;
  a.field = 0;
  a.bcm = L.bc_on ? (R *)L.bcm : nullptr;
  a.nbc = 2 * L.ny * L.nz;
  a.wl = nullptr;  // set by the pipelined launch when its lists are current
  a.wl_start = nullptr;
  return a;
}
template <class S, class R>
static Args<S, R> make_args(const Lattice &L) {
  return make_args<S, R>(L, (int)(L.step & 1));
}

// Boundary states of the open x planes for the state the next launch reads.
template <class S, class R>
static cudaError_t launch_xbc(Lattice &L, const Args<S, R> &a) {
  if (!L.bc_on) return cudaSuccess;
  const XbcSpec sp = xbc_spec(L, L.step);
  const int n = 2 * L.ny * L.nz, T = 128;
  if (L.step & 1)
    k_xbc<S, R, true><<<(n + T - 1) / T, T, 0, L.stream>>>(a, sp);
  else
    k_xbc<S, R, false><<<(n + T - 1) / T, T, 0, L.stream>>>(a, sp);
  return cudaGetLastError();
}

template <class S, class R>
cudaError_t set_model(Lattice &) { return cudaSuccess; }

template <class S, class R>
int max_block_threads() { return 256; }

template <class S, class R>
cudaError_t launch_init(Lattice &L, const double *d_phi0, double P0) {
  L.step = 0;
  L.ndiag = 0;
  L.last_diag_step = -1;
  Args<S, R> a = make_args<S, R>(L);
  cudaError_t e = cudaMemsetAsync(L.diag, 0, kDiagWords * sizeof(double), L.stream);
  if (e != cudaSuccess) return e;
  const int T = 256;
  const long long B = (L.N + T - 1) / T;
  k_init<S, R><<<(unsigned)B, T, 0, L.stream>>>(a, d_phi0, P0, (S *)L.h[0], (S *)L.wp[0]);
  return cudaGetLastError();
}

// The staged kernel (FP32, x extent a multiple of 4 and at least 64).
inline bool async_eligible(const Lattice &L) {
  return L.kernel == PFLB_KERNEL_FUSED_TMA && L.p.storage == PFLB_STORAGE_FP32 && L.tma_ok &&
         !L.bc_on;
}

template <bool ODD, bool DIAG>
static cudaError_t async_attrs() {
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_fused_async<ODD, DIAG>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AB_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_fused_async<ODD, DIAG>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  return cudaSuccess;
}

template <bool ODD, bool DIAG>
static cudaError_t launch_async_t(Lattice &L, Args<float, float> &a) {
  cudaError_t e0 = async_attrs<ODD, DIAG>();
  if (e0 != cudaSuccess) return e0;
  dim3 grid((L.nx + AB_X - 1) / AB_X, (L.ny + AB_Y - 1) / AB_Y, (L.nz + L.lz - 1) / L.lz);
  k_fused_async<ODD, DIAG><<<grid, AB_X * AB_Y, AB_SMEM, L.stream>>>(a, L.tmap[L.step & 1], L.err);
  return cudaGetLastError();
}

// The pipelined kernel (FP32 storage, periodic x, nx a multiple of 4).
template <class S>
constexpr bool pipe_storage() {
  return std::is_same<S, float>::value;
}
inline bool pipe_eligible(const Lattice &L) { return pipe_kernel_runs(L); }

// Dynamic shared memory above 48 KB is opted into once per device.
template <class S, class R, bool ODD, bool DIAG, bool FORCE>
static cudaError_t pipe_attrs() {
  static unsigned long long done = 0;  // bit d: set on device d
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit && (done & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(k_pipe<S, R, ODD, DIAG, FORCE>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sizeof(PipeSmem<S, R>));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_pipe<S, R, ODD, DIAG, FORCE>,
                           cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e != cudaSuccess) return e;
  done |= bit;
  return cudaSuccess;
}

template <class S, class R, bool ODD, bool DIAG, bool FORCE>
static cudaError_t launch_pipe_f(Lattice &L, Args<S, R> &a) {
  cudaError_t e = pipe_attrs<S, R, ODD, DIAG, FORCE>();
  if (e != cudaSuccess) return e;
  const dim3 grid((L.nx + PP_BX - 1) / PP_BX, (L.ny + PP_BY - 1) / PP_BY,
                  (L.nz + L.lz - 1) / L.lz);
  // the wall nodes of each block, listed for the planes per block in effect (a
  // list for another depth would have blocks update other blocks' nodes)
  if (L.nw > 0 && (!L.wl || L.wl_lz != L.lz)) return cudaErrorInvalidValue;
  a.wl = L.nw > 0 ? L.wl : nullptr;
  a.wl_start = L.nw > 0 ? L.wl_start : nullptr;
  k_pipe<S, R, ODD, DIAG, FORCE><<<grid, PP_NT, sizeof(PipeSmem<S, R>), L.stream>>>(a);
  return cudaGetLastError();
}

// The variant without body-force terms when F_ex = 0 (they vanish there).
template <class S, class R, bool ODD, bool DIAG>
static cudaError_t launch_pipe_t(Lattice &L, Args<S, R> &a) {
  if constexpr (std::is_same<R, float>::value) {
    if (a.m.Fx == R(0) && a.m.Fy == R(0) && a.m.Fz == R(0))
      return launch_pipe_f<S, R, ODD, DIAG, false>(L, a);
  }
  return launch_pipe_f<S, R, ODD, DIAG, true>(L, a);
}

// Launch that may be set up while the kernel before it on the stream still
// runs (the kernel itself waits for that one's end).
template <class... P, class... A>
static cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block,
                                    size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Phase 1 of one lattice.
template <class S, class R, bool ODD, bool XBC>
static cudaError_t launch_phi(Lattice &L, const Args<S, R> &a) {
  const long long V = phase1_vec<S>(L.N) ? 16 / (int)sizeof(S) : 1;
  const int nstate = XBC ? (2 * L.ny * L.nz + PH_NT1 - 1) / PH_NT1 : 0;
  const long long nphi = (L.N + PH_NT1 * V - 1) / (PH_NT1 * V);
  return launch_dependent(k_phase1<S, R, ODD, XBC>, (unsigned)(nstate + nphi), PH_NT1, 0, L.stream,
                          a, xbc_spec(L, L.step), nstate);
}

// The two-phase step of one lattice.
template <class S, class R, bool ODD, bool DIAG, bool XBC, int FORM>
static cudaError_t launch_phases_f(Lattice &L, const Args<S, R> &a) {
  cudaError_t e = launch_phi<S, R, ODD, XBC>(L, a);
  if (e != cudaSuccess) return e;
  const int plane2 = 2 * L.ny * L.nz;
  constexpr int NT = phase2_threads<R>();
  const int nwall = (L.nw + NT - 1) / NT, nedge = XBC ? (plane2 + NT - 1) / NT : 0;
  const long long grid = nwall + nedge + (L.N + NT - 1) / NT;
  return launch_dependent(k_phase2<S, R, ODD, DIAG, XBC, FORM>, (unsigned)grid, NT, 0, L.stream, a,
                          nwall, nedge);
}

// The variant without body-force terms when F_ex = 0 (they vanish there).
template <class S, class R, bool ODD, bool DIAG>
static cudaError_t launch_phases(Lattice &L, const Args<S, R> &a) {
  if (L.bc_on) return launch_phases_f<S, R, ODD, DIAG, true, open_form<S>()>(L, a);
  if constexpr (open_form<S>() == FORM_PLAIN) {
    if (a.plain) return launch_phases_f<S, R, ODD, DIAG, false, FORM_PLAIN>(L, a);
  }
  if (a.m.Fx == R(0) && a.m.Fy == R(0) && a.m.Fz == R(0))
    return launch_phases_f<S, R, ODD, DIAG, false, FORM_NOFORCE>(L, a);
  return launch_phases_f<S, R, ODD, DIAG, false, FORM_FORCE>(L, a);
}

template <class S, class R, bool ODD, bool DIAG>
static cudaError_t launch_fused_t(Lattice &L, Args<S, R> &a) {
  if (phase_kernel_runs(L)) return launch_phases<S, R, ODD, DIAG>(L, a);
  if constexpr (pipe_storage<S>()) {
    if (pipe_eligible(L)) return launch_pipe_t<S, R, ODD, DIAG>(L, a);
  }
  if constexpr (std::is_same<S, float>::value && std::is_same<R, float>::value) {
    if (async_eligible(L)) return launch_async_t<ODD, DIAG>(L, a);
  }
  const int bx = L.bx, by = L.by;
  dim3 grid((L.nx + bx - 1) / bx, (L.ny + by - 1) / by, (L.nz + L.lz - 1) / L.lz);
  const size_t smem = fused_smem_bytes<R>(bx, by, DIAG);
  if (L.bc_on)  // open x boundaries: the variant with boundary cells
    k_fused<S, R, ODD, DIAG, true><<<grid, bx * by, smem, L.stream>>>(a, bx, by);
  else
    k_fused<S, R, ODD, DIAG, false><<<grid, bx * by, smem, L.stream>>>(a, bx, by);
  return cudaGetLastError();
}

template <class S, class R, bool ODD, int MODE, bool DIAG>
static cudaError_t launch_cell_t(Lattice &L, Args<S, R> &a) {
  const int T = 256;
  const long long B = (L.N + T - 1) / T;
  if (L.bc_on)
    k_phi<S, R, true><<<(unsigned)B, T, 0, L.stream>>>(a, (R *)L.phi);
  else
    k_phi<S, R, false><<<(unsigned)B, T, 0, L.stream>>>(a, (R *)L.phi);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (L.bc_on)
    k_cell<S, R, ODD, MODE, DIAG, true><<<(unsigned)B, T, 0, L.stream>>>(a);
  else
    k_cell<S, R, ODD, MODE, DIAG, false><<<(unsigned)B, T, 0, L.stream>>>(a);
  return cudaGetLastError();
}

// Planes per block for the fused kernels.  Blocks all do the same work, so
// a launch takes ceil(blocks / resident slots) rounds of one block's time;
// a block of lz planes also recomputes phi on two halo planes (about 0.3 of
// a plane's cost each).  Chooses lz in [2, 32] minimising
// rounds x (lz + 0.6), e.g. 7 for 128^3 with 32 x 4 tiles on 152 SMs x 4
// blocks (19 chunks x 128 columns = 4 full rounds).
template <class S, class R>
int auto_lz(const Lattice &L) {
  int dev = 0, nsm = 0, per = 0;
  bool tma = false, pipe = false;
  if constexpr (std::is_same<S, float>::value && std::is_same<R, float>::value)
    tma = async_eligible(L);
  if constexpr (pipe_storage<S>()) pipe = pipe_eligible(L);
  const int bx = pipe ? PP_BX : (tma ? AB_X : L.bx), by = pipe ? PP_BY : (tma ? AB_Y : L.by);
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) {
    if (pipe) {
      if constexpr (pipe_storage<S>()) {
        e = pipe_attrs<S, R, false, true, true>();
        if (e == cudaSuccess)
          e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
              &per, k_pipe<S, R, false, true, true>, PP_NT, sizeof(PipeSmem<S, R>));
      }
    } else if (tma) {
      if constexpr (std::is_same<S, float>::value && std::is_same<R, float>::value) {
        e = async_attrs<false, true>();
        if (e == cudaSuccess)
          e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fused_async<false, true>,
                                                            bx * by, AB_SMEM);
      }
    } else {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fused<S, R, false, true>,
                                                        bx * by,
                                                        fused_smem_bytes<R>(bx, by, true));
    }
  }
  if (e != cudaSuccess || nsm < 1 || per < 1) {
    cudaGetLastError();
    return L.nz < 16 ? L.nz : 16;
  }
  const long long slots = (long long)nsm * per;
  const long long cols = (long long)((L.nx + bx - 1) / bx) * ((L.ny + by - 1) / by);
  int best = L.nz < 16 ? L.nz : 16;
  double best_cost = 1e300;
  for (int lz = (L.nz < 32 ? L.nz : 32); lz >= 2; --lz) {
    const long long blocks = cols * ((L.nz + lz - 1) / lz);
    const double cost = (double)((blocks + slots - 1) / slots) * (lz + 0.6);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = lz;
    }
  }
  return best;
}

template <class S, class R>
cudaError_t launch_step(Lattice &L, bool diag) {
  Args<S, R> a = make_args<S, R>(L);
  const bool odd = (L.step & 1) != 0;
  // (the two-phase step forms the boundary states itself)
  cudaError_t e = phase_kernel_runs(L) ? cudaSuccess : launch_xbc<S, R>(L, a);
  if (e != cudaSuccess) return e;
  if (diag) {
    // Diagnostic launch d accumulates into accumulator d&1 and zeroes the other.
    a.diag = diag_acc(L, (int)(L.ndiag & 1));
    a.diag_zero = diag_acc(L, (int)((L.ndiag + 1) & 1));
  }
  if (L.kernel != PFLB_KERNEL_TWOPASS) {  // fused, its TMA-staged and pipelined forms
    if (odd) e = diag ? launch_fused_t<S, R, true, true>(L, a) : launch_fused_t<S, R, true, false>(L, a);
    else e = diag ? launch_fused_t<S, R, false, true>(L, a) : launch_fused_t<S, R, false, false>(L, a);
  } else {
    if (odd) e = diag ? launch_cell_t<S, R, true, MODE_STEP, true>(L, a)
                      : launch_cell_t<S, R, true, MODE_STEP, false>(L, a);
    else e = diag ? launch_cell_t<S, R, false, MODE_STEP, true>(L, a)
                  : launch_cell_t<S, R, false, MODE_STEP, false>(L, a);
  }
  if (e == cudaSuccess) {
    if (diag) {
      L.last_diag_step = L.step;
      L.ndiag++;
    }
    L.step++;
  }
  return e;
}

// Diagnostics of the current state.
template <class S, class R>
cudaError_t launch_macro(Lattice &L) {
  Args<S, R> a = make_args<S, R>(L);
  a.diag = diag_acc(L, 2);
  a.diag_zero = nullptr;
  cudaError_t e = cudaMemsetAsync(a.diag, 0, 32 * kDiagCopies * sizeof(double), L.stream);
  if (e == cudaSuccess) e = launch_xbc<S, R>(L, a);
  if (e != cudaSuccess) return e;
  if (L.step & 1) return launch_cell_t<S, R, true, MODE_MACRO, true>(L, a);
  return launch_cell_t<S, R, false, MODE_MACRO, true>(L, a);
}

// One field of the current state into L.out.
template <class S, class R, bool ODD, bool XBC>
static cudaError_t launch_read_t(Lattice &L, int field) {
  Args<S, R> a = make_args<S, R>(L);
  a.out = L.out;
  a.field = field;
  if (field <= PFLB_FIELD_RHO) {
    const long long n = L.N / (phase1_vec<S>(L.N) ? 16 / (int)sizeof(S) : 1);
    return launch_dependent(k_read_phi<S, R, XBC>, (unsigned)((n + PH_NT1 - 1) / PH_NT1), PH_NT1, 0,
                            L.stream, a, xbc_spec(L, L.step));
  }
  cudaError_t e = launch_phi<S, R, ODD, XBC>(L, a);
  if (e != cudaSuccess) return e;
  constexpr int NT = phase2_threads<R>();
  const int nwall = (L.nw + NT - 1) / NT;
  const int nedge = XBC ? (2 * L.ny * L.nz + NT - 1) / NT : 0;
  const long long grid = nwall + nedge + (L.N + NT - 1) / NT;
  return launch_dependent(k_read_cell<S, R, ODD, XBC>, (unsigned)grid, NT, 0, L.stream, a, nwall,
                          nedge);
}

template <class S, class R>
cudaError_t launch_read(Lattice &L, int field) {
  if (L.step & 1)
    return L.bc_on ? launch_read_t<S, R, true, true>(L, field)
                   : launch_read_t<S, R, true, false>(L, field);
  return L.bc_on ? launch_read_t<S, R, false, true>(L, field)
                 : launch_read_t<S, R, false, false>(L, field);
}

template <class S, class R>
cudaError_t mark_xbc(Lattice &L, bool on) {
  const int plane = L.ny * L.nz, T = 128;
  k_mark_xbc<<<(2 * plane + T - 1) / T, T, 0, L.stream>>>(L.flags, L.nx, plane, on ? 1 : 0);
  return cudaGetLastError();
}

template <class S, class R>
size_t batch_desc_bytes() { return sizeof(Args<S, R>); }

template <class S, class R>
void batch_build_descs(Lattice *const *lats, int n, char *host) {
  for (int l = 0; l < n; ++l) {
    for (int p = 0; p < 2; ++p) {
      Args<S, R> a = make_args<S, R>(*lats[l], p);
      a.batch = 1;
      a.diag = diag_acc(*lats[l], (int)(lats[l]->ndiag & 1));
      a.diag_zero = diag_acc(*lats[l], (int)((lats[l]->ndiag + 1) & 1));
      std::memcpy(host + (2 * (size_t)l + p) * sizeof(Args<S, R>), &a, sizeof a);
    }
  }
}

// One step of a group of lattices: both phases of all of them.
template <class S, class R, bool XBC>
static cudaError_t batch_launch_group(const BatchDev &b, const BatchGroup &g, int gi, bool diag,
                                      int tpar) {
  const Args<S, R> *d = (const Args<S, R> *)b.descs;
  const int4 *it1 = (const int4 *)b.items + g.first1, *it2 = (const int4 *)b.items + g.first2;
  int *bstep = b.bstep + gi;
  cudaError_t e = launch_dependent(k_batch_phase1<S, R, XBC>, (unsigned)g.n1, PH_NT1, 0, b.stream,
                                   d, b.par0, it1, b.xspecs, bstep, tpar);
  if (e != cudaSuccess) return e;
  if (diag)
    return launch_dependent(k_batch_phase2<S, R, true, XBC>, (unsigned)g.n2, phase2_threads<R>(), 0, b.stream, d,
                            b.par0, it2, bstep, tpar);
  return launch_dependent(k_batch_phase2<S, R, false, XBC>, (unsigned)g.n2, phase2_threads<R>(), 0, b.stream, d,
                          b.par0, it2, bstep, tpar);
}

template <class S, class R>
cudaError_t batch_launch_step(const BatchDev &b, const BatchGroup &g, int gi, bool diag,
                              int tpar) {
  return g.open ? batch_launch_group<S, R, true>(b, g, gi, diag, tpar)
                : batch_launch_group<S, R, false>(b, g, gi, diag, tpar);
}

template <class S, class R>
int batch_blocks_per_sm() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_phase2<S, R, false, false>,
                                                    phase2_threads<R>(),
                                                    0) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

#define PFLB_INSTANTIATE(S, R)                                                   \
  template int batch_blocks_per_sm<S, R>();                                      \
  template size_t batch_desc_bytes<S, R>();                                      \
  template void batch_build_descs<S, R>(Lattice *const *, int, char *);         \
  template cudaError_t batch_launch_step<S, R>(const BatchDev &, const BatchGroup &, int, bool, \
                                               int);                             \
  template cudaError_t launch_init<S, R>(Lattice &, const double *, double);     \
  template cudaError_t launch_step<S, R>(Lattice &, bool);                       \
  template cudaError_t launch_macro<S, R>(Lattice &);                            \
  template cudaError_t launch_read<S, R>(Lattice &, int);                        \
  template cudaError_t set_model<S, R>(Lattice &);                               \
  template int max_block_threads<S, R>();                                        \
  template int auto_lz<S, R>(const Lattice &);                                  \
  template cudaError_t mark_xbc<S, R>(Lattice &, bool);

}  // namespace pflb
