// pflb_phase.cuh -- the step as two kernels (arXiv 2512.01032, Sec. II and
// Sec. III A): phase 1 sums phi = sum_i h_i of every cell into the phi field
// (and forms the boundary states of open x planes); phase 2 updates every
// cell, its neighbours' phi read from that field.
//
// Against the pipelined march (pflb_pipe.cuh) this reads h twice (389 B per
// FP32 cell instead of 305) but computes each phi once instead of once per
// tile it touches, keeps nothing in shared memory, has no barrier, takes any
// extent and any boundary, and hides the wall nodes' chains of loads behind
// the bulk cells of the same launch.  Where h stays in L2 between the two
// kernels the second read costs no DRAM traffic.  Measured (GB300, us per
// step, against the march, or the fused kernel where that could not run):
// FP32 drop 32^3 6.1 (10.3), sessile 64^3 14.6 (32.4), slit 1024 x 64 x 4 14.9
// (31.7), constricted duct w = 48 29 (56), channel 251 x 67 x 67 87 (153), sessile
// 128^3 136 (152); BF16 sessile 128^3 109 (138); FP64 sessile 64^3 303 (516).
// What bounds it: at 128^3 FP32 phase 1 takes 28.7 us, the copy bandwidth, and
// phase 2 runs at 82 to 90 % of it; at 16-bit storage the latency of the loads
// (14 warps per SM) and 872 instructions per cell; at FP64 the FP64 rate; below
// 64^3 the two launches and, in thin lattices, a wall node's chain of
// instructions.
//
// A unit of work is one lane per cell: bulk cells by their linear index, wall
// nodes by their record, boundary cells by their place in the two planes.
#pragma once
#include "pflb_kernels.cuh"
#include "pflb_pipe.cuh"

namespace pflb {

constexpr int PH_NT1 = 128;  // threads of a phase-1 block
// Threads of a phase-2 block: blocks of two warps leave fewer slots idle at
// the end of a launch than blocks of four (128^3: 116.7 against 118.8 us), and
// than blocks of one (117.6 against 116.0 us BF16, 142.1 against 143.8 FP32).
// At FP64 an SM issues one warp's operation in 16 clocks, so the warps per SM
// should be even: blocks of one.
template <class R>
__host__ __device__ constexpr int phase2_threads() {
  return sizeof(R) == 8 ? 32 : 64;
}
// Phase-2 blocks per SM that the compiler is asked for.  7 and 8 both give a
// thread 128 registers (14 warps put four on a quarter of the SM), with which
// nearly all loads of a cell (19 phi, 19 g, 19 h) are in flight at once; spill
// stores are 0 to 8 bytes in even FP32 and BF16 steps, 68 to 92 in odd ones, 44
// to 280 with diagnostics.  Sessile 128^3, us per step at 6 / 7 / 8 / 9 blocks:
// FP32 154 / 142 / 142 / 150, BF16 134 / 109 / 113 / 112.
template <class R>
__host__ __device__ constexpr int phase2_blocks() {
  return sizeof(R) == 8 ? 8 : 7;
}

// Forms of the collision in phase 2: pair form without and with a body force
// (packed at FP32, lean at FP64), and the per-direction form.
enum { FORM_NOFORCE = 0, FORM_FORCE = 1, FORM_PLAIN = 2 };
// Lattices in FP32 arithmetic that the march's layout does not take (open x
// boundaries, nx not a multiple of 4) have always had the per-direction form
// and keep it, with k_fused's roundings (COLL_FIXED), so that their results
// stay the same to the bit: through the switch of the mobility correction
// (Eq. 4) one rounding can become 1e-3 of phi at an interface cell within tens
// of steps.  Packed pairs / per direction, us per step: FP32 channel 251 x 67 x
// 67 76 / 87, open duct 192 x 50 x 50 39 / 44; BF16 66 / 72 and 34.5 / 38.3,
// sessile 98^3 48.6 / 59.1; FP16 72 / 84, 36 / 42, 52 / 68.
template <class S>
__host__ __device__ constexpr int open_form() {
  return sizeof(S) <= 4 ? FORM_PLAIN : FORM_FORCE;
}

// The h of a cell as stored, where COLL_FIXED needs them (FP16, the only
// storage whose decoding rounds).
template <class S, class R>
__device__ __forceinline__ const R *raw_h(const Args<S, R> &a, int c, R raw[Q]) {
  if constexpr (Codec<S>::scaled) {
#pragma unroll
    for (int i = 13; i <= 17; ++i) raw[i] = Codec<S>::template to<R>(a.hin[i][c]);
    return raw;
  }
  return nullptr;
}

// g of bulk cell c (A-A), for the packed forms: every weight's product rounded
// by itself, as when the march read them from shared memory.
template <class S, class R, bool ODD>
__device__ __forceinline__ void gather_bulk(const Args<S, R> &a, int c, const Nbr &nb, R g[Q]) {
#pragma unroll
  for (int k = 0; k < Q; ++k)
    g[k] = dec_pop_rn<S, R>(ODD ? a.g[opp_of(k)][c + nb.off(opp_of(k))] : a.g[k][c], k);
}

// Diagnostic sums of one cell per lane over a warp, added to one of the copies
// of the accumulator: eight sums by a butterfly that halves the quantities a
// lane carries at each of its first three exchanges (9 shuffles in place of
// 40), no shared memory and no barrier, so that the update's blocks stay
// small.  Measured on sessile 64^3 FP32 (15 us per step without): 20.4 us with
// sums over a block through shared memory, 28 us with resident blocks that
// keep per-thread sums (their fixed shares of the cells wait for the wall
// nodes).
template <class R>
__device__ __forceinline__ void phase_diag(double *diag, const DiagAcc<R> &d) {
  constexpr unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  R v[8] = {d.v[D_MASS],   d.v[D_KIN],    d.v[D_PH],  d.v[D_PL],
            d.v[D_REGION], d.v[D_NHEAVY], d.v[D_NPH], d.v[D_NPL]};
#pragma unroll
  for (int half = 4; half >= 1; half >>= 1) {
    const int o = 4 * half;  // 16, 8, 4
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const R send = hi ? v[j] : v[j + half], keep = hi ? v[j + half] : v[j];
      v[j] = keep + __shfl_xor_sync(all, send, o);
    }
  }
  v[0] += __shfl_xor_sync(all, v[0], 2);
  v[0] += __shfl_xor_sync(all, v[0], 1);
  if ((lane & 3) == 0 && v[0] != R(0)) {
    const int q = lane >> 2;  // bit 2: lane & 16, bit 1: lane & 8, bit 0: lane & 4
    const int slot = q == 0 ? D_MASS : q == 1 ? D_KIN : q == 2 ? D_PH : q == 3 ? D_PL
                   : q == 4 ? D_REGION : q == 5 ? D_NHEAVY : q == 6 ? D_NPH : D_NPL;
    atomicAdd(diag + slot, (double)v[0]);
  }
  // largest |u|^2: non-negative, so its bits order as integers
  if constexpr (sizeof(R) == 4) {
    const unsigned m = __reduce_max_sync(all, __float_as_uint(d.umax));
    if (lane == 1 && m)
      atomicMax((unsigned long long *)(diag + D_UMAX),
                (unsigned long long)__double_as_longlong((double)__uint_as_float(m)));
  } else {
    R m = d.umax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(all, m, o));
    if (lane == 1 && m > R(0))
      atomicMax((unsigned long long *)(diag + D_UMAX),
                (unsigned long long)__double_as_longlong((double)m));
  }
  // the rest is rare: contact line, interface crossings, non-finite values
  if (!__any_sync(all, d.v[D_CLN] != R(0) || d.front > R(0) || d.rear > R(0) ||
                           d.v[D_NONFINITE] != R(0)))
    return;
#pragma unroll
  for (int k = D_CLN; k <= D_NONFINITE; ++k) {
    if (k == D_KIN) continue;
    const R s = warp_sum(d.v[k]);
    if (lane == 0 && s != R(0)) atomicAdd(diag + k, (double)s);
  }
  R fr = d.front, re = d.rear;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fr = fmax(fr, __shfl_xor_sync(all, fr, o));
    re = fmax(re, __shfl_xor_sync(all, re, o));
  }
  if (lane < 2 && (lane ? re : fr) > R(0))
    atomicMax((unsigned long long *)(diag + (lane ? D_REAR : D_FRONT)),
              (unsigned long long)__double_as_longlong((double)(lane ? re : fr)));
}

// Dependent launches: a block lets the next kernel of the stream be set up
// at once, and itself waits here until the one before has finished.  So a
// block exists while the kernel before still writes phi, h, g or the
// diagnostic copies, and the read-only path (the read-only load intrinsic,
// ld_ro, restrict pointers to const) is only for memory that stays the same
// for as long as the kernel exists: every kernel that waits here, and every
// function that it calls, uses ordinary loads, which stay behind the wait.
__device__ __forceinline__ void launch_ready() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// phi of an open-boundary cell at plane x (reading R22), as xbc_cell forms it.
template <class S, class R>
__device__ __forceinline__ R edge_phi(const Args<S, R> &a, const XbcSpec &sp, int c, int x,
                                      long long t) {
  const int side = x == 0 ? 0 : 1;
  if (sp.type[side] != 1) return (R)xbc_value(sp, side, 4, t);
  const int ca = side ? c - 1 : c + 1;
  if (a.flags[ca] & F_SOLID) return R(0);
  R h[Q], s = R(0);
  ld_h_cell<S, R>(a.hin, ca, h);
#pragma unroll
  for (int i = 0; i < Q; ++i) s += h[i];
  return s;
}

// phi of the V cells from c on, summed in cell_phi's order: with V > 1 by
// 16-byte loads (c and the number of cells are multiples of V then, so every
// direction's address is aligned).  f returns the flags.
template <class S, class R, bool XBC, int V>
__device__ __forceinline__ void phi_cells(const Args<S, R> &a, const XbcSpec &sp, int c,
                                          long long t, R s[V], uint8_t f[V]) {
  if constexpr (V == 1) {
    R h[Q];
    f[0] = a.flags[c];
    ld_h_cell<S, R>(a.hin, c, h);
    s[0] = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) s[0] += h[i];
  } else {
    uint4 q[h_slots<S>()];
#pragma unroll
    for (int i = 0; i < h_slots<S>(); ++i)
      q[i] = *reinterpret_cast<const uint4 *>(a.hin[i] + c);
    if constexpr (V == 8) {
      const uint2 w = *reinterpret_cast<const uint2 *>(a.flags + c);
      memcpy(f, &w, 8);
    } else if constexpr (V == 4) {
      const uint32_t w = *reinterpret_cast<const uint32_t *>(a.flags + c);
      memcpy(f, &w, 4);
    } else {
      const uint16_t w = *reinterpret_cast<const uint16_t *>(a.flags + c);
      memcpy(f, &w, 2);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      S v[V], lo[V];
      memcpy(v, &q[i], 16);
      if constexpr (Codec<S>::narrow) memcpy(lo, &q[Q], 16);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        R d = dec_pop<S, R>(v[j], i);
        if constexpr (Codec<S>::narrow)
          if (i == 0) d += dec_pop<S, R>(lo[j], 0);
        s[j] = i == 0 ? d : s[j] + d;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (f[j] & F_SOLID) s[j] = R(0);
    if constexpr (XBC)
      if (f[j] & F_BC) s[j] = edge_phi<S, R>(a, sp, c + j, c + j - div_by(c + j, a.dx) * a.nx, t);
  }
}

template <class S, class R, bool XBC, int V>
__device__ __forceinline__ void phase1_cells(const Args<S, R> &a, const XbcSpec &sp, int c,
                                             long long t) {
  R s[V];
  uint8_t f[V];
  phi_cells<S, R, XBC, V>(a, sp, c, t, s, f);
  R *out = a.phi_w + c;
  if constexpr (V == 1) {
    *out = s[0];
  } else if constexpr (sizeof(R) == 8) {
    *reinterpret_cast<double2 *>(out) = make_double2(s[0], s[1]);
  } else {
#pragma unroll
    for (int j = 0; j < V; j += 4)
      *reinterpret_cast<float4 *>(out + j) = make_float4(s[j], s[j + 1], s[j + 2], s[j + 3]);
  }
}

// Phase 1 of cells [c0, c0 + n), by PH_NT1 threads.
template <class S, class R, bool XBC>
__device__ __forceinline__ void phase1_range(const Args<S, R> &a, const XbcSpec &sp, int c0, int n,
                                             bool vec, long long t) {
  constexpr int V = 16 / (int)sizeof(S);
  const unsigned end = (unsigned)c0 + n;
  if (vec) {
    for (unsigned c = c0 + threadIdx.x * V; c < end; c += PH_NT1 * V)
      phase1_cells<S, R, XBC, V>(a, sp, (int)c, t);
  } else {
    for (unsigned c = c0 + threadIdx.x; c < end; c += PH_NT1)
      phase1_cells<S, R, XBC, 1>(a, sp, (int)c, t);
  }
}

// Whether phase 1 may take 16 bytes per load.
template <class S>
__host__ __device__ inline bool phase1_vec(long long N) {
  return N % (16 / (int)sizeof(S)) == 0;
}

// Phase 2 of wall node rec.  Everything the update reads is loaded in two
// rounds of independent loads (the record, then what it indexes): a source
// across a solid link is chosen by address, not by branch.  A chain of
// conditional loads took 14 us per launch whatever the number of nodes.
template <class S, class R, bool ODD, int MODE, bool DIAG, bool XBC, int PAIRS>
__device__ __forceinline__ void wall_update(const Args<S, R> &a, int rec, DiagAcc<R> &acc) {
  const int nw = a.nw;
  const int c = a.wcell[rec];
  const uint32_t lm = a.wmask[rec];
#pragma unroll
  for (int k = 0; k < 5; ++k) prefetch_l1(a.wgeo + (k * nw + rec));
  const uint8_t f = a.flags[c];
  if constexpr (XBC)
    if (f & F_BC) return;
  const int z = div_by(c, a.dxy), r = c - z * (a.nx * a.ny), y = div_by(r, a.dx), x = r - y * a.nx;
  Nbr nb;
  nb.init(x, y, z, a.nx, a.ny, a.nz);
  R h[Q], g[Q], val[Q];
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const R *p = ((lm >> i) & 1u) ? a.ghost + ((i - 1) * nw + rec) : a.phi + (c + nb.off(i));
    val[i] = *p;
  }
  ld_h_cell<S, R>(a.hin, c, h);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const S *p = ODD ? a.g[opp_of(k)] + (c + nb.off(opp_of(k))) : a.g[k] + c;
    if (k != 0 && ((lm >> opp_of(k)) & 1u)) p = a.wp_rd + ((k - 1) * nw + rec);
    g[k] = ld_g<S, R>(p, k);
  }
  R phi = R(0), raw[Q];
  const R *hraw = nullptr;
  if constexpr (PAIRS == COLL_FIXED) {
    phi = a.phi[c];  // (as k_fused: the sum that the neighbours see)
    hraw = raw_h<S, R>(a, c, raw);
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) phi += h[i];
  }
  finish_cell<S, R, ODD, MODE, DIAG, false, PAIRS, true>(a, x, y, z, c, f, lm, rec, nb, h, g, phi,
                                                        val, acc, hraw);
}

// Phase 2 of a warp's wall nodes (every lane calls it; on: it has a record).
template <class S, class R, bool ODD, bool DIAG, bool XBC, int FORM>
__device__ __forceinline__ void phase2_wall(const Args<S, R> &a, int rec, bool on) {
  DiagAcc<R> acc;
  acc.zero();
  if (on)
    wall_update<S, R, ODD, MODE_STEP, DIAG, XBC, FORM == FORM_PLAIN ? COLL_FIXED : COLL_X2>(
        a, rec, acc);
  if (DIAG) phase_diag<R>(diag_copy(a.diag), acc);
}

// Phase 2 of boundary cell j (plane x = 0, then plane x = nx - 1).
template <class S, class R, bool ODD, int MODE = MODE_STEP>
__device__ __forceinline__ void phase2_edge(const Args<S, R> &a, int j) {
  const int plane = a.ny * a.nz, side = j >= plane, yz = j - side * plane;
  const int x = side ? a.nx - 1 : 0, y = yz % a.ny, z = yz / a.ny, c = x + a.nx * yz;
  const uint8_t f = a.flags[c];
  if (f & F_SOLID) return;
  Nbr nb;
  nb.init(x, y, z, a.nx, a.ny, a.nz);
  const int rec = (f & F_WALL) ? a.widx[c] : 0;
  const uint32_t lm = (f & F_WALL) ? a.wmask[rec] : 0u;
  boundary_cell<S, R, ODD, MODE>(a, x, y, z, c, lm, rec, nb);
}

// Phase 2 of bulk cell c (nothing for solid cells, wall nodes and boundary
// cells, which have units of their own).  All loads are issued before the
// flags decide, so that a warp waits for memory once (BF16 sessile 128^3:
// 112.6 against 117.6 us per step).  Every lane of the warp calls it, those
// past the last cell too.
template <class S, class R, bool ODD, bool DIAG, bool XBC, int FORM>
__device__ __forceinline__ void phase2_bulk(const Args<S, R> &a, unsigned cell) {
  // FP32 without diagnostics keeps the lanes of a warp together between the
  // fields and the update (sessile 128^3: 137 us per step against 142); at
  // 16-bit storage one branch is faster (109 against 119).  With diagnostics
  // the sums over the warp come last: at BF16 that is faster (127 us against
  // 131 with them before the update); at FP32 it is slower (154 against 146)
  // but leaves the update's contractions, and so the fields, as they are
  // without diagnostics and in the march.
  constexpr bool PLAIN = FORM == FORM_PLAIN;
  constexpr bool MID = sizeof(S) > 2 && !DIAG && !PLAIN;
  bool on = cell < (unsigned)a.N;
  if (!MID && !DIAG && !on) return;
  const int c = on ? (int)cell : 0;
  const int z = div_by(c, a.dxy), r = c - z * (a.nx * a.ny), y = div_by(r, a.dx), x = r - y * a.nx;
  const Model<R> &m = a.m;
  Nbr nb;
  nb.init(x, y, z, a.nx, a.ny, a.nz);
  R h[Q], g[Q], val[Q], gx, gy, gz, lap;
  Macro<R> mc;
  auto load = [&] {
    const uint8_t f = a.flags[c];
    val[0] = a.phi[c];
#pragma unroll
    for (int i = 1; i < Q; ++i) val[i] = a.phi[c + nb.off(i)];
    if constexpr (PLAIN)
      gather_g<S, R, ODD>(a, c, 0u, 0, nb, g);
    else
      gather_bulk<S, R, ODD>(a, c, nb, g);
    ld_h_cell<S, R>(a.hin, c, h);
    return !(f & (F_SOLID | F_WALL | (XBC ? F_BC : 0)));
  };
  auto fields = [&] {
    if constexpr (std::is_same<R, float>::value) {
      cd_stencil_x2(val, gx, gy, gz, lap);
      mc = macros_x2(m, g, val[0], gx, gy, gz, lap);
    } else {
      cd_stencil(val, gx, gy, gz, lap);
      mc = macros(m, g, val[0], gx, gy, gz, lap);
    }
  };
  auto update = [&] {
    if constexpr (std::is_same<R, float>::value)
      collide_pairs_x2<FORM == FORM_FORCE>(m, h, g, mc, val[0], gx, gy, gz, lap);
    else
      collide_pairs_lean<R, FORM == FORM_FORCE>(m, h, g, mc, val[0], gx, gy, gz, lap);
    store_cell<S, R, ODD>(a, c, 0u, 0, nb, h, g, val, false);
  };
  DiagAcc<R> acc;
  acc.zero();
  auto sums = [&] { diag_cell<S, R>(a, x, y, z, false, 0u, val[0], val[1], mc, acc); };
  if constexpr (MID) {
    if (on) on = load();
    if (on) fields();
    if (on) update();
  } else {
    if constexpr (PLAIN) {
      // finish_cell with the flags as read, not as known to have no F_WALL:
      // the sums that its wall corrections add to then stay uncontracted, as
      // in every build of this form (see open_form)
      if (on && load()) {
        R raw[Q];
        finish_cell<S, R, ODD, MODE_STEP, DIAG, XBC, COLL_FIXED>(
            a, x, y, z, c, a.flags[c], 0u, 0, nb, h, g, val[0], val, acc, raw_h<S, R>(a, c, raw));
      }
    } else if (on && load()) {
      fields();
      if (DIAG) sums();
      update();
    }
    if (DIAG) phase_diag<R>(diag_copy(a.diag), acc);
  }
}

// ------------------------------------------------------- one lattice
// Blocks below nstate form boundary states; the others take phi cells.
template <class S, class R, bool ODD, bool XBC>
__global__ void __launch_bounds__(PH_NT1)
    k_phase1(const __grid_constant__ Args<S, R> a, const __grid_constant__ XbcSpec sp, int nstate) {
  launch_ready();
  int b = blockIdx.x;
  if constexpr (XBC) {
    if (b < nstate) {
      const int j = b * PH_NT1 + threadIdx.x;
      if (j < 2 * a.ny * a.nz) xbc_cell<S, R, ODD>(a, sp, a.bcm, j, sp.step0);
      return;
    }
    b -= nstate;
  }
  const bool vec = phase1_vec<S>(a.N);
  const int per = PH_NT1 * (vec ? 16 / (int)sizeof(S) : 1), c0 = b * per;
  phase1_range<S, R, XBC>(a, sp, c0, min(per, a.N - c0), vec, sp.step0);
}

// Blocks of wall nodes, boundary cells or bulk cells, in that order (the
// wall nodes' loads take longest).  The bulk cells are taken from the last to
// the first: phase 1 read the last ones' h most recently, and the next phase
// 1 begins with the h written last (144^3 FP32: 201 instead of 210 us, BF16
// 166 instead of 172).
template <class S, class R, bool ODD, bool DIAG, bool XBC, int FORM>
__global__ void __launch_bounds__(phase2_threads<R>(), phase2_blocks<R>())
    k_phase2(const __grid_constant__ Args<S, R> a, int nwall, int nedge) {
  constexpr int NT = phase2_threads<R>();
  launch_ready();
  if (DIAG) zero_next_diag(a);
  const int u = blockIdx.x;
  if (u < nwall) {
    const int rec = u * NT + threadIdx.x;
    phase2_wall<S, R, ODD, DIAG, XBC, FORM>(a, rec, rec < a.nw);
  } else if (XBC && u < nwall + nedge) {
    const int j = (u - nwall) * NT + threadIdx.x;
    if (j < 2 * a.ny * a.nz) phase2_edge<S, R, ODD>(a, j);
  } else {
    phase2_bulk<S, R, ODD, DIAG, XBC, FORM>(a, (gridDim.x - 1 - u) * NT + threadIdx.x);
  }
}

// ------------------------------------------------------- field reads
// phi or rho of every cell straight from the h populations, as doubles (zero
// on solid cells): one pass over h, bound by its 76 + 8 bytes per FP32 cell.
template <class S, class R, bool XBC, int V>
__device__ __forceinline__ void read_cells(const Args<S, R> &a, const XbcSpec &sp, int c) {
  R s[V];
  uint8_t f[V];
  phi_cells<S, R, XBC, V>(a, sp, c, sp.step0, s, f);
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const double v = (double)(a.field == 0 ? s[j] : a.m.rho_L + s[j] * a.m.rho_dif);
    a.out[c + j] = (f[j] & F_SOLID) ? 0.0 : v;
  }
}
template <class S, class R, bool XBC>
__global__ void __launch_bounds__(PH_NT1)
    k_read_phi(const __grid_constant__ Args<S, R> a, const __grid_constant__ XbcSpec sp) {
  constexpr int V = 16 / (int)sizeof(S);
  launch_ready();
  const long long i = (long long)blockIdx.x * PH_NT1 + threadIdx.x;
  if (phase1_vec<S>(a.N)) {
    if (i * V < a.N) read_cells<S, R, XBC, V>(a, sp, (int)(i * V));
  } else if (i < a.N) {
    read_cells<S, R, XBC, 1>(a, sp, (int)i);
  }
}

// P or a velocity component of every cell, after phase 1: the units of phase
// 2, without the step.
template <class S, class R, bool ODD, bool XBC>
__global__ void __launch_bounds__(phase2_threads<R>())
    k_read_cell(const __grid_constant__ Args<S, R> a, int nwall, int nedge) {
  constexpr int NT = phase2_threads<R>();
  launch_ready();
  const unsigned u = blockIdx.x;
  if (u < (unsigned)nwall) {
    const int rec = u * NT + threadIdx.x;
    DiagAcc<R> acc;
    if (rec < a.nw) wall_update<S, R, ODD, MODE_MACRO, false, XBC, COLL_PLAIN>(a, rec, acc);
  } else if (XBC && u < (unsigned)(nwall + nedge)) {
    const int j = (u - nwall) * NT + threadIdx.x;
    if (j < 2 * a.ny * a.nz) phase2_edge<S, R, ODD, MODE_MACRO>(a, j);
  } else {
    const unsigned cell = (u - nwall - nedge) * NT + threadIdx.x;
    if (cell >= (unsigned)a.N) return;
    const int c = (int)cell;
    const uint8_t f = a.flags[c];
    if (f & (F_WALL | (XBC ? F_BC : 0))) return;
    if (f & F_SOLID) {
      a.out[c] = 0.0;
      return;
    }
    const int z = div_by(c, a.dxy), r = c - z * (a.nx * a.ny), y = div_by(r, a.dx),
              x = r - y * a.nx;
    Nbr nb;
    nb.init(x, y, z, a.nx, a.ny, a.nz);
    R g[Q], val[Q], gx, gy, gz, lap;
    val[0] = a.phi[c];
#pragma unroll
    for (int i = 1; i < Q; ++i) val[i] = a.phi[c + nb.off(i)];
    gather_g<S, R, ODD>(a, c, 0u, 0, nb, g);
    cd_stencil(val, gx, gy, gz, lap);
    const Macro<R> mc = macros(a.m, g, val[0], gx, gy, gz, lap);
    a.out[c] = field_of(a.field, val[0], mc.rho, mc.P, mc.ux, mc.uy, mc.uz);
  }
}

// ------------------------------------------------------ many lattices
// Items (lattice, kind, first, count), one per block.  The block copies the
// lattice's step descriptor for its A-A parity at this step into shared
// memory.  A lattice's cells see exactly the arithmetic that they see in a
// batch of their own.
enum { PHI_CELLS = 0, PHI_STATES = 1, UPD_BULK = 2, UPD_WALL = 3, UPD_EDGE = 4 };

template <class S, class R>
__device__ __forceinline__ const Args<S, R> &batch_args(unsigned char *smem,
                                                        const Args<S, R> *descs, int l, int p) {
  const int *src = reinterpret_cast<const int *>(descs + 2 * l + p);
  int *dst = reinterpret_cast<int *>(smem);
  for (int k = threadIdx.x; k < (int)(sizeof(Args<S, R>) / 4); k += blockDim.x) dst[k] = src[k];
  __syncthreads();
  return *reinterpret_cast<const Args<S, R> *>(smem);
}

// tpar: parity of the batch step; bstep: batch steps since the call began
// (boundary ramps), advanced by phase 2.
template <class S, class R, bool XBC>
__global__ void __launch_bounds__(PH_NT1)
    k_batch_phase1(const Args<S, R> *descs, const int *par0, const int4 *items,
                   const XbcSpec *specs, const int *bstep, int tpar) {
  __shared__ __align__(16) unsigned char smem[sizeof(Args<S, R>)];
  launch_ready();
  const int4 it = items[blockIdx.x];
  const int p = (par0[it.x] + tpar) & 1;
  const Args<S, R> &a = batch_args<S, R>(smem, descs, it.x, p);
  const XbcSpec &sp = specs[it.x];
  const long long t = XBC ? sp.step0 + *bstep : 0;
  if (it.y == PHI_CELLS) {
    phase1_range<S, R, XBC>(a, sp, it.z, it.w, phase1_vec<S>(a.N), t);
  } else if constexpr (XBC) {
    for (int j = it.z + (int)threadIdx.x; j < it.z + it.w; j += PH_NT1) {
      if (p)
        xbc_cell<S, R, true>(a, sp, a.bcm, j, t);
      else
        xbc_cell<S, R, false>(a, sp, a.bcm, j, t);
    }
  }
}

template <class S, class R, bool ODD, bool DIAG, bool XBC, int FORM>
__device__ __forceinline__ void batch_update(const Args<S, R> &a, const int4 &it) {
  for (int j0 = it.z; j0 < it.z + it.w; j0 += phase2_threads<R>()) {
    const int j = j0 + (int)threadIdx.x;
    // (an item of bulk cells ends at the lattice's last cell or at a multiple
    // of the block)
    if (it.y == UPD_BULK)
      phase2_bulk<S, R, ODD, DIAG, XBC, FORM>(a, j);
    else if (it.y == UPD_WALL)
      phase2_wall<S, R, ODD, DIAG, XBC, FORM>(a, j, j < it.z + it.w);
    else if (XBC && j < it.z + it.w)
      phase2_edge<S, R, ODD>(a, j);
  }
}

template <class S, class R, bool DIAG, bool XBC>
__global__ void __launch_bounds__(phase2_threads<R>(), phase2_blocks<R>())
    k_batch_phase2(const Args<S, R> *descs, const int *par0, const int4 *items, int *bstep,
                   int tpar) {
  __shared__ __align__(16) unsigned char smem[sizeof(Args<S, R>)];
  launch_ready();
  const int4 it = items[blockIdx.x];
  const int p = (par0[it.x] + tpar) & 1;
  const Args<S, R> &a = batch_args<S, R>(smem, descs, it.x, p);
  if (blockIdx.x == 0 && threadIdx.x == 0) *bstep += 1;
  // the first item of a lattice's bulk cells zeroes its next accumulator
  if (DIAG && it.y == UPD_BULK && it.z == 0) zero_diag(a.diag_zero);
  constexpr int FORM = XBC ? open_form<S>() : FORM_FORCE;
  if (!XBC && open_form<S>() == FORM_PLAIN && a.plain) {
    if (p)
      batch_update<S, R, true, DIAG, XBC, open_form<S>()>(a, it);
    else
      batch_update<S, R, false, DIAG, XBC, open_form<S>()>(a, it);
    return;
  }
  if (p)
    batch_update<S, R, true, DIAG, XBC, FORM>(a, it);
  else
    batch_update<S, R, false, DIAG, XBC, FORM>(a, it);
}

// Sum of the copies of an accumulator and the device error flag, as the record
// that a diagnostics read returns (256 threads).  out may be page-locked host
// memory: a synchronous read is then this kernel and a wait, without copies.
static __global__ void k_diag_fold(const double *copies, const int *err, int64_t step,
                                   pflb_diag_raw_t *out) {
  __shared__ double part[8][32];
  launch_ready();
  const int k = threadIdx.x & 31, w = threadIdx.x >> 5;
  double t = 0.0;
#pragma unroll 8
  for (int c = w; c < kDiagCopies; c += 8) {
    const double v = copies[32 * c + k];
    t = k >= D_UMAX ? fmax(t, v) : t + v;
  }
  part[w][k] = t;
  __syncthreads();
  if (w) return;
  for (int j = 1; j < 8; ++j) t = k >= D_UMAX ? fmax(t, part[j][k]) : t + part[j][k];
  out->acc[k] = k == D_UMAX ? sqrt(t) : t;  // accumulated as |u|^2
  if (k == 0) {
    out->step = step;
    out->err = *err;
    out->pad = 0;
  }
}

}  // namespace pflb
