// bcm_mg.cu -- geometric multigrid V-cycle, the preconditioner M^-1 of the pressure PCG
// (Eq. poisson; the paper solves the pressure equation with a multigrid on its cubes).
//
// Grids of one or two levels.  Per-cube levels l = 0 .. L coarsen every cube by two per
// level (B, B/2, ..., 1 cells per edge); a level-l+1 cell covers 2x2x2 cells of level l
// of the same cube.  Above level L (one cell per cube) the eight refined cubes of each
// level-0 position first join into one node, then the nodes of a sim are aggregated by
// their level-0 cube coordinates shifted right by m (m = 1 .. M).  Transfers are
// piecewise constant, restriction sums, and the coarse operators are the Galerkin
// products P^T K P.  For the flux-form K these are again flux-form operators: on
// per-cube level l a face carries 4^l fine faces, coefficient 4^l h of its cube, an
// outflow face twice that on the diagonal, other domain faces nothing, and a 2:1 face
// keeps the form of R7 (a coarse face cell against the four fine cells that touch it,
// weight 4/3 on the coarse side and 2/3 on the fine side, since the 2x2x2 aggregates on
// both sides keep the coarse cell / four fine cells pairing); the aggregate levels keep
// their Galerkin sums as small CSR tables built on the host.  The smoother is damped Jacobi
// S = omega D^-1 (omega = 0.8), one sweep before and one after the coarse correction,
// which is scaled by s = 1.75 (piecewise-constant transfers leave it too weak), so the
// V-cycle is symmetric positive definite and M^-1 suits CG:
//   V_l(r) = x + S (r - K x),  x = S r + s P V_{l+1}(P^T (r - K S r)),
//   V_top(r) = four damped-Jacobi sweeps from zero.
//
// Launches per V-cycle: the levels of 16^3 and 8^3 cells per cube on quad tiles
// (bcm_quad.cuh), the 4^3 and 2^3 levels of larger grids with a thread per cell, the rest
// down to one node per sim and back up in one launch of a cluster, and after the finest up
// launch the PCG's decisions (beta, convergence).  After pass A the finest down launch also
// does the PCG's pass B.
//
// What bounds it: the finest level moves 49 bytes a cell and iteration in FP32 (pass A 16,
// down with pass B 24.5, up 8.5; 60 before, when x = S r was stored and read).  On 83M cells
// (two levels) the three launches take 282, 416 and 280 us, 4.7, 4.9 and 2.5 TB/s (427, 470
// and 410 us with padded tiles); on 4.2M cells 20, 26 and 19 us (31, 31, 39).  In FP64
// they are bound by the FP64 pipe: 122, 160 and 144 us (138, 192, 151).  Below the finest
// level it is latency: 7 launches, 63 us serialised at 1024 cubes, where there were 9 in 80.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bcm_cube.cuh"
#include "bcm_internal.cuh"
#include "bcm_kernels.h"
#include "bcm_persist.cuh"
#include "bcm_quad.cuh"

namespace bcm {

template <int BL>
__device__ __forceinline__ int lcell(int i, int j, int k) { return (k * BL + j) * BL + i; }

// Per-sim constants of a level in the vector type: the FP32 path does no FP64
// arithmetic (FP64 runs at a small fraction of the FP32 rate on this GPU).
template <class TV>
__device__ __forceinline__ TV sim_inv(const SimParams& sp, int lvl, int s3);
template <>
__device__ __forceinline__ float sim_inv<float>(const SimParams& sp, int lvl, int s3) {
  return sp.invdiag32[lvl][s3];
}
template <>
__device__ __forceinline__ double sim_inv<double>(const SimParams& sp, int lvl, int s3) {
  return sp.invdiag[lvl][s3];
}
template <class TV>
__device__ __forceinline__ TV sim_h(const SimParams& sp);
template <>
__device__ __forceinline__ float sim_h<float>(const SimParams& sp) { return sp.h032; }
template <>
__device__ __forceinline__ double sim_h<double>(const SimParams& sp) { return sp.h0; }
// cell size of cube c (its refinement level halves the sim's level-0 size)
template <class TV>
__device__ __forceinline__ TV cube_h(const DevGrid& g, const SimParams& sp, int c) {
  return g.lvl[c] ? TV(0.5) * sim_h<TV>(sp) : sim_h<TV>(sp);
}

// The value across face f of cell (i, j, k) of cube c on per-cube level l (BL cells per
// edge) and the weight w of that face in the level's flux-form operator, whose
// coefficient 4^l h the caller carries (R7 on the coarser cells; the Galerkin product of
// the finer level keeps that form): a cell of this cube or of a same-level neighbour
// (w = 1), a domain ghost (w = 1; the cell itself, or minus it at an outflow face), the
// coarse cell across a 2:1 face (w = 2/3), or the mean of the four fine cells across it
// (w = 4/3).  val(cube, i, j, k) is a cell's value, xc this cell's.
template <int BL, class TV, class Val>
__device__ __forceinline__ TV mg_across(const DevGrid& g, int c, int l, int i, int j, int k,
                                        int f, TV xc, const Val& val, TV& w) {
  const int d = f >> 1, side = f & 1;
  int q[3] = {i, j, k};
  q[d] += side ? 1 : -1;
  w = TV(1);
  if (q[d] >= 0 && q[d] < BL) return val(c, q[0], q[1], q[2]);
  const int n = checked_nb(g, g.nb[6 * c + f]);
  if (n >= 0) {
    q[d] = side ? 0 : BL - 1;
    return val(n, q[0], q[1], q[2]);
  }
  if (n == NB_BOUNDARY) return g.sp[g.sim[c]].bc[f] == BC_OUTFLOW ? -xc : xc;
  const int t1 = tan1(d), t2 = tan2(d);
  const int a = t1 == 0 ? i : (t1 == 1 ? j : k), b = t2 == 0 ? i : (t2 == 1 ? j : k);
  int r3[3];
  r3[d] = side ? 0 : BL - 1;  // the cells across lie on the neighbour's facing layer
  if (n == NB_COARSE) {
    w = TV(2.0 / 3.0);
    const int C = g.aux[(6 * c + f) * 4];
    if (!bcm_expect(g, C >= 0 && C < g.n_cubes, CHK_AUX)) return xc;
    // corner coordinates in finest-cell units; a level-l cell spans 2^l level-0 cells
    const int sf = (1 << (g.max_level - g.lvl[c])) << l;
    const int sc = (1 << (g.max_level - g.lvl[C])) << l;
    r3[t1] = (g.ijk[3 * c + t1] + a * sf - g.ijk[3 * C + t1]) / sc;
    r3[t2] = (g.ijk[3 * c + t2] + b * sf - g.ijk[3 * C + t2]) / sc;
    if (!bcm_expect(g, r3[t1] >= 0 && r3[t1] < BL && r3[t2] >= 0 && r3[t2] < BL, CHK_CELL))
      return xc;
    return val(C, r3[0], r3[1], r3[2]);
  }
  w = TV(4.0 / 3.0);  // NB_FINE: the four fine cells that touch this coarse cell's face
  TV sum = TV(0);
#pragma unroll
  for (int bb = 0; bb < 2; ++bb)
#pragma unroll
    for (int aa = 0; aa < 2; ++aa) {
      const int ta = 2 * a + aa, tb = 2 * b + bb, qa = ta / BL, qb = tb / BL;
      const int F = g.aux[(6 * c + f) * 4 + qb * 2 + qa];
      if (!bcm_expect(g, F >= 0 && F < g.n_cubes && qa < 2 && qb < 2, CHK_AUX)) return xc;
      r3[t1] = ta - qa * BL;
      r3[t2] = tb - qb * BL;
      sum += val(F, r3[0], r3[1], r3[2]);
    }
  return TV(0.25) * sum;
}

// The sum over the six faces of w (xc - value across) for cell (i, j, k) of cube c, with every
// load of the cell in flight before the first use: the six face entries, then the six
// values at(cube, cell).  (Face by face, each behind its own branch, they are twelve
// dependent round trips: 4-9k cycles a level however few the cells.)  2:1 faces go through
// mg_across.
template <int BL, class TV, class At>
__device__ __forceinline__ TV mg_faces(const DevGrid& g, int c, int l, int i, int j, int k, TV xc,
                                       const At& at) {
  int nb[6];
#pragma unroll
  for (int f = 0; f < 6; ++f) nb[f] = checked_nb(g, g.nb[6 * c + f]);
  TV v[6];
  unsigned edge = 0u;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    int q[3] = {i, j, k};
    const int d = f >> 1, side = f & 1, o = q[d];
    const bool out = side ? o == BL - 1 : o == 0;
    if (out) edge |= 1u << f;
    const bool other = out && nb[f] >= 0;
    q[d] = out ? (other ? (side ? 0 : BL - 1) : o) : (side ? o + 1 : o - 1);
    v[f] = at(other ? nb[f] : c, lcell<BL>(q[0], q[1], q[2]));
  }
  TV acc = TV(0);
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    TV w = TV(1);
    if ((edge >> f & 1u) && nb[f] < 0) {
      if (nb[f] == NB_BOUNDARY) {
        v[f] = g.sp[g.sim[c]].bc[f] == BC_OUTFLOW ? -xc : xc;
      } else {
        auto val = [&](int cube, int a, int b, int e) { return at(cube, lcell<BL>(a, b, e)); };
        v[f] = mg_across<BL, TV>(g, c, l, i, j, k, f, xc, val, w);
      }
    }
    acc += w * (xc - v[f]);
  }
  return acc;
}

// omega / diag(K_l) of cell (i, j, k) of cube c on per-cube level l (BL cells per edge):
// diag(K_l) = 4^l diag(K) of a fine cell with the same boundary faces; wscale =
// omega / 4^l.  Neighbouring cubes belong to the same sim, so sp serves them too.
template <int BL, class TV>
__device__ __forceinline__ TV smooth_w(const DevGrid& g, const SimParams& sp, int c, int i, int j,
                                       int k, TV wscale) {
  return wscale * sim_inv<TV>(sp, g.lvl[c], s3_of<BL>(g.w3 + 6 * c, i, j, k));
}

// ---- down: x = S r, rr = r - K x, restriction of rr (P^T: sums), on levels of 4^3 and 2^3
// cells per cube that are too large for the coarse kernel below.
// One thread per fine cell: the eight children of a coarse cell are eight consecutive
// threads of one warp (child bits in the low three bits of the thread index), so the
// restriction is a three-step shuffle sum.  Threads of finished sims and of the tail take
// part in the shuffles with zeros.
// GIVEN: x = S r was formed by the finer level's launch, which knows each coarse cell once,
// where its six neighbours would each form it again (a launch of this kernel spends most
// of its instructions on that); else (the finest level of 4^3 cubes) it is formed here and
// stored.  The launch forms the next level's x the same way.
template <int BL, class TV>
__device__ __forceinline__ TV next_x(const DevGrid& g, const SimParams& sp, int c, int I, int J,
                                     int K, TV wscale, TV rc) {
  constexpr int CB = BL / 2;
  return smooth_w<CB, TV>(g, sp, c, I, J, K, TV(0.25) * wscale) * rc;
}
template <int BL, class TV, bool GIVEN>
__global__ __launch_bounds__(256) void k_mg_down_cell(DevGrid g, int l, TV wscale, TV cscale,
                                                      const TV* __restrict__ r,
                                                      TV* __restrict__ x, TV* __restrict__ rc,
                                                      TV* __restrict__ xn, int all) {
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  static_assert(BL >= 2, "restriction over 2x2x2 children");
  constexpr int CB = BL / 2, C3 = CB * CB * CB, B3 = BL * BL * BL;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long total = (long long)g.n_cubes * B3;
  const int c = (int)(t / B3), q = (int)(t - (long long)c * B3);
  const int d = q & 7, ci = q >> 3;
  const int I = ci % CB, J = (ci / CB) % CB, Kc = ci / (CB * CB);
  const bool on = t < total && (all || !g.ss[g.sim[c]].done);
  TV val = TV(0);
  if (on) {
    const int i = 2 * I + (d & 1), j = 2 * J + ((d >> 1) & 1), k = 2 * Kc + (d >> 2);
    const SimParams& sp = g.sp[g.sim[c]];
    const TV coef = cube_h<TV>(g, sp, c) * cscale;
    const size_t gi = (size_t)c * B3 + lcell<BL>(i, j, k);
    const TV rv = r[gi];
    auto sval = [&](int cube, int cell) {
      const size_t gn = (size_t)cube * B3 + cell;
      if constexpr (GIVEN) return x[gn];
      else
        return smooth_w<BL, TV>(g, sp, cube, cell % BL, (cell / BL) % BL, cell / (BL * BL), wscale) *
               r[gn];
    };
    const TV xc = sval(c, lcell<BL>(i, j, k));
    const TV acc = mg_faces<BL, TV>(g, c, l, i, j, k, xc, sval);
    if constexpr (!GIVEN) x[gi] = xc;
    val = rv - coef * acc;
  }
  val += __shfl_xor_sync(0xffffffffu, val, 1);
  val += __shfl_xor_sync(0xffffffffu, val, 2);
  val += __shfl_xor_sync(0xffffffffu, val, 4);
  if (d == 0 && on) {
    rc[(size_t)c * C3 + ci] = val;
    xn[(size_t)c * C3 + ci] = next_x<BL, TV>(g, g.sp[g.sim[c]], c, I, J, Kc, wscale, val);
  }
}

// ---- up: x~ = x + P y_coarse (on the fly for the cell and its neighbours), then
// y = x~ + S (r - K x~).  One thread per cell.
template <int BL, class TV>
__device__ __forceinline__ TV up_cell(const DevGrid& g, int l, TV wscale, TV cscale,
                                      const TV* __restrict__ r, const TV* __restrict__ x,
                                      const TV* __restrict__ yc, int c, int i, int j, int k,
                                      TV* rv_out) {
  constexpr int B3 = BL * BL * BL, CB = BL / 2;
  const SimParams& sp = g.sp[g.sim[c]];
  const TV coef = cube_h<TV>(g, sp, c) * cscale;
  auto uval = [&](int cube, int cell) {
    const int a = cell % BL, b = (cell / BL) % BL, e = cell / (BL * BL);
    return x[(size_t)cube * B3 + cell] +
           TV(kMgOver) * yc[(size_t)cube * CB * CB * CB + lcell<CB>(a >> 1, b >> 1, e >> 1)];
  };
  const TV rv = r[(size_t)c * B3 + lcell<BL>(i, j, k)];
  const TV xc = uval(c, lcell<BL>(i, j, k));
  const TV acc = mg_faces<BL, TV>(g, c, l, i, j, k, xc, uval);
  *rv_out = rv;
  return xc + smooth_w<BL, TV>(g, sp, c, i, j, k, wscale) * (rv - coef * acc);
}

template <int BL, class TV>
__device__ __forceinline__ void mg_up_item(const DevGrid& g, int l, TV wscale, TV cscale,
                                           const TV* __restrict__ r, const TV* __restrict__ x,
                                           const TV* __restrict__ yc,
                                           TV* __restrict__ y, int all, long long t) {
  constexpr int B3 = BL * BL * BL;
  const int c = (int)(t / B3), cell = (int)(t - (long long)c * B3);
  if (!all && g.ss[g.sim[c]].done) return;
  const int i = cell % BL, j = (cell / BL) % BL, k = cell / (BL * BL);
  TV rv;
  y[t] = up_cell<BL, TV>(g, l, wscale, cscale, r, x, yc, c, i, j, k, &rv);
}

template <int BL, class TV>
__global__ __launch_bounds__(256) void k_mg_up(DevGrid g, int l, TV wscale, TV cscale,
                                               const TV* __restrict__ r,
                                               const TV* __restrict__ x,
                                               const TV* __restrict__ yc,
                                               TV* __restrict__ y, int all) {
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)g.n_cubes * BL * BL * BL) return;
  mg_up_item<BL, TV>(g, l, wscale, cscale, r, x, yc, y, all, t);
}

// The last block of the finest up launch: mode 0 (start of a solve) takes <r, z> as
// the PCG's rz; mode 1 (after pass B) forms beta, counts the iteration and tests
// convergence on the <r, r> that pass B accumulated.
__device__ void mg_decide(const DevGrid& g, const SolveParams& prm, int mode, int nt) {
  int alive = 0;
  for (int q = threadIdx.x; q < g.n_sims; q += nt) {
    SimState& t = g.ss[q];
    const double rzs = acc_take(t, ACC_RZ);
    if (mode == 0) {
      if (!t.done) t.rz = rzs;
      alive |= !t.done;
      continue;
    }
    const double rr = acc_take(t, ACC_RR), pq = acc_take(t, ACC_PQ);
    if (t.done) continue;
    if (t.nonfinite || !isfinite(rr) || !isfinite(rzs) || !isfinite(pq)) {
      t.nonfinite = 1;
      t.done = 1;
      continue;
    }
    t.beta = (t.rz != 0.0) ? rzs / t.rz : 0.0;
    t.rz = rzs;
    t.rr = rr;
    t.iter += 1;
    t.total_iters += 1;
    const bool inner = prm.mixed != 0;
    const double tol2 = inner ? t.inner_tol2 : t.tol2;
    const bool ok = rr <= tol2;
    if (!inner) {
      t.rr64 = rr;
      t.converged = ok;
    }
    if (ok || t.iter >= (inner ? prm.inner_max_iter : prm.max_iter)) t.done = 1;
    alive |= !t.done;
  }
  alive = __syncthreads_or(alive);
  if (threadIdx.x == 0) {
    if (mode == 1) g.flags[0] = !alive;
    // a captured step: this launch ends the inner loop's body (mode 1) or starts an
    // inner solve (mode 0) and sets the loop's condition; mode 1 also keeps the guard
    // on the number of body executions
    if (prm.cond_inner) {
      unsigned int go = alive ? 1u : 0u;
      if (mode == 1 && atomicAdd(prm.guard, 1u) + 1u >= (unsigned int)prm.guard_limit) go = 0u;
      set_cond(prm.cond_inner, go);
      if (prm.body_count) atomicAdd(prm.body_count + (mode == 1 ? 0 : 1), 1u);
    }
  }
}

// ---- up on the finest level: z = y_0, <r, z> per sim, and the PCG's decisions.
// Blocks of NT = min(256, B^3) threads lie inside one cube, hence one sim.
template <int B, int NT, class TV>
__global__ __launch_bounds__(NT) void k_mg_up0(DevGrid g, const TV* __restrict__ r,
                                              const TV* __restrict__ x,
                                              const TV* __restrict__ yc,
                                              TV* __restrict__ z, SolveParams prm, int mode) {
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  constexpr int B3 = B * B * B, PER = B3 / NT;
  __shared__ double red[32];
  const int c = blockIdx.x / PER;
  const int s = g.sim[c];
  SimState& st = g.ss[s];
  const bool all = mode == 2;
  const bool active = all || !st.done;
  double rz = 0.0;
  if (active) {
    const int cell = (blockIdx.x - c * PER) * NT + threadIdx.x;
    const int i = cell % B, j = (cell / B) % B, k = cell / (B * B);
    TV rv;
    const TV zv = up_cell<B, TV>(g, 0, TV(kMgOmega), TV(1), r, x, yc, c, i, j,
                                 k, &rv);
    z[(size_t)c * B3 + cell] = zv;
    rz = double(rv * zv);
  }
  if (all) return;
  double vals[1] = {rz};
  block_sum<NT, 1>(vals, red);
  if (threadIdx.x == 0 && active) acc_add(st, ACC_RZ, vals[0]);
  if (last_block(g.counter)) mg_decide(g, prm, mode, NT);
}

// ---- levels of 8^3 / 16^3 cells per cube on quad tiles (bcm_quad.cuh): down stages
// x = S r with the face halo, forms rr = r - K x and sums its 2x2x2 children into r_{l+1};
// up stages x~ = S r + s P y_{l+1} (S r formed again from r: cheaper than storing and
// reading x), then y = x~ + S (r - K x~) and, on the finest level, <r, z>.  On level l,
// S = (omega / 4^l) D^-1 and K = 4^l h (sum of differences) with the finest level's D: the
// launch passes wl = omega / 4^l and cl = 4^l.  Same values as the per-cell kernels above.
//
// With FB the down launch also does the PCG's pass B (x_pcg += alpha p, r -= alpha q,
// <r, r>): it reads the residual r_in of the iteration and writes the new one to the
// other buffer r_out (blocks read their neighbours' r_in for the halo, so it is not
// updated in place), forming the halo's new residual on the fly.  The buffers swap
// with the parity of the sim's iteration count.
template <class TV>
struct PassB {
  TV* x;                 // PCG iterate
  const TV *p0, *p1, *q; // search directions (by iteration parity), q = K p
  TV *ra, *rb;           // residual: in ra, out rb at even iterations; swapped at odd
};

// alpha = <r, z> / <p, K p> of one sim (zero where the denominator is zero or not finite)
__device__ __forceinline__ double cg_alpha_of(double rz, double pq) {
  return pq != 0.0 && isfinite(pq) ? quick_div(rz, pq, quick_rcp(pq)) : 0.0;
}

template <int B, class TV, bool FB>
__global__ __launch_bounds__(QT<B, TV>::NT, QT<B, TV>::blocks) void k_mg_down_quad(DevGrid g, const TV* __restrict__ r0,
                                                            TV* __restrict__ r1,
                                                            TV* __restrict__ x1, int all,
                                                            PassB<TV> pb, TV wl, TV cl, int lsh) {
  using T = QT<B, TV>;
  constexpr int B3 = T::B3, BB = T::BB, CB = B / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CubeQ<TV> cqs[T::CPB];
  __shared__ TV alphas[T::CPB];
  const int cub = threadIdx.x / T::TPC, lt = threadIdx.x - cub * T::TPC;
  const int c = blockIdx.x * T::CPB + cub;
  TV* S = reinterpret_cast<TV*>(smem_raw) + cub * T::N;
  TV* gh = S + B3;
  CubeQ<TV>& cq = cqs[cub];
  const bool valid = c < g.n_cubes;
  const CubeLoad L = cube_lookup(g, valid ? c : 0, lt);
  Halo<B, TV> H;
  H.lookup(g, valid ? c : 0, lt);
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  poison_tile(reinterpret_cast<TV*>(smem_raw), T::CPB * T::N);
  if (!valid) return;
  SimState& st = g.ss[L.s];
  double pq = 0.0, rz = 0.0;
  if constexpr (FB) {  // the stripes of <p, K p>, and <r, z>
    if (lt < kStripes) pq = ld_acc(&st.acc[lt][ACC_PQ]);
    rz = st.rz;
  }
  if (!all && st.done) return;
  const TV* __restrict__ r = r0;
  TV* __restrict__ rout = nullptr;
  const TV* __restrict__ pn = nullptr;
  TV alpha = TV(0);
  if constexpr (FB) {
    const int it = st.iter;
    r = (it & 1) ? pb.rb : pb.ra;
    rout = (it & 1) ? pb.ra : pb.rb;
    pn = (it & 1) ? pb.p0 : pb.p1;
  }
  const int pos = lt % T::Q, i0 = (4 * pos) % B, j = (4 * pos) / B, k0 = T::NP * (lt / T::Q);
  const int cell0 = (k0 * B + j) * B + i0;
  const size_t base = (size_t)c * B3 + cell0;
  TV res[T::NP][4], v[T::NP][4];
#pragma unroll
  for (int m = 0; m < T::NP; ++m) {
    ld4(r + base + m * BB, res[m]);
    if constexpr (FB) ld4(pb.q + base + m * BB, v[m]);
  }
  TV ha[Halo<B, TV>::R][4], hb[FB ? Halo<B, TV>::R : 1][4];
  H.each(lt, [&](int u, int, int n, int cell, int stride) {
    const size_t gi = (size_t)n * B3 + cell;
    ldq(r + gi, stride, ha[u]);
    if constexpr (FB) ldq(pb.q + gi, stride, hb[u]);
  });
  cube_publish(cq, g, L, lt);
  if constexpr (FB) {  // alpha, by the cube's first warp while the cells are in flight
    if (lt < 32) {
#pragma unroll
      for (int o = 1; o < kStripes; o <<= 1) pq += __shfl_xor_sync(0xffffffffu, pq, o);
      if (lt == 0) alphas[cub] = TV(cg_alpha_of(rz, pq));
    }
  }
  T::sync();
  if constexpr (FB) alpha = alphas[cub];
  // S times the iteration's residual (FB: r_in - alpha q) on the halo
  auto make = [&](int u, int f, int, int cell, int stride, TV (&o)[4]) {
    TV inv[4];
    if constexpr (FB) axpy4(-alpha, hb[u], ha[u], ha[u]);
    nb_inv<B>(cq, g, c, f, cell, stride, inv);
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = (wl * inv[e]) * ha[u][e];
  };
  auto one = [&](int n, int cell) {
    const size_t gi = (size_t)n * B3 + cell;
    TV x = r[gi];
    if constexpr (FB) x -= alpha * pb.q[gi];
    return wl * inv_diag_any<B, TV>(g, n, cell) * x;
  };
  H.store(gh, g, c, lt, make, one, lsh);
  TV rr2 = TV(0);
#pragma unroll
  for (int m = 0; m < T::NP; ++m) {
    if constexpr (FB) {
      axpy4(-alpha, v[m], res[m], res[m]);
      rr2 += dot4(res[m], res[m]);
      st4(rout + base + m * BB, res[m]);
    }
    TV inv[4];
    quad_inv<B>(cq, i0, j, k0 + m, inv);
#pragma unroll
    for (int e = 0; e < 4; ++e) v[m][e] = (wl * inv[e]) * res[m][e];
    own_quad<B>(S, gh, cq, i0, j, k0 + m, v[m]);
  }
  T::sync();
  const TV h = cq.h * cl;
  quad_column<B>(S, gh, cq, i0, j, k0, v,
                 [&](int m, const TV (&acc)[4]) { axpy4(-h, acc, res[m], res[m]); });
  // 2x2x2 sums: planes and x within the thread, y from the lane B / 4 on
#pragma unroll
  for (int u = 0; u < T::NP / 2; ++u) {
    TV s0 = (res[2 * u][0] + res[2 * u][1]) + (res[2 * u + 1][0] + res[2 * u + 1][1]);
    TV s1 = (res[2 * u][2] + res[2 * u][3]) + (res[2 * u + 1][2] + res[2 * u + 1][3]);
    s0 += __shfl_xor_sync(0xffffffffu, s0, B / 4);
    s1 += __shfl_xor_sync(0xffffffffu, s1, B / 4);
    if ((j & 1) == 0) {
      const int I = i0 >> 1, J = j >> 1, K = (k0 >> 1) + u;
      const size_t o = (size_t)c * CB * CB * CB + (K * CB + J) * CB + I;
      r1[o] = s0;
      r1[o + 1] = s1;
      if (x1) {  // S r of the next level, where its kernel works cell by cell
        const TV w4 = TV(0.25) * wl;
        x1[o] = w4 * (cq.smask ? cq.inv[s3_of<CB>(cq.w3, I, J, K)] : cq.inv[18]) * s0;
        x1[o + 1] = w4 * (cq.smask ? cq.inv[s3_of<CB>(cq.w3, I + 1, J, K)] : cq.inv[18]) * s1;
      }
    }
  }
  if constexpr (FB) {  // x last: its loads would hold the registers of another block
    TV xv[T::NP][4], pv[T::NP][4];
#pragma unroll
    for (int m = 0; m < T::NP; ++m) {
      ld4(pb.x + base + m * BB, xv[m]);
      ld4(pn + base + m * BB, pv[m]);
    }
#pragma unroll
    for (int m = 0; m < T::NP; ++m) {
      axpy4(alpha, pv[m], xv[m], xv[m]);
      st4(pb.x + base + m * BB, xv[m]);
    }
  }
  if constexpr (FB) {  // (summed in FP64 from the threads on, as <r, z> below)
    const double sum = T::sum(double(rr2));
    if (lt == 0) acc_add_cube(st, ACC_RR, c, sum);
  }
}

template <int B, class TV>
__global__ __launch_bounds__(QT<B, TV>::NT, QT<B, TV>::blocks) void k_mg_up_quad(DevGrid g, const TV* __restrict__ ra,
                                                          const TV* __restrict__ rb,
                                                          const TV* __restrict__ y1,
                                                          TV* __restrict__ z, SolveParams prm,
                                                          int mode, TV wl, TV cl, int finest,
                                                          int lsh) {
  using T = QT<B, TV>;
  constexpr int B3 = T::B3, BB = T::BB, CB = B / 2, C3 = CB * CB * CB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ CubeQ<TV> cqs[T::CPB];
  const int cub = threadIdx.x / T::TPC, lt = threadIdx.x - cub * T::TPC;
  const int c = blockIdx.x * T::CPB + cub;
  TV* S = reinterpret_cast<TV*>(smem_raw) + cub * T::N;
  TV* gh = S + B3;
  CubeQ<TV>& cq = cqs[cub];
  const bool valid = c < g.n_cubes;
  const CubeLoad L = cube_lookup(g, valid ? c : 0, lt);
  Halo<B, TV> H;
  H.lookup(g, valid ? c : 0, lt);
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  poison_tile(reinterpret_cast<TV*>(smem_raw), T::CPB * T::N);
  SimState& st = g.ss[L.s];
  const bool active = valid && (mode == 2 || !st.done);
  TV part = TV(0);
  if (active) {
    // after a down launch with pass B (rb set) the new residual is in the buffer that
    // the iteration's parity selects, else in ra
    const TV* __restrict__ r = (mode == 1 && rb && !(st.iter & 1)) ? rb : ra;
    const int pos = lt % T::Q, i0 = (4 * pos) % B, j = (4 * pos) / B, k0 = T::NP * (lt / T::Q);
    const size_t base = (size_t)c * B3 + (k0 * B + j) * B + i0;
    auto coarse = [&](int cell) {
      return (((cell / BB) >> 1) * CB + (((cell / B) % B) >> 1)) * CB + ((cell % B) >> 1);
    };
    TV res[T::NP][4], v[T::NP][4], yc[T::NP / 2][2];
#pragma unroll
    for (int m = 0; m < T::NP; ++m) ld4(r + base + m * BB, res[m]);
#pragma unroll
    for (int u = 0; u < T::NP / 2; ++u) {
      const TV* y = y1 + (size_t)c * C3 + (((k0 >> 1) + u) * CB + (j >> 1)) * CB + (i0 >> 1);
      yc[u][0] = y[0];
      yc[u][1] = y[1];
    }
    TV ha[Halo<B, TV>::R][4], hy[Halo<B, TV>::R][2];
    H.each(lt, [&](int u, int, int n, int cell, int stride) {
      ldq(r + (size_t)n * B3 + cell, stride, ha[u]);
      hy[u][0] = y1[(size_t)n * C3 + coarse(cell)];
      hy[u][1] = y1[(size_t)n * C3 + coarse(cell + 2 * stride)];
    });
    cube_publish(cq, g, L, lt);
    T::sync();
    const TV over = TV(kMgOver);
    auto make = [&](int u, int f, int, int cell, int stride, TV (&o)[4]) {
      TV inv[4];
      nb_inv<B>(cq, g, c, f, cell, stride, inv);
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = (wl * inv[e]) * ha[u][e] + over * hy[u][e >> 1];
    };
    auto one = [&](int n, int cell) {
      return wl * inv_diag_any<B, TV>(g, n, cell) * r[(size_t)n * B3 + cell] +
             over * y1[(size_t)n * C3 + coarse(cell)];
    };
    H.store(gh, g, c, lt, make, one, lsh);
#pragma unroll
    for (int m = 0; m < T::NP; ++m) {
      TV inv[4];
      quad_inv<B>(cq, i0, j, k0 + m, inv);
      const TV ya = over * yc[m >> 1][0], yb = over * yc[m >> 1][1];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[m][e] = (wl * inv[e]) * res[m][e] + (e < 2 ? ya : yb);
      own_quad<B>(S, gh, cq, i0, j, k0 + m, v[m]);
    }
    T::sync();
    const TV h = cq.h * cl;
    quad_column<B>(S, gh, cq, i0, j, k0, v, [&](int m, const TV (&acc)[4]) {
      TV inv[4], t[4], zv[4];
      quad_inv<B>(cq, i0, j, k0 + m, inv);
      axpy4(-h, acc, res[m], t);
#pragma unroll
      for (int e = 0; e < 4; ++e) zv[e] = v[m][e] + (wl * inv[e]) * t[e];
      st4(z + base + m * BB, zv);
      part += dot4(res[m], zv);
    });
  }
  if (mode == 2 || !finest) return;
  const double sum = T::sum(double(part));
  if (lt == 0 && active) acc_add_cube(st, ACC_RZ, c, sum);
}

// The decisions of an iteration (mg_decide) after the quad kernels, in a launch of one block:
// electing a last block in the finest up launch instead keeps every block on its SM for two
// more round trips to memory.
__global__ void k_mg_decide(DevGrid g, SolveParams prm, int mode) {
  cudaGridDependencySynchronize();
  mg_decide(g, prm, mode, blockDim.x);
}

// ---- the coarse levels, in one cluster: the per-cube levels from lf on (BL = 4, 2, 1 cells
// per cube edge), the aggregate levels, and the way back up to level lf, with cluster
// barriers between the steps.  Each step is a short chain of dependent loads on few cells,
// so a launch of its own costs more than its work (9 launches, 57 us serialised at 1024
// cubes); one block of 1024 threads holds the aggregate levels that fit its shared memory
// (their tables are copied in while the previous kernel drains), the whole cluster the
// larger ones.  Values that other blocks wrote are read through L2.
struct AggLevel {
  int n;
  double *ar, *y, *at, *x;  // residual, result, scratch, S ar (shared memory, or the workspace)
  const double *diag, *inv, *val;  // K's diagonal, omega / diagonal, -off-diagonals
  const int *row, *col, *cptr, *cidx, *parent;  // parent: of this level's children
};

__host__ __device__ inline size_t top_piece(size_t bytes) { return (bytes + 15) & ~(size_t)15; }
// shared-memory bytes of aggregate levels k0 .. M-1
__host__ __device__ inline size_t agg_smem(const MgDev& mg, int n_cubes, int k0) {
  size_t b = 0;
  for (int k = k0; k < mg.M; ++k) {
    const size_t n = (size_t)mg.n[k], nnz = (size_t)mg.nnz[k], np = k ? mg.n[k - 1] : n_cubes;
    b += 6 * top_piece(8 * n) + top_piece(8 * nnz) + top_piece(4 * (n + 1)) + top_piece(4 * nnz);
    b += top_piece(4 * (n + 1)) + (k ? 2 : 1) * top_piece(4 * np);
  }
  return b;
}

// asynchronous global -> shared copy of `count` elements of 4 or 8 bytes, by the block
template <int E>
__device__ __forceinline__ void copy_async(const void* dst, const void* src, int count) {
  static_assert(E == 4 || E == 8, "element size");
  for (int a = threadIdx.x; a < count; a += blockDim.x) {
    const unsigned int d =
        (unsigned int)__cvta_generic_to_shared(static_cast<const char*>(dst) + (size_t)E * a);
    const char* s = static_cast<const char*>(src) + (size_t)E * a;
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(s), "n"(E) : "memory");
  }
}

// The V-cycle on the aggregate levels: W is the set of threads that runs a level (a block on
// shared memory, or the cluster on the workspace) with its index, size, barrier and loads.
// An FP64 operation takes a warp 64 cycles here, a barrier of the block about 40, so S ar is
// formed once per node and not once per edge, and the sums run in few chains.
struct BlockWorkers {
  __device__ __forceinline__ int id() const { return threadIdx.x; }
  __device__ __forceinline__ int count() const { return blockDim.x; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ double ld(const double* p) const { return *p; }
};
struct ClusterWorkers {
  int rank, ranks;
  __device__ __forceinline__ int id() const { return rank * blockDim.x + threadIdx.x; }
  __device__ __forceinline__ int count() const { return ranks * blockDim.x; }
  // the same threads numbered warp by warp over the blocks, so few cells use every SM
  __device__ __forceinline__ int spread() const {
    return (((int)threadIdx.x >> 5) * ranks + rank) * 32 + ((int)threadIdx.x & 31);
  }
  __device__ __forceinline__ void sync() const { cooperative_groups::this_cluster().sync(); }
  __device__ __forceinline__ double ld(const double* p) const { return __ldcg(p); }
};
// ar - K f on node a, f(b) a node's value: six entries at a time, loaded together, in two
// chains of additions (64 cycles each)
template <class W, class F>
__device__ __forceinline__ double agg_resid(const W& w, const AggLevel& L, int a, double r, const F& f) {
  double k0 = L.diag[a] * f(a), k1 = 0.0;
  const int e1 = L.row[a + 1];
  for (int e = L.row[a]; e < e1; e += 6) {
    double v[6], x[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const bool in = e + q < e1;
      v[q] = in ? L.val[e + q] : 0.0;
      x[q] = in ? f(L.col[e + q]) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 6; q += 2) {
      k0 -= v[q] * x[q];
      k1 -= v[q + 1] * x[q + 1];
    }
  }
  return r - (k0 + k1);
}
template <class W, class V>
__device__ __forceinline__ double agg_sum(const AggLevel& C, int a, const V& v) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  const int e0 = C.cptr[a], e1 = C.cptr[a + 1];
  for (int e = e0; e < e1; e += 4)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (e + q < e1) s[q] += v(C.cidx[e + q]);
  return (s[0] + s[1]) + (s[2] + s[3]);
}
// down on level L: x = S ar, at = ar - K x
template <class W>
__device__ __forceinline__ void agg_down(const W& w, const AggLevel& L) {
  for (int a = w.id(); a < L.n; a += w.count()) L.x[a] = L.inv[a] * w.ld(L.ar + a);
  w.sync();
  auto xv = [&](int b) { return w.ld(L.x + b); };
  for (int a = w.id(); a < L.n; a += w.count()) L.at[a] = agg_resid(w, L, a, w.ld(L.ar + a), xv);
}
// up on level L: x += s P yc, y = x + S (ar - K x)
template <class W, class Y>
__device__ __forceinline__ void agg_up(const W& w, const AggLevel& L, const int* parent, const Y& yc) {
  for (int a = w.id(); a < L.n; a += w.count()) L.x[a] = w.ld(L.x + a) + kMgOver * yc(parent[a]);
  w.sync();
  auto xv = [&](int b) { return w.ld(L.x + b); };
  for (int a = w.id(); a < L.n; a += w.count())
    L.y[a] = xv(a) + L.inv[a] * agg_resid(w, L, a, w.ld(L.ar + a), xv);
}
// kMgNuTop damped-Jacobi sweeps from zero (the first is S ar); result in y
template <class W>
__device__ __forceinline__ void agg_top(const W& w, const AggLevel& L) {
  double *x = L.at, *o = L.y;
  static_assert(kMgNuTop == 4, "an odd number of sweeps after the first ends in y");
  for (int a = w.id(); a < L.n; a += w.count()) x[a] = L.inv[a] * w.ld(L.ar + a);
  for (int sweep = 1; sweep < kMgNuTop; ++sweep) {
    w.sync();
    auto xv = [&](int b) { return w.ld(x + b); };
    for (int a = w.id(); a < L.n; a += w.count())
      o[a] = xv(a) + L.inv[a] * agg_resid(w, L, a, w.ld(L.ar + a), xv);
    double* t = x;
    x = o;
    o = t;
  }
}

// ---- per-cube levels inside the cluster (the same values as the per-cell kernels; r, x, y
// of the coarse levels are written and read by different blocks)
template <int BL, class TV>
__device__ __forceinline__ void coarse_down(const DevGrid& g, const MgDev& mg, int l, int all,
                                            const ClusterWorkers& w) {
  constexpr int B3 = BL * BL * BL, CB = BL > 1 ? BL / 2 : 1, C3 = CB * CB * CB;
  const TV *r = (const TV*)mg.r[l], *x = (const TV*)mg.x[l];
  TV* rc = BL > 1 ? (TV*)mg.r[l + 1] : (TV*)mg.rr;
  TV* xn = BL > 1 ? (TV*)mg.x[l + 1] : nullptr;
  const TV c4 = TV(1 << (2 * l)), wscale = TV(kMgOmega / double(1 << (2 * l)));
  const int total = g.n_cubes * B3, rounded = (total + 31) / 32 * 32;
  for (int t = w.spread(); t < rounded; t += w.count()) {
    const int c = t / B3, q = t - c * B3, d = BL > 1 ? q & 7 : 0, ci = BL > 1 ? q >> 3 : 0;
    const bool on = t < total && (all || !g.ss[g.n_sims == 1 ? 0 : g.sim[c]].done);
    const int I = ci % CB, J = (ci / CB) % CB, K = ci / (CB * CB);
    TV val = TV(0);
    if (on) {
      const int i = BL > 1 ? 2 * I + (d & 1) : 0, j = BL > 1 ? 2 * J + ((d >> 1) & 1) : 0;
      const int k = BL > 1 ? 2 * K + (d >> 2) : 0;
      const TV coef = cube_h<TV>(g, g.sp[g.sim[c]], c) * c4;
      auto xval = [&](int cube, int cell) { return __ldcg(x + (size_t)cube * B3 + cell); };
      const int cell = lcell<BL>(i, j, k);
      const TV rv = __ldcg(r + (size_t)c * B3 + cell), xc = xval(c, cell);
      const TV acc = mg_faces<BL, TV>(g, c, l, i, j, k, xc, xval);
      val = rv - coef * acc;
    }
    if constexpr (BL > 1) {
      val += __shfl_xor_sync(0xffffffffu, val, 1);
      val += __shfl_xor_sync(0xffffffffu, val, 2);
      val += __shfl_xor_sync(0xffffffffu, val, 4);
    }
    if (d == 0 && on) {
      rc[(size_t)c * C3 + ci] = val;
      if constexpr (BL > 1)
        xn[(size_t)c * C3 + ci] = next_x<BL, TV>(g, g.sp[g.sim[c]], c, I, J, K, wscale, val);
    }
  }
}
template <int BL, class TV>
__device__ __forceinline__ void coarse_up(const DevGrid& g, const MgDev& mg, int l, int all,
                                          const double* yagg, const ClusterWorkers& w) {
  constexpr int B3 = BL * BL * BL, CB = BL > 1 ? BL / 2 : 1;
  const TV *r = (const TV*)mg.r[l], *x = (const TV*)mg.x[l];
  const TV* yc = BL > 1 ? (const TV*)mg.y[l + 1] : nullptr;
  TV* y = (TV*)mg.y[l];
  const int* parent = mg.parent[0];
  const TV c4 = TV(1 << (2 * l)), wscale = TV(kMgOmega / double(1 << (2 * l)));
  const int total = g.n_cubes * B3;
  for (int t = w.spread(); t < total; t += w.count()) {
    const int c = t / B3, q = t - c * B3;
    if (!all && g.ss[g.n_sims == 1 ? 0 : g.sim[c]].done) continue;
    const int i = q % BL, j = (q / BL) % BL, k = q / (BL * BL);
    const SimParams& sp = g.sp[g.sim[c]];
    const TV coef = cube_h<TV>(g, sp, c) * c4;
    auto uval = [&](int cube, int cell) {  // S r + s P y
      const TV xv = __ldcg(x + (size_t)cube * B3 + cell);
      if constexpr (BL == 1) {
        return xv + TV(kMgOver * __ldcg(yagg + parent[cube]));
      } else {
        const int a = cell % BL, b = (cell / BL) % BL, e = cell / (BL * BL);
        return xv + TV(kMgOver) *
                        __ldcg(yc + (size_t)cube * CB * CB * CB + lcell<CB>(a >> 1, b >> 1, e >> 1));
      }
    };
    const TV xc = uval(c, q);
    const TV acc = mg_faces<BL, TV>(g, c, l, i, j, k, xc, uval);
    const TV rv = __ldcg(r + (size_t)c * B3 + q);
    y[(size_t)c * B3 + q] = xc + smooth_w<BL, TV>(g, sp, c, i, j, k, wscale) * (rv - coef * acc);
  }
}

// bl0: cells per cube edge on level lf; levels k < kd of the aggregates run on the cluster.
template <class TV>
__global__ __launch_bounds__(1024, 1) void k_mg_coarse(DevGrid g, MgDev mg, int lf, int bl0, int kd,
                                                       int all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ AggLevel lv[kMgMaxM];
  const int tid = threadIdx.x, NT = blockDim.x;
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const ClusterWorkers cw{(int)cl.block_rank(), (int)cl.num_blocks()};
  const BlockWorkers bw;
  const bool head = cw.rank == 0;
  if (tid == 0) {  // layout from the sizes alone (no memory reads)
    unsigned char* o = smem_raw;
    auto take = [&](size_t bytes) {
      unsigned char* p = o;
      o += top_piece(bytes);
      return p;
    };
    for (int k = 0; k < mg.M; ++k) {
      AggLevel& L = lv[k];
      const size_t n = mg.n[k], nnz = mg.nnz[k], np = k ? mg.n[k - 1] : g.n_cubes;
      L = AggLevel{mg.n[k], mg.ar[k], mg.ax[k], mg.at[k], mg.as[k], mg.diag[k], mg.inv[k], mg.val[k],
                   mg.row[k], mg.col[k], mg.cptr[k], mg.cidx[k], mg.parent[k]};
      if (k < kd) continue;
      L.ar = (double*)take(8 * n);
      L.y = (double*)take(8 * n);
      L.at = (double*)take(8 * n);
      L.x = (double*)take(8 * n);
      L.diag = (double*)take(8 * n);
      L.inv = (double*)take(8 * n);
      L.val = (double*)take(8 * nnz);
      L.row = (int*)take(4 * (n + 1));
      L.col = (int*)take(4 * nnz);
      L.cptr = (int*)take(4 * (n + 1));
      L.cidx = (int*)take(4 * np);
      if (k) L.parent = (int*)take(4 * np);
    }
  }
  __syncthreads();
  if (head) {
    for (int k = kd; k < mg.M; ++k) {
      const AggLevel& L = lv[k];
      const int n = L.n, nnz = mg.nnz[k], np = k ? mg.n[k - 1] : g.n_cubes;
      copy_async<8>(L.diag, mg.diag[k], n);
      copy_async<8>(L.inv, mg.inv[k], n);
      copy_async<8>(L.val, mg.val[k], nnz);
      copy_async<4>(L.row, mg.row[k], n + 1);
      copy_async<4>(L.col, mg.col[k], nnz);
      copy_async<4>(L.cptr, mg.cptr[k], n + 1);
      copy_async<4>(L.cidx, mg.cidx[k], np);
      if (k) copy_async<4>(L.parent, mg.parent[k], np);
    }
  }
  cudaGridDependencySynchronize();  // launched after the previous level's kernel
  int l = lf, bl = bl0;
  for (;; ++l, bl >>= 1) {
    if (bl == 4) coarse_down<4, TV>(g, mg, l, all, cw);
    else if (bl == 2) coarse_down<2, TV>(g, mg, l, all, cw);
    else coarse_down<1, TV>(g, mg, l, all, cw);
    cl.sync();
    if (bl == 1) break;
  }
  if (head) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
  }
  const int top = mg.M - 1;
  const TV* rr = (const TV*)mg.rr;
  auto cube_r = [&](int c) { return double(__ldcg(rr + c)); };
  // down: levels 0 .. kd-1 on the cluster, then the rest in the head block
  if (kd > 0) {
    for (int a = cw.id(); a < lv[0].n; a += cw.count()) lv[0].ar[a] = agg_sum<ClusterWorkers>(lv[0], a, cube_r);
    cl.sync();
    for (int k = 0; k < kd; ++k) {
      const AggLevel& L = lv[k];
      if (k == top) {
        agg_top(cw, L);
        cl.sync();
        break;
      }
      agg_down(cw, L);
      cl.sync();
      if (k + 1 < kd) {
        auto child = [&](int c) { return __ldcg(L.at + c); };
        for (int a = cw.id(); a < lv[k + 1].n; a += cw.count())
          lv[k + 1].ar[a] = agg_sum<ClusterWorkers>(lv[k + 1], a, child);
        cl.sync();
      }
    }
  }
  if (kd <= top) {
    if (head) {
      const AggLevel& F = lv[kd];
      if (kd == 0) {
        for (int a = tid; a < F.n; a += NT) F.ar[a] = agg_sum<BlockWorkers>(F, a, cube_r);
      } else {
        const AggLevel& L = lv[kd - 1];
        auto child = [&](int c) { return __ldcg(L.at + c); };
        for (int a = tid; a < F.n; a += NT) F.ar[a] = agg_sum<BlockWorkers>(F, a, child);
      }
      __syncthreads();
      for (int k = kd; k < top; ++k) {
        const AggLevel &L = lv[k], &C = lv[k + 1];
        agg_down(bw, L);
        __syncthreads();
        auto child = [&](int c) { return L.at[c]; };
        for (int a = tid; a < C.n; a += NT) C.ar[a] = agg_sum<BlockWorkers>(C, a, child);
        __syncthreads();
      }
      agg_top(bw, lv[top]);
      __syncthreads();
      for (int k = top - 1; k >= kd; --k) {
        const AggLevel& C = lv[k + 1];
        agg_up(bw, lv[k], C.parent, [&](int b) { return C.y[b]; });
        __syncthreads();
      }
      for (int a = tid; a < F.n; a += NT) mg.ax[kd][a] = F.y[a];  // for the other blocks
    }
    cl.sync();
  }
  for (int k = (kd <= top ? kd : top) - 1; k >= 0; --k) {
    const double* yc = mg.ax[k + 1];
    agg_up(cw, lv[k], mg.parent[k + 1], [&](int b) { return __ldcg(yc + b); });
    cl.sync();
  }
  for (;; --l, bl <<= 1) {
    if (bl == 4) coarse_up<4, TV>(g, mg, l, all, mg.ax[0], cw);
    else if (bl == 2) coarse_up<2, TV>(g, mg, l, all, mg.ax[0], cw);
    else coarse_up<1, TV>(g, mg, l, all, mg.ax[0], cw);
    if (l == lf) break;
    cl.sync();
  }
}

// ---------------------------------------------------------------- launcher

template <int BL, class TV>
static cudaError_t down_t(const Ctx& x, int l, int all) {
  const double c4 = double(1 << (2 * l));
  const long long n = (long long)x.g.n_cubes * BL * BL * BL;
  auto kern = l == 0 ? k_mg_down_cell<BL, TV, false> : k_mg_down_cell<BL, TV, true>;
  return launch_pdl(kern, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, x.stream, x.g, l,
                    TV(kMgOmega / c4), TV(c4), (const TV*)x.mg.r[l], (TV*)x.mg.x[l],
                    (TV*)x.mg.r[l + 1], (TV*)x.mg.x[l + 1], all);
}

template <int BL, class TV>
static cudaError_t up_t(const Ctx& x, int l, int all) {
  const long long n = (long long)x.g.n_cubes * BL * BL * BL;
  const TV* yc = (const TV*)x.mg.y[l + 1];
  const double c4 = double(1 << (2 * l));
  return launch_pdl(k_mg_up<BL, TV>, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, x.stream,
                    x.g, l, TV(kMgOmega / c4), TV(c4), (const TV*)x.mg.r[l], (const TV*)x.mg.x[l],
                    yc, (TV*)x.mg.y[l], all);
}

template <class TV>
static cudaError_t level_t(const Ctx& x, int l, bool down, int all) {
  const int BL = x.B >> l;
#define BCM_MG_LEVEL(V) \
  case V: return down ? down_t<V, TV>(x, l, all) : up_t<V, TV>(x, l, all);
  switch (BL) {
    BCM_MG_LEVEL(4)
    BCM_MG_LEVEL(2)
    default: return cudaErrorInvalidValue;
  }
#undef BCM_MG_LEVEL
}

template <int B, class TV>
static cudaError_t up0_t(const Ctx& x, const SolveParams& prm, int mode) {
  constexpr int B3 = B * B * B, NT = B3 < 256 ? B3 : 256;
  const TV* yc = (const TV*)x.mg.y[1];
  return launch_pdl(k_mg_up0<B, NT, TV>, dim3(x.g.n_cubes * (B3 / NT)), dim3(NT), 0, x.stream,
                    x.g, (const TV*)x.mg.r[0], (const TV*)x.mg.x[0], yc,
                    (TV*)x.mg.y[0], prm, mode);
}

template <int B, class TV>
static cudaError_t down_quad_t(const Ctx& x, int l, int all, bool fb) {
  using T = QT<B, TV>;
  const size_t sm = sizeof(TV) * (size_t)T::N * T::CPB;
  PassB<TV> pb{};
  if (fb) {
    pb.x = x.solve64 ? (TV*)x.f.p : (TV*)x.f.e;
    pb.p0 = (const TV*)x.f.p0;
    pb.p1 = (const TV*)x.f.p1;
    pb.q = (const TV*)x.f.q;
    pb.ra = (TV*)x.f.r;
    pb.rb = (TV*)x.f.s0;
  }
  const double c4 = double(1 << (2 * l));
  auto kern = fb ? k_mg_down_quad<B, TV, true> : k_mg_down_quad<B, TV, false>;
  cudaError_t e = allow_dynamic_smem(kern, sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((x.g.n_cubes + T::CPB - 1) / T::CPB), dim3(T::NT), sm, x.stream, x.g,
                    (const TV*)x.mg.r[l], (TV*)x.mg.r[l + 1],
                    B / 2 <= 4 ? (TV*)x.mg.x[l + 1] : (TV*)nullptr, all, pb, TV(kMgOmega / c4),
                    TV(c4), l);
}

template <int B, class TV>
static cudaError_t up_quad_t(const Ctx& x, int l, const SolveParams& prm, int mode, bool fb) {
  using T = QT<B, TV>;
  const size_t sm = sizeof(TV) * (size_t)T::N * T::CPB;
  const double c4 = double(1 << (2 * l));
  auto kern = k_mg_up_quad<B, TV>;
  cudaError_t e = allow_dynamic_smem(kern, sm);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((x.g.n_cubes + T::CPB - 1) / T::CPB), dim3(T::NT), sm, x.stream, x.g,
                    (const TV*)x.mg.r[l], fb ? (const TV*)x.f.s0 : (const TV*)nullptr,
                    (const TV*)x.mg.y[l + 1], (TV*)x.mg.y[l], prm, mode, TV(kMgOmega / c4), TV(c4),
                    l == 0 ? 1 : 0, l);
}

// First level of the coarse kernel: at most 4^3 cells per cube, and at most kCoarseCells cells
// (a launch over all SMs does more of them faster).  A block takes kCoarseBlock cells, up to
// the largest cluster: one SM does 1.7 FP64 operations a clock, so with 1024 cells a block
// these levels took longer than the launches they replaced.  FP64 steps in us (before the
// 8^3 tiles took two planes a thread) with a launch per level, with 16k cells and 1024 a block, and with these: 128 cubes of 4^3 2031, 2312,
// 1868; 1728 of 4^3 3408, 3485, 3128; 16 of 8^3 2577, 2998, 2556; 128 of 8^3 3341, 3592,
// 3084; 1024 of 16^3 31.4, 24.9, 24.3 ms.  2048 and 1024 cells, 256 and 64 a block: the same
// within 2 %.
constexpr long long kCoarseCells = 4096;
constexpr long long kCoarseBlock = 128;
static int coarse_from(const Ctx& x) {
  int l = 1;
  while (l < x.mg.L && ((x.B >> l) > 4 || (long long)x.g.n_cubes * (x.B >> l) * (x.B >> l) * (x.B >> l) >
                                              kCoarseCells))
    ++l;
  return l;
}
// aggregate levels of more than 1024 nodes, or that do not fit a block's shared memory, run on
// the cluster: levels k < coarse_kd
static int coarse_kd(const Ctx& x) {
  int kd = 0;
  while (kd < x.mg.M && (x.mg.n[kd] > 1024 || agg_smem(x.mg, x.g.n_cubes, kd) > 200 * 1024)) ++kd;
  return kd;
}
// The coarse kernel's launch as one cluster of `ranks` blocks; at: two attributes for cfg.
template <class TV>
static cudaError_t coarse_config(const Ctx& x, int ranks, cudaLaunchAttribute* at,
                                 cudaLaunchConfig_t* cfg) {
  const size_t sm = agg_smem(x.mg, x.g.n_cubes, coarse_kd(x));
  auto kern = k_mg_coarse<TV>;
  cudaError_t e = allow_dynamic_smem(kern, sm);
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
    return e;
  cfg->gridDim = dim3(ranks);
  cfg->blockDim = dim3(1024);
  cfg->dynamicSmemBytes = sm;
  cfg->stream = x.stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ranks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = at;
  cfg->numAttrs = 2;
  return cudaSuccess;
}
template <class TV>
static int coarse_limit_t(const Ctx& x) {
  for (int ranks = 16; ranks > 1; ranks /= 2) {
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg{};
    int n = 0;
    cudaError_t e = coarse_config<TV>(x, ranks, at, &cfg);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_mg_coarse<TV>, &cfg);
    if (e == cudaSuccess && n >= 1) return ranks;
    (void)cudaGetLastError();
  }
  return 1;
}
// Blocks of the largest cluster of the coarse kernel that the device runs for this grid: a
// device or partition may have fewer than 16 SMs in one GPC with the shared memory free (one
// block does all of it too).
int mg_cluster_limit(const Ctx& x) {
  return x.solve64 ? coarse_limit_t<double>(x) : coarse_limit_t<float>(x);
}
template <class TV>
static cudaError_t coarse_t(const Ctx& x, int lf, int all) {
  const int kd = coarse_kd(x);
  const long long bl = x.B >> lf, cells = x.g.n_cubes * bl * bl * bl;
  int ranks = 1;
  while (ranks < x.mg.cluster_max &&
         (cells > kCoarseBlock * ranks || (kd > 0 && x.mg.n[0] > 1024 * ranks)))
    ranks *= 2;
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg{};
  const cudaError_t e = coarse_config<TV>(x, ranks, at, &cfg);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_mg_coarse<TV>, x.g, x.mg, lf, (int)bl, kd, all);
}

template <class TV>
static cudaError_t vcycle_t(const Ctx& x, const SolveParams& prm, int mode) {
  const int all = mode == 2 ? 1 : 0;
  cudaError_t e;
  // the finest level of 8^3 and 16^3 cubes through the quad tile, which after
  // pass A also does the PCG's pass B; other cube sizes launch pass B first
  const bool tile = x.B == 8 || x.B == 16;
  const bool fb = tile && mode == 1;
  if (mode == 1 && !fb && (e = launch_cg_b(x, prm)) != cudaSuccess) return e;
  e = tile ? (x.B == 16 ? down_quad_t<16, TV>(x, 0, all, fb) : down_quad_t<8, TV>(x, 0, all, fb))
           : level_t<TV>(x, 0, true, all);
  if (e != cudaSuccess) return e;
  // levels of 8^3 cells per cube through the quad tile too, the smaller ones per cell down
  // to the level the coarse kernel takes over
  const int lf = coarse_from(x);
  for (int l = 1; l < lf; ++l)
    if ((e = (x.B >> l) == 8 ? down_quad_t<8, TV>(x, l, all, false)
                             : level_t<TV>(x, l, true, all)) != cudaSuccess)
      return e;
  if ((e = coarse_t<TV>(x, lf, all)) != cudaSuccess) return e;
  for (int l = lf - 1; l >= 1; --l)
    if ((e = (x.B >> l) == 8 ? up_quad_t<8, TV>(x, l, prm, mode, false)
                             : level_t<TV>(x, l, false, all)) != cudaSuccess)
      return e;
  if (tile) {
    e = x.B == 16 ? up_quad_t<16, TV>(x, 0, prm, mode, fb) : up_quad_t<8, TV>(x, 0, prm, mode, fb);
    if (e != cudaSuccess || mode == 2) return e;
    return launch_pdl(k_mg_decide, dim3(1), dim3(x.g.n_sims > 256 ? 256 : (x.g.n_sims + 31) / 32 * 32),
                      0, x.stream, x.g, prm, mode);
  }
  return x.B == 4 ? up0_t<4, TV>(x, prm, mode) : cudaErrorInvalidValue;
}

cudaError_t launch_mg_vcycle(const Ctx& x, const SolveParams& prm, int mode) {
  return x.solve64 ? vcycle_t<double>(x, prm, mode) : vcycle_t<float>(x, prm, mode);
}

}  // namespace bcm
