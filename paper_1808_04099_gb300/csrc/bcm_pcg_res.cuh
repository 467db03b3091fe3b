// bcm_pcg_res.cuh -- persistent Jacobi-PCG (Eq. poisson; Saad, Alg. 9.1) with the state of
// the iteration on chip, for grids whose vectors fit the registers and shared memory of
// one co-resident wave (one block per SM).
//
// Work items are z-slabs of cubes; block p owns a contiguous run of them (the paper's
// load-balanced linear distribution, Eq. loaddist), which is a contiguous range of the
// cube-major vectors.  Thread t keeps the quads (four cells along x) t, t + NT, ... of
// the range: in FP64 z = M^-1 r in registers (r itself is never stored: its recurrence scaled
// by the diagonal is z -= alpha M^-1 q), in FP32 r; the iterate x in registers where they
// suffice, the search direction p and K p / h in shared memory.  FP32 takes alpha over
// <p, K p> / h0 and adds up h0 x, so that one rounded factor steps both x and r: with z's
// factor rounded apart from x's, and r formed back from z in the sums, errors of one sign in
// all cells left a smooth error in the pressure that later iterations do not see (relative
// error at rtol 1e-12 on 246k cells 5.2e-13, now 1.6e-13; streaming form 1.4e-13).
// A cell's neighbours in other items are six ghost planes per item in shared memory, which
// hold the neighbours' p and are advanced by the same recurrence p = z + beta p as the cells
// themselves, so the only
// values that cross between blocks are the z of the items' face cells (fz, one plane per
// face, in L2).  An iteration is
//   pass A  p = z + beta p on the cells and the ghost planes; K p; <p, Kp>
//   wait for <p, Kp> of every block of the sim -> alpha
//   pass B  r (or z) -= alpha (M^-1) K p, x += alpha p; face z out; <r, z>, <r, r>
//   wait for <r, z>, <r, r> of every block of the sim -> beta, convergence.
//
// There is no grid barrier.  A block publishes each partial sum as one 16-byte word with
// the number of the iteration it belongs to, and a warp of every block that holds cells
// of the sim reads the words of that sim's blocks until all carry the iteration's number:
// the sum and the barrier are one message each way, sims do not wait for one another,
// and the order of the additions within a solve is fixed.  The waits end at
// barrier_timeout_ns (BCM_E_TIMEOUT).
//
// What bounds it: the two exchanges on small grids (2.2k cycles among 16 blocks, 3.1k
// among 152, with the sums 3-4k each); the FP64 pipe in FP64 (about 16 FP64 operations a
// cell and iteration, 20 counted on 64^3 with the ghost planes of its thin slabs; 1.7 a cycle
// and SM); instruction latency at 16 warps per SM on the largest FP32 grids.  Microseconds
// per iteration in two launches (FP64) or streaming (FP32), and here:
//   FP64  8k cells (16 cubes of 8^3) 28.8, 10.0; 64^3 48.2, 19.1; 524k (8^3) 47.9, 27.6
//   FP32  262k 13.0, 8.3; 524k (8^3) 15.1, 9.5; 24 sims, 312k cells 33.5, 10.4; 4.2M 32.5,
//         28.9
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "bcm_cube.cuh"
#include "bcm_internal.cuh"
#include "bcm_kernels.h"
#include "bcm_persist.cuh"
#include "bcm_quad.cuh"

namespace bcm {

namespace {

// A partial sum and the exchange it belongs to, one 128-bit access; each word has a line
// of its own.  Measured per exchange of one word among 152 blocks, cycles: words packed
// in shared lines 14.5k, in lines of their own read by one warp (five words a lane) 5.7k,
// by five warps (a word a lane) 3.1k; 2.2k among 16 blocks.
struct alignas(16) Word {
  double v;
  unsigned long long n;
};
struct alignas(256) WordLine {
  Word w;
};
constexpr int kWaitPer = 5;                 // words per lane of a warp that waits alone
constexpr int kResBlocks = 32 * kWaitPer;   // largest grid

__device__ __forceinline__ void word_put(Word* w, double v, unsigned long long n) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%0, %1};\n\tst.relaxed.gpu.global.b128 [%2], t;\n\t}" ::"l"(
                   __double_as_longlong(v)),
               "l"(n), "l"(w)
               : "memory");
}
__device__ __forceinline__ unsigned long long word_get(const Word* w, double& v) {
  long long a;
  unsigned long long n;
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(a), "=l"(n)
               : "l"(w)
               : "memory");
  v = __longlong_as_double(a);
  return n;
}
// After the block barrier and before a word: the block's writes come before the word.
// After the words of a wait: the other blocks' writes before their words are visible.
// (Acquire loads in the wait's loop instead would run one after another.)
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Shape of a launch, chosen on the host (res_shape).
struct ResShape {
  int lb, lk;          // log2 of the cube edge B and of the slab depth KS
  int ipb;             // items of the fullest block
  int mq;              // quads per thread whose K p / h is in shared memory (the rest: q)
  int multi;           // some block holds cells of several sims
  int o_g, o_q, o_item, o_21, o_tab, o_sim, o_red;  // byte offsets in dynamic shared memory
};

// Plane entries across the item's 2:1 faces (grids of two levels): of the coarse cell at the
// face's origin ([0]), or of the fine cells at the origin of each of its four parts (part
// 2 h + q: the half h of its rows, the half q of each row), which lie on one plane each.
struct ResFace21 {
  int at[6][4];
};

// Constants of one item.
template <class TV>
struct ResItem {
  int src[6];       // first entry of face f's source plane in fz, or -1: a 2:1 face
  int cube, slab;
  int sim;          // local index of its sim
  int tab;          // its 1/diag table
  unsigned w3;      // Jacobi face weights of the slab (3 bits each)
  unsigned flags;   // bit f: face f is a domain outflow (ghost -p); bits 8, 9, 10:
                    // some weight is not 3, some face is 2:1, an x face's weight is not 3; bits 16 + f / 24 + f: coarse, fine
  TV h, inv, dia;   // cell size (FP32: over the sim's h0), 1/diag and diag of a cell without
                    // special faces
};

struct ResSim {
  double alpha, beta, rz, rrz;  // rrz = 1 / rz
  double rz0, rr, tol2;         // <r, z> at entry, <r, r> of the last decision, the target
  double ih0;                   // 1 / h0
  int kdone;           // iterations this launch ran
  int done, first;
  int e0, cnt;         // the sim's words: first index and number of blocks
  int qa, qb;          // its quads in this block
};

// A waiting warp's view of the time: false when the wait ran out or another block's did.
__device__ __forceinline__ bool wait_on(int spin, unsigned long long& t0, volatile int* err,
                                        unsigned long long limit_ns) {
  int stop = 0;
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long t = global_ns();
    if (spin == 0) t0 = t;
    else if ((spin & 63) == 63 && *err) stop = 1;
    else if (t - t0 > limit_ns) {
      *err = 1;
      stop = 1;
    }
  }
  return !__any_sync(0xffffffffu, stop);
}
// The words of cnt blocks of one sim, read by one warp until all carry exchange number n
// (value a's words start at w + a * nE).
template <int NV, bool FENCE>
__device__ __forceinline__ bool warp_wait(const WordLine* __restrict__ w, int nE, int cnt,
                                          unsigned long long n, double (&v)[NV][kWaitPer],
                                          volatile int* err, unsigned long long limit_ns) {
  const int lane = threadIdx.x & 31;
  unsigned got = 0u, need = 0u;
#pragma unroll
  for (int u = 0; u < kWaitPer; ++u)
    if (lane + 32 * u < cnt) need |= ((1u << NV) - 1u) << (NV * u);
#pragma unroll
  for (int u = 0; u < kWaitPer; ++u)
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a][u] = 0.0;
  unsigned long long t0 = 0;
  for (int spin = 0;; ++spin) {
#pragma unroll
    for (int u = 0; u < kWaitPer; ++u)
#pragma unroll
      for (int a = 0; a < NV; ++a)
        if ((need & ~got) >> (NV * u + a) & 1u) {
          double x;
          if (word_get(&w[(size_t)a * nE + lane + 32 * u].w, x) == n) {
            v[a][u] = x;
            got |= 1u << (NV * u + a);
          }
        }
    if (__all_sync(0xffffffffu, got == need)) break;
    if (!wait_on(spin, t0, err, limit_ns)) return false;
  }
  if (FENCE) fence_gpu();
  return true;
}
// The same for a block of one sim: a word per lane, warps 0 .. ceil(cnt / 32) - 1 for each
// value; the values go to out[a * kResBlocks + block].
template <int NV, bool FENCE>
__device__ __forceinline__ bool block_wait(const WordLine* __restrict__ w, int nE, int cnt,
                                           unsigned long long n, double* out, volatile int* err,
                                           unsigned long long limit_ns) {
  const int per = (cnt + 31) >> 5, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int task = warp; task < NV * per; task += nw) {
    const int a = task / per, i = (task - a * per) * 32 + (threadIdx.x & 31);
    unsigned long long t0 = 0;
    for (int spin = 0;; ++spin) {
      double x = 0.0;
      const bool ok = i >= cnt || word_get(&w[(size_t)a * nE + i].w, x) == n;
      if (__all_sync(0xffffffffu, ok)) {
        if (i < cnt) out[a * kResBlocks + i] = x;
        break;
      }
      if (!wait_on(spin, t0, err, limit_ns)) return false;
    }
    if (FENCE) fence_gpu();
  }
  return true;
}
template <int NV>
__device__ __forceinline__ void words_sum(double (&v)[NV][kWaitPer], int cnt, double (&sum)[NV]) {
#pragma unroll
  for (int a = 0; a < NV; ++a) {
    double s = v[a][0];
    if (cnt > 32) s += v[a][1];
    if (cnt > 64) s += (v[a][2] + v[a][3]) + v[a][4];
    sum[a] = s;
  }
  const int lanes = cnt < 32 ? cnt : 32;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
    if (o < lanes) {
#pragma unroll
      for (int a = 0; a < NV; ++a) sum[a] += __shfl_xor_sync(0xffffffffu, sum[a], o);
    }
}

template <int NV>
__device__ __forceinline__ void wval_load(const double* wv, int cnt, double (&v)[NV][kWaitPer]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int a = 0; a < NV; ++a)
#pragma unroll
    for (int u = 0; u < kWaitPer; ++u)
      v[a][u] = lane + 32 * u < cnt ? wv[a * kResBlocks + lane + 32 * u] : 0.0;
}

// Block of item i under the linear distribution of N items over P blocks.
__device__ __forceinline__ int block_of_item(int i, int N, int P) {
  const int L = N / P, R = N % P;
  return i < R * (L + 1) ? i / (L + 1) : R + (i - R * (L + 1)) / L;
}

// Plane entry of cell (a, b) of face f of a cube in the items' face planes.
__device__ __forceinline__ int face_entry(const ResShape& sh, int cube, int f, int a, int b) {
  const int B = 1 << sh.lb, KS = 1 << sh.lk, G = 4 * KS * B + 2 * B * B, nsl = B >> sh.lk;
  if (f < 4) {
    const int s = b >> sh.lk;
    return (cube * nsl + s) * G + f * KS * B + ((b - s * KS) << sh.lb) + a;
  }
  return (cube * nsl + (f == 4 ? 0 : nsl - 1)) * G + 4 * KS * B + (f - 4) * B * B + (b << sh.lb) + a;
}

// The values of a 2:1 face's ghost at (a, b) (R7): fetch(cube, face, a, b) of the coarse
// cell across, or the mean over the four fine cells that touch the coarse face cell.
template <class TV, class Fetch>
__device__ __forceinline__ TV ghost_21(const DevGrid& g, const ResShape& sh, int c, int f, int a,
                                       int b, bool coarse, const Fetch& fetch) {
  const int d = f >> 1, B = 1 << sh.lb;
  if (coarse) {
    const int C = g.aux[(6 * c + f) * 4];
    if (!bcm_expect(g, C >= 0 && C < g.n_cubes, CHK_AUX)) return TV(0);
    const int sf = 1 << (g.max_level - g.lvl[c]), sc = 2 * sf;
    const int A = (g.ijk[3 * c + tan1(d)] + a * sf - g.ijk[3 * C + tan1(d)]) / sc;
    const int Bb = (g.ijk[3 * c + tan2(d)] + b * sf - g.ijk[3 * C + tan2(d)]) / sc;
    if (!bcm_expect(g, A >= 0 && A < B && Bb >= 0 && Bb < B, CHK_CELL)) return TV(0);
    return fetch(C, f ^ 1, A, Bb);
  }
  const int qa = (2 * a) >> sh.lb, qb = (2 * b) >> sh.lb;
  const int F = g.aux[(6 * c + f) * 4 + qb * 2 + qa];
  if (!bcm_expect(g, F >= 0 && F < g.n_cubes, CHK_AUX)) return TV(0);
  const int fa = 2 * a - qa * B, fb = 2 * b - qb * B;
  TV sum = TV(0);
  for (int bb = 0; bb < 2; ++bb)
    for (int aa = 0; aa < 2; ++aa) sum += fetch(F, f ^ 1, fa + aa, fb + bb);
  return TV(0.25) * sum;
}

// The entries of a ResFace21 for the R rows from b0 of face f of cube c.
__device__ __forceinline__ void face_21(const DevGrid& g, const ResShape& sh, int c, int f, int b0,
                                        int R, bool coarse, int (&at)[4]) {
  const int d = f >> 1, B = 1 << sh.lb;
  for (int u = 0; u < 4; ++u) at[u] = 0;
  if (coarse) {
    const int C = g.aux[(6 * c + f) * 4];
    if (!bcm_expect(g, C >= 0 && C < g.n_cubes, CHK_AUX)) return;
    const int sf = 1 << (g.max_level - g.lvl[c]), sc = 2 * sf;
    const int A = (g.ijk[3 * c + tan1(d)] - g.ijk[3 * C + tan1(d)]) / sc;
    const int Bb = (g.ijk[3 * c + tan2(d)] + b0 * sf - g.ijk[3 * C + tan2(d)]) / sc;
    if (!bcm_expect(g, A >= 0 && A < B && Bb >= 0 && Bb < B, CHK_CELL)) return;
    at[0] = face_entry(sh, C, f ^ 1, A, Bb);
    return;
  }
  for (int u = 0; u < 4; ++u) {
    const int tb = 2 * b0 + (u >> 1) * R, qb = tb >> sh.lb;
    const int F = g.aux[(6 * c + f) * 4 + 2 * qb + (u & 1)];
    if (bcm_expect(g, F >= 0 && F < g.n_cubes, CHK_AUX))
      at[u] = face_entry(sh, F, f ^ 1, 0, tb - qb * B);
  }
}

// v with its sign bit xor-ed by `sign` (an integer operation: FP64 ones are dear)
__device__ __forceinline__ float flip(float v, unsigned sign) {
  return __uint_as_float(__float_as_uint(v) ^ sign);
}
__device__ __forceinline__ double flip(double v, unsigned sign) {
  return __hiloint2double(__double2hiint(v) ^ (int)sign, __double2loint(v));
}

// face planes are read through L2, where the other blocks' stores are
__device__ __forceinline__ void ldcg4(const float* p, float (&v)[4]) {
  const float4 t = __ldcg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ldcg4(const double* p, double (&v)[4]) {
  const double2 a = __ldcg(reinterpret_cast<const double2*>(p));
  const double2 b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

__device__ __forceinline__ void ldcg2(const float* p, float (&v)[2]) {
  const float2 t = __ldcg(reinterpret_cast<const float2*>(p));
  v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void ldcg2(const double* p, double (&v)[2]) {
  const double2 t = __ldcg(reinterpret_cast<const double2*>(p));
  v[0] = t.x; v[1] = t.y;
}

// ---------------------------------------------------------------- the kernel
//
// M: quads per thread.  GEO: 0, or the cube edge B of whole-cube items, whose positions
// and shared-memory offsets are then compile-time functions of (thread, m).  XR: the
// iterate x in registers, else in global memory.  The K p of the last MQR quads stays in
// registers.
template <class TV, int NT, int M, int GEO, bool XR, int MQR>
__global__ __launch_bounds__(NT, 1) void k_pcg_res(DevGrid g, ResShape sh, TV* __restrict__ x,
                                                   const TV* __restrict__ r, TV* __restrict__ p,
                                                   TV* __restrict__ q, TV* __restrict__ fz,
                                                   WordLine* __restrict__ words,
                                                   SolveParams prm, int* err) {
  constexpr bool kD = sizeof(TV) == 8;
  // 2:1 ghosts through ResFace21, whose loads are independent, where registers are left for
  // them (the FP64 and the largest FP32 kernels spill), else cell by cell through the cubes'
  // tables, 4-5 us of an iteration: FP32 two-level grids of 188 cubes of 8^3 12.4 -> 8.1 us,
  // 1648 20.0 -> 12.5, 188 of 16^3 19.2 -> 11.8 (the streaming form takes 12.1, 29.8, 19.8)
  constexpr bool kTab = !kD && M <= 8;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int kLb = GEO == 16 ? 4 : GEO == 8 ? 3 : 2;
  const int lb = GEO ? kLb : sh.lb, lk = GEO ? kLb : sh.lk;
  const int B = 1 << lb, BB = B << lb, KS = 1 << lk;
  const int li = 2 * lb + lk, IC = 1 << li;       // cells per item
  const int FX = KS << lb, G = 4 * FX + 2 * BB;   // entries of an x/y face, per item
  TV* sp = reinterpret_cast<TV*>(sm);
  const int og = sh.o_g / (int)sizeof(TV);        // the ghost planes, from sp
  TV* sg = sp + og;
  TV* sq = reinterpret_cast<TV*>(sm + sh.o_q);
  ResItem<TV>* items = reinterpret_cast<ResItem<TV>*>(sm + sh.o_item);
  ResFace21* const f21 = reinterpret_cast<ResFace21*>(sm + sh.o_21);
  TV* tab = reinterpret_cast<TV*>(sm + sh.o_tab);
  ResSim* sims = reinterpret_cast<ResSim*>(sm + sh.o_sim);
  double* red = reinterpret_cast<double*>(sm + sh.o_red);
  __shared__ double wval[2 * kResBlocks];  // the words of a wait
  __shared__ int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool inner = prm.mixed != 0, multi = sh.multi != 0;
  const int kmax = inner ? prm.inner_max_iter : prm.max_iter;
  const int nsl = B >> lk;
  const int N = g.n_cubes * nsl, P = gridDim.x, bl = blockIdx.x;
  const int Lq = N / P, Rq = N % P;
  const int item0 = bl * Lq + min(bl, Rq), nit = Lq + (bl < Rq ? 1 : 0);
  const int NQ = (nit << li) >> 2;                // quads of this block
  const size_t base = (size_t)item0 << li;        // its first cell
  const int sim_lo = g.sim[item0 / nsl], nls = g.sim[(item0 + nit - 1) / nsl] - sim_lo + 1;
  const int nE = P + g.n_sims;                    // word lines per exchange

  // ---- tables of the block: items, sims, 1/diag and diag
  for (int it = tid; it < nit; it += NT) {
    ResItem<TV>& I = items[it];
    const int item = item0 + it, c = item / nsl, slab = item - c * nsl;
    int s = g.sim[c], lv = g.lvl[c];
    if (!bcm_expect(g, s >= 0 && s < g.n_sims && lv >= 0 && lv <= g.max_level, CHK_SIM)) s = lv = 0;
    const SimParams& P0 = g.sp[s];
    unsigned w3 = 0, fl = 0;
    for (int f = 0; f < 6; ++f) {
      // a face inside the cube (between its slabs) is a same-level face to the next slab
      const bool inside = (f == 4 && slab > 0) || (f == 5 && slab < nsl - 1);
      const int n = inside ? 0 : checked_nb(g, g.nb[6 * c + f]);
      const int w = inside ? 3 : g.w3[6 * c + f];
      w3 |= (unsigned)w << (3 * f);
      if (w != 3) fl |= f < 2 ? 5u << 8 : 1u << 8;
      const int off = f < 4 ? f * FX : 4 * FX + (f - 4) * BB;
      if (inside) {
        I.src[f] = (item + (f == 4 ? -1 : 1)) * G + 4 * FX + (f == 4 ? BB : 0);
      } else if (n >= 0) {
        const int fo = f ^ 1, oo = fo < 4 ? fo * FX : 4 * FX + (fo - 4) * BB;
        I.src[f] = (n * nsl + (f < 4 ? slab : f == 4 ? nsl - 1 : 0)) * G + oo;
      } else if (n == NB_BOUNDARY) {  // the ghost follows this item's own face cells
        I.src[f] = item * G + off;
        if (P0.bc[f] == BC_OUTFLOW) fl |= 1u << f;
      } else {
        I.src[f] = -1;
        fl |= (1u << 9) | (n == NB_COARSE ? 1u << (16 + f) : 1u << (24 + f));
        if (kTab) face_21(g, sh, c, f, f < 4 ? slab * KS : 0, f < 4 ? KS : B, n == NB_COARSE, f21[it].at[f]);
      }
    }
    I.cube = c;
    I.slab = slab;
    I.sim = s - sim_lo;
    I.tab = ((s - sim_lo) * (g.max_level + 1) + lv) * kW3;
    I.w3 = w3;
    I.flags = fl;
    I.h = TV((kD ? P0.h0 : 1.0) / double(1 << lv));
    I.inv = TV(P0.invdiag[lv][18]);
    I.dia = TV(1) / I.inv;
  }
  const int ntab = nls * (g.max_level + 1) * kW3;  // 1/diag, then diag
  for (int i = tid; i < ntab; i += NT) {
    const int w = i % kW3, sl = i / kW3;
    tab[i] = TV(g.sp[sim_lo + sl / (g.max_level + 1)].invdiag[sl % (g.max_level + 1)][w]);
    tab[ntab + i] = tab[i] > TV(0) ? TV(1) / tab[i] : TV(0);
  }
  for (int l = tid; l < nls; l += NT) {
    ResSim& S = sims[l];
    const int s = sim_lo + l;
    SimState& st = g.ss[s];
    const bool cont = st.cont != 0;
    S.alpha = S.beta = 0.0;
    S.rz = cont ? st.rz_last : st.rz;
    S.rz0 = st.rz;
    S.rr = st.rr;
    S.tol2 = inner ? st.inner_tol2 : st.tol2;
    S.rrz = S.rz != 0.0 ? 1.0 / S.rz : 0.0;
    S.ih0 = 1.0 / g.sp[s].h0;
    S.done = st.done ? 1 : 0;
    S.kdone = 0;
    S.first = cont ? 0 : 1;
    const int ia = g.sp[s].cube_begin * nsl, ib = g.sp[s].cube_end * nsl;
    const int b0 = block_of_item(ia, N, P), b1 = block_of_item(ib - 1, N, P);
    S.e0 = b0 + s;
    S.cnt = b1 - b0 + 1;
    S.qa = (max(ia - item0, 0) << li) >> 2;
    S.qb = (min(ib - item0, nit) << li) >> 2;
  }
  if (tid == 0) s_fail = 0;
  poison_tile(sp, nit << li);
  poison_tile(sg, nit * G);
  __syncthreads();
  bool any = false;
  for (int l = 0; l < nls; ++l) any |= !sims[l].done;
  if (bl == 0 && tid == 0) g.flags[0] = 1;
  if (!any) return;

  // item and position of quad m of thread tid; false beyond the block's cells.  Each pass
  // takes tid through opaque(): else the compiler keeps every quad's offsets in registers
  // across the iterations and spills.
  auto opaque = [&]() {
    int t = threadIdx.x;
    asm volatile("" : "+r"(t));
    return t;
  };
  // With GEO a thread's quads m = 2n, 2n + 1 lie one above the other (planes kk, kk + 1),
  // so pass A takes their common z neighbours from registers.
  auto quad = [&](int tid, int m, int& it, int& i0, int& j, int& kk) {
    if constexpr (GEO != 0) {
      constexpr int kT = GEO * GEO * GEO / 8;  // threads per item (two planes each)
      const int in = tid & (kT - 1);
      i0 = (4 * in) & (GEO - 1);
      j = ((4 * in) >> kLb) & (GEO - 1);
      kk = 2 * ((4 * in) >> (2 * kLb)) + (m & 1);
      it = (m >> 1) * (NT / kT) + tid / kT;
      return it < nit;
    } else {
      const int qd = tid + m * NT, cell = qd << 2, in = cell & (IC - 1);
      it = cell >> li;
      i0 = in & (B - 1);
      j = (in >> lb) & (B - 1);
      kk = in >> (2 * lb);
      return qd < NQ;
    }
  };
  auto cell0 = [&](int it, int i0, int j, int kk) {
    return (it << li) + (((kk << lb) + j) << lb) + i0;
  };
  // face-weight sums (thirds) of the four cells of a quad, 8 bits each
  auto s3q = [&](const ResItem<TV>& I, int i0, int j, int kk) {
    const unsigned w = I.w3;
    auto wf = [&](int f) { return (int)(w >> (3 * f) & 7u) - 3; };
    int sa = 18;
    if (j == 0) sa += wf(2);
    if (j == B - 1) sa += wf(3);
    if (kk == 0) sa += wf(4);
    if (kk == KS - 1) sa += wf(5);
    unsigned v = (unsigned)sa * 0x01010101u;
    if (i0 == 0) v += (unsigned)wf(0);
    if (i0 == B - 4) v += (unsigned)wf(1) << 24;
    return v;
  };
  // the cells' z on the item's faces, for the neighbours' ghosts
  auto put_faces = [&](int it, int i0, int j, int kk, const TV (&zv)[4]) {
    TV* F = fz + (size_t)(item0 + it) * G;
    if (i0 == 0) __stcg(F + (kk << lb) + j, zv[0]);
    if (i0 == B - 4) __stcg(F + FX + (kk << lb) + j, zv[3]);
    if (j == 0) st4(F + 2 * FX + (kk << lb) + i0, zv);
    if (j == B - 1) st4(F + 3 * FX + (kk << lb) + i0, zv);
    if (kk == 0) st4(F + 4 * FX + (j << lb) + i0, zv);
    if (kk == KS - 1) st4(F + 4 * FX + BB + (j << lb) + i0, zv);
  };
  // 1 / diag of the four cells of a quad
  auto quad_invs = [&](const ResItem<TV>& I, int i0, int j, int kk, TV (&iv)[4]) {
    if (I.flags >> 8 & 1u) {
      const unsigned v = s3q(I, i0, j, kk);
#pragma unroll
      for (int e = 0; e < 4; ++e) iv[e] = tab[I.tab + (int)(v >> (8 * e) & 255u)];
    } else {
      iv[0] = iv[1] = iv[2] = iv[3] = I.inv;
    }
  };
  auto live = [&](int it) { return !multi || !sims[items[it].sim].done; };
  auto sim_at = [&](int it) -> const ResSim& { return sims[multi ? items[it].sim : 0]; };

  // ---- state at entry
  TV z[M][4];  // FP64: z; FP32: r
  TV xr[XR ? M : 1][4];
  TV qr[MQR ? MQR : 1][4];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    int it, i0, j, kk;
    if (!quad(tid, m, it, i0, j, kk) || !live(it)) continue;
    const ResItem<TV>& I = items[it];
    const int c0 = cell0(it, i0, j, kk);
    TV rv[4], pv[4] = {TV(0), TV(0), TV(0), TV(0)};
    ld4(r + base + c0, rv);
    if (!sim_at(it).first) ld4(p + base + c0, pv);
    if constexpr (XR) {
      if (inner) xr[m][0] = xr[m][1] = xr[m][2] = xr[m][3] = TV(0);
      else ld4(x + base + c0, xr[m]);
    }
    st4(sp + c0, pv);
    TV iv[4], zv[4];
    quad_invs(I, i0, j, kk, iv);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      zv[e] = rv[e] * iv[e];
      z[m][e] = kD ? zv[e] : rv[e];
    }
    put_faces(it, i0, j, kk, zv);
  }
  // face f and position t on it of entry o of an item's planes
  auto plane = [&](int o, int& f, int& t) {
    f = o < 4 * FX ? o >> (lb + lk) : 4 + ((o - 4 * FX) >> (2 * lb));
    t = o - (f < 4 ? f * FX : 4 * FX + (f - 4) * BB);
  };
  // ghost planes of a kept search direction, from the neighbours' cells
  for (int e = tid; e < nit * G; e += NT) {
    const int it = e / G, o = e - it * G;
    const ResItem<TV>& I = items[it];
    TV v = TV(0);
    if (live(it) && !sim_at(it).first) {
      int f, t;
      plane(o, f, t);
      const int a = t & (B - 1), b = (t >> lb) + (f < 4 ? I.slab * KS : 0);
      auto cell = [&](int cube, int ff, int aa, int bb) {
        const int d = ff >> 1, n = (ff & 1) ? B - 1 : 0;
        int qq[3];
        qq[d] = n;
        qq[tan1(d)] = aa;
        qq[tan2(d)] = bb;
        return p[((size_t)cube << (3 * lb)) + (((qq[2] << lb) + qq[1]) << lb) + qq[0]];
      };
      if ((f == 4 && I.slab > 0) || (f == 5 && I.slab < nsl - 1)) {
        const int kz = f == 4 ? I.slab * KS - 1 : (I.slab + 1) * KS;
        v = p[((size_t)I.cube << (3 * lb)) + (((kz << lb) + (t >> lb)) << lb) + a];
      } else if (I.src[f] < 0) {
        v = ghost_21<TV>(g, sh, I.cube, f, a, b, I.flags >> (16 + f) & 1u, cell);
      } else {
        const int n = checked_nb(g, g.nb[6 * I.cube + f]);
        v = n >= 0 ? cell(n, f ^ 1, a, b) : cell(I.cube, f, a, b);
        if (I.flags >> f & 1u) v = -v;
      }
    }
    sg[e] = v;
  }

  // Sums of NV values per thread (several sims: per thread and quad), published under
  // exchange number n.  One sim: t[] is the thread's sum.  Several: each quad's values
  // were reduced over units of 16 quads, which never cross an item (res_shape), into red[].
  auto unit_sum = [&](int unit, int a, TV t) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((lane & 15) == 0 && unit < M * NT / 16) red[a * (M * NT / 16) + unit] = double(t);
  };
  auto publish = [&](auto NVc, WordLine* w, unsigned long long n, bool fence, const TV* t) {
    constexpr int NV = decltype(NVc)::value;
    if (!multi) {
      double s = 0.0;
      if constexpr (kD) {
        // FP64 adds are slow (16 cycles a warp, 64 of latency): each partial is added
        // once, by whole lanes
#pragma unroll
        for (int a = 0; a < NV; ++a) red[a * NT + tid] = t[a];
        __syncthreads();
        if (warp < NV) {
          double s4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
          for (int u = 0; u < NW; ++u) s4[u & 3] += red[warp * NT + 32 * u + lane];
          s = warp_sum((s4[0] + s4[1]) + (s4[2] + s4[3]));
        }
      } else {
#pragma unroll
        for (int a = 0; a < NV; ++a) {
          TV f = t[a];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
          if (lane == 0) red[a * NW + warp] = double(f);
        }
        __syncthreads();
        if (warp < NV) {
          s = red[warp * NW + (lane & (NW - 1))];
#pragma unroll
          for (int o = NW / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        }
      }
      if (warp < NV && lane == 0) {
        if (fence) fence_gpu();
        word_put(&w[(size_t)warp * nE + bl + sim_lo].w, s, n);
      }
    } else {
      __syncthreads();
      for (int l = warp; l < nls; l += NW) {
        if (sims[l].done) continue;
#pragma unroll
        for (int a = 0; a < NV; ++a) {
          double s = 0.0;
          for (int u = (sims[l].qa >> 4) + lane; u < sims[l].qb >> 4; u += 32)
            s += red[a * (M * NT / 16) + u];
          s = warp_sum(s);
          if (lane == 0) {
            if (fence) fence_gpu();
            word_put(&w[(size_t)a * nE + bl + sim_lo + l].w, s, n);
          }
        }
      }
    }
  };
  WordLine* const wa = words;       // <p, Kp>
  WordLine* const wb = words + nE;  // <r, z>, <r, r>
  using One = std::integral_constant<int, 1>;
  using Two = std::integral_constant<int, 2>;

  // the end of sim l after k iterations (lane 0 of a warp; the same in every block)
  auto finish = [&](int l, int k, double rr, bool ok, bool bad) {
    ResSim& S = sims[l];
    SimState& st = g.ss[sim_lo + l];
    S.done = 1;
    S.kdone = k;
    if (bl + sim_lo + l != S.e0) return;  // the sim's first block writes the results
    st.iter = k;
    st.total_iters += k;
    st.rr = rr;
    st.done = 1;
    st.rz_last = S.rz;
    st.p_off = 0;
    if (bad) st.nonfinite = 1;
    if (!inner) {
      st.rr64 = rr;
      st.converged = ok;
    }
  };
  // decisions of sim l from the sums of the previous pass B
  auto decide = [&](int l, int k, double rz, double rr) {
    ResSim& S = sims[l];
    if (k == 0) {
      rz = S.rz0;
      rr = S.rr;
    }
    const double tol2 = S.tol2;
    const bool bad = !isfinite(rr) || !isfinite(rz);
    if (bad || rr <= tol2 || k >= kmax) {
      finish(l, k, rr, !bad && rr <= tol2, bad);
      return;
    }
    S.rr = rr;
    S.beta = ((k == 0 && S.first) || S.rz == 0.0) ? 0.0 : quick_div(rz, S.rz, S.rrz);
    S.rz = rz;
  };

  {
    const TV t0[2] = {TV(0), TV(0)};
    if (multi) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        int it, i0, j, kk;
        quad(tid, m, it, i0, j, kk);
        unit_sum(cell0(it, i0, j, kk) >> 6, 0, TV(0));
        unit_sum(cell0(it, i0, j, kk) >> 6, 1, TV(0));
      }
    }
    publish(Two{}, wb, 1ull, true, t0);
  }
  // Ghost planes: thread t takes quad t % (G / 4) of the planes of items git, git + gips, ...
  // (the threads past the last whole item take none)
  constexpr int GU = M >= 8 ? 4 : 2;  // ghost quads in flight per thread
  const int gips = NT / (G >> 2), go = 4 * (tid % (G >> 2));
  const int git = tid / (G >> 2) < gips ? tid / (G >> 2) : nit;
  int gf, gt;
  plane(go, gf, gt);
  bool failed = false;
  for (int k = 0;; ++k) {
    // ---- wait for the sums of the previous pass B.  Once the words are there the
    // neighbours' face values are too: they are loaded while the sums are formed.
    double v[2][kWaitPer];
    const unsigned long long nb = (unsigned long long)k + 1;
    if (!multi) {
      if (!block_wait<2, true>(wb + sims[0].e0, nE, sims[0].cnt, nb, wval, err,
                               prm.barrier_timeout_ns))
        s_fail = 1;
    } else {
      for (int l = warp; l < nls; l += NW) {
        if (sims[l].done) continue;
        if (!warp_wait<2, true>(wb + sims[l].e0, nE, sims[l].cnt, nb, v, err, prm.barrier_timeout_ns)) {
          if (lane == 0) s_fail = 1;
          continue;
        }
        double s[2];
        words_sum<2>(v, sims[l].cnt, s);
        if (lane == 0) decide(l, k, s[0], s[1]);
      }
    }
    __syncthreads();
    if (s_fail) {
      failed = true;
      break;
    }
    const int tid = opaque();
    TV gz[GU][4];
    auto ghost_load = [&](int it, TV (&zv)[4]) {
      const ResItem<TV>& I = items[it];
      const int src = I.src[gf];
      if (src >= 0) {
        ldcg4(fz + src + gt, zv);
      } else {
        if constexpr (kTab) {
          const int* at = f21[it].at[gf];
          const int a = gt & (B - 1), b = gt >> lb;
          if (I.flags >> (16 + gf) & 1u) {
            TV w[2];
            ldcg2(fz + at[0] + ((b >> 1) << lb) + (a >> 1), w);
            zv[0] = zv[1] = w[0];
            zv[2] = zv[3] = w[1];
          } else {
            const int lr = gf < 4 ? lk : lb, hh = b >> (lr - 1), row = (2 * b - (hh << lr)) << lb;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int q = 2 * a + 4 * u, qa = q >> lb;
              const TV* F = fz + at[2 * hh + qa] + row + (q - (qa << lb));
              TV lo[4], hi[4];
              ldcg4(F, lo);
              ldcg4(F + B, hi);
              zv[2 * u] = TV(0.25) * (((lo[0] + lo[1]) + hi[0]) + hi[1]);
              zv[2 * u + 1] = TV(0.25) * (((lo[2] + lo[3]) + hi[2]) + hi[3]);
            }
          }
        } else {
          auto fetch = [&](int cube, int ff, int aa, int bb) {
            return __ldcg(fz + face_entry(sh, cube, ff, aa, bb));
          };
          const int b = (gt >> lb) + (gf < 4 ? I.slab * KS : 0);
#pragma unroll 1
          for (int u = 0; u < 4; ++u)
            zv[u] = ghost_21<TV>(g, sh, I.cube, gf, (gt & (B - 1)) + u, b, I.flags >> (16 + gf) & 1u, fetch);
        }
      }
    };
    auto ghost_step = [&](int it, TV (&zv)[4]) {
      if (!live(it)) return;
      const unsigned sign = (items[it].flags >> gf & 1u) << 31;
#pragma unroll
      for (int u = 0; u < 4; ++u) zv[u] = flip(zv[u], sign);
      TV pv[4];
      ld4(sg + it * G + go, pv);
      axpy4(TV(sim_at(it).beta), pv, zv, pv);
      st4(sg + it * G + go, pv);
    };
#pragma unroll
    for (int u = 0; u < GU; ++u)
      if (git + u * gips < nit) ghost_load(git + u * gips, gz[u]);
    if (!multi && warp == 0) {
      double s[2];
      wval_load<2>(wval, sims[0].cnt, v);
      words_sum<2>(v, sims[0].cnt, s);
      if (lane == 0) decide(0, k, s[0], s[1]);
    }
    __syncthreads();
    any = false;
    for (int l = 0; l < nls; ++l) any |= !sims[l].done;
    if (!any) break;
    // ---- pass A: p = z + beta p, on the ghost planes and the cells
#pragma unroll
    for (int u = 0; u < GU; ++u)
      if (git + u * gips < nit) ghost_step(git + u * gips, gz[u]);
    for (int it0 = git + GU * gips; it0 < nit; it0 += GU * gips) {
#pragma unroll
      for (int u = 0; u < GU; ++u)
        if (it0 + u * gips < nit) ghost_load(it0 + u * gips, gz[u]);
#pragma unroll
      for (int u = 0; u < GU; ++u)
        if (it0 + u * gips < nit) ghost_step(it0 + u * gips, gz[u]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
      int it, i0, j, kk;
      if (!quad(tid, m, it, i0, j, kk) || !live(it)) continue;
      const TV beta = TV(sim_at(it).beta);
      TV pv[4];
      const int c0 = cell0(it, i0, j, kk);
      ld4(sp + c0, pv);
      if constexpr (kD) {
        axpy4(beta, pv, z[m], pv);
      } else {
        TV iv[4];
        quad_invs(items[it], i0, j, kk, iv);
        mul4(z[m], iv, iv);
        axpy4(beta, pv, iv, pv);
      }
      st4(sp + c0, pv);
    }
    __syncthreads();
    // ---- pass A: K p / h, <p, Kp>
    // K p / h of a quad from its cells and neighbours; returns <p, K p / h>
    auto apply = [&](const ResItem<TV>& I, int i0, int j, int kk, const TV (&pc)[4], TV xl, TV xh,
                     const TV (&ym)[4], const TV (&yp)[4], const TV (&zm)[4], const TV (&zp)[4],
                     TV (&acc)[4]) {
      seven_point(pc, xl, xh, ym, yp, zm, zp, acc);
      if (I.flags >> 9 & 1u) {  // 2:1 faces: weight 2/3 on the fine side, 4/3 on the coarse
        auto wt = [&](int f) {
          return (I.flags >> (16 + f) & 1u) ? TV(2.0 / 3.0) - TV(1)
                 : (I.flags >> (24 + f) & 1u) ? TV(4.0 / 3.0) - TV(1) : TV(0);
        };
        if (i0 == 0) acc[0] += wt(0) * (pc[0] - xl);
        if (i0 == B - 4) acc[3] += wt(1) * (pc[3] - xh);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (j == 0) acc[e] += wt(2) * (pc[e] - ym[e]);
          if (j == B - 1) acc[e] += wt(3) * (pc[e] - yp[e]);
          if (kk == 0) acc[e] += wt(4) * (pc[e] - zm[e]);
          if (kk == KS - 1) acc[e] += wt(5) * (pc[e] - zp[e]);
        }
      }
      return dot4(pc, acc);
    };
    auto keep = [&](int m, int c0, const TV (&acc)[4]) {  // K p / h for pass B
      if (m >= M - MQR) {
        if constexpr (MQR > 0) {
#pragma unroll
          for (int e = 0; e < 4; ++e) qr[m >= M - MQR ? m - (M - MQR) : 0][e] = acc[e];
        }
      } else if (m < sh.mq) {  // the thread's own: any layout
        st4(sq + 4 * (m * NT + threadIdx.x), acc);
      } else {
        st4(q + base + c0, acc);
      }
    };
    TV pq[1] = {TV(0)};
    const int tid_a = opaque();
    if constexpr (GEO != 0) {
#pragma unroll
      for (int m = 0; m < M; m += 2) {
        TV part[2] = {TV(0), TV(0)};
        int it, i0, j, kk;
        // (an item takes whole warps, so the shuffles below are not divergent)
        if (quad(tid_a, m, it, i0, j, kk) && live(it)) {
          const ResItem<TV>& I = items[it];
          const int c0 = cell0(it, i0, j, kk), gi = og + it * G;
          TV pc[2][4], zm[4], zp[4];
          ld4(sp + c0, pc[0]);
          ld4(sp + c0 + BB, pc[1]);
          ld4(sp + (kk > 0 ? c0 - BB : gi + 4 * FX + (j << lb) + i0), zm);
          ld4(sp + (kk < KS - 2 ? c0 + 2 * BB : gi + 4 * FX + BB + (j << lb) + i0), zp);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int k2 = kk + u, cu = c0 + u * BB;
            TV ym[4], yp[4], acc[4];
            ld4(sp + (j > 0 ? cu - B : gi + 2 * FX + (k2 << lb) + i0), ym);
            ld4(sp + (j < B - 1 ? cu + B : gi + 3 * FX + (k2 << lb) + i0), yp);
            TV xl = __shfl_up_sync(0xffffffffu, pc[u][3], 1);
            TV xh = __shfl_down_sync(0xffffffffu, pc[u][0], 1);
            if (i0 == 0) xl = sp[gi + (k2 << lb) + j];
            if (i0 == B - 4) xh = sp[gi + FX + (k2 << lb) + j];
            if (u == 0) part[u] = apply(I, i0, j, k2, pc[0], xl, xh, ym, yp, zm, pc[1], acc);
            else part[u] = apply(I, i0, j, k2, pc[1], xl, xh, ym, yp, pc[0], zp, acc);
            part[u] *= I.h;
            keep(m + u, cu, acc);
          }
        }
        if (multi) {
          unit_sum(cell0(it, i0, j, kk) >> 6, 0, part[0]);
          unit_sum(cell0(it, i0, j, kk + 1) >> 6, 0, part[1]);
        } else {
          pq[0] += part[0] + part[1];
        }
      }
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        TV part = TV(0);
        int it, i0, j, kk;
        if (quad(tid_a, m, it, i0, j, kk) && live(it)) {
          const ResItem<TV>& I = items[it];
          const int c0 = cell0(it, i0, j, kk), gi = og + it * G;
          TV pc[4], ym[4], yp[4], zm[4], zp[4], acc[4];
          ld4(sp + c0, pc);
          ld4(sp + (j > 0 ? c0 - B : gi + 2 * FX + (kk << lb) + i0), ym);
          ld4(sp + (j < B - 1 ? c0 + B : gi + 3 * FX + (kk << lb) + i0), yp);
          ld4(sp + (kk > 0 ? c0 - BB : gi + 4 * FX + (j << lb) + i0), zm);
          ld4(sp + (kk < KS - 1 ? c0 + BB : gi + 4 * FX + BB + (j << lb) + i0), zp);
          const TV xl = sp[i0 > 0 ? c0 - 1 : gi + (kk << lb) + j];
          const TV xh = sp[i0 < B - 4 ? c0 + 4 : gi + FX + (kk << lb) + j];
          part = I.h * apply(I, i0, j, kk, pc, xl, xh, ym, yp, zm, zp, acc);
          keep(m, c0, acc);
        }
        if (multi) unit_sum(cell0(it, i0, j, kk) >> 6, 0, part);
        else pq[0] += part;
      }
    }
    // (no fence: nothing another block reads has been written since the last exchange)
    publish(One{}, wa, nb, false, pq);
    // A non-finite <p, Kp> ends an FP64 solve before it touches x, as in the two-launch form
    // (the FP32 inner solve runs on with alpha = 0, as the streaming form does).
    auto set_alpha = [&](int l, double (&va)[1][kWaitPer]) {
      ResSim& S = sims[l];
      double s[1];
      words_sum<1>(va, S.cnt, s);
      // lane 0: alpha = <r, z> / <p, Kp>; lane 1: 1 / <r, z> for the next beta
      const double d = lane == 0 ? s[0] : S.rz, y = quick_rcp(d);
      if (lane == 0) {
        S.alpha = (d != 0.0 && isfinite(d)) ? quick_div(S.rz, d, y) : 0.0;
        if (kD && !isfinite(d)) finish(l, k, S.rr, false, true);
      }
      if (lane == 1) S.rrz = y;
    };
    double va[1][kWaitPer];
    if (!multi) {
      if (!block_wait<1, false>(wa + sims[0].e0, nE, sims[0].cnt, nb, wval, err,
                                prm.barrier_timeout_ns))
        s_fail = 1;
      __syncthreads();
      if (warp == 0) {
        wval_load<1>(wval, sims[0].cnt, va);
        set_alpha(0, va);
      }
    } else {
      for (int l = warp; l < nls; l += NW) {
        if (sims[l].done) continue;
        if (!warp_wait<1, false>(wa + sims[l].e0, nE, sims[l].cnt, nb, va, err,
                                 prm.barrier_timeout_ns)) {
          if (lane == 0) s_fail = 1;
          continue;
        }
        set_alpha(l, va);
      }
    }
    __syncthreads();
    if (s_fail) {
      failed = true;
      break;
    }
    if (kD && !multi && sims[0].done) break;
    // ---- pass B: the residual's step, face planes, <r, z>, <r, r>
    TV rs[2] = {TV(0), TV(0)};
    const int tid_b = opaque();
#pragma unroll
    for (int m = 0; m < M; ++m) {
      TV rz = TV(0), rr = TV(0);
      int it, i0, j, kk;
      if (quad(tid_b, m, it, i0, j, kk) && live(it)) {
        const ResItem<TV>& I = items[it];
        const int c0 = cell0(it, i0, j, kk);
        TV acc[4];
        if (m < M - MQR) {
          if (m < sh.mq) ld4(sq + 4 * (m * NT + threadIdx.x), acc);
          else ld4(q + base + c0, acc);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = qr[m - (M - MQR) > 0 ? m - (M - MQR) : 0][e];
        }
        const TV ah = TV(sim_at(it).alpha) * I.h;
        if constexpr (kD) {
          // one diagonal value in the quad (bar its ends in a cube at an x domain face)
          const unsigned v4 = (I.flags >> 8 & 1u) ? s3q(I, i0, j, kk) : 0x12121212u;
          const int w = I.tab + (int)(v4 >> 8 & 255u);
          const TV t = ah * tab[w], dia = tab[ntab + w];
          if (!(I.flags >> 10 & 1u)) {
            axpy4(-t, acc, z[m], z[m]);
            rz = dot4(z[m], z[m]) * dia;
            rr = rz * dia;
          } else {
            const int w0 = I.tab + (int)(v4 & 255u), w1 = I.tab + (int)(v4 >> 24);
            z[m][0] -= ah * tab[w0] * acc[0];
            z[m][1] -= t * acc[1];
            z[m][2] -= t * acc[2];
            z[m][3] -= ah * tab[w1] * acc[3];
            const TV r0 = z[m][0] * tab[ntab + w0], r3 = z[m][3] * tab[ntab + w1];
            const TV r12 = (z[m][1] * z[m][1] + z[m][2] * z[m][2]) * dia;
            rz = z[m][0] * r0 + (z[m][3] * r3 + r12);
            rr = r0 * r0 + (r3 * r3 + r12 * dia);
          }
          put_faces(it, i0, j, kk, z[m]);
        } else {
          TV zv[4];
          quad_invs(I, i0, j, kk, zv);
          axpy4(-ah, acc, z[m], z[m]);
          mul4(z[m], zv, zv);
          rz = dot4(z[m], zv);
          rr = dot4(z[m], z[m]);
          put_faces(it, i0, j, kk, zv);
        }
      }
      if (multi) {
        unit_sum(cell0(it, i0, j, kk) >> 6, 0, rz);
        unit_sum(cell0(it, i0, j, kk) >> 6, 1, rr);
      } else {
        rs[0] += rz;
        rs[1] += rr;
      }
    }
    publish(Two{}, wb, nb + 1, true, rs);
    // ---- x += alpha p, while the sums travel
    const int tid_x = opaque();
#pragma unroll
    for (int m = 0; m < M; ++m) {
      int it, i0, j, kk;
      if (!quad(tid_x, m, it, i0, j, kk) || !live(it)) continue;
      const int c0 = cell0(it, i0, j, kk);
      const TV alpha = TV(sim_at(it).alpha);
      TV pv[4];
      ld4(sp + c0, pv);
      if constexpr (XR) {
        axpy4(alpha, pv, xr[m], xr[m]);
      } else {
        TV xv[4];
        ld4(x + base + c0, xv);
        axpy4(alpha, pv, xv, xv);
        st4(x + base + c0, xv);
      }
    }
    // Several sims: the warps of the next decisions set ResSim::done, which the loop above
    // reads, as soon as their sim's words are there (with one sim a barrier comes first).
    if (multi) __syncthreads();
  }
  if (failed) return;
  // ---- exit: the iterate (mixed: added to the FP64 one), and in mixed mode the search
  // direction, which the next correction cycle resumes
#pragma unroll
  for (int m = 0; m < M; ++m) {
    int it, i0, j, kk;
    if (!quad(tid, m, it, i0, j, kk) || sim_at(it).kdone == 0) continue;
    const int c0 = cell0(it, i0, j, kk);
    const size_t gi = base + c0;
    TV xv[4];
    if constexpr (XR) {
#pragma unroll
      for (int e = 0; e < 4; ++e) xv[e] = xr[m][e];
    } else {
      ld4(x + gi, xv);
    }
    if constexpr (kD) {
      if constexpr (XR) st4(x + gi, xv);
    } else {
      if (prm.x64_add) {
        double x64[4];
        ld4(prm.x64_add + gi, x64);
#pragma unroll
        for (int e = 0; e < 4; ++e) x64[e] = fma(double(xv[e]), sim_at(it).ih0, x64[e]);
        st4(prm.x64_add + gi, x64);
      }
      TV pv[4];
      ld4(sp + c0, pv);
      st4(p + gi, pv);
    }
  }
}

// ---------------------------------------------------------------- launcher

struct ResPlan {
  ResShape sh;
  int nt, m, geo, grid;
  size_t smem;
};

inline size_t up16(size_t b) { return (b + 15) & ~(size_t)15; }

// The launch shape of a grid, or false when its vectors do not fit on chip: the slab
// depth and the number of blocks of least estimated cycles per iteration.  An exchange is put
// at 1500 + 10 cycles per block (1.7k on 16 blocks, 3.0k on 152; measured without the sums 2.2k
// and 3.1k, see above), a cell at 1 cycle of an SM in FP32 and 8 in FP64, a ghost entry at 0.5
// and 1.
template <class TV>
bool res_shape(const Ctx& x, int nsm, size_t smem_max, ResPlan* out) {
  const int B = x.B, lb = B == 16 ? 4 : B == 8 ? 3 : 2;
  constexpr size_t E = sizeof(TV);
  constexpr int kMost = 4 * 512 * (E == 8 ? 6 : 14);
  const int blocks = nsm < kResBlocks ? nsm : kResBlocks;
  double best = -1.0;
  for (int lk = lb; lk >= 1; --lk) {
    const int KS = 1 << lk, IC = B * B * KS, G = 4 * KS * B + 2 * B * B;
    const long long N = (long long)x.g.n_cubes * (B / KS);
    if (N * G > 0x7fffffffLL) continue;
    // with several sims the sums run over units of 64 cells, which must not cross items
    if (x.g.n_sims > 1 && IC < 64) continue;
    for (int div = 1; div <= 16; ++div) {
      const int most = (blocks + div - 1) / div;
      const int grid = N < most ? (int)N : most;
      const int ipb = (int)((N + grid - 1) / grid);
      const long long cells = (long long)ipb * IC;
      if (cells > kMost) break;
      const int quads = (int)(cells / 4);
      const int need = (quads + 511) / 512;
      ResPlan P{};
      P.nt = quads <= 256 && grid <= 128 ? 256 : 512;
      P.geo = 0;
      P.m = need <= 1 ? 1 : need <= 2 ? 2 : need <= 4 ? 4 : need <= 8 ? 8 : 14;
      if (E == 8 && need > 4) P.m = 6;
      if (P.m >= 4 && KS == B && B >= 8) P.geo = B;  // the unrolled whole-cube kernels
      if (P.m > (E == 8 ? 4 : 8) && !P.geo) continue;
      const int nls = x.g.n_sims < ipb ? x.g.n_sims : ipb;
      const size_t units = (size_t)P.nt * P.m / 16;
      const size_t red = sizeof(double) * 2 * (x.g.n_sims > 1 ? units : E == 8 ? P.nt : P.nt / 32);
      ResShape& s = P.sh;
      s.lb = lb;
      s.lk = lk;
      s.ipb = ipb;
      s.multi = x.g.n_sims > 1 ? 1 : 0;
      size_t o = up16(E * (size_t)cells);
      s.o_g = (int)o;
      o += up16(E * (size_t)ipb * G);
      s.o_item = (int)o;
      o += up16(sizeof(ResItem<TV>) * (size_t)ipb);
      s.o_21 = (int)o;
      o += x.g.max_level && E == 4 ? up16(sizeof(ResFace21) * (size_t)ipb) : 0;
      s.o_tab = (int)o;
      o += up16(2 * E * (size_t)nls * (x.g.max_level + 1) * kW3);
      s.o_sim = (int)o;
      o += up16(sizeof(ResSim) * (size_t)nls);
      s.o_red = (int)o;
      o += up16(red);
      if (o > smem_max) break;
      s.o_q = (int)o;
      const size_t step = 4 * E * (size_t)P.nt, room = (smem_max - o) / step;
      s.mq = room < (size_t)P.m ? (int)room : P.m;
      o += step * (size_t)s.mq;
      P.grid = grid;
      P.smem = o;
      const double cost = (E == 8 ? 8.0 : 1.0) * (double)cells +
                          (E == 8 ? 1.0 : 0.5) * (double)ipb * G + 2.0 * (1500.0 + 10.0 * grid);
      if (best < 0.0 || cost < best) {
        best = cost;
        *out = P;
      }
    }
  }
  return best >= 0.0;
}

template <class TV, int NT, int M, int GEO>
cudaError_t res_launch(const Ctx& x, const SolveParams& prm, const ResPlan& P) {
  // x in registers up to four quads a thread (FP64: two), else in global memory; the
  // largest FP32 blocks keep K p of six quads in registers (the rest fills shared memory)
  constexpr bool XR = M <= (sizeof(TV) == 8 ? 2 : 4);
  constexpr int MQR = sizeof(TV) == 4 && M == 14 ? 4 : 0;
  auto kern = k_pcg_res<TV, NT, M, GEO, XR, MQR>;
  cudaError_t e = allow_dynamic_smem(kern, P.smem);
  if (e != cudaSuccess) return e;
  DevGrid gg = x.g;
  ResShape sh = P.sh;
  TV* xp;
  if constexpr (sizeof(TV) == 8) xp = x.f.p;
  else xp = x.f.e;
  const TV* rp = (const TV*)x.f.r;
  TV* pp = (TV*)x.f.p0;
  TV* qp = (TV*)x.f.q;
  TV* fz = (TV*)x.f.s0;  // face planes: idle vectors of the single-reduction form (s0, s1)
  WordLine* words = (WordLine*)x.f.words;
  SolveParams pr = prm;
  int* err = x.f.err;
  // exchange numbers start at one in every launch
  e = cudaMemsetAsync(words, 0, sizeof(WordLine) * 3 * (size_t)(P.grid + x.g.n_sims), x.stream);
  if (e != cudaSuccess) return e;
  void* args[] = {&gg, &sh, &xp, &rp, &pp, &qp, &fz, &words, &pr, &err};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(P.grid), dim3(NT), args, P.smem, x.stream);
}

template <class TV>
cudaError_t res_plan(const Ctx& x, ResPlan* P, bool* fits) {
  int dev = 0, nsm = 0, smax = 0;
  cudaError_t e;
  *fits = false;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
    return e;
  *fits = res_shape<TV>(x, nsm, (size_t)smax - sizeof(double) * 2 * kResBlocks - 64, P);
  return cudaSuccess;
}

}  // namespace

}  // namespace bcm
