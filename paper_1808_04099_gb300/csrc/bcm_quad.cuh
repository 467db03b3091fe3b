// bcm_quad.cuh -- pieces of the kernels that work on quads (four cells along x): packed FP32
// arithmetic, the 7-point operator on a quad, and the quad tile of a whole cube.
//
// A quad tile holds a cube's values densely (quads stay 16-byte aligned, unlike in a
// padded tile) and its six face halos as planes of their own.  A thread owns a column of
// two or four quads along z, so z neighbours are registers inside it, the x neighbours come
// from the lanes beside it, and every global load of a thread is issued before the first
// use: the padded-tile kernels load a few cells, store them, and load again, which made
// each cube a chain of about ten round trips to memory.
#pragma once

#include "bcm_cube.cuh"
#include "bcm_internal.cuh"

namespace bcm {

// 1 / d by Newton's iteration y <- y + y (1 - d y) from the hardware's approximate
// reciprocal (about 20 bits), two steps, and a quotient from it with one correction by its
// remainder: within an ulp or so of the division's.  An FP64 operation takes 64 cycles on
// this part and the compiler's division 1460; the reciprocal takes about 450, twice per
// iteration of the solver.  Exponents near the ends of the range go to the division.
__device__ __forceinline__ double quick_rcp(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const unsigned ex = (unsigned)__double2hiint(y) >> 20 & 0x7ffu;
  if (ex - 64u > 1920u) return 1.0 / d;
  y = fma(y, fma(-d, y, 1.0), y);
  return fma(y, fma(-d, y, 1.0), y);
}
__device__ __forceinline__ double quick_div(double a, double d, double y) {  // y = 1 / d
  double q = a * y;
  q = fma(fma(-d, q, a), y, q);
  return isfinite(q) ? q : a / d;
}

// Quads of cells in FP32 as two packed pairs (one instruction per pair), in FP64 plain.
__device__ __forceinline__ unsigned long long pk(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(unsigned long long r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// out = a x + y
__device__ __forceinline__ void axpy4(float a, const float (&x)[4], const float (&y)[4],
                                      float (&out)[4]) {
  const unsigned long long aa = pk(a, a);
  const unsigned long long l = fma2(aa, pk(x[0], x[1]), pk(y[0], y[1]));
  const unsigned long long h = fma2(aa, pk(x[2], x[3]), pk(y[2], y[3]));
  upk(l, out[0], out[1]);
  upk(h, out[2], out[3]);
}
__device__ __forceinline__ void axpy4(double a, const double (&x)[4], const double (&y)[4],
                                      double (&out)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) out[e] = fma(a, x[e], y[e]);
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ void mul4(const float (&x)[4], const float (&y)[4], float (&out)[4]) {
  const unsigned long long l = mul2(pk(x[0], x[1]), pk(y[0], y[1]));
  const unsigned long long h = mul2(pk(x[2], x[3]), pk(y[2], y[3]));
  upk(l, out[0], out[1]);
  upk(h, out[2], out[3]);
}
__device__ __forceinline__ float dot4(const float (&x)[4], const float (&y)[4]) {
  float a, b;
  upk(fma2(pk(x[2], x[3]), pk(y[2], y[3]), fma2(pk(x[0], x[1]), pk(y[0], y[1]), 0ull)), a, b);
  return a + b;
}
__device__ __forceinline__ double dot4(const double (&x)[4], const double (&y)[4]) {
  return fma(x[3], y[3], fma(x[2], y[2], fma(x[1], y[1], x[0] * y[0])));
}
// K p / h of a quad: its cells, the cells before and after it along x, the quads across y
// and z.  Both types sum differences, which are exact for close values (6 c minus the sum of
// the neighbours takes 6 FP64 operations a cell instead of 9.5, but its rounding grows with
// the value itself: 2.5e-14 of K p on a smooth 64^3 field, 1.6e-11 with the field offset by
// 100, against 2.7e-16).  A difference along x serves both its cells, and one along z too
// where the caller's next quad is this one's zp (the same expression).
__device__ __forceinline__ void seven_point(const double (&c)[4], double xl, double xh,
                                            const double (&ym)[4], const double (&yp)[4],
                                            const double (&zm)[4], const double (&zp)[4],
                                            double (&acc)[4]) {
  const double d01 = c[0] - c[1], d12 = c[1] - c[2], d23 = c[2] - c[3];
  const double x[4] = {(c[0] - xl) + d01, d12 - d01, d23 - d12, (c[3] - xh) - d23};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    acc[e] = (x[e] + ((c[e] - ym[e]) + (c[e] - yp[e]))) + ((c[e] - zp[e]) - (zm[e] - c[e]));
}
__device__ __forceinline__ void seven_point(const float (&c)[4], float xl, float xh,
                                            const float (&ym)[4], const float (&yp)[4],
                                            const float (&zm)[4], const float (&zp)[4],
                                            float (&acc)[4]) {
  const float d01 = c[0] - c[1], d12 = c[1] - c[2], d23 = c[2] - c[3];
  const float x[4] = {(c[0] - xl) + d01, d12 - d01, d23 - d12, (c[3] - xh) - d23};
#pragma unroll
  for (int u = 0; u < 4; u += 2) {
    const unsigned long long cc = pk(c[u], c[u + 1]);
    unsigned long long a = pk(x[u], x[u + 1]);
    a = add2(a, sub2(cc, pk(ym[u], ym[u + 1])));
    a = add2(a, sub2(cc, pk(yp[u], yp[u + 1])));
    a = add2(a, sub2(cc, pk(zm[u], zm[u + 1])));
    a = add2(a, sub2(cc, pk(zp[u], zp[u + 1])));
    upk(a, acc[u], acc[u + 1]);
  }
}

// ---- the quad tile

// A thread's column has NP planes: two on 8^3 in FP64, where the one warp that four planes
// leave a cube is a serial chain on one of the SM's four FP64 pipes (76 cycles an operation).
// FP64 multigrid steps with four planes and with two: 16 cubes of 8^3 2727, 2078 us, 128
// 3302, 2580, 1024 5658, 5373, 2880 14.1, 12.6 ms; 16 cubes of 16^3 5264, 4741 us.
template <int B, class TT>
struct QT {
  static constexpr int BB = B * B, B3 = B * BB, Q = BB / 4;  // quads per plane
  static constexpr int NP = B == 8 && sizeof(TT) == 8 ? 2 : 4;
  static constexpr int TPC = B3 / (4 * NP);                  // threads per cube
  static constexpr int CPB = TPC == 32 ? 4 : 1;              // cubes per block
  static constexpr int NT = TPC * CPB;
  static constexpr int N = B3 + 6 * BB;                      // tile elements
  // blocks per SM that the kernels are compiled for: 768 threads in FP32, 512 in FP64 (whose
  // passes are bound by the FP64 pipe)
  static constexpr int blocks = (sizeof(TT) == 4 ? 768 : 512) / NT;
  // threads of one cube: a warp or the block
  __device__ __forceinline__ static void sync() {
    if constexpr (TPC == 32) __syncwarp();
    else __syncthreads();
  }
  // sum of a cube's threads, valid in the cube's first
  __device__ __forceinline__ static double sum(double v) {
    if constexpr (TPC == 32) {
      return warp_sum(v);
    } else {
      __shared__ double red[NT];
      return block_sum_once<NT>(v, red);
    }
  }
};

// Constants of a block's cube.
template <class TV>
struct CubeQ {
  int nb[6];
  int w3[6];                 // Jacobi face weights (thirds)
  unsigned long long nbw;    // bit 6 f + e: face e of neighbour f has a weight other than 3
  int smask;                 // bit f: w3[f] is not 3
  int bnd, neg;              // bit f: domain face; with outflow (ghost -p)
  int c21;                   // bit f: coarse neighbour; bit 8 + f: fine neighbours
  TV inv[kW3];               // 1 / diag(K) by face-weight sum
  TV h;
};

// The constants of cube c, loaded by the 32 first threads of the cube (lt: thread within the
// cube) in two steps, so that the table lookups of the first are in flight together with a
// kernel's own first loads; QT::sync() publishes them.  Only tables that no kernel
// writes are read.
struct CubeLoad {
  int n, w, e0, e1, s, lv;
};
__device__ __forceinline__ CubeLoad cube_lookup(const DevGrid& g, int c, int lt) {
  CubeLoad L{0, 3, 3, 3, 0, 0};
  if (!bcm_expect(g, c >= 0 && c < g.n_cubes, CHK_CUBE)) c = 0;
  L.s = g.n_sims == 1 ? 0 : g.sim[c];
  if (lt >= 32) return L;
  L.lv = g.max_level == 0 ? 0 : g.lvl[c];
  if (lt < 6) {
    L.n = g.nb[6 * c + lt];
    L.w = g.w3[6 * c + lt];
  }
  L.e0 = g.nbw3[36 * c + lt];
  if (lt < 4) L.e1 = g.nbw3[36 * c + 32 + lt];
  return L;
}
template <class TV>
__device__ __forceinline__ void cube_publish(CubeQ<TV>& cq, const DevGrid& g, const CubeLoad& L, int lt) {
  if (lt >= 32) return;
  int s = L.s, lv = L.lv;
  if (!bcm_expect(g, s >= 0 && s < g.n_sims && lv >= 0 && lv <= g.max_level, CHK_SIM)) s = lv = 0;
  const SimParams& sp = g.sp[s];
  TV i0, i1 = TV(0), h;
  if constexpr (sizeof(TV) == 4) {
    i0 = sp.invdiag32[lv][lt];
    if (lt < kW3 - 32) i1 = sp.invdiag32[lv][32 + lt];
    h = lv ? 0.5f * sp.h032 : sp.h032;
  } else {
    i0 = sp.invdiag[lv][lt];
    if (lt < kW3 - 32) i1 = sp.invdiag[lv][32 + lt];
    h = lv ? 0.5 * sp.h0 : sp.h0;
  }
  const int bc = lt < 6 ? sp.bc[lt] : 0, n = lt < 6 ? checked_nb(g, L.n) : 0;
  const unsigned lo = __ballot_sync(0xffffffffu, L.e0 != 3), hi = __ballot_sync(0xffffffffu, L.e1 != 3);
  const unsigned sm = __ballot_sync(0xffffffffu, L.w != 3);
  const unsigned bn = __ballot_sync(0xffffffffu, lt < 6 && n == NB_BOUNDARY);
  const unsigned ng = __ballot_sync(0xffffffffu, lt < 6 && n == NB_BOUNDARY && bc == BC_OUTFLOW);
  const unsigned co = __ballot_sync(0xffffffffu, lt < 6 && n == NB_COARSE);
  const unsigned fi = __ballot_sync(0xffffffffu, lt < 6 && n == NB_FINE);
  if (lt < 6) {
    cq.nb[lt] = n;
    cq.w3[lt] = L.w;
  }
  cq.inv[lt] = i0;
  if (lt < kW3 - 32) cq.inv[32 + lt] = i1;
  if (lt == 0) {
    cq.nbw = (unsigned long long)lo | (unsigned long long)hi << 32;
    cq.smask = (int)sm;
    cq.bnd = (int)bn;
    cq.neg = (int)ng;
    cq.c21 = (int)(co | fi << 8);
    cq.h = h;
  }
}

// 1 / diag(K) of the cells of a quad of the cube
template <int B, class TV>
__device__ __forceinline__ void quad_inv(const CubeQ<TV>& cq, int i0, int j, int kk, TV (&v)[4]) {
  if (cq.smask == 0) {
    v[0] = v[1] = v[2] = v[3] = cq.inv[18];
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = cq.inv[s3_of<B>(cq.w3, i0 + e, j, kk)];
  }
}
// ... and of four cells of same-level neighbour f: cell0, cell0 + stride, ...
template <int B, class TV>
__device__ __forceinline__ void nb_inv(const CubeQ<TV>& cq, const DevGrid& g, int c, int f, int cell0,
                                       int stride, TV (&v)[4]) {
  if ((cq.nbw >> (6 * f) & 63ull) == 0) {
    v[0] = v[1] = v[2] = v[3] = cq.inv[18];
  } else {
    int w3[6];
    for (int e = 0; e < 6; ++e) w3[e] = g.nbw3[36 * c + 6 * f + e];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int cell = cell0 + e * stride;
      v[e] = cq.inv[s3_of<B>(w3, cell % B, (cell / B) % B, cell / (B * B))];
    }
  }
}

// four cells of a field: contiguous, or a stride apart (an x face)
template <class TV>
__device__ __forceinline__ void ldq(const TV* __restrict__ p, int stride, TV (&v)[4]) {
  if (stride == 1) {
    ld4(p, v);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = p[e * stride];
  }
}

// The tile's halo planes, each thread R quads of them, in two steps: the neighbour ids are
// looked up with the cube's other constants, so a kernel issues its halo loads together
// with those of its own cells, and forms the halo values once the constants are there.
template <int B, class TT>
struct Halo {
  using T = QT<B, TT>;
  static constexpr int R = (6 * T::Q + T::TPC - 1) / T::TPC;
  int n[R];
  __device__ __forceinline__ void lookup(const DevGrid& g, int c, int lt) {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int e = lt + u * T::TPC;
      n[u] = e < 6 * T::Q ? checked_nb(g, g.nb[6 * c + e / T::Q]) : NB_BOUNDARY;
    }
  }
  // fn(u, f, n, cell0, stride) for the thread's quads on same-level neighbours: cells cell0,
  // cell0 + stride, ... of cube n
  template <class Fn>
  __device__ __forceinline__ void each(int lt, const Fn& fn) const {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      if (n[u] < 0) continue;
      const int e = lt + u * T::TPC, f = e / T::Q, t = 4 * (e - f * T::Q), d = f >> 1;
      fn(u, f, n[u], cell_of<B>(d, (f & 1) ? 0 : B - 1, t % B, t / B), d == 0 ? B : 1);
    }
  }
  // the quads into the planes: make(u, f, n, cell0, stride, v), and one(cube, cell) for the
  // cells across 2:1 faces (domain faces are filled by own_quad)
  template <class TV, class Make, class One>
  __device__ __forceinline__ void store(TV* __restrict__ gh, const DevGrid& g, int c, int lt,
                                        const Make& make, const One& one, int lsh) const {
    each(lt, [&](int u, int f, int nn, int cell, int stride) {
      TV v[4];
      make(u, f, nn, cell, stride, v);
      st4(gh + 4 * (lt + u * T::TPC), v);
    });
#pragma unroll
    for (int u = 0; u < R; ++u) {
      if (n[u] >= NB_BOUNDARY) continue;
      const int e = lt + u * T::TPC, f = e / T::Q, t = 4 * (e - f * T::Q);
#pragma unroll 1
      for (int q = 0; q < 4; ++q)
        gh[4 * e + q] = poisson_ghost_21<B, TV>(g, c, f, t % B + q, t / B, n[u], one, lsh);
    }
  }
};

// A quad of the cube into the tile, with the ghosts it sets across domain faces.
template <int B, class TV, class CQ>
__device__ __forceinline__ void own_quad(TV* __restrict__ S, TV* __restrict__ gh, const CQ& cq,
                                         int i0, int j, int kk, const TV (&v)[4]) {
  constexpr int BB = B * B;
  st4(S + (kk * B + j) * B + i0, v);
  if (cq.bnd) {
    auto sg = [&](int f, TV x) { return (cq.neg >> f & 1) ? -x : x; };
    auto face = [&](int f, int o) {
      if (cq.bnd >> f & 1) {
        const TV w[4] = {sg(f, v[0]), sg(f, v[1]), sg(f, v[2]), sg(f, v[3])};
        st4(gh + f * BB + o, w);
      }
    };
    if (i0 == 0 && (cq.bnd & 1)) gh[kk * B + j] = sg(0, v[0]);
    if (i0 == B - 4 && (cq.bnd & 2)) gh[BB + kk * B + j] = sg(1, v[3]);
    if (j == 0) face(2, kk * B + i0);
    if (j == B - 1) face(3, kk * B + i0);
    if (kk == 0) face(4, j * B + i0);
    if (kk == B - 1) face(5, j * B + i0);
  }
}

// The 7-point sums (K v / h) of a thread's column of NP quads, planes k0 .. k0 + NP - 1, from
// the complete tile; out(m, acc) consumes plane k0 + m.  The threads of a warp call it
// together.
template <int B, class TV, int NP, class CQ, class Out>
__device__ __forceinline__ void quad_column(const TV* __restrict__ S, const TV* __restrict__ gh,
                                            const CQ& cq, int i0, int j, int k0,
                                            const TV (&v)[NP][4], const Out& out) {
  constexpr int BB = B * B;
  TV zm[4], zp[4];
  const int o = (k0 * B + j) * B + i0;
  ld4(k0 > 0 ? S + o - BB : gh + 4 * BB + j * B + i0, zm);
  ld4(k0 < B - NP ? S + o + NP * BB : gh + 5 * BB + j * B + i0, zp);
#pragma unroll
  for (int m = 0; m < NP; ++m) {
    const int kk = k0 + m, om = o + m * BB;
    TV ym[4], yp[4], acc[4];
    ld4(j > 0 ? S + om - B : gh + 2 * BB + kk * B + i0, ym);
    ld4(j < B - 1 ? S + om + B : gh + 3 * BB + kk * B + i0, yp);
    TV xl = __shfl_up_sync(0xffffffffu, v[m][3], 1);
    TV xh = __shfl_down_sync(0xffffffffu, v[m][0], 1);
    if (i0 == 0) xl = gh[kk * B + j];
    if (i0 == B - 4) xh = gh[BB + kk * B + j];
    TV b[4], t[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      b[e] = m == 0 ? zm[e] : v[m > 0 ? m - 1 : 0][e];
      t[e] = m == NP - 1 ? zp[e] : v[m < NP - 1 ? m + 1 : m][e];
    }
    seven_point(v[m], xl, xh, ym, yp, b, t, acc);
    if (cq.c21) {  // 2:1 faces: weight 2/3 on the fine side, 4/3 on the coarse (R7)
      auto wt = [&](int f) {
        return (cq.c21 >> f & 1) ? TV(2.0 / 3.0) - TV(1)
               : (cq.c21 >> (8 + f) & 1) ? TV(4.0 / 3.0) - TV(1) : TV(0);
      };
      if (i0 == 0) acc[0] += wt(0) * (v[m][0] - xl);
      if (i0 == B - 4) acc[3] += wt(1) * (v[m][3] - xh);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (j == 0) acc[e] += wt(2) * (v[m][e] - ym[e]);
        if (j == B - 1) acc[e] += wt(3) * (v[m][e] - yp[e]);
        if (kk == 0) acc[e] += wt(4) * (v[m][e] - b[e]);
        if (kk == B - 1) acc[e] += wt(5) * (v[m][e] - t[e]);
      }
    }
    out(m, acc);
  }
}

}  // namespace bcm
