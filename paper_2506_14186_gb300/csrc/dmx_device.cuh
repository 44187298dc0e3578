// Device code of the forward dynamics v' = F(q, v, u) and of one adaptive
// Dormand-Prince attempt, for one environment handled by a group of G lanes
// of a warp (G = 1, 2, 4, 8, 16, 32).  Every per-environment array lives in
// shared memory; the G lanes split loops over bodies, dofs, contact slots,
// constraint rows and matrix entries, and meet at __syncwarp(group mask).
//
// Method (arXiv 2506.14186):
//   Sec. 2, Eq. (EOM)       v' = M^-1 (tau - c + J^T f); M by the composite-
//                           rigid-body algorithm, c by recursive Newton-Euler
//                           (world-frame spatial vectors, Featherstone)
//   Sec. 2.1                signed distances r (active iff r < 0), pyramidal
//                           rows, a_ref = -b (J v) - k d(r) r, impedance d(r)
//                           (solimp spline), R = A_hat (1 - d) / d, and the
//                           relaxed Gauss principle solved by exact Newton
//   App. C.1                plane-box from the box vertices, pos = v - r/2 n
//   Sec. 4                  contacts from distance: d(r) continued for r > 0,
//                           softplus in place of the ReLU of a_ref (backward)
//   Sec. 3.1, App. B, C.2   adaptive Dormand-Prince 5(4), PID controller,
//                           quaternions integrated exactly
//   Fig. 12                 Tsitouras 5(4) and fixed-step semi-implicit Euler
//
// GB300 notes: an FP64 warp instruction takes 64 cycles of its SM
// sub-partition whatever its active lanes (a division 565, a reciprocal square
// root 350, a shared-memory read about 30, a model read through the L1 about
// 40), so the cost of a phase is the number of FP64 instructions on its
// longest path plus its dependent reads.  Work is therefore split into equal
// tasks of one matrix or vector component (branches inside a task cost the sum
// of their sides), tree recursions run along chains without meeting the other
// lanes, and indices come packed or from tables.  Every split keeps the
// operations of each result and their order: for a given final active set the
// results do not depend on the lane count.  (The line search, which only picks
// the next set to try, sums its slopes in lane order.)  The Newton search starts
// from the active set of the previous right-hand side of the same environment:
// the minimiser is unique, so the start changes the number of iterations, and the
// last bits where a row lies at the edge of the active set to rounding.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "dmx_model.h"

namespace dmx {

// ------------------------------------------------------------------ lane groups
template <int G>
struct Grp {
  int lane;
  int base;                          // first warp lane of the group
  unsigned mask;
  __device__ Grp() {
    const int l = threadIdx.x & 31;
    lane = l & (G - 1);
    base = l & ~(G - 1);
    mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << base);
  }
  // bit k: predicate of the group's lane k
  __device__ unsigned ballot(bool p) const {
    const unsigned b = __ballot_sync(mask, p);
    return G == 32 ? b : (b >> base) & ((1u << G) - 1u);
  }
  __device__ unsigned ior(unsigned x) const { return G == 1 ? x : __reduce_or_sync(mask, x); }
  __device__ void sync() const {
    if (G > 1) __syncwarp(mask);
  }
  __device__ double sum(double x) const {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(mask, x, o);
    return x;
  }
  __device__ int isum(int x) const {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(mask, x, o);
    return x;
  }
  __device__ int bcast(int x, int src) const { return G == 1 ? x : __shfl_sync(mask, x, src, G); }
  __device__ double bcast(double x, int src) const { return G == 1 ? x : __shfl_sync(mask, x, src, G); }
};

// Loop over n tasks spread over the group's lanes.  Not unrolled: the hot loop
// of a kernel (one right-hand side, its VJP) is a long run of such loops with
// one to five passes each, and unrolled copies push it out of the instruction
// caches (4096 box pushes 185 -> 176 ms, 2048 arm gradients 269 -> 250 ms).
#define DMX_TASKS(t, n) _Pragma("unroll 1") for (int t = g.lane; t < (n); t += G)

// (row, column) of the t-th entry of a lower triangle enumerated row by row
// ((0,0), (1,0), (1,1), (2,0), ...): the same for every matrix size.  In
// global memory (read through the L1): the lanes of a group read different
// entries, which the constant cache would serve one after the other.
constexpr int NTRI = (MAXV + 1) * (MAXV + 2) / 2;
struct TriTab {
  unsigned short e[NTRI];            // row << 8 | column
};
constexpr TriTab make_tri() {
  TriTab t{};
  int k = 0;
  for (int i = 0; i <= MAXV; ++i)
    for (int j = 0; j <= i; ++j) t.e[k++] = (unsigned short)(i << 8 | j);
  return t;
}
static __device__ const TriTab d_tri = make_tri();
struct Tri {
  int i, j;
};
__device__ __forceinline__ Tri tri(int t) {
  const int p = __ldg(&d_tri.e[t]);
  return {p >> 8, p & 255};
}

// ------------------------------------------------------------------ small helpers
// Comparisons on the bits of a double (an FP64 comparison takes 106 cycles of
// the FP64 unit's path, an fmax 210; integer ones about 15).  NaN compares
// false, as with the floating-point operators.
constexpr long long kInfBits = 0x7ff0000000000000ll;
__device__ __forceinline__ bool is_neg(double x) {            // x < 0
  const long long b = __double_as_longlong(x);
  return b < 0 && (unsigned long long)(b & 0x7fffffffffffffffll) - 1ull < (unsigned long long)kInfBits;
}
__device__ __forceinline__ bool is_pos(double x) {            // x > 0
  return (unsigned long long)__double_as_longlong(x) - 1ull < (unsigned long long)kInfBits;
}
__device__ __forceinline__ bool above(double x, double c) {   // x > c, c >= 0
  const long long b = __double_as_longlong(x);
  return b > __double_as_longlong(c) && b <= kInfBits;
}
__device__ __forceinline__ bool below(double x, double c) {   // x < c, x >= 0 or NaN, c > 0
  return __double_as_longlong(x) < __double_as_longlong(c);
}
// the larger of two numbers >= 0 (NaN if one is)
__device__ __forceinline__ double max_pos(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return __longlong_as_double(x > y ? x : y);
}
// x times sg = +-1
__device__ __forceinline__ double flip(double x, bool minus) {
  return __longlong_as_double(__double_as_longlong(x) ^ (minus ? (1ll << 63) : 0ll));
}
template <class A, class B, class C>
__device__ __forceinline__ void cross3(const A* a, const B* b, C* c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}
template <class A, class B>
__device__ __forceinline__ auto dot3(const A* a, const B* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
template <class A, class B, class C>
__device__ __forceinline__ void matvec3(const A* M, const B* x, C* y) {
  y[0] = M[0] * x[0] + M[1] * x[1] + M[2] * x[2];
  y[1] = M[3] * x[0] + M[4] * x[1] + M[5] * x[2];
  y[2] = M[6] * x[0] + M[7] * x[1] + M[8] * x[2];
}
template <class A, class B, class C>
__device__ __forceinline__ void matTvec3(const A* M, const B* x, C* y) {
  y[0] = M[0] * x[0] + M[3] * x[1] + M[6] * x[2];
  y[1] = M[1] * x[0] + M[4] * x[1] + M[7] * x[2];
  y[2] = M[2] * x[0] + M[5] * x[1] + M[8] * x[2];
}
// Single components (e = 0..5) of the spatial products above, so that the
// six components of a body's vector can go to six lanes.
__device__ __forceinline__ int nxt3(int k) { return k == 2 ? 0 : k + 1; }
__device__ __forceinline__ int prv3(int k) { return k == 0 ? 2 : k - 1; }
template <class T>
__device__ __forceinline__ T crm_comp(const T* a, const T* b, int e) {   // (a x b)_e, motion
  const int k = e < 3 ? e : e - 3, k1 = nxt3(k), k2 = prv3(k);
  const T* x = e < 3 ? b : b + 3;
  T r = a[k1] * x[k2] - a[k2] * x[k1];                                // (w x w2) or (w x v2)
  if (e >= 3) r += a[3 + k1] * b[k2] - a[3 + k2] * b[k1];             // + v x w2
  return r;
}
template <class T>
__device__ __forceinline__ T crf_comp(const T* a, const T* b, int e) {   // (a x* b)_e, force
  const int k = e < 3 ? e : e - 3, k1 = nxt3(k), k2 = prv3(k);
  const T* x = e < 3 ? b : b + 3;
  T r = a[k1] * x[k2] - a[k2] * x[k1];                                // (w x n) or (w x f)
  if (e < 3) r += a[3 + k1] * b[3 + k2] - a[3 + k2] * b[3 + k1];      // + v x f
  return r;
}
template <class T>
__device__ __forceinline__ T inertia_comp(const T* I, const T* x, int e) {   // (I x)_e, inertia_apply
  const int k = e < 3 ? e : e - 3, k1 = nxt3(k), k2 = prv3(k);
  if (e < 3)   // I_O row k (entry (k, j): 4 + k on the diagonal, else 6 + k + j) . w + h x v
    return I[k == 0 ? 4 : 6 + k] * x[0] + I[k == 1 ? 5 : 7 + k] * x[1] + I[k == 2 ? 6 : 8 + k] * x[2] +
           (I[1 + k1] * x[3 + k2] - I[1 + k2] * x[3 + k1]);
  return I[0] * x[3 + k] - (I[1 + k1] * x[k2] - I[1 + k2] * x[k1]);   // m v - h x w
}

// ------------------------------------------------------------------ workspace view
template <class T>
struct WsT {
  T* d;
  int* i;
  const Layout* L;
  // the right-hand-side VJP reads the contact records / Jacobian rows here
  // when set (a stage snapshot in device memory), else from the workspace
  const double* xct = nullptr;
  const double* xJ = nullptr;
  __device__ T* at(int off) const { return d + off; }
};

using Ws = WsT<double>;

// Entry e (row-major) of the rotation of the quaternion x (w, x, y, z) with
// s = 2 / |x|^2 (the normalisation folded into the products).  Every entry is
// s u1 u3 +- s u2 u4 (one minus it on the diagonal) with components picked by
// e, so that the nine lanes of a body run one instruction sequence: a switch
// over e costs the sum of its nine sides.
__device__ __forceinline__ double mul_add(double a, double b, double c) { return __fma_rn(a, b, c); }
template <class T>
__device__ __forceinline__ T quat_entry(const T* x, const T& s, int e) {
  // per entry 8 bits: u1, u3, u2, u4 (2 bits each, lowest first; 0 = w)
  const unsigned k = e < 8 ? (unsigned)(0x4E8D4EF5C98DC9FAull >> (8 * e)) & 255u : 0xA5u;
  const T t1 = s * x[k & 3], t2 = s * x[(k >> 4) & 3];
  T p = t2 * x[(k >> 6) & 3];
  if ((0x062u >> e) & 1u) p = -p;                      // entries 1, 5, 6
  const T v = mul_add(t1, x[(k >> 2) & 3], p);
  return ((0x111u >> e) & 1u) ? 1.0 - v : v;           // entries 0, 4, 8
}
// Entry (i, j) of the hinge rotation about the unit axis a by the angle with
// sine sn and cosine cs (Rodrigues: I + sin K + (1 - cos) K^2, K = [a]x).
template <class T>
__device__ __forceinline__ T hinge_entry(const double* a, const T& sn, const T& cs, int i, int j) {
  const T c1 = 1.0 - cs;
  T v = c1 * a[i] * a[j];
  if (i == j) return cs + v;
  const int k = 3 - i - j;                       // the third axis
  const bool pos = (j == nxt3(i));               // K_ij = -a_k for j = i + 1 (cyclic), else +a_k
  return pos ? v - sn * a[k] : v + sn * a[k];
}

// Sums along the body tree of one NC-component vector per body, in place, one
// lane per (chain, component): tree_down adds each body's parent into it
// (parents first), tree_up each body's children into it (children first, in
// order).  A chain is one loop of dependent additions in a register; the
// lanes meet once per chain level instead of once per body level.
template <int NC, int G, class T, class MD>
__device__ __forceinline__ void tree_down(const Grp<G>& g, const MD& m, T* X) {
  if (m.nlevel == 1) return;
  for (int cl = 0; cl < m.nchlev; ++cl) {
    const int c0 = m.chlev_start[cl], n = NC * (m.chlev_start[cl + 1] - c0);
    DMX_TASKS(t, n) {
      const int c = c0 + t / NC, e = t % NC;
      const int k0 = m.ch_start[c], k1 = m.ch_start[c + 1], par = m.ch_par[c];
      const int b0 = m.ch_list[k0];
      T x = X[NC * b0 + e];
      if (par >= 0) { x += X[NC * par + e]; X[NC * b0 + e] = x; }
      for (int k = k0 + 1; k < k1; ++k) {
        T* p = X + NC * m.ch_list[k] + e;
        x = *p + x;
        *p = x;
      }
    }
    g.sync();
  }
}
template <int NC, int G, class T, class MD>
__device__ __forceinline__ void tree_up(const Grp<G>& g, const MD& m, T* X) {
  if (m.nlevel == 1) return;
  for (int cl = m.nchlev - 1; cl >= 0; --cl) {
    const int c0 = m.chlev_start[cl], n = NC * (m.chlev_start[cl + 1] - c0);
    DMX_TASKS(t, n) {
      const int c = c0 + t / NC, e = t % NC;
      const int k0 = m.ch_start[c], k1 = m.ch_start[c + 1] - 1;
      const int tail = m.ch_list[k1], nc = m.child_count[tail], cs = m.child_start[tail];
      T x = X[NC * tail + e];
      if (nc > 0) {
        for (int j = 0; j < nc; ++j) x += X[NC * m.child_list[cs + j] + e];
        X[NC * tail + e] = x;
      }
      for (int k = k1 - 1; k >= k0; --k) {
        T* p = X + NC * m.ch_list[k] + e;
        x = *p + x;
        *p = x;
      }
    }
    g.sync();
  }
}

// Kinematics: body poses, COMs, dof motion vectors, body spatial inertias, geom poses.
// Work is split into small tasks so that a group's lanes stay busy even for a
// single body: per-body scalars (hinge sine and cosine, the free joint's
// quaternion normalisation), then every entry of every local transform, then
// the composition along the tree level by level (one entry per task), then
// COMs, geom poses and dof motion vectors, then spatial inertias.
template <int G, class T, class MD>
__device__ void kinematics(const Grp<G>& g, const MD& m, const WsT<T>& w, const T* q) {
  const Layout& L = *w.L;
  T* R = w.at(L.R); T* P = w.at(L.p); T* C = w.at(L.com);
  T* S = w.at(L.sd); T* Ib = w.at(L.Ib); T* Ic = w.at(L.Ic);
  T* X = w.at(L.xl); T* SC = w.at(L.sc);
  const int nb = m.nbody;
  DMX_TASKS(b, nb) {
    const BodyInfo bi = body_info(m, b);
    const T* x = q + bi.qadr;
    if (bi.jtype == JNT_FREE) {
      SC[2 * b] = 2.0 / (x[3] * x[3] + x[4] * x[4] + x[5] * x[5] + x[6] * x[6]);
    } else {
      T sn, cs;
      sincos(x[0], &sn, &cs);
      SC[2 * b] = sn; SC[2 * b + 1] = cs;
    }
  }
  g.sync();
  // local transforms: free joint = world pose; hinge = rotation in the parent frame.
  // Bodies at the root are written straight into the world arrays.
  DMX_TASKS(t, 12 * nb) {
    const int b = t / 12, e = t - 12 * b;
    const BodyInfo bi = body_info(m, b);
    const bool root = bi.parent < 0;
    T v;
    if (bi.jtype == JNT_FREE) {
      const T* x = q + bi.qadr;
      v = e < 9 ? quat_entry(x + 3, SC[2 * b], e) : x[e - 9];
    } else if (e >= 9) {
      v = m.b_pos[b][e - 9];
    } else {
      const int i = e / 3, j = e - 3 * (e / 3);
      const T sn = SC[2 * b], cs = SC[2 * b + 1];
      if (bi.ident) {
        v = hinge_entry(m.b_axis[b], sn, cs, i, j);
      } else {
        const double* Ro = m.b_Roff[b];
        v = Ro[3 * i] * hinge_entry(m.b_axis[b], sn, cs, 0, j) + Ro[3 * i + 1] * hinge_entry(m.b_axis[b], sn, cs, 1, j) +
            Ro[3 * i + 2] * hinge_entry(m.b_axis[b], sn, cs, 2, j);
      }
    }
    if (root) { if (e < 9) R[9 * b + e] = v; else P[3 * b + e - 9] = v; }
    else X[12 * b + e] = v;
  }
  g.sync();
  // world poses: R = R_parent R_local, p = p_parent + R_parent p_local: entries
  // 0..8 of R and 9..11 of p are the same product of a row of R_parent with a
  // column of the local transform
  for (int lev = 1; lev < m.nlevel; ++lev) {
    const int k0 = m.level_start[lev], n = 12 * (m.level_start[lev + 1] - k0);
    DMX_TASKS(t, n) {
      const int k = t / 12, e = t - 12 * k;
      const int pk = m.lv_pack[k0 + k], b = pk & 255, par = pk >> 8;
      const bool pos = e >= 9;
      const int i = pos ? e - 9 : e / 3, j = pos ? 9 : e - 3 * (e / 3), st = pos ? 1 : 3;
      const T* Rp = R + 9 * par + 3 * i; const T* xl = X + 12 * b + j;
      T v = Rp[0] * xl[0] + Rp[1] * xl[st] + Rp[2] * xl[2 * st];
      if (pos) v = P[3 * par + i] + v;
      *(pos ? P + 3 * b + i : R + 9 * b + e) = v;
    }
    g.sync();
  }
  // COMs and geom poses, one component per task, all of them a row of R times
  // a model vector (plus p): com, gpos, the columns of Roff
  T* gR = w.at(L.gR); T* gp = w.at(L.gp);
  const int n1 = 3 * nb, n2 = n1 + 12 * m.ngeom;
  DMX_TASKS(t, n2) {
    int b, i, st = 1;
    const double* c;
    T* out;
    bool rot = false, same = false;
    if (t < n1) {
      b = t / 3; i = t - 3 * b;
      c = m.b_com[b]; out = C + t;
    } else {
      const int gi = (t - n1) / 12, e = t - n1 - 12 * gi;
      b = m.g_body[gi];
      rot = e < 9;
      i = rot ? e / 3 : e - 9;
      const int j = e - 3 * i;
      c = rot ? m.g_Roff[gi] + j : m.g_pos[gi];
      if (rot) st = 3;
      same = rot ? m.g_ident[gi] : m.g_zpos[gi];
      out = rot ? gR + 9 * gi + e : gp + 3 * gi + i;
      if (same) { *out = rot ? R[9 * b + e] : P[3 * b + i]; continue; }
    }
    const T* Rb = R + 9 * b + 3 * i;
    T v = Rb[0] * c[0] + Rb[1] * c[st] + Rb[2] * c[2 * st];
    if (!rot) v = v + P[3 * b + i];
    *out = v;
  }
  // dof motion vectors (w; v at the world origin), one dof per task
  DMX_TASKS(i, m.nv) {
    const DofInfo di = dof_info(m, i);
    const int b = di.body;
    const T* Rb = R + 9 * b; const T* pb = P + 3 * b;
    T* st = S + 6 * i;
    if (di.free) {
      const int d = di.k;
      if (d < 3) {
        st[0] = 0.0; st[1] = 0.0; st[2] = 0.0; st[3] = d == 0 ? 1.0 : 0.0; st[4] = d == 1 ? 1.0 : 0.0;
        st[5] = d == 2 ? 1.0 : 0.0;
      } else {
        st[0] = Rb[d - 3]; st[1] = Rb[d]; st[2] = Rb[d + 3];
        cross3(pb, st, st + 3);
      }
    } else {
      matvec3(Rb, m.b_axis[b], st);
      cross3(pb, st, st + 3);
    }
  }
  g.sync();
  // spatial inertias about the world origin (m, m c, R diag(I) R^T + m (|c|^2 1 - c c^T)),
  // one entry per task: the six moments of every body first (12 operations
  // each), then mass and first moments, so that a pass of the lanes mostly
  // meets one kind.  Ic starts as a copy (composite inertias, crba).
  DMX_TASKS(k, 6 * nb) {
    const int b = k / 6, e = k - 6 * b;
    const double ms = m.b_mass[b];
    const T* c = C + 3 * b;
    const int i = e < 3 ? e : (e == 5 ? 1 : 0), j = e < 3 ? e : (e == 3 ? 1 : 2);   // xx yy zz xy xz yz
    const T* Rb = R + 9 * b;
    const double* In = m.b_inertia[b];
    T v = Rb[3 * i] * Rb[3 * j] * In[0] + Rb[3 * i + 1] * Rb[3 * j + 1] * In[1] + Rb[3 * i + 2] * Rb[3 * j + 2] * In[2];
    const T cc = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
    v += ms * ((i == j ? cc : T(0.0)) - c[i] * c[j]);
    Ib[10 * b + 4 + e] = v;
    Ic[10 * b + 4 + e] = v;
  }
  DMX_TASKS(k, 4 * nb) {
    const int b = k / 4, e = k - 4 * b;
    const double ms = m.b_mass[b];
    T v;
    if (e == 0) v = ms; else v = ms * C[3 * b + e - 1];
    Ib[10 * b + e] = v;
    Ic[10 * b + e] = v;
  }
  g.sync();
}

// Task t of 6 n tasks (n vectors of 6 components), angular components of
// every vector first: the two kinds of component have different formulas.
struct Comp6 {
  int i, e;
};
__device__ __forceinline__ Comp6 comp6(int t, int n) {
  const int h = t < 3 * n ? t : t - 3 * n, i = h / 3;
  return {i, h - 3 * i + (t < 3 * n ? 0 : 3)};
}

// Composite-rigid-body algorithm: M (dense, both triangles).
template <int G, class T, class MD>
__device__ void crba(const Grp<G>& g, const MD& m, const WsT<T>& w) {
  const Layout& L = *w.L;
  T* Ic = w.at(L.Ic);
  const T* S = w.at(L.sd); T* F = w.at(L.F); T* M = w.at(L.M);
  const int nv = m.nv;
  tree_up<10>(g, m, Ic);             // Ic starts as Ib (kinematics)
  DMX_TASKS(t, 6 * nv) {
    const Comp6 c = comp6(t, nv);
    F[6 * c.i + c.e] = inertia_comp(Ic + 10 * m.dof_body[c.i], S + 6 * c.i, c.e);
  }
  g.sync();
  DMX_TASKS(t, nv * (nv + 1) / 2) {   // lower triangle
    const Tri ij = tri(t);
    const int i = ij.i, j = ij.j;
    T v = 0.0;
    if ((m.b_anc[m.dof_body[i]] >> m.dof_body[j]) & 1u) {
      const T* s = S + 6 * j; const T* f = F + 6 * i;
      v = s[0] * f[0] + s[1] * f[1] + s[2] * f[2] + s[3] * f[3] + s[4] * f[4] + s[5] * f[5];
    }
    M[i * nv + j] = v;
    M[j * nv + i] = v;
  }
  g.sync();
}

// Recursive Newton-Euler with zero joint acceleration: rhs0 = tau - c.
// Body velocities and velocity-product accelerations are sums along the path
// from the root: each body's own joint term is computed for all bodies at
// once, then added down the tree.  The per-body work is split by component
// (one body component per task).
template <int G, class T, class MD>
__device__ void rne_and_forces(const Grp<G>& g, const MD& m, const WsT<T>& w, const T* q, const T* v,
                               const T* u) {
  const Layout& L = *w.L;
  const T* Ib = w.at(L.Ib); const T* S = w.at(L.sd);
  T* V = w.at(L.Vb); T* A = w.at(L.Ab); T* Fb = w.at(L.Fb); T* IV = w.at(L.iv);
  const int nb = m.nbody, nt = 6 * nb;
  // own joint velocity S v
  DMX_TASKS(t, nt) {
    const int b = t / 6, e = t - 6 * b;
    const BodyInfo bi = body_info(m, b);
    const int va = bi.vadr, nd = bi.nv;
    T x = 0.0;
    int d = 0;
    if (nd == 6) { d = 3; if (e >= 3) x = v[va + e - 3]; }   // unit translation vectors
    for (; d < nd; ++d) x += S[6 * (va + d) + e] * v[va + d];
    V[t] = x;
  }
  g.sync();
  tree_down<6>(g, m, V);
  // own velocity-product acceleration (vb x S_d) v_d (gravity at the roots)
  DMX_TASKS(t, nt) {
    const Comp6 c = comp6(t, nb);
    const int b = c.i, e = c.e;
    const BodyInfo bi = body_info(m, b);
    const int va = bi.vadr, nd = bi.nv;
    T x = (bi.parent < 0 && e >= 3) ? T(-m.grav[e - 3]) : T(0.0);
    const int d0 = (bi.jtype == JNT_FREE) ? 3 : 0;   // world-fixed translation axes
    for (int d = d0; d < nd; ++d) x += crm_comp(V + 6 * b, S + 6 * (va + d), e) * v[va + d];
    A[6 * b + e] = x;
  }
  g.sync();
  tree_down<6>(g, m, A);
  // body forces I a + v x* (I v)
  DMX_TASKS(t, nt) {
    const Comp6 c = comp6(t, nb);
    const int b = c.i, e = c.e;
    Fb[6 * b + e] = inertia_comp(Ib + 10 * b, A + 6 * b, e);
    IV[6 * b + e] = inertia_comp(Ib + 10 * b, V + 6 * b, e);
  }
  g.sync();
  DMX_TASKS(t, nt) {
    const Comp6 c = comp6(t, nb);
    const int b = c.i, e = c.e;
    Fb[6 * b + e] += crf_comp(V + 6 * b, IV + 6 * b, e);
  }
  g.sync();
  tree_up<6>(g, m, Fb);
  T* rhs0 = w.at(L.rhs0);
  DMX_TASKS(i, m.nv) {
    const int b = m.dof_body[i];
    const T* s = S + 6 * i; const T* f = Fb + 6 * b;
    const T c = s[0] * f[0] + s[1] * f[1] + s[2] * f[2] + s[3] * f[3] + s[4] * f[4] + s[5] * f[5];
    const T tau = -m.b_damping[b] * v[i];
    T x = tau - c;
    for (int a = m.dof_act[i]; a >= 0; a = m.act_next[a]) {
      if (m.a_type[a] == ACT_MOTOR) x += m.a_gear[a] * u[a];
      else x += m.a_kp[a] * (u[a] - q[m.a_qadr[a]]) - m.a_kd[a] * v[i];
    }
    rhs0[i] = x;
  }
  g.sync();
}

// ------------------------------------------------------------------ collision
// contact record (16 scalars): r, pos[3], n[3], t1[3], t2[3], d, pterm, D
template <class T, class H>
__device__ __forceinline__ T box_sdf(const T* y, const H* h, T* grad) {
  T qd[3];
  bool out = false;
  for (int i = 0; i < 3; ++i) { qd[i] = fabs(y[i]) - h[i]; out = out || qd[i] > 0; }
  if (out) {
    T ss = 0.0;
    for (int i = 0; i < 3; ++i) if (qd[i] > 0) ss += qd[i] * qd[i];
    const T d = sqrt(ss), inv = 1.0 / d;
    for (int i = 0; i < 3; ++i) {
      const T gg = qd[i] > 0 ? qd[i] * inv : T(0.0);
      grad[i] = y[i] < 0 ? -gg : gg;
    }
    return d;
  }
  int k = 0;
  if (qd[1] > qd[k]) k = 1;
  if (qd[2] > qd[k]) k = 2;
  grad[0] = 0.0; grad[1] = 0.0; grad[2] = 0.0;
  grad[k] = y[k] < 0 ? -1.0 : 1.0;
  return qd[k];
}
// A number with the sign of the slope of the box distance field along
// y0 + s wv: outside the box the gradient is (sgn y_i max(|y_i| - h_i, 0))_i
// divided by the (positive) distance, so the division and the square root
// are left out; inside it is sgn(y_k) e_k for the axis k of the largest
// |y_k| - h_k (the same tie rule as box_sdf).
__device__ __forceinline__ double box_sdf_slope(const double* y0, const double* wv, double s, const double* h) {
  const double y[3] = {y0[0] + s * wv[0], y0[1] + s * wv[1], y0[2] + s * wv[2]};
  const double qd[3] = {fabs(y[0]) - h[0], fabs(y[1]) - h[1], fabs(y[2]) - h[2]};
  if (qd[0] > 0 || qd[1] > 0 || qd[2] > 0) {
    double num = 0.0;
    for (int i = 0; i < 3; ++i)
      if (qd[i] > 0) num += (y[i] < 0 ? -qd[i] : qd[i]) * wv[i];
    return num;
  }
  int k = 0;
  if (qd[1] > qd[k]) k = 1;
  if (qd[2] > qd[k]) k = 2;
  return y[k] < 0 ? -wv[k] : wv[k];
}

// Minimiser over the capsule axis s in [-Lh, Lh] of the box distance field
// along y0 + s wv (box frame), by bisection on its slope (values only).
__device__ __forceinline__ double capsule_box_s(const double* y0v, const double* wvv, double Lh, const double* h) {
  if (box_sdf_slope(y0v, wvv, -Lh, h) >= 0) return -Lh;
  if (box_sdf_slope(y0v, wvv, Lh, h) <= 0) return Lh;
  double lo = -Lh, hi = Lh;
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (box_sdf_slope(y0v, wvv, mid, h) < 0) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}
// Curvature phi'' of the distance along the axis at an interior minimiser sv
// outside the box, where the minimiser moves with the poses (implicit
// function theorem: ds = -d(slope) / phi'').  Returns 0 where s is held
// constant (an end of the axis, inside the box, or a flat direction).
__device__ __forceinline__ double capsule_box_curv(const double* y0v, const double* wvv, double sv, double Lh,
                                                   const double* h) {
  double yv[3] = {y0v[0] + sv * wvv[0], y0v[1] + sv * wvv[1], y0v[2] + sv * wvv[2]}, gv[3];
  const double phi = box_sdf(yv, h, gv);
  bool outside = false;
  for (int i = 0; i < 3; ++i) outside = outside || (fabs(yv[i]) - h[i] > 0);
  if (!(outside && sv > -Lh && sv < Lh && phi > 0)) return 0.0;
  const double gw = gv[0] * wvv[0] + gv[1] * wvv[1] + gv[2] * wvv[2];
  double ww = 0;
  for (int i = 0; i < 3; ++i) if (fabs(yv[i]) > h[i]) ww += wvv[i] * wvv[i];
  const double phi2 = (ww - gw * gw) / phi;
  return phi2 > 1e-12 ? phi2 : 0.0;
}

// Capsule (geom g1) against box (geom g2): minimum over the capsule axis of
// the box distance field (convex along the axis; bisection on its slope, in
// values).
template <class T>
__device__ void capsule_box(const DevModel& m, const T* gR, const T* gp, int g1, int g2, double thr, T* ct,
                            T* s_out) {
  const double rc = m.g_size[g1][0], Lh = m.g_size[g1][1];
  const double* h = m.g_size[g2];
  const T* R1 = gR + 9 * g1; const T* R2 = gR + 9 * g2;
  const T* c1 = gp + 3 * g1; const T* c2 = gp + 3 * g2;
  T dc[3] = {c1[0] - c2[0], c1[1] - c2[1], c1[2] - c2[2]};
  const double reach = m.g_bound[g1] + m.g_bound[g2] + (thr > 0 ? thr : 0.0);
  const double dd = dc[0] * dc[0] + dc[1] * dc[1] + dc[2] * dc[2];
  if (dd > reach * reach) { ct[0] = 1e30; return; }   // cannot be within the threshold
  const T u[3] = {R1[0], R1[3], R1[6]};
  T y0[3], wv[3];
  matTvec3(R2, dc, y0);
  matTvec3(R2, u, wv);
  const double y0v[3] = {y0[0], y0[1], y0[2]}, wvv[3] = {wv[0], wv[1], wv[2]};
  const double sv = capsule_box_s(y0v, wvv, Lh, h);
  *s_out = T(sv);
  T s = sv;
  T y[3] = {y0[0] + s * wv[0], y0[1] + s * wv[1], y0[2] + s * wv[2]}, gr[3], n[3];
  const T dist = box_sdf(y, h, gr);
  matvec3(R2, gr, n);
  const T r = dist - rc;
  ct[0] = r;
  const T off = rc + 0.5 * r;
  for (int i = 0; i < 3; ++i) { ct[1 + i] = c1[i] + s * u[i] - off * n[i]; ct[4 + i] = n[i]; }
  // tangent frame: t1 perpendicular to n and world z (world x when n is near z)
  double ref[3] = {0, 0, 1};
  if (fabs(n[2]) >= 0.5) { ref[0] = 1; ref[2] = 0; }
  T t1[3], t2[3];
  cross3(n, ref, t1);
  const T il = rsqrt(dot3(t1, t1));
  t1[0] *= il; t1[1] *= il; t1[2] *= il;
  cross3(n, t1, t2);
  for (int i = 0; i < 3; ++i) { ct[7 + i] = t1[i]; ct[10 + i] = t2[i]; }
}

// Sphere / capsule pair (the billiard's ball-ball contact of Sec. 4, capsule
// pairs of App. C.1): geom g is the segment c + s u, |s| <= L along its local
// x (L = 0 for a sphere), radius rad.  Closest points: the least of the
// candidates of the box-constrained optimality conditions of
// |D + s ua - t ub|^2 (D = ca - cb): the interior point (non-parallel axes)
// and each edge with the other parameter clamped.  n from geom 2 to geom 1,
// r = |d| - ra - rb, pos = pa - (ra + r/2) n; tangent frame as for
// capsule-box.  st_out: s, t.
__device__ __forceinline__ double seg_half(const DevModel& m, int g) {
  return m.g_type[g] == GEOM_CAPSULE ? m.g_size[g][1] : 0.0;
}
__device__ __forceinline__ void seg_closest(double c, double Du, double Dv, double La, double Lb, const double* D,
                                            const double* ua, const double* ub, double* s_out, double* t_out) {
  double bs = 0.0, bt = 0.0, best = INFINITY;
  auto consider = [&](double s, double t) {
    if (fabs(s) > La || fabs(t) > Lb) return;
    double d2 = 0.0;
    for (int i = 0; i < 3; ++i) {
      const double di = D[i] + s * ua[i] - t * ub[i];
      d2 += di * di;
    }
    if (d2 < best) { best = d2; bs = s; bt = t; }
  };
  if (1.0 - c * c > 1e-12) {
    const double s0 = (c * Dv - Du) / (1.0 - c * c);
    consider(s0, Dv + s0 * c);
  }
  consider(-La, fmin(fmax(Dv - La * c, -Lb), Lb));
  consider(La, fmin(fmax(Dv + La * c, -Lb), Lb));
  consider(fmin(fmax(-Lb * c - Du, -La), La), -Lb);
  consider(fmin(fmax(Lb * c - Du, -La), La), Lb);
  *s_out = bs;
  *t_out = bt;
}
template <class T>
__device__ void seg_seg(const DevModel& m, const T* gR, const T* gp, int g1, int g2, double thr, T* ct, T* st_out) {
  const double ra = m.g_size[g1][0], rb = m.g_size[g2][0];
  const double La = seg_half(m, g1), Lb = seg_half(m, g2);
  const T* R1 = gR + 9 * g1; const T* R2 = gR + 9 * g2;
  const T* c1 = gp + 3 * g1; const T* c2 = gp + 3 * g2;
  const T D[3] = {c1[0] - c2[0], c1[1] - c2[1], c1[2] - c2[2]};
  const double reach = m.g_bound[g1] + m.g_bound[g2] + (thr > 0 ? thr : 0.0);
  const double Dv0[3] = {D[0], D[1], D[2]};
  if (Dv0[0] * Dv0[0] + Dv0[1] * Dv0[1] + Dv0[2] * Dv0[2] > reach * reach) { ct[0] = 1e30; return; }
  const T ua[3] = {R1[0], R1[3], R1[6]}, ub[3] = {R2[0], R2[3], R2[6]};
  const double uav[3] = {ua[0], ua[1], ua[2]}, ubv[3] = {ub[0], ub[1], ub[2]};
  const double cv = dot3(uav, ubv), Duv = dot3(Dv0, uav), Dvv = dot3(Dv0, ubv);
  double sv, tv;
  seg_closest(cv, Duv, Dvv, La, Lb, Dv0, uav, ubv, &sv, &tv);
  st_out[0] = T(sv);
  st_out[1] = T(tv);
  T s = sv, t = tv;
  T d[3], n[3];
  for (int i = 0; i < 3; ++i) d[i] = D[i] + s * ua[i] - t * ub[i];
  const T rho = sqrt(dot3(d, d));
  const T ir = 1.0 / rho;
  for (int i = 0; i < 3; ++i) n[i] = d[i] * ir;
  const T r = rho - (ra + rb);
  ct[0] = r;
  const T off = ra + 0.5 * r;
  for (int i = 0; i < 3; ++i) { ct[1 + i] = c1[i] + s * ua[i] - off * n[i]; ct[4 + i] = n[i]; }
  double ref[3] = {0, 0, 1};
  if (fabs(n[2]) >= 0.5) { ref[0] = 1; ref[2] = 0; }
  T t1[3], t2[3];
  cross3(n, ref, t1);
  const T il = rsqrt(dot3(t1, t1));
  t1[0] *= il; t1[1] *= il; t1[2] *= il;
  cross3(n, t1, t2);
  for (int i = 0; i < 3; ++i) { ct[7 + i] = t1[i]; ct[10 + i] = t2[i]; }
}

// Spline of the solimp shape on x in [0, 1] (midpoint mid, power pw).
template <class T>
__device__ __forceinline__ T spline_shape(const T& x, double mid, double pw) {
  if (x <= mid && mid > 0) {
    const T num = (pw == 2.0) ? x * x : (pw == 4.0 ? (x * x) * (x * x) : pow(x, pw));
    return num / ((pw == 2.0) ? mid : ::pow(mid, pw - 1.0));
  }
  const T y = 1.0 - x;
  const T num = (pw == 2.0) ? y * y : (pw == 4.0 ? (y * y) * (y * y) : pow(y, pw));
  return 1.0 - num / ((pw == 2.0) ? (1.0 - mid) : ::pow(1.0 - mid, pw - 1.0));
}
// a / b for a model constant b > 0 whose reciprocal rb was rounded on the host
// and 0 <= a <= 2 b: the quotient estimate a rb corrected by its exact
// remainder (Markstein 1990: with rb correctly rounded this is the rounded
// quotient).  Three FP64 instructions.
__device__ __forceinline__ double div_const(double a, double b, double rb) {
  const double q = a * rb;
  return __fma_rn(__fma_rn(-b, q, a), rb, q);
}
// impedance(r) of the forward right-hand side, r < 0, in doubles, for the
// quadratic spline (power 2, every shipped setting): the same value, with the
// divisions by the width and the midpoint done by div_const.
__device__ __forceinline__ double impedance_quadratic(const DevModel& m, double r) {
  const double width = m.solimp[2], mid = m.solimp[3], a = fabs(r);
  const double x = below(a, width) ? div_const(a, width, m.imp_rwidth) : 1.0;
  const bool low = is_pos(mid) && !above(x, mid);
  const double y = low ? x : 1.0 - x, den = low ? mid : 1.0 - mid;
  const double num = y * y;
  double sh = is_pos(den) ? div_const(num, den, low ? m.imp_rmid : m.imp_rmid1) : num / den;
  if (!low) sh = 1.0 - sh;
  const double d = m.solimp[0] + (m.solimp[1] - m.solimp[0]) * sh;
  if (is_neg(d)) return 0.0;
  if (above(d, 0.9999)) return 0.9999;
  return d;
}
template <class T>
__device__ __forceinline__ T impedance(const DevModel& m, const T& r, bool cfd) {
  T d;
  if (cfd && r >= 0) {
    T x = 1.0 - r / m.cfd[2];
    if (x < 0) x = 0.0;
    d = m.cfd[0] + (m.cfd[1] - m.cfd[0]) * spline_shape(x, m.cfd[3], m.cfd[4]);
  } else {
    const double d_o = m.solimp[0], d_w = m.solimp[1], width = m.solimp[2], mid = m.solimp[3];
    T x = fabs(r) / width;
    if (x > 1.0) x = 1.0;
    d = d_o + (d_w - d_o) * spline_shape(x, mid, m.solimp[4]);
  }
  if (d < 0.0) return T(0.0);
  if (d > 0.9999) return T(0.9999);
  return d;
}
template <class T>
__device__ __forceinline__ T softplus(const T& x) { return x > 0 ? x + log1p(exp(-x)) : log1p(exp(x)); }

// All contact slots, then the included ones (r < 0, or r < w_c for F~) and
// their per-slot impedance terms.
template <int G, class T, class MD>
__device__ void collide(const Grp<G>& g, const MD& m, const WsT<T>& w, bool cfd) {
  const Layout& L = *w.L;
  const T* gR = w.at(L.gR); const T* gp = w.at(L.gp);
  T* CT = w.at(L.ct);
  const double thr = cfd ? m.cfd[2] : 0.0;
  DMX_TASKS(s, m.nslot) {
    T* ct = CT + 16 * s;
    const SlotInfo si = slot_info(m, s);
    const int j = si.idx, g1 = si.g1;
    if (si.g2 >= 0) {
      if (m.g_type[si.g2] == GEOM_BOX) capsule_box(m, gR, gp, g1, si.g2, thr, ct, w.at(L.csv) + 2 * s);
      else seg_seg(m, gR, gp, g1, si.g2, thr, ct, w.at(L.csv) + 2 * s);
    } else {
      const T* Rg = gR + 9 * g1; const T* cg = gp + 3 * g1;
      T pt[3];
      double rad = 0.0;
      const int ty = m.g_type[g1];
      if (ty == GEOM_SPHERE) { pt[0] = cg[0]; pt[1] = cg[1]; pt[2] = cg[2]; rad = m.g_size[g1][0]; }
      else if (ty == GEOM_CAPSULE) {
        const double e = (j == 0) ? -m.g_size[g1][1] : m.g_size[g1][1];
        pt[0] = cg[0] + e * Rg[0]; pt[1] = cg[1] + e * Rg[3]; pt[2] = cg[2] + e * Rg[6];
        rad = m.g_size[g1][0];
      } else {
        T t[3];
        const double ex[3] = {(j & 1) ? m.g_size[g1][0] : -m.g_size[g1][0],
                              (j & 2) ? m.g_size[g1][1] : -m.g_size[g1][1],
                              (j & 4) ? m.g_size[g1][2] : -m.g_size[g1][2]};
        matvec3(Rg, ex, t);
        pt[0] = cg[0] + t[0]; pt[1] = cg[1] + t[1]; pt[2] = cg[2] + t[2];
      }
      const T r = pt[2] - rad;
      ct[0] = r;
      ct[1] = pt[0]; ct[2] = pt[1]; ct[3] = pt[2] - (rad + 0.5 * r);
      ct[4] = 0.0; ct[5] = 0.0; ct[6] = 1.0; ct[7] = 1.0; ct[8] = 0.0; ct[9] = 0.0; ct[10] = 0.0; ct[11] = 1.0;
      ct[12] = 0.0;
    }
    const bool inc = cfd ? ct[0] < thr : is_neg(ct[0]);
    w.i[L.sinc + s] = inc ? 1 : 0;
    if (inc) {
      const T r = ct[0];
      const T d = (!cfd && m.solimp[4] == 2.0) ? impedance_quadratic(m, r) : impedance(m, r, cfd);
      const int pr = si.pair;
      const double ahat = m.s_rows[s] == 1 ? m.p_ahat[pr] : m.p_ahat_edge[pr];
      const double kc = m.kcoef;
      ct[13] = d;
      ct[14] = cfd ? kc * d * (m.softplus * softplus(-r / m.softplus)) : -(kc * d * r);
      ct[15] = d / (ahat * (1.0 - d));
    }
  }
  g.sync();
}

// Constraint rows of the included contacts (compacted in slot order).
// Returns the number of rows, or -1 when they exceed the workspace.
template <int G, class T, class MD>
__device__ int make_rows(const Grp<G>& g, const MD& m, const WsT<T>& w, const T* v, bool cfd) {
  const Layout& L = *w.L;
  const T* CT = w.at(L.ct); const T* S = w.at(L.sd);
  int* slotrow = w.i + L.slotrow; int* rowid = w.i + L.rowid; int* slist = w.i + L.slist;
  const int nv = m.nv;
  int* rowslot = w.i + L.rowslot;
  const int* sinc = w.i + L.sinc;
  // row and slot prefixes by group ballots (every slot has 1 or 4 rows)
  int n = 0, ns = 0;
  for (int s0 = 0; s0 < m.nslot; s0 += G) {
    const int s = s0 + g.lane;
    const bool inc = s < m.nslot && sinc[s] != 0;
    const int nrow = s < m.nslot ? m.s_rows[s] : 0;
    const unsigned b1 = g.ballot(inc && nrow == 1), b4 = g.ballot(inc && nrow != 1);
    const unsigned below = (1u << g.lane) - 1u;
    const int r0 = n + __popc(b1 & below) + 4 * __popc(b4 & below);
    if (s < m.nslot) slotrow[s] = inc ? r0 : -1;
    if (inc) {
      for (int e = 0; e < nrow && r0 + e < L.rcap; ++e) rowslot[r0 + e] = s;
      slist[ns + __popc((b1 | b4) & below)] = s;
    }
    n += __popc(b1) + 4 * __popc(b4);
    ns += __popc(b1 | b4);
  }
  if (g.lane == 0) slotrow[m.nslot] = n;
  g.sync();
  const int nr = n, nincl = ns;
  if (nr > L.rcap) return -1;
  T* J = w.at(L.J);
#pragma unroll 1
  for (int idx = g.lane, si = g.lane / nv, i = g.lane - si * nv; idx < nincl * nv;   // included slots only
       idx += G, i += G % nv, si += G / nv + (i >= nv), i -= (i >= nv) ? nv : 0) {
    const int s = slist[si];
    const int r0 = slotrow[s];
    const T* ct = CT + 16 * s;
    const int p = m.s_pair[s];
    const unsigned mv2 = slot_move2(m, s);
    const int bi = dof_info(m, i).body;
    const bool mA = (m.s_move[s] >> bi) & 1u, mB = (mv2 >> bi) & 1u;
    T jn = 0.0, j1 = 0.0, j2 = 0.0;
    if (mA != mB) {
      const T* sv = S + 6 * i;
      T pv[3];
      cross3(sv, ct + 1, pv);
      pv[0] += sv[3]; pv[1] += sv[4]; pv[2] += sv[5];
      if (mv2 == 0u) {   // ground plane: the frame is the world's (z, x, y)
        jn = pv[2]; j1 = pv[0]; j2 = pv[1];
      } else {
        jn = flip(dot3(ct + 4, pv), mB); j1 = flip(dot3(ct + 7, pv), mB); j2 = flip(dot3(ct + 10, pv), mB);
      }
    }
    if (m.s_rows[s] == 1) {
      J[r0 * nv + i] = jn;
    } else {
      const double mu = m.p_mu[p];
      J[r0 * nv + i] = jn + mu * j1;
      J[(r0 + 1) * nv + i] = jn - mu * j1;
      J[(r0 + 2) * nv + i] = jn + mu * j2;
      J[(r0 + 3) * nv + i] = jn - mu * j2;
    }
  }
  g.sync();
  T* aref = w.at(L.aref); T* Dr = w.at(L.Dr);
  DMX_TASKS(r, nr) {   // one row per task
    const int s = rowslot[r];
    const int e = r - slotrow[s];
    const int p = m.s_pair[s];
    const int nrow = m.s_rows[s];
    const T* ct = CT + 16 * s;
    T jv = 0.0;
    for (int i = 0; i < nv; ++i) jv += J[r * nv + i] * v[i];
    aref[r] = -(m.bcoef * jv) + ct[14];
    Dr[r] = ct[15];
    rowid[r] = m.p_row0[p] + m.s_idx[s] * nrow + e;
  }
  g.sync();
  return nr;
}

// ------------------------------------------------------------------ dense kernels
// H <- its Cholesky factor below the diagonal, invd <- 1 / diagonal of the
// factor.  With rows = n + 1 the row after H's last (a right side) takes part
// as another row of the factor: it leaves as L^-1 of the right side, the
// forward half of the solve, without steps of its own.  Returns false if not SPD.
template <int G, class T>
__device__ bool cholesky(const Grp<G>& g, T* H, T* invd, int n, int rows) {
  bool ok = true;
  const Tri t0 = tri(g.lane);          // this lane's first entry of every trailing block
  const int e0 = t0.i * n + 1 + t0.j, r0 = t0.i * n, c0 = t0.j * n;
  for (int k = 0; k < n; ++k) {
    const T hkk = H[k * n + k];
    ok = ok && is_pos(hkk);
    const T il = rsqrt(hkk);   // the diagonal of the factor is kept as its reciprocal
    for (int i = k + 1 + g.lane; i < rows; i += G) H[i * n + k] *= il;
    if (g.lane == 0) invd[k] = il;
    g.sync();
    const int nt = rows - k - 1, cnt = nt * (nt + 1) / 2 - (rows - n);
    T* Hk = H + (k + 1) * n + k;   // column k below the diagonal
    // lower triangle of the trailing block
    if (g.lane < cnt) Hk[e0] -= Hk[r0] * Hk[c0];
#pragma unroll 1
    for (int t = g.lane + G; t < cnt; t += G) {
      const Tri ij = tri(t);
      Hk[ij.i * n + 1 + ij.j] -= Hk[ij.i * n] * Hk[ij.j * n];
    }
    g.sync();
  }
  return ok;
}
// x <- L^-T x (the backward half of the solve).  With a lane per component
// the vector stays in registers and each step broadcasts one of them (two
// shuffles instead of two group meetings and a trip through shared memory:
// 155 against 270 cycles a step).
template <int G>
__device__ __forceinline__ double chol_back_lanes(const Grp<G>& g, const double* H, const double* invd, double xi,
                                                  int n) {
  for (int k = n - 1; k >= 0; --k) {
    const double xk = g.bcast(xi, k) * invd[k];
    if (g.lane == k) xi = xk;
    else if (g.lane < k) xi -= H[k * n + g.lane] * xk;
  }
  return xi;
}
template <int G, class T>
__device__ void chol_back(const Grp<G>& g, const T* H, const T* invd, T* x, int n) {
  if constexpr (G > 1) {
    if (n <= G) {
      const double xi = chol_back_lanes(g, H, invd, g.lane < n ? x[g.lane] : 0.0, n);
      if (g.lane < n) x[g.lane] = xi;
      g.sync();
      return;
    }
  }
  for (int k = n - 1; k >= 0; --k) {
    const T xk = x[k] * invd[k];
    g.sync();
    if (g.lane == 0) x[k] = xk;
    DMX_TASKS(i, k) x[i] -= H[k * n + i] * xk;
    g.sync();
  }
}
// x <- H^-1 x with the factor from cholesky().
template <int G, class T>
__device__ void chol_solve(const Grp<G>& g, const T* H, const T* invd, T* x, int n) {
  if constexpr (G > 1) {
    if (n <= G) {
      double xi = g.lane < n ? x[g.lane] : 0.0;
      for (int k = 0; k < n; ++k) {
        const double xk = g.bcast(xi, k) * invd[k];
        if (g.lane == k) xi = xk;
        else if (g.lane > k && g.lane < n) xi -= H[g.lane * n + k] * xk;
      }
      xi = chol_back_lanes(g, H, invd, xi, n);
      if (g.lane < n) x[g.lane] = xi;
      g.sync();
      return;
    }
  }
  for (int k = 0; k < n; ++k) {
    const T xk = x[k] * invd[k];
    g.sync();
    if (g.lane == 0) x[k] = xk;
    for (int i = k + 1 + g.lane; i < n; i += G) x[i] -= H[i * n + k] * xk;
    g.sync();
  }
  chol_back(g, H, invd, x, n);
}

__device__ __forceinline__ bool mask_has(const int* mk, int id) { return (mk[id >> 5] >> (id & 31)) & 1; }

// H = M + J_A^T D_A J_A, b = rhs0 + J_A^T D_A a_ref,A; factor; an = H^-1 b.
template <int G, class T, class MD>
__device__ bool solve_active(const Grp<G>& g, const MD& m, const WsT<T>& w, int nr, const int* act) {
  const Layout& L = *w.L;
  const int nv = m.nv;
  const T* M = w.at(L.M); T* H = w.at(L.H);
  const T* J = w.at(L.J); const T* aref = w.at(L.aref); const T* Dr = w.at(L.Dr);
  const T* rhs0 = w.at(L.rhs0); T* an = w.at(L.an);
  const int* rowid = w.i + L.rowid;
  int* alist = w.i + L.alist;
  // compacted list of the active rows (in row order)
  int na = 0;
  for (int r0 = 0; r0 < nr; r0 += G) {
    const int r = r0 + g.lane;
    const bool a = r < nr && mask_has(act, rowid[r]);
    const unsigned bits = g.ballot(a);
    if (a) alist[na + __popc(bits & ((1u << g.lane) - 1u))] = r;
    na += __popc(bits);
  }
  g.sync();
  // Lower triangle of H, then b as its extra row: one entry per task, entry
  // (i, j) = M_ij + sum_r X_ri J_rj with the D-scaled rows X = (D J, D a_ref)
  // of hb active rows at a time, so that a row costs an entry one
  // multiply-add (scaling inside costs two and a second pass for b).
  T* X = w.at(L.xd);
  const int nx1 = nv + 1, nent = nv * (nv + 1) / 2 + nv;
  const int hb = L.hb;
  for (int k0 = 0; k0 == 0 || k0 < na; k0 += hb) {
    const int nk = min(hb, na - k0);
    DMX_TASKS(t, nk * nx1) {
      const int k = t / nx1, i = t - k * nx1;
      const int r = alist[k0 + k];
      X[t] = Dr[r] * (i < nv ? J[r * nv + i] : aref[r]);
    }
    g.sync();
    DMX_TASKS(t, nent) {
      const Tri ij = tri(t);
      const int i = ij.i, j = ij.j;
      T h = k0 ? H[i * nv + j] : (i < nv ? M[i * nv + j] : rhs0[j]);
      if (nk == HBLK) {
#pragma unroll
        for (int k = 0; k < HBLK; ++k) h += X[k * nx1 + i] * J[alist[k0 + k] * nv + j];
      } else {
        for (int k = 0; k < nk; ++k) h += X[k * nx1 + i] * J[alist[k0 + k] * nv + j];
      }
      H[i * nv + j] = h;
    }
    g.sync();
  }
  const bool ok = cholesky(g, H, w.at(L.tmp2), nv, nv + 1);
  chol_back(g, (const T*)H, (const T*)w.at(L.tmp2), an, nv);
  return ok;
}

// z = J a - a_ref for every row; returns the active set {z < 0} in newmask.
template <int G, class T, class MD>
__device__ void residual_set(const Grp<G>& g, const MD& m, const WsT<T>& w, int nr, const T* a, int* newmask) {
  const Layout& L = *w.L;
  const int nv = m.nv;
  const T* J = w.at(L.J); const T* aref = w.at(L.aref);
  T* z = w.at(L.z);
  const int* rowid = w.i + L.rowid;
  unsigned bits[MASKW] = {0u, 0u, 0u, 0u};
  DMX_TASKS(r, nr) {
    T t = 0.0;
    for (int i = 0; i < nv; ++i) t += J[r * nv + i] * a[i];
    const T zr = t - aref[r];
    z[r] = zr;
    const int id = rowid[r];
    const unsigned bit = is_neg(zr) ? 1u << (id & 31) : 0u;
#pragma unroll
    for (int k = 0; k < MASKW; ++k) bits[k] |= (id >> 5) == k ? bit : 0u;
  }
#pragma unroll
  for (int k = 0; k < MASKW; ++k) newmask[k] = 32 * k < m.nrowid ? (int)g.ior(bits[k]) : 0;
  g.sync();
}

// Exact line search along d = an - a: minimiser over alpha >= 0 of the convex
// piecewise quadratic primal cost; breakpoints compared without divisions.
// The search only selects the next Newton iterate, so it runs on values.
template <int G, class T, class MD>
__device__ double line_search(const Grp<G>& g, const MD& m, const WsT<T>& w, int nr) {
  const Layout& L = *w.L;
  const int nv = m.nv;
  const T* M = w.at(L.M); const T* J = w.at(L.J); const T* Dr = w.at(L.Dr);
  const T* a = w.at(L.a); const T* an = w.at(L.an); const T* rhs0 = w.at(L.rhs0);
  T* dl = w.at(L.tmp); T* z = w.at(L.z); T* s = w.at(L.s);
  DMX_TASKS(i, nv) dl[i] = an[i] - a[i];
  g.sync();
  double c0 = 0, c1 = 0;
  DMX_TASKS(i, nv) {
    double ma = 0, md = 0;
    for (int j = 0; j < nv; ++j) { ma += M[i * nv + j] * a[j]; md += M[i * nv + j] * dl[j]; }
    c0 += dl[i] * (ma - rhs0[i]);
    c1 += dl[i] * md;
  }
  const T* aref = w.at(L.aref);
  DMX_TASKS(r, nr) {
    double t = 0, u = 0;
    for (int i = 0; i < nv; ++i) { t += J[r * nv + i] * dl[i]; u += J[r * nv + i] * a[i]; }
    s[r] = t;
    z[r] = u - aref[r];
  }
  g.sync();
  double s0 = 0, s1 = 0;
  DMX_TASKS(r, nr) {
    const double zr = z[r], sr = s[r], dr = Dr[r];
    const bool act = zr < 0 || (zr == 0 && sr < 0);
    if (act) { s0 += dr * zr * sr; s1 += dr * sr * sr; }
  }
  double slope0 = g.sum(c0) + g.sum(s0), slope1 = g.sum(c1) + g.sum(s1);
  // sweep the breakpoints below the current root (each row toggles at most once)
  unsigned long long tog0 = 0ull, tog1 = 0ull;
  for (int iter = 0; iter <= nr; ++iter) {
    // candidate rows: active ones leaving (s > 0) or inactive ones entering (s < 0, z > 0)
    // with breakpoint -z/s below the root -slope0/slope1 (slope1 > 0)
    int best = -1;
    double bz = 0, bs = 1;
    DMX_TASKS(r, nr) {
      if (((r < 64 ? tog0 : tog1) >> (r & 63)) & 1ull) continue;
      const double zr = z[r], sr = s[r];
      const bool act = zr < 0 || (zr == 0 && sr < 0);
      const bool cand = act ? (sr > 0) : (sr < 0 && zr > 0);
      if (!cand) continue;
      // -z/s < -slope0/slope1  <=>  z slope1 > s slope0 (s > 0) or z slope1 < s slope0 (s < 0)
      const double lhs = zr * slope1, rhs = sr * slope0;
      const bool below = sr > 0 ? (lhs > rhs) : (lhs < rhs);
      if (!below) continue;
      // smaller breakpoint: -z/s < -bz/bs  <=>  z bs * sign > bz s * sign with sign(s bs)
      if (best < 0) { best = r; bz = zr; bs = sr; continue; }
      const double l2 = zr * bs, r2 = bz * sr;
      const bool smaller = (sr * bs > 0) ? (l2 > r2) : (l2 < r2);
      if (smaller) { best = r; bz = zr; bs = sr; }
    }
    // group arg-min over lanes
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const int ob = __shfl_xor_sync(g.mask, best, o);
      const double oz = __shfl_xor_sync(g.mask, bz, o), os = __shfl_xor_sync(g.mask, bs, o);
      if (ob >= 0) {
        bool take = best < 0;
        if (!take) {
          const double l2 = oz * bs, r2 = bz * os;
          take = (os * bs > 0) ? (l2 > r2) : (l2 < r2);
          if (!take && !(l2 != r2)) take = ob < best;   // tie: lowest row index
        }
        if (take) { best = ob; bz = oz; bs = os; }
      }
    }
    if (best < 0) break;
    const double zb = z[best], sb = s[best], db = Dr[best];
    const bool act = zb < 0 || (zb == 0 && sb < 0);
    const double dz = db * zb * sb, ds = db * sb * sb;
    if (act) { slope0 -= dz; slope1 -= ds; } else { slope0 += dz; slope1 += ds; }
    if (best < 64) tog0 |= 1ull << best; else tog1 |= 1ull << (best - 64);
  }
  const double alpha = -slope0 / slope1;
  return alpha < 0 ? 0.0 : alpha;
}

// Unique minimiser of the primal problem -> an (= v').  With the active set A
// of the current iterate, an = H_A^-1 b_A is the minimiser of A's quadratic;
// it is the solution as soon as its own active set is A (the gradient of the
// primal cost vanishes there).  Otherwise Newton moves to the exact line
// minimum between the iterate and an.  The first candidate set is the final
// set of the previous right-hand side of this environment (pmask): when it is
// still right, one factorisation finishes the solve; when not, Newton starts
// from its solution.  pmask receives the final set.
// Returns 0 or an ENV_* code.
template <int G, class T, class MD>
__device__ int solve_constraints(const Grp<G>& g, const MD& m, const WsT<T>& w, int nr) {
  const Layout& L = *w.L;
  const int nv = m.nv;
  int* pm = w.i + L.pmask; int* am = w.i + L.amask;
  T* a = w.at(L.a); const T* an = w.at(L.an);
  int cur[MASKW], nxt[MASKW];
  for (int k = 0; k < MASKW; ++k) cur[k] = pm[k];
  bool ok = true;
  int status = ENV_SOLVER_NOCONV;
  for (int it = 0; it <= 50; ++it) {
    ok = solve_active(g, m, w, nr, cur) && ok;
    residual_set(g, m, w, nr, an, nxt);
    bool same = true;
    for (int k = 0; k < MASKW; ++k) same = same && (nxt[k] == cur[k]);
    if (same) { status = ENV_OK; break; }
    if (it == 0) {
      // start point of the Newton search: the solution of the first candidate set
      DMX_TASKS(i, nv) a[i] = an[i];
      for (int k = 0; k < MASKW; ++k) cur[k] = nxt[k];
      g.sync();
      continue;
    }
    const double alpha = line_search(g, m, w, nr);
    const T* dl = w.at(L.tmp);
    DMX_TASKS(i, nv) a[i] += alpha * dl[i];
    g.sync();
    residual_set(g, m, w, nr, (const T*)a, cur);
  }
  g.sync();
  if (g.lane == 0)
    for (int k = 0; k < MASKW; ++k) { pm[k] = cur[k]; am[k] = cur[k]; }
  g.sync();
  if (!ok) return ENV_SOLVER_NOCONV;
  return status;
}

// v' = F(q, v, u) (or F~ with cfd) into out[nv].  Returns 0 or an ENV_* code.
template <int G, class T, class MD>
__device__ int rhs(const Grp<G>& g, const MD& m, const WsT<T>& w, const T* q, const T* v,
                                const T* u, bool cfd, T* out) {
  const Layout& L = *w.L;
  kinematics(g, m, w, q);
  crba(g, m, w);
  rne_and_forces(g, m, w, q, v, u);
  collide(g, m, w, cfd);
  const int nr = make_rows(g, m, w, v, cfd);
  if (nr < 0) return ENV_ROW_OVERFLOW;
  const int st = solve_constraints(g, m, w, nr);
  const T* an = w.at(L.an);
  DMX_TASKS(i, m.nv) out[i] = an[i];
  g.sync();
  return st;
}

// ------------------------------------------------------------------ integrator
// Explicit one-step schemes as partitioned tableaus on (q, v).  Stage s
// (s = 1 .. S-1) takes V_s = v_n + h sum_{j<s} av[s][j] K_j and
// Q_s = q_n (+) h sum_{j<=s} aq[s][j] V_j (V_0 = v_n; a diagonal position
// coefficient uses the stage's own new velocity), K_s = F(Q_s, V_s, u); the
// last stage is the step's result and its K the next step's K_0 (first same
// as last).  e = b - bhat: weights of the embedded error estimate of the
// adaptive schemes.  nzq / nzv / enz: bit j set where the coefficient is
// non-zero, so that the stage sums skip zeros with an integer test.
enum { METHOD_DOPRI5 = 0, METHOD_TSIT5 = 1, METHOD_EULER = 2, NMETHOD = 3 };
struct Tab {
  int S, adaptive;
  double aq[7][7], av[7][7];
  double e[7];
  unsigned nzq[7], nzv[7], enz;
};
__host__ __device__ constexpr void finish_tab(Tab& t) {
  for (int s = 0; s < 7; ++s) {
    t.nzq[s] = 0u; t.nzv[s] = 0u;
    for (int j = 0; j < 7; ++j) {
      if (t.aq[s][j] != 0.0) t.nzq[s] |= 1u << j;
      if (t.av[s][j] != 0.0) t.nzv[s] |= 1u << j;
    }
  }
  t.enz = 0u;
  for (int j = 0; j < 7; ++j)
    if (t.e[j] != 0.0) t.enz |= 1u << j;
}
// Dormand & Prince (1980) 5(4): row 7 = the 5th-order weights b.
__host__ __device__ constexpr Tab make_dopri5() {
  Tab t{7, 1,
        {},
        {{0, 0, 0, 0, 0, 0, 0},
         {1.0 / 5.0, 0, 0, 0, 0, 0, 0},
         {3.0 / 40.0, 9.0 / 40.0, 0, 0, 0, 0, 0},
         {44.0 / 45.0, -56.0 / 15.0, 32.0 / 9.0, 0, 0, 0, 0},
         {19372.0 / 6561.0, -25360.0 / 2187.0, 64448.0 / 6561.0, -212.0 / 729.0, 0, 0, 0},
         {9017.0 / 3168.0, -355.0 / 33.0, 46732.0 / 5247.0, 49.0 / 176.0, -5103.0 / 18656.0, 0, 0},
         {35.0 / 384.0, 0.0, 500.0 / 1113.0, 125.0 / 192.0, -2187.0 / 6784.0, 11.0 / 84.0, 0}},
        {35.0 / 384.0 - 5179.0 / 57600.0, 0.0, 500.0 / 1113.0 - 7571.0 / 16695.0, 125.0 / 192.0 - 393.0 / 640.0,
         -2187.0 / 6784.0 + 92097.0 / 339200.0, 11.0 / 84.0 - 187.0 / 2100.0, -1.0 / 40.0},
        {}, {}, 0u};
  for (int s = 0; s < 7; ++s)
    for (int j = 0; j < 7; ++j) t.aq[s][j] = t.av[s][j];
  finish_tab(t);
  return t;
}
// Tsitouras (2011) 5(4) (the paper's default solver): row 7 = b, e its
// published error weights.
__host__ __device__ constexpr Tab make_tsit5() {
  Tab t{7, 1,
        {},
        {{0, 0, 0, 0, 0, 0, 0},
         {0.161, 0, 0, 0, 0, 0, 0},
         {-0.008480655492356989, 0.335480655492357, 0, 0, 0, 0, 0},
         {2.897153057105493, -6.359448489975075, 4.3622954328695815, 0, 0, 0, 0},
         {5.325864828439257, -11.748883564062828, 7.4955393428898365, -0.09249506636175525, 0, 0, 0},
         {5.86145544294642, -12.92096931784711, 8.159367898576159, -0.071584973281401, -0.028269050394068383, 0, 0},
         {0.09646076681806523, 0.01, 0.4798896504144996, 1.379008574103742, -3.290069515436081, 2.324710524099774,
          0}},
        {-0.00178001105222577714, -0.0008164344596567469, 0.007880878010261995, -0.1447110071732629,
         0.5823571654525552, -0.45808210592918697, 0.015151515151515152},
        {}, {}, 0u};
  for (int s = 0; s < 7; ++s)
    for (int j = 0; j < 7; ++j) t.aq[s][j] = t.av[s][j];
  finish_tab(t);
  return t;
}
// Semi-implicit Euler with a fixed step (the MuJoCo XLA integrator the paper
// compares against): v_{n+1} = v_n + h K_0, q_{n+1} = q_n (+) h v_{n+1}.
__host__ __device__ constexpr Tab make_euler() {
  Tab t{2, 0, {}, {}, {}, {}, {}, 0u};
  t.av[1][0] = 1.0;
  t.aq[1][1] = 1.0;
  finish_tab(t);
  return t;
}
struct TabSet {
  Tab t[NMETHOD];
};
__host__ __device__ constexpr TabSet make_tabs() { return TabSet{{make_dopri5(), make_tsit5(), make_euler()}}; }
static __constant__ TabSet c_tabs = make_tabs();
#define TAB(mt) (c_tabs.t[(mt)])

// q (+) dq for every joint (free: translation + body-frame rotation exponential).
template <class T>
__device__ __forceinline__ void rot_exp(const T& th2, T& cw, T& sk) {   // cos(th / 2), sin(th / 2) / th
  if (th2 < 1e-2) {
    // |dq| < 0.1 rad: Taylor series of cos(th/2) and sin(th/2)/th in th^2
    // (the next terms are below 3e-20): no square root, sine or division
    cw = 1.0 + th2 * (-1.0 / 8.0 + th2 * (1.0 / 384.0 + th2 * (-1.0 / 46080.0 + th2 * (1.0 / 10321920.0))));
    sk = 0.5 + th2 * (-1.0 / 48.0 + th2 * (1.0 / 3840.0 + th2 * (-1.0 / 645120.0 + th2 * (1.0 / 185794560.0))));
  } else {
    const T th = sqrt(th2);
    T sn, cs;
    sincos(0.5 * th, &sn, &cs);
    cw = cs;
    sk = sn / th;
  }
}
// A free joint's quaternion takes four lanes, one component each: a lane
// evaluates one of the two series, the products of its component and the
// (shared) normalisation, 25 FP64 instructions on the longest path instead of
// 46 on one lane.
template <int G, class MD>
__device__ void integrate_pos_lanes(const Grp<G>& g, const MD& m, const double* q, const double* dq,
                                    double* out) {
  for (int t0 = 0; t0 < 4 * m.nbody; t0 += G) {
    const int t = t0 + g.lane, b = min(t >> 2, m.nbody - 1), c = t & 3;
    const bool live = t < 4 * m.nbody;
    const BodyInfo bi = body_info(m, b);
    const int qa = bi.qadr, va = bi.vadr;
    if (bi.jtype == JNT_HINGE) {
      if (live && c == 0) out[qa] = q[qa] + dq[va];
    } else if (live && c < 3) {
      out[qa + c] = q[qa + c] + dq[va + c];
    }
    const bool fr = live && bi.jtype == JNT_FREE;
    if (!g.ballot(fr)) continue;
    double cw = 1.0, sk = 0.5, d[3] = {0.0, 0.0, 0.0}, x[4] = {1.0, 0.0, 0.0, 0.0};
    if (fr) {
      for (int k = 0; k < 3; ++k) d[k] = dq[va + 3 + k];
      for (int k = 0; k < 4; ++k) x[k] = q[qa + 3 + k];
    }
    const double th2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const bool small = below(th2, 1e-2);
    // |dq| < 0.1 rad: the Taylor series of rot_exp, cos on even lanes, sine on odd ones
    const bool od = c & 1;
    const double k4 = od ? 1.0 / 185794560.0 : 1.0 / 10321920.0, k3 = od ? -1.0 / 645120.0 : -1.0 / 46080.0;
    const double k2 = od ? 1.0 / 3840.0 : 1.0 / 384.0, k1 = od ? -1.0 / 48.0 : -1.0 / 8.0, k0 = od ? 0.5 : 1.0;
    const double sr = k0 + th2 * (k1 + th2 * (k2 + th2 * (k3 + th2 * k4)));
    const double so = __shfl_xor_sync(g.mask, sr, 1);
    cw = od ? so : sr;
    sk = od ? sr : so;
    if (fr && !small) rot_exp(th2, cw, sk);
    const double e[4] = {cw, sk * d[0], sk * d[1], sk * d[2]};
    // component c of x (x) e: x0 e_c then the pairs (k, c ^ k), minus for k = c and along the cycle
    const double E0 = c == 0 ? e[0] : c == 1 ? e[1] : c == 2 ? e[2] : e[3];
    const double E1 = flip(c == 0 ? e[1] : c == 1 ? e[0] : c == 2 ? e[3] : e[2], c == 0 || c == 2);
    const double E2 = flip(c == 0 ? e[2] : c == 1 ? e[3] : c == 2 ? e[0] : e[1], c == 0 || c == 3);
    const double E3 = flip(c == 0 ? e[3] : c == 1 ? e[2] : c == 2 ? e[1] : e[0], c < 2);
    const double r = x[0] * E0 + x[1] * E1 + x[2] * E2 + x[3] * E3;
    const double rw = __shfl_sync(g.mask, r, 0, 4), rx = __shfl_sync(g.mask, r, 1, 4);
    const double ry = __shfl_sync(g.mask, r, 2, 4), rz = __shfl_sync(g.mask, r, 3, 4);
    const double in = rsqrt(rw * rw + rx * rx + ry * ry + rz * rz);
    if (fr) out[qa + 3 + c] = r * in;
  }
  g.sync();
}
template <int G, class T, class MD>
__device__ void integrate_pos(const Grp<G>& g, const MD& m, const T* q, const T* dq, T* out) {
  if constexpr (G >= 4) {
    integrate_pos_lanes(g, m, q, dq, out);
  } else {
    DMX_TASKS(b, m.nbody) {
      const int qa = m.b_qadr[b], va = m.b_vadr[b];
      if (m.b_jtype[b] == JNT_HINGE) { out[qa] = q[qa] + dq[va]; continue; }
      out[qa] = q[qa] + dq[va]; out[qa + 1] = q[qa + 1] + dq[va + 1]; out[qa + 2] = q[qa + 2] + dq[va + 2];
      const T* d = dq + va + 3;
      const T th2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
      T cw, sk;
      rot_exp(th2, cw, sk);
      const T ex = sk * d[0], ey = sk * d[1], ez = sk * d[2];
      const T w0 = q[qa + 3], a0 = q[qa + 4], b0 = q[qa + 5], c0 = q[qa + 6];
      const T rw = w0 * cw - a0 * ex - b0 * ey - c0 * ez;
      const T rx = w0 * ex + a0 * cw + b0 * ez - c0 * ey;
      const T ry = w0 * ey - a0 * ez + b0 * cw + c0 * ex;
      const T rz = w0 * ez + a0 * ey - b0 * ex + c0 * cw;
      const T in = rsqrt(rw * rw + rx * rx + ry * ry + rz * rz);
      out[qa + 3] = rw * in; out[qa + 4] = rx * in; out[qa + 5] = ry * in; out[qa + 6] = rz * in;
    }
    g.sync();
  }
}

// Magnitude used by the error norm for tangent component i of the positions.
template <class MD>
__device__ __forceinline__ double pos_mag(const MD& m, const double* q, int i) {
  const int b = m.dof_body[i];
  if (m.b_jtype[b] == JNT_HINGE) return fabs(q[m.b_qadr[b]]);
  const int d = i - m.b_vadr[b];
  return d < 3 ? fabs(q[m.b_qadr[b] + d]) : 1.0;
}

// The new stages of one step of scheme mt (TAB(mt)) of size h from (qn, vn)
// with ka[0] = F(qn, vn): stage velocities kv[s], derivatives ka[s], the
// result in (qs, vs) and its derivative in ka[(S-1) nv].  hook(s, status)
// runs after the right-hand side of stage s (the workspace then holds that
// evaluation).  Returns the worst stage status.
template <int G, class Hook, class MD>
__device__ int rk_stages(const Grp<G>& g, const MD& m, const Ws& w, const double* u, double h, int mt,
                         Hook&& hook) {
  const Layout& L = *w.L;
  const int nv = m.nv, S = TAB(mt).S;
  const double* qn = w.at(L.qn); const double* vn = w.at(L.vn);
  double* qs = w.at(L.qs); double* vs = w.at(L.vs);
  double* kv = w.at(L.kv); double* ka = w.at(L.ka); double* dq = w.at(L.dq);
  int st = 0;
  DMX_TASKS(i, nv) kv[i] = vn[i];
  g.sync();
  for (int s = 1; s < S; ++s) {
    const unsigned mq = TAB(mt).nzq[s], mv = TAB(mt).nzv[s];
    DMX_TASKS(i, nv) {
      double sq = 0, sv = 0;
      for (int j = 0; j < s; ++j) {
        if ((mq >> j) & 1u) sq += TAB(mt).aq[s][j] * kv[j * nv + i];
        if ((mv >> j) & 1u) sv += TAB(mt).av[s][j] * ka[j * nv + i];
      }
      const double vv = vn[i] + h * sv;
      if ((mq >> s) & 1u) sq += TAB(mt).aq[s][s] * vv;
      dq[i] = h * sq;
      vs[i] = vv;
      kv[s * nv + i] = vv;
    }
    g.sync();
    integrate_pos(g, m, qn, dq, qs);
    const int r = rhs(g, m, w, qs, vs, u, false, ka + s * nv);
    if (r > st) st = r;
    hook(s, r);
  }
  return st;
}

// Sum of x[0..n) (shared memory, consumed) in the order of a shuffle
// reduction over C lanes: component i first joins lane i mod C's partial sum,
// then the partial sums meet in a binary tree.  The order is C's whatever the
// group's own lane count, so that the lane count can follow the hardware
// without touching a single step decision.
template <int G>
__device__ double sum_as_lanes(const Grp<G>& g, double* x, int n, int C) {
  DMX_TASKS(c, min(C, n - C)) {
    double acc = x[c];
    for (int i = c + C; i < n; i += C) acc += x[i];
    x[c] = acc;
  }
  g.sync();
  const int np = min(n, C);          // partial sums that exist
  for (int o = C >> 1; o > 0; o >>= 1) {
    if (o >= np) continue;
    DMX_TASKS(c, min(o, np - o)) x[c] += x[c + o];
    g.sync();
  }
  return x[0];
}

// One attempt of scheme mt of size h from (qn, vn) with ka[0] = F(qn, vn).
// Leaves the result in (qs, vs) and its derivative in ka[(S-1) nv]; returns
// the RMS error norm of the embedded estimate (NaN-safe: non-finite -> +inf;
// 0 for a fixed-step scheme; summed in the order of `red` lanes) and the
// worst stage status.
template <int G, class Hook, class MD>
__device__ double rk_attempt(const Grp<G>& g, const MD& m, const Ws& w, const double* u, double h, int mt,
                             double rtol, double atol, int red, int* st_out, Hook&& hook) {
  const Layout& L = *w.L;
  const int nv = m.nv;
  const double* qn = w.at(L.qn); const double* vn = w.at(L.vn);
  const double* qs = w.at(L.qs); const double* vs = w.at(L.vs);
  const double* kv = w.at(L.kv); const double* ka = w.at(L.ka);
  const int st = rk_stages(g, m, w, u, h, mt, hook);
  *st_out = st;
  if (!TAB(mt).adaptive) return 0.0;
  const unsigned enz = TAB(mt).enz;
  double* terms = w.at(L.dq);        // free after the last stage
  DMX_TASKS(i, nv) {
    double ep = 0, ev = 0;
    for (int j = 0; j < 7; ++j) {
      if (!((enz >> j) & 1u)) continue;
      const double c = TAB(mt).e[j];
      ep += c * kv[j * nv + i];
      ev += c * ka[j * nv + i];
    }
    ep *= h; ev *= h;
    const double sp = atol + rtol * max_pos(pos_mag(m, qn, i), pos_mag(m, qs, i));
    const double sv = atol + rtol * max_pos(fabs(vn[i]), fabs(vs[i]));
    const double r1 = ep / sp, r2 = ev / sv;
    terms[i] = r1 * r1 + r2 * r2;
  }
  g.sync();
  const double acc = sum_as_lanes(g, terms, nv, red);
  g.sync();
  const double err = sqrt(acc / (2.0 * nv));
  return isfinite(err) ? err : INFINITY;
}

template <int G, class MD>
__device__ double rk_attempt(const Grp<G>& g, const MD& m, const Ws& w, const double* u, double h, int mt,
                             double rtol, double atol, int red, int* st_out) {
  return rk_attempt(g, m, w, u, h, mt, rtol, atol, red, st_out, [](int, int) {});
}
}  // namespace dmx
