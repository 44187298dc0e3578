// Compiled model and per-environment workspace layout, shared by the host
// runtime (which fills them) and the device kernels (which read them).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define DMX_HD __host__ __device__
#else
#define DMX_HD
#endif

namespace dmx {

// Capacity limits of the compiled model (checked by dmx_create_model).
constexpr int MAXB = 16;      // bodies
constexpr int MAXV = 24;      // dofs
constexpr int MAXQ = 32;      // position coordinates
constexpr int MAXG = 24;      // geoms
constexpr int MAXBOX = 4;     // box geoms (side-length parameters)
constexpr int MAXP = 24;      // contact pairs
constexpr int MAXS = 32;      // contact slots
constexpr int MAXU = 16;      // actuators
constexpr int MAXROWID = 128; // constraint rows over all slots (stable row ids)
// Constraint rows one right-hand side can hold (the included contacts' rows,
// compacted): the Jacobian and row arrays of the per-environment workspace
// are sized min(row ids, ROWCAP), which keeps shared memory per environment,
// hence warps per SM, independent of how many slots a model declares; a state
// with more included rows reports ENV_ROW_OVERFLOW.
constexpr int ROWCAP = 64;
constexpr int MAXLEV = 12;    // depth of the body tree
constexpr int MASKW = MAXROWID / 32;
constexpr int HBLK = 8;       // active rows per block of the Newton matrix assembly, at most

enum { JNT_FREE = 0, JNT_HINGE = 1 };
enum { GEOM_SPHERE = 0, GEOM_CAPSULE = 1, GEOM_BOX = 2 };
enum { ACT_MOTOR = 0, ACT_POSITION = 1 };
// Model parameters the adjoint differentiates (dmx_rollout_grad_params): solref
// (t_c, phi_d), solimp (d_o, d_w, width, midpoint), then the friction
// coefficient of every pair.
enum { PAR_TC = 0, PAR_DAMP = 1, PAR_DO = 2, PAR_DW = 3, PAR_WIDTH = 4, PAR_MID = 5, PAR_MU0 = 6 };
enum { ENV_OK = 0, ENV_MAX_STEPS = 1, ENV_H_UNDERFLOW = 2, ENV_NONFINITE = 3, ENV_SOLVER_NOCONV = 4,
       ENV_ROW_OVERFLOW = 5 };

struct DevModel {
  int nbody, ngeom, npair, nact, nq, nv, nu, nslot, nrowid, nlevel;
  double grav[3];
  double bcoef, kcoef;               // a_ref = -bcoef (J v) - kcoef d(r) r
  double solref[2];                  // t_c, phi_d (bcoef = 2 / (d_w t_c), kcoef = 1 / (d_w^2 t_c^2 phi_d^2))
  double solimp[5];                  // d_o, d_w, width, midpoint, power
  double cfd[5];                     // d_c, d_0, w_c, m_c, p_c
  double softplus;
  double imp_rwidth, imp_rmid, imp_rmid1;   // reciprocals of the spline's width, midpoint and 1 - midpoint
  // bodies (topological order)
  int b_parent[MAXB], b_jtype[MAXB], b_qadr[MAXB], b_vadr[MAXB], b_nv[MAXB];
  unsigned b_anc[MAXB];              // bit j: body j is this body or an ancestor
  double b_pos[MAXB][3], b_Roff[MAXB][9], b_axis[MAXB][3];
  double b_mass[MAXB], b_com[MAXB][3], b_inertia[MAXB][3], b_damping[MAXB];
  int b_ident[MAXB];                 // 1: b_Roff is exactly the identity
  int child_start[MAXB], child_count[MAXB], child_list[MAXB];
  int level_start[MAXLEV + 1], level_list[MAXB];
  int dof_body[MAXV];
  // Chains of the body tree: maximal runs in which every body but the last has
  // exactly one child, ordered by levels (a chain's head hangs on a chain of an
  // earlier level, or on the world), so that one lane can carry a component
  // down or up a whole run without meeting the others.
  int nchlev, chlev_start[MAXLEV + 1];                 // chain levels: ranges of chains
  int ch_start[MAXB + 1], ch_list[MAXB], ch_par[MAXB]; // bodies of each chain (head first), parent of its head (-1 = world)
  // the same tables packed, one read each (BodyInfo, DofInfo, SlotInfo)
  unsigned long long b_pack[MAXB];   // bytes: parent (255 = world), joint, qadr, vadr, nv, ident
  unsigned dof_pack[MAXV];           // bytes: body, index within its joint, joint
  unsigned s_pack[MAXS];             // bytes: pair, index within the pair, geom 1, geom 2 (255 = plane)
  unsigned s_move2[MAXS];            // bodies that move geom 2 of the slot (0: plane)
  int lv_pack[MAXB];                 // k-th body in level order: body | parent << 8 (parent 255 = world)
  int dof_act[MAXV], act_next[MAXU]; // first actuator on a dof (-1 = none), next one on the same dof
  // geoms
  int g_type[MAXG], g_body[MAXG];
  double g_pos[MAXG][3], g_Roff[MAXG][9], g_size[MAXG][3];
  double g_bound[MAXG];              // bounding-sphere radius about the geom centre
  int g_box[MAXG];                   // index among the box geoms (side-length parameter), else -1
  int nbox;
  int b_solebox[MAXB];               // geom index of the body's only geom when it is a box (its inertia follows the side), else -1
  int g_ident[MAXG], g_zpos[MAXG];   // 1: g_Roff is exactly the identity / g_pos is exactly zero
  // pairs and slots
  int p_g1[MAXP], p_g2[MAXP], p_condim[MAXP], p_slot0[MAXP], p_nslot[MAXP], p_row0[MAXP];
  double p_mu[MAXP], p_ahat[MAXP], p_ahat_edge[MAXP];
  double p_dahat[MAXP][MAXB + MAXBOX];   // d A_hat / d (mass of each body, then side of each box)
  int s_pair[MAXS], s_idx[MAXS];
  int s_rows[MAXS];                  // constraint rows of the slot (1 or 4)
  unsigned s_rdofs[MAXS];            // dofs with an angular motion vector that move geom 1 of the slot
  unsigned s_move[MAXS];             // bodies that move geom 1 of the slot (bit mask: its body and its ancestors)
  unsigned g_slots1[MAXG], g_slots2[MAXG];   // bit s: the geom is geom 1 / geom 2 of slot s
  unsigned b_geoms[MAXB];            // bit g: geom g is fixed to the body
  unsigned dof_anc[MAXV], dof_desc[MAXV];    // dofs j <= i of the dof's ancestor bodies, k >= i of its descendants (with its own)
  int s_barofs[MAXS], nslotbar;      // adjoint: offset / total of the per-slot pose cotangents
                                     // (12 doubles for a plane slot, 24 for a geom pair)
  // actuators
  int a_type[MAXU], a_qadr[MAXU], a_vadr[MAXU];
  double a_gear[MAXU], a_kp[MAXU], a_kd[MAXU];
};

// A model of one free body with ground-plane contacts only (ball, box, toss),
// as the device code sees it: the same data with the tree, dof and pair tables
// known to the compiler.  The functions over a model type then lose their
// loops over bodies and levels, joint types, index reads and geom pairs, and
// unroll the sums over six dofs (a right-hand side runs 13 instructions per
// FP64 instruction otherwise): 4096 box pushes 180 -> 135 ms, 20001 tosses 212 ->
// 155, 2048 toss gradients 127 -> 102.  The table members only hide the base's; they
// hold no data, and a DevModel is read through this type by a cast.
template <int V>
struct ConstTab {
  DMX_HD constexpr int operator[](int) const { return V; }
};
struct OneBody : DevModel {
  static constexpr int nbody = 1, nlevel = 1, nq = 7, nv = 6, nu = 0, nact = 0;
  ConstTab<-1> b_parent, p_g2, dof_act;
  ConstTab<JNT_FREE> b_jtype;
  ConstTab<0> b_qadr, b_vadr, dof_body, g_body, child_count;
  ConstTab<6> b_nv;
  ConstTab<1> b_anc, s_move;
};
// A model without geom pairs (the quadruped): the device code loses the
// capsule-box and segment-pair contacts (3000 quadrupeds 283 -> 278 ms).
struct PlaneOnly : DevModel {
  ConstTab<-1> p_g2;
};
enum { MODEL_GENERAL = 0, MODEL_ONE_BODY = 1, MODEL_PLANE_ONLY = 2 };   // DevModel, OneBody, PlaneOnly
template <class MD>
constexpr bool plane_only_v = false;
template <>
constexpr bool plane_only_v<OneBody> = true;
template <>
constexpr bool plane_only_v<PlaneOnly> = true;
template <class MD>
constexpr bool one_body_v = false;
template <>
constexpr bool one_body_v<OneBody> = true;
struct BodyInfo {
  int parent, jtype, qadr, vadr, nv, ident;
};
template <class MD>
DMX_HD inline BodyInfo body_info(const MD& m, int b) {
  if constexpr (one_body_v<MD>) return {-1, JNT_FREE, 0, 0, 6, 1};
  else {
    const unsigned long long x = m.b_pack[b];
    const int par = (int)(x & 255u);
    return {par == 255 ? -1 : par, (int)(x >> 8 & 255u), (int)(x >> 16 & 255u), (int)(x >> 24 & 255u),
            (int)(x >> 32 & 255u), (int)(x >> 40 & 255u)};
  }
}
struct DofInfo {
  int body, k;                       // its body and its index within the joint
  bool free, translation;            // of a free joint; one of its translations
};
template <class MD>
DMX_HD inline DofInfo dof_info(const MD& m, int i) {
  if constexpr (one_body_v<MD>) return {0, i, true, i < 3};
  else {
    const unsigned x = m.dof_pack[i];
    const int k = (int)(x >> 8 & 255u);
    const bool fr = (x >> 16 & 255u) == (unsigned)JNT_FREE;
    return {(int)(x & 255u), k, fr, fr && k < 3};
  }
}
struct SlotInfo {
  int pair, idx, g1, g2;             // g2 = -1: ground plane
};
template <class MD>
DMX_HD inline SlotInfo slot_info(const MD& m, int s) {
  const unsigned x = m.s_pack[s];
  const int g2 = (int)(x >> 24);
  return {(int)(x & 255u), (int)(x >> 8 & 255u), (int)(x >> 16 & 255u), plane_only_v<MD> || g2 == 255 ? -1 : g2};
}
template <class MD>
DMX_HD inline unsigned slot_move2(const MD& m, int s) {
  return plane_only_v<MD> ? 0u : m.s_move2[s];
}
inline bool is_plane_only(const DevModel& m) {
  for (int p = 0; p < m.npair; ++p)
    if (m.p_g2[p] >= 0) return false;
  return true;
}
inline bool is_one_body(const DevModel& m) {
  return m.nbody == 1 && m.b_jtype[0] == JNT_FREE && m.nact == 0 && is_plane_only(m);
}

// Offsets (in doubles / ints) of one environment's shared-memory workspace.
struct Layout {
  int qn, vn, qs, vs, kv, ka, dq;
  int R, p, com, sd, Ib, Ic, F, Vb, Ab, Fb, iv, gR, gp;
  int M, H, rhs0, a, an, tmp, tmp2;
  int ct, csv, J, aref, Dr, z, s, u;   // csv: closest-point parameters of each geom-pair slot (2 per slot)
  int xd, hb;                        // D-scaled rows (J, a_ref) of hb active rows (Newton matrix assembly)
  int nd;                            // doubles per environment (padded to even)
  int xl, sc;                        // kinematics scratch, aliases of Ab..Fb (12 per body) and iv (2 per body)
  int rowid, slotrow, slist, amask, pmask, misc;
  int sinc, rowslot, alist;          // slot included (0/1), slot of each row, compacted active rows
  int ni;                            // ints per environment
  int rcap;                          // constraint-row capacity
  int xbar;                          // adjoint layout: state cotangent (nq + nv), else -1
  int ovl;                           // adjoint layout: start of the arrays the VJP never reads, else nd
};

// Active rows per block of the Newton matrix assembly: as many D-scaled rows
// of nv + 1 as fit the larger of the arrays that are free meanwhile (residuals
// and line-search slopes, 2 per row; I V of the bias force, 6 per body).
DMX_HD inline int newton_block(int nv, int nb, int rcap) {
  const int h = (6 * nb > 2 * rcap ? 6 * nb : 2 * rcap) / (nv + 1);
  return h < 1 ? 1 : (h > HBLK ? HBLK : h);
}

DMX_HD inline Layout make_layout(const DevModel& m, int rcap) {
  Layout L{};
  int o = 0;
  const int nq = m.nq, nv = m.nv, nb = m.nbody, ng = m.ngeom, ns = m.nslot > 0 ? m.nslot : 1;
  auto take = [&](int n) { int r = o; o += n; return r; };
  L.qn = take(nq); L.vn = take(nv); L.qs = take(nq); L.vs = take(nv);
  L.kv = take(7 * nv); L.ka = take(7 * nv); L.dq = take(nv);
  L.R = take(9 * nb); L.p = take(3 * nb); L.com = take(3 * nb); L.sd = take(6 * nv);
  L.Ib = take(10 * nb); L.Ic = take(10 * nb); L.F = take(6 * nv);
  L.Vb = take(6 * nb); L.Ab = take(6 * nb); L.Fb = take(6 * nb); L.iv = take(6 * nb);
  // the bias-force arrays are free while the kinematics run: local transforms
  // (Ab and Fb are contiguous, 12 per body) and per-body scalars (iv)
  L.xl = L.Ab; L.sc = L.iv;
  L.gR = take(9 * ng); L.gp = take(3 * ng);
  L.M = take(nv * nv); L.H = take(nv * nv);
  L.an = take(nv);                   // directly after H: its extra row (cholesky)
  L.rhs0 = take(nv); L.a = take(nv); L.tmp = take(nv); L.tmp2 = take(nv);
  L.ct = take(16 * ns); L.csv = take(2 * ns);
  L.J = take(rcap * nv); L.aref = take(rcap); L.Dr = take(rcap); L.z = take(rcap); L.s = take(rcap);
  L.hb = newton_block(nv, nb, rcap);
  L.xd = 6 * nb > 2 * rcap ? L.iv : L.z;
  if (nv + 1 > 6 * nb && nv + 1 > 2 * rcap) L.xd = take(nv + 1);   // a free body with a row or two
  L.u = take(m.nu > 0 ? m.nu : 1);
  L.nd = (o + 1) & ~1;
  int i = 0;
  auto takei = [&](int n) { int r = i; i += n; return r; };
  L.rowid = takei(rcap); L.slotrow = takei(ns + 1); L.slist = takei(ns); L.amask = takei(MASKW);
  L.pmask = takei(MASKW);
  L.misc = takei(8);
  L.sinc = takei(ns); L.rowslot = takei(rcap); L.alist = takei(rcap);
  L.ni = (i + 3) & ~3;
  L.rcap = rcap;
  L.xbar = -1;
  L.ovl = L.nd;
  return L;
}

// Workspace of the reverse adjoint kernel when it restores stage snapshots:
// the same arrays, ordered so that everything the right-hand-side VJP reads
// (poses .. geom frames, the final Newton factor and solution, capsule-box
// minimisers, D and the residuals of the rows, controls) and the running
// state cotangent come first, and the arrays only the segment recompute uses
// (stage state, M, contact records, Jacobian rows, a_ref, line-search slopes)
// start at ovl.  During the reverse sweep the cotangent workspace occupies
// [ovl, ...): the VJP reads the contact records and Jacobian rows from the
// snapshot in device memory instead.
DMX_HD inline Layout make_layout_adj(const DevModel& m, int rcap) {
  Layout L = make_layout(m, rcap);
  int o = 0;
  const int nq = m.nq, nv = m.nv, nb = m.nbody, ng = m.ngeom, ns = m.nslot > 0 ? m.nslot : 1;
  auto take = [&](int n) { int r = o; o += n; return r; };
  L.R = take(9 * nb); L.p = take(3 * nb); L.com = take(3 * nb); L.sd = take(6 * nv);
  L.Ib = take(10 * nb); L.Ic = take(10 * nb); L.F = take(6 * nv);
  L.Vb = take(6 * nb); L.Ab = take(6 * nb); L.Fb = take(6 * nb); L.iv = take(6 * nb);
  L.xl = L.Ab; L.sc = L.iv;
  L.gR = take(9 * ng); L.gp = take(3 * ng);
  L.H = take(nv * nv);
  L.an = take(nv);                   // directly after H, as above
  L.rhs0 = take(nv); L.a = take(nv); L.tmp = take(nv); L.tmp2 = take(nv);
  L.csv = take(2 * ns); L.Dr = take(rcap); L.z = take(rcap);
  L.u = take(m.nu > 0 ? m.nu : 1);
  L.xbar = take(nq + nv);
  L.ovl = o;
  L.qn = take(nq); L.vn = take(nv); L.qs = take(nq); L.vs = take(nv);
  L.kv = take(7 * nv); L.ka = take(7 * nv); L.dq = take(nv);
  L.M = take(nv * nv);
  L.ct = take(16 * ns);
  L.J = take(rcap * nv); L.aref = take(rcap); L.s = take(rcap);
  L.xd = take(L.hb * (nv + 1));
  L.nd = (o + 1) & ~1;
  return L;
}

// Offsets (in doubles) of one environment's adjoint workspace (reverse-mode
// adjoint kernel): cotangents of the right-hand side's intermediates, then
// the stage data and cotangents of one Dormand-Prince step.
struct LayoutBar {
  int R, p, cR, cp, S, F, Ic, V, A, Fb, slot, y, jy, cz, cj, q, v, u;   // right-hand side
  int gb, iv, ivb;                   // geom pose cotangents, I V and its cotangent per body
  int sc, tk;                        // hinge sine and cosine, theta-cotangent terms per body
  int qn, vst, dq, dqb, Qs, kab, kvb, Qb, Vb, qnb, vnb, ub, xb;            // one step
  int pr, pd, pa;                    // model parameters: slot records (8 each), bcoef terms per dof, sums
  int nd;                            // doubles per environment (padded to even)
};
constexpr int SLOTBAR = 24;          // at most per slot: pose cotangents of its two geoms (R 9 + p 3 each)

DMX_HD inline LayoutBar make_bar_layout(const DevModel& m, int rcap, bool params = false) {
  LayoutBar B{};
  int o = 0;
  const int nq = m.nq, nv = m.nv, nb = m.nbody, ns = m.nslot > 0 ? m.nslot : 1, nu = m.nu > 0 ? m.nu : 1;
  auto take = [&](int n) { int r = o; o += n; return r; };
  B.R = take(9 * nb); B.p = take(3 * nb); B.cR = take(9 * nb); B.cp = take(3 * nb);
  B.S = take(6 * nv); B.F = take(6 * nv); B.Ic = take(10 * nb);
  B.V = take(6 * nb); B.A = take(6 * nb); B.Fb = take(6 * nb);
  B.slot = take(m.nslotbar > 0 ? m.nslotbar : SLOTBAR * ns);
  B.y = take(nv); B.jy = take(rcap); B.cz = take(rcap); B.cj = take(rcap);
  B.q = take(nq); B.v = take(nv); B.u = take(nu);
  B.gb = take(12 * (m.ngeom > 0 ? m.ngeom : 1)); B.iv = take(6 * nb); B.ivb = take(6 * nb);
  B.sc = take(2 * nb); B.tk = take(9 * nb);
  B.qn = take(nq); B.vst = take(7 * nv); B.dq = take(nv); B.dqb = take(nv); B.Qs = take(nq);
  B.kab = take(6 * nv); B.kvb = take(6 * nv); B.Qb = take(nq); B.Vb = take(nv);
  B.qnb = take(nq); B.vnb = take(nv); B.ub = take(nu); B.xb = take(nq + nv);
  B.pr = B.pd = B.pa = o;
  if (params) { B.pr = take(8 * ns); B.pd = take(nv); B.pa = take(PAR_MU0 + m.npair + m.nbody + m.nbox); }
  B.nd = (o + 1) & ~1;
  return B;
}

}  // namespace dmx
