// Step records of a taped rollout: what the reverse adjoint's segment recompute
// would otherwise evaluate again.  One record per accepted step: the snapshots
// of its S - 1 stage right-hand sides (the part of the workspace that the VJP
// reads), then the step's row (q_n, the stage velocities V_0..V_6, t_n).
// Records come in chunks of REC_STEPS steps, handed out while the rollout runs
// (the accepted steps are not known before); an environment that finds none
// left goes on without, and the adjoint recomputes those segments.
#pragma once
#include "dmx_model.h"

namespace dmx {

constexpr int REC_STEPS = 8;

// Offsets (doubles) of one stage snapshot: the part of a right-hand-side
// workspace that its VJP reads (poses .. geom frames, the Cholesky factor of
// the final Newton system with the solution, contact records, the used
// Jacobian rows with D and the residuals, then as ints: status, rows,
// slot->row map, row ids, final active set).
struct SnapOff {
  int n1, o2, n2, o3, o4, o5, o6, oi, size;
};
DMX_HD inline SnapOff snap_offsets(const DevModel& m, const Layout& L) {
  SnapOff o{};
  o.n1 = L.gp + 3 * m.ngeom - L.R;
  o.o2 = o.n1;
  o.n2 = L.tmp2 + m.nv - L.H;
  o.o3 = o.o2 + o.n2;
  o.o4 = o.o3 + 18 * m.nslot;          // contact records, then the closest-point parameters (2 per slot)
  o.o5 = o.o4 + L.rcap * m.nv;
  o.o6 = o.o5 + L.rcap;
  o.oi = o.o6 + L.rcap;
  const int nints = 3 + m.nslot + L.rcap + MASKW;
  o.size = (o.oi + (nints + 1) / 2 + 1) & ~1;
  return o;
}
// Doubles of a step's row: q_n, the stage velocities V_0..V_6, t_n.
DMX_HD inline int rev_row_doubles(const DevModel& m) { return m.nq + 7 * m.nv + 1; }

struct StepRecords {
  double* mem;              // [nchunk][REC_STEPS][stride], or null: no records
  int* chunk;               // [B][per_env]: 0 not asked for, -1 none left, else chunk index + 1
  int* next;                // chunks handed out
  int* owner;               // [nchunk][2]: environment and place (step / REC_STEPS) of a chunk
  int nchunk, per_env, stride, snap;   // capacity, table width, doubles per step, per snapshot
};

}  // namespace dmx
