// Step records of a taped rollout: what the reverse adjoint's segment recompute
// would otherwise evaluate again.  One record per accepted step: the snapshots
// of its S - 1 stage right-hand sides (the part of the workspace that the VJP
// reads), then the step's row (q_n, the stage velocities V_0..V_6, t_n).
// Every environment has records for its first `steps` steps; the adjoint
// recomputes the segments beyond.  A kept and a recomputed segment differ in the
// last bits where a contact row lies at the edge of the active set (the start of
// the Newton search decides there), so which ones are kept depends on the step
// and the size of the buffer alone, never on the order in which environments run.
#pragma once
#include "dmx_model.h"

namespace dmx {

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
// Offset (ints) of the final active set in a snapshot.
DMX_HD inline int snap_active(const DevModel& m, const Layout& L) {
  return 2 * snap_offsets(m, L).oi + 3 + m.nslot + L.rcap;
}
// Doubles of a step's row: q_n, the stage velocities V_0..V_6, t_n.
DMX_HD inline int rev_row_doubles(const DevModel& m) { return m.nq + 7 * m.nv + 1; }

struct StepRecords {
  double* mem;              // [steps][B][stride], or null: no records
  int steps, B;             // steps of every environment that have a record
  int stride, snap;         // doubles per step, per snapshot
  int active;               // offset (ints) of the final active set in a snapshot
};

}  // namespace dmx
