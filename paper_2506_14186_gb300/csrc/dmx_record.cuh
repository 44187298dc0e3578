// Device side of the step records (dmx_record.h): saving a right-hand side's
// workspace, and finding an environment's record of a step.
#pragma once
#include "dmx_device.cuh"
#include "dmx_record.h"

namespace dmx {

// dst[i] = src[i], i < n, eight loads in flight per lane (the snapshots live in
// device memory: one round trip per eight passes instead of one per pass).
template <int G>
__device__ __forceinline__ void copy_run(const Grp<G>& g, const double* __restrict__ src, double* __restrict__ dst,
                                         int n) {
  for (int i0 = g.lane; i0 < n; i0 += 8 * G) {
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k * G < n) x[k] = src[i0 + k * G];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k * G < n) dst[i0 + k * G] = x[k];
  }
}
// Workspace of the right-hand side just evaluated (status st) -> snapshot dst.
template <int G, class MD>
__device__ void snap_save(const Grp<G>& g, const MD& m, const Ws& w, double* dst, int st) {
  const Layout& L = *w.L;
  const SnapOff o = snap_offsets(m, L);
  const int nr = (st == ENV_ROW_OVERFLOW) ? 0 : w.i[L.slotrow + m.nslot];
  const double* d = w.d;
  DMX_TASKS(i, o.n1) dst[i] = d[L.R + i];
  DMX_TASKS(i, o.n2) dst[o.o2 + i] = d[L.H + i];
  DMX_TASKS(i, 16 * m.nslot) dst[o.o3 + i] = d[L.ct + i];
  DMX_TASKS(i, 2 * m.nslot) dst[o.o3 + 16 * m.nslot + i] = d[L.csv + i];
  DMX_TASKS(i, nr * m.nv) dst[o.o4 + i] = d[L.J + i];
  DMX_TASKS(i, nr) { dst[o.o5 + i] = d[L.Dr + i]; dst[o.o6 + i] = d[L.z + i]; }
  int* di = reinterpret_cast<int*>(dst + o.oi);
  if (g.lane == 0) { di[0] = st; di[1] = nr; }
  for (int i = g.lane; i <= m.nslot; i += G) di[2 + i] = w.i[L.slotrow + i];
  DMX_TASKS(i, nr) di[3 + m.nslot + i] = w.i[L.rowid + i];
  DMX_TASKS(i, MASKW) di[3 + m.nslot + L.rcap + i] = w.i[L.amask + i];
}
// Record of step n of an environment, null when there is none.  A step's
// records of all environments lie side by side: environments proceed at about
// the same pace, so what is written at a time spans few pages.
__device__ __forceinline__ double* step_record(const StepRecords& r, int env, int n) {
  return n < r.steps ? r.mem + ((size_t)n * r.B + env) * r.stride : nullptr;
}

}  // namespace dmx
