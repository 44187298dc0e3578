// Parameter block and launcher of the adjoint kernel (dmx_adjoint.cu).
#pragma once
#include <cuda_runtime.h>

#include "dmx_model.h"
#include "dmx_record.h"

namespace dmx {

struct AdjParams {
  const DevModel* model;
  Layout L;
  LayoutBar LB;           // reverse-mode kernel: cotangent workspace
  int B, NI, K, cfd;
  int method;             // METHOD_* integration scheme of the taped rollout
  const double* ckpt;     // [ncheck][nx+1][B] tape checkpoints (state, time)
  const double* hlog;     // [max_steps][B] accepted step sizes
  const int* tape_n;      // [B] accepted steps
  const double* ctrl;     // [NI][nu][B] controls of the taped rollout
  const double* T;        // [B] horizons
  const double* xT_bar;   // [nx][B]
  const double* xb_bar;   // [NI+1][nx][B] or null
  double* x0_bar;         // [nx][B]
  double* ctrl_bar;       // [NI][nu][B] or null
  double* segbuf;         // per warp (tangent) or group (reverse): recomputed steps of a segment
  double* snapbuf;        // reverse mode: per group, K steps x (S - 1) stage snapshots of SN doubles (or null)
  int SN;                 // doubles per snapshot
  StepRecords rec;        // records of the taped rollout
  double* cfdsnap;        // with cfd: snapshots of F~ at the stage states of ncfd recorded steps, or null
  int ncfd;
  int* cfdofs;            // [B + 1] first of an environment's steps among them (k_cfd_offsets)
  int kind;               // MODEL_* type of the kernels (OneBody: 8, 16, 32 lanes, PlaneOnly: 16, 32)
  int per, barofs;        // reverse mode: doubles per environment, offset of the cotangent workspace
  double* p_bar;          // [np][B] model-parameter gradients, or null
  int np;                 // model parameters differentiated when p_bar is set
  const int* touched;     // [B] or null (every environment): the reverse-mode kernel takes the environments whose
                          // taped steps met a contact, the tangent kernel the others
  int* queue;             // [2] next environment, next recorded step (cfd)
};

cudaError_t launch_adjoint(const AdjParams& P, int blocks, cudaStream_t st);
// out[k] = sum over e of x[k][e] (k < n, e < B): one block per row, fixed order.
cudaError_t launch_row_sums(const double* x, int n, int B, double* out, cudaStream_t st);
// d (translational inverse weight of every body at qpos0) / d (parameter
// pdir) into dinvw[nbody]; ws: Layout(rcap).nd derivative scalars (16 bytes)
// + ni ints of device memory, scratch: nq + 2 nv derivative scalars.
cudaError_t launch_body_invweight_tangent(const DevModel* m, const double* qpos0, int rcap, int pdir, void* ws,
                                          void* scratch, double* dinvw, cudaStream_t st);
// reverse-mode kernel, G lanes per environment (G = 2, 4, 8, 16, 32; with model
// parameters, P.p_bar set / par: 8, 16, 32)
cudaError_t launch_adjoint_rev(int G, const AdjParams& P, int blocks, int threads, size_t smem, cudaStream_t st);
int adjoint_rev_occupancy(int G, bool par, int kind, int threads, size_t smem);
cudaError_t launch_eval_rhs_vjp(int G, const AdjParams& P, const double* q, const double* v, const double* u,
                                const double* abar, double* qbar, double* vbar, double* ubar, int* status, int threads,
                                size_t smem, cudaStream_t st);
int adjoint_warps_per_block();
int adjoint_workspace_limit();
int adjoint_int_limit();

}  // namespace dmx
