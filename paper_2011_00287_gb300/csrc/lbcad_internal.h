// lbcad_internal.h -- types shared by the host runtime and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbcad_plan.h"

namespace lbcad {

// D3Q19 velocities (rest, six faces, twelve edges), the order published by
// lbcad_lattice().  constexpr so that fully unrolled loops fold them to immediates.
__host__ __device__ constexpr int lat_c(int i, int a) {
  return a == 0 ? (i == 1 ? 1 : i == 2 ? -1 : i == 7 ? 1 : i == 8 ? -1 : i == 9 ? 1 : i == 10 ? -1
                   : i == 11 ? 1 : i == 12 ? -1 : i == 13 ? 1 : i == 14 ? -1 : 0)
       : a == 1 ? (i == 3 ? 1 : i == 4 ? -1 : i == 7 ? 1 : i == 8 ? -1 : i == 9 ? -1 : i == 10 ? 1
                   : i == 15 ? 1 : i == 16 ? -1 : i == 17 ? 1 : i == 18 ? -1 : 0)
                : (i == 5 ? 1 : i == 6 ? -1 : i == 11 ? 1 : i == 12 ? -1 : i == 13 ? -1 : i == 14 ? 1
                   : i == 15 ? 1 : i == 16 ? -1 : i == 17 ? -1 : i == 18 ? 1 : 0);
}
// |c_i|^2: 0 rest, 1 face, 2 edge.
__host__ __device__ constexpr int lat_c2(int i) {
  return lat_c(i, 0) * lat_c(i, 0) + lat_c(i, 1) * lat_c(i, 1) + lat_c(i, 2) * lat_c(i, 2);
}
__host__ __device__ constexpr double lat_w(int i) {
  return lat_c2(i) == 0 ? 1.0 / 3.0 : lat_c2(i) == 1 ? 1.0 / 18.0 : 1.0 / 36.0;
}

// D3Q15 velocities of the LB populations (Sec. 3, Fig. 1): rest, six faces (as in D3Q19),
// eight corners; opposite velocities in adjacent slots.  Weights 2/9, 1/9, 1/72.
__host__ __device__ constexpr int lat15_c(int i, int a) {
  return i == 0 ? 0
       : i <= 6 ? lat_c(i, a)
       : a == 0 ? ((i == 7 || i == 9 || i == 11 || i == 14) ? 1 : -1)
       : a == 1 ? ((i == 7 || i == 9 || i == 12 || i == 13) ? 1 : -1)
                : ((i == 7 || i == 10 || i == 11 || i == 13) ? 1 : -1);
}
__host__ __device__ constexpr double lat15_w(int i) { return i == 0 ? 2.0 / 9.0 : i <= 6 ? 1.0 / 9.0 : 1.0 / 72.0; }

// Velocity sets of the populations as template arguments (the finite-difference stencils
// use D3Q19 in both cases).
struct VelD3Q19 {
  static constexpr int Q = 19;
  __host__ __device__ static constexpr int c(int i, int a) { return lat_c(i, a); }
  __host__ __device__ static constexpr double w(int i) { return lat_w(i); }
};
struct VelD3Q15 {
  static constexpr int Q = 15;
  __host__ __device__ static constexpr int c(int i, int a) { return lat15_c(i, a); }
  __host__ __device__ static constexpr double w(int i) { return lat15_w(i); }
};

// Per-instance coefficients in the compute type.
template <typename T>
struct Coef {
  T tau_inv, guo, rho0;
  T A0, chi0, chis, K, q0, gammaQ, xi, a, b, kphi, M, W, zeta;
  // products the kernels would otherwise form at every site
  T A0chi1, A0chis;        // A0 (chi0 + chis), A0 chis: A0 chi = A0chi1 + A0chis psi
  T cL, fQ2;               // A0 + 4 K q0^2, A0/2 + 2 K q0^2
  T K2, Kq, W2;            // 2 K, 2 K q0, 2 W
  T ah, bq, kh, zh;        // a/2, b/4, kphi/2, zeta/2
  T xi2, xi23, xi29;       // 2 xi, 2 xi/3, 2 xi/9
  T xip, xim;              // 1 + xi, 1 - xi
  T omc;                   // 1 - 1/tau
  T omw[3], gw3[3], gw9[3];  // per weight class (rest, faces, others): w/tau, 3 w guo, 9 w guo
};

// One instance of a launch: lattice, state buffers of this step parity, scratch.
template <typename T>
struct InstDesc {
  int nx, ny, nz;
  int vel;         // velocity set of the populations: 0 = D3Q19, 1 = D3Q15
  long long N;
  long long blk0;  // first block of this instance in per-site launches
  long long nblk;  // number of blocks of this instance
  const T* g_in;   // post-collision populations of the previous step [19][N]
  T* g_out;
  const T* q_in;   // [5][N]
  T* q_out;
  const T* psi_in; // [N]
  T* psi_out;
  const T* u_in;   // velocity of the previous step [3][N]
  T* u_out;
  T* sig;          // scratch: stress [9][N]
  T* mu;           // scratch: chemical potential [N]
  T* H;            // scratch: molecular field [5][N]
  T* rq;           // staged path, Heun: right-hand side R(Q, psi) at t [6][N] (Q 5, psi 1)
  T* qp;           // staged path, Heun: predicted Q, psi [6][N]
  const T* trig;   // (cos, sin) of 2 pi x/nx, 2 pi y/ny, 2 pi z/nz: [nx + ny + nz][2] (centroid sums)
  Coef<T> c;
};

// Launchers implemented per precision (lbcad_kernels_f32.cu / _f64.cu).
template <typename T, bool SHIFT>
struct Launch {
  static cudaError_t step(const InstDesc<T>* d_desc, int ninst, long long total_blocks, int bs, cudaStream_t s);
  // Staged step: fields -> LB -> order-parameter update (Euler), or fields -> LB ->
  // predictor -> fields at the predicted state -> corrector (Heun).  sync advects with the
  // velocity of this step instead of the previous one.
  // vel: 0 = D3Q19, 1 = D3Q15 populations; form: 0 = whole stress as a body force (Guo),
  // 1 = symmetric stress in the equilibrium, antisymmetric stress as forcing (Eqs. 9-11);
  // stencil: 0 = isotropic D3Q19 finite differences, 1 = fourth-order radius-2 differences.
  static cudaError_t staged(const InstDesc<T>* d_desc, int ninst, long long total_blocks, int bs, bool heun,
                            bool sync, int vel, int form, int stencil, cudaStream_t s);
  static cudaError_t get_fields(const InstDesc<T>& I, uint32_t mask, double* dst, cudaStream_t s);
  static cudaError_t set_fields(const InstDesc<T>& I, uint32_t mask, const double* src, T* g_target,
                                T* q_target, T* psi_target, T* u_target, cudaStream_t s);
  static cudaError_t observables(const InstDesc<T>& I, double* partial, int nblocks, double* out, cudaStream_t s);
};

// One instance as the marching kernels read it: sizes, coefficients, and a pointer to every component of every field.
// The kernels add a 32-bit site number to these pointers; k_march_lb takes only the first component of its
// populations and velocity from here and steps to the others by N (comp in lbcad_march.cuh).
template <typename T>
struct MarchDesc {
  int nx, ny, nz;
  unsigned plane;      // nx ny
  unsigned N;          // sites
  const T* g_in[19];   // as InstDesc, by component
  T* g_out[19];
  const T* q_in[5];
  T* q_out[5];
  const T* psi_in;
  T* psi_out;
  const T* u_in[3];
  T* u_out[3];
  // scratch of the default path: six arrays of pairs [sites][2] (see PairPlane in lbcad_march.cuh) over the planes of
  // the launch, sz0 the first of them; sync coupling and Heun use the first five
  T* S[6];
  int sz0;
  T* H[5];             // sync coupling, Heun: H at t
  T* F[3];             // replay of the adjoint: force
  T* rq[6];            // Heun: right-hand side at t, predicted state (Q, psi), H and mu there
  T* qp[6];
  T* Hp[6];
  const T* trig;       // (cos, sin) of 2 pi x/nx, 2 pi y/ny, 2 pi z/nz
  double mass0;        // N rho0 where the populations are stored shifted, else 0
  Coef<T> c;
};

// The instances of one launch, passed by value: kernels read them from the constant bank.  Read from device
// memory they stay in registers instead (FP32 Euler step at 32^3, 64^3, 128^3 and 256^3: 16.3, 33.9, 192 and 1362 us by
// value; 18.4, 40.7, 238 and 1680 us from device memory).  kPackMany instances fit a launch's argument space; larger
// batches take several launches.
template <typename T, int MI>
struct InstPack {
  MarchDesc<T> d[MI];
};
static_assert(sizeof(InstPack<double, kPackMany>) < 32000, "kernel arguments");

// A work item of a marching kernel: the planes [zb, ze) of one xy tile column of an instance (index within
// the launch).
struct MarchItem {
  int inst, x0, y0, zb, ze;
};

// The items of a launch, in slabs of planes: consecutive items are the tile columns of one slab, so that the
// blocks that run at the same time share the tiles' halos and the rows they straddle in L2.
// early: launched with programmatic dependent launch, for boxes whose step is short.
struct MarchWork {
  const MarchItem* items = nullptr;
  int nitems = 0, grid = 0;
  bool early = false;
};

// A tile shape of the step: tile sizes and resident blocks per SM of its kernels (see lbcad_march.cuh).
struct FusedCfg {
  int fx = 0, fy = 0, lx = 0, ly = 0;          // tiles of k_march_fields, of k_march_lb and the order-parameter kernels
  int fields_per_sm = 0, lb_per_sm = 0;        // k_march_fields, k_march_lb
  int pred_per_sm = 0, op_per_sm[2] = {0, 0};  // sync, Heun: fields at the predicted state, order-parameter kernels
};

// The work of one step for a group of instances (at most kPackMany).
struct StepWork {
  int first = 0, ninst = 0;  // instances of the group
  int sz0 = 0;               // first plane of the scratch
  MarchWork fields, lb, pred, op[2];
};

// What k_march_lb does: collision and psi (kFusedPlain), with the a6 sums (kFusedSums), or the collision
// alone (kFusedLbOnly: sync coupling, Heun); kFusedForce: kFusedPlain, and the force is written (replay of the adjoint).
constexpr int kFusedPlain = 0, kFusedSums = 1, kFusedLbOnly = 2, kFusedForce = 3;

// The FP64 conserved and centroid sums of the step (a6).  Each run of items of one instance that a block works
// on has a slot of 12 partial sums (block b, run j of the block: slot b * maxrun + j);
// slot_inst[slot] is its instance (-1: unused).  At the end of the kernel each block counts its
// slots on their instances (cnt; the kernel resets it), and the block whose count completes an
// instance sums the instance's slots in a fixed order into latest[inst][12]: mass, sum psi,
// momentum (3), sum phi_c cos (3), sum phi_c sin (3), sum phi_c.  Instances are numbered within the launch.
struct FusedObs {
  double* slots;
  const int* slot_inst;
  const int* nslot;    // [ninst] slots of each instance
  const int* slot_lo;  // [ninst] first slot of each instance
  const int* slot_hi;  // [ninst] one past its last slot
  unsigned* cnt;       // [ninst]
  double* latest;      // [ninst][12]
  int maxrun;
  int slot0;  // one instance, in several slabs: slots of the slabs before this one, and of all of them
  int total;
};

// The default path (lbcad_march.cuh), in several tile shapes, for each variant of the LB part:
// variant = (D3Q15 ? 1 : 0) + 2 * (Eq. 9-11 form ? 1 : 0).  prepare returns cudaErrorNotSupported for
// a tile shape the variant does not come in.
template <typename T, bool SHIFT>
struct LaunchFused {
  static int num_configs();
  // many: for launches of several instances
  static cudaError_t prepare(int variant, int k, bool many, bool split, bool heun, FusedCfg* cfg);
  // Euler with the velocity of the previous step; obs: also the a6 sums of the new state (FusedObs).
  // d: the descriptors of the group's instances (host memory, copied into the launch).
  static cudaError_t step(int variant, int k, const StepWork& w, const MarchDesc<T>* d, const FusedObs& ob, bool obs,
                          cudaStream_t s);
  // Sync coupling or Heun: fields, LB half (u of this step), then the order-parameter half: the update
  // (Euler), or predictor, fields at the predicted state and corrector (Heun).
  static cudaError_t split_step(int variant, int k, const StepWork& w, bool heun, bool sync, const MarchDesc<T>* d,
                                cudaStream_t s);
  // The adjoint's replay: one Euler step of D3Q19 with the body force, without the sums, that also leaves its
  // force (MarchDesc::F).
  static cudaError_t prepare_replay(int k);
  static cudaError_t replay(int k, const StepWork& w, const MarchDesc<T>* d, cudaStream_t s);
};

// Buffers of one reverse step of the adjoint (lbcad_adjoint.cuh).
template <typename T>
struct AdjDescHost {
  InstDesc<T> I;                 // state s_t (inputs)
  const T* F;                    // force of the step from it [3][N]
  const T *lg, *lq, *lp, *lu;    // cotangent of s_{t+1}
  T *A, *L, *B;                  // work: kAdjWorkA, kAdjWorkL and kAdjWorkB values per site
  MarchWork work;                // items of k_adj_fields
  T *og, *oq, *op, *ou;          // cotangent of s_t
  double* pgrad;                 // per-block sums over the reverse steps of d/dzeta, d/dq0
};
constexpr int kAdjWorkA = 20, kAdjWorkL = 12, kAdjWorkB = 24;  // (L holds 10, rounded up to whole quads)

template <typename T, bool SHIFT>
struct LaunchAdj {
  static cudaError_t reverse_step(const AdjDescHost<T>& h, cudaStream_t s);
  static cudaError_t seed(const InstDesc<T>& I, const double dX[3], const double ks[3], const double kc[3], T* lp,
                          cudaStream_t s);
  // tile and resident blocks per SM of k_adj_fields
  static cudaError_t fields_shape(int* tx, int* ty, int* per_sm);
  static cudaError_t export_fields(const InstDesc<T>& I, const T* lam, uint32_t mask, double* dst, cudaStream_t s);
};

// Adds the per-block partial sums of 2 values to total[0..1] (fixed order).
cudaError_t adj_accumulate(const double* pgrad, int nblocks, double* total, cudaStream_t s);

// Sets the message that lbcad_last_error(NULL) returns on this thread.
void set_thread_error(const char* msg);

constexpr int kStepBlock = 256;
constexpr int kObsBlock = 256;
constexpr int kObsMaxBlocks = 1024;
constexpr int kObsRowsPerBlock = 32;  // x rows per block of the separate a6 pass (4 per warp)

}  // namespace lbcad
