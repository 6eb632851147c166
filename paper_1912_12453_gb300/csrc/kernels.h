// Host-side launchers of the device kernels (element.cu, vector.cu).
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "chns_internal.h"

namespace chns {

template <typename T>
void launch_prep(const chns_mesh *m, const double *Un, const double *Uo, T *ut, T *dl, cudaStream_t st);
// F(U_new; U_old) with the constrained rows; E: the element-local buffer
void launch_residual(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo, const double *f,
                     const double *bc, double *E, double *F, cudaStream_t st);
// J.w with schedule `variant` (-1: the mesh's tuned schedule for float,
// schedule 0 for double); see element.cu for the schedules.  nv directions at
// a time: w and y hold nv vectors one after another, E nv element-local buffers
constexpr int kJacvecVariants = 7;
template <typename T>
void launch_jacvec(const chns_mesh *m, const PhysCoef &pc, const T *ut, const T *dl, const T *w, T *E, T *y,
                   cudaStream_t st, int variant = -1, int nv = 1);
// y = J w (float) at (U_new, U_old) without a preparation; false: not for this
// mesh, nothing launched
bool launch_jacvec_states(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo, const float *w,
                          float *E, float *y, cudaStream_t st);
// r = b - J x (r given), or one block-Jacobi sweep x += B (b - J x) with the
// nodal blocks B; E: the element-local buffer
template <typename T>
void launch_jacvec_defect(const chns_mesh *m, const PhysCoef &pc, const T *ut, const T *dl, const T *b, const T *B,
                          T *E, T *x, T *r, cudaStream_t st);
void launch_tau_floor_count(const chns_mesh *m, const PhysCoef &pc, const double *Un, const double *Uo,
                            unsigned long long *count, cudaStream_t st);
// x (the second of the six vectors of n_nodes doubles at v) = M^-1 (node sums of
// the element-local slots E), M the scalar Q1 mass matrix, by conjugate gradients
// in one cooperative kernel; part: cg_partials() doubles, ctr: zero.  Status in
// *s on the device: err 1: M not positive, 2: a grid barrier was given up, after `polls` polls (0: the
// default, about 20 s)
struct CgState {
  int err, its;
};
int cg_partials();
cudaError_t launch_cg(const chns_mesh *m, const PhysCoef &pc, double *E, double *v, double *part, unsigned *ctr,
                      CgState *s, int max_it, int polls, cudaStream_t st);
// the chemical-potential row of U into element-local slots (n_elem * 2^dim doubles)
void launch_mu_row(const chns_mesh *m, const PhysCoef &pc, const double *U, double *E, cudaStream_t st);
constexpr int kEnergyBlocks = 152 * 4;  // most blocks of the energy kernel
int64_t energy_blocks(const chns_mesh *m);
// per-instance element coefficients of a batched (union) mesh
chns_status upload_coef_tables(chns_mesh *m, const std::vector<PhysCoef> &pcs, cudaStream_t st);
chns_status copy_coef_tables(const chns_mesh *src, chns_mesh *dst);
// out3 (device): energy, integral of phi, volume with phi < 0; partial: 3 *
// energy_blocks(m) doubles
void launch_energy(const chns_mesh *m, const PhysCoef &pc, const double *U, double *partial, double *out3,
                   cudaStream_t st);

}  // namespace chns
