// Host launchers of the elementwise / reduction kernels (kernels.cu).
#pragma once

#include <cuda_runtime.h>
#include "internal.h"

namespace pt {

constexpr int kSlotMax = 20;   // deepest Anderson history (a multiple of four)
struct SlotList {
  int k;                       // valid entries
  int s[kSlotMax];             // history slots, oldest first
};

cudaError_t density(const double2* psi_r, long N, int ne, double* rho, cudaStream_t s);
cudaError_t density32(const float2* psi_r, long N, int ne, double* rho, cudaStream_t s);
cudaError_t rho_to_complex(const double* rho, double2* buf, long N, cudaStream_t s);
// the local potential from the Hartree potential vh_c (real parts; null without Hartree)
cudaError_t assemble_vloc(const double2* vh_c, const ConvSink& sink, long N, cudaStream_t s);
cudaError_t ion_potential(double* v, Grid3 g, const double* cell, const double* d_atoms, int na, double depth,
                          double sigma, cudaStream_t s);
cudaError_t hartree_factor(double* f, Grid3 g, const double* cell, cudaStream_t s);
cudaError_t half_step(const double2* psi, const double2* R, double hdt, double2* out, long n, cudaStream_t s);
cudaError_t precond_step(double2* x, const double2* R, const double* kin, int npw, long n, double tau, cudaStream_t s);
// r (holding r_prev) <- -(x + i hdt T - ph); dx = x - xp and dr = r - r_prev when have_prev
cudaError_t residual_push(const double2* x, const double2* T, const double2* ph, double hdt, const double2* xp,
                          double2* r, void* dx, void* dr, long n, int have_prev, int f32, cudaStream_t s);
// out = sum |r|^2; part: 1024 doubles
cudaError_t norm2(const double2* r, long n, double* part, double* out, cudaStream_t s);
// gram entries of the new slot and gamma per band; part: at least 8 * 4 * sl.k * ne doubles
cudaError_t anderson_gamma(const void* dR, long slot_stride, const SlotList& sl, int newslot, const double2* r,
                           int npw, int ne, int mdim, double2* gram, double2* gamma, void* part, int f32,
                           cudaStream_t s);
// out = x + beta r - sum_q gamma_q (dX_q + beta dR_q)
cudaError_t anderson_update(const double2* x, const double2* r, const void* dX, const void* dR, long slot_stride,
                            const SlotList& sl, const double2* gamma, int mdim, int npw, long n, double beta, int f32,
                            double2* out, cudaStream_t s);
cudaError_t kinetic_shifted(const double* gk3, int npw, double ax, double ay, double az, double* kin, cudaStream_t s);
cudaError_t rho_change(const double* a, const double* b, long N, double* part, double* out, cudaStream_t s);
// out8: [0] sum vion rho, [1] sum vh rho, [2] sum rho^{4/3}, [3..5] sum r rho,
//       [6] sum kin |c|^2, [7] Re tr(negM)   (grid sums without the dV factor)
cudaError_t energy_sums(const double* rho, const double* vion, const double* vh, int use_h, Grid3 g, const double* cell,
                        const double2* c, const double* kin, int npw, int ne, const double2* negM, double* part,
                        double* out8, cudaStream_t s);
cudaError_t axpy(double2 a, const double2* x, double2* y, long n, cudaStream_t s);
cudaError_t diff_to_complex(const double* a, const double* b, double2* buf, long N, cudaStream_t s);
cudaError_t add_real(const double2* buf, double* a, long N, cudaStream_t s);
cudaError_t kerker_factor(double* f, Grid3 g, const double* cell, double b, double q0, cudaStream_t s);

}  // namespace pt
