// Arguments and launchers of the two passes of the matrix-free operator (dg_face.cu, dg_volume.cu).
#pragma once

#include "dg_internal.h"

namespace dg {

// MODE_RES: residual; MODE_RES_LIN: residual that also fills the linearisation cache; MODE_TAN: exact
// Jacobian action. MODE_LINPART: the state-independent linear part of the Jacobian action (viscous
// and BR2 terms, pressure gradient, continuity); no convective product, no Riemann flux, no mass.
enum { MODE_RES = 0, MODE_RES_LIN = 1, MODE_TAN = 2, MODE_LINPART = 3 };

template <class R>
struct OpArgsT {
  MeshDev M;
  const R* in;
  R* out;
  R* face_buf;  // what the face pass hands to the volume pass (face_record)
  R* ubar;      // [ne][3][nq] velocity of the linearisation at the volume points
  R* dFlux;     // [faces][4][nqf][4] Jacobian of the Riemann flux at the face points (see dg_face.cu)
  R nu, eta8;  // viscosity; penalty / 8
  double c, inv_gdt;
  unsigned* status;
  int riemann_its;  // iteration cap of the star-state solve
};
using OpArgs = OpArgsT<double>;

// mode: MODE_*; FP32 passes exist for MODE_TAN only. t: the launch shape.
template <class R>
int face_pass(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st);
template <class R>
int volume_pass(Handle* h, const OpArgsT<R>& a, int mode, const OpTune& t, cudaStream_t st);

// CTAs of a kernel that one SM holds at once, by registers, shared memory and threads (cached per
// kernel and shape); 0: unknown
int resident_ctas(const void* kernel, int threads, size_t smem);

}  // namespace dg
