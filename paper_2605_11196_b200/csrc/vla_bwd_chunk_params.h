// Parameters of the chunked backward pass (vla_bwd_chunk.cuh), shared with the host code.
#pragma once

#include <stdint.h>

namespace vla {

struct BwdChunkParams {
  // the caller's tensors (flags: layout and reading)
  const void *q, *k, *v, *u;
  const float *S0, *d_out, *dS_T, *dA_T, *dz_T;
  float *dq, *dk, *dv, *du, *dS0, *dz0;
  // left by the A pass: [units, T, D], [units, T], [units, nch, D], per block operand image and scale, final A
  float *alpha, *zeta, *delta, *an, *zkc, *Asc, *A_T;
  unsigned char* Aimg;
  // per chunk: operand images, Tm and H; per token: 1 / scale of q, 1 / den, ||phi(k)||
  unsigned char *opK, *opQ, *opA;
  float *small, *qsi, *iden, *nrm;
  // e_t; S at block starts, its adjoint at block ends (images, a scale per 16 rows)
  float *e, *Ssc, *Dsc;
  unsigned char *Simg, *Dimg;
  // g_t, gradient of den_t, per block sums of the penalty side [D, D] and of dden q [D]
  float *g, *dden, *X, *Y, *XT, *XT2;
  // largest entries of X per block and of XT per unit; inverse scales of X's images (kept in Simg)
  float *Xmax, *XTmax, *Xsc;
  int* status;
  int T, units, nch, NB, heads;
  uint32_t flags, wait_limit;
  float eps;
};

}  // namespace vla
