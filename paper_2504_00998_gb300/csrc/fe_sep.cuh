// Separable preconditioner of the Poisson solve (Section 2.3, K phi = c): interface between the
// solver driver (fe_poisson.cu) and the transforms and iteration (fe_sep.cu).
#pragma once

#include "fe_internal.h"

namespace fe_sep {

// Buffers of one solve on the mesh's stream (n_phi entries each): the iterate, its masked
// residual, three work vectors, the constraint mask, two float work arrays, and room for the
// block partials and the scalars (part_doubles).
struct Buf {
  double *phi, *r, *z, *p, *q;
  const unsigned char* mask;
  float *ta, *tb;
  double* part;
};

// whether the mesh's chains are short enough for the host eigensolver
bool supported(const fe_mesh* m);
size_t part_doubles(const fe_mesh* m);
// Builds the eigenbases for the planes that hold free nodes (cnt[NZ]: free nodes per plane)
// into the mesh's workspace; m->sep_state becomes 1, or 2 when this constraint set has no
// separable form.  Synchronises.
fe_status plan(fe_mesh* m, const double* cnt, bool constant_null);
// CG in double with the separable preconditioner from phi and r until |r|^2 <= tol2, at most
// maxit iterations; *rr is the |r|^2 of the recurrence at return (rounding takes it below that of
// f - K phi).  *lost is set when the iteration stopped making progress or r is outside the
// floats' range, phi then being finite (the caller solves on from phi by other means).
fe_status solve(fe_mesh* m, const Buf& b, double tol2, int maxit, double* rr, int* iters,
                bool* lost);

}  // namespace fe_sep
