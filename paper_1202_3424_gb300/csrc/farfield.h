// Far-field amplitude kernels (farfield.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace dda {

// Right-hand sides in groups of NR (1 or 2) consecutive ones that share their
// directions; per group one table of the per-axis phases
//   tabs[(group*Lt + i)*ndp + d], i over the nx, ny and nz lattice indices of the
//   three axes one after another (Lt = nx + ny + nz), d < ndir padded to ndp:
//   exp(-i kd n_a (i_a - c_a)), c_a the lattice centre.
struct FarGeom {
    int nx, ny, nz;  // caller's lattice
    int ndir, ndp;
    int Lt() const { return nx + ny + nz; }
};
inline int far_padded(int ndir) { return (ndir + 127) / 128 * 128; }

// dirs[(group*ndir + d)*3 + a]: the unit vectors.  C = float2 or double2.
template <typename C>
cudaError_t launch_phase_tables(const FarGeom& f, int groups, double kd, const double* dirs, C* tabs, cudaStream_t st);

// F[r][d][a] (zeroed here) = kd^2 ((I - n n) sum_j P[r][.][j] phase_{r,d}(j))_a for groups*NR RHS;
// the sums in C's arithmetic, P rounded to it.
template <typename C>
cudaError_t launch_farfield(const Geom& g, const DevTarget& tg, const FarGeom& f, int groups, int NR, const double2* P,
                            const C* tabs, const double* dirs, double kd, double2* F, cudaStream_t st);

}  // namespace dda
