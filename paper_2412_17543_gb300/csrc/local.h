// Subdomain operators of the fast-diagonalization local solver (local.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "device.h"
#include "setup.h"

namespace dd {

// Assembled rows of the local stiffness matrices that touch the interface, in slices of 32
// rows (sliced ELL): pass 1 the interior rows with their interface columns (K_IG), pass 2
// the interface rows with all columns (K_GI, K_GG). Structure per subdomain type (pattern of
// interior, interface and absent nodes), coefficients per subdomain. Positions are those of
// the compact local vector: interface values, then interior values.
struct LocalRowsHost {
  std::vector<int> type;        // [S]
  std::vector<int> trange;      // [types][5]: slices of pass 1, slices of pass 2, first entry of the type in nb
  std::vector<int> sl_w;        // [slices] entries per row
  std::vector<int> sl_off;      // [slices] first entry, from the type's and the subdomain's base
  std::vector<int16_t> sl_out;  // [slices][32] output position (-1: none)
  std::vector<int16_t> sl_cnt;  // [slices][32] entries of the row
  std::vector<int16_t> nb;      // column position per entry, [slice][entry][32]
  std::vector<int64_t> coff;    // [S + 1] first coefficient of each subdomain
  std::vector<double> coef;     // per entry, FP64 sums over the bricks that hold both nodes
  std::vector<std::vector<int>> bnd;  // per type: interior unknowns next to the interface (rows of pass 1)
};
// boundary_only: the interior part of the compact vector holds the unknowns of bnd only (dense
// local solver), else all interior unknowns
LocalRowsHost build_local_rows(const Mesh1& M, const Level& L, bool boundary_only);

// rows of the dense local solver around the product s_B = K_BB t_B (vectors over rows.boff):
// t_B = K_BG x_G, then y_loc = K_GG x_G - K_GB s_B
void launch_rows_interior(const DevMesh& m, const double* xg, double* tB, cudaStream_t s);
void launch_rows_interface(const DevMesh& m, const double* xg, const double* sB, double* yloc, cudaStream_t s);

// mode ELEM_SCHUR: out = y_loc from xg; ELEM_CONDENSE: out = y_loc from f (free-node vector);
// ELEM_RECOVER: out = free-node solution from xg and f
void launch_local_apply(const DevMesh& m, int mode, const double* xg, const double* f, double* out, cudaStream_t s);
// the same for interleaved ensembles: members 0 .. nact - 1 (rounded up to rc = 4 or 8 per CTA; FP64 always 8);
// the other members' outputs are not written
void launch_local_apply_b(const DevMesh& m, int mode, int rc, int nact, const df64* xg, const df64* f, df64* out,
                          cudaStream_t s);

}  // namespace dd
