// Red/black SOR on A u = -rho for one box or many (gcv.cu, batch_gcv.cu).
#pragma once

#include <vector>

#include "internal.h"

namespace coulps {

// One box of a solve.  u and r are held colour by colour, rows of Wh sites
// (site x of a row at h = x >> 1) and one zero element, and a ghost row and
// plane of zeros at either end: element (z, y, h) of colour c at
// off + c * colour + ((z + 1) (Ly + 2) + y + 1) Ws + h.  A neighbour outside
// the box is then always a zero in memory (h = -1 is the previous row's zero).
struct SorBox {
  int Lx, Ly, Lz, Wh, Ws;
  long long off, colour;
  long long nat;  // first element in the natural-order arrays (x fastest)
  double a, b;    // u' = a u + b (S - rho): 1 - omega, omega / 6
};

// A box with its arrays from element `off` / natural-order element `nat` on.
SorBox sor_box(int Lx, int Ly, int Lz, long long off, long long nat);
inline long long sor_elems(const SorBox &b) { return 2 * b.colour; }

// A site's charge: element in the split arrays, in natural order, and value.
struct SorCharge {
  long long at, nat;
  double q, bq;  // charge, omega / 6 times it
};

// Appends box `b`'s charges (sites (x, y, z) and q, n of them), one entry per
// site with the charges of a site added in input order.
void sor_charges(const SorBox &b, int64_t n, const int32_t *sites, const double *q,
                 std::vector<SorCharge> &out);

// Solves every box: n_iter iterations from u = 0 (colour 0, then colour 1).
// Leaves u and the density in natural order in u_nat and rho_nat; works in
// split arrays and lists of its own from `alloc`, or where these do not fit in
// u_nat and rho_nat themselves (slower, the same u).  Synchronises s once (the
// host lists' uploads).
cudaError_t sor_solve(const std::vector<SorBox> &boxes, const std::vector<SorCharge> &charges,
                      int n_iter, double *u_nat, double *rho_nat, const Allocator &alloc,
                      cudaStream_t s);

}  // namespace coulps
