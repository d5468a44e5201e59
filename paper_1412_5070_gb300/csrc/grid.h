// grid.h -- building and sharing of the auxiliary grids (auxgrid.cuh).
#pragma once

#include <memory>
#include <vector>

#include <cuda_runtime.h>

#include "termlist.h"

namespace f12grid {

// The grids of one factor pair on one device: per class (2..6; 5 uses 3's) the
// cells, and per cell whether it reproduces the quadrature it was built from
// at a corner.  Immutable once built; contexts with the same factor share it.
struct AuxGrid {
  int device = 0;
  std::vector<f12::TermList> key;       // the kernels, by class
  double *cells[7] = {nullptr};         // device
  unsigned char *ok[7] = {nullptr};     // device, per cell
  std::vector<unsigned char> ok_host[7];
  double *xt = nullptr;                 // device: grid_point's values of every cell of xi
  size_t bytes = 0;
  AuxGrid() = default;
  AuxGrid(const AuxGrid &) = delete;
  AuxGrid &operator=(const AuxGrid &) = delete;
  ~AuxGrid();
};

// The grid of the kernels kt[2..6] (entry 5 unused) on the current device
// `device`, for the classes of `want`: an existing one of the same kernels if
// a context still holds it, else built now on `st` (which is synchronised).
// Classes the grid does not serve have null cells.  Null when the device
// memory for it is not there; the caller then evaluates directly.
std::shared_ptr<const AuxGrid> acquire(int device, const f12::TermList kt[7], const bool want[7], cudaStream_t st);

// Whether every cell of class cls that exponents xi in [xi_lo, xi_hi] and
// distances up to dmax can reach is there and in order.
bool covers(const AuxGrid &g, int cls, double xi_lo, double xi_hi, double dmax);

}  // namespace f12grid
