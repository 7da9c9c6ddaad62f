// FP64 transforms along one axis of the box at compiled edges (interface): the
// full-box FFTs of exact exchange and of the Hartree potential, the density, and
// the FP64 local part of H on boxes that are not cubic.  Each axis is dispatched
// by its own edge, so any combination of the sizes below is covered; kernels in
// fft_axis64_impl.cuh.
//
// All of them are bound by the FP64 pipe (about 0.49 T instructions a second
// measured), so what counts is the number of FP64 instructions: two register
// passes a transform with coprime factors where the edge has them (no twiddles
// between the passes: about 20 FP64 instructions a point at N = 90 against 29 in
// the radix-by-radix passes of the runtime plans), and no separate passes for the
// pair densities and the Coulomb factor: exact exchange of 32 bands on 8 at 90^3 78.4
// -> 57.9 ms.
//   Boxes with another edge (50 among them: as 5 x 10 it has no coprime factors, and
// no workload here has it) run the runtime plans.
#pragma once
#include "common.cuh"

namespace pwh {

#define PWH_AXIS_SIZES_A(X) X(90) X(20) X(64) X(120) X(54)
#define PWH_AXIS_SIZES_B(X) X(144) X(24) X(60) X(100) X(32)
#define PWH_AXIS_SIZES_C(X) X(128) X(30) X(72) X(96) X(36)
#define PWH_AXIS_SIZES_D(X) X(108) X(40) X(80) X(48)

enum AxisOp {
  AX_FWD,    // box <- forward transform
  AX_INV,    // box <- inverse transform
  AX_PAIR,   // box_j <- forward transform of conj(U_j) P
  AX_KERN    // box <- inverse of kern times forward
};
struct AxisArgs {
  double2* box;
  int64_t bstride;
  int nbox;
  int axis;             // 0, 1, 2: lines along i1, i2, i3 (C order, i3 fastest)
  const double2* U;     // AX_PAIR: boxes bstride apart
  const double2* P;     // AX_PAIR
  const double* kern;   // AX_KERN
};

enum PlaneOp {
  PL_YINV,     // sticks -> columns: inverse along y
  PL_XV,       // columns: inverse along x, times V, forward along x
  PL_XDENS,    // columns -> rho += occ |inverse along x|^2
  PL_YFWD      // columns -> sticks: forward along y
};
struct PlaneArgs {
  double2* W;       // sticks, [band][z][stick]
  int64_t wband;
  double2* C;       // columns, [band][z][column][y]
  int bb;           // bands
  const double* V;  // [z][y][x]
  const double* occ;
  int per_slice;    // PL_XDENS: bands a block
  double* rho;      // [z][y][x]
};

// True when edge n has compiled axis kernels.
bool axis64_size(int n);
// Both planar edges (and the z edge) have them.
inline bool axis64_planes(const System& s) {
  return axis64_size(s.n1) && axis64_size(s.n2) && axis64_size(s.n3);
}
// Each launches its kernel (the edge must be a compiled one).
void axis64_box(System& s, AxisOp op, const AxisArgs& a);
void axis64_plane(System& s, PlaneOp op, const PlaneArgs& a);
// z passes of a band batch (PassArgs as the compiled cubic passes): sticks <->
// sphere, FP64.
struct PassArgs;
void axis64_z(System& s, bool inverse, const PassArgs& a);

}  // namespace pwh
