// FP64 axis transforms: dispatch by edge over the translation units.
#include "fft_axis64.cuh"

#include "fft_spec.cuh"

namespace pwh {

#define PWH_AXIS_DECLARE(u)                                              \
  bool ax_has_##u(int n);                                                \
  bool ax_box_##u(System&, int n, AxisOp, const AxisArgs&);              \
  bool ax_plane_##u(System&, int n, PlaneOp, const PlaneArgs&);          \
  bool ax_z_##u(System&, int n, bool inverse, const PassArgs&);
PWH_AXIS_DECLARE(a)
PWH_AXIS_DECLARE(b)
PWH_AXIS_DECLARE(c)
PWH_AXIS_DECLARE(d)

static void missing() { throw Error{PWH_ERR_ARG, "FP64 axis transform needs a compiled edge"}; }

bool axis64_size(int n) { return ax_has_a(n) || ax_has_b(n) || ax_has_c(n) || ax_has_d(n); }
void axis64_box(System& s, AxisOp op, const AxisArgs& a) {
  const int n = a.axis == 0 ? s.n1 : a.axis == 1 ? s.n2 : s.n3;
  if (!ax_box_a(s, n, op, a) && !ax_box_b(s, n, op, a) && !ax_box_c(s, n, op, a) &&
      !ax_box_d(s, n, op, a))
    missing();
}
void axis64_plane(System& s, PlaneOp op, const PlaneArgs& a) {
  const int n = op == PL_YINV || op == PL_YFWD ? s.n2 : s.n1;
  if (!ax_plane_a(s, n, op, a) && !ax_plane_b(s, n, op, a) && !ax_plane_c(s, n, op, a) &&
      !ax_plane_d(s, n, op, a))
    missing();
}
void axis64_z(System& s, bool inverse, const PassArgs& a) {
  const int n = s.n3;
  if (!ax_z_a(s, n, inverse, a) && !ax_z_b(s, n, inverse, a) && !ax_z_c(s, n, inverse, a) &&
      !ax_z_d(s, n, inverse, a))
    missing();
}

}  // namespace pwh
