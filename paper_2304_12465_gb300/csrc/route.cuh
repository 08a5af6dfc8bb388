// Which kernel a float32 product launches (host only).
#pragma once

namespace krr {

enum ProductRoute { kRouteNone = -1, kRouteTcgen05 = 0, kRouteFma = 1, kRouteMmaSync = 2 };

// path: the process's choice (krr_set_product_path: 0 tcgen05, 1 FMA, 2
// mma.sync); tc5, mma, fma: the operands that the points were prepared with.
// The choice can change between the preparation and a product of the same
// solve, and the preparation builds only what its own choice needs, so a
// product takes the chosen kernel when it has operands and another that has
// them otherwise: never one without (its pointers would be NULL).
inline ProductRoute product_route(int path, bool tc5, bool mma, bool fma) {
  if (path == 0 && tc5) return kRouteTcgen05;
  if (path != 1 && mma) return kRouteMmaSync;
  if (fma) return kRouteFma;
  if (tc5) return kRouteTcgen05;
  return mma ? kRouteMmaSync : kRouteNone;
}

}  // namespace krr
