// Allocation with one retry (host only).
#pragma once

namespace krr {

// alloc() until it returns `ok`: once, and once more after trim() has given memory
// back to the system (false: there was none to give, and the first error stands).
template <typename Err, typename Alloc, typename Trim>
Err alloc_or_trim(Err ok, Alloc alloc, Trim trim) {
  const Err e = alloc();
  if (e == ok || !trim()) return e;
  return alloc();
}

}  // namespace krr
