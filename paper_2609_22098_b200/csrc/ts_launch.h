// The rule by which cooperative kernels are chained to the kernel before them.
#pragma once

namespace ts {

// launch(true) asks for a cooperative launch with programmatic stream serialization, launch(false) for a cooperative one
// only; both return an error code, 0 = launched.  A driver that does not take the two together is asked once: `refused`
// remembers it.  A launch that fails either way says nothing about the pair (an invalidated capture, too few SMs).
template <typename Launch>
inline auto launch_chained(int& refused, Launch launch) -> decltype(launch(true)) {
  using E = decltype(launch(true));
  if (!refused) {
    const E e = launch(true);
    if (e == E(0)) return e;
  }
  const E e = launch(false);
  if (e == E(0)) refused = 1;
  return e;
}

}  // namespace ts
