// sf_median_slots.h - which slot holds a window's resident medians, and when a
// consumer warp hands it back (tiled evidence pass), in the kernel and on the host alike.
#pragma once

#include <stdint.h>

#include "sf_host_device.h"

namespace sf {

// Window i of a CTA's range (0, 1, ...) lives in slot i % slots, as the slot's
// (i / slots)-th phase.
struct MedianPlace {
  int slots;  // 1 or 2
  SF_HOST_DEVICE uint32_t slot(int i) const { return slots == 2 ? static_cast<uint32_t>(i) & 1u : 0u; }
  SF_HOST_DEVICE uint32_t parity(int i) const { return static_cast<uint32_t>(slots == 2 ? i >> 1 : i) & 1u; }
};

// A consumer warp's place among the windows.  `wait(i)` waits for window i's medians;
// `arrive(i)` is the warp's one arrival on the `done` barrier of its slot, which the
// producer refills when every warp has arrived.  A wait knows a phase by its parity
// and a barrier counts arrivals, not warps, so both hold only for a warp that takes
// the windows one by one, those without a step of its own included: a wait for the
// slot's second phase passes before the first one has begun, and an arrival ahead of
// the phase before it stands in for a warp that still reads that one.
struct MedianWalk {
  int at = -1;  // window the warp is in
  template <typename Arrive, typename Wait>
  SF_HOST_DEVICE void enter(int i, Arrive arrive, Wait wait) {
    while (at < i) {
      if (at >= 0) arrive(at);
      wait(++at);
    }
  }
  // After the warp's last step; `last` is the range's last window.  Hands back the
  // windows whose slot takes another one, and no window that nothing follows.
  template <typename Arrive, typename Wait>
  SF_HOST_DEVICE void leave(int last, int slots, Arrive arrive, Wait wait) {
    enter(last + 1 - slots, arrive, wait);
  }
};

}  // namespace sf
