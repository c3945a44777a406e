// What a CTA still has in flight when it leaves after an expired wait (internal).
// Table images streamed through two shared-memory slots by bulk copies (sliced_hx.cu):
// Step i of a CTA uses image i: slot i & 1, phase i >> 1 of that slot's mbarrier; its MMAs complete
// phase i of the MMA barrier. A wait on a parity whose phase is not the next one returns at once,
// so whoever waits for a copy has to name the step it belongs to.
#pragma once

#include <cstdint>

namespace cs {

__host__ __device__ constexpr int image_slot(int step) { return step & 1; }
__host__ __device__ constexpr uint32_t image_parity(int step) {
  return (uint32_t)(step >> 1) & 1u;
}
__host__ __device__ constexpr uint32_t mma_parity(int step) { return (uint32_t)step & 1u; }

// One barrier whose phases are requested and waited for in turn, the parity moving on after each
// wait: the phase that a wait has just given up.
__host__ __device__ constexpr uint32_t given_up(uint32_t next_parity) { return next_parity ^ 1u; }

// Before a CTA frees its tensor memory and exits after `step` steps and `issued` images: waits for
// the last step's MMAs and image, whose own waits may have expired, and for the images requested
// ahead. Without an expired wait nothing is open and every wait would return at once.
template <class WaitImage, class WaitMma>
__host__ __device__ void settle_images(int step, int issued, WaitImage image, WaitMma mma) {
  for (int i = step > 0 ? step - 1 : 0; i < issued; ++i) image(image_slot(i), image_parity(i));
  if (step > 0) mma(mma_parity(step - 1));
}

}  // namespace cs
