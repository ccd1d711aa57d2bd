// vm.hpp -- host side of the precompiled eliminated walk: program images and
// kernel entry points.
#pragma once

#include <vector>

#include "elim.hpp"
#include "kernels.hpp"
#include "vm.h"

namespace perm {

// Per-lane slots and per-warp shared memory a program may take (two warps per
// SM at the least).
constexpr int kVmMaxSlotsPerLane = 320;
constexpr int kVmMaxWarpBytes = 100 * 1024;

// Bytes of per-warp shared memory a program needs beyond its image.
size_t vm_slot_area(int img, int limbs, int nslots, int nextra);

// Writes the program image of a planned matrix; img is kImgF64, kImgInt or
// kImgDD, limbs the exact ring (0 otherwise).  False when the program needs
// more than `max_slots` slots.
bool vm_image(const Matrix &m, const ElimPlan &E, int img, int limbs, int max_slots, std::pmr::vector<unsigned char> &out);

// The kernels of one arithmetic (kind as in generic_fns).
GenericFns vm_fns(int kind);

}  // namespace perm
