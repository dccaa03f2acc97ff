// line_pair_shapes.h -- the plane shapes (axis 2 x axis 3) the line-pair chain is compiled for: every
// pair of the lengths below within a factor of 1.5 of each other (any pair up to 32) whose plane fits in
// shared memory.
// Run-time shapes were tried (one kernel that selects the stages by length): twice the time per point
// (80^3: 6.4 against 3.4 ms, 100 x 108 x 90: 20.7 against 10.7 ms).  Other grids take the five pencil
// passes of pair_chain.cuh.  125 is not among the lengths: its plane passes have not been compiled or measured
// (128 orbitals on 125^3 take 183 ms in pencil passes).  The shapes make 32 objects and most of a library of 90 MB.
#pragma once

#define ACE_LP_PLANE_LENGTHS(X)                                                                             \
  X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60)      \
  X(64) X(72) X(75) X(80) X(81) X(90) X(96) X(100) X(108) X(120) X(128) X(135) X(144) X(150) X(160)
