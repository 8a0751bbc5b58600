// Rules that choose between kernels, as plain host functions: they can be checked without a GPU.
#pragma once

// Whether the gathers take five threads per atom (which add a stencil's z-planes in another order than one
// thread does): while they make at most one wave of the GPU's thread slots, 2,048 an SM (wide gather, one -> five: 9.8
// -> 6.1 us at 648 atoms, 10.0 -> 7.9 at 12,288, 11.9 -> 11.1 at 22,969; 14.2 -> 21.2 at 96,000). In the fixed-point
// mode, whose results are the same to the bit on every device, the line is that of 152 SMs whatever the device.
inline bool gather_five(long atoms, int sm_count, bool fixed) { return 5 * atoms <= 2048L * (fixed ? 152 : sm_count); }
