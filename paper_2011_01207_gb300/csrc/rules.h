// Rules that choose between kernels, and the places of the pair lists, as plain functions: they can be checked
// without a GPU.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define AP_HD __host__ __device__ __forceinline__
#else
#define AP_HD inline
#endif

#define AP_CHUNK 640               // candidate atoms of a block staged in shared memory at once
#define AP_LIST_PER_TILE 528       // capacity of the pair lists, entries per tile: 32 candidates x 16 target
                                   // pairs, and the padding of a chunk's 16 lists spread over its tiles
#define AP_LIST_PER_BLOCK 256

// Block I, whose tiles start at tile0, may have 32 mult candidates a tile (mult images an atom can appear in).
// Its lists start at entry
AP_HD size_t list_entry_base(int tile0, int I, int mult) {
    return (size_t)tile0 * mult * AP_LIST_PER_TILE + (size_t)I * AP_LIST_PER_BLOCK;
}
// and the places of its chunks' lists at
AP_HD size_t list_meta_base(int tile0, int I, int mult) { return ((size_t)tile0 * mult) / (AP_CHUNK / 32) + I; }
// chunks of n candidates, and the candidates of each but the last
AP_HD int list_chunks(int n) { return (n + AP_CHUNK - 1) / AP_CHUNK; }
AP_HD int list_chunk_size(int n) { return n ? (n + list_chunks(n) - 1) / list_chunks(n) : 0; }
// Warp w of the list kernel takes every fourth of a block's nt tiles, from tile w on: the first tile of its
// segment when the warps' tiles are laid one warp after the other
AP_HD int segment_tile(int nt, int w) { return w * (nt >> 2) + (w < (nt & 3) ? w : nt & 3); }
// While a block's lists are made, its candidates' masks (16 bytes each, eight entries) lie at the end of the room of
// its nt tiles, from this entry on. Chunk after chunk the masks are read and the lists written from the start; lists
// of as many entries as there can be reach no mask that is still to be read (tests/test_rules.py).
AP_HD size_t list_mask_base(int nt, int mult) {
    return (size_t)nt * mult * (AP_LIST_PER_TILE - 8 * 32) + AP_LIST_PER_BLOCK;
}

// Whether the gathers take five threads per atom (which add a stencil's z-planes in another order than one
// thread does): while they make at most one wave of the GPU's thread slots, 2,048 an SM (wide gather, one -> five: 9.8
// -> 6.1 us at 648 atoms, 10.0 -> 7.9 at 12,288, 11.9 -> 11.1 at 22,969; 14.2 -> 21.2 at 96,000). In the fixed-point
// mode, whose results are the same to the bit on every device, the line is that of 152 SMs whatever the device.
inline bool gather_five(long atoms, int sm_count, bool fixed) { return 5 * atoms <= 2048L * (fixed ? 152 : sm_count); }
