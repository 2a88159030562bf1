// The turns of the 3D residual + full weighting (k_resrestrict3 in kernels_mg.cu).  A block's warps
// march its fine planes; once per coarse plane every warp stores into a shared plane and one of
// R3_TURNS groups of warps sums it.  For the c-th coarse plane of the block (c = 0, 1, ...) a warp
//   1. stores its part of shared plane r3_plane(c);
//   2. arrives at named barrier 1 + r3_turn(c), and waits there only if that is its own group's turn
//      (r3_turn(c) == r3_group(warp));
//   3. in its own turn reads the whole shared plane.
// A store into a shared plane must come after every read of what it held before.  The reader of plane c
// arrives at the barriers c + 1, c + 2, ... after its read, so the storing warp has to have waited in a
// turn between the two uses: with a period of P shared planes, in one of c + 1 .. c + P - 1.  A group's turns
// are R3_TURNS apart, so P = R3_TURNS + 1 is the least that gives every group such a turn; with P = R3_TURNS the
// reading group itself has none (its own turns are c and c + P), and one of its warps could store while
// another still reads.
// No CUDA here: the host compiles it too, to check that order for every pair of warps.
#pragma once

#ifdef __CUDACC__
#define R3_HD __host__ __device__ __forceinline__
#else
#define R3_HD inline
#endif

constexpr int R3_TURNS = 4;              // groups of warps, and named barriers 1 .. R3_TURNS
constexpr int R3_PLANES = R3_TURNS + 1;  // shared planes

R3_HD int r3_group(int warp) { return (warp >> 2) % R3_TURNS; }
R3_HD int r3_turn(int c) { return c % R3_TURNS; }
R3_HD int r3_plane(int c) { return c % R3_PLANES; }
