// chunk_split.h -- how accept_chunks_kernel divides a batch's chunks (1024
// tokens of one target row each, numbered row by row) among warps.  Plain
// integer code, so that it also compiles for the host, where it is checked.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SF_HOST_DEVICE inline
#endif

namespace sf {

// The NW warps that share U chunks: at most one per chunk, so that each of them
// owns at least one (a row's runs are then exactly the warps between its first
// and last chunk's owners), and at most `most`.
SF_HOST_DEVICE int chunk_warps(long long U, long long most) { return static_cast<int>(U < most ? U : most); }

// Warp g's chunks [u0, u1): [g U / NW, (g + 1) U / NW), and none for the warps
// that only fill up the last CTA (g >= NW).
struct ChunkRange {
  int u0, u1;
};

SF_HOST_DEVICE ChunkRange chunk_range(int g, int U, int NW) {
  if (g >= NW) return ChunkRange{U, U};
  return ChunkRange{static_cast<int>(static_cast<long long>(g) * U / NW),
                    static_cast<int>(static_cast<long long>(g + 1) * U / NW)};
}

// The warp owning chunk u: the largest g with g U / NW <= u.
SF_HOST_DEVICE int chunk_owner(int u, int U, int NW) {
  const unsigned long long n = static_cast<unsigned long long>(u + 1) * static_cast<unsigned>(NW) - 1;
  if ((n >> 32) == 0) return static_cast<int>(static_cast<uint32_t>(n) / static_cast<uint32_t>(U));
  return static_cast<int>(n / static_cast<unsigned>(U));
}

}  // namespace sf
