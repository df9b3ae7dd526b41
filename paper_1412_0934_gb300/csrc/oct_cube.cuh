// Indexing of a 4^3 cube of octs in a list in Morton order and of its 6^3-oct neighbourhood, shared by the
// kernel that finds the cubes (octs_build.cu) and the one that steps them (kernels_impl.cuh).
#pragma once
#include <cuda_runtime.h>

namespace hydro {

// Oct t = (c*6 + b)*6 + a of the 6^3 neighbourhood of a cube whose 64 octs are member[] in Morton order:
// the member at (a, b, c) - 1, or a member's neighbour beyond the cube's sides.
__device__ __forceinline__ int cube_slot(int i, int j, int k) {  // Morton index of 0 .. 3 per axis
  return (i & 1) | (j & 1) << 1 | (k & 1) << 2 | (i & 2) << 2 | (j & 2) << 3 | (k & 2) << 4;
}
__device__ __forceinline__ int cube_oct(const int* member, const int* nbr, int t) {
  const int a = t % 6, b = t / 6 % 6, c = t / 36;
  const int i = min(max(a, 1), 4), j = min(max(b, 1), 4), k = min(max(c, 1), 4);
  const int o = __ldg(member + cube_slot(i - 1, j - 1, k - 1));
  return (a == i && b == j && c == k) ? o : __ldg(nbr + 27LL * o + ((c - k + 1) * 3 + b - j + 1) * 3 + a - i + 1);
}

}  // namespace hydro
