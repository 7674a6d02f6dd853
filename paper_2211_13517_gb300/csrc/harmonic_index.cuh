// Index arithmetic of the top-harmonic indexed sum, shared by its kernels:
// harmonic j of H of the cell (ir, iz), o = iz - iz0, reads the cell
//     (iz0 + src_off(H, o, j),  (ir j + H/2)/H).
#pragma once

namespace fdas {

__host__ __device__ constexpr int ilog2h(int n) { return n <= 1 ? 0 : 1 + ilog2h(n >> 1); }

// harmonic visited at position idx of the stage order
__host__ __device__ constexpr int j_at(int H, int idx) {
    return idx == 0 ? H : ((2 * (idx - (1 << ilog2h(idx))) + 1) * H) >> (ilog2h(idx) + 1);
}

__host__ __device__ constexpr int src_off(int H, int o, int j) {
    return o < 0 ? -(((-o) * j + H / 2) / H) : ((o * j + H / 2) / H);
}

}  // namespace fdas
