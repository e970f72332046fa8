// Contraction with the su(3) structure constants, shared by the kinetic-force kernels.
#pragma once

namespace rm {

// G_a += sum_c f_acd rc_c for one column d (d a compile-time constant after unrolling)
template <typename T>
__device__ __forceinline__ void f_contract(int d, const T (&rc)[8], T (&G)[8]) {
    constexpr int tr[9][3] = {{0, 1, 2}, {0, 3, 6}, {0, 4, 5}, {1, 3, 5}, {1, 4, 6},
                              {2, 3, 4}, {2, 5, 6}, {3, 4, 7}, {5, 6, 7}};
    constexpr double fv[9] = {1.0, 0.5, -0.5, 0.5, 0.5, 0.5, -0.5, 0.86602540378443864676, 0.86602540378443864676};
#pragma unroll
    for (int t = 0; t < 9; t++) {
        const int i = tr[t][0], j = tr[t][1], k = tr[t][2];
        const T v = (T)fv[t];
        if (d == k) { G[i] = fma(v, rc[j], G[i]); G[j] = fma(-v, rc[i], G[j]); }
        else if (d == j) { G[k] = fma(v, rc[i], G[k]); G[i] = fma(-v, rc[k], G[i]); }
        else if (d == i) { G[j] = fma(v, rc[k], G[j]); G[k] = fma(-v, rc[j], G[k]); }
    }
}

// the same by rows: G_a = sum_t v_t (RC[c_t][d_t] - RC[d_t][c_t]) over the triples that hold a
struct FTerm { int c, d; double v; };
__constant__ FTerm kFTerms[8][4] = {
    {{1, 2, 1.0}, {3, 6, 0.5}, {4, 5, -0.5}, {0, 0, 0.0}},
    {{2, 0, 1.0}, {3, 5, 0.5}, {4, 6, 0.5}, {0, 0, 0.0}},
    {{0, 1, 1.0}, {3, 4, 0.5}, {5, 6, -0.5}, {0, 0, 0.0}},
    {{6, 0, 0.5}, {5, 1, 0.5}, {4, 2, 0.5}, {4, 7, 0.86602540378443864676}},
    {{5, 0, -0.5}, {6, 1, 0.5}, {2, 3, 0.5}, {7, 3, 0.86602540378443864676}},
    {{0, 4, -0.5}, {1, 3, 0.5}, {6, 2, -0.5}, {6, 7, 0.86602540378443864676}},
    {{0, 3, 0.5}, {1, 4, 0.5}, {2, 5, -0.5}, {7, 5, 0.86602540378443864676}},
    {{3, 4, 0.86602540378443864676}, {5, 6, 0.86602540378443864676}, {0, 0, 0.0}, {0, 0, 0.0}}};

}  // namespace rm
