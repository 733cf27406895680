// moment_tables.cuh -- compile-time index tables behind the group-of-lanes form of the SMRT
// collision (lane_tables.cuh): where the per-thread code in core.cuh unrolls over the multi-index
// slots at compile time, a lane holds run-time slots.
//   es   the ordered pairs of order-2 slots adding up to each order-4 slot (ES-BGK target)
#pragma once

#include "core.cuh"

namespace smrt {

// Multi-index components and orders of every slot, computed once (the mi_* helpers loop).
template <int N>
struct SlotIndex {
    static constexpr int M = nmom(N);
    int c[M][3] = {};
    int ord[M] = {};
    constexpr SlotIndex() {
        for (int p = 0; p < M; ++p) {
            for (int k = 0; k < 3; ++k) c[p][k] = mi_comp(p, k);
            ord[p] = c[p][0] + c[p][1] + c[p][2];
        }
    }
};

constexpr double fact_small(int n) {
    double v = 1.0;
    for (int i = 2; i <= n; ++i) v *= i;
    return v;
}
// coefficient of x^j in He_n(x) (Appendix B), loop form
constexpr double he_coef_l(int n, int j) {
    if (j > n || ((n - j) & 1)) return 0.0;
    const int l = (n - j) / 2;
    return ((l & 1) ? -1.0 : 1.0) * fact_small(n) / (fact_small(l) * fact_small(j) * double(1 << l));
}

// es: the ordered pairs of order-2 slots adding up to each order-4 slot
template <int N>
struct EsTables {
    static constexpr int M = nmom(N);
    int n[M] = {};
    int q1[M][8] = {};
    int q2[M][8] = {};
    constexpr EsTables() {
        const SlotIndex<N> s;
        for (int p = 0; p < M; ++p) {
            if (s.ord[p] != 4) continue;
            for (int a = ord_off(2); a < ord_off(3); ++a)
                for (int b = ord_off(2); b < ord_off(3); ++b)
                    if (s.c[a][0] + s.c[b][0] == s.c[p][0] && s.c[a][1] + s.c[b][1] == s.c[p][1] &&
                        s.c[a][2] + s.c[b][2] == s.c[p][2]) {
                        q1[p][n[p]] = a;
                        q2[p][n[p]] = b;
                        ++n[p];
                    }
        }
    }
};

}  // namespace smrt
